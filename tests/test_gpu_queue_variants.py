"""The queue's launch against the launches per iteration, for every association
variant and storage type: batches of one pair more than a team launch takes.
The same bits in every pose, count and trace.
"""
import os
import re

import pytest

from tests import test_gpu_team as TT

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module", autouse=True)
def _built():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1802_03980_gb300 import build
    build()


def _most_team_pairs():
    with open(os.path.join(ROOT, "paper_1802_03980_gb300", "csrc", "kf_internal.cuh")) as f:
        return int(re.search(r"constexpr int kTeamMaxPairs = (\d+);", f.read()).group(1))


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("kw", [
    {}, dict(cos_angle_min=0.9), dict(shoot_radius=2, normal_mode=1), dict(shoot_radius=1, cos_angle_min=0.8),
    dict(hist_bins=1), dict(hist_bins=1023, band_kappa=0.5), dict(hist_bins=4096, band_kappa=1.25)],
    ids=lambda kw: "-".join(kw) or "projective")
def test_queue_equals_per_iteration_launches(kw, precision):
    sizes = ([(160, 120), (97, 75), (161, 123), (64, 48)] * 16)[:_most_team_pairs() + 1]
    pairs = TT._pairs(sizes, empty=(5,))
    queue = TT._run(7, pairs, 3, (5, 4, 3), 2, precision=precision, **kw)
    assert queue[0] == queue[1]
    assert queue[0] == TT._run(7 | 16, pairs, 3, (5, 4, 3), 1, precision=precision, **kw)[0]

"""kf_debug_wait_timeout after an alignment that ended with too few matches: the
counts that it left behind are not taken for the empty launch's own.
"""
import numpy as np
import pytest

from oracle import kf_oracle as O
from synth import scenes as S
from tests import kfhelp as H

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1802_03980_gb300 import build
    build()


def test_the_wait_runs_out_after_an_alignment_without_matches():
    k = H.kf()
    pr = S.config2_kinect(64, 160, 120)
    p, _ = H.params(levels=2, caps=(3, 3))
    with H.Tracker(p, 160, 120) as t:
        t.set_pair(pr)
        want = t.align(pr)
        t.set_pair(pr, depth=np.zeros_like(pr.depth))
        assert t.align(pr)[0] == O.TOO_FEW_INLIERS
        assert k.kf_debug_wait_timeout(t.h, 20.0) == k.KF_ERR_TIMEOUT
        t.set_pair(pr)
        got = t.align(pr)
        assert want[0] == got[0] and (want[1] == got[1]).all()

"""Trackers of different histogram sizes in one process: a tracker with the most
bins goes on as before after one with few was created, through the team launch,
the queue and the launches per iteration, for both storage types.
"""
import os
import re

import numpy as np
import pytest

from tests import kfhelp as H
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


def _align(trk, pairs):
    st, poses, res = H.kf().kf_align_batch(
        [t.h for t in trk], np.stack([pr.prior_R for pr in pairs]),
        np.stack([pr.init_pose for pr in pairs]), [pr.lam for pr in pairs])
    return st, poses.tolist(), [bytes(r) for r in res]


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("launch", ["team", "queue", "iterations"])
def test_a_small_histogram_leaves_a_large_ones_launches_alone(launch, precision):
    k = H.kf()
    n = _most_team_pairs() + 1 if launch == "queue" else 2
    pairs = TT._pairs([(64, 48), (97, 75)] * ((n + 1) // 2))[:n]
    flags = 7 | (k.KF_LAUNCH_PER_ITERATION if launch == "iterations" else 0)

    def trackers(bins):
        p, _ = H.params(levels=2, caps=(3, 3), flags=flags, hist_bins=bins, precision=precision)
        trk = [H.Tracker(p, pr.K.width, pr.K.height) for pr in pairs]
        for t, pr in zip(trk, pairs):
            t.set_pair(pr)
        return trk

    alone = []
    for bins in (4096, 16):
        trk = trackers(bins)
        try:
            alone.append(_align(trk, pairs))
        finally:
            for t in trk:
                t.close()
    large, small = trackers(4096), trackers(16)
    try:
        for _ in range(2):
            assert _align(large, pairs) == alone[0]
            assert _align(small, pairs) == alone[1]
    finally:
        for t in large + small:
            t.close()

"""The FP64 solve and pose update of one iteration against numpy.

band_kappa 0.5 gives a band that does not start at bin 0, so the iteration and
kf_debug_reduce take the same way over the same rows: the hook's sums are the
ones the iteration solved, and H x = g can be checked to the solver's own
rounding.
"""
import math

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


@pytest.mark.parametrize("lam", [0.0, 5.0, 1e3, 1e12])
@pytest.mark.parametrize("rot_deg", [2.0, 25.0])
def test_increment_and_update_are_the_systems_solution(lam, rot_deg):
    k = H.kf()
    K = S.Intrinsics(160, 120, 140.0, 140.0, 80.0, 60.0)
    pr = S.make_pair(S.room_scene(), K, S.rng_for(1, 7), rot_deg, 0.03, 0.5)
    # unseeded: the start is off by the whole motion, so large increments occur
    p, op = H.params(levels=1, caps=(1,), flags=O.USE_FILTER, band_kappa=0.5, d_max=1.0)
    with H.Tracker(p, 160, 120) as t:
        t.set_pair(pr)
        _, pose, _ = t.align(pr, lam=lam, prior=False)
        (rec,) = k.kf_debug_trace(t.h)
        assert rec.klo > 0
        sums = k.kf_debug_reduce(t.h, 0, pr.init_pose, rec.klo, rec.khi)
    assert int(sums[27]) == rec.n
    A = np.zeros((6, 6))
    A[np.triu_indices(6)] = sums[:21]
    A = A + np.triu(A, 1).T
    A[:3, :3] += 2.0 * lam * rec.n * np.eye(3)
    x = np.array(rec.x[:])
    # backward error of the elimination: a few dozen roundings of 2^-53
    resid = np.abs(A @ x - sums[21:27])
    scale = np.abs(A) @ np.abs(x) + np.abs(sums[21:27])
    assert (resid <= 64 * 2.0 ** -53 * scale).all(), (resid / scale)
    # the update, to the rounding of its few products of numbers of order one
    want = O.apply_increment(x, pr.init_pose)
    assert np.abs(pose - want).max() < 1e-14, (np.linalg.norm(x[:3]), math.degrees(np.linalg.norm(x[:3])))

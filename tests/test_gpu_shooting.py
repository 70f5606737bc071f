"""Normal shooting at the edges of its candidate groups against the oracle:
every window radius, images smaller than a window or a warp, windows that leave
the image on each side, and holes: matched pixel, bin and histogram bit for bit.
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


@pytest.mark.parametrize("w,size", [(1, (40, 30)), (2, (8, 6)), (2, (47, 33)), (2, (100, 75)), (3, (47, 33)),
                                    (4, (8, 6)), (4, (61, 40))])
def test_windows_at_the_border_match_the_oracle(w, size):
    pr = S.config2_kinect(31, *size)
    holes = np.random.default_rng(w).random(pr.model_vertex.shape[:2]) < 0.05
    pr.model_vertex[holes] = np.nan
    p, op = H.params(levels=2, caps=(2, 2), shoot_radius=w)
    with H.Tracker(p, *size) as t:
        t.set_pair(pr)
        fr, mo = H.oracle_levels_from_gpu(t, pr, 2)
        T0 = O.seed_pose(pr.prior_R, pr.init_pose, op)
        for l in range(2):
            for shift in ((0.0, 0.0), (0.3, 0.2), (-0.3, -0.2)):   # windows over each side of the image
                T = O.apply_increment(np.r_[0.0, 0.0, 0.0, shift, 0.0], T0)
                idx, b, hist = H.kf().kf_debug_associate(t.h, l, T, fr[l].V.shape[:2], p.hist_bins)
                a = O.associate(fr[l], mo[l], T, O.f32_transforms(T, pr.model_pose), op)
                want = np.where(a.valid, a.vi * mo[l].cam.width + a.ui, -1)
                assert np.array_equal(idx, want), (l, shift)
                assert np.array_equal(b, np.where(a.valid, a.k, -1)), (l, shift)
                assert np.array_equal(hist.astype(np.int64), O.histogram(a, p.hist_bins)), (l, shift)

"""The front end's instances against the oracle: each number of levels with the
default filter radius, and the radii that share an instance, on images that end
one pixel into or before a 32-pixel tile, with holes and depths on the border.

Bars as for the other front-end comparisons: the filter within its float32
rounding, the pyramid on the device's own level above with its decisions exact
and its mean within three float32 roundings of the largest depth, the
back-projected vertices bit for bit.
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


@pytest.mark.parametrize("levels,radius,size", [
    (1, 2, (33, 31)), (2, 2, (67, 65)), (3, 2, (131, 97)), (4, 2, (129, 72)), (4, 2, (200, 161)),
    (4, 4, (65, 80)), (3, 0, (64, 36)), (2, 1, (97, 33)), (1, 3, (40, 47)), (3, 4, (95, 100))])
def test_frontend_instances_match_oracle_stages(levels, radius, size):
    pr = S.config2_kinect(21, *size)
    dep = pr.depth.copy()
    rng = np.random.default_rng(levels * 8 + radius)
    dep[rng.random(dep.shape) < 0.1] = 0.0
    dep[0, ::3], dep[-1, 1::3], dep[2::3, 0] = np.inf, -1.0, np.nan
    p, op = H.params(levels=levels, caps=(2,) * levels, bilateral_radius=radius)
    with H.Tracker(p, *size) as t:
        t.set_pair(pr, depth=dep)
        lv = t.frame_levels(levels)
    cams = O.frame_level_cams(O.Cam(*pr.K.as_tuple()), levels)
    Db = O.bilateral_filter(dep, op.bilateral_sigma_s, op.bilateral_sigma_r, radius)
    assert ((lv[0][0] > 0) == (Db > 0)).all()
    assert np.abs(lv[0][0] - Db).max() < 5e-6
    for l, (D, V, N) in enumerate(lv):
        if l > 0:
            Dd = O.downsample(lv[l - 1][0], op.bilateral_sigma_r)
            assert ((D > 0) == (Dd > 0)).all(), l
            assert np.abs(D - Dd).max() <= 3 * 2.0 ** -24 * 4 * float(Dd.max()), l
        V32 = O.vertex_map32(D, cams[l])
        No = O.normal_map(O.vertex_map(D, cams[l]), V32)
        ok = np.isfinite(V32).all(-1) & np.isfinite(No).all(-1)
        assert (np.isfinite(V).all(-1) == ok).all(), l
        assert (np.isfinite(N).all(-1) == ok).all(), l
        assert (V[ok] == V32[ok]).all(), l

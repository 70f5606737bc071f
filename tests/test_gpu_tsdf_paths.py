"""The volume's short ways against its general ones, bit for bit.

The raycast leaps over bricks that hold no observed value <= 0, unless a ray
has more than 65536 samples: a z_far far behind the cube asks for the same
samples with and without leaps. The integration uses branch-free divisions
unless a pose entry is tiny but not zero: 1e-30 in place of a zero changes no
rounded sum and takes the general division.
"""
import numpy as np
import pytest

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


def _volume(k, res, side, origin, mu):
    p = k.kf_volume_default_params()
    p.res, p.side, p.mu = res, side, mu
    for a in range(3):
        p.origin[a] = origin[a]
    return k.kf_volume_create(p, 0)


def _frame(seed, w, h, pose):
    rng = S.rng_for(9, seed)
    K = S.kinect_intrinsics(w, h)
    return K.as_tuple(), S.render_depth(S.room_scene(), pose, K, rng, outliers=0.1, dropout=0.05)


# (res, side, origin, mu, frame size, ray step): whole and ragged bricks and superbricks, one brick
@pytest.mark.parametrize("res,side,origin,mu,size,dz", [
    (9, 4.0, (-2.0, -2.0, 0.5), 0.9, (67, 45), 0.1),
    (64, 4.5, (-2.3, -1.8, 0.2), 0.25, (160, 120), 0.05),
    (131, 5.0, (-2.5, -2.0, -0.5), 0.12, (161, 119), 0.03),
])
def test_leaps_and_short_divisions_change_no_bit(res, side, origin, mu, size, dz):
    k = H.kf()
    path = [S.look_at((0.1 * i, -0.05 * i, 0.1), (0.2 * i - 0.2, 0.1, 3.0)) for i in range(4)]
    frames = [_frame(i, *size, T) for i, T in enumerate(path)]
    vols = [_volume(k, res, side, origin, mu) for _ in range(2)]
    try:
        for (K, D), T in zip(frames, path):
            tiny = np.where(T == 0.0, 1e-30, T)
            tiny[3] = T[3]
            assert (tiny != T).any()
            D = np.ascontiguousarray(D)
            for v, pose in zip(vols, (T, tiny)):
                k.kf_volume_integrate(v, D.ctypes.data, K, pose, False)
        (F0, W0), (F1, W1) = (k.kf_volume_read(v, res) for v in vols)
        assert (F0 == F1).all() and (W0 == W1).all() and (W0 > 0).any()
        # seen from the path, from outside the cube and along its floor
        views = path + [S.look_at((-4.0, 0.3, 2.0), (1.0, 0.0, 2.2)), S.look_at((-1.2, 0.9, 1.0), (1.5, 1.1, 3.0)),
                        S.look_at((0.3, 0.2, 7.0), (0.0, 0.0, 2.0))]
        hits = 0
        for T in views:
            for near in (0.05, 0.6):
                far = near + dz * 1000
                V, N = k.kf_volume_raycast(vols[0], frames[0][0], T, near, far, dz)
                Vg, Ng = k.kf_volume_raycast(vols[0], frames[0][0], T, near, near + dz * 70000, dz)
                assert np.array_equal(V, Vg, equal_nan=True) and np.array_equal(N, Ng, equal_nan=True)
                hits += int(np.isfinite(V).all(-1).sum())
        assert hits > 0
    finally:
        for v in vols:
            k.kf_volume_destroy(v)

"""A volume's first integration of a device frame inside a stream capture: the
call queues kernels only, so the replayed graph gives the field of a direct
call. Frames of one tile of depths, of many, and beyond the largest number of
tiles that a volume holds."""
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


@pytest.mark.parametrize("size", [(16, 16), (161, 119), (65536, 272)])
def test_a_captured_first_integration_equals_a_direct_one(size):
    import torch
    k = H.kf()
    w, h = size
    T = S.look_at((0.1, -0.1, 0.0), (0.0, 0.1, 3.0))
    depth = S.render_depth(S.room_scene(), T, S.kinect_intrinsics(160, 120), S.rng_for(9, 3), outliers=0.1, dropout=0.05)
    K = S.kinect_intrinsics(160, 120)
    # the same view at any size: pixels repeated, intrinsics scaled
    depth = depth[np.arange(h) * 120 // h][:, np.arange(w) * 160 // w]
    K = (w, h, K.fx * w / 160, K.fy * h / 120, K.cx * w / 160, K.cy * h / 120)
    D = torch.from_numpy(np.ascontiguousarray(depth, np.float32)).cuda()
    p = k.kf_volume_default_params()
    p.res, p.side, p.mu = 41, 4.5, 0.3
    p.origin[0], p.origin[1], p.origin[2] = -2.3, -1.8, 0.2
    s = torch.cuda.Stream()
    torch.cuda.synchronize()
    vols = [k.kf_volume_create(p, s.cuda_stream) for _ in range(2)]
    try:
        k.kf_volume_integrate(vols[0], D.data_ptr(), K, T, True)
        torch.cuda.synchronize()
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=s):
            k.kf_volume_integrate(vols[1], D.data_ptr(), K, T, True)
        with torch.cuda.stream(s):
            g.replay()
        torch.cuda.synchronize()
        (F0, W0), (F1, W1) = (k.kf_volume_read(v, p.res) for v in vols)
        assert (F0 == F1).all() and (W0 == W1).all() and (W0 > 0).any()
    finally:
        for v in vols:
            k.kf_volume_destroy(v)

"""Batches of page-locked host frames over several front-end launches, each
copying the next one's frames: the maps of device frames, bit for bit. Groups
that end at the frame limit and at the pixel limit, a large group after tiles
too few to copy it with one layer of blocks, frames off a 16-byte boundary, and
pageable frames between page-locked ones.
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


@pytest.mark.parametrize("sizes,pageable,off", [
    ([(37, 33)] * 33 + [(1280, 960), (64, 48)], (), ()),
    ([(640, 480)] * 9, (4, 8), (1, 5)),
    ([(1280, 960), (31, 29), (1280, 960), (333, 251)], (1,), (0, 3))])
def test_pulled_batches_equal_device_frames(sizes, pageable, off):
    import torch
    k = H.kf()
    p, _ = H.params(levels=2, caps=(2, 2))
    pairs = [S.config2_kinect(90 + i % 5, *sz) for i, sz in enumerate(sizes)]
    host = [np.ascontiguousarray(pr.depth, np.float32).reshape(-1) for pr in pairs]
    maps = {}
    for mode in ("device", "host"):
        trk = [H.Tracker(p, *sz) for sz in sizes]
        try:
            keep, ptrs = [], []
            for i, f in enumerate(host):
                if mode == "device":
                    b = torch.from_numpy(f).cuda()
                    ptrs.append(b.data_ptr())
                elif i in pageable:
                    b = f
                    ptrs.append(f.ctypes.data)
                else:  # off: one float past the buffer's boundary
                    b = torch.from_numpy(np.r_[np.zeros(int(i in off), np.float32), f]).pin_memory()
                    ptrs.append(b.data_ptr() + 4 * int(i in off))
                keep.append(b)
            torch.cuda.synchronize()
            k.kf_set_frame_batch([t.h for t in trk], ptrs, [pr.K.as_tuple() for pr in pairs],
                                 k.KF_FRAME_DEVICE if mode == "device" else k.KF_FRAME_HOST)
            torch.cuda.synchronize()
            maps[mode] = [t.frame_levels(2) for t in trk]
        finally:
            for t in trk:
                t.close()
    for a, b in zip(maps["device"], maps["host"]):
        for la, lb in zip(a, b):
            for x, y in zip(la, lb):
                assert np.array_equal(x, y, equal_nan=True)

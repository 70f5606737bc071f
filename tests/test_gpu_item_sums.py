"""The sum over work items at large item counts.

kf_reduce_noalloc with one valid pixel per item: an item's products of the
normal's components are then single rounded float32 products, and their sum over
the items is known exactly. And the largest frames that a team takes, whose sums
fold, against the launches per iteration.
"""
from fractions import Fraction

import numpy as np
import pytest

from tests import kfhelp as H
from tests import test_gpu_team as TT

pytestmark = pytest.mark.gpu

ITEM = 4096  # frame pixels


@pytest.fixture(scope="module", autouse=True)
def _built():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1802_03980_gb300 import build
    build()


@pytest.mark.parametrize("items", [1, 9, 75, 320, 321, 1024])
@pytest.mark.parametrize("signed", [True, False])
def test_the_sum_over_items_is_as_near_as_a_float64_one(items, signed):
    import torch
    k = H.kf()
    rng = np.random.Generator(np.random.PCG64(7 * items + signed))
    w, h = 4096, items
    fv = np.full((h * w, 3), np.nan, np.float32)
    fv[::ITEM, 2] = 1.0
    # every item's pixel looks at a model pixel of its own
    mw, mh = 64, 16
    u, v = np.arange(items) % mw, np.arange(items) // mw
    fv[::ITEM, 0] = (u - 32) / np.float32(64.0)
    fv[::ITEM, 1] = (v - 8) / np.float32(64.0)
    n = rng.normal(size=(items, 3))
    if not signed:
        n = np.abs(n)
    n = (n * 10.0 ** rng.uniform(-3, 2, (items, 1))).astype(np.float32)
    mv = np.full((mh * mw, 3), np.nan, np.float32)
    mn = np.zeros((mh * mw, 3), np.float32)
    mv[v * mw + u] = fv[::ITEM]
    mn[v * mw + u] = n
    dev = [torch.from_numpy(np.ascontiguousarray(x)).cuda() for x in (fv, mv, mn)]
    sums = torch.zeros(29, dtype=torch.float64, device="cuda")
    torch.cuda.synchronize()
    eye = np.eye(4)
    st = k.kf_reduce_noalloc(dev[0].data_ptr(), w, h, dev[1].data_ptr(), dev[2].data_ptr(),
                             (mw, mh, 64.0, 64.0, 32.0, 8.0), eye, eye, 0.16, 512, 0, 511,
                             sums.data_ptr(), torch.cuda.current_stream().cuda_stream)
    assert st == k.KF_OK
    torch.cuda.synchronize()
    got = sums.cpu().numpy()
    assert got[27] == items
    # upper-triangle places of the normal's products: rows 3, 4, 5
    at = {(3, 3): 15, (3, 4): 16, (3, 5): 17, (4, 4): 18, (4, 5): 19, (5, 5): 20}
    for (r, c), place in at.items():
        terms = n[:, r - 3] * n[:, c - 3]  # float32, rounded once
        exact = sum(map(Fraction, map(float, terms)))
        big = float(np.abs(terms).max())
        running = float(np.abs(np.cumsum(terms.astype(np.float64))).max())
        # a float64 sum: one rounding of the running sum an addition, their
        # errors of either sign
        bound = np.sqrt(items) * 2.0 ** -53 * max(big, running)
        err = abs(float(Fraction(float(got[place])) - exact))
        assert err <= bound, (r, c, err / big, bound / big)


def test_a_large_team_adds_as_the_launches_per_iteration():
    pairs = TT._pairs([(2048, 1152)])  # 576 items
    assert TT._run(7, pairs, 2, (2, 2), 1)[0] == TT._run(7 | 16, pairs, 2, (2, 2), 1)[0]

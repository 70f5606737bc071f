"""Team launches of two trackers on two streams at the same time, from two
threads: each alignment's bits are those of the tracker on its own."""
import threading

import pytest

from tests import kfhelp as H
from tests import test_gpu_team as TT

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1802_03980_gb300 import build
    build()


@pytest.mark.parametrize("sizes", [[(640, 480), (640, 480)], [(640, 480), (161, 123)]])
def test_two_trackers_at_the_same_time_change_no_bit(sizes):
    p, _ = H.params()
    pairs = TT._pairs(sizes)
    trk = [H.Tracker(p, *sz) for sz in sizes]  # each with a stream of its own
    try:
        for t, pr in zip(trk, pairs):
            t.set_pair(pr)

        def once(i):
            st, pose, res = trk[i].align(pairs[i])
            return st, pose.tolist(), bytes(res)

        alone = [once(i) for i in range(2)]
        got = [[], []]

        def run(i):
            for _ in range(100):
                got[i].append(once(i))

        threads = [threading.Thread(target=run, args=(i,)) for i in range(2)]
        for th in threads:
            th.start()
        for th in threads:
            th.join()
        for i in range(2):
            assert got[i] == [alone[i]] * 100
    finally:
        for t in trk:
            t.close()

"""Workers of a team launch that come late to a message.

A worker without half items at the pair's level only waits for the next
message, and the leader does not wait for it, so it may sleep through messages
and has to go on from the one it finds. A build whose idle workers sleep some
60 us between two looks (an iteration takes about 9) misses several in every
alignment: the same bits as the ordinary build's, and no time-out. The last
case runs more iterations than there are rotating histograms; its bits are also
those of the launches per iteration, which have none.
"""
import json
import os
import subprocess
import sys

import numpy as np
import pytest

from synth import scenes as S
from tests import kfhelp as H

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

# batches whose coarse levels leave workers without items; flags
CASES = [([(640, 480)], 3, (10, 5, 4), 7), ([(1280, 960)], 4, (4, 3, 3, 2), 7),
         ([(640, 480), (333, 251), (160, 120)], 3, (10, 5, 4), 7),
         ([(640, 480), (160, 120)], 3, (19, 9, 11), 3)]

CHILD = r"""
import json, sys
sys.path.insert(0, {root!r})
from tests.test_gpu_team_late import alignments
print("RESULT " + json.dumps(alignments()))
"""


def alignments(cases=CASES):
    k = H.kf()
    out = []
    for sizes, levels, caps, flags in cases:
        p, _ = H.params(levels=levels, caps=caps, flags=flags)
        pairs = [S.config2_kinect(60 + i, *sz) for i, sz in enumerate(sizes)]
        trk = [H.Tracker(p, *sz) for sz in sizes]
        try:
            for t, pr in zip(trk, pairs):
                t.set_pair(pr)
            for _ in range(8):
                st, poses, res = k.kf_align_batch(
                    [t.h for t in trk], np.stack([pr.prior_R for pr in pairs]),
                    np.stack([pr.init_pose for pr in pairs]), [pr.lam for pr in pairs])
                out.append([int(st), poses.tolist(), [bytes(r).hex() for r in res]])
        finally:
            for t in trk:
                t.close()
    return out


def test_workers_that_sleep_through_messages_change_no_bit(tmp_path):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1802_03980_gb300 import build
    build()
    lib = build(defines=["KF_TEAM_IDLE_NS=60000"], out=str(tmp_path / "libkftrack_late.so"))
    r = subprocess.run([sys.executable, "-c", CHILD.format(root=ROOT)], cwd=ROOT,
                       env=dict(os.environ, KF_TRACK_LIB=lib), capture_output=True, text=True, timeout=600)
    assert r.returncode == 0, r.stderr[-2000:]
    late = json.loads([x for x in r.stdout.splitlines() if x.startswith("RESULT ")][-1][len("RESULT "):])
    assert late == alignments()
    sizes, levels, caps, flags = CASES[-1]
    general = alignments([(sizes, levels, caps, flags | H.kf().KF_LAUNCH_PER_ITERATION)])
    assert late[-8:] == general

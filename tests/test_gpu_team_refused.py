"""A team launch that the device refuses (its blocks cannot all be resident, as in
a context with a part of the SMs): the call goes through the queue, with the
same bits. The build under test counts on 64 blocks an SM, so that the runtime
refuses the larger of its launches.
"""
import json
import os
import subprocess
import sys

import pytest

from tests import test_gpu_team as TT

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

CHILD = r"""
import json, sys
sys.path.insert(0, {root!r})
from tests.test_gpu_team_refused import alignments
print("RESULT " + json.dumps(alignments()))
"""


def alignments():
    out = []
    # refused (600 and 900 half items), then one that fits
    for sizes in ([(1280, 960)], [(640, 480)] * 6, [(320, 240)]):
        for st, poses, res, _ in TT._run(7, TT._pairs(sizes), 3, (5, 4, 3), 3):
            out.append([int(st), poses, [r.hex() for r in res]])
    return out


def test_a_refused_team_launch_goes_through_the_queue(tmp_path):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1802_03980_gb300 import build
    build()
    lib = build(defines=["KF_TEAM_PER_SM=64"], out=str(tmp_path / "libkftrack_many.so"))
    r = subprocess.run([sys.executable, "-c", CHILD.format(root=ROOT)], cwd=ROOT,
                       env=dict(os.environ, KF_TRACK_LIB=lib), capture_output=True, text=True, timeout=600)
    assert r.returncode == 0, r.stderr[-2000:]
    refused = json.loads([x for x in r.stdout.splitlines() if x.startswith("RESULT ")][-1][len("RESULT "):])
    assert refused == alignments()

"""The guarded build (-DKF_CHECKED) on batches that take the team launch.

Every form of tests/test_gpu_team.py, run by a child process that loads the
guarded library: no guard fires (one that did would turn the status into
KF_ERR_INTERNAL), and every bit is the unguarded build's.
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
from tests.test_gpu_checked_team import alignments
print("RESULT " + json.dumps(alignments()))
"""


def alignments():
    out = {}
    for name, (sizes, levels, caps, kw) in TT.CASES.items():
        st, poses, res, trace = TT._run(7, TT._pairs(sizes), levels, caps, 1, **kw)[0]
        out[name] = [int(st), poses, [r.hex() for r in res], [[list(x) for x in t] for t in trace]]
    return out


def test_no_guard_fires_in_a_team_launch(tmp_path):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1802_03980_gb300 import build
    build()
    lib = build(defines=["KF_CHECKED"], out=str(tmp_path / "libkftrack_checked.so"))
    r = subprocess.run([sys.executable, "-c", CHILD.format(root=ROOT)], cwd=ROOT,
                       env=dict(os.environ, KF_TRACK_LIB=lib), capture_output=True, text=True, timeout=600)
    assert r.returncode == 0, r.stderr[-2000:]
    checked = json.loads([x for x in r.stdout.splitlines() if x.startswith("RESULT ")][-1][len("RESULT "):])
    assert checked == json.loads(json.dumps(alignments()))

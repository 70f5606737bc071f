"""The tuner times the kernel that its knobs shape (no GPU): every knob of the
default grid belongs to the queue's launch, and a batch of any size takes it.
"""
import os
import re

import pytest

from paper_1802_03980_gb300 import tune

CSRC = os.path.join(os.path.dirname(tune.__file__), "csrc")


def _source(name):
    with open(os.path.join(CSRC, name)) as f:
        return f.read()


def test_default_knobs_are_the_queue_launch_s_own():
    # kf_icp.cu holds the queue and its ring; the register gathers' knobs are in
    # the header that the other launches share
    text = _source("kf_icp.cu")
    for name in tune.GRID:
        assert f"#ifndef {name}\n" in text, name


@pytest.mark.parametrize("pairs", [1, 6, 16, 17, 64])
def test_a_timed_batch_is_too_large_for_a_team(pairs):
    most = int(re.search(r"kTeamMaxPairs = (\d+);", _source("kf_internal.cuh")).group(1))
    of = tune.queue_batch(pairs)
    assert len(of) > most and len(of) >= pairs
    assert of[:pairs] == list(range(pairs)) and set(of) == set(range(pairs))

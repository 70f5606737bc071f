"""The team launch of small batches against the per-iteration launches (the
general path): the same bits in every pose and count, over the forms it
accepts, at the edges of its work split: one item, ragged items, one and two
half items a worker, teams that share the device, every storage type and
association variant, the fewest and most bins, and a pair that stops early.
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


def _run(flags, pairs, levels, caps, again, **kw):
    k = H.kf()
    p, _ = H.params(levels=levels, caps=caps, flags=flags, **kw)
    trk = [H.Tracker(p, pr.K.width, pr.K.height) for pr in pairs]
    try:
        for t, pr in zip(trk, pairs):
            t.set_pair(pr)
        out = []
        for _ in range(again):
            st, poses, res = k.kf_align_batch(
                [t.h for t in trk], np.stack([pr.prior_R for pr in pairs]),
                np.stack([pr.init_pose for pr in pairs]), [pr.lam for pr in pairs])
            out.append((st, poses.tolist(), [bytes(r) for r in res],
                        [[(r.level, r.N, r.kmed, r.khi, r.n, r.passes, r.w0, r.w1) for r in k.kf_debug_trace(t.h)]
                         for t in trk]))
        return out
    finally:
        for t in trk:
            t.close()


def _pairs(sizes, empty=()):
    out = [S.config2_kinect(60 + i, *sz) for i, sz in enumerate(sizes)]
    for i in empty:
        out[i].depth = np.zeros_like(out[i].depth)
    return out


CASES = {
    "one_item": ([(64, 48)], 1, (5,), {}),
    "ragged": ([(333, 251)], 3, (10, 5, 4), {}),
    "full_frame": ([(640, 480)], 3, (10, 5, 4), {}),
    "two_halves_a_worker": ([(1280, 960)], 4, (4, 3, 3, 2), {}),
    "fp16_gate": ([(640, 480), (161, 123)], 3, (10, 5, 4), dict(precision=1, cos_angle_min=0.9)),
    "shooting": ([(320, 240), (97, 75)], 2, (4, 3), dict(shoot_radius=2, normal_mode=1)),
    "shooting_gate_fp16": ([(97, 75)], 2, (4, 3), dict(shoot_radius=1, cos_angle_min=0.8, precision=1)),
    "shared_device": ([(640, 480), (333, 251), (160, 120), (640, 480)], 3, (10, 5, 4), {}),
    "one_bin": ([(160, 120)], 2, (3, 3), dict(hist_bins=1)),
    "odd_bins_narrow_band": ([(160, 120)], 2, (3, 3), dict(hist_bins=1023, band_kappa=0.5)),
    "most_bins": ([(160, 120)], 2, (3, 3), dict(hist_bins=4096, band_kappa=1.25)),
    "tiny_distances": ([(160, 120)], 1, (2,), dict(d_max=1e-16)),
}


@pytest.mark.parametrize("name", CASES)
def test_team_equals_per_iteration_launches(name):
    sizes, levels, caps, kw = CASES[name]
    pairs = _pairs(sizes)
    team = _run(7, pairs, levels, caps, 2, **kw)
    assert team[0] == team[1]
    assert team[0] == _run(7 | 16, pairs, levels, caps, 1, **kw)[0]


def test_a_pair_without_matches_ends_alone_and_the_next_call_is_unharmed():
    pairs = _pairs([(320, 240), (320, 240), (160, 120)], empty=(1,))
    team = _run(7, pairs, 3, (10, 5, 4), 3)
    assert team[0] == team[1] == team[2]
    assert team[0] == _run(7 | 16, pairs, 3, (10, 5, 4), 1)[0]
    assert team[0][0] == O.TOO_FEW_INLIERS


def test_a_leader_without_workers_times_out_and_the_tracker_goes_on():
    k = H.kf()
    (pr,) = _pairs([(320, 240)])
    p, _ = H.params()
    with H.Tracker(p, 320, 240) as t:
        t.set_pair(pr)
        before = t.align(pr)
        assert k.kf_debug_wait_timeout(t.h, 20.0) == k.KF_ERR_TIMEOUT
        after = t.align(pr)
        assert before[0] == after[0] and (before[1] == after[1]).all()

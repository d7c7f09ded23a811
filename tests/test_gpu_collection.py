"""Hypothesis collection when the group budget is spent: budgets within one coarse count of
solutions (2048 groups), one group to either side of it, and over ten of them. The
hypotheses are those of the groups in order, and a smaller budget's are the first of a
larger one's, bit for bit."""
import numpy as np
import pytest

from tests.helpers import f32_state, small_window

pytestmark = pytest.mark.gpu


def test_spent_budgets():
    from paper_2104_06789_gb300 import build, voldor as vd
    build.build()
    w = small_window(seed=1600, W=120, H=90, f=90.0, T=2)
    depth, rig = f32_state(np.random.default_rng(6), w)
    runs = []
    for groups in (1, 7, 9, 500, 2047, 2048, 2049, 4100, 20001):
        p = vd.default_params(hyps_per_frame=65536, groups_per_frame=groups, inv_depth_min=w.inv_depth_range[0],
                              inv_depth_max=w.inv_depth_range[1])
        g = vd.Window(w.flows.astype(np.float32), w.K, p)
        g.set_state(poses=w.poses, depth=depth, rigidness=rig, iteration=0)
        for _ in range(2):                                # the counts of one frame do not reach the next
            g.set_state(poses=w.poses)
            g.pose_update(0, 2)
        runs.append((groups, g.hypotheses()))
        g.destroy()
    last = runs[-1][1]
    assert 15000 < len(last["t"]) < 65536
    for groups, h in runs:
        n = len(h["t"])
        assert n == np.searchsorted(last["group"], groups)
        for key in ("group", "slot", "R", "t", "weight"):
            assert np.array_equal(h[key], last[key][:n]), (groups, key)
    new = np.concatenate([[True], np.diff(last["group"]) > 0])
    assert np.all(np.diff(last["group"]) >= 0)
    first = np.maximum.accumulate(np.where(new, np.arange(len(new)), 0))
    assert np.array_equal(last["slot"], np.arange(len(new)) - first)      # slots 0, 1, ... of each group

"""Dense scores do not depend on what a window scored before: an odd number of
hypotheses after a larger call (the last one shares a reciprocal with the operand row
after it), also where that row held a hypothesis that is not finite in FP32, and the
hypotheses of a pose update after one. A window with a history and a fresh one agree
bit for bit."""
import numpy as np
import pytest

from tests.helpers import f32_hypotheses, f32_state, small_window

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def vd():
    from paper_2104_06789_gb300 import build, voldor
    build.build()
    return voldor


def _window(vd, w, depth, rig, crit, **kw):
    p = vd.default_params(hyps_per_frame=255, inv_depth_min=w.inv_depth_range[0], inv_depth_max=w.inv_depth_range[1],
                          criterion=crit, **kw)
    g = vd.Window(w.flows.astype(np.float32), w.K, p)
    g.set_state(poses=w.poses, depth=depth, rigidness=rig, iteration=0)
    return g


@pytest.mark.parametrize("crit", [0, 1])
@pytest.mark.parametrize("n", [1, 31, 33, 129, 253])
@pytest.mark.parametrize("far", [0.0, 1e39])
def test_scores_after_another_call(vd, crit, n, far):
    w = small_window(seed=1300, W=80, H=61, f=60.0, T=2)
    depth, rig = f32_state(np.random.default_rng(1), w)
    g, fresh = _window(vd, w, depth, rig, crit), _window(vd, w, depth, rig, crit)
    R, tv = f32_hypotheses(np.random.default_rng(n), w.poses[1][:3, :3], w.poses[1][:3, 3], 255)
    before = tv[::-1].copy()
    before[1::2] += far                  # every odd row, the partners of the last of an odd number
    g.score_hypotheses(2, R[::-1].copy(), before)
    assert np.array_equal(g.score_hypotheses(2, R[:n], tv[:n]), fresh.score_hypotheses(2, R[:n], tv[:n]))
    g.destroy()
    fresh.destroy()


def test_pose_update_after_another_call(vd):
    w = small_window(seed=1301, W=80, H=61, f=60.0, T=2)
    depth, rig = f32_state(np.random.default_rng(2), w)
    R, tv = f32_hypotheses(np.random.default_rng(3), np.eye(3), np.zeros(3), 255)
    counts = []
    for groups in range(40, 52):         # a spent budget: about 60 hypotheses, some counts odd
        out = []
        for history in (False, True):
            g = _window(vd, w, depth, rig, 0, groups_per_frame=groups)
            if history:
                g.score_hypotheses(1, R, tv + 1e39)
            g.pose_update(0, 2)
            out.append((g.hypotheses()["L"], g.get_pose_depth_rigidness(depth=False, rigidness=False)[0]))
            g.destroy()
        assert np.array_equal(out[0][0], out[1][0]) and np.array_equal(out[0][1], out[1][1]), groups
        counts.append(len(out[0][0]))
    assert max(counts) < 255 and any(c % 2 for c in counts)

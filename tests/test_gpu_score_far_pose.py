"""Dense scores do not depend on the frame's current pose: with T_t far from every
hypothesis (a translation a million times theirs, a half turn) they agree with the oracle to
1e-5 relative, the package's bound on dense scores, and a pose update finds the
pose it finds from the true one to the bound on poses after the meanshift (1e-6)."""
import numpy as np
import pytest

from tests.helpers import f32_hypotheses, f32_state, oracle_window, pose_close, small_window

pytestmark = pytest.mark.gpu


def _far(poses, t, far):
    out = poses.copy()
    if far == "turn":
        out[t - 1, :3, :3] = np.diag([-1.0, 1.0, -1.0])
    else:
        out[t - 1, :3, 3] += np.array([1.0, -2.0, 0.5]) * far
    return out


@pytest.mark.parametrize("crit,res", [(0, 0), (1, 0), (0, 1), (1, 1)])
@pytest.mark.parametrize("far", [30.0, 1e5, 1e12, 1e30, "turn"])
def test_scores(oracle_lib, crit, res, far):
    from paper_2104_06789_gb300 import build, voldor as vd
    build.build()
    w = small_window(seed=1700, W=80, H=61, f=60.0, T=2)
    depth, rig = f32_state(np.random.default_rng(1), w)
    p = vd.default_params(hyps_per_frame=64, inv_depth_min=w.inv_depth_range[0], inv_depth_max=w.inv_depth_range[1],
                          criterion=crit, residual=res)
    g = vd.Window(w.flows.astype(np.float32), w.K, p)
    g.set_state(poses=_far(w.poses, 2, far), depth=depth, rigidness=rig, iteration=0)
    ow = oracle_window(oracle_lib, w, w.flows.astype(np.float32).astype(np.float64), 64, depth, rig, w.poses,
                       criterion=crit, residual=res)
    R, tv = f32_hypotheses(np.random.default_rng(2), w.poses[1][:3, :3], w.poses[1][:3, 3], 40)
    L, ref = g.score_hypotheses(2, R, tv), ow.score(2, R, tv)
    g.destroy()
    assert np.all(np.abs(L - ref) <= 1e-5 * np.abs(ref))


@pytest.mark.parametrize("far", [1e5, "turn"])
def test_pose_update(far):
    from paper_2104_06789_gb300 import build, voldor as vd
    build.build()
    w = small_window(seed=1701, W=80, H=61, f=60.0, T=2)
    depth, rig = f32_state(np.random.default_rng(3), w)
    p = vd.default_params(hyps_per_frame=256, inv_depth_min=w.inv_depth_range[0], inv_depth_max=w.inv_depth_range[1])
    out = []
    for poses in (w.poses, _far(w.poses, 2, far)):
        g = vd.Window(w.flows.astype(np.float32), w.K, p)
        g.set_state(poses=poses, depth=depth, rigidness=rig, iteration=0)
        g.pose_update(0, 2)
        out.append(g.get_pose_depth_rigidness(depth=False, rigidness=False)[0][1])
        g.destroy()
    assert pose_close(out[1], out[0])[0]

"""Dense scores of far fewer hypotheses than a frame may hold, whose pixel chunks are
chosen for their number: one group of 128 and a part, up to one group less than all,
on images of one tile, of fewer tiles than chunks fit, and of more. Against the
oracle; bound 1e-5 relative, the package's bound on dense scores."""
import numpy as np
import pytest

from tests.helpers import f32_hypotheses, f32_state, oracle_window, small_window

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("W,H", [(16, 8), (60, 31), (230, 97)])
@pytest.mark.parametrize("n", [1, 128, 129, 400, 896, 897])
def test_few_hypotheses(oracle_lib, W, H, n):
    from paper_2104_06789_gb300 import build, voldor as vd
    build.build()
    w = small_window(seed=1500 + W, W=W, H=H, f=W * 0.75, T=2)
    depth, rig = f32_state(np.random.default_rng(W), w)
    p = vd.default_params(hyps_per_frame=1024, inv_depth_min=w.inv_depth_range[0], inv_depth_max=w.inv_depth_range[1])
    g = vd.Window(w.flows.astype(np.float32), w.K, p)
    g.set_state(poses=w.poses, depth=depth, rigidness=rig, iteration=0)
    ow = oracle_window(oracle_lib, w, w.flows.astype(np.float32).astype(np.float64), 64, depth, rig, w.poses)
    R, tv = f32_hypotheses(np.random.default_rng(n), w.poses[1][:3, :3], w.poses[1][:3, 3], n)
    L, ref = g.score_hypotheses(2, R, tv), ow.score(2, R, tv)
    assert np.all(np.abs(L - ref) <= 1e-5 * np.abs(ref))
    g.destroy()

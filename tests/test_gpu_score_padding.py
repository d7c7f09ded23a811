"""Dense scores when the last pixel tile is not full and the residual's floor
underflows in the scoring's FP32 scale (x_min / fx^2 = 0): lanes past the last pixel
add nothing. Bound: 1e-5 relative, the package's bound on dense scores."""
import numpy as np
import pytest

from tests.helpers import f32_hypotheses, f32_state, oracle_window, small_window

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("crit,res", [(0, 0), (1, 0), (0, 1), (1, 1)])
@pytest.mark.parametrize("W,H", [(127, 3), (33, 20), (64, 4)])
def test_lanes_past_the_last_pixel(oracle_lib, W, H, crit, res):
    from paper_2104_06789_gb300 import build, voldor as vd
    build.build()
    w = small_window(seed=1400 + W, W=W, H=H, f=W * 0.75, T=2)
    depth, rig = f32_state(np.random.default_rng(W), w)
    p = vd.default_params(hyps_per_frame=64, inv_depth_min=w.inv_depth_range[0], inv_depth_max=w.inv_depth_range[1],
                          criterion=crit, residual=res, x_min=1e-44)
    g = vd.Window(w.flows.astype(np.float32), w.K, p)
    g.set_state(poses=w.poses, depth=depth, rigidness=rig, iteration=0)
    ow = oracle_window(oracle_lib, w, w.flows.astype(np.float32).astype(np.float64), 64, depth, rig, w.poses,
                       criterion=crit, residual=res)
    R, tv = f32_hypotheses(np.random.default_rng(3), w.poses[0][:3, :3], w.poses[0][:3, 3], 40)
    L = g.score_hypotheses(1, R, tv)
    ref = ow.score(1, R, tv)             # (its floor of 1e-6 px^2 moves no score by 1e-8)
    g.destroy()
    assert np.all(np.abs(L - ref) <= 1e-5 * np.abs(ref))

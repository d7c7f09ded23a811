"""Dense scores with flows of thousands of pixels and a Fisk shape whose floor is not small:
the outlier density's exponent passes 128 at such pixels, whether they lie before or behind
the camera under a hypothesis. Bound: 1e-5 relative, the package's bound on dense scores."""
import numpy as np
import pytest

from tests.helpers import f32_hypotheses, f32_state, oracle_window, small_window

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("crit", [0, 1])
@pytest.mark.parametrize("beta_min", [0.05, 0.33, 0.8])
@pytest.mark.parametrize("back", [0.0, 12.0, 1e3])
def test_exponents_beyond_128(oracle_lib, crit, beta_min, back):
    from paper_2104_06789_gb300 import build, voldor as vd
    build.build()
    w = small_window(seed=1800, W=80, H=61, f=60.0, T=2)
    rng = np.random.default_rng(7)
    depth, rig = f32_state(rng, w)
    flows = w.flows.astype(np.float32)
    o = rng.random(flows.shape[:3]) < 0.1
    way = rng.uniform(0, 2 * np.pi, o.sum())
    flows[o] = (rng.uniform(300, 9000, o.sum()) * np.stack([np.cos(way), np.sin(way)])).T
    p = vd.default_params(hyps_per_frame=64, inv_depth_min=w.inv_depth_range[0], inv_depth_max=w.inv_depth_range[1],
                          criterion=crit, beta_min=beta_min)
    g = vd.Window(flows, w.K, p)
    g.set_state(poses=w.poses, depth=depth, rigidness=rig, iteration=0)
    ow = oracle_window(oracle_lib, w, flows.astype(np.float64), 64, depth, rig, w.poses, criterion=crit, beta_min=beta_min)
    R, tv = f32_hypotheses(rng, w.poses[0][:3, :3], w.poses[0][:3, 3], 40)
    tv[::2, 2] = np.float32(-back)       # a part of the scene, or all of it, behind camera t
    L, ref = g.score_hypotheses(1, R, tv), ow.score(1, R, tv)
    g.destroy()
    assert np.all(np.isfinite(L))
    assert np.all(np.abs(L - ref) <= 1e-5 * np.abs(ref))

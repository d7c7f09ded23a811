"""Rigidness smoothing on strips whose longer chains leave an SM room for two blocks or one
(16 and 32 warps to a block instead of 8), along both sides, with chain counts that are
no multiple of a block's. Bound: 2e-5 absolute, the package's bound on smoothed rigidness."""
import numpy as np
import pytest

from tests.helpers import f32_state, oracle_window, small_window

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("W,H,T", [(2047, 5, 2), (5, 2100, 2), (3001, 9, 1), (37, 4096, 1)])
def test_strips(oracle_lib, W, H, T):
    from paper_2104_06789_gb300 import build, voldor as vd
    build.build()
    w = small_window(seed=W + H, W=W, H=H, f=max(W, H) * 0.75, T=T)
    depth, rig = f32_state(np.random.default_rng(W), w)
    p = vd.default_params(hyps_per_frame=64, inv_depth_min=w.inv_depth_range[0], inv_depth_max=w.inv_depth_range[1])
    ow = oracle_window(oracle_lib, w, w.flows.astype(np.float32).astype(np.float64), 64, depth, rig, w.poses)
    for k in (0, 1):
        g = vd.Window(w.flows.astype(np.float32), w.K, p)
        g.set_state(poses=w.poses, depth=depth, rigidness=rig, iteration=k)
        g.rigidness_smooth(k)
        q = g.get_buffer(vd.BUF_SMOOTHED, (w.T, w.H, w.W), np.float32)
        g.destroy()
        assert np.abs(q - ow.smooth(k, ow.emissions())).max() < 2e-5, k

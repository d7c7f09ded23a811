"""The depth sweep's resolution at the edges of its parts: chains one position
shorter than, as long as and one longer than a chain's sixteen parts and its
multiples, frame counts that fill one, two, four and eight lanes of a test and one
over (T = 1, 2, 3, 5, 8, 9, 16), and smoothed weights below zero, where a partial
score no longer bounds the whole.

Teacher-forced against the FP64 oracle like the sweep on extreme shapes: labels and
depths equal at every pixel outside the runs that follow a near tie (at most a
quarter of the pixels)."""
import numpy as np
import pytest

from tests.helpers import f32_state, oracle_window, small_window, tie_runs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("W,H,T,low", [(15, 17, 3, 0.0), (16, 33, 9, 0.0), (31, 16, 5, 0.0), (49, 32, 8, 0.0),
                                       (65, 47, 2, 0.0), (33, 20, 16, 0.0), (40, 18, 1, 0.0), (48, 21, 4, -0.5)])
def test_sweep_equals_the_sequential_one(oracle_lib, W, H, T, low):
    from paper_2104_06789_gb300 import build, voldor as vd
    build.build()
    w = small_window(seed=W * H + T, W=W, H=H, f=max(W, H) * 0.75, T=T)
    rng = np.random.default_rng(W + H)
    p = vd.default_params(hyps_per_frame=64, inv_depth_min=w.inv_depth_range[0], inv_depth_max=w.inv_depth_range[1])
    for k in range(4):                                 # L->R, T->B, R->L, B->T
        depth, rig = f32_state(rng, w)
        g = vd.Window(w.flows.astype(np.float32), w.K, p)
        g.set_state(poses=w.poses, depth=depth, rigidness=rig, iteration=k)
        ow = oracle_window(oracle_lib, w, w.flows.astype(np.float32).astype(np.float64), 64, depth, rig, w.poses)
        q = rng.uniform(low, 1, size=(w.T, w.H, w.W)).astype(np.float32)
        g.set_buffer(vd.BUF_SMOOTHED, q)
        g.depth_update(k)
        lab_gpu = g.get_buffer(vd.BUF_LABELS, (w.H, w.W), np.uint8)
        _, D_gpu, _ = g.get_pose_depth_rigidness(poses=False, rigidness=False)
        th0 = ow.theta.copy()
        lab_ref = ow.mie_sweep(k, q.astype(np.float64))
        tied = tie_runs(ow, k, q.astype(np.float64), th0, lab_ref, lab_gpu)
        assert tied.mean() <= 0.25, (k, tied.mean())
        assert np.all((lab_gpu == lab_ref)[~tied]), k
        assert np.all((np.abs(D_gpu - ow.theta) <= 1e-5 * ow.theta)[~tied]), k
        g.destroy()

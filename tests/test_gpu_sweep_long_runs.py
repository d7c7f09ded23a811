"""The depth sweep where one value is carried far: a fronto-parallel plane seen with
quiet flows from a poor depth, so that a good sample holds for hundreds of positions,
past the ends of the chain's sixteen parts and of what a warp follows by itself, to the
end of the chain too. Frame counts of one, two, four and eight lanes to a test and one over.

Every step of the sweep is checked by itself, given the value it was handed: the depth
of a pixel is its previous one, its sample or its predecessor's, whichever the FP64
oracle scores highest. Two FP32 scores within 1e-5 each (the per-pixel likelihood's
bound) may swap places, so the choice may be worse than the best by 2e-5 relative."""
import numpy as np
import pytest

from tests.conftest import fronto_parallel_window

import oracle

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("W,H,T", [(900, 3, 4), (3, 700, 9), (1300, 2, 2), (640, 4, 1), (4096, 2, 3)])
def test_long_runs(oracle_lib, W, H, T):
    from paper_2104_06789_gb300 import build, voldor as vd
    build.build()
    rng = np.random.default_rng(W + H + T)
    shifts = [tuple(v) for v in rng.uniform(0.05, 0.2, (T, 2)) * rng.choice([-1, 1], (T, 2))]
    flows, K, poses, _ = fronto_parallel_window(W, H, T, f=0.8 * max(W, H), shifts=shifts)
    flows = (flows + rng.normal(0, 0.1, flows.shape)).astype(np.float32)
    depth = np.full((H, W), 30.0, np.float32)
    rig = np.ones((T, H, W), np.float32)
    kw = dict(inv_depth_min=1 / 40.0, inv_depth_max=1.0)
    ow = oracle.OracleWindow(flows.astype(np.float64), K, S=64, **kw)
    ow.poses[:] = poses
    q = rig.astype(np.float64)
    longest = 0
    for k in range(4):
        g = vd.Window(flows, K, vd.default_params(hyps_per_frame=64, **kw))
        g.set_state(poses=poses, depth=depth, rigidness=rig, iteration=k)
        g.set_buffer(vd.BUF_SMOOTHED, rig)
        g.depth_update(k)
        lab = g.get_buffer(vd.BUF_LABELS, (H, W), np.uint8)
        smp = g.get_buffer(vd.BUF_DEPTH_SAMPLES, (H, W), np.float32)
        _, D, _ = g.get_pose_depth_rigidness(poses=False, rigidness=False)
        g.destroy()
        rows = k % 2 == 0
        for c in range(H if rows else W):
            run, carried = 0, None
            for i in range(W if rows else H):
                x, y = [(i, c), (c, i), (W - 1 - i, c), (c, H - 1 - i)][k % 4]
                choices = [depth[y, x], carried, smp[y, x]]
                assert D[y, x] == choices[lab[y, x]], (k, x, y)
                scores = [ow.mie_score(q, y * W + x, float(v)) for v in choices if v is not None]
                chosen = ow.mie_score(q, y * W + x, float(D[y, x]))
                assert chosen >= max(scores) - 2e-5 * abs(max(scores)), (k, x, y)
                run = run + 1 if lab[y, x] == 1 else 0
                longest = max(longest, run)
                carried = D[y, x]
    assert longest > max(W, H) // 4

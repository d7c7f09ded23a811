"""Dense scores at the edges of the scoring kernel's tiles against the oracle:
128-pixel tiles, stages of 32 and groups of 128 hypotheses, chunks without a
tile, every criterion and residual model, hypotheses that put pixels behind the
camera, and hypotheses so far away that a pair's shared reciprocal would
overflow. Bound: 1e-5 relative, the package's bound on dense scores."""
import numpy as np
import pytest

from tests.helpers import f32_hypotheses, f32_state, oracle_window, small_window

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def vd():
    from paper_2104_06789_gb300 import build, voldor
    build.build()
    return voldor


def _check(vd, oracle_lib, W, H, t, R, tv, crit=0, res=0, shape=None, T=2):
    w = small_window(seed=1200 + W, W=W, H=H, f=W * 0.75, T=T)
    depth, rig = f32_state(np.random.default_rng(W), w)
    p = vd.default_params(hyps_per_frame=max(64, len(R)), inv_depth_min=w.inv_depth_range[0],
                          inv_depth_max=w.inv_depth_range[1], criterion=crit, residual=res)
    g = vd.Window(w.flows.astype(np.float32), w.K, p)
    if shape:
        g.set_score_shape(*shape)
    g.set_state(poses=w.poses, depth=depth, rigidness=rig, iteration=0)
    ow = oracle_window(oracle_lib, w, w.flows.astype(np.float32).astype(np.float64), 64, depth, rig, w.poses,
                       criterion=crit, residual=res)
    R, tv = R @ w.poses[t - 1][:3, :3], tv + w.poses[t - 1][:3, 3]
    R = np.eye(3) + (R - np.eye(3)).astype(np.float32)          # exact in the scoring's FP32 form
    tv = tv.astype(np.float32).astype(np.float64)
    L_gpu, L_ref = g.score_hypotheses(t, R, tv), ow.score(t, R, tv)
    g.destroy()
    err = np.abs(L_gpu - L_ref)          # (a hypothesis with every pixel behind camera t scores 0 under MLE)
    assert np.all(err <= 1e-5 * np.abs(L_ref)), int((err - 1e-5 * np.abs(L_ref)).argmax())


def _near(n, seed=0):
    return f32_hypotheses(np.random.default_rng(seed), np.eye(3), np.zeros(3), n)


# 127, 128, 129 and 256 valid pixels on frame 1 (every pixel of the first frame is valid), one and two groups
@pytest.mark.parametrize("W,H", [(127, 2), (64, 2), (43, 3), (128, 2)])
@pytest.mark.parametrize("n", [1, 31, 33, 129])
def test_tile_and_stage_edges(vd, oracle_lib, W, H, n):
    _check(vd, oracle_lib, W, H, 1, *_near(n, n))


@pytest.mark.parametrize("crit,res", [(0, 0), (1, 0), (0, 1), (1, 1)])
@pytest.mark.parametrize("n,chunks", [(128, 1), (257, 3), (96, 40)])
def test_variants_and_chunks(vd, oracle_lib, crit, res, n, chunks):
    _check(vd, oracle_lib, 80, 61, 2, *_near(n, 7), crit=crit, res=res, shape=(8, chunks))


@pytest.mark.parametrize("crit", [0, 1])
@pytest.mark.parametrize("far", [0.0, 1.0e11])
def test_behind_the_camera_and_far_away(vd, oracle_lib, crit, far):
    R, tv = _near(64, 3)
    tv[::3, 2] -= 12.0                   # the nearer half of the scene passes behind camera t
    if far:                              # beyond 2^30: the frame's path with a reciprocal per lane
        tv[1::4] = np.random.default_rng(5).normal(size=tv[1::4].shape) * far
    _check(vd, oracle_lib, 80, 61, 2, R, tv, crit=crit)

"""The median Sampson errors of the epipolar bootstrap where their selection
changes its way: images smaller than, as large as and just above the 16384 pixels
of the bracketing subset, a subset of every third pixel, errors that are small
at the subset's places and large elsewhere (the bracket misses: selection over
all pixels), and 1, 9 and 24 samples (a part group, a full
group and a part group, three full groups).

The medians are FP32 order statistics of FP32 errors; against the oracle's FP64
errors they move by no more than the largest perturbation of the values, ~1e-6
relative for the cancellation-free form: bound 2e-5 relative."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu

SUBSET = 16384                       # pixels in the bracketing subset at most


def _flows(W, H, K, rng):
    """A sideways motion over random depths, with Gaussian noise of 0.2 pixels."""
    x, y = np.meshgrid(np.arange(W, dtype=np.float64), np.arange(H, dtype=np.float64))
    z = rng.uniform(2.0, 10.0, (H, W))
    fx, fy, cx, cy = K
    X = np.stack([(x - cx) / fx * z, (y - cy) / fy * z, z], -1)
    a = 0.02
    R = np.array([[np.cos(a), 0, np.sin(a)], [0, 1, 0], [-np.sin(a), 0, np.cos(a)]])
    Y = X @ R.T + np.array([0.1, 0.03, 0.05])
    f = np.stack([fx * Y[..., 0] / Y[..., 2] + cx - x, fy * Y[..., 1] / Y[..., 2] + cy - y], -1)
    return (f + rng.normal(0.0, 0.2, f.shape)).astype(np.float32)


@pytest.mark.parametrize("W,H,M,miss", [(24, 20, 24, False), (128, 128, 9, False), (145, 113, 24, False),
                                        (181, 181, 1, False), (207, 194, 24, False), (207, 194, 9, True)])
def test_medians_match_the_oracle(W, H, M, miss):
    from paper_2104_06789_gb300 import build, voldor as vd
    build.build()
    rng = np.random.default_rng(W * H + M)
    K = (0.9 * W, 0.9 * W, 0.5 * (W - 1), 0.5 * (H - 1))
    flows = np.repeat(_flows(W, H, K, rng)[None], 2, 0)
    if miss:
        step = -(-W * H // SUBSET)
        k = np.arange(W * H // step)
        rough = np.ones(W * H, bool)
        rough[k * step + (k * 5) % step] = False
        assert 0.55 < rough.mean() < 0.75
        flows.reshape(2, -1, 2)[:, rough] += rng.normal(0.0, 4.0, (rough.sum(), 2)).astype(np.float32)
    p = vd.default_params(inv_depth_min=0.05, inv_depth_max=1.0, hyps_per_frame=64)
    g = vd.Window(flows, K, p)
    ow = oracle.OracleWindow(flows.astype(np.float64), K, inv_depth_min=0.05, inv_depth_max=1.0)
    try:
        g.bootstrap_epipolar(M, 1.0)
    except vd.VoldorError as err:                  # the medians stand whether or not a sample wins
        assert err.status == vd.ERR_DEGENERATE
    r = g.epipolar_results()
    scores = ow.epipolar_bootstrap(M, 1.0)[2]
    assert np.array_equal(np.isfinite(scores), np.isfinite(r["medians"]))
    n = 0
    for m in np.flatnonzero(np.isfinite(scores)):
        assert r["medians"][m] == pytest.approx(scores[m], rel=2e-5), m
        n += 1
    assert n >= max(1, M // 4)
    g.destroy()

"""The median Sampson errors of the epipolar bootstrap on images whose first bracket holds
more errors than there is room for (above 1.4 and above 1.87 million pixels), where a
second, larger subset narrows it; with errors that are small at the second subset's places
and large elsewhere the narrowed bracket misses and all pixels are selected from.

The medians are FP32 order statistics of FP32 errors; against the oracle's FP64
errors they move by no more than the largest perturbation of the values, ~1e-6
relative for the cancellation-free form: bound 2e-5 relative."""
import numpy as np
import pytest

import oracle
from tests.test_gpu_epipolar_median import _flows

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("W,H,M,miss", [(1500, 1000, 9, False), (1433, 1367, 9, False), (1433, 1367, 6, True)])
def test_medians_of_large_images(oracle_lib, W, H, M, miss):
    from paper_2104_06789_gb300 import build, voldor as vd
    build.build()
    rng = np.random.default_rng(W * H + M)
    K = (0.9 * W, 0.9 * W, 0.5 * (W - 1), 0.5 * (H - 1))
    flows = _flows(W, H, K, rng)[None]
    if miss:
        N = W * H
        step = N // int(min((6 * N / 65536) ** 2, 24 * 65536, N))
        k = np.arange(N // step)
        rough = np.ones(N, bool)
        rough[k * step + (k * 5) % step] = False
        assert rough.mean() > 0.9
        flows.reshape(-1, 2)[rough] += rng.normal(0.0, 4.0, (rough.sum(), 2)).astype(np.float32)
    p = vd.default_params(inv_depth_min=0.05, inv_depth_max=1.0, hyps_per_frame=64)
    g = vd.Window(flows, K, p)
    ow = oracle.OracleWindow(flows.astype(np.float64), K, inv_depth_min=0.05, inv_depth_max=1.0)
    try:
        g.bootstrap_epipolar(M, 1.0)
    except vd.VoldorError as err:                  # the medians stand whether or not a sample wins
        assert err.status == vd.ERR_DEGENERATE
    r = g.epipolar_results()
    g.destroy()
    scores = ow.epipolar_bootstrap(M, 1.0)[2]
    assert np.array_equal(np.isfinite(scores), np.isfinite(r["medians"]))
    good = np.isfinite(scores)
    assert good.sum() >= M // 4
    assert np.allclose(r["medians"][good], scores[good], rtol=2e-5, atol=0.0)

"""The weight gradient's work items at their edges: images narrower than, as wide as
and one column wider than an item of 64 columns, one and two rows (fewer items than
CTAs), several images, and more items than CTAs; every layer shape (16 -> 32, 32 ->
32, 32 -> 2 channels) is in each.

Against the network with BF16 rounding at the kernels' storage points the kernels
differ by FP32 accumulation order and the rare BF16 rounding it flips: 1e-2 relative
L2 per parameter block."""
import numpy as np
import pytest

from test_gpu_net import _blocks, _case, _emulated, _rel

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("T,B,H,W", [(3, 1, 1, 7), (8, 1, 2, 64), (4, 2, 7, 65), (8, 1, 40, 129), (2, 3, 19, 128),
                                     (5, 1, 90, 300)])
def test_gradients_at_segment_edges(T, B, H, W):
    import torch

    from paper_2104_06789_gb300 import build, voldor as vd
    build.build()
    cases = [_case(T, H, W, seed=10 * W + b) for b in range(B)]
    params = cases[0][0]
    net = vd.Net(T, params)
    flows = torch.from_numpy(np.stack([c[1] for c in cases])).cuda()
    target = torch.from_numpy(np.stack([c[2] for c in cases])).cuda()
    net.train_step(flows, target, lr=0.0, lam_r=0.5)
    g = net.get_grads().astype(np.float64)
    ref = np.mean([_emulated(params, c[1], c[2], T, 0.5)[1] for c in cases], axis=0)
    for (key, a), (_, r) in zip(_blocks(T, g), _blocks(T, ref)):
        assert _rel(a, r) < 1e-2, (key, _rel(a, r))
    net.destroy()

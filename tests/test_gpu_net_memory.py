"""A network that only infers holds its parameters (under 2 MB) and no training buffers: the
weight gradient's partial sums (84 MB) come with the first training step. Device memory
is taken in granules of 2 MB, one for each of the thirteen allocations at most."""
import pytest

pytestmark = pytest.mark.gpu


def test_training_buffers_come_with_training():
    torch = pytest.importorskip("torch")
    from paper_2104_06789_gb300 import build, voldor as vd
    build.build()
    flows = torch.randn(1, 8, 16, 16, 2, device="cuda")
    target = torch.rand(1, 16, 16, 2, device="cuda")
    vd.Net(8).destroy()                                   # what loading the library takes is not the network's
    torch.cuda.synchronize()
    free = torch.cuda.mem_get_info()[0]
    net = vd.Net(8)
    assert free - torch.cuda.mem_get_info()[0] <= 28 << 20
    net.train_step(flows, target, 0.0)
    assert free - torch.cuda.mem_get_info()[0] >= 84 << 20
    net.destroy()

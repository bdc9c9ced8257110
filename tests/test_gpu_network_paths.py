"""The one-kernel BF16 network (tcgen05) and the launch per layer (mma.sync), which serves the same network where the
rows are not 8-byte aligned: the same bits.  Both round inputs, weights and activations to BF16 at the same
places and sum K steps of 16 in the same order in FP32."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_1706_07632_gb300 as fh  # noqa: E402


@pytest.mark.parametrize("hidden,layers,rows", [(64, 1, 1), (64, 3, 127), (128, 2, 129), (192, 8, 640), (256, 3, 1000),
                                                (320, 3, 30011)])
def test_one_kernel_equals_launch_per_layer(hidden, layers, rows):
    net = fh.WSNet(hidden, layers, seed=hidden)
    g = torch.Generator("cuda").manual_seed(rows)
    p = torch.randn(net.num_params(), generator=torch.Generator().manual_seed(rows)).numpy() * 0.05
    net.set_params(net.get_params() + p)
    X = torch.rand(rows, 6, device="cuda", generator=g) * 2 - 1
    shifted = torch.empty(rows * 6 + 1, device="cuda")[1:].view(rows, 6)
    shifted.copy_(X)
    assert X.data_ptr() % 8 == 0 and shifted.data_ptr() % 8 == 4
    one, per_layer = torch.empty(rows, device="cuda"), torch.empty(rows, device="cuda")
    n0 = fh.wsnet_launches()
    net.forward(X, one, bf16=True)
    n1 = fh.wsnet_launches()
    net.forward(shifted, per_layer, bf16=True)
    assert n1 - n0 == 2 and fh.wsnet_launches() - n1 > 2  # weights packed and one kernel; the other path
    assert torch.equal(one, per_layer)

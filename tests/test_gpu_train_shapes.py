"""Gradients of the warm-start network and its one-launch BF16 inference on ragged batch and layer widths (edges of the GEMM tiles, of the
16-byte loads and of the row splits), against the float64 oracle.

Tolerance: every entry is a chain of at most 2 layers + 1 = 9 dot products; a float32 dot product of
length K <= 1000 with rounding errors adding up at random is off by about sqrt(K) 2^-24 = 1.9e-6 of its
terms' size, the activations' fast exponential by a few 2^-23 each, and cancellation in the weight
gradients costs a small factor: 5e-5 of the gradient's norm."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_1706_07632_gb300 as fh  # noqa: E402
from oracle import nn  # noqa: E402


@pytest.mark.parametrize("hidden,layers,batch", [(8, 1, 1), (8, 2, 63), (67, 2, 65), (64, 4, 64), (130, 3, 257),
                                                 (200, 3, 1000), (320, 3, 4097)])
def test_loss_and_gradient_on_ragged_shapes(hidden, layers, batch):
    net = fh.WSNet(hidden, layers, seed=3)
    rng = np.random.default_rng(hidden + batch)
    X = rng.uniform(-1, 1, (batch, 6)).astype(np.float32)
    Y = rng.uniform(0, 1, batch).astype(np.float32)
    loss, g = net.loss_grad(torch.as_tensor(X, device="cuda"), torch.as_tensor(Y, device="cuda"))
    ref_loss, ref = nn.loss_grad(net.get_params(), nn.widths(hidden, layers), X, Y)
    assert abs(loss - ref_loss) <= 5e-5 * ref_loss
    assert np.linalg.norm(g - ref) <= 5e-5 * np.linalg.norm(ref)
    off = 0
    w = nn.widths(hidden, layers)
    for l in range(len(w) - 1):  # layer by layer, so that no small gradient hides behind a large one
        n = w[l] * w[l + 1] + w[l + 1]
        assert np.linalg.norm(g[off:off + n] - ref[off:off + n]) <= 5e-5 * np.linalg.norm(ref[off:off + n])
        off += n


def _bf16(x):
    return torch.as_tensor(np.asarray(x, dtype=np.float32)).to(torch.bfloat16).to(torch.float64).numpy()


@pytest.mark.parametrize("hidden,layers,rows", [(64, 1, 1), (64, 8, 129), (128, 2, 127), (192, 3, 128), (256, 4, 640),
                                                (320, 1, 257), (320, 3, 50001)])
def test_bf16_network_in_one_launch(hidden, layers, rows):
    """Every width the one-launch network serves (row blocks of 128, several per CTA at 50001 rows; no
    hidden product at one layer) against a layer-by-layer emulation.  An activation whose FP32 sum lies
    near a rounding boundary may round to the neighbouring BF16 value (2^-8 relative), in a small share
    of the terms of the next sum: 5e-3 of max|y|."""
    net = fh.WSNet(hidden, layers, seed=5)
    rng = np.random.default_rng(rows)
    X = rng.uniform(-1, 1, (rows, 6)).astype(np.float32)
    y = torch.empty(rows, dtype=torch.float32, device="cuda")
    net.forward(torch.as_tensor(X, device="cuda"), y, bf16=True)
    w = nn.widths(hidden, layers)
    a = _bf16(X)
    for l, (W, b) in enumerate(nn.unpack(net.get_params(), w)):
        z = a @ _bf16(W).T + b.astype(np.float64)
        a = _bf16(z / (1 + np.exp(-z))) if l < layers else z
    assert np.max(np.abs(y.cpu().numpy() - a[:, 0])) <= 5e-3 * np.max(np.abs(a))

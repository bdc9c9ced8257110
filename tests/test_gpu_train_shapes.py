"""Gradients of the warm-start network on ragged batch and layer widths (edges of the GEMM tiles, of the
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

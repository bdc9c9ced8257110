"""The buffers a network keeps for its batches: one network over batches of changing size gives the gradients and
values of a fresh one, bit for bit."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import numpy as np  # noqa: E402

import paper_1706_07632_gb300 as fh  # noqa: E402


def _batch(n):
    g = torch.Generator("cuda").manual_seed(n)
    return torch.rand(n, 6, device="cuda", generator=g), torch.rand(n, device="cuda", generator=g)


@pytest.mark.parametrize("hidden,layers", [(67, 3), (320, 2), (512, 1)])
def test_gradients_over_batches_of_changing_size(hidden, layers):
    used = fh.WSNet(hidden, layers, seed=6)
    for n in (5, 300, 64, 4097, 1000, 4097, 9000):
        X, Y = _batch(n)
        _, got = used.loss_grad(X, Y)
        _, want = fh.WSNet(hidden, layers, seed=6).loss_grad(X, Y)
        assert np.array_equal(got, want), n

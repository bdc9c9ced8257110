"""The buffers a network keeps for its batches: one network over batches of changing size gives the gradients and
values of a fresh one, bit for bit, holds no more memory than one that has seen the largest batch only, and survives
an allocation that fails."""
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


def _values(net, X):
    y = torch.empty(X.shape[0], device="cuda")
    net.forward(X, y)
    return y


def test_buffers_do_not_pile_up():
    """Batches doubling to 32000 rows of 320 x 3: 471 MB at the largest, as much again if every size stayed."""
    X, Y = _batch(32000)
    used = []
    for sizes in ((32000,), (1000, 2000, 4000, 8000, 16000, 32000)):
        torch.cuda.synchronize()
        before = torch.cuda.mem_get_info()[0]
        net = fh.WSNet(320, 3, seed=1)
        for n in sizes:
            net.loss_grad(X[:n], Y[:n])
        used.append(before - torch.cuda.mem_get_info()[0])
        del net
    assert used[1] <= 1.1 * used[0], used


def test_failed_growth_leaves_the_network_usable():
    net = fh.WSNet(320, 3, seed=1)
    X, _ = _batch(20000)  # 295 MB of activations
    small = _values(net, X[:100])
    y, again = torch.empty(20000, device="cuda"), torch.empty(100, device="cuda")
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    hog = torch.empty(torch.cuda.mem_get_info()[0] - (96 << 20), dtype=torch.uint8, device="cuda")
    try:
        with pytest.raises(fh.FhmgError) as e:
            net.forward(X, y)
        assert e.value.status == -3
        net.forward(X[:100], again)
    finally:
        del hog
        torch.cuda.empty_cache()
    assert torch.equal(again, small)
    net.forward(X, y)
    assert torch.equal(y, _values(fh.WSNet(320, 3, seed=1), X))

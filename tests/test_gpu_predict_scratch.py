"""A prediction's scratch stays with the network, buffer by buffer in the order of use: a network that has served
other problems (larger, smaller, the other dimension, other streams), or whose prediction failed half-way
for want of memory, predicts what a fresh one predicts, bit for bit."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_1706_07632_gb300 as fh  # noqa: E402

SIZES = [(2, 63, 64, 9), (1, 127, 256, 31), (2, 127, 128, 31), (1, 7, 64, 9), (2, 31, 256, 31), (2, 63, 64, 9)]


def _problem(dim, N, M, stream=None):
    P = fh.Problem(fh.HMatrix(0.5, 2.0, 1.0, M, 64, 0, 1e-10), dim, N, stream=stream)
    g = torch.Generator("cuda").manual_seed(N + M)
    s = torch.randn((N,) * dim, dtype=torch.float64, device="cuda", generator=g)
    return P, s.expand((M,) + s.shape).contiguous()


@pytest.mark.parametrize("hidden,bf16", [(64, True), (64, False), (40, True)])
def test_one_network_over_many_problems(hidden, bf16):
    used = fh.WSNet(hidden, 3, seed=4)
    for i, (dim, N, M, K) in enumerate(SIZES):
        stream = torch.cuda.Stream() if i % 2 else None
        P, f = _problem(dim, N, M, stream)
        torch.cuda.synchronize()
        want = fh.WSNet(hidden, 3, seed=4).predict(P, f, 0.5, K=K, bf16=bf16)
        got = used.predict(P, f, 0.5, K=K, bf16=bf16)
        assert torch.equal(got, want), (dim, N, M, K)


def test_failed_growth_leaves_the_network_usable():
    net = fh.WSNet(64, 3, seed=4)
    P1, f1 = _problem(2, 63, 64)
    P2, f2 = _problem(2, 255, 1024, torch.cuda.Stream())  # K = 32: rows 25 MB + 8 MB, synthesis 33 MB
    u1 = net.predict(P1, f1, 0.5, K=9)
    u2, again = torch.empty_like(f2), torch.empty_like(f1)
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    hog = torch.empty(torch.cuda.mem_get_info()[0] - (48 << 20), dtype=torch.uint8, device="cuda")
    try:
        with pytest.raises(fh.FhmgError) as e:  # the synthesis buffer does not fit, with the rows' kernels under way
            net.predict(P2, f2, 0.5, K=32, u0=u2)
        assert e.value.status == -3
        net.predict(P1, f1, 0.5, K=9, u0=again)
    finally:
        del hog
        torch.cuda.empty_cache()
    assert torch.equal(again, u1)
    want = fh.WSNet(64, 3, seed=4).predict(P2, f2, 0.5, K=32)
    assert torch.equal(net.predict(P2, f2, 0.5, K=32, u0=u2), want)
    assert torch.equal(net.predict(P1, f1, 0.5, K=9), u1)

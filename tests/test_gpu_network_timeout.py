"""The one-kernel BF16 network's bounded waits: a withheld weight tile makes them give up.  The kernel returns,
the rows it has not computed are NaN, the failure is reported by the call it belongs to (a forward pass: by
status(); a prediction: by itself) and by no other, and the next call gives the clean result."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_1706_07632_gb300 as fh  # noqa: E402


def _timed_out(call):
    with pytest.raises(fh.FhmgError) as e:
        call()
    return e.value.status == fh.FHMG_ETIMEOUT


@pytest.mark.parametrize("hidden,layers,rows", [(64, 2, 100), (320, 3, 128 * 152 + 131), (128, 8, 129)])
def test_forward_timeout_is_reported_by_status(hidden, layers, rows):
    net = fh.WSNet(hidden, layers, seed=2)
    X = torch.rand(rows, 6, device="cuda")
    clean, y = torch.empty(rows, device="cuda"), torch.zeros(rows, device="cuda")
    net.forward(X, clean, bf16=True)
    net.status()
    net.inject_timeout(512)
    net.forward(X, y, bf16=True)
    assert _timed_out(net.status)
    assert bool(torch.isnan(y).all())  # the withheld tile belongs to every CTA's first rows
    net.status()                       # reported once
    net.forward(X, y, bf16=True)
    net.status()
    assert torch.equal(y, clean)


def test_prediction_timeout_is_its_own():
    net = fh.WSNet(64, 2, seed=2)
    H = fh.HMatrix(0.5, 2.0, 1.0, 64, 64, 0, 1e-10)
    P = fh.Problem(H, 1, 63)
    f = torch.rand(1, 63, dtype=torch.float64, device="cuda").expand(64, 63).contiguous()
    clean = net.predict(P, f, 0.5, K=9)
    net.inject_timeout(512)
    assert _timed_out(lambda: net.predict(P, f, 0.5, K=9))
    net.status()                       # not a forward pass's
    assert torch.equal(net.predict(P, f, 0.5, K=9), clean)
    X, y = torch.rand(100, 6, device="cuda"), torch.empty(100, device="cuda")
    net.inject_timeout(512)
    net.forward(X, y, bf16=True)
    assert torch.equal(net.predict(P, f, 0.5, K=9), clean)  # an earlier forward pass's is not the prediction's
    assert _timed_out(net.status)


def test_inject_rejects_what_it_cannot_arm():
    for net, spin in ((fh.WSNet(64, 1), 512), (fh.WSNet(96, 2), 512), (fh.WSNet(64, 2), 0), (fh.WSNet(64, 2), 1 << 30)):
        with pytest.raises(fh.FhmgError) as e:
            net.inject_timeout(spin)
        assert e.value.status == fh.FHMG_EINVAL

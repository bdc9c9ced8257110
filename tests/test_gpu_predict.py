"""The predicted warm start, element by element, against the float64 oracle: features, network and synthesis over
the exact sine coefficients of the source, in 1D and 2D, at odd mode counts (ragged tiles of the synthesis) and
at more modes than grid points.

Tolerance.  u0 = sum_k s_k c_k y_k / lam_k with |s_k| <= 1, so its error is at most the sum over the modes of
* |c_k| / lam_k times the network's error.  FP32: its dot products of K <= 320 terms are off by about sqrt(K) 2^-24 =
  1.1e-6 of the sum of their terms' sizes, which through up to four layers and their cancellation stays below
  5e-5 of the sum of the output's terms (the bound of the gradient tests).  BF16, against an emulation that
  rounds at the same places: 5e-3 of max|y| (the bound of the inference tests);
* max|y| / lam_k times the projection's error: source, sines and two dot products of N <= 1023 terms in FP32, each
  off by about sqrt(N) 2^-24 = 1.9e-6 of its terms: 6e-6 of (2 / (N + 1))^dim sum |f|;
* |a_k| = |c_k y_k| / lam_k times that of the synthesis, K <= 33 terms per dimension: 2e-6."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_1706_07632_gb300 as fh  # noqa: E402
from oracle import direct, l1, nn  # noqa: E402


def _bf16(x):
    return torch.as_tensor(np.asarray(x, dtype=np.float32)).to(torch.bfloat16).to(torch.float64).numpy()


def _network(params, w, X, bf16):
    """(y, size of the output's terms): float64, or with inputs, weights and activations rounded to BF16."""
    r = _bf16 if bf16 else (lambda v: v)
    a = r(X)
    layers = nn.unpack(params, w)
    for W, b in layers[:-1]:
        z = a @ r(W).T + b
        a = r(z / (1.0 + np.exp(-z)))
    W, b = layers[-1]
    return (a @ r(W).T + b)[:, 0], (np.abs(a) @ np.abs(W).T + np.abs(b))[:, 0]


@pytest.mark.parametrize("bf16", [False, True])
@pytest.mark.parametrize("dim,N,M,K,hidden", [(1, 63, 64, 9, 320), (1, 1023, 64, 33, 64), (1, 7, 64, 9, 64),
                                              (2, 63, 64, 9, 320), (2, 127, 64, 31, 64), (2, 31, 128, 31, 40)])
def test_prediction_against_oracle(dim, N, M, K, hidden, bf16):
    alpha, gamma = 0.45, 1.7
    rng = np.random.default_rng(N + K)
    net = fh.WSNet(hidden, 3, seed=8)
    params = (net.get_params() + 0.05 * rng.standard_normal(net.num_params())).astype(np.float32)
    net.set_params(params)
    # a source with c_k = sqrt(lam_k) g_k on more modes than are predicted, so that every mode counts in u0
    n = min(N, K + 3)
    lam1 = direct.laplacian_eigs_1d(N, 1.0 / (N + 1))[:n]
    S = np.sin(np.pi * np.outer(np.arange(1, n + 1), np.arange(1, N + 1)) / (N + 1))
    lam = lam1 if dim == 1 else lam1[:, None] + lam1[None]
    c = np.sqrt(lam) * rng.standard_normal(lam.shape)
    field = c @ S if dim == 1 else S.T @ c @ S
    k = min(N, K)
    keep = (slice(0, k),) * dim
    lam, c = lam[keep].ravel(), c[keep].ravel()
    t = l1.graded_mesh(1.0, M, gamma)[1:]
    X = nn.features(lam[:, None], alpha, t[None]).reshape(-1, 6).astype(np.float32).astype(np.float64)
    y, terms = _network(params.astype(np.float64), nn.widths(hidden, 3), X, bf16)
    y = y.reshape(len(lam), M)
    a = (y * (c / lam)[:, None]).T
    want = a @ S[:k] if dim == 1 else S[:k].T @ a.reshape(M, k, k) @ S[:k]
    net_err = 5e-3 * np.abs(y).max() if bf16 else 5e-5 * terms.max()
    coef_err = 6e-6 * (2.0 / (N + 1)) ** dim * np.abs(field).sum()
    tol = net_err * np.sum(np.abs(c) / lam) + coef_err * np.abs(y).max() * np.sum(1 / lam) + 2e-6 * np.abs(a).sum(1).max()

    H = fh.HMatrix(alpha, gamma, 1.0, M, 64, 0, 1e-10)
    P = fh.Problem(H, dim, N)
    f = torch.as_tensor(field, device="cuda").expand((M,) + field.shape).contiguous()
    got = net.predict(P, f, alpha, K=K, bf16=bf16).cpu().numpy()
    assert np.abs(got - want).max() <= tol, (np.abs(got - want).max(), tol, np.abs(want).max())

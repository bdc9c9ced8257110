"""Restriction and prolongation of a batch share launches (64 instances each): more instances than one
launch holds, grids from the smallest to several blocks per row, 1D and 2D side by side, against
single-instance solves."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_1706_07632_gb300 as fh  # noqa: E402


@pytest.mark.parametrize("count", [1, 67])
def test_batched_transfers_match_single_solves(count):
    # FP64: both sides do the same operations, the products' sums at most in another order (tile width), so
    # that the solutions agree to a few hundred rounding errors of 1.1e-16 times the 1e3..1e4 by which
    # the cycles' residual bound may see them: 1e-11, as in the other comparisons of batched and single solves
    rng = np.random.default_rng(5)
    shapes = [(1, 3, 64), (1, 1023, 64), (2, 3, 64), (1, 255, 128), (2, 31, 64), (1, 7, 256), (2, 7, 128)]
    Ps, us, fs, keep = [], [], [], []
    for i in range(count):
        dim, N, M = shapes[i % len(shapes)]
        H = fh.HMatrix(float(rng.uniform(0.2, 0.9)), 2.0, 1.0, M, 64, 0, 1e-10)
        keep.append(H)
        Ps.append(fh.Problem(H, dim, N))
        f = torch.as_tensor(rng.standard_normal((M, N**dim)), device="cuda")
        fs.append(f)
        us.append(torch.zeros_like(f))
    k, _ = fh.solve_batched(Ps, us, fs, 1, 1, 1e-8, 60)
    for i in range(count):
        u1 = torch.zeros_like(us[i])
        k1, _ = Ps[i].solve(u1, fs[i], None, 1, 1, 1e-8, 60)
        assert k[i] == k1
        assert float((us[i] - u1).abs().max() / u1.abs().max()) < 1e-11

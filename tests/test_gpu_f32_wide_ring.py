"""FP32-product walks on the tensor cores with the deepest ring of x tiles (a dense lower triangle of eight
leaves: every earlier leaf stays in shared memory, so that the tiles' TF32 pairs do not fit at tile
32), against the FP64 oracle.  Bars as for the other FP32 walks: FP32 entries and x tiles (6e-8) and FP32
accumulation of a few hundred terms give 2e-6 for products, 2e-5 for the recurrence of a line solve."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_1706_07632_gb300 as fh  # noqa: E402
from oracle import direct, l1  # noqa: E402
from paper_1706_07632_gb300 import inputs  # noqa: E402


@pytest.mark.parametrize("M", [256, 512])
@pytest.mark.parametrize("tile", [16, 32])
@pytest.mark.parametrize("ncols", [37, 1029])
def test_wide_ring(M, tile, ncols):
    alpha, gamma = 0.8, 1.5
    R = l1.l1_matrix(l1.graded_mesh(1.0, M, gamma), alpha)
    P = fh.Problem(fh.HMatrix(alpha, gamma, 1.0, M, 64, 0, 0.0), 1, 63, prec=fh.MIXED_FP32)
    B = inputs.random_field(41, (M, ncols))
    Bd = torch.as_tensor(B, dtype=torch.float64, device="cuda")
    X = torch.empty_like(Bd)

    def rel(ref):
        return float(np.abs(X.cpu().numpy() - ref).max() / np.abs(ref).max())

    P.line_solve_f32(3, X, Bd, tile)
    assert rel(direct.solve_o2_mode(R, 2.0 * 16.0**2, B)) < 2e-5
    P.hmatvec_f32(X, Bd, tile)
    assert rel(R @ B) < 2e-6

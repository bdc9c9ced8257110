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


@pytest.mark.parametrize("M,rank,tile", [(1024, 12, 32), (1024, 20, 32), (1024, 30, 32), (4096, 12, 16), (4096, 36, 16)])
def test_many_live_z_values(M, rank, tile):
    # the Taylor form keeps hundreds of z values alive: shared memory holds the TF32 pairs and the buffers of
    # right-hand sides, only the buffers, or neither; against the SIMT walk at tile 1 (bar as for the
    # other comparisons of the two kernels)
    P = fh.Problem(fh.HMatrix(0.5, 2.0, 1.0, M, 64, rank, 0.0), 1, 63, prec=fh.MIXED_FP32)
    B = torch.as_tensor(inputs.random_field(43, (M, 333)), dtype=torch.float64, device="cuda")
    X, Y = torch.empty_like(B), torch.empty_like(B)
    for product in (False, True):
        for tc, out, t in ((True, X, tile), (False, Y, 1)):
            P.set_tensor_cores(tc)
            P.hmatvec_f32(out, B, t) if product else P.line_solve_f32(4, out, B, t)
        assert float((X - Y).abs().max() / Y.abs().max()) < 1e-5

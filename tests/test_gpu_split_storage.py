"""Storage by colour of the 2D FP32 grid functions (inner cycles of the mixed forms): the same solve with
FP64 storage (rows) and FP32 storage (by colour) on the smallest grids and the smallest tile edges.

The inner cycles differ by FP32 rounding only, so a V(1,1) cycle contracts alike: FP32 storage may need
one outer round more (two inner cycles a round at the default), and a wrong neighbour, weight or boundary
row costs far more.  The solutions meet the same residual target: they agree to a few 1e-8 of the
largest value."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_1706_07632_gb300 as fh  # noqa: E402
from paper_1706_07632_gb300 import inputs  # noqa: E402


@pytest.mark.parametrize("N,M,direct,prec", [(3, 64, 0, fh.MIXED_FP32), (7, 128, 3, fh.MIXED_FP32),
                                             (31, 64, 0, fh.MIXED_FP32), (63, 128, 31, fh.MIXED_FP32),
                                             (127, 128, 0, fh.MIXED_BF16), (255, 64, 31, fh.MIXED_BF16)])
def test_fp32_storage_solves_like_fp64_storage(N, M, direct, prec):
    H = fh.HMatrix(0.5, 2.0, 1.0, M, 64, 0, 1e-10)
    t, _ = H.mesh()
    a, s, _ = inputs.grf_2d(3, t[1:], N, 0.1)
    f = (torch.as_tensor(a, device="cuda")[:, None, None] * torch.as_tensor(s, device="cuda")[None]).contiguous()
    got = {}
    for storage in (1, 2):
        P = fh.Problem(H, 2, N, 1.0, prec)
        P.set_mixed_storage(storage)
        P.set_inner(2)
        if direct:
            P.set_coarse_direct(direct)
        u = torch.zeros_like(f)
        k, rr = P.solve(u, f, None, 1, 1, 1e-8, 60)
        got[storage] = (k, u)
    assert got[2][0] <= got[1][0] + 2, (got[1][0], got[2][0])
    assert float((got[2][1] - got[1][1]).abs().max() / got[1][1].abs().max()) < 1e-7

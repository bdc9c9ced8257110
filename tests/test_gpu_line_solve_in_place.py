"""Line solves in place (X aliases B, which the header allows): the same bits as into an array of its own,
on the tcgen05 walk (its memory warps load the right-hand sides a leaf ahead of the results), on the TF32
walk of both tiles and on the narrow SIMT walk; one leaf, two (both leaf buffers once) and several."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_1706_07632_gb300 as fh  # noqa: E402

WIDE = 128 * 152 + 1029  # a 128-column tile for every SM, and a ragged last tile


@pytest.mark.parametrize("prec,cols", [(fh.MIXED_BF16, WIDE), (fh.MIXED_FP32, WIDE), (fh.MIXED_FP32, 2501),
                                       (fh.MIXED_FP32, 37)])
@pytest.mark.parametrize("M", [64, 128, 512])
def test_in_place_equals_out_of_place(prec, cols, M):
    H = fh.HMatrix(0.55, 2.0, 1.0, M, 64, 0, 1e-10)
    P = fh.Problem(H, 2, 63, 1.0, prec)
    g = torch.Generator("cuda").manual_seed(cols + M)
    B = torch.randn(M, cols, dtype=torch.float32, device="cuda", generator=g)
    X = torch.empty_like(B)
    P.line_solve_s(P.levels - 1, X, B)
    P.line_solve_s(P.levels - 1, B, B)
    assert torch.equal(B, X)


@pytest.mark.parametrize("cols,tile", [(2501, 16), (2501, 32), (37, 4)])
@pytest.mark.parametrize("M", [64, 512])
def test_in_place_equals_out_of_place_fp64_storage(cols, tile, M):
    H = fh.HMatrix(0.55, 2.0, 1.0, M, 64, 0, 1e-10)
    P = fh.Problem(H, 1, 255, 1.0, fh.MIXED_FP32)
    g = torch.Generator("cuda").manual_seed(cols + tile)
    B = torch.randn(M, cols, dtype=torch.float64, device="cuda", generator=g)
    X = torch.empty_like(B)
    P.line_solve_f32(P.levels - 1, X, B, tile=tile)
    P.line_solve_f32(P.levels - 1, B, B, tile=tile)
    assert torch.equal(B, X)

"""The split defect's fixed-point stencil (sp_stencil in csrc/split.cuh) against exact rational arithmetic: zero for
equal values of either sign, odd in its values, and within its bound.

Bound: 2 NX terms (the point counts NX times) are off by half a unit of at most 2^(e - 59), 2^e the largest
value's power of two, and the sum is rounded once to FP64: |S - exact| <= NX 2^(e - 59) + 2^-53 |exact| (and,
S being that sum plus its error, 2^-53 of the error)."""
import ctypes
import os
import subprocess
from fractions import Fraction

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_1706_07632_gb300 import build  # noqa: E402
from tests.conftest import ROOT  # noqa: E402


@pytest.fixture(scope="module")
def stencil(tmp_path_factory):
    so = str(tmp_path_factory.mktemp("stencil") / "stencil.so")
    subprocess.check_call([build.NVCC] + build.ARCH + build.NVCC_FLAGS
                          + ["-shared", os.path.join(ROOT, "tests", "cuda", "stencil.cu"), "-o", so])
    lib = ctypes.CDLL(so)

    def call(v):
        v = torch.as_tensor(np.ascontiguousarray(v), device="cuda")
        out = torch.empty(v.shape[0], dtype=torch.float64, device="cuda")
        torch.cuda.synchronize()
        assert lib.stencil(v.shape[1] - 1, ctypes.c_void_p(v.data_ptr()), ctypes.c_void_p(out.data_ptr()),
                           v.shape[0]) == 0
        return out.cpu().numpy()

    return call


@pytest.mark.parametrize("nx", [2, 4])
def test_equal_values_give_zero(stencil, nx):
    rng = np.random.default_rng(nx)
    v = rng.standard_normal(400) * 10.0 ** rng.integers(-200, 200, 400)
    assert np.all(stencil(np.repeat(v[:, None], nx + 1, axis=1)) == 0.0)


@pytest.mark.parametrize("nx", [2, 4])
@pytest.mark.parametrize("spread", [0, 4, 70])
def test_odd_and_within_its_bound(stencil, nx, spread):
    rng = np.random.default_rng(10 * nx + spread)
    n = 500
    v = rng.standard_normal((n, nx + 1)) * 2.0 ** rng.integers(-spread, spread + 1, (n, nx + 1))
    if spread == 0:  # neighbours of a smooth grid function: the stencil cancels
        v = v[:, :1] * (1 + 1e-7 * rng.standard_normal((n, nx + 1)))
    v[:20, 1] = 0.0
    s = stencil(v)
    assert np.all(stencil(-v) == -s)
    for row, got in zip(v, s):
        exact = nx * Fraction(row[0]) - sum(Fraction(x) for x in row[1:])
        e = int(np.frexp(np.abs(row).max())[1]) - 1
        err = nx * Fraction(2) ** (e - 59)
        assert abs(Fraction(float(got)) - exact) <= err + (abs(exact) + err) / 2 ** 53

"""The reciprocal of the network's activations (csrc/rcp.cuh) is the division's result, bit for bit, for every
float of its range, 1 to 2^125 (1.05e9 of them): the function is compiled from its header into a small library
of its own (tests/cuda/rcp_all.cu)."""
import ctypes
import os
import subprocess

import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_1706_07632_gb300 import build  # noqa: E402
from tests.conftest import ROOT  # noqa: E402


def test_reciprocal_of_every_float_of_the_range(tmp_path):
    so = str(tmp_path / "rcp_all.so")
    subprocess.check_call([build.NVCC] + build.ARCH + build.NVCC_FLAGS
                          + ["-shared", os.path.join(ROOT, "tests", "cuda", "rcp_all.cu"), "-o", so])
    lib = ctypes.CDLL(so)
    bad = torch.zeros(1, dtype=torch.int64, device="cuda")
    worst = torch.zeros(1, dtype=torch.int32, device="cuda")
    torch.cuda.synchronize()
    first, last = 127 << 23, (127 + 125) << 23
    rc = lib.rcp_compare(ctypes.c_uint(first), ctypes.c_uint(last), ctypes.c_void_p(bad.data_ptr()),
                         ctypes.c_void_p(worst.data_ptr()))
    assert rc == 0
    assert int(bad) == 0, (int(bad), hex(int(worst)))

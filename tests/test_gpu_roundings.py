"""The library's own roots and quotients against correctly rounded ones: rho_root (the radius of
the normals) over every 32-bit word, exactly; the reflectors' root and quotient over 2^26
norms of all exponents, never more than one unit in the last place off and off at all in fewer than
one case in 10^6 (2^-25 from the error before the last rounding, some times that allowed)."""
import ctypes
import os
import subprocess

import pytest
import torch

from paper_2111_10448_gb300 import build

pytestmark = pytest.mark.gpu


def test_roundings(tmp_path):
    so = str(tmp_path / "roundings.so")
    src = os.path.join(os.path.dirname(os.path.abspath(__file__)), "roundings.cu")
    subprocess.run([build.nvcc()] + build.ARCH + build.FLAGS + ["-I", build.CSRC, "-shared", "-o", so, src], check=True)
    lib = ctypes.CDLL(so)
    lib.count_roundings.argtypes = [ctypes.c_void_p, ctypes.c_ulonglong]
    out = torch.zeros(5, dtype=torch.int64, device="cuda")
    total = 1 << 26
    assert lib.count_roundings(out.data_ptr(), total) == 0
    rho, roots, quotients, dr, dq = out.tolist()
    assert rho == 0
    assert dr <= 1 and dq <= 1
    assert roots <= total * 1e-6 and quotients <= total * 1e-6, (roots, quotients)

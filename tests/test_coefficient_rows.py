"""The differentiation coefficients handed to the kernels: with 1/dx in them and
rounded, each row still adds up to zero (a uniform flux has no residual) but for
the rounding of the one entry that closes it, half an ulp; the sum is taken
exactly.  Reads the tables through the library's own table function (no GPU).
"""
import ctypes
from fractions import Fraction

import numpy as np
import pytest

from paper_2604_02125_gb300 import crkfr

FILL = "_ZN3crk15fill_ref_tablesEiiRKNS_8MeshArgsEPNS_6RefTabIdEEPNS3_IfEE"
INV_DX = 72   # byte offset of inv_dx in MeshArgs: E, cells and their three divisors come first


def _tables(N, eq, inv_dx):
    """[direction][p][q] coefficients B in FP64 and FP32 (direction 3: without 1/dx)."""
    fill = getattr(crkfr.load_library(), FILL)
    fill.restype = None
    mesh, t64, t32 = (ctypes.create_string_buffer(16384) for _ in range(3))
    ctypes.memmove(ctypes.addressof(mesh) + INV_DX, np.array(inv_dx, dtype=np.float64).ctypes.data, 24)
    fill(N, eq, mesh, t64, t32)
    B64 = np.frombuffer(t64.raw, dtype=np.float64, count=144, offset=8 * 144).reshape(4, 6, 6)
    packed = 2 * 2 * 36 * 2   # FP32: two arrays of pairs come first
    B32 = np.frombuffer(t32.raw, dtype=np.float32, count=144, offset=4 * (packed + 144)).reshape(4, 6, 6)
    return B64[:, :N + 1, :N + 1], B32[:, :N + 1, :N + 1]


@pytest.mark.parametrize("eq", [0, 1])
@pytest.mark.parametrize("N", [1, 2, 3, 4, 5])
def test_rows_add_up_to_zero(N, eq):
    rng = np.random.default_rng(N)
    for _ in range(40):
        inv_dx = 10.0 ** rng.uniform(-2.0, 3.0, 3)
        for B in _tables(N, eq, inv_dx):
            for d in range(3):
                assert np.allclose(B[d], B[3] * inv_dx[d], rtol=1e-6, atol=1e-6 * np.abs(B[d]).max())
            # the entry that closes a row: the diagonal of an end row, the smallest other one of an inner row
            for T in B:
                for p in range(N + 1):
                    m = p if p in (0, N) else min((q for q in range(N + 1) if q != p), key=lambda q: abs(T[p][q]))
                    total = abs(sum(Fraction(float(x)) for x in T[p]))
                    assert total <= Fraction(float(np.spacing(abs(T[p][m])))) / 2, (N, p, T[p])
                    assert p in (0, N) or T[p][p] == 0.0

"""GLM-MHD at rest in exact balance: a uniform field B = (1, 0, 0) with p = 1/2, so
that the flux of x momentum along x, p + |B|^2/2 - B_x^2, is zero and that of y
momentum along y is one, while the non-conservative product B(u) g(u) = |B|^2
at every x face is not zero.  All values are small powers of two, c_h = 0, and at degree 1
D = +-1, so every flux difference and face jump is exactly zero in both
precisions: the state stays as it is, bit for bit, if the large products
cancel before they are scaled and rounded.  1/dx and dt are no powers of two.
"""
import numpy as np
import pytest

from paper_2604_02125_gb300 import crkfr, inputs

pytestmark = pytest.mark.gpu

CASES = [("rkfr", "reduced"), ("crkfr", "reduced"), ("crkfr", "stages")]


@pytest.mark.parametrize("vol", ["ec", "central"])
@pytest.mark.parametrize("prec", ["fp64", "fp32"])
@pytest.mark.parametrize("scheme,ncflux", CASES)
def test_balanced_field_stays(scheme, ncflux, prec, vol):
    N = 1
    mesh = inputs.mesh_dict("glm_mhd", 2, N, [7, 5], [0.0, 0.0], [1.0, 0.7], 1.5, vol=vol, c_h=0.0)
    one = np.ones((35, (N + 1) ** 2))
    zero = np.zeros_like(one)
    U = inputs.mhd_cons(1.5, one, [zero] * 3, 0.5 * one, [one, zero, zero], zero)
    with crkfr.Solver(dict(mesh, ncflux=ncflux), prec=prec, dt_fixed=0.0123, scheme=scheme) as s:
        s.set_state(U)
        s.step(3)
        G = s.get_state()
    assert np.array_equal(G, U), np.max(np.abs(G - U))

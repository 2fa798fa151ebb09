"""The branches of the logarithmic means in the two-point fluxes (GPU against
the FP64 oracle): node values whose pairs sit just below and just above each
branch's bound on u = ((a-b)/(a+b))^2, far below and far above.

One step from a saw of two densities per element (every pair of a line has
u = 0 or the stated u), with the pressure constant (rho/p jumps with rho) or
proportional to the density (rho/p constant).  Bars: the pair fluxes carry a
few units in the last place (FP64 1e-16, the oracle's log mean 1.2e-15, FP32
6e-8), amplified by the sums of |D_pq f| over the residual, below 1e2 on these
saws, over up to six stages: 1e-12 and 4e-5, rounded up; the subtraction
u1 - u0 adds 1e-16 |u| / |du| < 1e-13.
"""
import numpy as np
import pytest

import oracle
from paper_2604_02125_gb300 import crkfr, inputs
from parity_util import check_increment

pytestmark = pytest.mark.gpu

EDGES = [0.0, 1e-12, 2.0 ** -13 * (1 - 1e-9), 2.0 ** -13 * (1 + 1e-9), 1e-3, 0.05 * (1 - 1e-5), 0.05 * (1 + 1e-5),
         0.0625 * (1 - 1e-9), 0.0625 * (1 + 1e-9), 0.3]


# the FP64 form's two-part series: on both sides of its bound, across the
# exponents its fixed-point sum spans, and where the corrections vanish
SERIES_EDGES = [2.0 ** -11 * (1 - 1e-9), 2.0 ** -11 * (1 + 1e-9), 2.0 ** -12, 3e-5, 1e-7, 1e-16, 1e-24, 1e-31]


@pytest.mark.parametrize("eq,N", [("euler", 3), ("glm_mhd", 3)])
@pytest.mark.parametrize("scale", [1.0, 1e-60, 1e60])
@pytest.mark.parametrize("u", SERIES_EDGES)
def test_two_part_series(u, scale, eq, N):
    """scale: density and pressure (and the magnetic energy) far outside the FP32 range."""
    test_log_mean_branches(u, eq, N, "fp64", 1e-11, scale)


@pytest.mark.parametrize("prec,tol", [("fp64", 1e-11), ("fp32", 1e-4)])
@pytest.mark.parametrize("eq,N", [("euler", 3), ("euler", 4), ("glm_mhd", 3)])
@pytest.mark.parametrize("u", EDGES)
def test_log_mean_branches(u, eq, N, prec, tol, scale=1.0):
    oracle.build()
    dim = 2
    mesh = inputs.mesh_dict(eq, dim, N, [5, 3], [0.0, 0.0], [1.0, 0.7], 1.4, c_h=0.0 if eq == "euler" else 2.0)
    n = N + 1
    f = np.sqrt(u)
    p = np.arange(n * n)
    odd = ((p % n + p // n) % 2)[None, :]
    rho = scale * np.where(odd == 1, (1 + f) / (1 - f), 1.0) * np.ones((15, 1))
    pr = np.where(np.arange(15)[:, None] % 2 == 0, scale, rho)
    root = np.sqrt(scale)
    v = [0.3 + 0.05 * odd * np.ones_like(rho), -0.2 * np.ones_like(rho)]
    if eq == "euler":
        U = inputs.euler_cons(1.4, rho, v, pr)
    else:
        one = np.ones_like(rho)
        U = inputs.mhd_cons(1.4, rho, v + [0.1 * one], pr, [0.4 * root * one, 0.3 * root * one, 0.2 * root * one], 0.1 * root * one)
    s = crkfr.Solver(mesh, prec=prec)
    s.set_state(U)
    s.step(1)
    G = s.get_state()
    dt = s.info()["dt"]
    s.close()
    check_increment(G, oracle.step(mesh, U, dt), U, tol, "%s N=%d u=%g %s" % (eq, N, u, prec))

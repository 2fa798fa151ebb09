"""States whose FP64 reciprocals leave the range of the reciprocal unit, which
takes subnormal operands and results for zero: the step takes the reciprocal of rho^2 p
(EC flux, GLM-MHD) or of rho and p, here just below 2^-1022 and just above 2^1022, and
well inside both for comparison.

Against the FP64 oracle.  The reciprocals are subnormal or of a subnormal, exact to
2^-50 at the sizes chosen; the bar of the other FP64 steps' branches (1e-11) stays.
"""
import numpy as np
import pytest

import oracle
from paper_2604_02125_gb300 import crkfr, inputs
from parity_util import check_increment

pytestmark = pytest.mark.gpu

# (rho, p) with rho^2 p: inside, below 2^-1022 (2.2e-308), above 2^1022 (4.5e307)
SCALES = [(1e-100, 1e-104), (1e-100, 1.5e-108), (1e-100, 0.9e-108), (1e100, 1e104), (1e100, 0.6e108), (1e100, 1.2e108)]


@pytest.mark.parametrize("rho0,p0", SCALES)
@pytest.mark.parametrize("eq,dim,N,vol", [("euler", 1, 3, "ec"), ("euler", 2, 3, "ec"), ("euler", 2, 4, "ec"),
                                          ("euler", 3, 2, "ec"), ("euler", 2, 3, "kep"), ("glm_mhd", 2, 3, "ec")])
def test_reciprocals_at_the_ends_of_the_range(eq, dim, N, vol, rho0, p0):
    oracle.build()
    cells = [5, 3, 4][:dim]
    c = np.sqrt(p0 / rho0)
    mesh = inputs.mesh_dict(eq, dim, N, cells, [0.0] * dim, [1.0, 0.7, 0.9][:dim], 1.4, c_h=0.0 if eq == "euler" else 2.0 * c)
    mesh["vol"] = vol
    E, NP = int(np.prod(cells)), (N + 1) ** dim
    rng = np.random.default_rng(3)
    wave = lambda a: 1.0 + a * rng.uniform(-1.0, 1.0, (E, NP))
    rho, pr = rho0 * wave(0.02), p0 * wave(0.02)
    v = [0.3 * c * wave(0.1) for _ in range(dim)]
    if eq == "euler":
        U = inputs.euler_cons(1.4, rho, v, pr)
    else:
        b = np.sqrt(p0)
        U = inputs.mhd_cons(1.4, rho, v + [0.1 * c * wave(0.1)], pr, [0.4 * b * wave(0.1) for _ in range(3)], 0.1 * b * wave(0.1))
    with crkfr.Solver(mesh, prec="fp64") as s:
        s.set_state(U)
        s.step(1)
        G = s.get_state()
        dt = s.info()["dt"]
    assert np.all(np.isfinite(G)) and dt > 0.0
    R = oracle.step(mesh, U, dt)
    # variable by variable in units of the state's own, so that no square leaves the range
    scale = np.abs(U).reshape(U.shape[0], -1).max(axis=1).reshape((-1,) + (1,) * (U.ndim - 1))
    check_increment(G / scale, R / scale, U / scale, 1e-11, "%s %dD N=%d %s rho=%g p=%g" % (eq, dim, N, vol, rho0, p0))

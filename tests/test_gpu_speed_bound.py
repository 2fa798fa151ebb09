"""The FP64 form's time step where the face kernel decides from FP32 bounds
which nodes' wave speeds it evaluates in FP64: dt must be the CFL rule on the
FP64 maximum over every node, whatever the states.

Random node states over many decades of Mach number, plasma beta, scale and
gamma - 1; a step with a tiny fixed-point dt (cfl 1e-11: the increments are
small, so the states stay physical) gives u^1, whose dt the next step reports.
Bar 1e-13: the formula's own rounding (p from a cancelling difference is
evaluated from the same FP64 values by the same formula; a node dropped by a
wrong bound would move the maximum by 1e-7 or more).
"""
import numpy as np
import pytest

from paper_2604_02125_gb300 import crkfr, inputs

pytestmark = pytest.mark.gpu


def _max_speed(mesh, U):
    g, dim = mesh["gamma"], mesh["dim"]
    idx = [mesh["cells"][d] / (mesh["hi"][d] - mesh["lo"][d]) for d in range(dim)]
    rho = U[0]
    if mesh["eq"] == "euler":
        v = [U[1 + d] / rho for d in range(dim)]
        p = (g - 1) * (U[dim + 1] - 0.5 * sum(U[1 + d] ** 2 for d in range(dim)) / rho)
        c = np.sqrt(g * p / rho)
        return np.max(sum((np.abs(v[d]) + c) * idx[d] for d in range(dim)))
    v = [U[1 + k] / rho for k in range(3)]
    BB = U[5] ** 2 + U[6] ** 2 + U[7] ** 2
    p = (g - 1) * (U[4] - 0.5 * rho * sum(x * x for x in v) - 0.5 * BB - 0.5 * U[8] ** 2)
    a2, b2 = g * p / rho, BB / rho
    s = a2 + b2
    tot = 0
    for d in range(2):
        cf = np.sqrt(0.5 * (s + np.sqrt(np.maximum(s * s - 4 * a2 * U[5 + d] ** 2 / rho, 0))))
        tot = tot + (np.abs(v[d]) + np.maximum(cf, mesh["c_h"])) * idx[d]
    return np.max(tot)


@pytest.mark.parametrize("scale", [1.0, 1e-18, 1e18, 1e-40])
@pytest.mark.parametrize("gamma", [1.4, 5.0 / 3.0, 1.0 + 1e-6])
@pytest.mark.parametrize("eq,dim,N,cells", [("euler", 1, 3, [70]), ("euler", 2, 3, [9, 11]), ("euler", 2, 5, [7, 5]),
                                            ("euler", 3, 2, [4, 5, 3]), ("glm_mhd", 2, 3, [9, 7])])
def test_dt_is_the_fp64_maximum(eq, dim, N, cells, gamma, scale):
    for seed in range(6):
        rng = np.random.default_rng(seed)
        mesh = inputs.mesh_dict(eq, dim, N, cells, [0.0] * dim, [1.0, 0.7, 1.3][:dim], gamma, vol="central", cfl=1e-11,
                                c_h=0.3 if eq == "glm_mhd" else 0.0)
        shape = (int(np.prod(cells)), (N + 1) ** dim)
        dec = lambda lo, hi: 10.0 ** rng.uniform(lo, hi, shape)  # noqa: E731
        spread = [0.0, 0.5, 1.5][seed % 3]
        rho, p = scale * dec(-spread, spread), scale * dec(-spread, spread)
        v = [dec(-2, 1.5) * rng.choice([-1.0, 1.0], shape) for _ in range(3)]
        if eq == "euler":
            U = inputs.euler_cons(gamma, rho, v[:dim], p)
        else:
            B = [np.sqrt(scale) * dec(-1, 1) * rng.choice([-1.0, 1.0], shape) for _ in range(3)]
            U = inputs.mhd_cons(gamma, rho, v, p, B, np.sqrt(scale) * 0.1 * np.ones(shape))
        s = crkfr.Solver(mesh, prec="fp64")
        s.set_state(U)
        s.step(1)
        U1 = s.get_state(check=False)
        s.step(1)
        info = s.info()
        s.close()
        want = mesh["cfl"] / _max_speed(mesh, U1)
        assert np.isfinite(want)
        assert abs(info["dt"] - want) <= 1e-13 * want, (seed, info["dt"], want)

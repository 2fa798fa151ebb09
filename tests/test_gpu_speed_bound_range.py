"""The FP64 form's wave-speed filter (the face kernel evaluates in FP64 only the
nodes whose FP32 bound could be the maximum) where the bound's FP32 parts leave
the normal range: tiny and huge densities, p/rho far below one, momenta whose
squares underflow, meshes whose 1/dx has no normal FP32 value.

dt has to be the CFL rule on the FP64 maximum over every node, and a state
that is not physical has to be reported.  Bar 1e-13 as in
test_gpu_speed_bound.py (the formula's own rounding; a node dropped by a wrong
bound moves the maximum by far more on these states).
"""
import numpy as np
import pytest

import oracle
from paper_2604_02125_gb300 import crkfr, inputs
from test_gpu_speed_bound import _max_speed

pytestmark = pytest.mark.gpu


def _check_dt(mesh, U, what):
    with crkfr.Solver(mesh, prec="fp64") as s:
        s.set_state(U)
        s.step(1)
        U1 = s.get_state(check=False)
        s.step(1)
        dt = s.info()["dt"]
    want = mesh["cfl"] / _max_speed(mesh, U1)
    assert np.isfinite(want), what
    assert abs(dt - want) <= 1e-13 * want, (what, dt, want)


def _decades(rng, lo, hi, shape):
    return 10.0 ** rng.uniform(lo, hi, shape)


@pytest.mark.parametrize("scale", [1.0, 1e3, 1e-10])
@pytest.mark.parametrize("theta", [1e-30, 1e-25, 1e-22, 1e-20, 1e-19, 1e-18, 1e-15])
def test_cold_mhd_gas(theta, scale):
    """GLM-MHD at rest, no field, no cleaning speed: p/rho = theta, s^2 below the FP32 range."""
    mesh = inputs.mesh_dict("glm_mhd", 2, 3, [9, 7], [0.0, 0.0], [1.0, 0.7], 5.0 / 3.0, vol="central", cfl=1e-11)
    for seed in range(3):
        rng = np.random.default_rng(seed)
        shape = (63, 16)
        rho = scale * _decades(rng, -0.3, 0.3, shape)
        zero = np.zeros(shape)
        U = inputs.mhd_cons(5.0 / 3.0, rho, [zero] * 3, theta * rho * _decades(rng, -0.5, 0.5, shape), [zero] * 3, zero)
        _check_dt(mesh, U, (theta, scale, seed))


@pytest.mark.parametrize("dim", [1, 2])
@pytest.mark.parametrize("scale", [1e30, 1e36, 1e38, 2e38])
def test_dense_gas_at_rest(scale, dim):
    """Densities whose FP32 reciprocal is not a normal number, in pressure equilibrium
    (a momentum would overflow the FP32 squares and so be seen)."""
    mesh = inputs.mesh_dict("euler", dim, 3, {1: [70], 2: [9, 7]}[dim], [0.0] * dim, [1.0, 0.7][:dim], 1.4, vol="central", cfl=1e-11)
    for seed in range(3):
        rng = np.random.default_rng(seed)
        shape = (int(np.prod(mesh["cells"][:dim])), 4 ** dim)
        rho, p = scale * rng.uniform(0.9, 1.5, shape), np.full(shape, 0.5 * scale)
        _check_dt(mesh, inputs.euler_cons(1.4, rho, [np.zeros(shape)] * dim, p), (scale, dim, seed))


@pytest.mark.parametrize("eq,dim", [("euler", 1), ("euler", 2), ("euler", 3), ("glm_mhd", 2)])
@pytest.mark.parametrize("scale", [1e-18, 1e-21, 1e-24, 1e-27, 1e-28, 1e-29, 1e-31, 1e24])
def test_fast_thin_gas(scale, eq, dim):
    """Velocities up to 1e7 in a thin gas: squares of the momenta below the FP32 range."""
    cells = {1: [40], 2: [7, 5], 3: [4, 3, 3]}[dim]
    mesh = inputs.mesh_dict(eq, dim, 3, cells, [0.0] * dim, [1.0, 0.7, 1.3][:dim], 1.4, vol="central", cfl=1e-11,
                            c_h=0.3 if eq == "glm_mhd" else 0.0)
    for seed in range(4):
        rng = np.random.default_rng(seed)
        shape = (int(np.prod(cells)), 4 ** dim)
        speed = [1e2, 1e5, 1e6, 1e7][seed]
        rho = scale * _decades(rng, -0.3, 0.3, shape)
        v = [speed * rng.uniform(-1.0, 1.0, shape) for _ in range(3)]
        p = rho * speed ** 2 * _decades(rng, -2.0, 0.0, shape)
        if eq == "euler":
            U = inputs.euler_cons(1.4, rho, v[:dim], p)
        else:
            B = [np.sqrt(scale) * speed * rng.uniform(-0.5, 0.5, shape) for _ in range(3)]
            U = inputs.mhd_cons(1.4, rho, v, p, B, np.sqrt(scale) * 0.1 * np.ones(shape))
        _check_dt(mesh, U, (scale, eq, dim, seed))


def test_cells_beyond_the_fp32_range():
    """1/dx without a normal FP32 value."""
    mesh = inputs.mesh_dict("euler", 1, 3, [70], [0.0], [1e44], 1.4, vol="central", cfl=1e-11)
    for seed in range(6):
        rng = np.random.default_rng(seed)
        shape = (70, 4)
        rho, v = rng.uniform(0.9, 1.1, shape), 1e15 * rng.uniform(-0.1, 0.1, shape)
        p = 1e30 * rng.uniform(0.99, 1.01, shape)
        _check_dt(mesh, inputs.euler_cons(1.4, rho, [v], p), seed)


@pytest.mark.parametrize("scale", [1.0, 1e-24, 1e-29])
def test_negative_pressure_is_reported(scale):
    """A step that drives the pressure below zero in a thin gas whose kinetic
    energy has no FP32 squares, while faster nodes hold the maximum."""
    oracle.build()
    mesh = inputs.mesh_dict("euler", 1, 3, [32], [0.0], [1.0], 1.4, cfl=0.4, vol="kep")
    (x,) = inputs.node_coords(mesh)
    rng = np.random.default_rng(0)
    fast, cold = np.exp(-((x - 0.125) / 0.06) ** 2), np.exp(-((x - 0.65) / 0.15) ** 2)
    v = 1e6 * (1.0 + 3.0 * fast) + 3e5 * cold * rng.uniform(-1.0, 1.0, x.shape)
    p = scale * 1e12 * (0.05 + 2.0 * fast) * (1.0 - 0.999 * cold)
    U = inputs.euler_cons(1.4, scale * np.ones_like(x), [v], p)
    G = oracle.step(mesh, U, oracle.cfl_dt(mesh, U))
    assert np.min(0.4 * (G[2] - 0.5 * G[1] ** 2 / G[0])) < -1e-5 * np.max(0.4 * G[2])
    with crkfr.Solver(mesh, prec="fp64") as s:
        s.set_state(U)
        s.sync()
        assert s.info()["status"] == crkfr.CR_OK
        s.step(1)
        with pytest.raises(crkfr.CrError) as ei:
            s.sync()
            s.get_state()
        assert ei.value.status == crkfr.CR_ENONPHYSICAL

"""The forms of the volume kernel for small meshes against the general one, on
the same flow: a state on a small mesh, and copies of it side by side on a
periodic mesh large enough for the general form, advanced by the same steps.
The cells have the same size (a power of two), so both take the same dt and
differ by the rounding of the volume form alone: a step's increment is at most
a tenth of the state, so FP64 1e-13 stands for about a thousand roundings of
it, FP32 1e-6 (increments in single precision) for about a hundred.
"""
import numpy as np
import pytest

from paper_2604_02125_gb300 import crkfr, inputs
from parity_util import check_close

pytestmark = pytest.mark.gpu

# (system, dimension, cells of the small mesh, copies); 4864 = 32 x 152 elements in 2D and 3D
MESHES = [("euler", 1, [96], [512]), ("euler", 1, [77], [640]),
          ("euler", 2, [16, 19], [4, 4]), ("euler", 3, [8, 8, 19], [2, 2, 1]),
          ("glm_mhd", 2, [16, 19], [4, 4])]


def _run(eq, dim, N, cells, vol, prec, U):
    mesh = inputs.mesh_dict(eq, dim, N, cells, [0.0] * dim, [c * 0.125 for c in cells], 1.4, vol=vol,
                            c_h=2.0 if eq == "glm_mhd" else 0.0)
    if U is None:
        U = inputs.smooth_random_field(mesh, seed=5 + N, amp=0.1)
    with crkfr.Solver(mesh, prec=prec) as s:
        s.set_state(U)
        s.step(2)
        return U, s.get_state(), s.info()["dt"]


@pytest.mark.parametrize("vol", ["ec", "kep", "central"])
@pytest.mark.parametrize("prec", ["fp64", "fp32"])
@pytest.mark.parametrize("eq,dim,cells,copies", MESHES)
def test_copies(eq, dim, cells, copies, prec, vol):
    if eq == "glm_mhd" and vol == "kep":
        pytest.skip("no such flux")
    if dim > 1 and prec == "fp32":
        pytest.skip("one form")
    for N in range(1, 6):
        U, G, dt = _run(eq, dim, N, cells, vol, prec, None)
        tile = [1] + copies[::-1] + [1]

        def repeat(X):
            M, NP = X.shape[0], X.shape[-1]
            return np.ascontiguousarray(np.tile(X.reshape([M] + cells[::-1] + [NP]), tile).reshape(M, -1, NP))

        _, Gc, dtc = _run(eq, dim, N, [c * k for c, k in zip(cells, copies)], vol, prec, repeat(U))
        what = "%s%dd N=%d %s %s" % (eq, dim, N, vol, prec)
        assert abs(dt - dtc) <= 1e-13 * dt if prec == "fp64" else abs(dt - dtc) <= 1e-6 * dt, what
        check_close(Gc, repeat(G), 1e-13 if prec == "fp64" else 1e-6, what)

"""The kernel forms reported for a mesh are those its step launches: the forms for
small meshes and the general one, with sizes taken from the device's SM count, and
the two forms of the 1D volume kernel against each other bit for bit.
"""
import numpy as np
import pytest

from paper_2604_02125_gb300 import crkfr, inputs

pytestmark = pytest.mark.gpu


def _info(eq, cells, N, prec, vol="ec", **kw):
    dim = len(cells)
    mesh = inputs.mesh_dict(eq, dim, N, cells, [0.0] * dim, [c * 0.125 for c in cells], 1.4, vol=vol,
                            c_h=2.0 if eq == "glm_mhd" else 0.0)
    with crkfr.Solver(mesh, prec=prec, **kw) as s:
        t = s.tuning_info()
    return t["volume"], t["elements_per_cta"], t["face"]


def _sms():
    import torch
    return torch.cuda.get_device_properties(0).multi_processor_count


@pytest.mark.parametrize("N", [2, 3, 4, 5])
@pytest.mark.parametrize("prec", ["fp64", "fp32"])
def test_1d(N, prec):
    few, many = 24 * _sms(), 24 * _sms() + 1
    per_warp = {2: 8, 3: 4, 4: 2, 5: 2}[N]       # groups of lanes that hold n (n-1)/2 pairs
    assert _info("euler", [few], N, prec)[:2] == ("pairs", per_warp)
    assert _info("euler", [many], N, prec)[:2] == ("lanes", 32)
    assert _info("euler", [few], N, prec, vol="central")[:2] == ("lanes", 32)
    assert _info("euler", [few], N, prec, scheme="rkfr") == ("lanes", 32, "line")
    by_line = prec == "fp64" or N <= 3
    assert _info("euler", [few], N, prec)[2] == ("line" if by_line else "lanes")


@pytest.mark.parametrize("eq,cells,N", [("euler", [16, 19], 3), ("euler", [16, 19], 5), ("euler", [300, 300], 1),
                                        ("glm_mhd", [16, 19], 3), ("euler", [8, 9, 11], 3)])
def test_fp64_tiles(eq, cells, N):
    assert _info(eq, cells, N, "fp64")[:2] == ("small tiles", 8 if (N + 1) ** (len(cells) - 1) % 4 == 0 or len(cells) == 3 else 16)
    assert _info(eq, cells, N, "fp32")[0] == "lanes"


def test_fp64_tiles_by_the_busiest_sm():
    sms = _sms()
    # degree 4, tiles of 32 elements in 5 warps against 16 in 3: one tile per SM, and a whole number of them
    assert _info("euler", [sms, 16], 4, "fp64")[:2] == ("small tiles", 16)
    assert _info("euler", [sms, 32], 4, "fp64")[:2] == ("lanes", 32)


@pytest.mark.parametrize("N", [2, 3, 4, 5])
@pytest.mark.parametrize("vol", ["ec", "kep"])
@pytest.mark.parametrize("prec", ["fp64", "fp32"])
def test_1d_forms_give_the_same_bits(N, vol, prec):
    """A periodic state on the form with a lane per pair, and 64 copies of it on the form
    with a thread per element, one step of the same dt (the cells are of the same size, a
    power of two): the same arithmetic in the same order."""
    cells = _sms()
    copies = 64

    def step(c, U):
        mesh = inputs.mesh_dict("euler", 1, N, [c], [0.0], [c * 0.125], 1.4, vol=vol)
        if U is None:
            U = inputs.smooth_random_field(mesh, seed=5 + N, amp=0.1)
        with crkfr.Solver(mesh, prec=prec, dt_fixed=2.0 ** -9) as s:
            s.set_state(U)
            s.step(1)
            return U, s.get_state(), s.tuning_info()["volume"]

    U, G, form = step(cells, None)
    assert form == "pairs"
    _, Gc, form = step(cells * copies, np.tile(U, (1, copies, 1)))
    assert form == "lanes"
    assert np.array_equal(Gc.reshape(U.shape[0], copies, cells, N + 1),
                          np.broadcast_to(G[:, None], (U.shape[0], copies, cells, N + 1)))

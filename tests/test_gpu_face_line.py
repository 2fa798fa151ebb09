"""The 1D face / update kernel with a thread per line of an element, and the
volume form with a lane per pair of nodes, against the forms that large meshes
take: a state on a small mesh, and copies of it side by side on a periodic mesh
beyond the bounds of both rules (24 and 1024 elements per SM), advanced with the
same fixed dt.  The forms do the same arithmetic in the same order, so the
states are equal bit for bit.  And the same step from buffers that start on an
odd 8-byte boundary, which the forms' 16-byte accesses have to leave alone.
"""
import numpy as np
import pytest

from paper_2604_02125_gb300 import crkfr, inputs

pytestmark = pytest.mark.gpu

CELLS = 45


def _mesh(N, cells, vol="ec"):
    return inputs.mesh_dict("euler", 1, N, [cells], [0.0], [cells * 0.125], 1.4, vol=vol)


def _run(mesh, U, prec, steps=3, **kw):
    with crkfr.Solver(mesh, prec=prec, dt_fixed=1e-3, **kw) as s:
        s.set_state(U)
        s.step(steps)
        return s.get_state()


@pytest.mark.parametrize("vol", ["ec", "kep", "central"])
@pytest.mark.parametrize("prec", ["fp64", "fp32"])
@pytest.mark.parametrize("N", [1, 2, 3, 4, 5])
def test_small_and_large_mesh_bit_for_bit(N, prec, vol):
    import torch
    copies = 1025 * torch.cuda.get_device_properties(0).multi_processor_count // CELLS + 1
    U = inputs.smooth_random_field(_mesh(N, CELLS, vol), seed=N, amp=0.1)
    big = np.ascontiguousarray(np.tile(U, (1, copies, 1)))
    G, Gb = _run(_mesh(N, CELLS, vol), U, prec), _run(_mesh(N, CELLS * copies, vol), big, prec)
    assert np.array_equal(Gb, np.tile(G, (1, copies, 1)))


@pytest.mark.parametrize("prec", ["fp64", "fp32"])
@pytest.mark.parametrize("N", [1, 2, 3, 4, 5])
def test_buffers_on_an_8_byte_boundary(N, prec):
    import torch
    mesh = _mesh(N, CELLS)
    U = inputs.smooth_random_field(mesh, seed=N, amp=0.1)
    ref = _run(mesh, U, prec, steps=1)
    for off_in, off_out in ((0, 1), (1, 0), (1, 1)):
        a, b = (torch.zeros(U.size + 1, dtype=torch.float64, device="cuda") for _ in range(2))
        u, out = a[off_in:off_in + U.size], b[off_out:off_out + U.size]
        u.copy_(torch.from_numpy(U).reshape(-1))
        crkfr.step_noalloc(mesh, u, out, prec=prec, dt_fixed=1e-3)
        torch.cuda.synchronize()
        assert np.array_equal(out.cpu().numpy().reshape(U.shape), ref), (off_in, off_out)

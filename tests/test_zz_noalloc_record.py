"""cr_step_noalloc's step record, which every call on a device reuses and each
call leaves clean for the next: calls of different systems, degrees and
precisions in turn, in place and out of place, with and without the dt output,
after a state whose wave speeds are far larger, on two streams one after the
other, against the regular path (dt 1e-14, state 1e-12: the same kernels on the
same data; a stale maximum or status would change dt or skip the update).
"""
import numpy as np
import pytest

from paper_2604_02125_gb300 import crkfr, inputs

pytestmark = pytest.mark.gpu


def _cases():
    fast, U = inputs.shear_layer_2d(cells=(6, 5), N=3)
    yield fast, inputs.euler_cons(1.4, U[0], [40.0 + U[1] / U[0], U[2] / U[0]], 900.0 * np.ones_like(U[0]))
    yield inputs.shear_layer_2d(cells=(6, 5), N=3)
    yield inputs.mhd_vortex_2d(cells=(5, 4), N=4)
    yield inputs.density_wave_1d(cells=33, N=5)
    yield inputs.tgv_3d(cells=(3, 4, 3), N=4)


def test_record_is_clean_for_the_next_call():
    import torch
    streams = [torch.cuda.Stream(), torch.cuda.Stream()]
    for rep in range(2):
        for k, (mesh, U) in enumerate(_cases()):
            for prec in ("fp64", "fp32"):
                with crkfr.Solver(mesh, prec=prec) as s:
                    s.set_state(U)
                    s.step(1)
                    ref, dt_ref = s.get_state(), s.info()["dt"]
                u = torch.from_numpy(U).cuda()
                out = u if (k + rep) % 2 else torch.full_like(u, 7.0)
                dt = torch.zeros(1, dtype=torch.float64, device="cuda")
                torch.cuda.synchronize()
                crkfr.step_noalloc(mesh, u, out, dt, prec=prec, stream=streams[(k + rep) % 2])
                torch.cuda.synchronize()
                assert abs(dt.item() - dt_ref) <= 1e-14 * dt_ref, (k, prec)
                got = out.cpu().numpy()
                assert np.linalg.norm(got - ref) <= 1e-12 * np.linalg.norm(ref), (k, prec)
                if out is not u:
                    assert np.array_equal(u.cpu().numpy(), U)

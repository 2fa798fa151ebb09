"""The face / update kernel's node mapping at its edges: ragged last tiles of
every remainder class, fewer elements than a tile, one element, elements whose
neighbour lies in another tile or wraps around, for every degree (a tile's
values are N+1 rounds of the CTA; the rounds cut through elements differently
for every N).  One step against the FP64 oracle, node by node, both
precisions, and the RKFR stage form of the same kernel.

Bars as in the variant matrix: state 1e-12 / 1e-5, in FP64 also the increment,
1e-10.  (In FP32 the increment's own rounding grows with the number of elements
across the box, as eps |D| / dx against |u_x|: 1.4e-3 for 95 elements at N = 5,
before and after the node mapping; a misplaced node moves the state by the
increment itself, 1e-3 to 1e-2, which the state's bar shows.  One element of
degree 1 has equal node values on a periodic box: its increment is zero.)
"""
import numpy as np
import pytest

import oracle
from paper_2604_02125_gb300 import crkfr, inputs
from parity_util import check_close, check_increment

pytestmark = pytest.mark.gpu

CELLS = {1: [[1], [31], [33], [95]], 2: [[1, 1], [31, 1], [3, 11], [8, 8], [13, 5]],
         3: [[1, 1, 1], [3, 11, 1], [4, 4, 4], [5, 3, 7]]}
CASES = [("euler", d, c) for d in (1, 2, 3) for c in CELLS[d]] + [("glm_mhd", 2, c) for c in CELLS[2]]


@pytest.mark.parametrize("scheme", ["crkfr", "rkfr"])
@pytest.mark.parametrize("prec", ["fp64", "fp32"])
@pytest.mark.parametrize("eq,dim,cells", CASES)
def test_edges(eq, dim, cells, prec, scheme):
    oracle.build()
    for N in range(1, 6):
        mesh = inputs.mesh_dict(eq, dim, N, cells, [0.0] * dim, [1.0, 0.8, 1.2][:dim], 1.4,
                                c_h=2.0 if eq == "glm_mhd" else 0.0)
        mesh["scheme"] = scheme
        U = inputs.smooth_random_field(mesh, seed=17 + N, amp=0.1)
        s = crkfr.Solver(mesh, prec=prec)
        s.set_state(U)
        s.step(1)
        G, dt = s.get_state(), s.info()["dt"]
        s.close()
        O = (oracle.rkfr_step if scheme == "rkfr" else oracle.step)(mesh, U, dt)
        what = "%s%dd %s N=%d %s %s" % (eq, dim, cells, N, prec, scheme)
        check_close(G, O, 1e-12 if prec == "fp64" else 1e-5, what)
        if prec == "fp64" and np.max(np.abs(O - U)) > 1e-13:
            check_increment(G, O, U, 1e-10, what)

"""PPM edges clipped to a neighbour's value are that value, however small beside
the cell's own: densities rising from e through 1, 10 to 20 within three cells
(the cell of density 1 has its low edge clipped to e), for e down to where 1 - e
rounds to 1, pressure and velocity uniform.  One step against the oracle at the
bar of the FP64 form, which holds D to 1e-12 of itself in every cell."""
import numpy as np
import pytest

import oracle
import problems as pb
from problems import ct
from tests.test_gpu_parity import TOL64, assert_parity, gb  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("divb", ["glm", "ct"])
@pytest.mark.parametrize("axis", [0, 1, 2])
@pytest.mark.parametrize("e", [1e-4, 1e-8, 1e-12, 1e-20])
def test_clipped_edges(gb, e, axis, divb):  # noqa: F811
    g = pb.periodic_box(ndim=3).with_(nx=(16, 16, 16), nroot=(1, 1, 1), blocks=None, divb=divb, rho_floor=1e-30)
    P = pb.empty_prims(g)
    shape = [1, 1, 1, 1]
    shape[3 - axis] = 16
    P[:, 0] = np.asarray([e] * 6 + [1.0, 10.0] + [20.0] * 8).reshape(shape)
    P[:, 1] = 1.0
    P[:, 2 + axis] = -0.3
    s, o = gb.Solver(g), oracle.Oracle(g)
    for x in (s, o):
        x.set_prims(P)
        if divb == "ct":
            x.set_faces(np.zeros(ct.face_count(g)))
    dt = o.cfl_dt()
    for x in (s, o):
        x.step(dt)
    assert_parity(s.cons(), o.cons(), TOL64, f"{e} {axis} {divb}", g)

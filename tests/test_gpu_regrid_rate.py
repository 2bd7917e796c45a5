"""The CFL step of a context that held another state before it received a
transferred one is that of the transferred state."""
import pytest

import problems as pb
from problems import ct
from tests.test_gpu_parity import gb  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("divb", ["glm", "ct"])
def test_rate_of_the_transferred_state(gb, divb):  # noqa: F811
    g = pb.periodic_box(ndim=3).with_(divb=divb, ch=0.1)
    P = pb.random_periodic_prims(g)
    cold = P.copy()
    cold[:, 1] *= 1e-3
    F = ct.random_potential_faces(g)
    held, other, alone = (gb.Solver(g) for _ in range(3))
    for s, prims, scale in ((held, cold, 0.1), (other, P, 1.0), (alone, P, 1.0)):
        s.set_prims(prims)
        if divb == "ct":
            s.set_faces(scale * F)
        s.cfl_dt()
    gb.bhac_regrid_transfer(other.ctx, held.ctx)
    # the inversion recovers the primitives to its tolerance
    assert held.cfl_dt() == pytest.approx(alone.cfl_dt(), rel=1e-10)

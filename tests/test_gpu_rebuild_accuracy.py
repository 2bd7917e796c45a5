"""The conserved state that FP64 cells are given from their primitives (floored
cells in every stage) is as accurate as the oracle's: the rms difference of S_1
and tau after three steps of a torus that is mostly floored atmosphere.

Bar: sqrt(2) times the oracle's own rms distance from the same scheme in long
double arithmetic on these inputs (S_1 3.54e-15 and tau 2.03e-16 with the cleaning
form, 2.85e-14 and 1.40e-15 with constrained transport, each relative to the
variable's size plus tau + D): what two equally accurate results differ by."""
import numpy as np
import pytest

import oracle
import problems as pb
from problems import ct
from tests.test_gpu_parity import gb  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("divb,dt,s1,tau", [("glm", 0.006281302310526371, 3.54e-15, 2.03e-16),
                                            ("ct", 0.05545652285218239, 2.85e-14, 1.40e-15)])
def test_rebuilt_states(gb, divb, dt, s1, tau):  # noqa: F811
    g = pb.torus_3d(nroot=(4, 2, 2)).with_(divb=divb)
    P = pb.fm_torus_prims(g)
    s, o = gb.Solver(g), oracle.Oracle(g)
    for x in (s, o):
        x.set_prims(P)
        if divb == "ct":
            x.set_faces(ct.fm_torus_faces(g, P))
        for _ in range(3):
            x.step(dt)
    ref, got = o.cons(), s.cons()
    E = np.abs(ref[:, 4] + ref[:, 0])
    for v, own in ((1, s1), (4, tau)):
        rms = np.sqrt(np.mean((np.abs(got[:, v] - ref[:, v]) / (np.abs(ref[:, v]) + E)) ** 2))
        assert rms <= np.sqrt(2.0) * own, (v, rms)

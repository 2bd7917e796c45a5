"""The light-cone test that leaves wave speeds out of the CFL maximum: the time
step with cleaning speeds below one and with constrained transport (none at
all), on hot magnetised states whose largest rate is not the innermost cell's,
for an adiabatic index on either side of the test's limit, equals the oracle's.
The bar is that of test_cfl_matches_oracle for the load (same formulas); the
stand-alone reduction after a step sees states that agree to 1e-12."""
import numpy as np
import pytest

import oracle
import problems as pb
from problems import ct
from tests.test_gpu_parity import gb  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("form", ["fp64", "mixed"])
@pytest.mark.parametrize("gamma_ad", [4.0 / 3.0, 2.2])
@pytest.mark.parametrize("kind", ["glm", "ct"])
def test_cfl_below_light_speed(gb, kind, gamma_ad, form):  # noqa: F811
    g = pb.torus_3d(nblock=(8, 8, 8), nroot=(4, 2, 4)).with_(gamma_ad=gamma_ad, ch=0.3, divb=kind)
    P = pb.fm_torus_prims(g.with_(gamma_ad=4.0 / 3.0))
    rng = np.random.default_rng(3)
    hot = rng.random(P[:, 0].shape) < 0.02
    P[:, 1] = np.where(hot, 50.0 * P[:, 0], P[:, 1])
    s, o = gb.Solver(g, form), oracle.Oracle(g)
    s.set_prims(P)
    o.set_prims(P)
    if kind == "ct":
        F = ct.fm_torus_faces(g, P)
        s.set_faces(F)
        o.set_faces(F)
    dt = o.cfl_dt()
    assert s.cfl_dt() == pytest.approx(dt, rel=1e-14)
    s.step(dt)
    o.step(dt)
    assert s.cfl_dt() == pytest.approx(o.cfl_dt(), rel=1e-11 if form == "fp64" else 1e-4)

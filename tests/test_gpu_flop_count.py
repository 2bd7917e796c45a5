"""The CFL rate in the operation count: below the light speed the cleaning form's
cells form their wave speeds in the second stage, at or above it the rate is
tabulated and none is formed."""
import pytest

import problems as pb
from tests.test_gpu_parity import gb  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("form", ["fp64", "mixed"])
@pytest.mark.parametrize("name", ["torus", "box"])
def test_wave_speeds_are_counted(gb, name, form):  # noqa: F811
    out = []
    for ch in (1.0, 0.5):
        g = (pb.torus_3d(nroot=(4, 3, 2)) if name == "torus" else pb.periodic_box(ndim=3)).with_(ch=ch)
        s = gb.Solver(g, form)
        s.set_prims(pb.fm_torus_prims(g) if name == "torus" else pb.random_periodic_prims(g))
        # a step so short that the inversions do not depend on ch
        out.append(s.count_flops(1e-9, nsamples=2000, seed=3)["fp64_flops"])
    # three directions' speeds, one of every two stages: at least ten operations each
    assert out[1] - out[0] > 15.0

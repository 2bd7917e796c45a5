"""A launch shape set with threads = 0 on a grid whose default CTA is smaller than
256 threads: the calls that a 256-thread CTA allows are accepted, the others are
refused, and the state does not depend on it."""
import numpy as np
import pytest

import problems as pb
from tests.test_gpu_parity import gb  # noqa: F401

pytestmark = pytest.mark.gpu


def _run(gb, g, P, *shape):  # noqa: F811
    s = gb.Solver(g, "mixed")
    if shape:
        s.set_launch(*shape)
    s.set_prims(P)
    s.cfl_dt()
    s.step(0.0)
    return s.cons()


@pytest.mark.parametrize("shape", [(0, 0, 0, 0, 0, 2), (0, 0, 0, 0, 1, 7), (8, 8, 0, 0, 1, 4), (8, 4, 0, 0, 0, 0),
                                   (0, 0, 0, 1, 0, 0)])
def test_default_threads(gb, shape):  # noqa: F811
    g = pb.torus_3d(nroot=(2, 2, 2), nblock=(8, 8, 8))
    P = pb.fm_torus_prims(g)
    assert np.array_equal(_run(gb, g, P, *shape), _run(gb, g, P))


@pytest.mark.parametrize("shape", [(0, 0, 0, 0, 0, 8), (0, 0, 64, 0, 0, 2), (0, 0, 288, 0, 0, 0)])
def test_refused(gb, shape):  # noqa: F811
    s = gb.Solver(pb.torus_3d(nroot=(2, 2, 2), nblock=(8, 8, 8)), "mixed")
    with pytest.raises(gb.BhacError) as e:
        s.set_launch(*shape)
    assert e.value.status == 1

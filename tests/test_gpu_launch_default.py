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


@pytest.mark.parametrize("nx,nroot", [((24, 20, 4), (6, 6, 4)), ((50, 44, 1), (12, 12, 1)), ((23, 29, 3), (5, 6, 5))])
@pytest.mark.parametrize("form", ["fp64", "mixed"])
def test_default_fits_any_block(gb, nx, nroot, form):  # noqa: F811
    """Block faces that no standard tile divides and that are too large for the
    shared memory as a whole, on grids of many blocks."""
    from paper_2108_12240_gb300 import autotune
    from tests.test_gpu_parity import TOL64, TOLMIX, assert_parity, one_step
    g = pb.periodic_box(ndim=3 if nx[2] > 1 else 2).with_(nx=nx, nroot=nroot, blocks=None)
    tx, ty = autotune.default_shape(g, form, 152)[:2]
    assert nx[0] % tx == 0 and nx[1] % ty == 0
    assert autotune.smem_bytes(tx, ty, g.ndim, form) <= autotune.SMEM_LIMIT
    s, o, _ = one_step(gb, g, pb.random_periodic_prims(g), form)
    assert_parity(s.cons(), o.cons(), TOL64 if form == "fp64" else TOLMIX, f"{nx} {form}", g)

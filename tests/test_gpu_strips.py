"""The stage kernel's strip reconstruction at the edges of its ranges: block
extents below, at and above a strip's six cells and the default tiles, with
every remainder of (extent + 2) / 6, against the oracle.  The bars are those
of test_gpu_parity (rounding order only): 1e-12 in FP64, 1e-5 mixed."""
import pytest

import problems as pb
from tests.test_gpu_parity import TOL64, TOLMIX, assert_parity, gb, one_step  # noqa: F401

pytestmark = pytest.mark.gpu

BLOCKS = [(3, 4, 3), (5, 7, 4), (6, 10, 5), (8, 3, 7), (11, 5, 3), (16, 6, 4), (22, 9, 3),
          (20, 16, 4)]  # the last: too large a tile for a third z-face plane in FP64


@pytest.mark.parametrize("form,tol", [("fp64", TOL64), ("mixed", TOLMIX)])
@pytest.mark.parametrize("recon", ["ppm", "minmod"])
@pytest.mark.parametrize("nx", BLOCKS)
def test_odd_blocks_3d(gb, nx, recon, form, tol):  # noqa: F811
    g = pb.periodic_box(ndim=3).with_(nx=nx, nroot=(2, 2, 2), blocks=None, recon=recon)
    s, o, _ = one_step(gb, g, pb.random_periodic_prims(g), form)
    assert_parity(s.cons(), o.cons(), tol, f"{nx} {recon} {form}", g)


@pytest.mark.parametrize("form,tol", [("fp64", TOL64), ("mixed", TOLMIX)])
@pytest.mark.parametrize("nx", [(3, 5), (7, 3), (20, 13), (40, 9)])
def test_odd_blocks_2d_torus(gb, nx, form, tol):  # noqa: F811
    g = pb.torus_2d().with_(nx=(*nx, 1), nroot=(4, 4, 1), blocks=None)
    s, o, _ = one_step(gb, g, pb.fm_torus_prims(g), form)
    assert_parity(s.cons(), o.cons(), tol, f"{nx} {form}", g)


@pytest.mark.parametrize("form,tol", [("fp64", TOL64), ("mixed", TOLMIX)])
@pytest.mark.parametrize("nx,ndim", [((3, 4, 5), 3), ((7, 6, 3), 3), ((17, 5, 4), 3), ((70, 3, 1), 2), ((5, 130, 1), 2)])
def test_constrained_transport_lines(gb, nx, ndim, form, tol):  # noqa: F811
    """Lines of the face-flux kernel below and above one segment (64 faces),
    CTAs whose lines span blocks, and remainders of the strips."""
    import numpy as np

    import oracle
    from problems import ct
    g = pb.periodic_box(ndim=ndim).with_(nx=nx, nroot=(2, 2, 2 if ndim == 3 else 1), blocks=None, divb="ct")
    P, F = pb.random_periodic_prims(g), ct.random_potential_faces(g)
    P[:, 8] = 0.0
    s, o = gb.Solver(g, form), oracle.Oracle(g)
    for x in (s, o):
        x.set_prims(P)
        x.set_faces(F)
    dt = o.cfl_dt()
    for x in (s, o):
        x.step(dt)
    assert_parity(s.cons(), o.cons(), tol, f"{nx} {form}", g)
    ref = o.faces()
    assert np.abs(s.faces() - ref).max() <= tol * np.abs(ref).max()

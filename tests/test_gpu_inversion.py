"""The inversion's root against the root in extended precision, where the
iteration has the least room: energy densities far below one, strong fields.

Random cells in a flat box: the conserved state of one set of primitives is
inverted (a stage of size 1e-30, which adds nothing to it) from another set that
differs by up to 20%, and again with numpy's long double, started at the
primitives found.  Bar on the pressure, per cell: the error that rounding alone
can cause.  E = tau + D is one addition and, with the field along x, B^2 and B.S
are one product each: these are taken as the library rounds them.  Each residual
of the system in (Z, v^2) is then a sum of products with at most eight roundings
per term (B^2/2 - E being one term), so it is known to 8 eps times the sum of
its terms' magnitudes; the inverse Jacobian carries that to (Z, v^2), 2 eps are added
for their own updates, and p = g (Z (1 - v^2) - D sqrt(1 - v^2)) carries it on
with four roundings of its own."""
import numpy as np
import pytest

import problems as pb
from tests.test_gpu_parity import gb  # noqa: F401

pytestmark = pytest.mark.gpu

LD = np.longdouble
EPS = 2.0 ** -53


def box(rho, p_over_rho, sigma, u, c2p):
    """A grid and random primitives of these sizes (spreads of 30%, velocities in
    random directions, the field along x)."""
    g = pb.periodic_box(ndim=2).with_(nx=(16, 16, 1), nroot=(4, 4, 1), blocks=None, c2p=c2p, rho_floor=1e-6 * rho,
                                      p_floor=1e-12 * rho)
    rng = np.random.default_rng(5)
    P = pb.empty_prims(g)

    def spread():
        return 1.0 + 0.3 * (2.0 * rng.random(P[:, 0].shape) - 1.0)

    d = rng.standard_normal(P[:, :3].shape)
    P[:, 0] = rho * spread()
    P[:, 1] = p_over_rho * P[:, 0] * spread()
    P[:, 2:5] = u * d / np.sqrt((d * d).sum(1, keepdims=True))
    P[:, 5] = np.sqrt(sigma * rho * (1.0 + 2.5 * p_over_rho)) * spread()
    return g, P


def pressure_and_bar(g, U, P, stop=0.0):
    """The pressure of the root nearest the primitives P for the conserved
    state U (flat), and the bar on its error."""
    gf = LD((g.gamma_ad - 1.0) / g.gamma_ad)
    D, S, E = U[:, 0].astype(LD), U[:, 1:4].astype(LD), (U[:, 4] + U[:, 0]).astype(LD)
    B2, BS = (U[:, 5] * U[:, 5]).astype(LD), (U[:, 5] * U[:, 1]).astype(LD)
    S2, ec = (S * S).sum(1), B2 / 2 - E
    W2 = 1 + (P[:, 2:5].astype(LD) ** 2).sum(1)
    Z, v2 = (P[:, 0] + P[:, 1] / gf) * W2, 1 - 1 / W2
    for _ in range(30):
        om, ZB, h = 1 - v2, Z + B2, BS * BS / (2 * Z * Z)
        sq = np.sqrt(om)
        f1 = ZB * ZB * v2 / 2 - h * (Z + ZB) - S2 / 2
        f2 = Z + ec + B2 * v2 / 2 - h - gf * Z * om + gf * D * sq
        j11, j12 = ZB * (v2 + 2 * h / Z), ZB * ZB / 2
        j21, j22 = 1 - gf * om + 2 * h / Z, gf * Z + B2 / 2 - gf * D / (2 * sq)
        det = j11 * j22 - j12 * j21
        Z, v2 = Z + (f2 * j12 - f1 * j22) / det, v2 + (f1 * j21 - f2 * j11) / det
    r1 = 8 * EPS * (ZB * ZB * v2 / 2 + h * (Z + ZB) + S2 / 2)
    r2 = 8 * EPS * (Z + abs(ec) + B2 * v2 / 2 + h + gf * Z * om + gf * D * sq)
    dZ = (abs(j22) * r1 + j12 * r2) / abs(det) + (2 * EPS + stop) * Z
    dv2 = (j21 * r1 + abs(j11) * r2) / abs(det) + 2 * EPS + stop * v2
    om = 1 - v2
    sq = np.sqrt(om)
    bar = gf * (dZ * om + dv2 * (Z + D / (2 * sq)) + 4 * EPS * (Z * om + D * sq))
    return gf * (Z * om - D * sq), bar


def check(gb, rho, p_over_rho, sigma, u, c2p, form, spread=0.2):  # noqa: F811
    g, P1 = box(rho, p_over_rho, sigma, u, c2p)
    s = gb.Solver(g, form)
    s.set_prims(P1)
    U1 = s.cons()
    s.set_prims(P1 * (1.0 + spread * (2.0 * np.random.default_rng(6).random(P1.shape) - 1.0)))
    s.set_cons(U1)
    s.stage(1, 1e-30)
    P, U, st = s.prims(), s.cons(), s.c2p_status()
    p, bar = pressure_and_bar(g, U, P, g.c2p_tol if c2p == "nk" else 0.0)
    ok = st.reshape(p.shape) == 0
    assert ok.mean() > 0.95
    err = np.abs(P[:, 1] - p)[ok]
    assert np.all(err <= bar[ok]), (float((err / bar[ok]).max()), float((err / p[ok]).max()))


# (products of two 1e-30 densities leave the FP32 range of the mixed form's fluxes)
@pytest.mark.parametrize("rho,form", [(r, f) for r in (1.0, 1e-11, 1e-13, 1e-14, 2e-15, 1e-16, 1e-30)
                                      for f in ("fp64", "mixed") if not (r < 1e-20 and f == "mixed")])
@pytest.mark.parametrize("c2p", ["newton", "nk"])
def test_small_densities(gb, rho, c2p, form):  # noqa: F811
    check(gb, rho, 1e-2, 0.1, 0.3, c2p, form)


@pytest.mark.parametrize("form", ["fp64", "mixed"])
@pytest.mark.parametrize("c2p", ["newton", "nk"])
@pytest.mark.parametrize("sigma", [1e2, 1e3, 1e5])
@pytest.mark.parametrize("u,spread", [(1e-3, 0.03), (1e-3, 0.2), (0.05, 0.001), (0.3, 0.01), (0.3, 0.2), (5.0, 0.2)])
def test_strong_magnetisation(gb, u, spread, sigma, c2p, form):  # noqa: F811
    check(gb, 1.0, 1e-2, sigma, u, c2p, form, spread)


@pytest.mark.parametrize("form", ["fp64", "mixed"])
@pytest.mark.parametrize("c2p", ["newton", "nk"])
@pytest.mark.parametrize("sigma,u", [(0.1, 1.0), (1e2, 0.3), (1e3, 1.0)])
def test_kernels_share_the_bits(gb, sigma, u, c2p, form):  # noqa: F811
    """Three and more steps in most cells: the fused kernel (solver fixed at compile
    time) and the split form (solver chosen at run time) agree bit for bit."""
    g, P = box(1.0, 1e-2, sigma, u, c2p)
    outs = []
    for chunks in (0, 3):
        s = gb.Solver(g, form)
        s.set_split(chunks)
        s.set_prims(P)
        s.cfl_dt()
        for _ in range(2):
            s.step(0.0)
        outs.append((s.prims(), s.cons(), s.c2p_status()))
    for a, b in zip(*outs):
        assert np.array_equal(a, b)

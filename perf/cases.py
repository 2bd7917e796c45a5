"""Performance cases: what a program does with this library, timed through its
public entry points.

One pass is an output interval of a run: the primitives (and, with constrained
transport, the face fields) are loaded from device memory, the CFL step is
reduced, the state advances by ``steps`` RK2 steps with the device's own time
step, directly or as one captured CUDA graph, and the primitives, the conserved
state (and the faces) are read back to device memory.  The plan a program keeps
(Solver: arena, ghost maps, metric tables, graph) is made in ``prepare``.

``exact`` restates the scheme on one global array in plain FP64 torch (no
blocks, no library code); grids with refinement levels have no such form there.
"""
import math

import numpy as np
import torch

import paper_2108_12240_gb300 as gb
import problems as pb
from problems import ct

NV = 9


def listed():
    return [
        # the smallest calls: the shock tube of the smoke check, 4 blocks, ten
        # steps between outputs (launches and latency are everything)
        dict(name="shock_small_fp64", kind="shock", nx=16, ny=16, rx=2, ry=2, form="fp64", steps=10),
        # the 2-D relativistic shock tube workload, 16 blocks of 32 x 32
        dict(name="shock_tube_fp64", kind="shock", nx=32, ny=32, rx=4, ry=4, form="fp64", steps=10),
        # the axisymmetric torus workload, 256 blocks of 16 x 16: direct launches
        # in FP64, and a captured graph of ten steps in the mixed form
        dict(name="torus_2d_fp64", kind="torus", nx=16, ny=16, rx=16, ry=16, form="fp64", steps=5),
        dict(name="torus_2d_mixed_graph", kind="torus", nx=16, ny=16, rx=16, ry=16, form="mixed", steps=10, graph=True),
        # the 3-D torus workload, 432 blocks of 16^3, both forms
        dict(name="torus_3d_fp64", kind="torus", nx=16, ny=16, nz=16, rx=12, ry=6, rz=6, form="fp64", steps=2),
        dict(name="torus_3d_mixed", kind="torus", nx=16, ny=16, nz=16, rx=12, ry=6, rz=6, form="mixed", steps=4),
        # the benchmark's torus in its block shape (32 x 32 x 16), at the largest
        # sizes whose inputs are quick to make: above 4 M cells the rate no longer
        # depends on the size
        dict(name="torus_3d_large_fp64", kind="torus", nx=32, ny=32, nz=16, rx=8, ry=4, rz=8, form="fp64", steps=2),
        dict(name="torus_3d_large_mixed", kind="torus", nx=32, ny=32, nz=16, rx=16, ry=4, rz=8, form="mixed", steps=2),
        # constrained transport (the method's own div B control), both forms
        dict(name="torus_3d_ct_fp64", kind="torus", nx=16, ny=16, nz=16, rx=8, ry=4, rz=4, form="fp64", divb="ct", steps=2),
        dict(name="torus_3d_ct_mixed", kind="torus", nx=16, ny=16, nz=16, rx=12, ry=6, rz=6, form="mixed", divb="ct",
             steps=2),
        # three refinement levels, 16^3 blocks (the AMR workload at a fifth of its leaves)
        dict(name="amr_torus_mixed", kind="amr", nx=16, rx=8, ry=2, rz=2, form="mixed", steps=2),
        # a flat periodic box in ragged blocks, with the second limiter and
        # Riemann solver
        dict(name="box_3d_ragged_mixed", kind="box", nx=12, ny=20, nz=9, rx=8, ry=4, rz=8, form="mixed", recon="minmod",
             riemann="tvdlf", steps=2),
    ]


def draw(rng):
    """A case of the same ranges: forms, schemes and launch modes that are used, 2-D from 1e3 to 3e5 cells and 3-D from
    1e4 to 4e6 (FP64: 2e6), in even, odd and ragged blocks."""
    form = rng.choice(["fp64", "mixed"])
    case = dict(kind=rng.choice(["shock", "torus", "torus3", "torus3", "ct3", "amr", "box"]), form=form)
    if case["kind"] in ("shock", "torus"):
        case.update(nx=rng.choice([8, 12, 16, 20, 32]), ny=rng.choice([8, 11, 16, 24, 32]))
        cells = math.exp(rng.uniform(math.log(1e3), math.log(3e5)))
        r = max(1.0, cells / (case["nx"] * case["ny"]))
        a = math.exp(rng.uniform(-0.5, 0.5))
        case.update(rx=max(2, round(math.sqrt(r) * a)), ry=max(2, round(math.sqrt(r) / a)), steps=rng.choice([2, 4, 7, 10]))
        if rng.random() < 0.4:
            case["graph"] = True
    elif case["kind"] == "amr":
        case.update(nx=rng.choice([8, 16]), rx=8, ry=2, rz=rng.choice([1, 2]), steps=rng.choice([1, 2]))
    else:
        if case["kind"] == "box":
            case.update(nx=rng.choice([7, 12, 16, 24]), ny=rng.choice([9, 16, 20]), nz=rng.choice([5, 9, 16]))
        else:
            case.update(nx=rng.choice([8, 16, 32]), ny=rng.choice([8, 16, 24, 32]), nz=rng.choice([8, 16]))
        top = 1.2e6 if case["kind"] == "ct3" else (2e6 if form == "fp64" else 4e6)
        cells = math.exp(rng.uniform(math.log(1e4), math.log(top)))
        r = max(1.0, cells / (case["nx"] * case["ny"] * case["nz"])) ** (1.0 / 3.0)
        b = [r * math.exp(rng.uniform(-0.3, 0.3)) for _ in range(2)]
        b.append(r ** 3 / (b[0] * b[1]))
        case.update(rx=max(2, int(b[0])), ry=max(2, int(b[1])), rz=max(2, int(b[2])), steps=rng.choice([1, 2]))
        if case["kind"] == "ct3":
            case.update(divb="ct")
        if case["kind"] in ("torus3", "ct3"):
            case["kind"] = "torus"
            if case["rz"] * case["nz"] % 2:
                case["rz"] += 1
    if case["kind"] != "amr":
        case["recon"] = rng.choice(["ppm", "ppm", "minmod"])
        case["riemann"] = rng.choice(["hll", "hll", "tvdlf"])
        if rng.random() < 0.15 and not case.get("divb"):
            case["c2p"] = "nk"
    return case


def grid_of(case):
    opt = {k: case[k] for k in ("recon", "riemann", "divb", "c2p") if k in case}
    n, r = (case["nx"], case.get("ny", 1), case.get("nz", 1)), (case["rx"], case["ry"], case.get("rz", 1))
    if case["kind"] == "amr":
        return pb.amr_torus(root=r, nblock=case["nx"], **opt)
    if case["kind"] == "shock":
        return pb.shock_tube_2d().with_(nx=n, nroot=r, blocks=None, **opt)
    if case["kind"] == "box":
        return pb.periodic_box(ndim=3).with_(nx=n, nroot=r, blocks=None, **opt)
    g = pb.torus_3d() if n[2] > 1 else pb.torus_2d()
    return g.with_(nx=n, nroot=r, blocks=None, **opt)


def inputs(case, grid, seed):
    """Initial primitives (and faces) on the GPU, from the seed alone."""
    gen = torch.Generator(device="cuda").manual_seed(seed)
    faces = None
    if case["kind"] == "shock":
        P = torch.from_numpy(pb.shock_tube_prims(grid)).cuda()
        # the two states with a seeded 1% spread, so that no two runs are alike
        xi = 1.0 + 0.01 * (2.0 * torch.rand(P[:, :2].shape, generator=gen, device="cuda", dtype=torch.float64) - 1.0)
        P[:, :2] *= xi
    elif case["kind"] == "box":
        P = torch.from_numpy(pb.random_periodic_prims(grid, seed)).cuda()
    else:
        # the torus does not depend on phi: one plane per block, repeated, then
        # the +-2% pressure perturbation of the torus cells
        plane = pb.fm_torus_prims(grid.with_(nx=(grid.nx[0], grid.nx[1], 1)), pert=0.0)
        if case.get("divb") == "ct":
            thin = grid.with_(nx=(grid.nx[0], grid.nx[1], 1))
            parts = ct.split_faces(thin, ct.fm_torus_faces(thin, plane)) if grid.ndim == 3 else None
            if parts is None:
                faces = torch.from_numpy(ct.fm_torus_faces(grid, plane)).cuda()
            else:
                nz = grid.nx[2]
                up = [torch.from_numpy(parts[d]).cuda().expand(-1, nz, -1, -1) for d in (0, 1)]
                up.append(torch.zeros((grid.nb, nz + 1, grid.nx[1], grid.nx[0]), dtype=torch.float64, device="cuda"))
                faces = torch.cat([p.reshape(grid.nb, -1) for p in up], dim=1).reshape(-1).contiguous()
        P = torch.from_numpy(plane).cuda().repeat(1, 1, grid.nx[2], 1, 1)
        x1 = torch.from_numpy(pb.cell_centres(grid.with_(nx=(grid.nx[0], 1, 1)))[0]).cuda()
        torus = P[:, 0] > 10.0 * grid.rho_floor * torch.exp(x1) ** grid.rho_floor_pow
        xi = torch.rand(P[:, 1].shape, generator=gen, device="cuda", dtype=torch.float64)
        P[:, 1] = torch.where(torus, P[:, 1] * (1.0 + 0.02 * (2.0 * xi - 1.0)), P[:, 1])
    return P.contiguous(), faces


def prepare(case, seed):
    grid = grid_of(case)
    P, faces = inputs(case, grid, seed)
    state = dict(prims=P, faces=faces, steps=case["steps"], graph=bool(case.get("graph")), cons=torch.empty_like(P),
                 faces_out=None if faces is None else torch.empty_like(faces))
    if not state["graph"]:
        state["solver"] = gb.Solver(grid, case["form"])
        return state
    stream = torch.cuda.Stream()  # a graph is captured on a stream of its own
    stream.wait_stream(torch.cuda.current_stream())
    s = state["solver"] = gb.Solver(grid, case["form"], stream=stream)
    s.set_prims(P)
    gb.bhac_cfl_dt(s.ctx, False)
    s.capture(case["steps"])
    return state


def run(state):
    if state["graph"]:
        with torch.cuda.stream(state["solver"].stream):
            return interval(state)
    return interval(state)


def interval(state):
    s = state["solver"]
    s.set_prims(state["prims"])
    if state["faces"] is not None:
        gb.bhac_set_faces(s.ctx, state["faces"].data_ptr(), True)
    gb.bhac_cfl_dt(s.ctx, False)
    if state["graph"]:
        s.replay()
    else:
        for _ in range(state["steps"]):
            s.step()
    out = dict(prims=s.prims_device(), cons=state["cons"])
    gb.bhac_get_cons(s.ctx, state["cons"].data_ptr(), True)
    if state["faces"] is not None:
        gb.bhac_get_faces(s.ctx, state["faces_out"].data_ptr(), True)
        out["faces"] = state["faces_out"]
    return out


def work(case):
    """Per zone and stage, the FP64 state read and written once (288 B; 252 B where the flux side reads the FP32
    primitives) and the scheme's operations (about 2200 in 3-D, 1600 in 2-D); the load and the read-back once a pass."""
    g = grid_of(case)
    stages = 2 * case["steps"] * g.ncells
    three = g.ndim == 3
    state = 288 if case["form"] == "fp64" else 252
    if case.get("divb") == "ct":
        state += 48 if three else 32
    return {"bytes": stages * state + g.ncells * 72 * 3, "flops": stages * (2200 if three else 1600)}


# ---------------------------------------------------------------------------
# The scheme in plain FP64 torch on one global array [var, k, j, i].
# ---------------------------------------------------------------------------
RHO, PRS, U1, B1, PSI = 0, 1, 2, 5, 8


def _metric(g, x1, x2, grad=False):
    """alpha, beta^1, the spatial metric's non-zero components (11, 13, 22, 33) and their derivatives along x1 and x2
    by the complex step."""
    def values(y1, y2):
        if g.coords == "mks":
            r, th, dr, dth = torch.exp(y1), math.pi * y2, torch.exp(y1), math.pi
        else:
            r, th, dr, dth = y1, y2, torch.ones_like(y1), 1.0
        s2, c = torch.sin(th) ** 2, torch.cos(th)
        Sig = r * r + g.spin ** 2 * c * c
        z = 2.0 * g.mass * r / Sig
        return [1.0 / torch.sqrt(1.0 + z), z / (1.0 + z) / dr, (1.0 + z) * dr * dr, -g.spin * s2 * (1.0 + z) * dr,
                Sig * dth * dth, s2 * (Sig + g.spin ** 2 * s2 * (1.0 + z))]
    x1, x2 = torch.broadcast_tensors(x1, x2)
    if g.coords == "cart":
        one, zero = torch.ones_like(x1), torch.zeros_like(x1)
        v = [one, zero, one, zero, one, one]
        d = [[zero] * 6, [zero] * 6]
    else:
        v, h = values(x1, x2), 1e-30
        d = [[q.imag / h for q in values(torch.complex(x1, torch.full_like(x1, h)), x2.to(torch.complex128))],
             [q.imag / h for q in values(x1.to(torch.complex128), torch.complex(x2, torch.full_like(x2, h)))]] if grad else None
    m = dict(zip(("al", "be", "g11", "g13", "g22", "g33"), v))
    det = m["g11"] * m["g33"] - m["g13"] ** 2
    m.update(i11=m["g33"] / det, i13=-m["g13"] / det, i33=m["g11"] / det, i22=1.0 / m["g22"], sg=torch.sqrt(m["g22"] * det), d=d)
    return m


def _lower(m, a):
    return [m["g11"] * a[0] + m["g13"] * a[2], m["g22"] * a[1], m["g13"] * a[0] + m["g33"] * a[2]]


def _raise(m, a):
    return [m["i11"] * a[0] + m["i13"] * a[2], m["i22"] * a[1], m["i13"] * a[0] + m["i33"] * a[2]]


def _dot(a, b):
    return a[0] * b[0] + a[1] * b[1] + a[2] * b[2]


def _derived(g, m, P):
    q = dict(m=m, P=P)
    u, B = P[U1:U1 + 3], P[B1:B1 + 3]
    ul, Bl = _lower(m, u), _lower(m, B)
    W = torch.sqrt(1.0 + _dot(u, ul))
    v, vl = [x / W for x in u], [x / W for x in ul]
    Bsq, Bv = _dot(B, Bl), _dot(B, vl)
    b2 = Bsq / W ** 2 + Bv ** 2
    rhoh = P[RHO] + g.gamma_ad / (g.gamma_ad - 1.0) * P[PRS]
    Z = rhoh * W * W
    D = P[RHO] * W
    S = [(Z + Bsq) * a - Bv * b for a, b in zip(vl, Bl)]
    tau = Z - P[PRS] + Bsq - 0.5 * b2 - D
    q.update(W=W, v=v, vl=vl, B=B, Bl=Bl, Bsq=Bsq, Bv=Bv, b2=b2, rhoh=rhoh, ptot=P[PRS] + 0.5 * b2, S=S, D=D, tau=tau,
             U=torch.stack([D, *S, tau, B[0], B[1], B[2], P[PSI]]))
    return q


def _stress(q, i, j):
    """W^i_j."""
    return q["S"][j] * q["v"][i] + (q["ptot"] if i == j else 0.0) - q["B"][i] * q["Bl"][j] / q["W"] ** 2 - q["Bv"] * q["B"][i] * q["vl"][j]


def _flux(q, d, ch):
    m, v, B, psi = q["m"], q["v"], q["B"], q["P"][PSI]
    al, be = m["al"], [m["be"], 0.0, 0.0]
    gi = [[m["i11"], 0.0, m["i13"]], [0.0, m["i22"], 0.0], [m["i13"], 0.0, m["i33"]]][d]
    Sd = _raise(m, q["S"])[d]
    F = [q["D"] * (al * v[d] - be[d])]
    F += [al * _stress(q, d, j) - be[d] * q["S"][j] for j in range(3)]
    F += [al * (Sd - q["D"] * v[d]) - be[d] * q["tau"]]
    F += [(al * v[d] - be[d]) * B[j] - (al * v[j] - be[j]) * B[d] + al * gi[j] * psi for j in range(3)]
    F += [al * ch * ch * B[d] - be[d] * psi]
    return torch.stack(F)


def _speeds(g, q, d):
    m, vsq = q["m"], 1.0 - 1.0 / q["W"] ** 2
    cs2, ca2 = g.gamma_ad * q["P"][PRS] / q["rhoh"], q["b2"] / (q["rhoh"] + q["b2"])
    a2 = cs2 + ca2 - cs2 * ca2
    gdd, vd, be = (m["i11"], m["i22"], m["i33"])[d], q["v"][d], m["be"] if d == 0 else 0.0
    den = 1.0 - vsq * a2
    disc = torch.clamp(a2 * (1.0 - vsq) * (gdd * den - vd * vd * (1.0 - a2)), min=0.0)
    c, s = vd * (1.0 - a2), torch.sqrt(disc)
    return m["al"] * (c - s) / den - be, m["al"] * (c + s) / den - be


def _edges(g, P, ax):
    """Low and high edge values along axis ``ax`` of every cell two or more from that axis's ends."""
    n = P.shape[ax]
    a = [P.narrow(ax, k, n - 4) for k in range(5)]
    if g.recon == "minmod":
        dm, dp = a[2] - a[1], a[3] - a[2]
        mm = torch.where(dm * dp <= 0.0, torch.zeros_like(dm), torch.where(dm.abs() < dp.abs(), dm, dp))
        return a[2] - 0.5 * mm, a[2] + 0.5 * mm

    def face(p, q, r, s):
        v = 7.0 / 12.0 * (q + r) - 1.0 / 12.0 * (p + s)
        return torch.minimum(torch.maximum(v, torch.minimum(q, r)), torch.maximum(q, r))
    L, R, c = face(*a[:4]), face(*a[1:]), a[2]
    flat = (R - c) * (c - L) <= 0.0
    L, R = torch.where(flat, c, L), torch.where(flat, c, R)
    dd, m6 = R - L, 6.0 * (c - 0.5 * (L + R))
    lo, hi = dd * dd < dd * m6, dd * m6 < -dd * dd
    return torch.where(lo, 3.0 * c - 2.0 * R, L), torch.where(hi, 3.0 * c - 2.0 * L, R)


class _Plain:
    def __init__(self, g):
        self.g, dev = g, dict(dtype=torch.float64, device="cuda")
        self.N = [g.nroot[d] * g.nx[d] for d in range(3)]
        self.dx = [(g.xmax[d] - g.xmin[d]) / self.N[d] for d in range(3)]
        self.ct = g.divb == "ct"
        self.ch, self.kappa = (0.0, 0.0) if self.ct else (g.ch, g.kappa)
        self.at = lambda d, lo, n, off: g.xmin[d] + (torch.arange(lo, lo + n, **dev) + off) * self.dx[d]
        self.mc = _metric(g, self.at(0, 0, self.N[0], 0.5), self.at(1, 0, self.N[1], 0.5)[:, None], grad=True)
        r = torch.exp(self.at(0, 0, self.N[0], 0.5)) if g.coords == "mks" else self.at(0, 0, self.N[0], 0.5) * 0.0 + 1.0
        self.floor = [g.rho_floor * r ** g.rho_floor_pow, g.p_floor * r ** g.p_floor_pow]

    def to_global(self, blocks):
        g = self.g
        x = blocks.reshape(g.nroot[2], g.nroot[1], g.nroot[0], NV, g.nx[2], g.nx[1], g.nx[0])
        return x.permute(3, 0, 4, 1, 5, 2, 6).reshape(NV, *self.N[::-1]).contiguous()

    def to_blocks(self, x):
        g = self.g
        x = x.reshape(NV, g.nroot[2], g.nx[2], g.nroot[1], g.nx[1], g.nroot[0], g.nx[0])
        return x.permute(1, 3, 5, 0, 2, 4, 6).reshape(g.nb, NV, g.nx[2], g.nx[1], g.nx[0])

    def faces_global(self, faces):
        """Block face arrays -> one array per direction, N + 1 along it."""
        g, out = self.g, [torch.zeros([self.N[e] + (e == d) for e in (2, 1, 0)], dtype=torch.float64, device="cuda")
                          for d in range(self.g.ndim)]
        for b, d, at, part in self._face_parts(faces.reshape(g.nb, -1)):
            out[d][at] = part
        return out

    def faces_blocks(self, parts):
        g = self.g
        n = sum(int(np.prod(s)) for s in ct.face_shapes(g))
        out = torch.empty((g.nb, n), dtype=torch.float64, device="cuda")
        for b, d, at, part in self._face_parts(out):
            part.copy_(parts[d][at])
        return out.reshape(-1)

    def _face_parts(self, flat):
        g = self.g
        for b in range(g.nb):
            c, o = [int(v) for v in g.blocks[b][1:]], 0
            for d, shape in enumerate(ct.face_shapes(g)):
                n = int(np.prod(shape))
                at = tuple(slice(c[e] * g.nx[e], c[e] * g.nx[e] + g.nx[e] + (e == d)) for e in (2, 1, 0))
                yield b, d, at, flat[b, o:o + n].view(shape)
                o += n

    def pad(self, X, w, skip=None, prims=True):
        """Boundary rules: ``w`` cells on each side of every active dimension but ``skip`` (a face direction)."""
        g = self.g
        for d in range(g.ndim):
            if d == skip:
                continue
            ax, N = X.dim() - 1 - d, self.N[d]
            i = torch.arange(-w, N + w, device="cuda")
            lo, hi = i < 0, i >= N
            kinds = g.bc[d]
            src = i.clone()
            for m, kind, mirror, edge in ((lo, kinds[0], -1 - i, 0), (hi, kinds[1], 2 * N - 1 - i, N - 1)):
                src = torch.where(m, i % N if kind == "periodic" else mirror if kind == "axis" else torch.full_like(i, edge), src)
            Y = X.index_select(ax, src)
            for m, kind, side in ((lo, kinds[0], 0), (hi, kinds[1], 1)):
                k = m.nonzero().flatten()
                if kind == "axis":
                    part = Y.index_select(ax, k)
                    if g.ndim == 3:
                        # phi + pi; a face array normal to phi has its last plane equal to the first
                        za = X.dim() - 3
                        n = self.N[2]
                        p = torch.roll(part.narrow(za, 0, n), n // 2, za)
                        part = p if part.shape[za] == n else torch.cat([p, p.narrow(za, 0, 1)], za)
                    if prims:
                        part = part.clone()
                        part[U1 + 1].neg_()
                        part[B1 + 1].neg_()
                    Y = Y.index_copy(ax, k, part)
                elif kind == "noinflow" and prims:
                    part = Y.index_select(ax, k)
                    part[U1 + d] = torch.clamp(part[U1 + d], max=0.0) if side == 0 else torch.clamp(part[U1 + d], min=0.0)
                    Y = Y.index_copy(ax, k, part)
            X = Y
        return X

    def face_fluxes(self, P, faces):
        """Densitized fluxes through the faces normal to each active direction, 0..N along it and, across, the cells
        (with constrained transport one more on each side)."""
        g, ring, out = self.g, 1 if self.ct else 0, []
        Q = self.pad(P, 3)
        for d in range(g.ndim):
            X = Q
            for e in range(g.ndim):
                if e != d:
                    X = X.narrow(3 - e, 3 - ring, self.N[e] + 2 * ring)
            ax = 3 - d
            lowE, highE = _edges(g, X, ax)       # of cells -1 .. N
            n = self.N[d] + 1
            L, R = highE.narrow(ax, 0, n).clone(), lowE.narrow(ax, 1, n).clone()
            bad = (L[RHO] <= 0) | (L[PRS] <= 0) | (R[RHO] <= 0) | (R[PRS] <= 0)
            L, R = torch.where(bad, X.narrow(ax, 2, n), L), torch.where(bad, X.narrow(ax, 3, n), R)
            lo = [0 if e == d else -ring for e in range(2)]
            num = [n if e == d else self.N[e] + 2 * ring for e in range(2)]
            m = _metric(g, self.at(0, lo[0], num[0], 0.0 if d == 0 else 0.5), self.at(1, lo[1], num[1], 0.0 if d == 1 else 0.5)[:, None])
            if self.ct:
                Bn = self.pad(faces[d], 1, skip=d, prims=False) / m["sg"]
                L[B1 + d], R[B1 + d] = Bn, Bn
            F = self.riemann(m, L, R, d)
            if d == 1:
                rows = [r for r, kind in ((0, g.bc[1][0]), (n - 1, g.bc[1][1])) if kind == "axis"]
                if rows:
                    F[:, :, rows] = 0.0
            out.append(F)
        return out

    def riemann(self, m, L, R, d):
        g, ch = self.g, self.ch
        q, r = _derived(g, m, L), _derived(g, m, R)
        FL, FR = _flux(q, d, ch), _flux(r, d, ch)
        lm, lp = zip(_speeds(g, q, d), _speeds(g, r, d))
        be = m["be"] if d == 0 else 0.0
        c = m["al"] * torch.sqrt((m["i11"], m["i22"], m["i33"])[d]) * ch
        glm = torch.tensor([v in (PSI, B1 + d) for v in range(NV)], device="cuda").reshape(NV, 1, 1, 1)
        if g.riemann == "hll":
            p = torch.clamp(torch.maximum(*lp), min=0.0)
            s = torch.clamp(torch.minimum(*lm), max=0.0)
            p, s = torch.where(glm, torch.maximum(p, c - be), p), torch.where(glm, torch.minimum(s, -c - be), s)
            w = p - s
            F = torch.where(w > 0, (p * (FL - s * q["U"]) - s * (FR - p * r["U"])) / w, 0.5 * (FL + FR))
        else:
            a = torch.stack([x.abs() for x in (*lm, *lp)]).amax(0)
            a = torch.where(glm, torch.maximum(a, torch.maximum((c - be).abs(), (-c - be).abs())), a)
            F = 0.5 * (FL + FR) - 0.5 * a * (r["U"] - q["U"])
        return m["sg"] * F

    def sources(self, P):
        m, q = self.mc, _derived(self.g, self.mc, P)
        if self.g.coords == "cart":
            S = torch.zeros_like(P)
            S[PSI] = -self.kappa * P[PSI]
            return S
        Su = _raise(m, q["S"])
        W = [Su[i] * q["v"][j] + q["ptot"] * a - q["B"][i] * q["B"][j] / q["W"] ** 2 - q["Bv"] * q["B"][j] * q["v"][i]
             for i, j, a in ((0, 0, m["i11"]), (0, 2, m["i13"]), (1, 1, m["i22"]), (2, 2, m["i33"]))]
        E, S = q["tau"] + q["D"], torch.zeros_like(P)
        G = [W[0] * d[2] + 2.0 * W[1] * d[3] + W[2] * d[4] + W[3] * d[5] for d in m["d"]]
        for k, d in enumerate(m["d"]):
            S[1 + k] = 0.5 * m["al"] * G[k] + q["S"][0] * d[1] - E * d[0]
        (a1, b1), (a2, b2) = m["d"][0][:2], m["d"][1][:2]
        S[4] = 0.5 * m["be"] * G[0] + _stress(q, 0, 0) * b1 + _stress(q, 1, 0) * b2 - (Su[0] * a1 + Su[1] * a2)
        S[PSI] = -m["al"] * self.kappa * P[PSI] - P[PSI] * b1 + self.ch ** 2 * (q["B"][0] * a1 + q["B"][1] * a2)
        return m["sg"] * S

    def invert(self, U, P):
        """Newton in (Z, v^2) from the previous primitives, then the floors; U keeps its densitized form."""
        g, m, gf = self.g, self.mc, (self.g.gamma_ad - 1.0) / self.g.gamma_ad
        u = U / m["sg"]
        D, S, E, B = u[0], u[1:4], u[4] + u[0], u[5:8]
        Su = _raise(m, S)
        S2, Bsq, BS = _dot(Su, S), _dot(B, _lower(m, B)), _dot(B, S)
        old = _dot(P[U1:U1 + 3], _lower(m, P[U1:U1 + 3]))
        Z, v2 = (P[RHO] + P[PRS] / gf) * (1.0 + old), old / (1.0 + old)
        done = torch.zeros_like(Z, dtype=torch.bool)
        for _ in range(30):
            sq = torch.sqrt(1.0 - v2)
            f1 = (Z + Bsq) ** 2 * v2 - BS ** 2 * (2.0 * Z + Bsq) / Z ** 2 - S2
            f2 = Z - gf * (Z * (1.0 - v2) - D * sq) + 0.5 * Bsq * (1.0 + v2) - 0.5 * BS ** 2 / Z ** 2 - E
            j11 = 2.0 * (Z + Bsq) * v2 + 2.0 * BS ** 2 * (Z + Bsq) / Z ** 3
            j12, j21 = (Z + Bsq) ** 2, 1.0 - gf * (1.0 - v2) + BS ** 2 / Z ** 3
            j22 = gf * (Z - 0.5 * D / sq) + 0.5 * Bsq
            det = j11 * j22 - j12 * j21
            Zn, vn = Z + (f2 * j12 - f1 * j22) / det, v2 + (f1 * j21 - f2 * j11) / det
            Zn = torch.where(Zn > 0, Zn, 0.5 * Z)
            vn = torch.where(vn < 0, 0.5 * v2, torch.where(vn >= 1, 0.5 * (v2 + 1.0), vn))
            now = (Zn - Z).abs() <= 1e-12 * Zn
            Z, v2 = torch.where(done, Z, Zn), torch.where(done, v2, vn)
            done = done | now
        ok = done & torch.isfinite(Z) & (D > 0)
        sq = torch.sqrt(1.0 - v2)
        Q = torch.stack([D * sq, gf * (Z * (1.0 - v2) - D * sq)] + [(a + BS / Z * b) / ((Z + Bsq) * sq) for a, b in zip(Su, B)])
        Q = torch.where(ok, Q, P[:5])
        fl = (Q[RHO] < self.floor[0]) | (Q[PRS] < self.floor[1])
        Q[RHO], Q[PRS] = torch.maximum(Q[RHO], self.floor[0]), torch.maximum(Q[PRS], self.floor[1])
        usq = _dot(Q[2:5], _lower(m, Q[2:5]))
        fast = 1.0 + usq > g.w_max ** 2
        Q[2:5] = torch.where(fast, Q[2:5] * torch.sqrt((g.w_max ** 2 - 1.0) / usq), Q[2:5])
        Q = torch.cat([Q, u[5:]])
        return torch.where(fl | fast | ~ok, m["sg"] * _derived(g, m, Q)["U"], U), Q

    def rate(self, P):
        g, q, total = self.g, _derived(self.g, self.mc, P), 0.0
        for d in range(g.ndim):
            be = self.mc["be"].abs() if d == 0 else 0.0
            c = self.mc["al"] * torch.sqrt((self.mc["i11"], self.mc["i22"], self.mc["i33"])[d]) * self.ch + be
            total = total + torch.stack([*(s.abs() for s in _speeds(g, q, d)), c.expand_as(P[0])]).amax(0) / self.dx[d]
        return float(total.max())

    def curl(self, F):
        """d_t of the face fields: edge EMFs are means of four face fluxes."""
        n, g = self.N, self.g
        cut = lambda d, v, lo: F[d][v][tuple(slice(lo[e] + (0 if e == d or e >= g.ndim else 1),
                                                   lo[e] + (0 if e == d or e >= g.ndim else 1) + self._en[e]) for e in (2, 1, 0))]
        E = {}
        for a, (d, e) in ((2, (0, 1)), (0, (1, 2)), (1, (2, 0))):
            if g.ndim == 2 and a != 2:
                continue
            self._en = [n[k] if k == a else n[k] + 1 for k in range(3)]
            back = lambda k: [-1 if q == k else 0 for q in range(3)]
            E[a] = 0.25 * (cut(e, B1 + d, [0, 0, 0]) + cut(e, B1 + d, back(d)) - cut(d, B1 + e, [0, 0, 0]) - cut(d, B1 + e, back(e)))
        diff = lambda a, d: E[a].diff(dim=2 - d) / self.dx[d]
        R = [-diff(2, 1), diff(2, 0)]
        if g.ndim == 3:
            R = [R[0] + diff(1, 2), R[1] - diff(0, 2), -diff(1, 0) + diff(0, 1)]
        for r, kind in ((0, g.bc[1][0]), (n[1], g.bc[1][1])):
            if kind == "axis":
                R[1][:, r] = 0.0
        return R

    def stage(self, P, U, faces, dt, Un=None, fn=None):
        g, F = self.g, self.face_fluxes(P, faces)
        rhs = self.sources(P)
        for d in range(g.ndim):
            X = F[d]
            for e in range(g.ndim):
                if e != d and self.ct:
                    X = X.narrow(3 - e, 1, self.N[e])
            rhs = rhs - X.diff(dim=3 - d) / self.dx[d]
        V = U + dt * rhs
        if Un is not None:
            V = 0.5 * Un + 0.5 * V
        new = None
        if self.ct:
            new = [f + dt * r for f, r in zip(faces, self.curl(F))]
            if fn is not None:
                new = [0.5 * a + 0.5 * b for a, b in zip(fn, new)]
            V = torch.cat([V[:5], self.cell_field(new, V)])
        V, Q = self.invert(V, P)
        return Q, V, new

    def cell_field(self, faces, V):
        B = [0.5 * (f.narrow(2 - d, 0, self.N[d]) + f.narrow(2 - d, 1, self.N[d])) for d, f in enumerate(faces)]
        B += [V[B1 + 2]] * (3 - len(B))
        return torch.stack(B + [torch.zeros_like(B[0])])

    def run(self, P, faces, steps):
        P = self.to_global(P)
        if self.ct:
            faces = self.faces_global(faces)
            sg = self.mc["sg"]
            P = torch.cat([P[:5], self.cell_field(faces, P * sg) / sg])
        U = self.mc["sg"] * _derived(self.g, self.mc, P)["U"]
        for _ in range(steps):
            dt = self.g.cfl / self.rate(P)
            Q, V, new = self.stage(P, U, faces, dt)
            P, U, faces = self.stage(Q, V, new, dt, Un=U, fn=faces)
        out = dict(prims=self.to_blocks(P), cons=self.to_blocks(U))
        if self.ct:
            out["faces"] = self.faces_blocks(faces)
        return out


def exact(case, seed):
    grid = grid_of(case)
    if grid.nlevels > 1:
        return None
    P, faces = inputs(case, grid, seed)
    return _Plain(grid).run(P, faces, case["steps"])

// Staggered-mesh constrained transport (the div B control of the method's
// Sec. 2), in the FP64 form or the mixed form (T = float: the
// face states and fluxes in FP32 from the FP32 primitives, the fluxes stored,
// the EMFs, the face update and the face field in FP64, so the discrete
// divergence stays at FP64 round-off; the cell sources in FP32 and the
// inversion as in the mixed stage kernel).
//
// Evolved field: Phi^d = sqrt(gamma) B^d at the centre of every face normal to
// an active direction d.  A stage runs, after the usual ghost-cell fill:
//   ring   the faces one cell outside each block (across, in every active
//          transverse direction) copied from the neighbour that owns them;
//   flux   every face of the block and its ring: PPM/minmod states from the
//          ghosted primitives, the normal field of both states set to the
//          face's own Phi^d / sqrt(gamma), HLL/TVDLF flux (densitized);
//   faces  d_t Phi = -curl E on the block's faces, the edge EMF the mean of
//          the four face fluxes of B around the edge (E_3 = F^2(B^1) =
//          -F^1(B^2), and cyclically), then the RK stage combination;
//   cells  flux divergence, sources and RK combination of D, S_i, tau (and of
//          B^3 in 2-D), cell field sqrt(gamma) B^d = (Phi^d_low + Phi^d_high)/2,
//          then the inversion, floors and CFL rate of the stage kernel.
// Both blocks sharing a face compute its update from identical inputs (their
// ghost cells and ring faces hold the same values), so their copies agree and
// the discrete divergence sum_d dPhi^d/dx_d of every cell stays at round-off.
// Across refinement levels a ring face is a copy, or the mean of the two faces
// of the coarser cell it cuts, or of the finer faces on it; after the fluxes,
// a coarse face on a level boundary takes the mean of the finer fluxes, every
// edge EMF is stored, and an edge that a finer leaf touches takes the mean of
// the finer EMFs along it before the face update (host-built maps), so the
// coarse copy of a level-boundary face changes by the mean of the changes of
// the finer faces covering it.
// psi is not evolved (zero), and no cleaning speed enters the fluxes.
#include <algorithm>
#include <thread>

#include "ct.h"
#include "stage_impl.cuh"

namespace bhac {

CtGeom ct_geom(const bhac_grid_desc* d) {
  CtGeom g;
  g.ndim = d->ndim;
  for (int e = 0; e < 3; ++e) g.nx[e] = d->nx[e];
  long long off = 0, own = 0;
  for (int dd = 0; dd < 3; ++dd) {
    long long nf = 1, no = 1;
    for (int e = 0; e < 3; ++e) {
      const bool across = e != dd && e < d->ndim;
      g.fe[dd][e] = e == dd ? d->nx[e] + 1 : d->nx[e] + (across ? 2 : 0);
      g.fo[dd][e] = across ? 1 : 0;
      nf *= g.fe[dd][e];
      no *= d->nx[e] + (e == dd ? 1 : 0);
    }
    if (dd >= d->ndim) nf = no = 0;
    g.foff[dd] = off;
    g.nfd[dd] = nf;
    off += nf;
    g.own_off[dd] = own;
    g.nown_d[dd] = no;
    own += no;
  }
  g.nfb = off;
  g.nown_b = own;
  long long eo = 0;
  for (int a = 0; a < 3; ++a) {
    const bool active = d->ndim == 3 || a == 2;
    long long n = active ? 1 : 0;
    for (int e = 0; e < 3; ++e) {
      g.ee[a][e] = e == a ? d->nx[e] : d->nx[e] + (e < d->ndim ? 1 : 0);
      n *= g.ee[a][e];
    }
    g.eoff[a] = eo;
    eo += n;
  }
  g.nEb = eo;
  return g;
}


bool ct_ring_map(const bhac_grid_desc* desc, const bhac_block_desc* blocks, int nb, const CtGeom& g,
                 std::vector<long long>& dst, std::vector<long long>& src) {
  const int* nr = desc->nroot;
  std::vector<int> lut((size_t)nr[0] * nr[1] * nr[2], -1);
  for (int b = 0; b < nb; ++b) lut[((size_t)blocks[b].iz * nr[1] + blocks[b].iy) * nr[0] + blocks[b].ix] = b;
  long long N[3];
  for (int e = 0; e < 3; ++e) N[e] = (long long)nr[e] * desc->nx[e];
  dst.clear();
  src.clear();
  for (int b = 0; b < nb; ++b) {
    const int bc[3] = {blocks[b].ix, blocks[b].iy, blocks[b].iz};
    for (int d = 0; d < desc->ndim; ++d)
      for (int k = -g.fo[d][2]; k < g.fe[d][2] - g.fo[d][2]; ++k)
        for (int j = -g.fo[d][1]; j < g.fe[d][1] - g.fo[d][1]; ++j)
          for (int i = -g.fo[d][0]; i < g.fe[d][0] - g.fo[d][0]; ++i) {
            const int f[3] = {i, j, k};
            bool ring = false;
            for (int e = 0; e < 3; ++e)
              if (e != d && (f[e] < 0 || f[e] >= desc->nx[e])) ring = true;
            if (!ring) continue;
            long long G[3];
            for (int e = 0; e < 3; ++e) G[e] = (long long)bc[e] * desc->nx[e] + f[e];
            // boundary rules across the face (the along-d index is a face index and stays)
            for (int e = 0; e < desc->ndim; ++e) {
              if (e == d) continue;
              const int side = G[e] < 0 ? 0 : (G[e] >= N[e] ? 1 : -1);
              if (side < 0) continue;
              const int kind = desc->bc[e][side];
              if (kind == BHAC_BC_PERIODIC) {
                G[e] = ((G[e] % N[e]) + N[e]) % N[e];
              } else if (kind == BHAC_BC_OUTFLOW || kind == BHAC_BC_NOINFLOW) {
                G[e] = side == 0 ? 0 : N[e] - 1;
              } else {  // polar axis (x2): mirror, and phi + pi in 3-D
                G[e] = side == 0 ? -1 - G[e] : 2 * N[e] - 1 - G[e];
                if (desc->ndim == 3) G[2] = ((G[2] + N[2] / 2) % N[2] + N[2]) % N[2];
              }
            }
            if (desc->ndim == 3 && d != 2 && desc->bc[2][0] == BHAC_BC_PERIODIC) G[2] = ((G[2] % N[2]) + N[2]) % N[2];
            int ob[3], lf[3];
            for (int e = 0; e < 3; ++e) {
              if (G[e] < 0 || G[e] > N[e] || (e != d && G[e] == N[e])) return false;
              ob[e] = (int)(G[e] / desc->nx[e]);
              if (e == d && ob[e] >= nr[e]) ob[e] = nr[e] - 1;
              lf[e] = (int)(G[e] - (long long)ob[e] * desc->nx[e]);
            }
            const int o = lut[((size_t)ob[2] * nr[1] + ob[1]) * nr[0] + ob[0]];
            if (o < 0) return false;
            dst.push_back((long long)b * g.nfb + ring_index(g, d, i, j, k));
            src.push_back((long long)o * g.nfb + ring_index(g, d, lf[0], lf[1], lf[2]));
          }
  }
  return true;
}

namespace {

// Leaf blocks by (level, block coordinates): one dense table per level.
struct LeafFinder {
  std::vector<std::vector<int>> lut;
  void build(const bhac_grid_desc* d, const bhac_block_desc* blocks, int nb) {
    lut.resize(d->nlevels);
    for (int L = 0; L < d->nlevels; ++L) {
      size_t n = 1;
      for (int e = 0; e < 3; ++e) n *= (size_t)d->nroot[e] << (e < d->ndim ? L : 0);
      lut[L].assign(n, -1);
    }
    for (int b = 0; b < nb; ++b) {
      const int L = blocks[b].level;
      const size_t n0 = (size_t)d->nroot[0] << L, n1 = (size_t)d->nroot[1] << L;
      lut[L][((size_t)blocks[b].iz * n1 + blocks[b].iy) * n0 + blocks[b].ix] = b;
    }
  }
  int get(const bhac_grid_desc* d, int L, const long long bc[3]) const {
    if (L < 0 || L >= d->nlevels) return -1;
    long long n[3];
    for (int e = 0; e < 3; ++e) {
      n[e] = (long long)d->nroot[e] << (e < d->ndim ? L : 0);
      if (bc[e] < 0 || bc[e] >= n[e]) return -1;
    }
    return lut[L][(size_t)((bc[2] * n[1] + bc[1]) * n[0] + bc[0])];
  }
};

struct LevelCtx {
  const bhac_grid_desc* d;
  const CtGeom* g;
  LeafFinder leaves;
  long long ncell(int e, int L) const { return ((long long)d->nroot[e] * d->nx[e]) << (e < d->ndim ? L : 0); }
  // 0: a level-L leaf holds cell G; -1: a coarser leaf covers it; +1: finer leaves do
  int cover(int L, const long long G[3]) const {
    long long bc[3];
    for (int e = 0; e < 3; ++e) bc[e] = G[e] / d->nx[e];
    if (leaves.get(d, L, bc) >= 0) return 0;
    for (int Lc = L - 1; Lc >= 0; --Lc) {
      for (int e = 0; e < 3; ++e) bc[e] = (e < d->ndim ? G[e] >> (L - Lc) : G[e]) / d->nx[e];
      if (leaves.get(d, Lc, bc) >= 0) return -1;
    }
    return 1;
  }
  // Phi indices (ring layout, whole arena) whose mean is face G of direction dd
  // at level L (a face index along dd, cell indices across, inside the domain):
  // the face of the level-L leaf above it along dd, else below; the coarse face
  // it lies on or the two faces of the coarse cell it cuts; the finer faces on
  // it.  Returns the count (1, 2 or 4), 0 if the levels do not resolve it.
  int face_sources(int dd, int L, const long long G[3], long long src[4]) const {
    const long long Nd = ncell(dd, L);
    long long bc[3];
    int lf[3];
    for (int e = 0; e < 3; ++e)
      if (e != dd) {
        bc[e] = G[e] / d->nx[e];
        lf[e] = (int)(G[e] % d->nx[e]);
      }
    for (int above = 1; above >= 0; --above) {
      const long long cell = above ? G[dd] : G[dd] - 1;
      if (cell < 0 || cell >= Nd) continue;
      bc[dd] = cell / d->nx[dd];
      lf[dd] = (int)(G[dd] - bc[dd] * d->nx[dd]);
      const int b = leaves.get(d, L, bc);
      if (b >= 0) {
        src[0] = (long long)b * g->nfb + ring_index(*g, dd, lf[0], lf[1], lf[2]);
        return 1;
      }
    }
    long long cell[3] = {G[0], G[1], G[2]};
    if (cell[dd] >= Nd) cell[dd] = Nd - 1;
    const int cov = cover(L, cell);
    if (cov < 0 && L > 0) {
      long long H[3], H1[3];
      for (int e = 0; e < 3; ++e) H[e] = H1[e] = e < d->ndim ? G[e] >> 1 : G[e];
      if (!(G[dd] & 1)) return face_sources(dd, L - 1, H, src) == 1 ? 1 : 0;
      H1[dd] += 1;
      long long s1[4];
      if (face_sources(dd, L - 1, H, src) != 1 || face_sources(dd, L - 1, H1, s1) != 1) return 0;
      src[1] = s1[0];
      return 2;
    }
    if (cov <= 0 || L + 1 >= d->nlevels) return 0;
    int t[2], nt = 0;
    for (int e = 0; e < d->ndim; ++e)
      if (e != dd) t[nt++] = e;
    for (int q = 0; q < (1 << nt); ++q) {
      long long F[3] = {G[0], G[1], G[2]}, s1[4];
      F[dd] = 2 * G[dd];
      for (int u = 0; u < nt; ++u) F[t[u]] = 2 * G[t[u]] + ((q >> u) & 1);
      if (face_sources(dd, L + 1, F, s1) != 1) return 0;
      src[q] = s1[0];
    }
    return 1 << nt;
  }
  // cell q (0..3) around the edge along a at G (level L): across each active
  // transverse direction below (bit 0) or above (bit 1); periodic wrap; false
  // where it leaves the domain across another boundary
  bool edge_cell(int a, int L, const long long G[3], int q, long long C[3], int s[3]) const {
    int u = 0;
    for (int e = 0; e < 3; ++e) {
      C[e] = G[e];
      s[e] = 0;
      if (e == a || e >= d->ndim) continue;
      s[e] = (q >> u++) & 1;
      C[e] = G[e] - 1 + s[e];
      const long long N = ncell(e, L);
      if (C[e] < 0 || C[e] >= N) {
        if (d->bc[e][C[e] < 0 ? 0 : 1] != BHAC_BC_PERIODIC) return false;
        C[e] = ((C[e] % N) + N) % N;
      }
    }
    return true;
  }
};


// flux of variable v through face (d; i, j, k) of block b
__device__ __forceinline__ double xf_at(const CtArgs& c, int b, int d, int v, int i, int j, int k) {
  return c.xf[(long long)b * NV * c.g.nfb + NV * c.g.foff[d] + v * c.g.nfd[d] + (ring_index(c.g, d, i, j, k) - c.g.foff[d])];
}

__global__ void __launch_bounds__(256) ct_ring_kernel(const long long* __restrict__ dst, const long long* __restrict__ src,
                                                      long long n, double* phi) {
  for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < n; t += (long long)gridDim.x * blockDim.x)
    phi[dst[t]] = phi[src[t]];
}

__global__ void __launch_bounds__(256) ct_ring_mean_kernel(const long long* __restrict__ dst,
                                                           const long long* __restrict__ src, long long n,
                                                           double* phi) {
  for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < n; t += (long long)gridDim.x * blockDim.x) {
    double s = 0.0;
    int m = 0;
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const long long o = src[4 * t + q];
      if (o >= 0) {
        s += phi[o];
        ++m;
      }
    }
    phi[dst[t]] = s / m;
  }
}

// Coarse fluxes on level boundaries: the mean of the finer faces' fluxes, every variable.
__global__ void __launch_bounds__(256) ct_reflux_kernel(CtArgs c) {
  for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < c.nxr;
       t += (long long)gridDim.x * blockDim.x) {
    const long long stride = c.g.nfd[c.xr_d[t]];
    for (int v = 0; v < NV; ++v) {
      double s = 0.0;
      int m = 0;
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const long long o = c.xr_src[4 * t + q];
        if (o >= 0) {
          s += c.xf[o + v * stride];
          ++m;
        }
      }
      c.xf[c.xr_dst[t] + v * stride] = s / m;
    }
  }
}

__device__ __forceinline__ double to_t(double x, double) { return x; }
__device__ __forceinline__ float to_t(double x, float) { return narrow_f64(x); }

// Lines of cells along each direction d, the work units of the flux kernel: the
// ns[d] segments of nf[d] faces of every line through a block and its ring.  A
// CTA takes nu[d] units; CTAs [g0[d], g0[d + 1]) run direction d, one direction
// after the other, since the three directions' code together is larger than
// an SM's instruction cache.
struct CtLines {
  int nu[3], nf[3], ns[3];
  unsigned units[3], g0[4];
};
constexpr int kCtThreads = 256, kCtLine = 64;  // most faces of one segment

// Flux through face (D; i, j, k) of block b from the states PL, PR (D a
// compile-time direction, so they stay in registers); T the flux arithmetic
// (double: FP64 form; float: mixed form).
template <typename T, int D, bool FLAT>
__device__ __forceinline__ void ct_one_face(const StageArgs& a, const CtArgs& c, int b, int i, int j, int k,
                                            const T* EL, const T* ER, int es) {
  const int L = a.blk[4 * b];
  const int G1 = a.blk[4 * b + 1] * a.nx + i, G2 = a.blk[4 * b + 2] * a.ny + j;
  const int N1 = a.N1l[L];
  T F[NV];
  const long long face = ring_index(c.g, D, i, j, k);
  const bool axis = !FLAT && D == 1 && ((G2 == 0 && c.axis_lo) || (G2 == a.N2l[L] && c.axis_hi));
  if (axis) {
#pragma unroll
    for (int v = 0; v < NV; ++v) F[v] = T(0.0);
  } else {
    const int sd = D == 0 ? 1 : (D == 1 ? a.Nx : a.Nx * a.Ny);
    const int c0 = ((k + a.gz) * a.Ny + (j + a.gy)) * a.Nx + (i + a.gx);  // the cell above the face
    const T* Pb = (sizeof(T) == 8 ? reinterpret_cast<const T*>(a.P_in) : reinterpret_cast<const T*>(a.P32_in)) +
                  (size_t)b * NV * a.ncell;
    const double phi = c.phi_in[(long long)b * c.g.nfb + face];
    T PL[NV], PR[NV];
#pragma unroll
    for (int v = 0; v < NV; ++v) {
      PL[v] = ER[v * es];
      PR[v] = EL[v * es];
    }
    positivity_fallback(a, Pb, sd, c0, PL, PR);
    Met<T> m;
    T acg = T(1.0);
    if (FLAT) {
      m = flat_metric<T>();
    } else if (D == 0) {
      const size_t r = ((size_t)c.teo_f1[L] + (size_t)(G2 + 1) * (N1 + 3) + (G1 + 1)) * FREC;
      if (sizeof(T) == 8) {
        m = load_face_metric<T>(c.te_f1 + r);
        acg = T(c.te_f1[r + F_ACG]);
      } else {
        m = load_face_metric<T>(c.te_f1_32 + r);
        acg = T(c.te_f1_32[r + F_ACG]);
      }
    } else if (D == 1) {
      const size_t r = ((size_t)c.teo_f2[L] + (size_t)(G2 + 1) * (N1 + 2) + (G1 + 1)) * FREC;
      if (sizeof(T) == 8) {
        m = load_face_metric<T>(c.te_f2 + r);
        acg = T(c.te_f2[r + F_ACG]);
      } else {
        m = load_face_metric<T>(c.te_f2_32 + r);
        acg = T(c.te_f2_32[r + F_ACG]);
      }
    } else {
      const size_t r = ((size_t)c.teo_c[L] + (size_t)(G2 + 1) * (N1 + 2) + (G1 + 1)) * CREC;
      if (sizeof(T) == 8) {
        m = load_centre_metric<T>(c.te_c + r);
        acg = T(c.te_c[r + C_ACG3]);
      } else {
        m = load_centre_metric<T>(c.te_c32 + r);
        acg = T(c.te_c32[r + C_ACG3]);
      }
    }
    const T Bn = to_t(phi, T(0)) / m.sg;
    PL[B1 + D] = Bn;
    PR[B1 + D] = Bn;
    riemann_flux(m, acg, PL, PR, D, a.riemann, pick<T>(a.gam, a.gam_f), pick<T>(a.gam_fac, a.gam_fac_f), T(0.0), F);
  }
  const long long o = (long long)b * NV * c.g.nfb + NV * c.g.foff[D] + (face - c.g.foff[D]);
#pragma unroll
  for (int v = 0; v < NV; ++v) c.xf[o + v * c.g.nfd[D]] = to_double(F[v]);
}

// The units [u0, u0 + nu) of direction D: both edges of every cell of each
// line into shared memory, by strips of one variable (as the stage kernel's R),
// then the faces between them.  Edge (v, cell m, unit u) sits where consecutive
// lanes of a phase read and write consecutive words: cells fastest along x,
// units (consecutive in x) fastest otherwise.  A face used to reconstruct both
// its cells from six loads per variable; sharing a cell's edges halves that.
// Flux kernel on 128x64x64 cells FP64 1.35 -> 1.16 ms, on 192x96x96 mixed 0.54
// -> 0.44 ms (from the step: 7.69 -> 6.94 and 7.26 -> 6.88 ms per interval).
template <typename T, int D, bool FLAT>
__device__ __forceinline__ void ct_lines(const StageArgs& a, const CtArgs& c, const CtLines& w, unsigned u0, T* E,
                                         int4* unit) {
  const int nu = w.nu[D], nf = w.nf[D], nc = nf + 1, ns = w.ns[D], nces = nu * nc;
  constexpr int e1 = D == 0 ? 1 : 0, e2 = D == 2 ? 1 : 2;
  const int n1 = c.g.fe[D][e1], n2 = c.g.fe[D][e2], nd = c.g.fe[D][D];
  for (int t = threadIdx.x; t < nu; t += kCtThreads) {
    const unsigned u = u0 + t;
    int4 q = make_int4(-1, 0, 0, 0);  // block (-1: none), transverse indices, first face
    if (u < w.units[D]) {
      const unsigned r1 = u / (unsigned)n1, r2 = r1 / (unsigned)n2;
      q.y = (int)(u - r1 * n1) - c.g.fo[D][e1];
      q.z = (int)(r1 - r2 * n2) - c.g.fo[D][e2];
      q.x = (int)(r2 / (unsigned)ns);
      q.w = (int)(r2 - (unsigned)q.x * ns) * nf;
    }
    unit[t] = q;
  }
  __syncthreads();
  T* EL = E;
  T* ER = E + NV * nces;
  const int sd = D == 0 ? 1 : (D == 1 ? a.Nx : a.Nx * a.Ny), so = D == 0 ? 1 : nu;
  const T* P_all = sizeof(T) == 8 ? reinterpret_cast<const T*>(a.P_in) : reinterpret_cast<const T*>(a.P32_in);
  const int nst = (nc + kStrip - 1) / kStrip, nl = nu * nst;
  const FastDiv dv(nl), din(D == 0 ? nst : nu), dfa(D == 0 ? nf : nu);
  for (int t = threadIdx.x; t < NV * nl; t += kCtThreads) {
    int v, r, hi, lo;
    dv.split(t, v, r);
    din.split(r, hi, lo);
    const int m = D == 0 ? hi : lo, s = (D == 0 ? lo : hi) * kStrip;
    const int4 q = unit[m];
    const int n = (nd - q.w < nf ? nd - q.w : nf) + 1 - s;  // cells of the line from this strip on
    if (q.x < 0 || n <= 0) continue;
    const int first = q.w - 1 + s;
    const int i = D == 0 ? first : q.y, j = D == 0 ? q.y : (D == 1 ? first : q.z), k = D == 2 ? first : q.z;
    const T* p = P_all + ((size_t)q.x * NV + v) * a.ncell + ((k + a.gz) * a.Ny + (j + a.gy)) * a.Nx + (i + a.gx);
    const int o = v * nces + (D == 0 ? m * nc + s : s * nu + m);
    strip_edges<T, kStrip>(a.recon, p, sd, n, EL + o, ER + o, so);
  }
  __syncthreads();
  for (int t = threadIdx.x; t < nu * nf; t += kCtThreads) {
    int hi, lo;
    dfa.split(t, hi, lo);
    const int m = D == 0 ? hi : lo, f = D == 0 ? lo : hi;
    const int4 q = unit[m];
    const int face = q.w + f;
    if (q.x < 0 || face >= nd) continue;
    const int i = D == 0 ? face : q.y, j = D == 0 ? q.y : (D == 1 ? face : q.z), k = D == 2 ? face : q.z;
    const int o = D == 0 ? m * nc + f : f * nu + m;
    ct_one_face<T, D, FLAT>(a, c, q.x, i, j, k, EL + o + so, ER + o, nces);
  }
}

// Fluxes through every face of every block and its ring.
template <typename T, bool FLAT>
__global__ void __launch_bounds__(kCtThreads) ct_flux_kernel(StageArgs a, CtArgs c, CtLines w) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ int4 unit[kCtThreads / 2];
  T* E = reinterpret_cast<T*>(smem_raw);
  const unsigned g = blockIdx.x;
  if (g < w.g0[1])
    ct_lines<T, 0, FLAT>(a, c, w, g * w.nu[0], E, unit);
  else if (g < w.g0[2])
    ct_lines<T, 1, FLAT>(a, c, w, (g - w.g0[1]) * w.nu[1], E, unit);
  else
    ct_lines<T, 2, FLAT>(a, c, w, (g - w.g0[2]) * w.nu[2], E, unit);
}

// Four times the edge EMFs: E_3 at (i-1/2, j-1/2) of cell layer k, E_1 at
// (j-1/2, k-1/2) of column i, E_2 at (k-1/2, i-1/2) of row j.  (The quarter is
// exact wherever it is applied; the face update, bound by its 20 FP64
// instructions per face, applies it to 1/dx and needs 16.)
__device__ __forceinline__ double emf3x4(const CtArgs& c, int b, int i, int j, int k) {
  return xf_at(c, b, 1, B1, i, j, k) + xf_at(c, b, 1, B1, i - 1, j, k) - xf_at(c, b, 0, B2, i, j, k) -
         xf_at(c, b, 0, B2, i, j - 1, k);
}
__device__ __forceinline__ double emf1x4(const CtArgs& c, int b, int i, int j, int k) {
  return xf_at(c, b, 2, B2, i, j, k) + xf_at(c, b, 2, B2, i, j - 1, k) - xf_at(c, b, 1, B3, i, j, k) -
         xf_at(c, b, 1, B3, i, j, k - 1);
}
__device__ __forceinline__ double emf2x4(const CtArgs& c, int b, int i, int j, int k) {
  return xf_at(c, b, 0, B3, i, j, k) + xf_at(c, b, 0, B3, i, j, k - 1) - xf_at(c, b, 2, B1, i, j, k) -
         xf_at(c, b, 2, B1, i - 1, j, k);
}


// Four times the change of E_A from the edge at (i, j, k) to the next along e.
// E_A = (F^q(B^p) - F^p(B^q)) / 4 summed over the four faces around the edge,
// (p, q) the next directions after A: two flux arrays, whose elements are
// addressed by strides from the edge's (16 separate indices took most of the
// kernel's instructions).
template <int A>
__device__ __forceinline__ double emf_diff(const CtArgs& c, int b, int i, int j, int k, int e) {
  constexpr int p = (A + 1) % 3, q = (A + 2) % 3;  // E_3: p = 1, q = 2 (1-based)
  const CtGeom& g = c.g;
  const int sp[3] = {1, g.fe[p][0], g.fe[p][0] * g.fe[p][1]};  // strides of the arrays of direction p, q
  const int sq[3] = {1, g.fe[q][0], g.fe[q][0] * g.fe[q][1]};
  const double* X = c.xf + (long long)b * NV * g.nfb;
  const double* Q = X + NV * g.foff[q] + (B1 + p) * g.nfd[q] + (k + g.fo[q][2]) * sq[2] + (j + g.fo[q][1]) * sq[1] + (i + g.fo[q][0]);
  const double* P = X + NV * g.foff[p] + (B1 + q) * g.nfd[p] + (k + g.fo[p][2]) * sp[2] + (j + g.fo[p][1]) * sp[1] + (i + g.fo[p][0]);
  const int oq = sel3(e, sq[0], sq[1], sq[2]), op = sel3(e, sp[0], sp[1], sp[2]);
  const double lo = Q[0] + Q[-sq[p]] - P[0] - P[-sp[q]];
  return (Q[oq] + Q[oq - sq[p]] - P[op] - P[op - sp[q]]) - lo;
}

// d_t Phi = -curl E and the stage combination, one thread per owned face.
template <int DIM>
__global__ void __launch_bounds__(256) ct_face_kernel(StageArgs a, CtArgs c) {
  const double dt = block_dt(a);
  const unsigned n = (unsigned)a.nblocks * (unsigned)c.g.nown_b;
  for (unsigned t = blockIdx.x * blockDim.x + threadIdx.x; t < n; t += gridDim.x * blockDim.x) {
    const int b = (int)(t / (unsigned)c.g.nown_b);
    int d, i, j, k;
    owned_face(c.g, (int)(t - (unsigned)b * (unsigned)c.g.nown_b), d, i, j, k);
    const long long o = (long long)b * c.g.nfb + ring_index(c.g, d, i, j, k);
    const int G2 = a.blk[4 * b + 2] * a.ny + j;
    if (!a.flat && d == 1 && ((G2 == 0 && c.axis_lo) || (G2 == a.N2g && c.axis_hi))) {
      c.phi_out[o] = 0.0;  // sqrt(gamma) = 0 on the axis
      continue;
    }
    const double qx = 0.25 * a.idx[0], qy = 0.25 * a.idx[1], qz = 0.25 * a.idx[2];
    double R;
    if (d == 0) {
      R = -emf_diff<2>(c, b, i, j, k, 1) * qy;
      if (DIM == 3) R += emf_diff<1>(c, b, i, j, k, 2) * qz;
    } else if (d == 1) {
      R = emf_diff<2>(c, b, i, j, k, 0) * qx;
      if (DIM == 3) R -= emf_diff<0>(c, b, i, j, k, 2) * qz;
    } else {
      R = -emf_diff<1>(c, b, i, j, k, 0) * qx + emf_diff<0>(c, b, i, j, k, 1) * qy;
    }
    if (a.stage == 1)
      c.phi_out[o] = c.phi_in[o] + dt * R;
    else
      c.phi_out[o] = half_t(c.phi_n[o] + fma_t(dt, R, c.phi_in[o]));
  }
}

// Every edge EMF of every block into c.emf (grids with refinement levels).
__global__ void __launch_bounds__(256) ct_emf_kernel(StageArgs a, CtArgs c) {
  const unsigned n = (unsigned)a.nblocks * (unsigned)c.g.nEb;
  for (unsigned t = blockIdx.x * blockDim.x + threadIdx.x; t < n; t += gridDim.x * blockDim.x) {
    const int b = (int)(t / (unsigned)c.g.nEb);
    const int r = (int)(t - (unsigned)b * (unsigned)c.g.nEb);
    const int e = r >= c.g.eoff[2] ? 2 : (r >= c.g.eoff[1] ? 1 : 0);
    const int q = r - (int)c.g.eoff[e];
    const int i = q % c.g.ee[e][0], j = (q / c.g.ee[e][0]) % c.g.ee[e][1], k = q / (c.g.ee[e][0] * c.g.ee[e][1]);
    c.emf[t] = 0.25 * (e == 0 ? emf1x4(c, b, i, j, k) : (e == 1 ? emf2x4(c, b, i, j, k) : emf3x4(c, b, i, j, k)));
  }
}

// Edges that a finer leaf touches: the mean of the finer EMFs along them (the
// finer entries are never corrected themselves, so the order does not matter).
__global__ void __launch_bounds__(256) ct_emf_fix_kernel(CtArgs c) {
  for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < c.nef;
       t += (long long)gridDim.x * blockDim.x) {
    const long long s1 = c.ef_src[2 * t + 1];
    const double e0 = c.emf[c.ef_src[2 * t]];
    c.emf[c.ef_dst[t]] = s1 >= 0 ? (e0 + c.emf[s1]) / 2.0 : e0;
  }
}

__device__ __forceinline__ double emf_at(const CtArgs& c, int b, int e, int i, int j, int k) {
  return c.emf[(long long)b * c.g.nEb + c.g.eoff[e] + ((long long)k * c.g.ee[e][1] + j) * c.g.ee[e][0] + i];
}

// d_t Phi = -curl E from the stored (corrected) EMFs with the block's level
// spacing, and the stage combination, one thread per owned face.
template <int DIM>
__global__ void __launch_bounds__(256) ct_face_level_kernel(StageArgs a, CtArgs c) {
  const double dt = block_dt(a);
  const unsigned n = (unsigned)a.nblocks * (unsigned)c.g.nown_b;
  for (unsigned t = blockIdx.x * blockDim.x + threadIdx.x; t < n; t += gridDim.x * blockDim.x) {
    const int b = (int)(t / (unsigned)c.g.nown_b);
    int d, i, j, k;
    owned_face(c.g, (int)(t - (unsigned)b * (unsigned)c.g.nown_b), d, i, j, k);
    const long long o = (long long)b * c.g.nfb + ring_index(c.g, d, i, j, k);
    const int L = a.blk[4 * b];
    const int G2 = a.blk[4 * b + 2] * a.ny + j;
    if (!a.flat && d == 1 && ((G2 == 0 && c.axis_lo) || (G2 == a.N2l[L] && c.axis_hi))) {
      c.phi_out[o] = 0.0;  // sqrt(gamma) = 0 on the axis
      continue;
    }
    const double ix = a.idxl[L][0], iy = a.idxl[L][1], iz = a.idxl[L][2];
    double R;
    if (d == 0) {
      R = -(emf_at(c, b, 2, i, j + 1, k) - emf_at(c, b, 2, i, j, k)) * iy;
      if (DIM == 3) R += (emf_at(c, b, 1, i, j, k + 1) - emf_at(c, b, 1, i, j, k)) * iz;
    } else if (d == 1) {
      R = (emf_at(c, b, 2, i + 1, j, k) - emf_at(c, b, 2, i, j, k)) * ix;
      if (DIM == 3) R -= (emf_at(c, b, 0, i, j, k + 1) - emf_at(c, b, 0, i, j, k)) * iz;
    } else {
      R = -(emf_at(c, b, 1, i + 1, j, k) - emf_at(c, b, 1, i, j, k)) * ix +
          (emf_at(c, b, 0, i, j + 1, k) - emf_at(c, b, 0, i, j, k)) * iy;
    }
    if (a.stage == 1)
      c.phi_out[o] = c.phi_in[o] + dt * R;
    else
      c.phi_out[o] = half_t(c.phi_n[o] + fma_t(dt, R, c.phi_in[o]));
  }
}

// Flux divergence, sources, RK combination, the cell field from the updated
// faces, then the stage kernel's inversion, floors, outputs and CFL rate.  T:
// the arithmetic of the sources (float in the mixed form, from the FP32
// primitives and metric records).  Two CTAs per SM as the register bound (a
// few spilled values; the mixed form's stage 2.5% faster than at one CTA).
// NKM: the inversion's solver (0 analytic Newton, 1 Newton-Krylov), compiled in:
// both in one kernel cost spilled registers.
template <typename T, int DIM, bool FLAT, int NKM>
__global__ void __launch_bounds__(256, 2) ct_cell_kernel(StageArgs a, CtArgs c) {
  const double dt = block_dt(a);
  if (a.stage == 1 && blockIdx.x == 0 && threadIdx.x == 0) *a.dt_dev = dt;
  unsigned cnt[4] = {0u, 0u, 0u, 0u};
  double rate_max = 0.0;
  const unsigned n = (unsigned)a.nblocks * (unsigned)a.nint;
  for (unsigned t = blockIdx.x * blockDim.x + threadIdx.x; t < n; t += gridDim.x * blockDim.x) {
    const int b = (int)(t / (unsigned)a.nint);
    const LevelGeo geo = level_geo(a, a.blk[4 * b]);
    const int ci = (int)(t - (unsigned)b * (unsigned)a.nint);
    const int i = ci % a.nx, j = (ci / a.nx) % a.ny, k = ci / (a.nx * a.ny);
    const int cg = ((k + a.gz) * a.Ny + (j + a.gy)) * a.Nx + (i + a.gx);
    const int I1 = a.blk[4 * b + 1] * a.nx + i, I2 = a.blk[4 * b + 2] * a.ny + j;
    double rhs[NV];
#pragma unroll
    for (int v = 0; v < NV; ++v) rhs[v] = 0.0;
#pragma unroll
    for (int d = 0; d < DIM; ++d) {
      const int ih = i + (d == 0), jh = j + (d == 1), kh = k + (d == 2);
#pragma unroll
      for (int v = 0; v < NV; ++v) rhs[v] += -(xf_at(c, b, d, v, ih, jh, kh) - xf_at(c, b, d, v, i, j, k)) * geo.idx[d];
    }
    if (!FLAT) {
      const T* crec = (sizeof(T) == 8 ? reinterpret_cast<const T*>(geo.tc) : reinterpret_cast<const T*>(geo.tc32)) +
                      (size_t)(I2 * geo.N1 + I1) * CREC;
      const T* Pin = sizeof(T) == 8 ? reinterpret_cast<const T*>(a.P_in) : reinterpret_cast<const T*>(a.P32_in);
      T Pc[NV], S[NV];
#pragma unroll
      for (int v = 0; v < NV; ++v) Pc[v] = Pin[(size_t)b * NV * a.ncell + (size_t)v * a.ncell + cg];
      const Met<T> m = load_centre_metric<T>(crec);
      const T sg = crec[C_SG];
      if constexpr (sizeof(T) == 8) {
        sources_direct(m, crec, Pc, a.gam_fac, T(0.0), T(0.0), S);
        rhs[CS1] = fma_t(sg, S[0], rhs[CS1]);
        rhs[CS2] = fma_t(sg, S[1], rhs[CS2]);
        rhs[CTAU] = fma_t(sg, S[2], rhs[CTAU]);
      } else {
        T Uc[NV];
        Derived<T> s;
        derive(m, Pc, a.gam_fac_f, s);
        cons_of(Pc, s, Uc);
        sources_of(m, crec, Pc, s, Uc, T(0.0), T(0.0), S);
        // (D, S_3 and B have no source)
        rhs[CS1] += to_double(sg * S[CS1]);
        rhs[CS2] += to_double(sg * S[CS2]);
        rhs[CTAU] += to_double(sg * S[CTAU]);
      }
    }
    const size_t ub = (size_t)b * NV * a.nint + ci;
    double U[NV];
#pragma unroll
    for (int v = 0; v < NV; ++v) {
      const double un = a.Un[ub + (size_t)v * a.nint];
      U[v] = a.stage == 1 ? fma_t(dt, rhs[v], un) : half_t(un + fma_t(dt, rhs[v], a.U1[ub + (size_t)v * a.nint]));
    }
#pragma unroll
    for (int d = 0; d < DIM; ++d) {
      const long long lo = (long long)b * c.g.nfb + ring_index(c.g, d, i, j, k);
      const long long hi = (long long)b * c.g.nfb + ring_index(c.g, d, i + (d == 0), j + (d == 1), k + (d == 2));
      U[B1 + d] = half_t(c.phi_out[lo] + c.phi_out[hi]);
    }
    U[PSI] = 0.0;
    finish_cell<T, DIM, FLAT, (sizeof(T) == 4), NKM, true>(a, geo, b, ci, cg, I1, I2, U, cnt, rate_max);
  }
  reduce_outputs(a, cnt, rate_max);
}

// After a face load, in one pass over the interior cells (three passes, one of
// them for the rate, took 565 us on 1.8 M cells): the cell field of the
// loaded primitives from its faces (psi = 0), the conserved state, and the CFL
// rate of the state reduced into smax_out.
template <int DIM, bool FLAT>
__global__ void __launch_bounds__(256) ct_load_kernel(StageArgs a, CtArgs c, double* P, float* P32, double* U) {
  double rate_max = 0.0;
  const unsigned n = (unsigned)a.nblocks * (unsigned)a.nint;
  for (unsigned t = blockIdx.x * blockDim.x + threadIdx.x; t < n; t += gridDim.x * blockDim.x) {
    const int b = (int)(t / (unsigned)a.nint);
    const int ci = (int)(t - (unsigned)b * (unsigned)a.nint);
    const int i = ci % a.nx, j = (ci / a.nx) % a.ny, k = ci / (a.nx * a.ny);
    const int cg = ((k + a.gz) * a.Ny + (j + a.gy)) * a.Nx + (i + a.gx);
    const LevelGeo geo = level_geo(a, a.blk[4 * b]);
    const unsigned long long seen = cfl_seen(a);
    Met<double> m = flat_metric<double>();
    const double* rec = nullptr;
    const float* rec32 = nullptr;
    double sg = 1.0, isg = 1.0;
    if (!FLAT) {
      const int I1 = a.blk[4 * b + 1] * a.nx + i, I2 = a.blk[4 * b + 2] * a.ny + j;
      rec = geo.tc + (size_t)(I2 * geo.N1 + I1) * CREC;
      rec32 = geo.tc32 + (size_t)(I2 * geo.N1 + I1) * CREC;
      m = load_centre_metric<double>(rec);
      sg = rec[C_SG];
      isg = rec[C_ISG];
    }
    double* Pb = P + (size_t)b * NV * a.ncell + cg;
    double Pc[NV], Uc[NV];
#pragma unroll
    for (int v = 0; v < NV; ++v) Pc[v] = Pb[(size_t)v * a.ncell];
#pragma unroll
    for (int d = 0; d < DIM; ++d) {
      const long long lo = (long long)b * c.g.nfb + ring_index(c.g, d, i, j, k);
      const long long hi = (long long)b * c.g.nfb + ring_index(c.g, d, i + (d == 0), j + (d == 1), k + (d == 2));
      // the quotient by sqrt(gamma): the product with its reciprocal and one correction
      const double x = half_t(c.phi_in[lo] + c.phi_in[hi]), q = x * isg;
      Pc[B1 + d] = fma(fma(-q, sg, x), isg, q);
    }
    Pc[PSI] = 0.0;
    cons_direct(m, Pc, a.gam_fac, Uc);
#pragma unroll
    for (int v = 0; v < NV; ++v) {
      U[((size_t)b * NV + v) * a.nint + ci] = FLAT ? Uc[v] : sg * Uc[v];
      if ((v >= B1 && v < B1 + DIM) || v == PSI) {
        Pb[(size_t)v * a.ncell] = Pc[v];
        if (P32) P32[(size_t)b * NV * a.ncell + cg + (size_t)v * a.ncell] = narrow_f64(Pc[v]);
      }
    }
    cfl_max<DIM, FLAT, true>(a, geo, m, rec, rec32, Pc, seen, rate_max);
  }
  const double w = warp_max_d(rate_max);
  if ((threadIdx.x & 31u) == 0) atomicMax(a.smax_out, (unsigned long long)__double_as_longlong(w));
}

__global__ void __launch_bounds__(256) ct_copy_kernel(int nblocks, CtGeom g, const double* __restrict__ src, double* dst,
                                                      int to_ring) {
  const unsigned n = (unsigned)nblocks * (unsigned)g.nown_b;  // below the ring-extended count, which fits 31 bits
  for (unsigned t = blockIdx.x * blockDim.x + threadIdx.x; t < n; t += gridDim.x * blockDim.x) {
    const int b = (int)(t / (unsigned)g.nown_b);
    int d, i, j, k;
    owned_face(g, (int)(t - (unsigned)b * (unsigned)g.nown_b), d, i, j, k);
    const long long o = (long long)b * g.nfb + ring_index(g, d, i, j, k);
    if (to_ring)
      dst[o] = src[t];
    else
      dst[t] = src[o];
  }
}

int grid_of(long long n) {
  int dev = 0, nsm = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
  long long g = (n + 255) / 256;
  const long long cap = 32LL * nsm;
  if (g > cap) g = cap;
  return g < 1 ? 1 : (int)g;
}

}  // namespace

CtLevelMaps ct_level_maps(const bhac_grid_desc* d, const bhac_block_desc* blocks, int nb, const CtGeom& g) {
  CtLevelMaps M;
  M.ok = false;
  LevelCtx X;
  X.d = d;
  X.g = &g;
  X.leaves.build(d, blocks, nb);
  const int* nx = d->nx;
  // ring faces: the boundary rules across (at the block's level), then the
  // sources; blocks in contiguous ranges on host threads, joined in order
  struct RingOut {
    std::vector<long long> copy_dst, copy_src, mean_dst, mean_src;
    bool ok = true;
  };
  auto ring_block = [&](int b, RingOut& R) {
    const int L = blocks[b].level;
    const long long bo[3] = {blocks[b].ix, blocks[b].iy, blocks[b].iz};
    long long N[3];
    for (int e = 0; e < 3; ++e) N[e] = X.ncell(e, L);
    for (int dd = 0; dd < d->ndim; ++dd)
      for (int k = -g.fo[dd][2]; k < g.fe[dd][2] - g.fo[dd][2]; ++k)
        for (int j = -g.fo[dd][1]; j < g.fe[dd][1] - g.fo[dd][1]; ++j)
          for (int i = -g.fo[dd][0]; i < g.fe[dd][0] - g.fo[dd][0]; ++i) {
            const int f[3] = {i, j, k};
            bool ring = false;
            for (int e = 0; e < 3; ++e)
              if (e != dd && (f[e] < 0 || f[e] >= nx[e])) ring = true;
            if (!ring) continue;
            long long G[3];
            for (int e = 0; e < 3; ++e) G[e] = bo[e] * nx[e] + f[e];
            for (int e = 0; e < d->ndim; ++e) {
              if (e == dd) continue;
              const int side = G[e] < 0 ? 0 : (G[e] >= N[e] ? 1 : -1);
              if (side < 0) continue;
              const int kind = d->bc[e][side];
              if (kind == BHAC_BC_PERIODIC) {
                G[e] = ((G[e] % N[e]) + N[e]) % N[e];
              } else if (kind == BHAC_BC_OUTFLOW || kind == BHAC_BC_NOINFLOW) {
                G[e] = side == 0 ? 0 : N[e] - 1;
              } else {  // polar axis (x2): mirror, and phi + pi in 3-D
                G[e] = side == 0 ? -1 - G[e] : 2 * N[e] - 1 - G[e];
                if (d->ndim == 3) G[2] = ((G[2] + N[2] / 2) % N[2] + N[2]) % N[2];
              }
            }
            if (d->ndim == 3 && dd != 2 && d->bc[2][0] == BHAC_BC_PERIODIC) G[2] = ((G[2] % N[2]) + N[2]) % N[2];
            for (int e = 0; e < 3; ++e)
              if (G[e] < 0 || G[e] > N[e] || (e != dd && G[e] == N[e])) {
                R.ok = false;
                return;
              }
            long long src[4];
            const int n = X.face_sources(dd, L, G, src);
            if (n == 0) {
              R.ok = false;
              return;
            }
            const long long dst = (long long)b * g.nfb + ring_index(g, dd, i, j, k);
            if (n == 1) {
              R.copy_dst.push_back(dst);
              R.copy_src.push_back(src[0]);
            } else {
              R.mean_dst.push_back(dst);
              for (int q = 0; q < 4; ++q) R.mean_src.push_back(q < n ? src[q] : -1);
            }
          }
  };
  {
    const int nt = std::max(1, std::min(16, std::min(nb / 64, (int)std::thread::hardware_concurrency())));
    std::vector<RingOut> part(nt);
    std::vector<std::thread> pool;
    for (int t = 0; t < nt; ++t)
      pool.emplace_back([&, t] {
        for (int b = (int)((long long)nb * t / nt); b < (int)((long long)nb * (t + 1) / nt) && part[t].ok; ++b)
          ring_block(b, part[t]);
      });
    for (auto& th : pool) th.join();
    for (const RingOut& R : part) {
      if (!R.ok) return M;
      M.copy_dst.insert(M.copy_dst.end(), R.copy_dst.begin(), R.copy_dst.end());
      M.copy_src.insert(M.copy_src.end(), R.copy_src.begin(), R.copy_src.end());
      M.mean_dst.insert(M.mean_dst.end(), R.mean_dst.begin(), R.mean_dst.end());
      M.mean_src.insert(M.mean_src.end(), R.mean_src.begin(), R.mean_src.end());
    }
  }
  // coarse fluxes on level boundaries: the mean of the finer ones (the finer
  // faces in the order: first transverse direction (d + 1) % 3 outer, (d + 2) % 3 inner)
  auto xf_index = [&](int b, int dd, int i, int j, int k) {
    return (long long)b * NV * g.nfb + NV * g.foff[dd] + (ring_index(g, dd, i, j, k) - g.foff[dd]);
  };
  for (int b = 0; b < nb; ++b) {
    const int L = blocks[b].level;
    const long long bo[3] = {blocks[b].ix, blocks[b].iy, blocks[b].iz};
    for (int dd = 0; dd < d->ndim; ++dd)
      for (int side = 0; side < 2; ++side) {
        long long nbc[3] = {bo[0], bo[1], bo[2]};
        nbc[dd] += side == 0 ? -1 : 1;
        const long long nbd = (long long)d->nroot[dd] << L;
        if (nbc[dd] < 0 || nbc[dd] >= nbd) {
          if (d->bc[dd][side] != BHAC_BC_PERIODIC) continue;
          nbc[dd] = (nbc[dd] + nbd) % nbd;
        }
        if (X.leaves.get(d, L, nbc) >= 0) continue;
        long long chb[3];
        for (int e = 0; e < 3; ++e) chb[e] = e < d->ndim ? 2 * nbc[e] : nbc[e];
        if (side == 0) chb[dd] += 1;
        if (X.leaves.get(d, L + 1, chb) < 0) continue;
        const int t1 = (dd + 1) % 3, t2 = (dd + 2) % 3;
        const int fcoarse = side == 0 ? 0 : nx[dd], ffine = side == 0 ? nx[dd] : 0;
        for (int a = 0; a < nx[t1]; ++a)
          for (int bb = 0; bb < nx[t2]; ++bb) {
            long long src[4] = {-1, -1, -1, -1};
            int cnt = 0;
            for (int s1 = 0; s1 < (t1 < d->ndim ? 2 : 1); ++s1)
              for (int s2 = 0; s2 < (t2 < d->ndim ? 2 : 1); ++s2) {
                const long long gc1 = bo[t1] * nx[t1] + a, gc2 = bo[t2] * nx[t2] + bb;
                const long long Gf1 = t1 < d->ndim ? 2 * gc1 + s1 : gc1, Gf2 = t2 < d->ndim ? 2 * gc2 + s2 : gc2;
                long long fb[3];
                fb[dd] = chb[dd];
                fb[t1] = Gf1 / nx[t1];
                fb[t2] = Gf2 / nx[t2];
                const int bf = X.leaves.get(d, L + 1, fb);
                if (bf < 0) continue;
                int li[3];
                li[dd] = ffine;
                li[t1] = (int)(Gf1 % nx[t1]);
                li[t2] = (int)(Gf2 % nx[t2]);
                src[cnt++] = xf_index(bf, dd, li[0], li[1], li[2]);
              }
            if (cnt == 0) continue;
            int lc[3];
            lc[dd] = fcoarse;
            lc[t1] = a;
            lc[t2] = bb;
            M.xr_dst.push_back(xf_index(b, dd, lc[0], lc[1], lc[2]));
            for (int q = 0; q < 4; ++q) M.xr_src.push_back(src[q]);
            M.xr_d.push_back(dd);
          }
      }
  }
  // EMFs of edges that a finer leaf touches: the mean of the finer EMFs along them
  for (int b = 0; b < nb; ++b) {
    const int L = blocks[b].level;
    const long long bo[3] = {blocks[b].ix, blocks[b].iy, blocks[b].iz};
    for (int a = 0; a < 3; ++a) {
      if (!(d->ndim == 3 || a == 2)) continue;
      const int* ee = g.ee[a];
      for (int k = 0; k < ee[2]; ++k)
        for (int j = 0; j < ee[1]; ++j)
          for (int i = 0; i < ee[0]; ++i) {
            const int loc[3] = {i, j, k};
            bool inner = true;  // all four cells around the edge are the block's own
            for (int e = 0; e < d->ndim; ++e)
              if (e != a && (loc[e] == 0 || loc[e] == nx[e])) inner = false;
            if (inner) continue;
            long long G[3], C[3];
            int sgn[3];
            for (int e = 0; e < 3; ++e) G[e] = bo[e] * nx[e] + loc[e];
            bool finer = false;
            for (int q = 0; q < 4 && !finer; ++q)
              if (X.edge_cell(a, L, G, q, C, sgn) && X.cover(L, C) > 0) finer = true;
            if (!finer || L + 1 >= d->nlevels) continue;
            const int na = a < d->ndim ? 2 : 1;
            long long src[2] = {-1, -1};
            int n = 0;
            for (int t = 0; t < na; ++t) {
              long long F[3];
              for (int e = 0; e < 3; ++e) F[e] = e >= d->ndim ? G[e] : 2 * G[e] + (e == a ? t : 0);
              for (int q = 0; q < 4; ++q) {
                if (!X.edge_cell(a, L + 1, F, q, C, sgn)) continue;
                long long bc[3];
                for (int e = 0; e < 3; ++e) bc[e] = C[e] / nx[e];
                const int bf = X.leaves.get(d, L + 1, bc);
                if (bf < 0) continue;
                int lf[3];
                for (int e = 0; e < 3; ++e)
                  lf[e] = (int)(C[e] - bc[e] * nx[e]) + (e != a && e < d->ndim && !sgn[e] ? 1 : 0);
                src[n++] = (long long)bf * g.nEb + g.eoff[a] + ((long long)lf[2] * g.ee[a][1] + lf[1]) * g.ee[a][0] + lf[0];
                break;
              }
            }
            if (n != na) continue;
            M.ef_dst.push_back((long long)b * g.nEb + g.eoff[a] + ((long long)k * ee[1] + j) * ee[0] + i);
            M.ef_src.push_back(src[0]);
            M.ef_src.push_back(src[1]);
          }
    }
  }
  M.ok = true;
  return M;
}

}  // namespace bhac

// Host self-check of the constrained-transport ring maps (test utility).
extern "C" bhac_status bhac_ct_ring_faces_host(const bhac_grid_desc* d, const bhac_block_desc* b, int nb,
                                               const double* owned, double* ring) {
  using namespace bhac;
  if (!d || !b || !owned || !ring || nb <= 0 || d->divb != BHAC_DIVB_CT || d->ndim < 2 || d->ndim > 3 ||
      d->nlevels < 1 || d->nlevels > MAXLEV)
    return BHAC_ERR_ARG;
  const CtGeom g = ct_geom(d);
  std::vector<long long> cd, cs, md, ms;
  if (d->nlevels == 1) {
    if (!ct_ring_map(d, b, nb, g, cd, cs)) return BHAC_ERR_ARG;
  } else {
    CtLevelMaps M = ct_level_maps(d, b, nb, g);
    if (!M.ok) return BHAC_ERR_ARG;
    cd.swap(M.copy_dst);
    cs.swap(M.copy_src);
    md.swap(M.mean_dst);
    ms.swap(M.mean_src);
  }
  for (long long t = 0; t < (long long)nb * g.nfb; ++t) ring[t] = 0.0;
  for (int q = 0; q < nb; ++q)
    for (long long r = 0; r < g.nown_b; ++r) {
      int dd, i, j, k;
      owned_face(g, (int)r, dd, i, j, k);
      ring[(long long)q * g.nfb + ring_index(g, dd, i, j, k)] = owned[(long long)q * g.nown_b + r];
    }
  for (size_t t = 0; t < cd.size(); ++t) ring[cd[t]] = ring[cs[t]];
  for (size_t t = 0; t < md.size(); ++t) {
    double s = 0.0;
    int m = 0;
    for (int q = 0; q < 4; ++q)
      if (ms[4 * t + q] >= 0) {
        s += ring[ms[4 * t + q]];
        ++m;
      }
    ring[md[t]] = s / m;
  }
  return BHAC_OK;
}

namespace bhac {

cudaError_t launch_ct_ring(const long long* dst, const long long* src, long long n, double* phi, cudaStream_t st) {
  if (n <= 0) return cudaSuccess;
  ct_ring_kernel<<<grid_of(n), 256, 0, st>>>(dst, src, n, phi);
  return cudaGetLastError();
}

cudaError_t launch_ct_ring_mean(const long long* dst, const long long* src, long long n, double* phi,
                                cudaStream_t st) {
  if (n <= 0) return cudaSuccess;
  ct_ring_mean_kernel<<<grid_of(n), 256, 0, st>>>(dst, src, n, phi);
  return cudaGetLastError();
}

// Segments of at most kCtLine faces, and as many lines per CTA as its threads
// have faces for: at most 320 cells (segments of four faces) and 46080 bytes of
// edges, which needs no opt-in shared memory.
static CtLines ct_line_plan(const StageArgs& a, const CtGeom& g) {
  CtLines w;
  w.g0[0] = 0;
  for (int d = 0; d < 3; ++d) {
    w.nu[d] = w.nf[d] = w.ns[d] = 1;
    w.units[d] = 0;
    unsigned groups = 0;
    if (d < g.ndim) {
      const int nd = g.fe[d][d];
      w.ns[d] = (nd + kCtLine - 1) / kCtLine;
      w.nf[d] = (nd + w.ns[d] - 1) / w.ns[d];
      w.nu[d] = kCtThreads / w.nf[d];
      w.units[d] = (unsigned)a.nblocks * (unsigned)(g.nfd[d] / nd) * (unsigned)w.ns[d];
      groups = (w.units[d] + w.nu[d] - 1) / w.nu[d];
    }
    w.g0[d + 1] = w.g0[d] + groups;
  }
  return w;
}

template <typename T, bool FLAT>
static cudaError_t launch_ct_flux(const StageArgs& a, const CtArgs& c, const CtLines& w, cudaStream_t st) {
  size_t smem = 0;
  for (int d = 0; d < c.g.ndim; ++d) {
    const size_t n = 2 * NV * sizeof(T) * (size_t)w.nu[d] * (w.nf[d] + 1);
    smem = n > smem ? n : smem;
  }
  ct_flux_kernel<T, FLAT><<<w.g0[3], kCtThreads, smem, st>>>(a, c, w);
  return cudaGetLastError();
}

template <typename T, int DIM, bool FLAT>
static void launch_ct_cell(const StageArgs& a, const CtArgs& c, int grid, cudaStream_t st) {
  if (a.c2p_nk)
    ct_cell_kernel<T, DIM, FLAT, 1><<<grid, 256, 0, st>>>(a, c);
  else
    ct_cell_kernel<T, DIM, FLAT, 0><<<grid, 256, 0, st>>>(a, c);
}

template <typename T>
static cudaError_t launch_ct_cells(const StageArgs& a, const CtArgs& c, int grid, cudaStream_t st) {
  if (a.ndim == 3)
    a.flat ? launch_ct_cell<T, 3, true>(a, c, grid, st) : launch_ct_cell<T, 3, false>(a, c, grid, st);
  else
    a.flat ? launch_ct_cell<T, 2, true>(a, c, grid, st) : launch_ct_cell<T, 2, false>(a, c, grid, st);
  return cudaGetLastError();
}

cudaError_t launch_ct_stage(const StageArgs& a, const CtArgs& c, bool mixed, cudaStream_t st) {
  const long long no = (long long)a.nblocks * c.g.nown_b,
                  nc = (long long)a.nblocks * a.nint;
  const CtLines w = ct_line_plan(a, c.g);
  cudaError_t e = mixed ? (a.flat ? launch_ct_flux<float, true>(a, c, w, st) : launch_ct_flux<float, false>(a, c, w, st))
                        : (a.flat ? launch_ct_flux<double, true>(a, c, w, st) : launch_ct_flux<double, false>(a, c, w, st));
  if (e != cudaSuccess) return e;
  if (c.amr) {
    // refinement levels: coarse fluxes corrected, every EMF stored and the
    // touched coarse ones corrected, then the face update from them
    if (c.nxr > 0) ct_reflux_kernel<<<grid_of(c.nxr), 256, 0, st>>>(c);
    ct_emf_kernel<<<grid_of((long long)a.nblocks * c.g.nEb), 256, 0, st>>>(a, c);
    if (c.nef > 0) ct_emf_fix_kernel<<<grid_of(c.nef), 256, 0, st>>>(c);
    if (a.ndim == 3)
      ct_face_level_kernel<3><<<grid_of(no), 256, 0, st>>>(a, c);
    else
      ct_face_level_kernel<2><<<grid_of(no), 256, 0, st>>>(a, c);
  } else if (a.ndim == 3) {
    ct_face_kernel<3><<<grid_of(no), 256, 0, st>>>(a, c);
  } else {
    ct_face_kernel<2><<<grid_of(no), 256, 0, st>>>(a, c);
  }
  e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  return mixed ? launch_ct_cells<float>(a, c, grid_of(nc), st) : launch_ct_cells<double>(a, c, grid_of(nc), st);
}

cudaError_t launch_ct_load(const StageArgs& a, const CtArgs& c, double* P, float* P32, double* U, cudaStream_t st) {
  int grid = grid_of((long long)a.nblocks * a.nint) / 4;  // about eight CTAs per SM: few atomics on the one rate word
  if (grid < 1) grid = 1;
  if (a.ndim == 3)
    a.flat ? ct_load_kernel<3, true><<<grid, 256, 0, st>>>(a, c, P, P32, U)
           : ct_load_kernel<3, false><<<grid, 256, 0, st>>>(a, c, P, P32, U);
  else
    a.flat ? ct_load_kernel<2, true><<<grid, 256, 0, st>>>(a, c, P, P32, U)
           : ct_load_kernel<2, false><<<grid, 256, 0, st>>>(a, c, P, P32, U);
  return cudaGetLastError();
}

cudaError_t launch_ct_copy_faces(const StageArgs& a, const CtGeom& g, const double* src, double* dst, int to_ring,
                                 cudaStream_t st) {
  ct_copy_kernel<<<grid_of((long long)a.nblocks * g.nown_b), 256, 0, st>>>(a.nblocks, g, src, dst, to_ring);
  return cudaGetLastError();
}

}  // namespace bhac

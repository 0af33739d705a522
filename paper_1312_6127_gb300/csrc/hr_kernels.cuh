// Kernels of one RK3 sub-step (Sec. 4.2 of McKinney et al. 2014) for sm_103a.
//
// Data layout in HBM: structure of arrays, one FP64 plane per primitive,
// [12][N3][N2][N1] with 4 ghost zones on each side of every active direction
// (i fastest, so a warp reads 32 consecutive x1 zones of one variable).
// Face fluxes of direction d share the cell indexing: the flux stored at cell
// t is the flux through t's lower d-face.
//
// A context holds one or more grids (the boxes of a batch).  Every array is
// the concatenation of per-grid blocks, each laid out as above; BoxGeo gives a
// grid's sizes and its offsets.  Every kernel loops over the grids and, inside
// a grid, over its index space with a grid-stride loop, so one launch advances
// all grids of a batch.  Grids are sized by the host in multiples of the SM
// count.
#pragma once
#include "hr_common.cuh"
#include "hr_implicit.cuh"

namespace hr {

struct Bufs {
  double* P;       // [12][ntot] primitives, ghosts included (per grid)
  double* K;       // [ntot] per-zone absorption opacity (opacity field mode), ghosts included
  double* Un;      // [12][nact] conserved state at the start of the step
  double* Sn;      // RK3, null otherwise.  FP64: [2][nact] rho0 and u_g at the start of the
                   // step; split: [nact] the conserved entropy there
  void* F[3];      // [12][ntot] face fluxes (real type of the precision mode)
  void* FS[3];     // RK3, null otherwise: [ntot] FP64: left state's share of the mass flux;
                   // split: the entropy face flux
  double* ES[3];   // FP64: [4][ntot] edges of rho0 and u_g of each direction (EdgeSet)
  void* spd[3];    // [ntot] per-face max signal speed
  void* aux;       // [10][ntot] per-cell gdet, sqrt(-g) u^d gas/rad, tau weights
  void* flat[3];   // [2][ntot] flattener, max over the sub-steps of the step
  void* emf;       // [3][ntot] edge EMFs of the pairs of directions
  double* dt;      // [nbox] time step of each grid
  unsigned char* status;  // [nact] worst outcome over the sub-steps
  int* iters;             // [nact] Newton steps summed over the sub-steps
  unsigned char* failed;  // [nact] back-up flag of the current sub-step
  int* qcount;            // [4] lengths: retry queue, back-up list, Newton continuation queue, its finite-difference end
  int* qzone;             // [nact] retry queue: zone index within its grid
  int* qbox;              // [nact] retry queue: grid of the entry
  double* qdata;          // [nact][19] retry queue payload: U*, PMHD best x, e_T, h, S*
  int* fzone;             // [nact] back-up list: zone index within its grid
  int* fbox;              // [nact] back-up list: grid of the entry
  double* ftmp;           // [nact][12] averaged primitives of back-up zones
  int* czone;             // [nact] Newton continuation queue: zone index within its grid
  int* cbox;              // [nact] Newton continuation queue: grid of the entry
  double* cdata;          // [nact][CSTRIDE] continuation payload: U*, Newton state
  int ncont;              // nact of the context: the queue's finite-difference zones fill it from the end
  unsigned long long* stats;  // [8] counters
  unsigned long long* dtmin;  // [nbox] CFL minimum (ordered bits of a positive double)
  const double* geo;          // metric tables of Kerr-Schild grids (null otherwise)
  // records of the sub-step for the adjoint's recomputation of a step and for
  // the IMEX sources (null otherwise); planes per grid, grid b at 12 aoff_b:
  double* ust_rec;            // [12][nact] U* of every zone of the sub-step
  unsigned char* meth_rec;    // [nact] outcome of every zone of the sub-step
  double* psol_rec;           // [12][nact] solution of every zone before the floors
  double* sst_rec;            // [nact] explicit entropy S* of the zones whose retry read it in the sub-step
  double* imexM;              // IMEX: [4 stages][4 gas rows][nact] per grid, grid b at 16 aoff_b
  double* Bf[3];              // staggered field: sqrt(-g) B^d on the d-faces [ntot] (null: flux-CT)
};


// FP64 edge values of one direction: [lower, upper][q - 2][ntot] of the primitives
// q >= 2 in E and [lower, upper][q][ntot] of rho0 and u_g in S, from which the
// entropy fluxes are formed where a zone needs them (entropy_flux).
struct EdgeSet {
  double* E;
  double* S;
  __device__ __forceinline__ EdgeSet box(const BoxGeo& b) const { return {E + 20 * b.coff, S + 4 * b.coff}; }
  // plane of primitive q's lower (up = 0) or upper (1) edges
  __device__ __forceinline__ double* plane(int up, int q, long long nt) const {
    return q < U1 ? S + (2 * up + q) * nt : E + (10 * up + q - U1) * nt;
  }
};

struct EdgeSets {
  EdgeSet d[3];
};

// Counter update aggregated over the converged lanes of a warp.
__device__ __forceinline__ void warp_add(unsigned long long* dst, unsigned v) {
  unsigned mask = __activemask();
  unsigned s = __reduce_add_sync(mask, v);
  if ((int)(threadIdx.x & 31) == __ffs(mask) - 1 && s) atomicAdd(dst, (unsigned long long)s);
}

#define HR_TID (blockIdx.x * (long long)blockDim.x + threadIdx.x)
#define HR_STRIDE ((long long)gridDim.x * blockDim.x)

// ------------------------------------------------------------ work split
// First item of this thread among the items of a grid whose predecessors in
// the context hold `done` items: the grids' items form one sequence dealt to
// the threads in turn, so that a batch of small grids loads every block alike.
// (The FP32 kernels of split precision pass over each grid from its first item:
// with another loop around them their sums are fused and rounded differently, and
// the FP32 stages answer round-off with up to 3e-7.)
__device__ __forceinline__ long long first_item(long long done) {
  if (done == 0) return HR_TID;
  const long long r = HR_TID - done % HR_STRIDE;
  return r < 0 ? r + HR_STRIDE : r;
}

// Opacity-field value of a cell (1 when the opacity is not a field).
__device__ __forceinline__ double kfield(const DevParams& p, const double* K, long long t) {
  return p.opacity == 2 ? K[t] : 1.0;
}

// ------------------------------------------------------------ metric tables
// The Kerr-Schild metric depends on (x1, x2) only.  A Kerr-Schild grid keeps,
// per (i, j), the metric at the cell centres, its x1 and x2 derivatives (for
// the geometric source) and the metric at the x1 and x2 faces, evaluated once
// when the context is created by the same functions the kernels would call.
// The FP64 kernels then read 16 doubles (L2-resident: a few MB per grid)
// instead of evaluating exp, sin, cos and four divisions per zone and face,
// which matters because the step is bound by FP64 arithmetic.
// Layout of a grid's table (offset BoxGeo::goff, in doubles): [GEO_C][N2][N1]
// centres, [16][N2][N1] centre derivatives, [GEO_F][N2][n1+1] x1 faces,
// [GEO_F][n2+1][N1] x2 faces, sqrt(-g) on the x1-x2 edges [n2+1][n1+1]; fields in the order of Geo (g00 g01 g03 g11 g13
// g22 g33 G00 G01 G11 G13 G22 G33 gdet alpha ialpha) and of MetricDeriv.
// Centres add 1/sqrt(-g) (plane 16), sqrt(g_dd) of the three directions
// (17..19), sqrt(gamma^{kk}) of the ZAMO slice (20..22), the density and
// internal-energy floors (23, 24) and the longest active proper edge of the
// cell (25); faces add 1/sqrt(-g) (16) and sqrt(g_dd) of their direction (17).
// Each saves divisions, square roots or exponentials per zone or face.  The
// derivatives are stored as the geometric source contracts them (split
// precision: plain): 1/2 sqrt(-g) d_nu g_{mu kappa}, off-diagonals doubled, and
// d_nu sqrt(-g).
constexpr int GEO_C = 26, GEO_F = 18;
struct GeoTab {
  const double* C;
  const double* M;
  const double* F0;
  const double* F1;
  const double* E;         // [n2+1][n1+1]
  long long sC, sF0, sF1;  // plane sizes
};

__host__ __device__ __forceinline__ long long geotab_size(const BoxGeo& b) {
  const long long sC = (long long)b.N[0] * b.N[1];
  return (GEO_C + 16) * sC + GEO_F * ((long long)(b.n[0] + 1) * b.N[1] + (long long)b.N[0] * (b.n[1] + 1)) +
         (long long)(b.n[0] + 1) * (b.n[1] + 1);
}

__device__ __forceinline__ GeoTab geotab(const double* base, const BoxGeo& b) {
  GeoTab t;
  t.sC = (long long)b.N[0] * b.N[1];
  t.sF0 = (long long)(b.n[0] + 1) * b.N[1];
  t.sF1 = (long long)b.N[0] * (b.n[1] + 1);
  t.C = base + b.goff;
  t.M = t.C + GEO_C * t.sC;
  t.F0 = t.M + 16 * t.sC;
  t.F1 = t.F0 + GEO_F * t.sF0;
  t.E = t.F1 + GEO_F * t.sF1;
  return t;
}

// entry of (i, j) (active indices, ghosts negative): centres, x1 faces
// (i = face index 0..n1), x2 faces (j = face index 0..n2)
__device__ __forceinline__ long long gidx_c(const BoxGeo& b, int i, int j) {
  return (long long)(j + b.ng[1]) * b.N[0] + (i + b.ng[0]);
}
__device__ __forceinline__ long long gidx_f0(const BoxGeo& b, int i, int j) {
  return (long long)(j + b.ng[1]) * (b.n[0] + 1) + i;
}
__device__ __forceinline__ long long gidx_f1(const BoxGeo& b, int i, int j) {
  return (long long)j * b.N[0] + (i + b.ng[0]);
}

template <int MET>
__device__ __forceinline__ Geo<MET, double> geo_load(const double* __restrict__ t, long long s, long long x) {
  Geo<MET, double> g;
  g.g00 = __ldg(t + x);
  g.g01 = __ldg(t + s + x);
  g.g03 = __ldg(t + 2 * s + x);
  g.g11 = __ldg(t + 3 * s + x);
  g.g13 = __ldg(t + 4 * s + x);
  g.g22 = __ldg(t + 5 * s + x);
  g.g33 = __ldg(t + 6 * s + x);
  g.G00 = __ldg(t + 7 * s + x);
  g.G01 = __ldg(t + 8 * s + x);
  g.G11 = __ldg(t + 9 * s + x);
  g.G13 = __ldg(t + 10 * s + x);
  g.G22 = __ldg(t + 11 * s + x);
  g.G33 = __ldg(t + 12 * s + x);
  g.gdet = __ldg(t + 13 * s + x);
  g.alpha = __ldg(t + 14 * s + x);
  g.ialpha = __ldg(t + 15 * s + x);
  return g;
}

template <int MET>
__device__ __forceinline__ void geo_store(double* t, long long s, long long x, const Geo<MET, double>& g) {
  const double v[16] = {g.g00, g.g01, g.g03, g.g11, g.g13, g.g22, g.g33, g.G00,
                        g.G01, g.G11, g.G13, g.G22, g.G33, g.gdet, g.alpha, g.ialpha};
  for (int f = 0; f < 16; ++f) t[f * s + x] = v[f];
}

// Metric of the centre of cell (i, j): from the table when the grid has one
// (FP64 kernels), else evaluated.
template <int MET, typename R>
__device__ __forceinline__ Geo<MET, R> geo_centre(const DevParams& p, const BoxGeo& bx, const double* geo0, int i,
                                                  int j) {
  if constexpr (MET == KS && std::is_same<R, double>::value) {
    if (geo0 && bx.goff >= 0) {
      const GeoTab T = geotab(geo0, bx);
      return geo_load<MET>(T.C, T.sC, gidx_c(bx, i, j));
    }
  }
  return make_geo<MET, R>(p, R(xcen(bx, 0, i)), R(xcen(bx, 1, j)));
}

// ----------------------------------------------------------- ghost fill
// One direction at a time, in the order 1, 2, 3, so that edges and corners
// come from already-filled cells.  Periodic wraps; outflow copies the last
// active zone and clamps the normal velocities (gas and radiation) so nothing
// enters from the ghost; polar mirrors across the axis from the zone half a
// turn away in phi, negating the theta components.  The opacity field, when
// present, is copied like a scalar primitive.
// NQ variables per thread, blockIdx.y the first of them.  The fill moves little:
// its time is the latency of a thread's chain, so one grid takes a thread per
// value (NQ = 1: 64x32x16 0.113 -> 0.063 ms per RK3 step), and a batch, whose
// threads pass over all its boxes, one per cell (12 boxes: 0.43 ms, 0.93 with
// NQ = 1).
template <int d, int NQ>
__global__ void k_bc_fill(DevParams p, const BoxGeo* __restrict__ boxes, int nbox, double* __restrict__ P0,
                          double* __restrict__ K0) {
  const int q0 = NQ == 1 ? blockIdx.y : 0;
  long long done = 0;
  for (int bi = 0; bi < nbox; ++bi) {
    const BoxGeo& bx = boxes[bi];
    double* P = P0 + 12 * bx.coff;
    double* K = K0 && q0 == 0 ? K0 + bx.coff : nullptr;
    // directions before d include their ghosts, those after it do not
    constexpr int e0 = d == 0 ? 1 : 0, e1 = d == 2 ? 1 : 2;
    const int g0 = e0 < d ? bx.ng[e0] : 0, g1 = e1 < d ? bx.ng[e1] : 0;
    const int l0 = bx.n[e0] + 2 * g0, l1 = bx.n[e1] + 2 * g1, ng = bx.ng[d];
    const long long total = 2LL * ng * l0 * l1;
    for (long long id = first_item(done); id < total; id += HR_STRIDE) {
      // x1 fastest: for d = 0 the ghost index, else e0 = x1
      unsigned r = (unsigned)id;
      int c[3], g, side;
      if (d == 0) {
        g = r % ng;
        r /= ng;
        c[e0] = r % l0;
        r /= l0;
        c[e1] = r % l1;
        side = r / l1;
      } else {
        c[e0] = r % l0;
        r /= l0;
        g = r % ng;
        r /= ng;
        c[e1] = r % l1;
        side = r / l1;
      }
      c[e0] -= g0;
      c[e1] -= g1;
      const int bc = bx.bc[2 * d + side];
      if (bc == 4) continue;  // fixed ghosts keep the values they were given
      int src[3];
      src[e0] = c[e0];
      src[e1] = c[e1];
      c[d] = side == 0 ? -1 - g : bx.n[d] + g;
      double sgn = 1.0;
      int clamp = 0;
      if (bc == 0) {
        src[d] = side == 0 ? bx.n[d] - 1 - g : g;
      } else if (bc == 1 || bc == 3) {
        src[d] = side == 0 ? 0 : bx.n[d] - 1;
        clamp = bc == 3 ? 0 : (side == 0 ? -1 : 1);
      } else {
        src[d] = side == 0 ? g : bx.n[d] - 1 - g;
        if (bx.n[2] > 1) src[2] = ((d == 2 ? g : c[2]) + bx.n[2] / 2) % bx.n[2];
        sgn = -1.0;
      }
      const long long s = cell_index(bx, src[0], src[1], src[2]);
      const long long t = cell_index(bx, c[0], c[1], c[2]);
#pragma unroll
      for (int e = 0; e < NQ; ++e) {
        const int q = q0 + e;
        const bool normal = q == U1 + d || q == UR1 + d;
        double v = P[q * bx.ntot + s];
        if (normal || q == B1 + d) v *= sgn;
        if (clamp != 0 && normal) {
          const double vc = clamp < 0 ? fmin(v, 0.0) : fmax(v, 0.0);
          if (p.sig) sig_put(p, bx.coff + t, 50 + d, (unsigned long long)q << 8 | (vc != v ? 1u : 0u));
          v = vc;
        }
        P[q * bx.ntot + t] = v;
      }
      if (K) K[t] = K[s];
    }
    done += total;
  }
}

// --------------------------------------------------------------- cell prep
// Per cell: sqrt(-g), and for every active direction d the flattener inputs
// sqrt(-g) u^d (gas, radiation) and the weight w_d = min(1, 2 tau_d) of the
// optical depth of the cell along d (Sec. 4.3).
template <int MET, typename R>
__global__ void k_prep(DevParams p, const BoxGeo* __restrict__ boxes, int nbox,
                       const double* __restrict__ P0, const double* __restrict__ K0,
                       R* __restrict__ aux0, const double* __restrict__ geo0) {
  for (int bi = 0; bi < nbox; ++bi) {
    const BoxGeo& bx = boxes[bi];
    const double* P = P0 + 12 * bx.coff;
    const double* K = K0 + bx.coff;
    R* aux = aux0 + 10 * bx.coff;
    for (long long t = HR_TID; t < bx.ntot; t += HR_STRIDE) {
      long long r = t;
      int i = (int)(r % bx.N[0]) - bx.ng[0];
      r /= bx.N[0];
      int j = (int)(r % bx.N[1]) - bx.ng[1];
      const Geo<MET, R> g = geo_centre<MET, R>(p, bx, geo0, i, j);
      R ucon[4], ucov[4], gm, urc[4], urv[4], gr;
      fourvel<MET, R>(g, R(P[U1 * bx.ntot + t]), R(P[U2 * bx.ntot + t]), R(P[U3 * bx.ntot + t]), ucon, ucov, &gm);
      fourvel<MET, R>(g, R(P[UR1 * bx.ntot + t]), R(P[UR2 * bx.ntot + t]), R(P[UR3 * bx.ntot + t]), urc, urv, &gr);
      R kabs, ksca;
      opacity<R>(p, R(P[RHO * bx.ntot + t]), R(P[UU * bx.ntot + t]), R(kfield(p, K, t)), &kabs, &ksca);
      aux[t] = g.gdet;
#pragma unroll
      for (int d = 1; d <= 3; ++d) {
        aux[(1 + 3 * (d - 1)) * bx.ntot + t] = g.gdet * ucon[d];
        aux[(2 + 3 * (d - 1)) * bx.ntot + t] = g.gdet * urc[d];
        R tau = (kabs + ksca) * sqrt(g.gdd(d)) * R(bx.dx[d - 1]);
        R w = R(2) * tau;
        aux[(3 + 3 * (d - 1)) * bx.ntot + t] = w < R(1) ? w : R(1);
      }
    }
  }
}

// The same in FP64: the metric factors it needs come from the table, the
// 4-velocities' time components from gamma^2 = 1 + u~^i g_ij u~^j, and only
// active directions are formed (none with MC, which has no flattener).
// Measured over an RK3 step: 256x128x64 torus 1.51 -> 1.02 ms.
template <int MET>
__global__ void k_prep64(DevParams p, const BoxGeo* __restrict__ boxes, int nbox, const double* __restrict__ P0,
                         const double* __restrict__ K0, double* __restrict__ aux0, const double* __restrict__ geo0) {
  for (int bi = 0; bi < nbox; ++bi) {
    const BoxGeo& bx = boxes[bi];
    const double* P = P0 + 12 * bx.coff;
    const double* K = K0 + bx.coff;
    double* aux = aux0 + 10 * bx.coff;
    const long long nt = bx.ntot;
    for (long long t = first_item(bx.coff); t < nt; t += HR_STRIDE) {
      Geo<MET, double> g;
      double gd = 1.0, a01 = 0.0, sd[3] = {1.0, 1.0, 1.0};
      if constexpr (MET == KS) {
        const GeoTab T = geotab(geo0, bx);
        const long long x = (unsigned)t % (unsigned)T.sC, s = T.sC;
        gd = __ldg(T.C + 13 * s + x);
        if (p.recon == 0) {
          g.g11 = __ldg(T.C + 3 * s + x);
          g.g13 = __ldg(T.C + 4 * s + x);
          g.g22 = __ldg(T.C + 5 * s + x);
          g.g33 = __ldg(T.C + 6 * s + x);
          a01 = __ldg(T.C + 14 * s + x) * __ldg(T.C + 8 * s + x);
          for (int e = 0; e < 3; ++e) sd[e] = __ldg(T.C + (17 + e) * s + x);
        }
      }
      aux[t] = gd;
      if (p.recon != 0) continue;
      double u[3], r[3], l[3];
#pragma unroll
      for (int e = 0; e < 3; ++e) {
        u[e] = P[(U1 + e) * nt + t];
        r[e] = P[(UR1 + e) * nt + t];
      }
      if constexpr (MET == KS) {
        if (p.act[0]) {  // u^1 = u~^1 - gamma alpha g^{t1}; u^2, u^3 are u~^2, u~^3
          lower3<MET>(g, u[0], u[1], u[2], l);
          u[0] = fma(-sqrt64(fma(u[0], l[0], fma(u[1], l[1], fma(u[2], l[2], 1.0)))), a01, u[0]);
          lower3<MET>(g, r[0], r[1], r[2], l);
          r[0] = fma(-sqrt64(fma(r[0], l[0], fma(r[1], l[1], fma(r[2], l[2], 1.0)))), a01, r[0]);
        }
      }
      const double rho = P[RHO * nt + t], ug = P[UU * nt + t];
      const double k2 = 2.0 * opacity_sum(p, rho, [&] { return p.gm1 * ug * rcp(rho); }, kfield(p, K, t));
#pragma unroll
      for (int e = 0; e < 3; ++e) {
        if (!p.act[e]) continue;
        aux[(1 + 3 * e) * nt + t] = gd * u[e];
        aux[(2 + 3 * e) * nt + t] = gd * r[e];
        const double w = k2 * sd[e] * bx.dx[e];
        aux[(3 + 3 * e) * nt + t] = w < 1.0 ? w : 1.0;
      }
    }
  }
}

// ----------------------------------------------------------- flattener
// Shock flattener of Sec. 4.3 (SP0 = 0.75): for GAS (gas pressure and
// sqrt(-g) u^d) and RAD (radiation pressure and sqrt(-g) u^d_rad), each
// pressure blended toward the total by the cell's w; flattening where
// |dp| > 0.33 min p and the flow compresses, with the shock parameter
// dp1/dp2 mapped by 10 (Sp - 0.75) to [0, 1]; the upstream neighbour's value
// is max-ed in; GAS and RAD are blended to their maximum by w; and the result
// is max-ed with the values of the earlier sub-steps of the step.
template <typename R>
struct FlatCell {
  R pg, pr, vg, vr, w;
};

template <typename R>
__device__ __forceinline__ R ftilde(const FlatCell<R>* c, int m, bool gas, R w) {
  R pe1 = gas ? c[m + 1].pg + w * c[m + 1].pr : c[m + 1].pr + w * c[m + 1].pg;
  R pem = gas ? c[m - 1].pg + w * c[m - 1].pr : c[m - 1].pr + w * c[m - 1].pg;
  R pe2 = gas ? c[m + 2].pg + w * c[m + 2].pr : c[m + 2].pr + w * c[m + 2].pg;
  R pe2m = gas ? c[m - 2].pg + w * c[m - 2].pr : c[m - 2].pr + w * c[m - 2].pg;
  R dp1 = pe1 - pem, dp2 = pe2 - pe2m;
  R dv = gas ? c[m + 1].vg - c[m - 1].vg : c[m + 1].vr - c[m - 1].vr;
  R mn = pe1 < pem ? pe1 : pem;
  if (fabs(dp1) > R(0.33) * mn && dv < R(0)) {
    R sp = dp2 != R(0) ? dp1 / dp2 : R(0);
    R f = R(10) * (sp - R(0.75));
    return f < R(0) ? R(0) : (f > R(1) ? R(1) : f);
  }
  return R(0);
}

// Flattener of the centre cell c[3] of a 7-cell stencil (GAS, RAD).
template <typename R>
__device__ __forceinline__ void flatten_cell(const FlatCell<R>* c, R* Fg, R* Fr) {
  const R w = c[3].w;
  R g0 = ftilde<R>(c, 3, true, w), r0 = ftilde<R>(c, 3, false, w);
  R pg1 = c[4].pg + w * c[4].pr, pgm = c[2].pg + w * c[2].pr;
  R pr1 = c[4].pr + w * c[4].pg, prm = c[2].pr + w * c[2].pg;
  int sg = (pg1 - pgm) < R(0) ? 1 : -1;
  int sr = (pr1 - prm) < R(0) ? 1 : -1;
  R gn = ftilde<R>(c, 3 + sg, true, c[3 + sg].w);
  R rn = ftilde<R>(c, 3 + sr, false, c[3 + sr].w);
  R fg = g0 > gn ? g0 : gn;
  R fr = r0 > rn ? r0 : rn;
  R mx = fg > fr ? fg : fr;
  *Fg = (R(1) - w) * fg + w * mx;
  *Fr = (R(1) - w) * fr + w * mx;
}

// Branches of the flattener of cell 3 of c[0..6] (flatten_cell): each
// ftilde's compression test and clamp, the neighbour chosen, the maxima taken.
template <typename R>
__device__ __forceinline__ unsigned ftilde_code(const FlatCell<R>* c, int m, bool gas, R w) {
  auto pe = [&](int o) { return gas ? c[m + o].pg + w * c[m + o].pr : c[m + o].pr + w * c[m + o].pg; };
  auto ve = [&](int o) { return gas ? c[m + o].vg : c[m + o].vr; };
  R dp1 = pe(1) - pe(-1), dp2 = pe(2) - pe(-2);
  R dv = ve(1) - ve(-1);
  R p1 = pe(1), pm = pe(-1);
  if (!(fabs(dp1) > R(0.33) * (p1 < pm ? p1 : pm) && dv < R(0))) return 0u;
  R sp = dp2 != R(0) ? dp1 / dp2 : R(0);
  R f = R(10) * (sp - R(0.75));
  return f <= R(0) ? 1u : (f >= R(1) ? 3u : 2u);
}
template <typename R>
__device__ __forceinline__ unsigned flatten_code(const FlatCell<R>* c, R og, R orr) {
  const R w = c[3].w;
  R g0 = ftilde<R>(c, 3, true, w), r0 = ftilde<R>(c, 3, false, w);
  R pg1 = c[4].pg + w * c[4].pr, pgm = c[2].pg + w * c[2].pr;
  R pr1 = c[4].pr + w * c[4].pg, prm = c[2].pr + w * c[2].pg;
  int sg = (pg1 - pgm) < R(0) ? 1 : -1;
  int sr = (pr1 - prm) < R(0) ? 1 : -1;
  R gn = ftilde<R>(c, 3 + sg, true, c[3 + sg].w);
  R rn = ftilde<R>(c, 3 + sr, false, c[3 + sr].w);
  R fg = g0 > gn ? g0 : gn, fr = r0 > rn ? r0 : rn;
  R Fg = (R(1) - w) * fg + w * (fg > fr ? fg : fr), Fr = (R(1) - w) * fr + w * (fg > fr ? fg : fr);
  unsigned k = ftilde_code<R>(c, 3, true, w) | ftilde_code<R>(c, 3, false, w) << 2 |
               ftilde_code<R>(c, 3 + sg, true, c[3 + sg].w) << 4 | ftilde_code<R>(c, 3 + sr, false, c[3 + sr].w) << 6;
  k |= (sg > 0 ? 1u : 0u) << 8 | (sr > 0 ? 1u : 0u) << 9 | (g0 > gn ? 1u : 0u) << 10 | (r0 > rn ? 1u : 0u) << 11;
  k |= (fg > fr ? 1u : 0u) << 12 | (Fg > og ? 1u : 0u) << 13 | (Fr > orr ? 1u : 0u) << 14;
  return k;
}

template <typename R>
__global__ void k_flatten(DevParams p, const BoxGeo* __restrict__ boxes, int nbox,
                          const double* __restrict__ P0, const R* __restrict__ aux0,
                          R* __restrict__ flat0, int d) {
  for (int bi = 0; bi < nbox; ++bi) {
    const BoxGeo& bx = boxes[bi];
    const double* P = P0 + 12 * bx.coff;
    const R* aux = aux0 + 10 * bx.coff;
    R* flat = flat0 + 2 * bx.coff;
    int len[3], off[3];
    for (int e = 0; e < 3; ++e) {
      if (bx.n[e] > 1) {
        len[e] = bx.n[e] + 2;
        off[e] = -1;
      } else {
        len[e] = 1;
        off[e] = 0;
      }
    }
    long long total = (long long)len[0] * len[1] * len[2];
    const long long st = bx.str[d];
    for (long long id = HR_TID; id < total; id += HR_STRIDE) {
      long long r = id;
      int i = (int)(r % len[0]) + off[0];
      r /= len[0];
      int j = (int)(r % len[1]) + off[1];
      int k = (int)(r / len[1]) + off[2];
      long long t = cell_index(bx, i, j, k);
      FlatCell<R> c[7];
#pragma unroll
      for (int m = 0; m < 7; ++m) {
        long long cm = t + (m - 3) * st;
        c[m].pg = R((p.gam - 1.0) * P[UU * bx.ntot + cm]);
        c[m].pr = R(P[ER * bx.ntot + cm] * (1.0 / 3.0));
        c[m].vg = aux[(1 + 3 * d) * bx.ntot + cm];
        c[m].vr = aux[(2 + 3 * d) * bx.ntot + cm];
        c[m].w = aux[(3 + 3 * d) * bx.ntot + cm];
      }
      R Fg, Fr;
      flatten_cell<R>(c, &Fg, &Fr);
      R og = flat[t], orr = flat[bx.ntot + t];
      if (p.sig) sig_put(p, bx.coff + t, 30 + d, flatten_code<R>(c, og, orr));
      flat[t] = Fg > og ? Fg : og;
      flat[bx.ntot + t] = Fr > orr ? Fr : orr;
    }
  }
}

// The flattener in FP64.  Each cell's own value f(m) (ftilde) is formed once
// and handed to the neighbours: a thread walks along x2 or x3 with a window in
// registers, or, along x1, a warp passes values between its lanes.  With
// X = dp_gas and Y = dp_rad across the cell the blended differences are X + w Y
// and Y + w X; the rest of the test is formed only where the flow compresses,
// the wider difference only where the jump is a shock.  About 12 FP64
// instructions per cell where nothing compresses.  `fresh`: the first sub-step
// (no earlier value to keep).  Measured over an RK3 step: 256x128x64 torus
// 3.05 -> 1.38 ms, 64x32x16 0.18 -> 0.10.

// f(m) from the jump dp across the cell and the wider jump d2.
__device__ __forceinline__ double flat_value(double dp, double d2) {
  const double f = d2 != 0.0 ? 10.0 * (dp / d2 - 0.75) : -7.5;
  return f < 0.0 ? 0.0 : (f > 1.0 ? 1.0 : f);
}
// The jump dp is a shock beside the blended pressures pp, pm.
__device__ __forceinline__ bool flat_shock(double dp, double pp, double pm) {
  return fabs(dp) > 0.33 * (pp < pm ? pp : pm);
}

// The cell's flattener from f of the cell and its two neighbours (gas, rad).
__device__ __forceinline__ void flat_store(const DevParams& p, double w, const double fg[3], const double fr[3],
                                           bool gup, bool rup, bool fresh, double* F, double* R) {
  const double ng = gup ? fg[2] : fg[0], nr = rup ? fr[2] : fr[0];
  const double a = fg[1] > ng ? fg[1] : ng, b = fr[1] > nr ? fr[1] : nr;
  if (a == 0.0 && b == 0.0) {
    if (fresh) *F = *R = 0.0;
    return;
  }
  const double mx = a > b ? a : b;
  const double g = (1.0 - w) * a + w * mx, r = (1.0 - w) * b + w * mx;
  if (fresh || g > *F) *F = g;
  if (fresh || r > *R) *R = r;
}

// The branch signature of the flattener of the cell at t (a test instrument).
__device__ __forceinline__ void flat_sig(const DevParams& p, const BoxGeo& bx, const double* P, const double* aux,
                                             long long t, int d, double og, double orr) {
  FlatCell<double> c[7];
  for (int m = 0; m < 7; ++m) {
    const long long x = t + (m - 3) * bx.str[d];
    c[m].pg = (p.gam - 1.0) * P[UU * bx.ntot + x];
    c[m].pr = P[ER * bx.ntot + x] * (1.0 / 3.0);
    c[m].vg = aux[(1 + 3 * d) * bx.ntot + x];
    c[m].vr = aux[(2 + 3 * d) * bx.ntot + x];
    c[m].w = aux[(3 + 3 * d) * bx.ntot + x];
  }
  sig_put(p, bx.coff + t, 30 + d, flatten_code<double>(c, og, orr));
}

template <int d, bool SIG>
__device__ __forceinline__ void flat_cols(const DevParams& p, const BoxGeo* __restrict__ boxes, int nbox,
                                          const double* __restrict__ P0, const double* __restrict__ aux0,
                                          double* __restrict__ flat0, int chunk, bool fresh) {
  constexpr int o = 3 - d;
  long long done = 0;
  for (int bi = 0; bi < nbox; ++bi) {
    const BoxGeo& bx = boxes[bi];
    const double* P = P0 + 12 * bx.coff;
    const double* aux = aux0 + 10 * bx.coff;
    double* flat = flat0 + 2 * bx.coff;
    const int wx = bx.n[0] > 1 ? bx.n[0] + 2 : 1, wo = bx.n[o] > 1 ? bx.n[o] + 2 : 1;
    const int nd = bx.n[d] + 2, nch = (nd + chunk - 1) / chunk, cols = wx * wo;
    const long long total = (long long)nch * cols, st = bx.str[d], nt = bx.ntot;
    const double* Ug = P + UU * nt;
    const double* Er = P + ER * nt;
    const double* vg = aux + (1 + 3 * d) * nt;
    const double* vr = aux + (2 + 3 * d) * nt;
    const double* wt = aux + (3 + 3 * d) * nt;
    for (long long id = first_item(done); id < total; id += HR_STRIDE) {
      const int ch = (int)(id / cols), col = (int)(id - (long long)ch * cols);
      const int c0 = ch * chunk - 1, c1 = min(c0 + chunk, bx.n[d] + 1);  // cells c0 .. c1 - 1
      int ii[3];
      ii[0] = col % wx + (bx.n[0] > 1 ? -1 : 0);
      ii[o] = col / wx + (bx.n[o] > 1 ? -1 : 0);
      ii[d] = c0 - 1;
      long long t = cell_index(bx, ii[0], ii[1], ii[2]);
      // pressures of cells m-2 .. m+2 around m = c0 - 1, velocities of m-1 .. m+1
      double pg[5], pr[5], ug[3], ur[3], fg[3], fr[3], wc = 0.0, wm = 0.0;
      bool gu = false, ru = false;  // f's neighbour lies at m + 1, of cell m - 1
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        pg[e + 1] = p.gm1 * Ug[t + (e - 2) * st];
        pr[e + 1] = Er[t + (e - 2) * st] * (1.0 / 3.0);
      }
      ug[1] = vg[t - st];
      ug[2] = vg[t];
      ur[1] = vr[t - st];
      ur[2] = vr[t];
      fg[1] = fg[2] = fr[1] = fr[2] = 0.0;
      for (int m = c0 - 1; m <= c1; ++m, t += st) {
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          pg[e] = pg[e + 1];
          pr[e] = pr[e + 1];
        }
        pg[4] = p.gm1 * Ug[t + 2 * st];
        pr[4] = Er[t + 2 * st] * (1.0 / 3.0);
        ug[0] = ug[1];
        ug[1] = ug[2];
        ug[2] = vg[t + st];
        ur[0] = ur[1];
        ur[1] = ur[2];
        ur[2] = vr[t + st];
        wm = wc;  // of cell m - 1
        wc = wt[t];
        fg[0] = fg[1];
        fg[1] = fg[2];
        fr[0] = fr[1];
        fr[1] = fr[2];
        const double X = pg[3] - pg[1], Y = pr[3] - pr[1];
        const double dg = fma(wc, Y, X), dr = fma(wc, X, Y);
        fg[2] = fr[2] = 0.0;
        if (ug[2] < ug[0] && flat_shock(dg, fma(wc, pr[3], pg[3]), fma(wc, pr[1], pg[1])))
          fg[2] = flat_value(dg, fma(wc, pr[4] - pr[0], pg[4] - pg[0]));
        if (ur[2] < ur[0] && flat_shock(dr, fma(wc, pg[3], pr[3]), fma(wc, pg[1], pr[1])))
          fr[2] = flat_value(dr, fma(wc, pg[4] - pg[0], pr[4] - pr[0]));
        if (m > c0) {
          const long long c = t - st;
          if (SIG) flat_sig(p, bx, P, aux, c, d, fresh ? 0.0 : flat[c], fresh ? 0.0 : flat[nt + c]);
          flat_store(p, wm, fg, fr, gu, ru, fresh, flat + c, flat + nt + c);
        }
        gu = dg < 0.0;
        ru = dr < 0.0;
      }
    }
    done += total;
  }
}

// d = 0: a warp takes 26 consecutive cells of the joined rows (as k_recon_rows),
// one per lane, three lanes on either side for the neighbours only.
template <bool SIG>
__device__ __forceinline__ void flat_rows(const DevParams& p, const BoxGeo* __restrict__ boxes, int nbox,
                                          const double* __restrict__ P0, const double* __restrict__ aux0,
                                          double* __restrict__ flat0, bool fresh) {
  const int lane = threadIdx.x & 31;
  const unsigned full = 0xffffffffu;
  long long done = 0;
  for (int bi = 0; bi < nbox; ++bi) {
    const BoxGeo& bx = boxes[bi];
    const double* P = P0 + 12 * bx.coff;
    const double* aux = aux0 + 10 * bx.coff;
    double* flat = flat0 + 2 * bx.coff;
    const int w1 = bx.n[1] > 1 ? bx.n[1] + 2 : 1, w2 = bx.n[2] > 1 ? bx.n[2] + 2 : 1;
    const int o1 = bx.n[1] > 1 ? -1 : 0, o2 = bx.n[2] > 1 ? -1 : 0;
    const int N0 = bx.N[0], cells = w1 * w2 * N0, ntask = (cells + 25) / 26;
    const long long total = 32LL * ntask, nt = bx.ntot;
    for (long long id = first_item(done); id < total; id += HR_STRIDE) {
      const int f0 = 26 * (int)(id >> 5) - 3 + lane, f = min(max(f0, 0), cells - 1), row = f / N0;
      const int x = f - row * N0 - 4;
      const long long t = cell_index(bx, x, row % w1 + o1, row / w1 + o2);
      const double pg = p.gm1 * P[UU * nt + t], pr = P[ER * nt + t] * (1.0 / 3.0);
      const double vg = aux[nt + t], vr = aux[2 * nt + t], w = aux[3 * nt + t];
      const double pgp = __shfl_down_sync(full, pg, 1), pgm = __shfl_up_sync(full, pg, 1);
      const double prp = __shfl_down_sync(full, pr, 1), prm = __shfl_up_sync(full, pr, 1);
      const bool cg = __shfl_down_sync(full, vg, 1) < __shfl_up_sync(full, vg, 1);
      const bool cr = __shfl_down_sync(full, vr, 1) < __shfl_up_sync(full, vr, 1);
      const double X = pgp - pgm, Y = prp - prm, dg = fma(w, Y, X), dr = fma(w, X, Y);
      const bool hg = cg && flat_shock(dg, fma(w, prp, pgp), fma(w, prm, pgm));
      const bool hr = cr && flat_shock(dr, fma(w, pgp, prp), fma(w, pgm, prm));
      double fg[3] = {0.0, 0.0, 0.0}, fr[3] = {0.0, 0.0, 0.0};
      if (__any_sync(full, hg || hr)) {
        const double X2 = __shfl_down_sync(full, pg, 2) - __shfl_up_sync(full, pg, 2);
        const double Y2 = __shfl_down_sync(full, pr, 2) - __shfl_up_sync(full, pr, 2);
        if (hg) fg[1] = flat_value(dg, fma(w, Y2, X2));
        if (hr) fr[1] = flat_value(dr, fma(w, X2, Y2));
        fg[0] = __shfl_up_sync(full, fg[1], 1);
        fg[2] = __shfl_down_sync(full, fg[1], 1);
        fr[0] = __shfl_up_sync(full, fr[1], 1);
        fr[2] = __shfl_down_sync(full, fr[1], 1);
      }
      if (lane < 3 || lane > 28 || f0 >= cells || x < -1 || x > bx.n[0]) continue;
      if (SIG) flat_sig(p, bx, P, aux, t, 0, fresh ? 0.0 : flat[t], fresh ? 0.0 : flat[nt + t]);
      flat_store(p, w, fg, fr, dg < 0.0, dr < 0.0, fresh, flat + t, flat + nt + t);
    }
    done += total;
  }
}

// One launch for the directions d0 + blockIdx.y: a grid that does not fill the
// GPU runs them side by side.
struct FlatSet {
  double* f[3];
};
struct Chunks {
  int c[3];
};
template <bool SIG>
__global__ void __launch_bounds__(128) k_flat(DevParams p, const BoxGeo* __restrict__ boxes, int nbox,
                                              const double* __restrict__ P0, const double* __restrict__ aux0,
                                              FlatSet flat, Chunks ch, bool fresh, int d0) {
  const int d = d0 + blockIdx.y;
  if (!p.act[d]) return;
  if (d == 0) flat_rows<SIG>(p, boxes, nbox, P0, aux0, flat.f[0], fresh);
  else if (d == 1) flat_cols<1, SIG>(p, boxes, nbox, P0, aux0, flat.f[1], ch.c[1], fresh);
  else flat_cols<2, SIG>(p, boxes, nbox, P0, aux0, flat.f[2], ch.c[2], fresh);
}

// ------------------------------------------------------------- reconstruction
template <typename R>
__device__ __forceinline__ R mc_slope(R qm, R q0, R qp) {
  R dl = q0 - qm, dr = qp - q0, dc = R(0.5) * (qp - qm);
  if (dl * dr <= R(0)) return R(0);
  R m = fabs(dc);
  R a = R(2) * fabs(dl), b = R(2) * fabs(dr);
  m = m < a ? m : a;
  m = m < b ? m : b;
  return dc > R(0) ? m : -m;
}

// PPM edge values of the centre of s[0..4] (Colella & Woodward 1984, no
// contact steepening), flattened toward the cell mean by chi, then limited.
// sm, s0, sp: the cell and its neighbours; dm, d0, dp: their MC slopes.
template <typename R>
__device__ __forceinline__ void ppm_slopes(R sm, R s0, R sp, R dm, R d0, R dp, R chi, R* aL, R* aR) {
  const R sixth = R(1.0 / 6.0);
  R l = R(0.5) * (sm + s0) - (d0 - dm) * sixth;
  R r = R(0.5) * (s0 + sp) - (dp - d0) * sixth;
  R q = s0;
  l = (R(1) - chi) * l + chi * q;
  r = (R(1) - chi) * r + chi * q;
  if ((r - q) * (q - l) <= R(0)) {
    l = q;
    r = q;
  } else {
    R dd = r - l;
    R m6 = R(6) * (q - R(0.5) * (l + r));
    if (dd * m6 > dd * dd) l = R(3) * q - R(2) * r;
    else if (-dd * dd > dd * m6) r = R(3) * q - R(2) * l;
  }
  *aL = l;
  *aR = r;
}

template <typename R>
__device__ __forceinline__ void ppm_cell(const R s[5], R chi, R* aL, R* aR) {
  R dm = mc_slope<R>(s[0], s[1], s[2]);
  R d0 = mc_slope<R>(s[1], s[2], s[3]);
  R dp = mc_slope<R>(s[2], s[3], s[4]);
  ppm_slopes<R>(s[1], s[2], s[3], dm, d0, dp, chi, aL, aR);
}

// ------------------------------------------------------- edge reconstruction
// FP64 reconstruction of one direction: the PPM parabola (or MC line) of every
// primitive in every cell of the face range (cells -1..n_d along d, transverse
// range widened by one layer), flattened by the cell's GAS or RAD flattener and
// stored as its two edge values (EdgeSet); the face kernel reads the upper edge
// of cell f-1 and the lower edge of cell f.  In r and phi on the Kerr-Schild grid
// the velocity and field components are reconstructed as sqrt(-g) times the
// primitive (Sec. 4.3).
//
// Bound by FP64 instructions (each holds an SM's FP64 pipe for 16 clocks), so
// nothing is computed twice: neighbouring cells share the difference, the MC
// slope and the interface value between them (a thread walks along d with
// them in registers, or, along x1, a warp passes them between its lanes), and
// the limiters work on differences: with a = |r - q|, b = |q - l| the
// monotonicity tests of Colella & Woodward read b > 2 a and a > 2 b, and twice
// the MC slope is min(|dl + dr|, 4 |dl|, 4 |dr|).  About 11 FP64 instructions
// per cell and variable.  One thread (or warp) takes one variable: few
// registers, many warps, and small grids still fill the SMs.  Measured over an
// RK3 step (GB300, PPM, event time of the class) against a slope pass plus a
// parabola pass of one thread per cell: Kerr-Schild torus 256x128x64 17.2 -> 7.8
// ms, 64x32x16 0.75 -> 0.19, 256 zones in 1D 0.125 -> 0.024.

// The limiters' comparisons and powers of two act on the bit patterns, off the
// FP64 pipe: twice a double's bits (the sign shifted out) order like its
// magnitude.  (A mask in place of the shift is compiled to an FP64 |x|.)
__device__ __forceinline__ unsigned long long mag_key(double x) {
  return (unsigned long long)__double_as_longlong(x) << 1;
}
// |a| < 2^k |b|, for normal numbers and zero (a subnormal b counts as up to
// 2^(k-1022); a slope limited by it is off by that much at most)
__device__ __forceinline__ bool mag_less(double a, double b, int k = 0) {
  return mag_key(a) < mag_key(b) + ((unsigned long long)k << 53);
}
__device__ __forceinline__ bool opposite(double a, double b) { return (__double2hiint(a) ^ __double2hiint(b)) < 0; }

// Twice the MC slope from the differences to the left and right neighbour.
__device__ __forceinline__ double mc_twice(double dm, double dp) {
  const double s = dm + dp, m = mag_less(dm, dp) ? dm : dp;  // central, smaller one-sided
  if (opposite(dm, dp) || mag_key(m) == 0) return 0.0;
  return mag_less(s, m, 2) ? s : __hiloint2double(__double2hiint(m) + (2 << 20), __double2loint(m));
}
// Branch of mc_twice: 0 opposite or zero differences (no slope), 1 central, 2 twice
// the left, 3 twice the right difference.
__device__ __forceinline__ unsigned mc_twice_code(double dm, double dp) {
  const bool left = mag_less(dm, dp);
  const double m = left ? dm : dp;
  if (opposite(dm, dp) || mag_key(m) == 0) return 0u;
  if (mag_less(dm + dp, m, 2)) return 1u;
  return left ? 2u : 3u;
}
// PPM interface value between cells of values sm and sm + d whose doubled MC
// slopes are Dm and D0 (third-order with limited slopes).
__device__ __forceinline__ double ppm_face(double sm, double d, double Dm, double D0) {
  return fma(Dm - D0, 1.0 / 12.0, fma(0.5, d, sm));
}
// Flattening and monotonicity of the parabola of a cell of value q with edge
// values l, r; returns the branch: 0 none, 1 flat, 2 left edge moved, 3 right edge
// moved.
__device__ __forceinline__ unsigned ppm_limit(double q, double chi, double& l, double& r) {
  if (mag_key(chi) != 0) {
    l = (1.0 - chi) * l + chi * q;
    r = (1.0 - chi) * r + chi * q;
  }
  const double A = r - q, B = q - l, l2 = fma(-2.0, A, q), r2 = fma(2.0, B, q);
  const bool flat = opposite(A, B), left = !mag_less(B, A, 1), right = !mag_less(A, B, 1);  // b >= 2 a, a >= 2 b
  l = flat ? q : (left ? l2 : l);
  r = flat ? q : (!left && right ? r2 : r);
  // an edge on the cell's value is flat too: the same values, but the adjoint and
  // the branch signature tell it from a monotone parabola
  return flat || mag_key(A) == 0 || mag_key(B) == 0 ? 1u : (left ? 2u : (right ? 3u : 0u));
}

// d = 1, 2: a thread walks `chunk` cells of one column along d for one
// variable; lanes are neighbours along x1, so every load is coalesced.  A
// chunk's start repeats two slopes and one interface: about one cell's work.
// SIG: folds its decisions into the branch signature (a test instrument; a
// variant of its own, so that the hot one holds no registers for it).
template <int MET, int d, bool SIG>
__device__ __forceinline__ void recon_cols(const DevParams& p, const BoxGeo* __restrict__ boxes, int nbox,
                                           const double* __restrict__ P0, const double* __restrict__ aux0,
                                           const double* __restrict__ flat0, const EdgeSet& E0, int chunk) {
  const bool weighted = (MET == KS) && (d != 1);
  constexpr int o = 3 - d;  // the other transverse direction beside x1
  long long done = 0;
  for (int bi = 0; bi < nbox; ++bi) {
    const BoxGeo& bx = boxes[bi];
    const double* P = P0 + 12 * bx.coff;
    const double* aux = aux0 + 10 * bx.coff;
    const double* flat = flat0 + 2 * bx.coff;
    const EdgeSet E = E0.box(bx);
    const int wx = bx.n[0] > 1 ? bx.n[0] + 2 : 1, wo = bx.n[o] > 1 ? bx.n[o] + 2 : 1;
    const int nd = bx.n[d] + 2, nch = (nd + chunk - 1) / chunk, cols = wx * wo;
    const long long total = 12LL * nch * cols, st = bx.str[d], nt = bx.ntot;
    for (long long id = first_item(done); id < total; id += HR_STRIDE) {
      const int qc = (int)(id / cols), col = (int)(id - (long long)qc * cols);
      const int q = qc / nch, c0 = (qc - q * nch) * chunk - 1;
      const int c1 = min(c0 + chunk, bx.n[d] + 1);  // cells c0 .. c1 - 1
      int ii[3];
      ii[0] = col % wx + (bx.n[0] > 1 ? -1 : 0);
      ii[o] = col / wx + (bx.n[o] > 1 ? -1 : 0);
      ii[d] = c0;
      long long t = cell_index(bx, ii[0], ii[1], ii[2]);
      const bool wq = weighted && ((q >= U1 && q <= B3) || q >= UR1);
      const double* Pq = P + q * nt;
      const double* chi = flat + (q < ER ? 0 : nt);
      double* __restrict__ El = E.plane(0, q, nt);
      double* __restrict__ Er = E.plane(1, q, nt);
      auto ld = [&](long long x) { return wq ? aux[x] * Pq[x] : Pq[x]; };
      double s0 = ld(t), sp = ld(t + st), dp = sp - s0;
      const double sm = ld(t - st), dm = s0 - sm;
      double D0 = mc_twice(dm, dp), aL = 0.0;
      if (p.recon == 0) {
        const double dmm = sm - ld(t - 2 * st);
        aL = ppm_face(sm, dm, mc_twice(dmm, dm), D0);
        if (SIG && c0 == -1)
          sig_put(p, bx.coff + t - st, 10 + d, (unsigned long long)q << 8 | mc_twice_code(dmm, dm));
      }
      double dl = dm;  // kept for the branch signature only
#pragma unroll 2
      for (int c = c0; c < c1; ++c, t += st) {
        if (SIG) sig_put(p, bx.coff + t, 10 + d, (unsigned long long)q << 8 | mc_twice_code(dl, dp));
        const double s2 = ld(t + 2 * st), d2 = s2 - sp, Dp = mc_twice(dp, d2);
        double l, r;
        if (p.recon == 0) {
          const double aR = ppm_face(s0, dp, D0, Dp);
          l = aL;
          r = aR;
          const unsigned code = ppm_limit(s0, chi[t], l, r);
          if (SIG) sig_put(p, bx.coff + t, 20 + d, (unsigned long long)q << 8 | code);
          aL = aR;
        } else {
          l = fma(-0.25, D0, s0);
          r = fma(0.25, D0, s0);
        }
        El[t] = l;
        Er[t] = r;
        if (SIG && c == bx.n[d])
          sig_put(p, bx.coff + t + st, 10 + d, (unsigned long long)q << 8 | mc_twice_code(dp, d2));
        s0 = sp;
        sp = s2;
        dl = dp;
        dp = d2;
        D0 = Dp;
      }
    }
    done += total;
  }
}

// d = 0: a warp takes 60 consecutive cells of the rows of the transverse range
// (rows joined end to end, ghosts included) for one variable, two cells per
// lane, the first and last lane for the neighbours only; differences, slopes
// and interface values pass between lanes.  Values that cross a row's end
// reach ghost cells that are not stored.
template <int MET, bool SIG>
__device__ __forceinline__ void recon_rows(const DevParams& p, const BoxGeo* __restrict__ boxes, int nbox,
                                           const double* __restrict__ P0, const double* __restrict__ aux0,
                                           const double* __restrict__ flat0, const EdgeSet& E0) {
  const bool weighted = (MET == KS);
  const int lane = threadIdx.x & 31;
  const unsigned full = 0xffffffffu;
  long long done = 0;
  for (int bi = 0; bi < nbox; ++bi) {
    const BoxGeo& bx = boxes[bi];
    const double* P = P0 + 12 * bx.coff;
    const double* aux = aux0 + 10 * bx.coff;
    const double* flat = flat0 + 2 * bx.coff;
    const EdgeSet E = E0.box(bx);
    const int w1 = bx.n[1] > 1 ? bx.n[1] + 2 : 1, w2 = bx.n[2] > 1 ? bx.n[2] + 2 : 1;
    const int o1 = bx.n[1] > 1 ? -1 : 0, o2 = bx.n[2] > 1 ? -1 : 0;
    const int N0 = bx.N[0], cells = w1 * w2 * N0, ntask = (cells + 59) / 60;
    const long long total = 12LL * ntask * 32, nt = bx.ntot;
    for (long long id = first_item(done); id < total; id += HR_STRIDE) {
      const int task = (int)(id >> 5), q = task / ntask, seg = task - q * ntask;
      // this lane's two cells and their places in memory
      int x[2];
      long long t[2];
      const int f0 = 60 * seg - 2 + 2 * lane;
#pragma unroll
      for (int e = 0; e < 2; ++e) {
        const int f = min(max(f0 + e, 0), cells - 1), row = f / N0;
        x[e] = f - row * N0 - 4;
        t[e] = cell_index(bx, x[e], row % w1 + o1, row / w1 + o2);
      }
      const bool wq = weighted && ((q >= U1 && q <= B3) || q >= UR1);
      const double* Pq = P + q * nt;
      double s[2];
#pragma unroll
      for (int e = 0; e < 2; ++e) s[e] = wq ? aux[t[e]] * Pq[t[e]] : Pq[t[e]];
      const double sm = __shfl_up_sync(full, s[1], 1);
      const double d0 = s[0] - sm, d1 = s[1] - s[0], d2 = __shfl_down_sync(full, d0, 1);
      const double D0 = mc_twice(d0, d1), D1 = mc_twice(d1, d2);
      double l[2], r[2], chi[2] = {0.0, 0.0};
      const bool mine = lane >= 1 && lane <= 30 && f0 < cells;
      unsigned code[2] = {0u, 0u};
      if (p.recon == 0) {
        const double* ch = flat + (q < ER ? 0 : nt);
#pragma unroll
        for (int e = 0; e < 2; ++e)
          if (x[e] >= -1 && x[e] <= bx.n[0]) chi[e] = ch[t[e]];
        const double Dm = __shfl_up_sync(full, D1, 1);
        l[0] = ppm_face(sm, d0, Dm, D0);
        l[1] = ppm_face(s[0], d1, D0, D1);
        r[0] = l[1];
        r[1] = __shfl_down_sync(full, l[0], 1);
#pragma unroll
        for (int e = 0; e < 2; ++e) code[e] = ppm_limit(s[e], chi[e], l[e], r[e]);
      } else {
        l[0] = fma(-0.25, D0, s[0]);
        r[0] = fma(0.25, D0, s[0]);
        l[1] = fma(-0.25, D1, s[1]);
        r[1] = fma(0.25, D1, s[1]);
      }
#pragma unroll
      for (int e = 0; e < 2; ++e) {
        if (!mine || f0 + e >= cells) continue;
        if (SIG && x[e] >= -2 && x[e] <= bx.n[0] + 1)
          sig_put(p, bx.coff + t[e], 10, (unsigned long long)q << 8 | (e ? mc_twice_code(d1, d2) : mc_twice_code(d0, d1)));
        if (x[e] < -1 || x[e] > bx.n[0]) continue;
        if (SIG && p.recon == 0) sig_put(p, bx.coff + t[e], 20, (unsigned long long)q << 8 | code[e]);
        E.plane(0, q, nt)[t[e]] = l[e];
        E.plane(1, q, nt)[t[e]] = r[e];
      }
    }
    done += total;
  }
}

// One launch per direction: fewer registers (the merged kernel holds 88), which a
// grid that fills the GPU needs (256x128x64 per RK3 step 7.8 ms, merged 8.0;
// batch of 12 boxes 5.16 against 5.31).
template <int MET, bool SIG>
__global__ void __launch_bounds__(256) k_recon_rows(DevParams p, const BoxGeo* __restrict__ boxes, int nbox,
                                                    const double* __restrict__ P0, const double* __restrict__ aux0,
                                                    const double* __restrict__ flat0, EdgeSet E0) {
  recon_rows<MET, SIG>(p, boxes, nbox, P0, aux0, flat0, E0);
}
template <int MET, int d, bool SIG>
__global__ void __launch_bounds__(256) k_recon_cols(DevParams p, const BoxGeo* __restrict__ boxes, int nbox,
                                                    const double* __restrict__ P0, const double* __restrict__ aux0,
                                                    const double* __restrict__ flat0, EdgeSet E0, int chunk) {
  recon_cols<MET, d, SIG>(p, boxes, nbox, P0, aux0, flat0, E0, chunk);
}
// One launch for the directions d0 + blockIdx.y: a grid that does not fill the GPU
// runs them side by side (64x32x16 per RK3 step 0.22 -> 0.19 ms).
template <int MET>
__global__ void __launch_bounds__(256) k_recon_all(DevParams p, const BoxGeo* __restrict__ boxes, int nbox,
                                                   const double* __restrict__ P0, const double* __restrict__ aux0,
                                                   FlatSet flat, EdgeSets E, Chunks ch, int d0) {
  const int d = d0 + blockIdx.y;
  if (!p.act[d]) return;
  if (d == 0) recon_rows<MET, false>(p, boxes, nbox, P0, aux0, flat.f[0], E.d[0]);
  else if (d == 1) recon_cols<MET, 1, false>(p, boxes, nbox, P0, aux0, flat.f[1], E.d[1], ch.c[1]);
  else recon_cols<MET, 2, false>(p, boxes, nbox, P0, aux0, flat.f[2], E.d[2], ch.c[2]);
}

// FP32 reconstruction (split precision), one thread per cell of the face range
// and all 12 primitives: FP32 arithmetic is cheap, so each cell computes its
// own slopes.
template <int MET, int d>
__global__ void __launch_bounds__(256) k_edges(DevParams p, const BoxGeo* __restrict__ boxes, int nbox,
                                               const double* __restrict__ P0, const float* __restrict__ aux0,
                                               const float* __restrict__ flat0, float* __restrict__ E0) {
  typedef float R;
  const bool weighted = (MET == KS) && (d != 1);
  for (int bi = 0; bi < nbox; ++bi) {
    const BoxGeo& bx = boxes[bi];
    const double* P = P0 + 12 * bx.coff;
    const R* aux = aux0 + 10 * bx.coff;
    const R* flat = flat0 + 2 * bx.coff;
    R* E = E0 + 24 * bx.coff;
    int len[3], off[3];
    for (int e = 0; e < 3; ++e) {
      if (bx.n[e] > 1) {
        len[e] = bx.n[e] + 2;
        off[e] = -1;
      } else {
        len[e] = 1;
        off[e] = 0;
      }
    }
    long long total = (long long)len[0] * len[1] * len[2];
    const long long st = bx.str[d];
    for (long long id = HR_TID; id < total; id += HR_STRIDE) {
      long long r = id;
      int i = (int)(r % len[0]) + off[0];
      r /= len[0];
      int j = (int)(r % len[1]) + off[1];
      int k = (int)(r / len[1]) + off[2];
      long long t = cell_index(bx, i, j, k);
      R chg = R(0), chr = R(0);
      if (p.recon == 0) {
        chg = flat[t];
        chr = flat[bx.ntot + t];
      }
      R gw[5];
      if (weighted) {
#pragma unroll
        for (int m = 0; m < 5; ++m) gw[m] = aux[t + (m - 2) * st];
      }
#pragma unroll
      for (int q = 0; q < NPR; ++q) {
        const bool wq = weighted && ((q >= U1 && q <= B3) || q >= UR1);
        R s[5];
#pragma unroll
        for (int m = 0; m < 5; ++m) {
          R v = R(P[q * bx.ntot + t + (m - 2) * st]);
          s[m] = wq ? gw[m] * v : v;
        }
        R aL, aR;
        if (p.recon == 0) {
          ppm_cell<R>(s, q < ER ? chg : chr, &aL, &aR);
        } else {
          R dq = mc_slope<R>(s[1], s[2], s[3]);
          aL = s[2] - R(0.5) * dq;
          aR = s[2] + R(0.5) * dq;
        }
        E[q * bx.ntot + t] = aL;
        E[(NPR + q) * bx.ntot + t] = aR;
      }
    }
  }
}

// Riemann flux through one face of direction d (0-based) from the two
// reconstructed states: both states' gas and radiation signal speeds, then
// HLL or LAXF (Eqs. hll, lax), the gas and radiation groups with their own
// speeds; F[B_d] = 0.  smax: the largest signal speed (for the CFL step).
// Split precision's face kernel (FP64: face_flux64).
template <int MET, typename R, int d>
__device__ __forceinline__ void face_flux(const DevParams& p, const Geo<MET, R>& g, R dxd, R kL, R kR, R ks,
                                          const R PL[NPR], const R PR[NPR], R out[NPR], R* smax,
                                          unsigned* code = nullptr, R* fs = nullptr, R* gas = nullptr) {
  R sL[4], sR[4];
  unsigned cL = 0, cR = 0;
  R lL[3], lR[3];  // Lorentz factors and 1/u^t of the states, for face_accum
  const R dl = sqrt(g.gdd(d + 1)) * dxd;  // proper cell length along d, for the optical depth
  face_speeds<MET, R>(p, g, d + 1, dl, kL, ks, PL, sL, code ? &cL : nullptr, lL);
  face_speeds<MET, R>(p, g, d + 1, dl, kR, ks, PR, sR, code ? &cR : nullptr, lR);
  R cmaxg = fmax(R(0), fmax(sL[1], sR[1]));
  R cming = -fmin(R(0), fmin(sL[0], sR[0]));
  R cmaxr = fmax(R(0), fmax(sL[3], sR[3]));
  R cminr = -fmin(R(0), fmin(sL[2], sR[2]));
  if (code) {  // which signal speed each maximum took, and the speed caps
    unsigned c = cL | (cR << 3);
    c |= (sL[1] >= sR[1] ? 0u : 1u) << 6 | (R(0) > fmax(sL[1], sR[1]) ? 1u : 0u) << 7;
    c |= (sL[0] <= sR[0] ? 0u : 1u) << 8 | (R(0) < fmin(sL[0], sR[0]) ? 1u : 0u) << 9;
    c |= (sL[3] >= sR[3] ? 0u : 1u) << 10 | (R(0) > fmax(sL[3], sR[3]) ? 1u : 0u) << 11;
    c |= (sL[2] <= sR[2] ? 0u : 1u) << 12 | (R(0) < fmin(sL[2], sR[2]) ? 1u : 0u) << 13;
    c |= (cmaxg > cming ? 1u : 0u) << 14 | (cmaxr > cminr ? 1u : 0u) << 15;
    *code = c;
  }
  // weights of (F_L, U_L) and (F_R, U_R) in the flux, gas and radiation groups
  R fLg, uLg, fRg, uRg, fLr, uLr, fRr, uRr;
  if (p.flux == 0) {  // LAXF: 1/2 (F_L + F_R - c (U_R - U_L))
    R cg = cmaxg > cming ? cmaxg : cming, cr = cmaxr > cminr ? cmaxr : cminr;
    fLg = fRg = fLr = fRr = R(0.5);
    uLg = R(0.5) * cg;
    uRg = -uLg;
    uLr = R(0.5) * cr;
    uRr = -uLr;
  } else {  // HLL: (c- F_R + c+ F_L - c- c+ (U_R - U_L)) / (c- + c+)
    R sg = cmaxg + cming, sr = cmaxr + cminr;
    if (sg > R(0)) {
      R isg = R(1) / sg;
      fLg = cmaxg * isg;
      fRg = cming * isg;
      uLg = cming * cmaxg * isg;
      uRg = -uLg;
    } else {
      fLg = fRg = R(0.5);
      uLg = uRg = R(0);
    }
    if (sr > R(0)) {
      R isr = R(1) / sr;
      fLr = cmaxr * isr;
      fRr = cminr * isr;
      uLr = cminr * cmaxr * isr;
      uRr = -uLr;
    } else {
      fLr = fRr = R(0.5);
      uLr = uRr = R(0);
    }
  }
#pragma unroll
  for (int q = 0; q < NPR; ++q) out[q] = R(0);
  if (fs) *fs = R(0);
  face_accum<MET, R>(p, g, d + 1, PL, fLg, uLg, fLr, uLr, out, fs, lL);
  face_accum<MET, R>(p, g, d + 1, PR, fRg, uRg, fRr, uRr, out, fs, lR);
  out[B1 + d] = R(0);
  *smax = fmax(fmax(cmaxg, cming), fmax(cmaxr, cminr));
  if (gas) {
    gas[0] = cmaxg;
    gas[1] = cming;
  }
}

// ----------------------------------------------------------------- fluxes
// One thread per face of direction d (faces 0..n_d, transverse range widened
// by one layer for the EMF averages).  Reads the two reconstructed states
// (upper edge of cell f-1, lower edge of cell f), evaluates the metric at the
// face in registers, the gas and radiation signal speeds of both states and
// the HLL or LAXF flux (Eqs. hll, lax), gas and radiation groups with their own
// speeds.  The direction is a template parameter so that every index into a
// 4-vector or the primitive array is resolved at compile time.
// FP32 fluxes of one direction (split precision).
template <int MET, int d>
__global__ void __launch_bounds__(128) k_face32(DevParams p, const BoxGeo* __restrict__ boxes, int nbox,
                                                const float* __restrict__ E0, const double* __restrict__ K0,
                                                float* __restrict__ F0, float* __restrict__ spd0,
                                                float* __restrict__ FS0, float* __restrict__ gsp0) {
  typedef float R;
  const bool weighted = (MET == KS) && (d != 1);
  for (int bi = 0; bi < nbox; ++bi) {
    const BoxGeo& bx = boxes[bi];
    const R* E = E0 + 24 * bx.coff;
    const double* K = K0 + bx.coff;
    R* F = F0 + 12 * bx.coff;
    R* spd = spd0 + bx.coff;
    R* FS = FS0 ? FS0 + bx.coff : nullptr;
    R* gsp = gsp0 ? gsp0 + 2 * bx.coff : nullptr;  // gas v_max, v_min per face (staggered field)
    int len[3], off[3];
    for (int e = 0; e < 3; ++e) {
      if (e == d) {
        len[e] = bx.n[e] + 1;
        off[e] = 0;
      } else if (bx.n[e] > 1) {
        len[e] = bx.n[e] + 2;
        off[e] = -1;
      } else {
        len[e] = 1;
        off[e] = 0;
      }
    }
    long long total = (long long)len[0] * len[1] * len[2];
    const long long st = bx.str[d];
    const R dxd = R(bx.dx[d]);
    for (long long id = HR_TID; id < total; id += HR_STRIDE) {
      long long r = id;
      int ii[3];
      ii[0] = (int)(r % len[0]) + off[0];
      r /= len[0];
      ii[1] = (int)(r % len[1]) + off[1];
      ii[2] = (int)(r / len[1]) + off[2];
      long long t = cell_index(bx, ii[0], ii[1], ii[2]);
      const int f = ii[d];
      if (MET == KS && d == 1 && ((f == 0 && bx.bc[2] == 2) || (f == bx.n[1] && bx.bc[3] == 2))) {
#pragma unroll
        for (int q = 0; q < NPR; ++q) F[q * bx.ntot + t] = R(0);
        spd[t] = R(0);
        if (FS) FS[t] = R(0);
        if (gsp) gsp[t] = gsp[bx.ntot + t] = R(0);
        continue;
      }
      Geo<MET, R> g;
      R igf = R(1);
      R xf[3];
      for (int e = 0; e < 3; ++e) xf[e] = R(bx.x0[e] + (ii[e] + (e == d ? 0.0 : 0.5)) * bx.dx[e]);
      g = make_geo<MET, R>(p, xf[0], xf[1]);
      igf = weighted ? R(1) / g.gdet : R(1);
      R PL[NPR], PR[NPR];
#pragma unroll
      for (int q = 0; q < NPR; ++q) {
        const bool wq = weighted && ((q >= U1 && q <= B3) || q >= UR1);
        R aR, bL;  // upper edge of cell f-1, lower edge of cell f
        aR = E[(NPR + q) * bx.ntot + t - st];
        bL = E[q * bx.ntot + t];
        PL[q] = wq ? aR * igf : aR;
        PR[q] = wq ? bL * igf : bL;
      }
      const R kL = R(kfield(p, K, t - st)), kR = R(kfield(p, K, t));
      R out[NPR], smax;
      unsigned fcode = 0;
      R fsv, gs[2];
      face_flux<MET, R, d>(p, g, dxd, kL, kR, R(p.kscale), PL, PR, out, &smax, p.sig ? &fcode : nullptr,
                           FS ? &fsv : nullptr, gs);
      if (p.sig) sig_put(p, bx.coff + t, 40 + d, fcode);
      if (FS) FS[t] = fsv;
      if (gsp) {
        gsp[t] = gs[0];
        gsp[bx.ntot + t] = gs[1];
      }
#pragma unroll
      for (int q = 0; q < NPR; ++q) F[q * bx.ntot + t] = out[q];
      spd[t] = smax;
    }
  }
}

template <int MET, int d>
__device__ __forceinline__ void face_dir(const DevParams& p, const BoxGeo* __restrict__ boxes, int nbox, EdgeSet E0,
                                         const double* __restrict__ K0, double* __restrict__ F0,
                                         double* __restrict__ spd0, const double* __restrict__ geo0,
                                         double* __restrict__ FS0, double* __restrict__ gsp0) {
  const bool weighted = (MET == KS) && (d != 1);
  long long done = 0;
  for (int bi = 0; bi < nbox; ++bi) {
    const BoxGeo& bx = boxes[bi];
    const EdgeSet E = E0.box(bx);
    const double* K = K0 + bx.coff;
    double* F = F0 + 12 * bx.coff;
    double* spd = spd0 + bx.coff;
    double* FS = FS0 ? FS0 + bx.coff : nullptr;
    double* gsp = gsp0 ? gsp0 + 2 * bx.coff : nullptr;  // gas v_max, v_min per face (staggered field)
    int len[3], off[3];
    for (int e = 0; e < 3; ++e) {
      if (e == d) {
        len[e] = bx.n[e] + 1;
        off[e] = 0;
      } else if (bx.n[e] > 1) {
        len[e] = bx.n[e] + 2;
        off[e] = -1;
      } else {
        len[e] = 1;
        off[e] = 0;
      }
    }
    long long total = (long long)len[0] * len[1] * len[2];
    const long long st = bx.str[d];
    const double dxd = bx.dx[d];
    for (long long id = first_item(done); id < total; id += HR_STRIDE) {
      long long r = id;
      int ii[3];
      ii[0] = (int)(r % len[0]) + off[0];
      r /= len[0];
      ii[1] = (int)(r % len[1]) + off[1];
      ii[2] = (int)(r / len[1]) + off[2];
      long long t = cell_index(bx, ii[0], ii[1], ii[2]);
      const int f = ii[d];
      if (MET == KS && d == 1 && ((f == 0 && bx.bc[2] == 2) || (f == bx.n[1] && bx.bc[3] == 2))) {
#pragma unroll
        for (int q = 0; q < NPR; ++q) F[q * bx.ntot + t] = 0.0;
        spd[t] = 0.0;
        if (FS) FS[t] = 0.0;
        if (gsp) gsp[t] = gsp[bx.ntot + t] = 0.0;
        continue;
      }
      Geo<MET, double> g;
      double igf = 1.0, dl = dxd;  // 1/sqrt(-g) and the cell's proper length along d
      if constexpr (MET == KS) {
        const GeoTab T = geotab(geo0, bx);
        const double* tab = d == 0 ? T.F0 : (d == 1 ? T.F1 : T.C);
        const long long sz = d == 0 ? T.sF0 : (d == 1 ? T.sF1 : T.sC);
        const long long x = d == 0 ? gidx_f0(bx, ii[0], ii[1])
                                   : (d == 1 ? gidx_f1(bx, ii[0], ii[1]) : gidx_c(bx, ii[0], ii[1]));
        g = geo_load<MET>(tab, sz, x);
        if (weighted) igf = __ldg(tab + 16 * sz + x);
        dl = dxd * __ldg(tab + (d == 2 ? 19 : 17) * sz + x);
      } else {
        g = make_geo<MET, double>(p, 0.0, 0.0);
      }
      double PL[NPR], PR[NPR];
#pragma unroll
      for (int q = 0; q < NPR; ++q) {
        const bool wq = weighted && ((q >= U1 && q <= B3) || q >= UR1);
        const double aR = E.plane(1, q, bx.ntot)[t - st];  // upper edge of cell f-1
        const double bL = E.plane(0, q, bx.ntot)[t];       // lower edge of cell f
        PL[q] = wq ? aR * igf : aR;
        PR[q] = wq ? bL * igf : bL;
      }
      const double kL = kfield(p, K, t - st), kR = kfield(p, K, t);
      double out[NPR], smax;
      unsigned fcode = 0;
      double fsv, gs[2];
      face_flux64<MET, d + 1>(p, g, dl, kL, kR, PL, PR, out, &smax, p.sig ? &fcode : nullptr, FS ? &fsv : nullptr,
                              gsp ? gs : nullptr);
      if (p.sig) sig_put(p, bx.coff + t, 40 + d, fcode);
      if (FS) FS[t] = fsv;
      if (gsp) {
        gsp[t] = gs[0];
        gsp[bx.ntot + t] = gs[1];
      }
#pragma unroll
      for (int q = 0; q < NPR; ++q) F[q * bx.ntot + t] = out[q];
      spd[t] = smax;
    }
    done += total;
  }
}

// FP64: one launch per direction for the grids that fill the GPU.
template <int MET, int d>
__global__ void __launch_bounds__(128) k_face(DevParams p, const BoxGeo* __restrict__ boxes, int nbox, EdgeSet E0,
                                              const double* __restrict__ K0, double* __restrict__ F0,
                                              double* __restrict__ spd0, const double* __restrict__ geo0,
                                              double* __restrict__ FS0, double* __restrict__ gsp0) {
  face_dir<MET, d>(p, boxes, nbox, E0, K0, F0, spd0, geo0, FS0, gsp0);
}
// One launch for the directions d0 + blockIdx.y, as k_recon_all (64x32x16 per RK3
// step 0.35 -> 0.27 ms; grids that fill the GPU gain nothing).  gsp: gas v_max,
// v_min per face (staggered field; null otherwise).
struct FaceArgs {
  EdgeSets E;
  double* F[3];
  double* spd[3];
  double* FS[3];
  double* gsp[3];
};
template <int MET>
__global__ void __launch_bounds__(128) k_face_all(DevParams p, const BoxGeo* __restrict__ boxes, int nbox,
                                                  const double* __restrict__ K0, const double* __restrict__ geo0,
                                                  FaceArgs a, int d0) {
  const int d = d0 + blockIdx.y;
  if (!p.act[d]) return;
  if (d == 0) face_dir<MET, 0>(p, boxes, nbox, a.E.d[0], K0, a.F[0], a.spd[0], geo0, a.FS[0], a.gsp[0]);
  else if (d == 1) face_dir<MET, 1>(p, boxes, nbox, a.E.d[1], K0, a.F[1], a.spd[1], geo0, a.FS[1], a.gsp[1]);
  else face_dir<MET, 2>(p, boxes, nbox, a.E.d[2], K0, a.F[2], a.spd[2], geo0, a.FS[2], a.gsp[2]);
}

// ----------------------------------------------------------------- flux-CT
// Toth (2000) constrained transport for the pair (a, b) of active directions:
// edge EMF = 1/4 (F_a[B_b] + F_a[B_b](b-1) - F_b[B_a] - F_b[B_a](a-1)), zero on
// the polar axis; then F_a[B_b] and F_b[B_a] become averages of the two
// adjacent edge EMFs (with opposite signs).
// blockIdx.y = 0, 1, 2: the pairs (0, 1), (0, 2), (1, 2); emf1 holds one plane per
// pair, `planes` apart.
template <typename R>
struct FluxSet {
  R* f[3];
};
template <typename R>
__global__ void k_emf(DevParams p, const BoxGeo* __restrict__ boxes, int nbox, FluxSet<R> F, R* __restrict__ emf1,
                      long long planes) {
  const int a = blockIdx.y == 2 ? 1 : 0, b = blockIdx.y == 0 ? 1 : 2;
  if (!p.act[a] || !p.act[b]) return;
  const R* Fa0 = F.f[a];
  const R* Fb0 = F.f[b];
  R* emf0 = emf1 + blockIdx.y * planes;
  long long done = 0;
  for (int bi = 0; bi < nbox; ++bi) {
    const BoxGeo& bx = boxes[bi];
    const R* fab = Fa0 + 12 * bx.coff + (B1 + b) * bx.ntot;
    const R* fba = Fb0 + 12 * bx.coff + (B1 + a) * bx.ntot;
    R* emf = emf0 + bx.coff;
    int len[3];
    for (int e = 0; e < 3; ++e) len[e] = bx.n[e] + ((e == a || e == b) ? 1 : 0);
    long long total = (long long)len[0] * len[1] * len[2];
    const long long sa = bx.str[a], sb = bx.str[b];
    for (long long id = first_item(done); id < total; id += HR_STRIDE) {
      long long r = id;
      int ii[3];
      ii[0] = (int)(r % len[0]);
      r /= len[0];
      ii[1] = (int)(r % len[1]);
      ii[2] = (int)(r / len[1]);
      long long t = cell_index(bx, ii[0], ii[1], ii[2]);
      bool pole = p.metric == KS && (a == 1 || b == 1) &&
                  ((ii[1] == 0 && bx.bc[2] == 2) || (ii[1] == bx.n[1] && bx.bc[3] == 2));
      emf[t] = pole ? R(0) : R(0.25) * (fab[t] + fab[t - sb] - fba[t] - fba[t - sa]);
    }
    done += total;
  }
}

template <typename R>
__global__ void k_ct(DevParams p, const BoxGeo* __restrict__ boxes, int nbox, const R* __restrict__ emf1,
                     FluxSet<R> F, long long planes) {
  const int a = blockIdx.y == 2 ? 1 : 0, b = blockIdx.y == 0 ? 1 : 2;
  if (!p.act[a] || !p.act[b]) return;
  R* Fa0 = F.f[a];
  R* Fb0 = F.f[b];
  const R* emf0 = emf1 + blockIdx.y * planes;
  long long done = 0;
  for (int bi = 0; bi < nbox; ++bi) {
    const BoxGeo& bx = boxes[bi];
    R* fab = Fa0 + 12 * bx.coff + (B1 + b) * bx.ntot;
    R* fba = Fb0 + 12 * bx.coff + (B1 + a) * bx.ntot;
    const R* emf = emf0 + bx.coff;
    // two index spaces: a-faces (a in [0,n_a], b in [0,n_b)) then b-faces
    int la[3], lb[3];
    for (int e = 0; e < 3; ++e) {
      la[e] = bx.n[e] + (e == a ? 1 : 0);
      lb[e] = bx.n[e] + (e == b ? 1 : 0);
    }
    long long na = (long long)la[0] * la[1] * la[2];
    long long nb = (long long)lb[0] * lb[1] * lb[2];
    const long long sa = bx.str[a], sb = bx.str[b];
    for (long long id = first_item(done); id < na + nb; id += HR_STRIDE) {
      const int* L = id < na ? la : lb;
      long long r = id < na ? id : id - na;
      int i0 = (int)(r % L[0]);
      r /= L[0];
      int i1 = (int)(r % L[1]);
      int i2 = (int)(r / L[1]);
      long long t = cell_index(bx, i0, i1, i2);
      if (id < na) fab[t] = R(0.5) * (emf[t] + emf[t + sb]);
      else fba[t] = R(-0.5) * (emf[t] + emf[t + sa]);
    }
    done += na + nb;
  }
}

// ----------------------------------------------------------------- floors
// Lorentz-factor caps, density and internal-energy floors f0 r^pow,
// magnetisation caps b^2/rho, b^2/u_g, u_g/rho, and Ebar > 0.

// The floors f0 r^pow at x1 as f0 exp(pow ln r), with ln r = x1 itself when
// r = e^x1 (R0 = 0); on the Minkowski grid r = 1.
template <int MET>
__device__ __forceinline__ void floor_values(const DevParams& p, double x1, double* rfl, double* ufl) {
  double lr = 0.0;
  if constexpr (MET == KS) lr = p.R0 == 0.0 ? x1 : log(p.R0 + exp(x1));
  *rfl = p.rf0 * (p.rfp == 0.0 ? 1.0 : exp(p.rfp * lr));
  *ufl = p.uf0 * (p.ufp == 0.0 ? 1.0 : exp(p.ufp * lr));
}

// b^2 of u~^i and B^i by b^2 = (B^i B_i + (B^i u_i)^2) / (u^t)^2, and
// gamma^2 of u~^i; both in FP64 or on dual numbers.
template <int MET, typename T>
__device__ __forceinline__ T floor_bsq(const Geo<MET, T>& g, const T P[NPR], T* g2) {
  if constexpr (std::is_same<T, double>::value) {
    double l[3], m[3];
    lower3<MET>(g, P[U1], P[U2], P[U3], l);
    lower3<MET>(g, P[B1], P[B2], P[B3], m);
    *g2 = fma(P[U1], l[0], fma(P[U2], l[1], fma(P[U3], l[2], 1.0)));
    const double bt = fma(P[B1], l[0], fma(P[B2], l[1], P[B3] * l[2]));
    const double BB = fma(P[B1], m[0], fma(P[B2], m[1], P[B3] * m[2]));
    return fma(bt, bt, BB) * (MET == MINK ? rcp(*g2) : (g.alpha * g.alpha) * rcp(*g2));
  } else {
    T ucon[4], ucov[4], bcon[4], bcov[4], bsq, gm;
    fourvel<MET, T>(g, P[U1], P[U2], P[U3], ucon, ucov, &gm);
    bvec<MET, T>(g, ucon, ucov, P[B1], P[B2], P[B3], bcon, bcov, &bsq);
    *g2 = gm * gm;
    return bsq;
  }
}

template <int MET, typename T = double>
__device__ __forceinline__ void apply_floors(const DevParams& p, const Geo<MET, T>& g, double rf0, double uf0,
                                             T P[NPR], unsigned* code = nullptr) {
  T g2, bsq = floor_bsq<MET, T>(g, P, &g2);
  const T r2 = 1.0 + g.sq3(P[UR1], P[UR2], P[UR3]);
  const double gc = p.ggas_max * p.ggas_max, rc = p.grad_max * p.grad_max;
  if (code) *code = (g2 > gc ? 1u : 0u) | (r2 > rc ? 2u : 0u);  // which floors act (the branch signature)
  if (g2 > gc) {
    T f = sqrt((gc - 1.0) / (g2 - 1.0));
    P[U1] *= f;
    P[U2] *= f;
    P[U3] *= f;
    bsq = floor_bsq<MET, T>(g, P, &g2);
  }
  if (r2 > rc) {
    T f = sqrt((rc - 1.0) / (r2 - 1.0));
    P[UR1] *= f;
    P[UR2] *= f;
    P[UR3] *= f;
  }
  const T rb = bsq * p.ibsq_rho, ub = bsq * p.ibsq_u;
  const T rfl = fmax(T(rf0), rb), ufl = fmax(T(uf0), ub);
  if (code) {
    const T u1 = fmax(P[UU], ufl);
    *code |= (rb > rf0 ? 4u : 0u) | (ub > uf0 ? 8u : 0u) | (rfl > P[RHO] ? 16u : 0u) | (ufl > P[UU] ? 32u : 0u) |
             (u1 * p.iu_rho > fmax(P[RHO], rfl) ? 64u : 0u) | (!(P[ER] > 0.0) ? 128u : 0u);
  }
  P[RHO] = fmax(P[RHO], rfl);
  P[UU] = fmax(P[UU], ufl);
  P[RHO] = fmax(P[RHO], P[UU] * p.iu_rho);
  if (!(P[ER] > 0.0)) P[ER] = T(1e-150);
}

// Final primitives of an accepted PMHD iterate: gas from x, B fixed, radiation
// re-inverted with BASIC if the TYPE2 branch saw a negative energy (Sec. 4.10).
// Final primitives from the error function's state at x (pmhd_res), without
// evaluating it again: gas from x, B fixed, radiation re-inverted with BASIC
// if the TYPE2 branch saw a negative energy (Sec. 4.10).
template <int MET, bool FAST>
__device__ __forceinline__ void pmhd_final_state(const DevParams& p, const ImpSys<MET, FAST>& s, const double x[4],
                                                 const ImpState& st, double P[NPR]) {
  P[RHO] = st.rho;
  P[UU] = x[0];
  P[U1] = x[1];
  P[U2] = x[2];
  P[U3] = x[3];
  P[B1] = s.B[0];
  P[B2] = s.B[1];
  P[B3] = s.B[2];
  double Pr[4] = {st.Pr[0], st.Pr[1], st.Pr[2], st.Pr[3]};
  if (st.negE) rad_invert<MET, double>(p, s.g, st.Rt_pre, 0, Pr);
  P[ER] = Pr[0];
  P[UR1] = Pr[1];
  P[UR2] = Pr[2];
  P[UR3] = Pr[3];
}

template <int MET, typename T = double, bool FAST>
__device__ __forceinline__ void pmhd_final(const DevParams& p, const ImpSysT<MET, T, FAST>& s, const T x[4], T P[NPR],
                                           T* Eg = nullptr, unsigned* code = nullptr) {
  ImpResT<T> r;
  ImpStateT<T> stt;
  pmhd_res<MET, T>(p, s, x, r, &stt, false);
  if (code) {  // the TYPE2 limiter's branch at the solution (the branch signature)
    T Prt[4];
    int lim = 0;
    rad_invert<MET, T>(p, s.g, stt.Rt_pre, 2, Prt, &lim);
    *code = (unsigned)r.negE | (unsigned)lim << 1;
  }
  if (Eg)
    for (int k = 0; k < 4; ++k) Eg[k] = r.Eg[k];
  P[RHO] = stt.rho;
  P[UU] = x[0];
  P[U1] = x[1];
  P[U2] = x[2];
  P[U3] = x[3];
  P[B1] = s.B[0];
  P[B2] = s.B[1];
  P[B3] = s.B[2];
  T Pr[4] = {stt.Pr[0], stt.Pr[1], stt.Pr[2], stt.Pr[3]};
  if (r.negE) rad_invert<MET, T>(p, s.g, stt.Rt_pre, 0, Pr);
  P[ER] = Pr[0];
  P[UR1] = Pr[1];
  P[UR2] = Pr[2];
  P[UR3] = Pr[3];
}

// Optical depth of a cell along its longest active proper edge, from the
// primitives P (the tau < 2/3 guess rules of Sec. 4.10).
template <int MET>
__device__ __forceinline__ double zone_tau(const DevParams& p, const Geo<MET, double>& g, const double dx[3],
                                           const double P[NPR], double kf) {
  double kabs, ksca;
  opacity<double>(p, P[RHO], P[UU], kf, &kabs, &ksca);
  double dl = 0.0;
#pragma unroll
  for (int d = 1; d <= 3; ++d)
    if (p.act[d - 1]) dl = fmax(dl, sqrt(g.gdd(d)) * dx[d - 1]);
  return (kabs + ksca) * dl;
}

// The retry methods after PMHD (Sec. 4.10-4.11).  URAD from the PMHD iterate
// where its e_T < 1e-4, else from P_s; then PRAD if neither reached 1e-9,
// guessed from the better earlier solution where its e_T < 1e-4, else from
// the optically thin limit (the M1 inversion of R*, no source) where
// tau < 2/3, else from P_s.  The lowest-error solution wins (the earlier
// method on ties); its primitives before the floors go to Pn.  px / peT: the
// PMHD iterate and its error (inf if none).  Returns the outcome: ST_PMHD,
// ST_URAD (URAD or PRAD), or ST_BACKUP when no residual was finite or the
// best e_T exceeds 1e-7; *eT_out its error, *steps_out the Newton steps.
template <int MET, bool FAST>
__device__ int retry_sequence(const DevParams& p, const Geo<MET, double>& g, const ImpSys<MET, FAST>& s,
                              const double Ps[NPR], const double px[4], double peT, double tau, double Pn[NPR],
                              double* eT_out, int* steps_out, bool subdom = false, double Sst = NAN) {
  const bool pfin = isfinite(peT);
  double Pb[NPR];
  if (pfin) {  // the PMHD iterate as its error function left it (TYPE2 radiation)
    ImpRes rr;
    ImpState stt;
    pmhd_res<MET>(p, s, px, rr, &stt, false);
    Pb[RHO] = stt.rho;
    Pb[UU] = px[0];
    Pb[U1] = px[1];
    Pb[U2] = px[2];
    Pb[U3] = px[3];
    Pb[B1] = s.B[0];
    Pb[B2] = s.B[1];
    Pb[B3] = s.B[2];
    for (int q = 0; q < 4; ++q) Pb[ER + q] = stt.Pr[q];
  }
  const double* Pg = (pfin && peT < 1e-4) ? Pb : Ps;
  double urc[4], urv[4], gr;
  fourvel<MET, double>(g, Pg[UR1], Pg[UR2], Pg[UR3], urc, urv, &gr);
  const double e43 = (4.0 / 3.0) * Pg[ER];
  double xr[4];
  xr[0] = e43 * urc[0] * urv[0] + Pg[ER] * (1.0 / 3.0);
  for (int n = 1; n < 4; ++n) xr[n] = e43 * urc[0] * urv[n];
  double gas[5] = {Pg[RHO], Pg[UU], Pg[U1], Pg[U2], Pg[U3]};
  double ux[4], ugas[5], ueT;
  int steps = newton_urad<MET>(p, s, xr, gas, ux, ugas, &ueT);
  int best = pfin ? 0 : -1;
  double beT = pfin ? peT : HUGE_VAL;
  if (isfinite(ueT) && (best < 0 || ueT < beT)) {
    best = 1;
    beT = ueT;
  }
  double qx[4], qgas[5], qeT = HUGE_VAL;
  if (!(beT < 1e-9)) {
    double xq[4], gq[5];
    if (best >= 0 && beT < 1e-4) {
      if (best == 0) {
        for (int q = 0; q < 4; ++q) xq[q] = Pb[ER + q];
        for (int q = 0; q < 5; ++q) gq[q] = Pb[q];
      } else {
        rad_invert<MET>(p, g, ux, 2, xq);
        for (int q = 0; q < 5; ++q) gq[q] = ugas[q];
      }
    } else {
      if (tau < 2.0 / 3.0) {
        rad_invert<MET>(p, g, s.Rs, 2, xq);
      } else {
        for (int q = 0; q < 4; ++q) xq[q] = Ps[ER + q];
      }
      for (int q = 0; q < 5; ++q) gq[q] = Ps[q];
    }
    steps += newton_rad<MET, true>(p, s, xq, gq, qx, qgas, &qeT);
    if (isfinite(qeT) && (best < 0 || qeT < beT)) {
      best = 2;
      beT = qeT;
    }
  }
  double sx[4];
  if (subdom && !(beT < 1e-9)) {
    // staged PMHD (Sec. 4.10): guessed from the gas of the best earlier
    // solution if its e_T < 1e-4 (else P_s), u_g from the specific entropy
    // S* / (rho0 u^t)* at the density of P_s where S* is given
    const double* gsrc = Ps;
    if (best >= 0 && beT < 1e-4) gsrc = best == 0 ? Pb : (best == 1 ? ugas : qgas);
    double xs[4] = {gsrc[UU], gsrc[U1], gsrc[U2], gsrc[U3]};
    entropy_ug_guess(p, Sst, s.Dlab * g.gdet, Ps[RHO], xs);
    double seT;
    steps += newton_pmhd_staged<MET>(p, s, xs, sx, &seT);
    if (isfinite(seT) && (best < 0 || seT < beT)) {
      best = 3;
      beT = seT;
    }
  }
  // then the staged URAD and PRAD, each from the primitives of the
  // lowest-error solution so far if its e_T < 1e-4 (as its error function
  // formed them), else from P_s
  double tx[2][4], tgas[2][5];
#pragma unroll 1
  for (int pr = 0; pr < 2 && subdom && !(beT < 1e-9); ++pr) {
    double Pq[NPR];
    for (int q = 0; q < NPR; ++q) Pq[q] = Ps[q];
    if (best >= 0 && beT < 1e-4) {
      if (best == 0 || best == 3) {
        ImpRes rr;
        ImpState stt;
        const double* bx = best == 0 ? px : sx;
        pmhd_res<MET>(p, s, bx, rr, &stt, false);
        Pq[RHO] = stt.rho;
        for (int c = 0; c < 4; ++c) Pq[UU + c] = bx[c];
        for (int c = 0; c < 4; ++c) Pq[ER + c] = stt.Pr[c];
      } else if (best == 1 || best == 4) {
        const double* gg = best == 1 ? ugas : tgas[0];
        for (int c = 0; c < 5; ++c) Pq[c] = gg[c];
        rad_invert<MET>(p, g, best == 1 ? ux : tx[0], 2, Pq + ER);
      } else {
        const double* gg = best == 2 ? qgas : tgas[1];
        const double* xx = best == 2 ? qx : tx[1];
        for (int c = 0; c < 5; ++c) Pq[c] = gg[c];
        for (int c = 0; c < 4; ++c) Pq[ER + c] = xx[c];
      }
    }
    double gq[5] = {Pq[RHO], Pq[UU], Pq[U1], Pq[U2], Pq[U3]}, x4[4], reT;
    if (pr == 1) {
      for (int c = 0; c < 4; ++c) x4[c] = Pq[ER + c];
      steps += newton_rad_staged<MET, true>(p, s, x4, gq, tx[1], tgas[1], &reT);
    } else {
      double urc2[4], urv2[4], gr2;
      fourvel<MET, double>(g, Pq[UR1], Pq[UR2], Pq[UR3], urc2, urv2, &gr2);
      const double e43q = (4.0 / 3.0) * Pq[ER];
      x4[0] = e43q * urc2[0] * urv2[0] + Pq[ER] * (1.0 / 3.0);
      for (int c = 1; c < 4; ++c) x4[c] = e43q * urc2[0] * urv2[c];
      steps += newton_rad_staged<MET, false>(p, s, x4, gq, tx[0], tgas[0], &reT);
    }
    if (isfinite(reT) && (best < 0 || reT < beT)) {
      best = 4 + pr;
      beT = reT;
    }
  }
  int method = ST_URAD;
  if (best == 0) {
    pmhd_final<MET>(p, s, px, Pn);
    method = ST_PMHD;
  } else if (best == 1) {
    for (int q = 0; q < 5; ++q) Pn[q] = ugas[q];
    double Pr[4];
    if (rad_invert<MET>(p, g, ux, 2, Pr)) rad_invert<MET>(p, g, ux, 0, Pr);
    for (int q = 0; q < 4; ++q) Pn[ER + q] = Pr[q];
  } else if (best == 2) {
    for (int q = 0; q < 5; ++q) Pn[q] = qgas[q];
    for (int q = 0; q < 4; ++q) Pn[ER + q] = qx[q];
  } else if (best == 3) {
    pmhd_final<MET>(p, s, sx, Pn);
  } else if (best == 4) {
    for (int q = 0; q < 5; ++q) Pn[q] = tgas[0][q];
    double Pr[4];
    if (rad_invert<MET>(p, g, tx[0], 2, Pr)) rad_invert<MET>(p, g, tx[0], 0, Pr);
    for (int q = 0; q < 4; ++q) Pn[ER + q] = Pr[q];
  } else if (best == 5) {
    for (int q = 0; q < 5; ++q) Pn[q] = tgas[1][q];
    for (int q = 0; q < 4; ++q) Pn[ER + q] = tx[1][q];
  } else {
    for (int q = 0; q < NPR; ++q) Pn[q] = Ps[q];
    method = ST_BACKUP;
    beT = HUGE_VAL;
  }
  Pn[B1] = s.B[0];
  Pn[B2] = s.B[1];
  Pn[B3] = s.B[2];
  if (beT > 1e-7) method = ST_BACKUP;
  *eT_out = beT;
  *steps_out = steps;
  return method;
}

// Metric derivatives for the geometric source: forward-mode pair (d/dx1, d/dx2).
struct D2 {
  double v, a, b;
};
__device__ __forceinline__ D2 operator+(D2 x, D2 y) { return {x.v + y.v, x.a + y.a, x.b + y.b}; }
__device__ __forceinline__ D2 operator-(D2 x, D2 y) { return {x.v - y.v, x.a - y.a, x.b - y.b}; }
__device__ __forceinline__ D2 operator*(D2 x, D2 y) {
  return {x.v * y.v, x.a * y.v + x.v * y.a, x.b * y.v + x.v * y.b};
}
__device__ __forceinline__ D2 operator*(double c, D2 y) { return {c * y.v, c * y.a, c * y.b}; }
__device__ __forceinline__ D2 operator/(D2 x, D2 y) {
  double iy = 1.0 / y.v;
  double q = x.v * iy;
  return {q, (x.a - q * y.a) * iy, (x.b - q * y.b) * iy};
}

// d_nu g_{mu kappa} (nu = x1, x2) of the covariant Kerr-Schild metric in the
// internal chart and d_nu sqrt(-g).
struct MetricDeriv {
  double g00[2], g01[2], g03[2], g11[2], g13[2], g22[2], g33[2], sg[2];
};
__device__ __forceinline__ MetricDeriv ks_derivs(const DevParams& p, double x1, double x2) {
  const double a = p.a, hh = p.h, pi = 3.14159265358979323846;
  double ex = exp(x1);
  D2 r = {p.R0 + ex, ex, 0.0};
  double s2x, c2x;
  sincospi(2.0 * x2, &s2x, &c2x);
  D2 th = {pi * x2 + 0.5 * (1.0 - hh) * s2x, 0.0, pi + (1.0 - hh) * pi * c2x};
  double st, ct;
  sincos(th.v, &st, &ct);
  D2 sth = {st, 0.0, ct * th.b}, cth = {ct, 0.0, -st * th.b};
  D2 J1 = {ex, ex, 0.0};
  D2 J2 = {pi * (1.0 + (1.0 - hh) * c2x), 0.0, -2.0 * pi * pi * (1.0 - hh) * s2x};
  const double J3 = 2.0 * pi;
  D2 s2 = sth * sth;
  D2 S = r * r + (a * a) * (cth * cth);
  D2 tr = (2.0 * r) / S;
  D2 one = {1.0, 0.0, 0.0};
  D2 m00 = tr - one;
  D2 m01 = tr * J1;
  D2 m03 = (-a * J3) * (tr * s2);
  D2 m11 = (one + tr) * J1 * J1;
  D2 m13 = (-a * J3) * (s2 * (one + tr) * J1);
  D2 m22 = S * J2 * J2;
  D2 m33 = (J3 * J3) * (s2 * (S + (a * a) * (s2 * (one + tr))));
  D2 sg = J3 * (S * sth * J1 * J2);
  MetricDeriv md;
  md.g00[0] = m00.a; md.g00[1] = m00.b;
  md.g01[0] = m01.a; md.g01[1] = m01.b;
  md.g03[0] = m03.a; md.g03[1] = m03.b;
  md.g11[0] = m11.a; md.g11[1] = m11.b;
  md.g13[0] = m13.a; md.g13[1] = m13.b;
  md.g22[0] = m22.a; md.g22[1] = m22.b;
  md.g33[0] = m33.a; md.g33[1] = m33.b;
  md.sg[0] = sg.a; md.sg[1] = sg.b;
  return md;
}

// v^mu v^kappa d_nu g_{mu kappa}
template <typename T>
__device__ __forceinline__ T qform(const MetricDeriv& m, int n, const T v[4]) {
  return m.g00[n] * v[0] * v[0] + 2.0 * m.g01[n] * v[0] * v[1] + 2.0 * m.g03[n] * v[0] * v[3] +
         m.g11[n] * v[1] * v[1] + 2.0 * m.g13[n] * v[1] * v[3] + m.g22[n] * v[2] * v[2] +
         m.g33[n] * v[3] * v[3];
}

__device__ __forceinline__ MetricDeriv md_load(const double* __restrict__ t, long long s, long long x) {
  MetricDeriv m;
  double* v = reinterpret_cast<double*>(&m);  // the 16 doubles of MetricDeriv, in declaration order
  for (int f = 0; f < 16; ++f) v[f] = __ldg(t + f * s + x);
  return m;
}

// Fills the metric tables of the Kerr-Schild grids of a context.
static __global__ void k_geo_init(DevParams p, const BoxGeo* __restrict__ boxes, int nbox, double* geo0) {
  for (int bi = 0; bi < nbox; ++bi) {
    const BoxGeo& bx = boxes[bi];
    if (bx.goff < 0) continue;
    const GeoTab T = geotab(geo0, bx);
    double* C = const_cast<double*>(T.C);
    double* M = const_cast<double*>(T.M);
    double* F0 = const_cast<double*>(T.F0);
    double* F1 = const_cast<double*>(T.F1);
    double* Ed = const_cast<double*>(T.E);
    const long long total = T.sC + T.sF0 + T.sF1 + (long long)(bx.n[0] + 1) * (bx.n[1] + 1);
    for (long long id = HR_TID; id < total; id += HR_STRIDE) {
      if (id < T.sC) {  // centres and their derivatives
        const int i = (int)(id % bx.N[0]) - bx.ng[0], j = (int)(id / bx.N[0]) - bx.ng[1];
        const double x1 = xcen(bx, 0, i), x2 = xcen(bx, 1, j);
        const Geo<KS, double> g = make_geo<KS, double>(p, x1, x2);
        geo_store<KS>(C, T.sC, id, g);
        C[16 * T.sC + id] = 1.0 / g.gdet;
        C[17 * T.sC + id] = sqrt(g.g11);
        C[18 * T.sC + id] = sqrt(g.g22);
        C[19 * T.sC + id] = sqrt(g.g33);
        double dl = 0.0;
        for (int k = 1; k < 4; ++k) {
          C[(19 + k) * T.sC + id] = sqrt(g.Gdd(k) - g.Gt(k) * g.Gt(k) / g.Gtt());
          if (p.act[k - 1]) dl = fmax(dl, sqrt(g.gdd(k)) * bx.dx[k - 1]);
        }
        floor_values<KS>(p, x1, &C[23 * T.sC + id], &C[24 * T.sC + id]);
        C[25 * T.sC + id] = dl;
        const MetricDeriv md = ks_derivs(p, x1, x2);
        const double* v = reinterpret_cast<const double*>(&md);
        for (int f = 0; f < 16; ++f) {
          const int c = f / 2;  // g00 g01 g03 g11 g13 g22 g33 sg, two derivatives each
          const double w = c == 7 || p.precision ? 1.0 : (c == 1 || c == 2 || c == 4 ? g.gdet : 0.5 * g.gdet);
          M[f * T.sC + id] = w * v[f];
        }
      } else if (id < T.sC + T.sF0) {  // x1 faces
        const long long e = id - T.sC;
        const int i = (int)(e % (bx.n[0] + 1)), j = (int)(e / (bx.n[0] + 1)) - bx.ng[1];
        const double x1 = bx.x0[0] + (i + 0.0) * bx.dx[0], x2 = bx.x0[1] + (j + 0.5) * bx.dx[1];
        const Geo<KS, double> g = make_geo<KS, double>(p, x1, x2);
        geo_store<KS>(F0, T.sF0, e, g);
        F0[16 * T.sF0 + e] = 1.0 / g.gdet;
        F0[17 * T.sF0 + e] = sqrt(g.g11);
      } else if (id < T.sC + T.sF0 + T.sF1) {  // x2 faces
        const long long e = id - T.sC - T.sF0;
        const int i = (int)(e % bx.N[0]) - bx.ng[0], j = (int)(e / bx.N[0]);
        const double x1 = bx.x0[0] + (i + 0.5) * bx.dx[0], x2 = bx.x0[1] + (j + 0.0) * bx.dx[1];
        const Geo<KS, double> g = make_geo<KS, double>(p, x1, x2);
        geo_store<KS>(F1, T.sF1, e, g);
        F1[16 * T.sF1 + e] = 1.0 / g.gdet;
        F1[17 * T.sF1 + e] = sqrt(g.g22);
      } else {  // x1-x2 edges
        const long long e = id - T.sC - T.sF0 - T.sF1;
        const int i = (int)(e % (bx.n[0] + 1)), j = (int)(e / (bx.n[0] + 1));
        Ed[e] = make_geo<KS, double>(p, bx.x0[0] + i * bx.dx[0], bx.x0[1] + j * bx.dx[1]).gdet;
      }
    }
  }
}

// U(P) and the geometric source SM(P) of one zone (X = SM on return):
// SM_nu = 1/2 sqrt(-g) T^{mu kappa} d_nu g_{mu kappa}, equal to
// sqrt(-g) T^kappa_lambda Gamma^lambda_{nu kappa} for a symmetric T and nonzero
// only for nu = x1, x2 on the stationary axisymmetric metric.
template <int MET, typename T>
__device__ __forceinline__ void cons_source(const DevParams& p, const Geo<MET, T>& g, double x1, double x2,
                                            const T Ps[NPR], T Us[NPR], T X[NPR],
                                            const MetricDeriv* mdp = nullptr) {
  T ucon[4], ucov[4], gm, bcon[4], bcov[4], bsq, urc[4], urv[4], gr;
  fourvel<MET, T>(g, Ps[U1], Ps[U2], Ps[U3], ucon, ucov, &gm);
  bvec<MET, T>(g, ucon, ucov, Ps[B1], Ps[B2], Ps[B3], bcon, bcov, &bsq);
  fourvel<MET, T>(g, Ps[UR1], Ps[UR2], Ps[UR3], urc, urv, &gr);
  const T pg = (p.gam - 1.0) * Ps[UU];
  const T wb = Ps[RHO] + Ps[UU] + pg + bsq, pt = pg + 0.5 * bsq;
  const T gd = g.gdet, mt = Ps[RHO] * ucon[0];
  const T E = Ps[ER], e43 = (4.0 / 3.0) * E;
  Us[0] = gd * mt;
  Us[1] = gd * (wb * ucon[0] * ucov[0] + pt - bcon[0] * bcov[0] + mt);
#pragma unroll
  for (int n = 1; n < 4; ++n) Us[1 + n] = gd * (wb * ucon[0] * ucov[n] - bcon[0] * bcov[n]);
  Us[5] = gd * Ps[B1];
  Us[6] = gd * Ps[B2];
  Us[7] = gd * Ps[B3];
  Us[8] = gd * (e43 * urc[0] * urv[0] + E * (1.0 / 3.0));
#pragma unroll
  for (int n = 1; n < 4; ++n) Us[8 + n] = gd * (e43 * urc[0] * urv[n]);
#pragma unroll
  for (int q = 0; q < NPR; ++q) X[q] = T(0.0);
  if constexpr (MET == KS) {
    const MetricDeriv md = mdp ? *mdp : ks_derivs(p, x1, x2);
#pragma unroll
    for (int n = 0; n < 2; ++n) {
      T qu = qform(md, n, ucon), qb = qform(md, n, bcon), qr = qform(md, n, urc);
      X[2 + n] = 0.5 * gd * (wb * qu - qb) + pt * md.sg[n];
      X[9 + n] = 0.5 * gd * e43 * qr + E * (1.0 / 3.0) * md.sg[n];
    }
  }
  (void)x1;
  (void)x2;
}

// The same in FP64 with the metric derivatives of the table (md: 1/2 sqrt(-g)
// d_nu g_{mu kappa}, off-diagonals doubled): the source contracts T^{mu kappa}
// once per nu, and the rows of U take the two-scalar form of pmhd_res64.
template <int MET>
__device__ __forceinline__ void cons_source64(const DevParams& p, const Geo<MET, double>& g, const double Ps[NPR],
                                              double Us[NPR], double X[NPR], const MetricDeriv& md) {
  double l[3], m[3], k[3], igm;
  lower3<MET>(g, Ps[U1], Ps[U2], Ps[U3], l);
  lower3<MET>(g, Ps[B1], Ps[B2], Ps[B3], m);
  lower3<MET>(g, Ps[UR1], Ps[UR2], Ps[UR3], k);
  const double gm = sqrt_rsqrt(fma(Ps[U1], l[0], fma(Ps[U2], l[1], fma(Ps[U3], l[2], 1.0))), &igm);
  const double gr = sqrt64(fma(Ps[UR1], k[0], fma(Ps[UR2], k[1], fma(Ps[UR3], k[2], 1.0))));
  const double bt = fma(Ps[B1], l[0], fma(Ps[B2], l[1], Ps[B3] * l[2]));
  const double BB = fma(Ps[B1], m[0], fma(Ps[B2], m[1], Ps[B3] * m[2]));
  double u0 = gm, l0 = -gm, iut = igm, r0 = gr, k0 = -gr, m0 = 0.0, a01 = 0.0;
  if constexpr (MET == KS) {
    a01 = g.alpha * g.G01;
    const double b1 = g.alpha * a01;
    u0 = gm * g.ialpha;
    l0 = fma(b1, l[0], -g.alpha * gm);
    iut = g.alpha * igm;
    r0 = gr * g.ialpha;
    k0 = fma(b1, k[0], -g.alpha * gr);
    m0 = b1 * m[0];
  }
  const double bu = bt * iut, bsq = fma(bt, bt, BB) * (iut * iut);
  const double pg = p.gm1 * Ps[UU], wb = Ps[RHO] + fma(p.gam, Ps[UU], bsq), pt = fma(0.5, bsq, pg);
  const double wu = wb * u0, Z = fma(-bt, bu, wu), mt = Ps[RHO] * u0;
  const double E = Ps[ER], e43 = (4.0 / 3.0) * E, e13 = E * (1.0 / 3.0), er = e43 * r0, gd = g.gdet;
  Us[0] = gd * mt;
  Us[1] = gd * fma(Z, l0, fma(-bu, m0, pt + mt));
#pragma unroll
  for (int n = 0; n < 3; ++n) {
    Us[2 + n] = gd * fma(Z, l[n], -bu * m[n]);
    Us[5 + n] = gd * Ps[B1 + n];
    Us[9 + n] = gd * (er * k[n]);
  }
  Us[8] = gd * fma(er, k0, e13);
#pragma unroll
  for (int q = 0; q < NPR; ++q) X[q] = 0.0;
  if constexpr (MET == KS) {
    const double u1 = fma(-gm, a01, Ps[U1]), u2 = Ps[U2], u3 = Ps[U3];
    const double b1 = fma(bt, u1, Ps[B1]) * iut, b2 = fma(bt, u2, Ps[B2]) * iut, b3 = fma(bt, u3, Ps[B3]) * iut;
    const double w1 = wb * u1;
    const double T[7] = {fma(wu, u0, -bt * bt), fma(wu, u1, -bt * b1),      fma(wu, u3, -bt * b3),
                         fma(w1, u1, -b1 * b1), fma(w1, u3, -b1 * b3),      fma(wb * u2, u2, -b2 * b2),
                         fma(wb * u3, u3, -b3 * b3)};
    const double r1 = fma(-gr, a01, Ps[UR1]), r2 = Ps[UR2], r3 = Ps[UR3], e1 = e43 * r1;
    const double R[7] = {er * r0, er * r1, er * r3, e1 * r1, e1 * r3, e43 * r2 * r2, e43 * r3 * r3};
    const double* d = reinterpret_cast<const double*>(&md);
#pragma unroll
    for (int n = 0; n < 2; ++n) {
      double xg = pt * md.sg[n], xr = e13 * md.sg[n];
#pragma unroll
      for (int c = 0; c < 7; ++c) {
        xg = fma(T[c], d[2 * c + n], xg);
        xr = fma(R[c], d[2 * c + n], xr);
      }
      X[2 + n] = xg;
      X[9 + n] = xr;
    }
  }
}

constexpr int CSTRIDE = NPR + 23;  // continuation queue record: U*, Newton state, S*

__device__ __forceinline__ void newton_state_store(const NewtonState& st, double* d) {
  for (int i = 0; i < 4; ++i) {
    d[i] = st.x[i];
    d[4 + i] = st.best_x[i];
  }
  d[8] = st.best_eT;
  d[9] = st.hs.t1;
  d[10] = st.hs.t2;
  d[11] = st.hs.t3;
  d[12] = st.hs.t4;
  d[13] = st.hs.i1;
  d[14] = st.hs.i2;
  d[15] = st.hs.i3;
  d[16] = st.hs.i4;
  d[17] = st.eps;
  d[18] = (double)st.hs.rises;
  d[19] = (double)st.k;
  d[20] = (double)st.steps;
  d[21] = (double)st.jac32;
}

__device__ __forceinline__ void newton_state_load(const double* d, NewtonState& st) {
  for (int i = 0; i < 4; ++i) {
    st.x[i] = d[i];
    st.best_x[i] = d[4 + i];
  }
  st.best_eT = d[8];
  st.hs.t1 = d[9];
  st.hs.t2 = d[10];
  st.hs.t3 = d[11];
  st.hs.t4 = d[12];
  st.hs.i1 = d[13];
  st.hs.i2 = d[14];
  st.hs.i3 = d[15];
  st.hs.i4 = d[16];
  st.eps = d[17];
  st.hs.rises = (int)d[18];
  st.k = (int)d[19];
  st.steps = (int)d[20];
  st.jac32 = (int)d[21];
}

// End of a zone's PMHD solve: accept (e_T < 1e-9: final primitives, floors,
// write) or queue the zone for URAD.  Returns whether it was accepted.
template <int MET, bool FAST>
__device__ __forceinline__ bool pmhd_finish(const DevParams& p, const BoxGeo& bx, int bi, long long z, long long t,
                                            const double fl[2], const Geo<MET, double>& g, const ImpSys<MET, FAST>& s,
                                            const double Ust[NPR], double h, const double best_x[4],
                                            double beT, int steps, double* P, const Bufs& b, double Sst,
                                            double acc_tol = 1e-9, const ImpState* bst = nullptr) {
  const long long zg = bx.aoff + z;
  b.iters[zg] += steps;
  const bool accept = beT >= 0.0 && beT < acc_tol;  // beT < 0: sub-dominant radiation, URAD first
  if (accept) {
    double Pn[NPR];
    unsigned lcode = 0;
    if (bst && !p.sig)  // the state the Newton loop kept for its best iterate
      pmhd_final_state<MET>(p, s, best_x, *bst, Pn);
    else
      pmhd_final<MET, double>(p, s, best_x, Pn, nullptr, p.sig ? &lcode : nullptr);
    if (b.psol_rec)
      for (int q = 0; q < NPR; ++q) b.psol_rec[12 * bx.aoff + q * bx.nact + z] = Pn[q];
    unsigned fcode = 0;
    apply_floors<MET>(p, g, fl[0], fl[1], Pn, p.sig ? &fcode : nullptr);
    if (p.sig) sig_put(p, bx.coff + t, 60, (fcode << 2 | lcode) << 4 | ST_PMHD);
#pragma unroll
    for (int q = 0; q < NPR; ++q) P[q * bx.ntot + t] = Pn[q];
    if (b.meth_rec) b.meth_rec[zg] = ST_PMHD;
  } else {
    int slot = atomicAdd(&b.qcount[0], 1);
    b.qzone[slot] = (int)z;
    b.qbox[slot] = bi;
    double* qd = b.qdata + (long long)slot * QSTRIDE;
#pragma unroll
    for (int q = 0; q < NPR; ++q) qd[q] = Ust[q];
    for (int q = 0; q < 4; ++q) qd[12 + q] = isfinite(beT) ? best_x[q] : 0.0;
    qd[16] = beT;
    qd[17] = h;
    qd[18] = Sst;
  }
  return accept;
}

// The radiation of a zone is "extremely sub-dominant" (Sec. 4.10) when its
// conserved energy in U* or its fluid-frame energy density
// Ehat = Ebar (4/3 gamma_rel^2 - 1/3) is below 10 eps_m of the gas's (u_g for
// Ehat).  PMHD recovers the radiation from the gas's round-off there, so such
// zones start with URAD.  (The relative change of the energy row over the
// explicit update, which the paper also lists, would flag every zone whose
// radiation the update left unchanged, whatever its size; it is not used.)
template <int MET>
__device__ __forceinline__ bool radiation_subdominant(const Geo<MET, double>& g, const double Ust[NPR],
                                                      const double Ps[NPR]) {
  const double tiny = 10.0 * 2.220446049250313e-16;
  if (fabs(Ust[ER]) < tiny * fabs(Ust[UU])) return true;
  if (!(Ps[ER] < tiny * Ps[UU])) return false;  // Ehat >= Ebar (gamma_rel >= 1)
  double uc[4], uv[4], gm, rc[4], rv[4], gr;
  fourvel<MET, double>(g, Ps[U1], Ps[U2], Ps[U3], uc, uv, &gm);
  fourvel<MET, double>(g, Ps[UR1], Ps[UR2], Ps[UR3], rc, rv, &gr);
  const double grel = -(rc[0] * uv[0] + rc[1] * uv[1] + rc[2] * uv[2] + rc[3] * uv[3]);
  return Ps[ER] * ((4.0 / 3.0) * grel * grel - 1.0 / 3.0) < tiny * Ps[UU];
}

// Sec. 4.11: the cold-MHD equations are tried only for a cold, momentum-
// dominated zone: u_g < 0.1 rho0 u~^i u~_i of the guess primitives, and for
// the gas t^t_mu = T^t_mu + rho0 u^t delta^t_mu and the radiation R^t_mu of
// U* alike, |t_t t^t| < 0.1 |sum_i t_i t^i| with t^mu = g^{mu nu} t_nu.
template <int MET>
__device__ __forceinline__ bool cold_allowed(const Geo<MET, double>& g, const double Ust[NPR],
                                             const double Ps[NPR]) {
  if (!(Ps[UU] < 0.1 * Ps[RHO] * g.sq3(Ps[U1], Ps[U2], Ps[U3]))) return false;
  const double igd = 1.0 / g.gdet;
#pragma unroll
  for (int w = 0; w < 2; ++w) {
    const int o = w == 0 ? UU : ER;
    const double t[4] = {Ust[o] * igd, Ust[o + 1] * igd, Ust[o + 2] * igd, Ust[o + 3] * igd};
    double up[3];
    g.raise3(t, up);
    const double at = fabs(t[0] * g.raise_t(t));
    const double as = fabs(t[1] * up[0] + t[2] * up[1] + t[3] * up[2]);
    if (!(at < 0.1 * as)) return false;
  }
  return true;
}

// The back-up equations of Sec. 4.11 for a zone that the energy methods left
// without a solution.  First the entropy equation (Eq. source6) in place of
// the gas energy equation, where the explicit S* (sqrt(-g) S u^t) is finite,
// by the energy methods' sequence: PMHD (emode 1; with emode 2 the update
// kernel ran it already and px / peT are its best iterate and error), then
// URAD and PRAD while the best entropy solution has e_T >= 1e-9, each from the
// primitives of that solution if its e_T < 1e-4, else from P_s.  Then, for a
// cold momentum-dominated zone (cold_allowed), the cold-MHD equations: PMHD
// on the three momentum equations with u_g held at the guess.  The PMHD
// attempts start from the energy PMHD's guess (P_s, or where tau < 2/3 the
// gas inversion of U*); a solution is accepted at e_T <= 1e-7.  Returns
// METH_ENTROPY (the entropy PMHD's solution), METH_ENTROPY_RAD (the entropy
// URAD's or PRAD's) or METH_COLD with Pn and *eT set, 0 if none gives a
// solution; adds the Newton steps to *steps.  emode 0: no entropy equation.
template <int MET, bool FAST>
__device__ int backup_equations(const DevParams& p, const Geo<MET, double>& g, const ImpSys<MET, FAST>& s,
                                const double Ust[NPR], const double Ps[NPR], double Sst, int emode,
                                double tau, double Pn[NPR], double* eT, int* steps,
                                const double* px = nullptr, double peT = HUGE_VAL) {
  const bool ent = emode != 0 && isfinite(Sst);
  const bool cold = cold_allowed<MET>(g, Ust, Ps);
  if (!ent && !cold) return 0;
  double x0[4] = {Ps[UU], Ps[U1], Ps[U2], Ps[U3]};
  if (tau < 2.0 / 3.0) {
    double go[5], T3[3] = {s.Ts[1], s.Ts[2], s.Ts[3]};
    if (gas_invert_sys<MET>(p, s, s.Ts[0], T3, Ps, 1e-9, go) == 0)
      for (int c = 0; c < 4; ++c) x0[c] = go[1 + c];
  }
  if (ent) {
    ImpSys<MET, FAST> se = s;
    se.entropy = true;
    se.Sstar = Sst / g.gdet;
    double bxe[4] = {0.0, 0.0, 0.0, 0.0}, beT = HUGE_VAL;
    int who = -1;  // 0 PMHD, 1 URAD, 2 PRAD
    if (emode == 1) {
      double xe[4] = {x0[0], x0[1], x0[2], x0[3]};
      entropy_ug_guess(p, Sst, s.Dlab * g.gdet, Ps[RHO], xe);
      *steps += newton_pmhd<MET>(p, se, xe, bxe, &beT);
    } else if (px && isfinite(peT)) {
      for (int c = 0; c < 4; ++c) bxe[c] = px[c];
      beT = peT;
    }
    if (isfinite(beT)) who = 0;
    double rx[2][4], rgas[2][5];
#pragma unroll 1
    for (int pr = 0; pr < 2 && !(beT < 1e-9); ++pr) {
      double Pq[NPR];
      for (int q = 0; q < NPR; ++q) Pq[q] = Ps[q];
      if (who >= 0 && beT < 1e-4) {
        if (who == 0) {
          ImpRes rr;
          ImpState stt;
          pmhd_res<MET>(p, se, bxe, rr, &stt, false);
          Pq[RHO] = stt.rho;
          for (int c = 0; c < 4; ++c) Pq[UU + c] = bxe[c];
          for (int c = 0; c < 4; ++c) Pq[ER + c] = stt.Pr[c];
        } else if (who == 1) {
          for (int c = 0; c < 5; ++c) Pq[c] = rgas[0][c];
          rad_invert<MET>(p, g, rx[0], 2, Pq + ER);
        } else {
          for (int c = 0; c < 5; ++c) Pq[c] = rgas[1][c];
          for (int c = 0; c < 4; ++c) Pq[ER + c] = rx[1][c];
        }
      }
      double gq[5] = {Pq[RHO], Pq[UU], Pq[U1], Pq[U2], Pq[U3]}, x4[4], reT;
      if (pr == 1) {
        for (int c = 0; c < 4; ++c) x4[c] = Pq[ER + c];
        *steps += newton_rad<MET, true>(p, se, x4, gq, rx[1], rgas[1], &reT);
      } else {
        double urc2[4], urv2[4], gr2;
        fourvel<MET, double>(g, Pq[UR1], Pq[UR2], Pq[UR3], urc2, urv2, &gr2);
        const double e43q = (4.0 / 3.0) * Pq[ER];
        x4[0] = e43q * urc2[0] * urv2[0] + Pq[ER] * (1.0 / 3.0);
        for (int c = 1; c < 4; ++c) x4[c] = e43q * urc2[0] * urv2[c];
        *steps += newton_rad<MET, false>(p, se, x4, gq, rx[0], rgas[0], &reT);
      }
      if (isfinite(reT) && (who < 0 || reT < beT)) {
        who = 1 + pr;
        beT = reT;
      }
    }
    if (beT <= 1e-7) {
      if (who == 0) {
        pmhd_final<MET>(p, se, bxe, Pn);
      } else {
        for (int q = 0; q < 5; ++q) Pn[q] = rgas[who - 1][q];
        if (who == 1) {
          double Pr[4];
          if (rad_invert<MET>(p, g, rx[0], 2, Pr)) rad_invert<MET>(p, g, rx[0], 0, Pr);
          for (int q = 0; q < 4; ++q) Pn[ER + q] = Pr[q];
        } else {
          for (int q = 0; q < 4; ++q) Pn[ER + q] = rx[1][q];
        }
        for (int c = 0; c < 3; ++c) Pn[B1 + c] = s.B[c];
      }
      *eT = beT;
      return who == 0 ? METH_ENTROPY : METH_ENTROPY_RAD;
    }
  }
  if (cold) {
    ImpSys<MET, FAST> sc = s;
    sc.entropy = false;
    sc.cold = true;
    double bxc[4] = {0.0, 0.0, 0.0, 0.0}, beT = HUGE_VAL;
    *steps += newton_pmhd<MET>(p, sc, x0, bxc, &beT);
    if (beT <= 1e-7) {
      pmhd_final<MET>(p, sc, bxc, Pn);
      *eT = beT;
      return METH_COLD;
    }
  }
  return 0;
}

// The explicit entropy S* = a_s S^n + b_s (S(P_s) + dt X_S) of a zone (FP64,
// RK3), formed where it is read: by the zones that reach the entropy equation
// (Sec. 4.7, 4.11), few in any run, or by all zones in the entropy-everywhere
// mode.  Two logarithms per face were a quarter of the face kernel when every
// face formed its flux (256x128x64 torus, per RK3 step: faces 17.4 -> 13.8 ms,
// update 21.7 -> 20.5 ms without, at 16 blocks per SM); the face kernel keeps the
// left state's mass flux mL, and the flux is s_L mL + s_R (F_rho - mL) with the
// entropy per baryon s of the kept edges (Sec. 2, Eq. S).  The mode that reads it
// everywhere forms each face's flux from either side and still gains with the rest
// (128x64x32 torus, step: 16.9 -> 11.2 ms).
static __device__ __forceinline__ double entropy_flux(const DevParams& p, const BoxGeo& bx, const Bufs& b, int d,
                                                      long long t) {
  const double* S = b.ES[d] + 4 * bx.coff;
  const long long nt = bx.ntot, tm = t - bx.str[d];
  const double mL = ((const double*)b.FS[d])[bx.coff + t], m = ((const double*)b.F[d])[12 * bx.coff + t];
  return entropy_per_baryon<double>(p, S[2 * nt + tm], S[3 * nt + tm]) * mL +
         entropy_per_baryon<double>(p, S[t], S[nt + t]) * (m - mL);
}
// Us0 = sqrt(-g) rho0 u^t of the sub-step's input, rho, ug its density and
// internal energy; z, t the zone's active and cell index.
__device__ __forceinline__ double entropy_star(const DevParams& p, const BoxGeo& bx, const Bufs& b, long long z,
                                               long long t, int stage, double dt, double Us0, double rho,
                                               double ug) {
  const double A = stage == 0 ? 0.0 : (stage == 1 ? 0.75 : 1.0 / 3.0);
  const double Bc = stage == 0 ? 1.0 : (stage == 1 ? 0.25 : 2.0 / 3.0);
  const double Su = Us0 * entropy_per_baryon<double>(p, rho, ug);
  const double* Sn = b.Sn + 2 * bx.aoff;
  const double sn =
      stage == 0 ? Su : b.Un[12 * bx.aoff + z] * entropy_per_baryon<double>(p, Sn[z], Sn[bx.nact + z]);
  double div = 0.0;
#pragma unroll 1
  for (int f = 0; f < 6; ++f) {  // the upper and the lower face of each direction
    const int d = f >> 1;
    if (!p.act[d]) continue;
    const double v = entropy_flux(p, bx, b, d, t + (f & 1 ? 0 : bx.str[d])) / bx.dx[d];
    div += f & 1 ? -v : v;
  }
  return A * sn + Bc * (Su - dt * div);
}

// ------------------------------------------------------- update + implicit
// One thread per active zone: U(P_s), the geometric source
// SM_nu = 1/2 sqrt(-g) T^{mu kappa} d_nu g_{mu kappa}  (equal to
// sqrt(-g) T^kappa_lambda Gamma^lambda_{nu kappa} for a symmetric T, nonzero
// only for nu = x1, x2 on the stationary axisymmetric metric), the explicit
// update X = -sum_d dF_d/dx_d + SM, the RK3 combination
// U* = a_s U^n + b_s (U(P_s) + dt X) (Sec. 4.1), the PMHD Newton solve, floors.
// Zones whose PMHD error exceeds 1e-9 go to the retry queue, and so do zones
// whose radiation is extremely sub-dominant (URAD only, Sec. 4.10).
template <int MET, typename R, bool CONT, bool IMEX>
__device__ __forceinline__ void update_box(const DevParams& p, const BoxGeo& bx, int bi, const Bufs& b,
                                           int stage, int split, const ImexStage& im) {
  const double A = stage == 0 ? 0.0 : (stage == 1 ? 0.75 : 1.0 / 3.0);
  const double Bc = stage == 0 ? 1.0 : (stage == 1 ? 0.25 : 2.0 / 3.0);
  {
    const double dt = b.dt[bi];
    double* P = b.P + 12 * bx.coff;
    const double* K = b.K + bx.coff;
    double* Un = b.Un + 12 * bx.aoff;
    const R* Fd[3] = {(const R*)b.F[0] + 12 * bx.coff, (const R*)b.F[1] + 12 * bx.coff,
                      (const R*)b.F[2] + 12 * bx.coff};
    const double idx[3] = {1.0 / bx.dx[0], 1.0 / bx.dx[1], 1.0 / bx.dx[2]};
    for (long long z = first_item(bx.aoff); z < bx.nact; z += HR_STRIDE) {
      long long r = z;
      int i = (int)(r % bx.n[0]);
      r /= bx.n[0];
      int j = (int)(r % bx.n[1]);
      int k = (int)(r / bx.n[1]);
      long long t = cell_index(bx, i, j, k);
      // the zone's metric, 1/sqrt(-g), sqrt(gamma^{kk}), floors and longest edge
      Geo<MET, double> g;
      MetricDeriv mdt{};
      double igd, sgk[3], fl[2], dl;
      if constexpr (MET == KS) {
        const GeoTab T = geotab(b.geo, bx);
        const long long gi = gidx_c(bx, i, j);
        g = geo_load<MET>(T.C, T.sC, gi);
        mdt = md_load(T.M, T.sC, gi);
        igd = __ldg(T.C + 16 * T.sC + gi);
        for (int e = 0; e < 3; ++e) sgk[e] = __ldg(T.C + (20 + e) * T.sC + gi);
        fl[0] = __ldg(T.C + 23 * T.sC + gi);
        fl[1] = __ldg(T.C + 24 * T.sC + gi);
        dl = __ldg(T.C + 25 * T.sC + gi);
      } else {
        g = make_geo<MET, double>(p, 0.0, 0.0);
        igd = sgk[0] = sgk[1] = sgk[2] = 1.0;
        fl[0] = p.rf0;
        fl[1] = p.uf0;
        dl = 0.0;
        for (int e = 0; e < 3; ++e)
          if (p.act[e]) dl = fmax(dl, bx.dx[e]);
      }
      double Ps[NPR];
#pragma unroll
      for (int q = 0; q < NPR; ++q) Ps[q] = P[q * bx.ntot + t];
      const double kz = kfield(p, K, t);
      double Us[NPR], X[NPR];
      constexpr bool FAST = std::is_same<R, double>::value;
      if constexpr (FAST) cons_source64<MET>(p, g, Ps, Us, X, mdt);
      else cons_source<MET, double>(p, g, 0.0, 0.0, Ps, Us, X, &mdt);
      // flux divergence (an IMEX stage without flux term reads no fluxes)
      const bool rhs = !IMEX || im.d != 0.0;
#pragma unroll
      for (int d = 0; d < 3; ++d) {
        if (!p.act[d] || !rhs) continue;
        const long long s = bx.str[d];
#pragma unroll
        for (int q = 0; q < NPR; ++q) {
          if (q == B1 + d) continue;  // F_d[B_d] = 0
          R df = Fd[d][q * bx.ntot + t + s] - Fd[d][q * bx.ntot + t];
          X[q] -= double(df) * idx[d];
        }
      }
      double Ust[NPR];
#pragma unroll
      for (int q = 0; q < NPR; ++q) {
        double un;
        if (stage == 0) {
          Un[q * bx.nact + z] = Us[q];
          un = Us[q];
        } else {
          un = Un[q * bx.nact + z];
        }
        if constexpr (IMEX)
          Ust[q] = im.an * un + im.ap * Us[q] + im.d * dt * X[q];
        else
          Ust[q] = A * un + Bc * (Us[q] + dt * X[q]);
      }
      if (b.Bf[0]) {  // staggered field: B from the evolved faces (average of the two)
#pragma unroll
        for (int d = 0; d < 3; ++d) {
          const double* Bfd = b.Bf[d] + bx.coff;
          Ust[B1 + d] = p.act[d] ? 0.5 * (Bfd[t] + Bfd[t + bx.str[d]]) : Bfd[t];
        }
      }
      if (IMEX && stage > 0) {
        // earlier stages' implicit sources: +M on the gas rows, -M on the radiation rows
        const double* M = b.imexM + 16 * bx.aoff + z;
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          if (j >= stage) break;
          const double cj = im.c[j];
#pragma unroll
          for (int r = 0; r < 4; ++r) {
            const double m = M[(4 * j + r) * bx.nact];
            Ust[UU + r] += dt * cj * m;
            Ust[ER + r] -= dt * cj * m;
          }
        }
      }
      if (b.ust_rec) {
#pragma unroll
        for (int q = 0; q < NPR; ++q) b.ust_rec[12 * bx.aoff + q * bx.nact + z] = Ust[q];
      }
      // RK3: what the explicit entropy needs of the step's start (FP64,
      // entropy_star; where every zone takes the entropy equation it is formed
      // here), or, in split precision, the explicit entropy
      // S* = a_s S^n + b_s (S(P_s) + dt X_S) itself; NaN: none
      double Sst = NAN;
      if (!IMEX && b.Sn) {
        if constexpr (std::is_same<R, double>::value) {
          if (stage == 0) {
            b.Sn[2 * bx.aoff + z] = Ps[RHO];
            b.Sn[2 * bx.aoff + bx.nact + z] = Ps[UU];
          }
          if (p.implicit_eq == 1) Sst = entropy_star(p, bx, b, z, t, stage, dt, Us[RHO], Ps[RHO], Ps[UU]);
        } else {
          const double Su = Us[RHO] * entropy_per_baryon<double>(p, Ps[RHO], Ps[UU]);
          double* Sn = b.Sn + bx.aoff;
          double sn;
          if (stage == 0) {
            Sn[z] = Su;
            sn = Su;
          } else {
            sn = Sn[z];
          }
          double divS = 0.0;
#pragma unroll
          for (int d = 0; d < 3; ++d) {
            if (!p.act[d]) continue;
            const R* FSd = (const R*)b.FS[d] + bx.coff;
            divS += double(FSd[t + bx.str[d]] - FSd[t]) * idx[d];
          }
          Sst = A * sn + Bc * (Su - dt * divS);
        }
      }
      // implicit solve
      const double h = IMEX ? im.g * dt : Bc * dt;
      // extremely sub-dominant radiation: no PMHD attempt; the zone goes to
      // the retry queue for URAD with a negative PMHD error as the mark
      const bool subdom = radiation_subdominant<MET>(g, Ust, Ps);
      ImpSys<MET, FAST> s;
      build_sys_with<MET, double>(p, g, igd, sgk, Ust, h, kz, s);
      double x0[4] = {Ps[UU], Ps[U1], Ps[U2], Ps[U3]}, kt;
      if constexpr (FAST) {
        kt = opacity_sum(p, Ps[RHO], [&] { return p.gm1 * Ps[UU] * rcp(Ps[RHO]); }, kz);
      } else {
        double kabs, ksca;
        opacity<double>(p, Ps[RHO], Ps[UU], kz, &kabs, &ksca);
        kt = kabs + ksca;
      }
      if (kt * dl < 2.0 / 3.0) {
        double go[5];
        double T3[3] = {s.Ts[1], s.Ts[2], s.Ts[3]};
        const int rc = FAST ? gas_invert<MET>(p, g, s.Dlab, s.Ts[0], T3, s.B, Ps, 1e-9, go)
                            : gas_invert_ieee<MET>(p, g, s.Dlab, s.Ts[0], T3, s.B, Ps, 1e-9, go);
        if (rc == 0) {
          x0[0] = go[1];
          x0[1] = go[2];
          x0[2] = go[3];
          x0[3] = go[4];
        }
      }
      bool accept = false;
      unsigned done_steps = 0;
      if (p.implicit_eq == 1) {
        // the entropy equation in every zone (Eq. source6), PMHD iterates;
        // e_T >= 1e-9 goes to the retry queue for the entropy URAD and PRAD
        // (the methods' sequence, Sec. 4.10-4.11)
        s.entropy = true;
        s.Sstar = Sst * igd;
        double bxn[4] = {0.0, 0.0, 0.0, 0.0}, beT = HUGE_VAL;
        double xe[4] = {x0[0], x0[1], x0[2], x0[3]};
        entropy_ug_guess(p, Sst, s.Dlab * g.gdet, Ps[RHO], xe);
        const int steps = newton_pmhd<MET>(p, s, xe, bxn, &beT);
        accept = pmhd_finish<MET>(p, bx, bi, z, t, fl, g, s, Ust, h, bxn, beT, steps, P, b, Sst, 1e-9);
        done_steps = (unsigned)steps;
        warp_add(&b.stats[ST_ENTROPY], accept ? 1u : 0u);
      } else if constexpr (!CONT) {
        double bxn[4] = {0.0, 0.0, 0.0, 0.0}, beT = -1.0;
        ImpState bst;
        const int steps = subdom ? 0 : newton_pmhd<MET>(p, s, x0, bxn, &beT, &bst);
        accept = pmhd_finish<MET>(p, bx, bi, z, t, fl, g, s, Ust, h, bxn, beT, steps, P, b, Sst, 1e-9,
                                  subdom ? nullptr : &bst);
        done_steps = (unsigned)steps;
      } else {
        // the first `split` iterations here; a zone that needs more
        // continues in the compacted queue (k_newton_cont), so that the
        // heavy tail of iteration counts runs in full warps
        NewtonState ns;
        newton_pmhd_init(x0, ns);
        if (subdom) ns.best_eT = -1.0;
        if (subdom || newton_pmhd_run<MET>(p, s, ns, split)) {
          accept = pmhd_finish<MET>(p, bx, bi, z, t, fl, g, s, Ust, h, ns.best_x, ns.best_eT, ns.steps, P, b, Sst);
          done_steps = (unsigned)ns.steps;
        } else {
          const int slot = ns.jac32 ? atomicAdd(&b.qcount[2], 1) : b.ncont - 1 - atomicAdd(&b.qcount[3], 1);
          b.czone[slot] = (int)z;
          b.cbox[slot] = bi;
          double* cd = b.cdata + (long long)slot * CSTRIDE;
#pragma unroll
          for (int q = 0; q < NPR; ++q) cd[q] = Ust[q];
          newton_state_store(ns, cd + NPR);
          cd[NPR + 22] = Sst;
        }
      }
      warp_add(&b.stats[ST_PMHD], accept ? 1u : 0u);
      warp_add(&b.stats[ST_ITERS], done_steps);
      warp_add(&b.stats[ST_SOLVES], 1u);
    }
  }
}

// Zones whose PMHD Newton iteration did not end within the update kernel's
// `split` iterations: a persistent grid over the compacted queue
// resumes each iteration from its saved state (same arithmetic as an
// uninterrupted iteration) and finishes the zone as the update kernel would.
// Bound by FP64 warp instructions, which cost the same with one lane as with 32:
// zones on finite differences (five residuals an iteration) come from the
// queue's other end, into warps of their own.  Update class of 12 boxes per RK3
// step 43.9 -> 29.9 ms (11 lanes of 32 were active in an FP64 instruction of the
// update kernel, 18 now).
// FAST: the functions of the context's update kernel (ImpSysT), so that a queue
// changes no byte of the result, in split precision (false) as in FP64.
template <int MET, bool FAST>
__global__ void __launch_bounds__(128) k_newton_cont(DevParams p, const BoxGeo* __restrict__ boxes, Bufs b,
                                                     double hfac) {
  // the finite-difference zones first, in warps of their own
  const int nfd = b.qcount[3], pad = (nfd + 31) & ~31, nq = pad + b.qcount[2];
  for (int it = blockIdx.x * blockDim.x + threadIdx.x; it < nq; it += gridDim.x * blockDim.x) {
    if (it >= nfd && it < pad) continue;
    const int e = it < nfd ? b.ncont - 1 - it : it - pad;
    const int bi = b.cbox[e];
    const BoxGeo& bx = boxes[bi];
    const long long z = b.czone[e];
    long long r = z;
    const int i = (int)(r % bx.n[0]);
    r /= bx.n[0];
    const int j = (int)(r % bx.n[1]);
    const int k = (int)(r / bx.n[1]);
    const long long t = cell_index(bx, i, j, k);
    const Geo<MET, double> g = geo_centre<MET, double>(p, bx, b.geo, i, j);
    double fl[2];
    floor_values<MET>(p, xcen(bx, 0, i), &fl[0], &fl[1]);
    const double* cd = b.cdata + (long long)e * CSTRIDE;
    double Ust[NPR];
    for (int q = 0; q < NPR; ++q) Ust[q] = cd[q];
    NewtonState ns;
    newton_state_load(cd + NPR, ns);
    const double h = hfac * b.dt[bi];  // the sub-step's implicit step fraction
    ImpSys<MET, FAST> s;
    build_sys<MET>(p, g, Ust, h, kfield(p, b.K + bx.coff, t), s);
    newton_pmhd_run<MET>(p, s, ns, INT_MAX);
    const bool accept = pmhd_finish<MET>(p, bx, bi, z, t, fl, g, s, Ust, h, ns.best_x, ns.best_eT, ns.steps,
                                         b.P + 12 * bx.coff, b, cd[NPR + 22]);
    if (accept) atomicAdd(&b.stats[ST_PMHD], 1ULL);
    atomicAdd(&b.stats[ST_ITERS], (unsigned long long)ns.steps);
  }
}

// IMEX: the sub-step of an IMEX scheme with coefficients im (otherwise RK3).
// ONE: a single grid whose geometry travels in the kernel's parameter space
// (no registers held for it across the Newton solve); otherwise the boxes of
// a batch, read from the device table.  CONT: PMHD iterations beyond `split`
// continue in k_newton_cont (the queue costs registers; it pays where the
// iteration counts are heavy-tailed, which the autotuner measures).
template <int MET, typename R, bool ONE, bool CONT, bool IMEX>
__global__ void __launch_bounds__(128) k_update(DevParams p, BoxGeo one, const BoxGeo* __restrict__ boxes,
                                                int nbox, Bufs b, int stage, int split, ImexStage im) {
  if constexpr (ONE) {
    update_box<MET, R, CONT, IMEX>(p, one, 0, b, stage, split, im);
  } else {
    for (int bi = 0; bi < nbox; ++bi) update_box<MET, R, CONT, IMEX>(p, boxes[bi], bi, b, stage, split, im);
  }
}

// IMEX: the implicit source of stage j on the gas rows,
// M^j = (U(P) - U*) / (g dt), with P the stage's implicit solution before the
// floors (the change the implicit stage made, Sec. 4.8); the radiation rows
// take -M^j, so gas plus radiation stays conserved.
template <int MET>
__global__ void k_imex_store(DevParams p, const BoxGeo* __restrict__ boxes, int nbox, Bufs b, int j, double gj) {
  for (int bi = 0; bi < nbox; ++bi) {
    const BoxGeo& bx = boxes[bi];
    const double h = gj * b.dt[bi];
    const double* Ps = b.psol_rec + 12 * bx.aoff;
    const double* Us = b.ust_rec + 12 * bx.aoff;
    double* M = b.imexM + 16 * bx.aoff;
    for (long long z = first_item(bx.aoff); z < bx.nact; z += HR_STRIDE) {
      long long r = z;
      const int i = (int)(r % bx.n[0]);
      r /= bx.n[0];
      const int jj = (int)(r % bx.n[1]);
      const double x1 = xcen(bx, 0, i), x2 = xcen(bx, 1, jj);
      const Geo<MET, double> g = geo_centre<MET, double>(p, bx, b.geo, i, jj);
      double Pz[NPR], Uz[NPR], Xz[NPR];
#pragma unroll
      for (int q = 0; q < NPR; ++q) Pz[q] = Ps[q * bx.nact + z];
      cons_source<MET, double>(p, g, x1, x2, Pz, Uz, Xz);
#pragma unroll
      for (int q = 0; q < 4; ++q) M[(4 * j + q) * bx.nact + z] = (Uz[UU + q] - Us[(UU + q) * bx.nact + z]) / h;
    }
  }
}

// ----------------------------------------------------------- retry (URAD)
// Persistent grid over the retry queue (its length is read on the device, so
// the launch needs no host round trip and can live in a CUDA graph): URAD,
// then PRAD (retry_sequence); e_T > 1e-7 sends the zone to the
// neighbour-average back-up.  FAST: as k_newton_cont.
template <int MET, bool FAST>
__global__ void __launch_bounds__(128) k_retry(DevParams p, const BoxGeo* __restrict__ boxes, Bufs b, int stage) {
  const int nq = b.qcount[0];
  for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < nq; e += gridDim.x * blockDim.x) {
    const long long z = b.qzone[e];
    const int bi = b.qbox[e];
    const BoxGeo& bx = boxes[bi];
    double* P = b.P + 12 * bx.coff;
    const double* K = b.K + bx.coff;
    const double* qd = b.qdata + (long long)e * QSTRIDE;
    long long r = z;
    int i = (int)(r % bx.n[0]);
    r /= bx.n[0];
    int j = (int)(r % bx.n[1]);
    int k = (int)(r / bx.n[1]);
    long long t = cell_index(bx, i, j, k);
    double x1 = xcen(bx, 0, i), x2 = xcen(bx, 1, j);
    Geo<MET, double> g = make_geo<MET, double>(p, x1, x2);
    double Ust[NPR], Ps[NPR], px[4];
    for (int q = 0; q < NPR; ++q) {
      Ust[q] = qd[q];
      Ps[q] = P[q * bx.ntot + t];
    }
    for (int q = 0; q < 4; ++q) px[q] = qd[12 + q];
    // qd[16] < 0: radiation extremely sub-dominant, URAD only (no PMHD iterate)
    const bool subdom = qd[16] < 0.0;
    const double peT = subdom ? HUGE_VAL : qd[16];
    const double h = qd[17];
    ImpSys<MET, FAST> s;
    build_sys<MET>(p, g, Ust, h, kfield(p, K, t), s);
    const long long zg = bx.aoff + z;
    double Pn[NPR], eT;
    int steps;
    const double tau = zone_tau<MET>(p, g, bx.dx, Ps, kfield(p, K, t));
    int method;
    double Sst = qd[18];
    // FP64: the explicit entropy, where the sequence reads it
    auto entropy = [&] {
      if (!FAST || !b.Sn) return;
      double u[4], v[4], gm;
      fourvel<MET, double>(g, Ps[U1], Ps[U2], Ps[U3], u, v, &gm);
      Sst = entropy_star(p, bx, b, z, t, stage, b.dt[bi], g.gdet * Ps[RHO] * u[0], Ps[RHO], Ps[UU]);
      if (b.sst_rec) b.sst_rec[zg] = Sst;
    };
    if (p.implicit_eq == 1) {  // the entropy PMHD of the update kernel left e_T >= 1e-9
      for (int q = 0; q < NPR; ++q) Pn[q] = Ps[q];
      for (int c = 0; c < 3; ++c) Pn[B1 + c] = s.B[c];
      eT = HUGE_VAL;
      steps = 0;
      method = ST_BACKUP;
    } else {
      if (subdom) entropy();
      method = retry_sequence<MET>(p, g, s, Ps, px, peT, tau, Pn, &eT, &steps, subdom, Sst);
    }
    // no energy-based solution: the entropy, then the cold-MHD equations
    int by = 0;
    if (method == ST_BACKUP) {
      if (p.implicit_eq != 1 && !subdom) entropy();
      by = p.implicit_eq == 1 ? backup_equations<MET>(p, g, s, Ust, Ps, Sst, 2, tau, Pn, &eT, &steps, px, peT)
                              : backup_equations<MET>(p, g, s, Ust, Ps, Sst, 1, tau, Pn, &eT, &steps);
      // a retry method's solution, except that in the entropy-everywhere
      // mode the entropy PMHD is the first method
      if (by) method = (p.implicit_eq == 1 && by == METH_ENTROPY) ? ST_PMHD : ST_URAD;
    }
    b.iters[zg] += steps;
    if (b.psol_rec)
      for (int q = 0; q < NPR; ++q) b.psol_rec[12 * bx.aoff + q * bx.nact + z] = Pn[q];
    unsigned fcode = 0;
    double fl[2];
    floor_values<MET>(p, x1, &fl[0], &fl[1]);
    apply_floors<MET>(p, g, fl[0], fl[1], Pn, p.sig ? &fcode : nullptr);
    if (p.sig) sig_put(p, bx.coff + t, 60, fcode << 4 | (unsigned)method);
    for (int q = 0; q < NPR; ++q) P[q * bx.ntot + t] = Pn[q];
    unsigned char m = (unsigned char)method;
    if (m > b.status[zg]) b.status[zg] = m;
    // the adjoint differentiates every entropy solution through the entropy
    // PMHD's system (the URAD and PRAD solve the same equations)
    if (b.meth_rec) b.meth_rec[zg] = by ? (unsigned char)(by == METH_ENTROPY_RAD ? METH_ENTROPY : by) : m;
    if (by == METH_ENTROPY || by == METH_ENTROPY_RAD) atomicAdd(&b.stats[ST_ENTROPY], 1ULL);
    if (by == METH_COLD) atomicAdd(&b.stats[ST_COLD], 1ULL);
    if (method == ST_BACKUP || by == METH_COLD) {
      // the back-up average: all primitives but B, or u_g alone for a
      // cold-MHD solution (Sec. 4.11); either counts as not good for its
      // neighbours' averages
      b.failed[zg] = method == ST_BACKUP ? 1 : 2;
      int slot = atomicAdd(&b.qcount[1], 1);
      b.fzone[slot] = (int)z;
      b.fbox[slot] = bi;
    }
    if (method == ST_BACKUP) {
      atomicAdd(&b.stats[ST_BACKUP], 1ULL);
    } else if (method == ST_URAD) {
      atomicAdd(&b.stats[ST_URAD], 1ULL);
    } else {
      atomicAdd(&b.stats[ST_PMHD], 1ULL);
    }
    atomicAdd(&b.stats[ST_ITERS], (unsigned long long)steps);
  }
}

// ------------------------------------------------------------- back-up
// Average of the good active face neighbours (all active neighbours if none
// is good); B keeps its constrained-transport value, and a zone solved by the
// cold-MHD equations takes the average for u_g alone (Sec. 4.11).  All
// averages are formed before any is written back (k_backup_apply).
static __global__ void k_backup_avg(DevParams p, const BoxGeo* __restrict__ boxes, Bufs b) {
  const int nf = b.qcount[1];
  for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < nf; e += gridDim.x * blockDim.x) {
    const BoxGeo& bx = boxes[b.fbox[e]];
    const double* P = b.P + 12 * bx.coff;
    long long z = b.fzone[e];
    long long r = z;
    int ii[3];
    ii[0] = (int)(r % bx.n[0]);
    r /= bx.n[0];
    ii[1] = (int)(r % bx.n[1]);
    ii[2] = (int)(r / bx.n[1]);
    double sg[NPR], sa[NPR];
    for (int q = 0; q < NPR; ++q) sg[q] = sa[q] = 0.0;
    int ng = 0, na = 0;
    for (int d = 0; d < 3; ++d) {
      if (bx.n[d] == 1) continue;
      for (int side = -1; side <= 1; side += 2) {
        int nb[3] = {ii[0], ii[1], ii[2]};
        nb[d] += side;
        if (nb[d] < 0 || nb[d] >= bx.n[d]) continue;
        long long zn = ((long long)nb[2] * bx.n[1] + nb[1]) * bx.n[0] + nb[0];
        long long tn = cell_index(bx, nb[0], nb[1], nb[2]);
        bool good = !b.failed[bx.aoff + zn];
        for (int q = 0; q < NPR; ++q) {
          double v = P[q * bx.ntot + tn];
          sa[q] += v;
          if (good) sg[q] += v;
        }
        ++na;
        if (good) ++ng;
      }
    }
    long long t = cell_index(bx, ii[0], ii[1], ii[2]);
    if (p.sig) sig_put(p, bx.coff + t, 61, (unsigned)ng << 4 | (unsigned)na);
    const bool cold = b.failed[bx.aoff + z] == 2;
    for (int q = 0; q < NPR; ++q) {
      double v = P[q * bx.ntot + t];
      if (na > 0 && !(q >= B1 && q <= B3) && (!cold || q == UU)) v = ng > 0 ? sg[q] / ng : sa[q] / na;
      b.ftmp[(long long)e * NPR + q] = v;
    }
  }
}

template <int MET>
__global__ void k_backup_apply(DevParams p, const BoxGeo* __restrict__ boxes, Bufs b) {
  const int nf = b.qcount[1];
  for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < nf; e += gridDim.x * blockDim.x) {
    const BoxGeo& bx = boxes[b.fbox[e]];
    double* P = b.P + 12 * bx.coff;
    long long z = b.fzone[e];
    long long r = z;
    int i = (int)(r % bx.n[0]);
    r /= bx.n[0];
    int j = (int)(r % bx.n[1]);
    int k = (int)(r / bx.n[1]);
    long long t = cell_index(bx, i, j, k);
    double x1 = xcen(bx, 0, i), x2 = xcen(bx, 1, j);
    Geo<MET, double> g = make_geo<MET, double>(p, x1, x2);
    double Pn[NPR];
    for (int q = 0; q < NPR; ++q) Pn[q] = b.ftmp[(long long)e * NPR + q];
    unsigned fcode = 0;
    double fl[2];
    floor_values<MET>(p, x1, &fl[0], &fl[1]);
    apply_floors<MET>(p, g, fl[0], fl[1], Pn, p.sig ? &fcode : nullptr);
    if (p.sig) sig_put(p, bx.coff + t, 62, fcode);
    for (int q = 0; q < NPR; ++q) P[q * bx.ntot + t] = Pn[q];
  }
}

// --------------------------------------------------------------- CFL dt
// dt = C min_zones 1 / sum_d (v_d/dx_d), v_d = larger face speed of the zone
// along d, per grid.  Block minimum by warp shuffles, then one atomicMin on
// the bit pattern (positive doubles order like unsigned integers).
template <typename R>
__global__ void k_cfl(DevParams p, const BoxGeo* __restrict__ boxes, int nbox, Bufs b) {
  __shared__ double sm[32];
  for (int bi = 0; bi < nbox; ++bi) {
    const BoxGeo& bx = boxes[bi];
    double best = HUGE_VAL;
    for (long long z = first_item(bx.aoff); z < bx.nact; z += HR_STRIDE) {
      long long r = z;
      int i = (int)(r % bx.n[0]);
      r /= bx.n[0];
      int j = (int)(r % bx.n[1]);
      int k = (int)(r / bx.n[1]);
      long long t = cell_index(bx, i, j, k);
      double sum = 0.0;
      for (int d = 0; d < 3; ++d) {
        if (bx.n[d] == 1) continue;
        const R* sp = (const R*)b.spd[d] + bx.coff;
        double v = fmax((double)sp[t], (double)sp[t + bx.str[d]]);
        sum += v / bx.dx[d];
      }
      if (sum > 0.0) best = fmin(best, 1.0 / sum);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) best = fmin(best, __shfl_down_sync(0xffffffffu, best, o));
    int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    __syncthreads();
    if (lane == 0) sm[w] = best;
    __syncthreads();
    if (w == 0) {
      best = lane < (int)(blockDim.x >> 5) ? sm[lane] : HUGE_VAL;
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) best = fmin(best, __shfl_down_sync(0xffffffffu, best, o));
      if (lane == 0 && best < HUGE_VAL)
        atomicMin(&b.dtmin[bi], (unsigned long long)__double_as_longlong(best));
    }
  }
}

static __global__ void k_cfl_init(Bufs b, int nbox) {
  for (int i = threadIdx.x; i < nbox; i += blockDim.x) b.dtmin[i] = 0x7FF0000000000000ULL;  // +inf
}

static __global__ void k_cfl_finish(DevParams p, Bufs b, int nbox) {
  for (int i = threadIdx.x; i < nbox; i += blockDim.x)
    b.dt[i] = p.courant * __longlong_as_double((long long)b.dtmin[i]);
}

}  // namespace hr

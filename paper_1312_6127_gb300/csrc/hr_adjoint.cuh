// Adjoint (reverse-mode derivative) of one full RK3 step, FP64, one grid.
//
// The reverse sweep visits the sub-steps of Sec. 4.1-4.2 in reverse order and,
// inside each, the operations of the sub-step in reverse: implicit solve,
// explicit update, flux-CT, Riemann fluxes, reconstruction, flattener, cell
// factors and ghost fill.  Each kernel applies the transpose of its forward
// operation's local Jacobian to the incoming cotangent along the branches
// (limiters, wave-speed maxima, flattener clamps) that the forward step took:
// by a reverse sweep written out by hand for the fluxes, the reconstruction,
// the explicit update and the implicit solve; by evaluating the forward device
// functions on dual numbers (Dn<N>) for the flattener, the cell factors, the
// floors where one acts, and the zones that the entropy equation solved.
//
// The implicit solve is differentiated through its solution, not through the
// Newton iterations (implicit-function theorem): at the root x* of the PMHD
// error E(x; U*, kappa) = 0, dx*/dU* = -J_x^{-1} dE/dU*, so the cotangent of
// U* is  gU = (dP/dU*)^T gP - (dE/dU*)^T lambda  with  J_x^T lambda = (dP/dx)^T gP,
// one transposed 4x4 solve per zone.  The floors act on the solution: their
// Jacobian (identity for the components they leave alone, the derivative of
// the floor value for those they set) is applied first.  Zones that took the
// neighbour-average back-up pass their cotangent to the neighbours they
// averaged (B, which is U*[B]/sqrt(-g), excepted).  The time step is held
// fixed.
#pragma once
#include "hr_kernels.cuh"

namespace hr {

struct AdjBufs {
  double* Pst;          // [4][12][ntot] sub-step inputs P_0, P_1, P_2 and the result P^{n+1}
  double* chi;          // [3][3][2][ntot] flattener after sub-step s, per direction (PPM)
  double* Ust;          // [3][12][nact] U* of every zone and sub-step
  unsigned char* meth;  // [3][nact] outcome per sub-step: 0 PMHD, 1 URAD, 2 back-up, 3 entropy
  double* Psol;         // [3][12][nact] solution of every zone before the floors
  double* gP;           // [12][ntot] cotangent of the current sub-step's input (ghosts included)
  double* gN;           // [12][nact] cotangent of the current sub-step's output
  double* gUn;          // [12][nact] cotangent of U^n
  double* gU;           // [12][nact] cotangent of U*
  double* gX;           // [12][nact] cotangent of the explicit rate X
  double* gF[3];        // [12][ntot] cotangent of the face fluxes
  double* gE;           // [24][ntot] cotangent of the reconstructed edges of one direction
  double* gchi;         // [2][ntot] cotangent of the flattener used by one direction's edges
  double* carry;        // [3][2][ntot] flattener cotangent passed to the earlier sub-step
  double* gaux;         // [3][ntot] cotangent of sqrt(-g) u^d (gas, rad) and w_d of one direction
  double* gemf;         // [ntot] cotangent of the edge EMFs of one pair of directions
  double* gk;           // [1] cotangent of kappa_scale
  // the entropy (Sec. 2, Eq. S), for zones solved by the entropy equation
  double* Sst;          // [3][nact] explicit entropy S* of the zones whose retry read it (valid where meth is 3)
  double* gS;           // [nact] cotangent of S*
  double* gSn;          // [nact] cotangent of S^n, the step's initial conserved entropy
  double* gXS;          // [nact] cotangent of the entropy's explicit rate X_S = -div F_S
  double* gFS[3];       // [ntot] cotangent of the entropy face fluxes
};

__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// Adds v of every lane of a full warp to *dst (one atomic per warp).  Called
// by all 32 lanes (no early exit between the grid-stride loop and this call).
__device__ __forceinline__ void warp_atomic_add(double* dst, double v) {
  v = warp_sum(v);
  if ((threadIdx.x & 31) == 0 && v != 0.0) atomicAdd(dst, v);
}

__device__ __forceinline__ void zone_ijk(const BoxGeo& bx, long long z, int& i, int& j, int& k) {
  long long r = z;
  i = (int)(r % bx.n[0]);
  r /= bx.n[0];
  j = (int)(r % bx.n[1]);
  k = (int)(r / bx.n[1]);
}

__device__ __forceinline__ long long zone_of(const BoxGeo& bx, int i, int j, int k) {
  return ((long long)k * bx.n[1] + j) * bx.n[0] + i;
}

// Sets *flag when any of the n method records equals m.
static __global__ void ka_find_meth(const unsigned char* __restrict__ meth, long long n, unsigned char m, int* flag) {
  for (long long z = HR_TID; z < n; z += HR_STRIDE)
    if (meth[z] == m) *flag = 1;
}

// ------------------------------------------------------------ back-up (T)
// A back-up zone's non-B primitives are the average of its good neighbours'
// solutions: its cotangent moves to those neighbours.
static __global__ void ka_backup_T(BoxGeo bx, const unsigned char* __restrict__ meth, double* gN) {
  for (long long z = HR_TID; z < bx.nact; z += HR_STRIDE) {
    if (meth[z] != 2) continue;
    int ii[3];
    zone_ijk(bx, z, ii[0], ii[1], ii[2]);
    long long nb_z[6];
    int ng = 0;
    for (int d = 0; d < 3; ++d) {
      if (bx.n[d] == 1) continue;
      for (int side = -1; side <= 1; side += 2) {
        int nb[3] = {ii[0], ii[1], ii[2]};
        nb[d] += side;
        if (nb[d] < 0 || nb[d] >= bx.n[d]) continue;
        long long zn = zone_of(bx, nb[0], nb[1], nb[2]);
        if (meth[zn] != 2) nb_z[ng++] = zn;
      }
    }
    for (int q = 0; q < NPR; ++q) {
      if (q >= B1 && q <= B3) continue;
      double g = gN[q * bx.nact + z];
      gN[q * bx.nact + z] = 0.0;
      if (ng == 0 || g == 0.0) continue;
      g /= ng;
      for (int e = 0; e < ng; ++e) atomicAdd(&gN[q * bx.nact + nb_z[e]], g);
    }
  }
}

// ------------------------------------------------------------- frames (T)
// 4-velocities, field and b^2 of a state transposed (FaceSide, Frame): from the
// cotangents of u^t, u^1, u_t, u_i, B_t, B_i, b^t, 1/u^t, b^2 and the radiation's
// u^t, u^1, u_t, u_i to those of u~^i, B^i and u~_rad^i (added to gP).
template <int MET, class S>
__device__ __forceinline__ void gas_frame_T(const Geo<MET, double>& g, double a01, double b1, const S& s,
                                            const double P[NPR], double gu0, double gu1, double gl0,
                                            const double gl[3], double gm0, const double gmv[3], double gbt,
                                            double giut, double gbsq, double gP[NPR]) {
  const double ia = MET == MINK ? 1.0 : g.ialpha, al = MET == MINK ? 1.0 : g.alpha;
  const double gBB = gbsq * (s.iut * s.iut);
  gbt = fma(2.0 * gBB, s.bt, gbt);
  giut = fma(2.0 * gbsq, s.bsq * rcp(s.iut), giut);
  // gamma: u^t = gamma / alpha, u^1 = u~^1 - gamma a01, u_t = b1 l_1 - alpha gamma, 1/u^t = alpha / gamma
  double ggm = fma(-giut * s.iut, s.igm, gu0 * ia) - al * gl0;
  ggm = fma(-gu1, a01, ggm);
  gP[U1] += gu1;
  const double gg = 0.5 * ggm * s.igm;
  double a[3], b[3], t[3];
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    gP[B1 + i] = fma(gbt, s.l[i], fma(gBB, s.m[i], gP[B1 + i]));
    a[i] = fma(gbt, P[B1 + i], fma(gg, P[U1 + i], gl[i]));
    b[i] = fma(gBB, P[B1 + i], gmv[i]);
    gP[U1 + i] = fma(gg, s.l[i], gP[U1 + i]);
  }
  a[0] = fma(b1, gl0, a[0]);
  b[0] = fma(b1, gm0, b[0]);
  lower3<MET>(g, a[0], a[1], a[2], t);
#pragma unroll
  for (int i = 0; i < 3; ++i) gP[U1 + i] += t[i];
  lower3<MET>(g, b[0], b[1], b[2], t);
#pragma unroll
  for (int i = 0; i < 3; ++i) gP[B1 + i] += t[i];
}
template <int MET, class S>
__device__ __forceinline__ void frame_T(const Geo<MET, double>& g, double a01, double b1, const S& s,
                                        const double P[NPR], double gu0, double gu1, double gl0, const double gl[3],
                                        double gm0, const double gmv[3], double gbt, double giut, double gbsq,
                                        double gr0, double gr1, double gk0, const double gk[3], double gP[NPR]) {
  gas_frame_T<MET>(g, a01, b1, s, P, gu0, gu1, gl0, gl, gm0, gmv, gbt, giut, gbsq, gP);
  const double ia = MET == MINK ? 1.0 : g.ialpha, al = MET == MINK ? 1.0 : g.alpha;
  double a[3], t[3];
  gP[UR1] += gr1;
  const double ggr = fma(-gr1, a01, fma(gr0, ia, -al * gk0));
  const double gq = 0.5 * ggr * rcp(s.gr);
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    gP[UR1 + i] = fma(gq, s.k[i], gP[UR1 + i]);
    a[i] = fma(gq, P[UR1 + i], gk[i]);
  }
  a[0] = fma(b1, gk0, a[0]);
  lower3<MET>(g, a[0], a[1], a[2], t);
#pragma unroll
  for (int i = 0; i < 3; ++i) gP[UR1 + i] += t[i];
}

// The frames of a zone's state, as FaceSide forms them.
template <int MET>
struct Frame {
  double gm, igm, gr, u0, u1, l0, l[3], bt, m0, m[3], iut, bsq, r0, r1, k0, k[3];
  __device__ __forceinline__ Frame(const Geo<MET, double>& g, double a01, double b1, const double P[NPR]) {
    const double ia = MET == MINK ? 1.0 : g.ialpha, al = MET == MINK ? 1.0 : g.alpha;
    lower3<MET>(g, P[U1], P[U2], P[U3], l);
    lower3<MET>(g, P[B1], P[B2], P[B3], m);
    lower3<MET>(g, P[UR1], P[UR2], P[UR3], k);
    gm = sqrt_rsqrt(fma(P[U1], l[0], fma(P[U2], l[1], fma(P[U3], l[2], 1.0))), &igm);
    gr = sqrt64(fma(P[UR1], k[0], fma(P[UR2], k[1], fma(P[UR3], k[2], 1.0))));
    bt = fma(P[B1], l[0], fma(P[B2], l[1], P[B3] * l[2]));
    u0 = gm * ia;
    u1 = fma(-gm, a01, P[U1]);
    l0 = fma(b1, l[0], -al * gm);
    iut = al * igm;
    m0 = b1 * m[0];
    r0 = gr * ia;
    r1 = fma(-gr, a01, P[UR1]);
    k0 = fma(b1, k[0], -al * gr);
    bsq = fma(bt, bt, fma(P[B1], m[0], fma(P[B2], m[1], P[B3] * m[2]))) * (iut * iut);
  }
};

// U(P) and the geometric source of cons_source64 transposed: gU the cotangents
// of U, gX those of the source rows (2, 3 gas, 9, 10 radiation), gs that of the
// conserved entropy U_rho s; md the scaled metric derivatives.  Adds to gP.
template <int MET>
__device__ __forceinline__ void cons_T(const DevParams& p, const Geo<MET, double>& g, const MetricDeriv& md,
                                       const double P[NPR], const double gU[NPR], const double gX[NPR], double gs,
                                       double gP[NPR]) {
  const double a01 = MET == MINK ? 0.0 : g.alpha * g.G01, b1 = MET == MINK ? 0.0 : g.alpha * a01;
  const Frame<MET> s(g, a01, b1, P);
  const double wb = P[RHO] + fma(p.gam, P[UU], s.bsq), bu = s.bt * s.iut, wu = wb * s.u0, Z = fma(-s.bt, bu, wu);
  const double E = P[ER], e43 = (4.0 / 3.0) * E, er = e43 * s.r0;
  double o[NPR];
#pragma unroll
  for (int q = 0; q < NPR; ++q) o[q] = g.gdet * gU[q];
  double gmt = o[0] + o[1], gpt = o[1], gZ = o[1] * s.l0, gbu = -o[1] * s.m0, gl0 = o[1] * Z, gm0 = -o[1] * bu;
  double ger = o[8] * s.k0, gk0 = o[8] * er, ge13 = o[8], gl[3], gmv[3], gk[3];
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    gZ = fma(o[2 + i], s.l[i], gZ);
    gbu = fma(-o[2 + i], s.m[i], gbu);
    gl[i] = o[2 + i] * Z;
    gmv[i] = -o[2 + i] * bu;
    ger = fma(o[9 + i], s.k[i], ger);
    gk[i] = o[9 + i] * er;
    gP[B1 + i] += o[5 + i];
  }
  double gwb = 0.0, gu0 = 0.0, gu1 = 0.0, gbt = 0.0, giut = 0.0, gr0 = 0.0, gr1 = 0.0, ge43 = 0.0;
  if (gs != 0.0) {  // U_rho s: d s = n d ug / ug - (n + 1) d rho / rho
    const double n = 1.0 / (p.gam - 1.0), w = gs * g.gdet * P[RHO] * s.u0;
    gmt = fma(gs * g.gdet, entropy_per_baryon<double>(p, P[RHO], P[UU]), gmt);
    gP[UU] += w * n / P[UU];
    gP[RHO] -= w * (n + 1.0) / P[RHO];
  }
  if constexpr (MET == KS) {
    const double* dm = reinterpret_cast<const double*>(&md);
    const double u2 = P[U2], u3 = P[U3], r2 = P[UR2], r3 = P[UR3];
    const double c1 = fma(s.bt, s.u1, P[B1]) * s.iut, c2 = fma(s.bt, u2, P[B2]) * s.iut,
                 c3 = fma(s.bt, u3, P[B3]) * s.iut;  // b^i
    double G[7], H[7];
#pragma unroll
    for (int c = 0; c < 7; ++c) {
      G[c] = fma(gX[2], dm[2 * c], gX[3] * dm[2 * c + 1]);
      H[c] = fma(gX[9], dm[2 * c], gX[10] * dm[2 * c + 1]);
    }
    gpt += fma(gX[2], md.sg[0], gX[3] * md.sg[1]);
    ge13 += fma(gX[9], md.sg[0], gX[10] * md.sg[1]);
    // contractions G(v) of a vector and their halved gradients
    const double a0 = fma(G[0], s.u0, 0.5 * fma(G[1], s.u1, G[2] * u3));
    const double a1 = fma(G[3], s.u1, 0.5 * fma(G[1], s.u0, G[4] * u3));
    const double a2 = G[5] * u2, a3 = fma(G[6], u3, 0.5 * fma(G[2], s.u0, G[4] * s.u1));
    gwb += a0 * s.u0 + a1 * s.u1 + a2 * u2 + a3 * u3;
    gu0 += 2.0 * wb * a0;
    gu1 += 2.0 * wb * a1;
    gP[U2] += 2.0 * wb * a2;
    gP[U3] += 2.0 * wb * a3;
    const double d0 = -2.0 * fma(G[0], s.bt, 0.5 * fma(G[1], c1, G[2] * c3));
    const double d1 = -2.0 * fma(G[3], c1, 0.5 * fma(G[1], s.bt, G[4] * c3));
    const double d2 = -2.0 * G[5] * c2, d3 = -2.0 * fma(G[6], c3, 0.5 * fma(G[2], s.bt, G[4] * c1));
    // b^i = (B^i + b^t u^i) / u^t
    gbt += d0 + s.iut * (d1 * s.u1 + d2 * u2 + d3 * u3);
    const double bi = s.bt * s.iut;
    gu1 = fma(d1, bi, gu1);
    gP[U2] = fma(d2, bi, gP[U2]);
    gP[U3] = fma(d3, bi, gP[U3]);
    gP[B1] = fma(d1, s.iut, gP[B1]);
    gP[B2] = fma(d2, s.iut, gP[B2]);
    gP[B3] = fma(d3, s.iut, gP[B3]);
    giut += (d1 * c1 + d2 * c2 + d3 * c3) * rcp(s.iut);
    const double e0 = fma(H[0], s.r0, 0.5 * fma(H[1], s.r1, H[2] * r3));
    const double e1 = fma(H[3], s.r1, 0.5 * fma(H[1], s.r0, H[4] * r3));
    const double e2 = H[5] * r2, e3 = fma(H[6], r3, 0.5 * fma(H[2], s.r0, H[4] * s.r1));
    ge43 += e0 * s.r0 + e1 * s.r1 + e2 * r2 + e3 * r3;
    gr0 += 2.0 * e43 * e0;
    gr1 += 2.0 * e43 * e1;
    gP[UR2] += 2.0 * e43 * e2;
    gP[UR3] += 2.0 * e43 * e3;
  }
  ge43 = fma(ger, s.r0, ge43);
  gr0 = fma(ger, e43, gr0);
  gP[ER] += fma(4.0 / 3.0, ge43, ge13 * (1.0 / 3.0));
  // Z = wu - b^t bu, bu = b^t / u^t, wu = wb u^t, mt = rho u^t
  gbt = fma(-gZ, bu, gbt);
  gbu = fma(-gZ, s.bt, gbu);
  gbt = fma(gbu, s.iut, gbt);
  giut = fma(gbu, s.bt, giut);
  gwb = fma(gZ, s.u0, gwb);
  gu0 = fma(gZ, wb, fma(gmt, P[RHO], gu0));
  gP[RHO] += fma(gmt, s.u0, gwb);
  gP[UU] += fma(p.gam, gwb, p.gm1 * gpt);
  frame_T<MET>(g, a01, b1, s, P, gu0, gu1, gl0, gl, gm0, gmv, gbt, giut, gwb + 0.5 * gpt, gr0, gr1, gk0, gk, gP);
}

// Metric and scaled metric derivatives of the centre of cell (i, j).
template <int MET>
__device__ __forceinline__ Geo<MET, double> centre_tables(const DevParams& p, const BoxGeo& bx, const double* geo,
                                                          int i, int j, MetricDeriv* md) {
  if constexpr (MET == KS) {
    const GeoTab T = geotab(geo, bx);
    const long long x = gidx_c(bx, i, j);
    *md = md_load(T.M, T.sC, x);
    return geo_load<MET>(T.C, T.sC, x);
  } else {
    return make_geo<MET, double>(p, 0.0, 0.0);
  }
}

// ------------------------------------------------------- implicit solve (T)
// The error function and the final primitives of a zone at its solution
// (pmhd_res64), with every intermediate the reverse sweep reads.
template <int MET>
struct PmhdEval {
  double l[3], gm, igm, u0, iut, l0, rho, bt, bu, bsq, pg, pt, wb, Z, m0, m[3];
  double Rt[4], t[3], Er, ie, U2, y, sq, sm1, sp2, rr, E, fa, gr, v0, v[3];
  double T, ka, ksca, kt, uru, e43, c1, c2, lam, hA, hC;  // ka: absorption over kappa_scale
  bool neg, lim;

  __device__ __forceinline__ PmhdEval(const DevParams& p, const ImpSys<MET>& s, const double x[4]) {
    const auto& g = s.g;
    const auto& c = s.pre;
    const double al = MET == MINK ? 1.0 : g.alpha;
    lower3<MET>(g, x[1], x[2], x[3], l);
    gm = sqrt_rsqrt(fma(x[1], l[0], fma(x[2], l[1], fma(x[3], l[2], 1.0))), &igm);
    u0 = MET == MINK ? gm : gm * g.ialpha;
    iut = al * igm;
    l0 = fma(c.b1, l[0], -al * gm);
    rho = s.Dlab * iut;
    bt = fma(s.B[0], l[0], fma(s.B[1], l[1], s.B[2] * l[2]));
    bu = bt * iut;
    bsq = fma(bt, bt, c.BB) * (iut * iut);
    pg = p.gm1 * x[0];
    pt = fma(0.5, bsq, pg);
    wb = rho + fma(p.gam, x[0], bsq);
    Z = fma(-bt, bu, wb * u0);
    m0 = c.m0;
    for (int k = 0; k < 3; ++k) m[k] = c.m[k];
    Rt[0] = s.Rs[0] - (fma(rho, u0, fma(Z, l0, fma(-bu, m0, pt))) - s.Ts[0]);
#pragma unroll
    for (int k = 0; k < 3; ++k) Rt[1 + k] = s.Rs[1 + k] - (fma(Z, l[k], -bu * m[k]) - s.Ts[1 + k]);
    raise3(g, c, Rt + 1, t);
    U2 = c.a2 * fma(Rt[1], t[0], fma(Rt[2], t[1], Rt[3] * t[2]));
    Er = fma(c.b1, Rt[1], -Rt[0]);
    neg = !(Er > 0.0);
    y = neg ? HUGE_VAL : (U2 > 0.0 ? U2 / (Er * Er) : 0.0);
    lim = y > p.ymax_rad;
    if (lim) {
      Er = 1e-150 + sqrt(U2 / p.ymax_rad);
      y = U2 / (Er * Er);
    }
    ie = 1.0 / Er;
    sq = sqrt64(fma(-3.0, y, 4.0));
    sm1 = sq - 1.0;
    sp2 = sq + 2.0;
    rr = rsqrt64(sp2 * sm1);
    E = Er * sm1;
    fa = 1.5 * ie * rr * al;
    gr = 0.5 * sp2 * rr;
#pragma unroll
    for (int k = 0; k < 3; ++k) v[k] = fa * Rt[1 + k];
    v0 = fma(c.b1, v[0], -al * gr);
    T = pg * u0 * s.iDlab;
    if (p.opacity == 2) {
      ka = s.kf;
    } else if (p.opacity == 1) {
      const double Tl = T > p.Tmin ? T : p.Tmin, T2 = Tl * Tl;
      ka = p.kabs0 * rho * rho * rsqrt64(T2 * T2 * T2 * Tl);
    } else {
      ka = p.kabs0 * rho;
    }
    ksca = s.ks * p.kes0 * rho;
    kt = fma(s.ks, ka, ksca);
    uru = fma(v[0], x[1], fma(v[1], x[2], fma(v[2], x[3], -gr * gm)));
    e43 = (4.0 / 3.0) * E;
    c1 = e43 * uru;
    c2 = E * (1.0 / 3.0);
    lam = s.ks * ka * p.a_rad * (T * T) * (T * T);
    hA = -s.h * (kt * c1);
    hC = -s.h * (fma(kt, c2, lam) + ksca * fma(c1, uru, -c2));
  }
  // gamma^{ij} w_j
  __device__ __forceinline__ static void raise3(const Geo<MET, double>& g, const ImpPre<double>& c, const double w[3],
                                                double o[3]) {
    if constexpr (MET == MINK) {
      for (int k = 0; k < 3; ++k) o[k] = w[k];
    } else {
      o[0] = fma(g.G13, w[2], c.c11 * w[0]);
      o[1] = g.G22 * w[1];
      o[2] = fma(g.G33, w[2], g.G13 * w[0]);
    }
  }

  // Reverse sweep: gE the cotangents of the error rows, gp those of the final
  // primitives -> gx of x, gU of U* (times sqrt(-g)), *gks of kappa_scale.
  __device__ __forceinline__ void reverse(const DevParams& p, const ImpSys<MET>& s, const double x[4],
                                          const double gE[4], const double gp[NPR], double gx[4], double gU[NPR],
                                          double* gks) const {
    const auto& g = s.g;
    const auto& c = s.pre;
    const double al = MET == MINK ? 1.0 : g.alpha, a01 = MET == MINK ? 0.0 : g.alpha * g.G01;
    double gEf = 0.0, gfa = 0.0, gt[3] = {0.0, 0.0, 0.0};
    if (!neg) {
      gEf = gp[ER];
#pragma unroll
      for (int k = 0; k < 3; ++k) {
        gfa = fma(gp[UR1 + k], t[k], gfa);
        gt[k] = gp[UR1 + k] * fa;
      }
    }
    // E_k = dT_k - hG_k, hG = hA v + hC u
    const double ghA = -fma(gE[0], v0, fma(gE[1], v[0], fma(gE[2], v[1], gE[3] * v[2])));
    const double ghC = -fma(gE[0], l0, fma(gE[1], l[0], fma(gE[2], l[1], gE[3] * l[2])));
    const double gv0 = -gE[0] * hA;
    double gl0 = -gE[0] * hC, gv[3], gl[3];
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      gv[k] = -gE[1 + k] * hA;
      gl[k] = -gE[1 + k] * hC;
    }
    // four-force
    const double hc = -s.h * ghC, ha = -s.h * ghA, T3 = T * T * T;
    const double gc1 = fma(ha, kt, hc * ksca * uru), gkt = fma(ha, c1, hc * c2), gc2 = hc * (kt - ksca);
    const double gka = fma(hc * p.a_rad, T3 * T, gkt), gks_ = fma(hc, fma(c1, uru, -c2), gkt);  // of ks ka, ks kes0 rho
    double guru = fma(hc * ksca, c1, gc1 * e43);
    double gT = 4.0 * hc * s.ks * ka * p.a_rad * T3;
    *gks += fma(gka, ka, gks_ * p.kes0 * rho);
    double grho = fma(gks_ * s.ks, p.kes0, gp[RHO]);
    if (p.opacity == 1) {
      grho = fma(2.0 * gka * s.ks, ka / rho, grho);
      if (T > p.Tmin) gT = fma(-3.5 * gka * s.ks, ka / T, gT);
    } else if (p.opacity == 0) {
      grho = fma(gka * s.ks, p.kabs0, grho);
    }
    const double gpg = gT * u0 * s.iDlab;
    double gu0 = gT * pg * s.iDlab, gD = -gT * pg * u0 * (s.iDlab * s.iDlab);
    gEf += fma(gc1 * uru, 4.0 / 3.0, gc2 * (1.0 / 3.0));
    // u_r.u = v_i u~^i - gamma_r gamma
    double ggr = fma(-guru, gm, -al * gv0);
    const double ggm = -guru * gr;
    gv[0] = fma(c.b1, gv0, gv[0]);
    double gR[4];
    gR[0] = 0.0;
    double gxu[3];
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      gxu[k] = guru * v[k];
      gv[k] = fma(guru, x[1 + k], gv[k]);
      gfa = fma(gv[k], Rt[1 + k], gfa);
      gR[1 + k] = gv[k] * fa;
    }
    // radiation frame
    double gie = 1.5 * gfa * rr * al;
    const double grr = fma(1.5 * gfa * ie, al, 0.5 * ggr * sp2), gpr = -0.5 * rr * rr * rr * grr;
    const double gsp2 = fma(0.5 * ggr, rr, gpr * sm1), gsm1 = fma(gpr, sp2, gEf * Er);
    double gEr = gEf * sm1, gU2;
    if (lim) {
      gEr = fma(-gie, ie * ie, gEr);
      gU2 = 0.5 * gEr * ie / p.ymax_rad;
    } else {
      const double gy = -1.5 * (gsp2 + gsm1) * rcp(sq);
      gU2 = gy * ie * ie;
      gie = fma(2.0 * gy * U2, ie, gie);
      gEr = fma(-gie, ie * ie, gEr);
      gR[0] -= gEr;
      gR[1] = fma(c.b1, gEr, gR[1]);
    }
    double rt[3];
    raise3(g, c, gt, rt);
#pragma unroll
    for (int k = 0; k < 3; ++k) gR[1 + k] += fma(2.0 * gU2 * c.a2, t[k], rt[k]);
    // R = R* - (T - T*): T's and the conserved inputs' cotangents
    double gTc[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      gTc[k] = gE[k] - gR[k];
      gU[UU + k] = -gTc[k];
      gU[ER + k] = gR[k];
    }
    double gZ = gTc[0] * l0, gbu = -gTc[0] * m0, gmv[3];
    const double gm0 = -gTc[0] * bu;
    gl0 = fma(gTc[0], Z, gl0);
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      gZ = fma(gTc[1 + k], l[k], gZ);
      gbu = fma(-gTc[1 + k], m[k], gbu);
      gl[k] = fma(gTc[1 + k], Z, gl[k]);
      gmv[k] = -gTc[1 + k] * bu;
    }
    const double gwb = gZ * u0, gpt = gTc[0];
    gu0 = fma(gZ, wb, fma(gTc[0], rho, gu0));
    grho += fma(gTc[0], u0, gwb);
    double gbt = -gZ * bu;
    gbu = fma(-gZ, bt, gbu);
    gbt = fma(gbu, iut, gbt);
    double giut = fma(gbu, bt, grho * s.Dlab);
    gD = fma(grho, iut, gD);
    gx[0] = gp[UU] + fma(p.gam, gwb, p.gm1 * (gpt + gpg));
    double P[NPR], gP[NPR];
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      P[U1 + k] = x[1 + k];
      P[B1 + k] = s.B[k];
      gP[U1 + k] = gp[U1 + k] + gxu[k];
      gP[B1 + k] = gp[B1 + k];
    }
    gas_frame_T<MET>(g, a01, c.b1, *this, P, fma(ggm, al, gu0), 0.0, gl0, gl, gm0, gmv, gbt, giut,
                     fma(0.5, gpt, gwb), gP);
    gU[RHO] = gD;
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      gx[1 + k] = gP[U1 + k];
      gU[B1 + k] = gP[B1 + k];
    }
  }
};

// Bound by FP64 instructions (64x32x16 torus, per step: 1.64 ms on dual numbers
// over sixteen inputs, 0.47 so).
// One zone per thread: the floors' transpose (identity unless one acts), then
// the implicit-function theorem with reverse sweeps of PmhdEval: four for the
// rows of dE/dx, one for the primitives, one for the solved lambda.  Zones
// solved by the entropy equation follow in ka_implicit_entropy.
template <int MET>
__global__ void __launch_bounds__(128) ka_implicit(DevParams p, BoxGeo bx, AdjBufs a, int s, double dt,
                                                   const double* __restrict__ K, const double* __restrict__ geo) {
  const double Bc = s == 0 ? 1.0 : (s == 1 ? 0.25 : 2.0 / 3.0);
  const double h = Bc * dt;
  const double* Ust0 = a.Ust + (long long)s * 12 * bx.nact;
  const unsigned char* meth = a.meth + (long long)s * bx.nact;
  const double* Psol0 = a.Psol + (long long)s * 12 * bx.nact;
  double gk = 0.0;
  for (long long z = HR_TID; z < bx.nact; z += HR_STRIDE) {
    double gq[NPR];
    bool any = false;
#pragma unroll
    for (int q = 0; q < NPR; ++q) {
      gq[q] = a.gN[q * bx.nact + z];
      any = any || gq[q] != 0.0;
      a.gU[q * bx.nact + z] = 0.0;
    }
    a.gS[z] = 0.0;
    const int m = meth[z];
    if (!any || m == METH_ENTROPY) continue;
    int i, j, k;
    zone_ijk(bx, z, i, j, k);
    const long long t = cell_index(bx, i, j, k);
    Geo<MET, double> g;
    double igd = 1.0, fl[2] = {p.rf0, p.uf0};
    const double sgk[3] = {1.0, 1.0, 1.0};  // the error's norms are not read here
    if constexpr (MET == KS) {
      const GeoTab T = geotab(geo, bx);
      const long long x = gidx_c(bx, i, j);
      g = geo_load<MET>(T.C, T.sC, x);
      igd = __ldg(T.C + 16 * T.sC + x);
      fl[0] = __ldg(T.C + 23 * T.sC + x);
      fl[1] = __ldg(T.C + 24 * T.sC + x);
    } else {
      g = make_geo<MET, double>(p, 0.0, 0.0);
    }
    if (m == ST_BACKUP) {  // only B = U*[B] / sqrt(-g) is the zone's own
      for (int c = 0; c < 3; ++c) a.gU[(B1 + c) * bx.nact + z] = gq[B1 + c] * igd;
      continue;
    }
    double Us[NPR], Ps[NPR];
#pragma unroll
    for (int q = 0; q < NPR; ++q) {
      Us[q] = Ust0[q * bx.nact + z];
      Ps[q] = Psol0[q * bx.nact + z];
    }
    {  // floors: gq <- (d floors / d P)^T gq at the solution
      double Pf[NPR];
      bool acts = false;
      for (int q = 0; q < NPR; ++q) Pf[q] = Ps[q];
      apply_floors<MET>(p, g, fl[0], fl[1], Pf);
#pragma unroll
      for (int q = 0; q < NPR; ++q) acts = acts || Pf[q] != Ps[q];
      if (acts) {
        typedef Dn<4> D4;
        const Geo<MET, D4> g4 = geo_cast<D4>(g);
        double gs[NPR];
#pragma unroll 1
        for (int ch = 0; ch < 3; ++ch) {
          D4 PD[NPR];
          for (int q = 0; q < NPR; ++q) PD[q] = D4::seed(Ps[q], q - 4 * ch);
          apply_floors<MET, D4>(p, g4, fl[0], fl[1], PD);
          for (int c = 0; c < 4; ++c) {
            double v = 0.0;
            for (int q = 0; q < NPR; ++q) v += gq[q] * PD[q].d[c];
            gs[4 * ch + c] = v;
          }
        }
        for (int q = 0; q < NPR; ++q) gq[q] = gs[q];
      }
    }
    ImpSys<MET> sys;
    build_sys_with<MET, double>(p, g, igd, sgk, Us, h, kfield(p, K, t), sys);
    const double x[4] = {Ps[UU], Ps[U1], Ps[U2], Ps[U3]};
    const PmhdEval<MET> ev(p, sys, x);
    double J[4][4], lam[4], gx[4], gU[NPR], sum[NPR], ks = 0.0;
    bool ok = true;
#pragma unroll 1
    for (int it = 0; it < 6; ++it) {
      double gE[4], gp[NPR];
#pragma unroll
      for (int c = 0; c < 4; ++c) gE[c] = it < 4 ? (c == it ? 1.0 : 0.0) : (it == 4 ? 0.0 : -lam[c]);
#pragma unroll
      for (int q = 0; q < NPR; ++q) gp[q] = it == 4 ? gq[q] : 0.0;
      ks = 0.0;
      ev.reverse(p, sys, x, gE, gp, gx, gU, &ks);
      if (it < 4) {
#pragma unroll
        for (int r = 0; r < 4; ++r)
          if (r == it)
            for (int c = 0; c < 4; ++c) J[c][r] = gx[c];  // transposed
      } else if (it == 4) {
        for (int q = 0; q < NPR; ++q) sum[q] = gU[q];
        ok = solve4(J, gx, lam);
        if (!ok) break;
      }
    }
    if (!ok) continue;
    gk += ks;
#pragma unroll
    for (int q = 0; q < NPR; ++q) a.gU[q * bx.nact + z] = (sum[q] + gU[q]) * igd;
  }
  warp_atomic_add(a.gk, gk);
}

// The zones solved by the entropy equation (by the entropy PMHD, URAD or PRAD,
// which solve the same equations; few in any step), on dual numbers: the same
// transposed solve on the entropy system (Eq. source6), which also depends on
// S*.
template <int MET>
__global__ void ka_implicit_entropy(DevParams p, BoxGeo bx, AdjBufs a, int s, double dt,
                                    const double* __restrict__ K) {
  const double Bc = s == 0 ? 1.0 : (s == 1 ? 0.25 : 2.0 / 3.0);
  const double h = Bc * dt;
  const double* Ust0 = a.Ust + (long long)s * 12 * bx.nact;
  const unsigned char* meth = a.meth + (long long)s * bx.nact;
  const double* Psol0 = a.Psol + (long long)s * 12 * bx.nact;
  typedef Dn<4> D4;
  typedef Dn<1> D1;
  double gk = 0.0;
  for (long long z = HR_TID; z < bx.nact; z += HR_STRIDE) {
    if (meth[z] != METH_ENTROPY) continue;
    double gq[NPR];
    bool any = false;
    for (int q = 0; q < NPR; ++q) {
      gq[q] = a.gN[q * bx.nact + z];
      any = any || gq[q] != 0.0;
    }
    if (!any) continue;
    int i, j, k;
    zone_ijk(bx, z, i, j, k);
    const long long t = cell_index(bx, i, j, k);
    const double x1 = xcen(bx, 0, i), x2 = xcen(bx, 1, j);
    const Geo<MET, double> g = make_geo<MET, double>(p, x1, x2);
    const double igd = 1.0 / g.gdet;
    double Us[NPR], Ps[NPR];
    for (int q = 0; q < NPR; ++q) {
      Us[q] = Ust0[q * bx.nact + z];
      Ps[q] = Psol0[q * bx.nact + z];
    }
    const double kz = kfield(p, K, t);
    const double Sz = a.Sst[(long long)s * bx.nact + z];
    const Geo<MET, D4> g4 = geo_cast<D4>(g);
    {  // floors: gq <- (d floors / d P)^T gq at the solution
      double fl[2];
      floor_values<MET>(p, x1, &fl[0], &fl[1]);
      double gs[NPR];
      for (int ch = 0; ch < 3; ++ch) {
        D4 PD[NPR];
        for (int q = 0; q < NPR; ++q) PD[q] = D4::seed(Ps[q], q - 4 * ch);
        apply_floors<MET, D4>(p, g4, fl[0], fl[1], PD);
        for (int c = 0; c < 4; ++c) {
          double v = 0.0;
          for (int q = 0; q < NPR; ++q) v += gq[q] * PD[q].d[c];
          gs[4 * ch + c] = v;
        }
      }
      for (int q = 0; q < NPR; ++q) gq[q] = gs[q];
    }
    const double x[4] = {Ps[UU], Ps[U1], Ps[U2], Ps[U3]};
    double J[4][4], gx[4] = {0.0, 0.0, 0.0, 0.0};
    {  // derivatives with respect to x
      D4 xs[4], UsD[NPR], PsD[NPR], Eg[4];
      for (int c = 0; c < 4; ++c) xs[c] = D4::seed(x[c], c);
      for (int q = 0; q < NPR; ++q) UsD[q] = D4(Us[q]);
      ImpSysT<MET, D4> sys;
      build_sys<MET, D4>(p, g4, UsD, h, D4(kz), sys);
      sys.entropy = true;
      sys.Sstar = D4(Sz * igd);
      pmhd_final<MET, D4>(p, sys, xs, PsD, Eg);
      for (int r = 0; r < 4; ++r)
        for (int c = 0; c < 4; ++c) J[c][r] = Eg[r].d[c];  // transposed
      for (int q = 0; q < NPR; ++q)
        for (int c = 0; c < 4; ++c) gx[c] += gq[q] * PsD[q].d[c];
    }
    double lam[4];
    if (!solve4(J, gx, lam)) continue;
    double gU[NPR];
    for (int ch = 0; ch < 3; ++ch) {  // derivatives with respect to U*, four at a time
      D4 xs[4], UsD[NPR], PsD[NPR], Eg[4];
      for (int c = 0; c < 4; ++c) xs[c] = D4(x[c]);
      for (int q = 0; q < NPR; ++q) UsD[q] = D4::seed(Us[q], q - 4 * ch);
      ImpSysT<MET, D4> sys;
      build_sys<MET, D4>(p, g4, UsD, h, D4(kz), sys);
      sys.entropy = true;
      sys.Sstar = D4(Sz * igd);
      pmhd_final<MET, D4>(p, sys, xs, PsD, Eg);
      for (int c = 0; c < 4; ++c) {
        double v = 0.0;
        for (int q = 0; q < NPR; ++q) v += gq[q] * PsD[q].d[c];
        for (int r = 0; r < 4; ++r) v -= lam[r] * Eg[r].d[c];
        gU[4 * ch + c] = v;
      }
    }
    {  // derivative with respect to kappa_scale (E only; P depends on it through x*)
      const Geo<MET, D1> g1 = geo_cast<D1>(g);
      D1 xs[4], UsD[NPR], PsD[NPR], Eg[4];
      for (int c = 0; c < 4; ++c) xs[c] = D1(x[c]);
      for (int q = 0; q < NPR; ++q) UsD[q] = D1(Us[q]);
      ImpSysT<MET, D1> sys;
      build_sys<MET, D1>(p, g1, UsD, h, D1(kz), sys);
      sys.ks = D1::seed(p.kscale, 0);
      sys.entropy = true;
      sys.Sstar = D1(Sz * igd);
      pmhd_final<MET, D1>(p, sys, xs, PsD, Eg);
      for (int r = 0; r < 4; ++r) gk -= lam[r] * Eg[r].d[0];
    }
    for (int q = 0; q < NPR; ++q) a.gU[q * bx.nact + z] = gU[q];
    // S* enters the entropy row only, E_0 = T (S u^t(x) - S*/sqrt(-g)) +
    // h G_mu u^mu with T = p/rho0 at the solution (the factor F_13)
    a.gS[z] = lam[0] * ((p.gam - 1.0) * Ps[UU] / Ps[RHO]) * igd;
  }
  warp_atomic_add(a.gk, gk);
}

// --------------------------------------------------- explicit update (T)
// U* = a_s U^n + b_s (U(P_s) + dt X),  X = -sum_d dF_d/dx_d + SM(P_s).  Bound by
// FP64 instructions: one reverse sweep with tabulated metric, 64x32x16 torus per
// step 1.26 ms on three passes of dual numbers, 0.10 so.
template <int MET>
__global__ void __launch_bounds__(128) ka_update(DevParams p, BoxGeo bx, AdjBufs a, int s, double dt,
                                                 const double* __restrict__ Ps0, const double* __restrict__ geo) {
  const double A = s == 0 ? 0.0 : (s == 1 ? 0.75 : 1.0 / 3.0);
  const double Bc = s == 0 ? 1.0 : (s == 1 ? 0.25 : 2.0 / 3.0);
  for (long long z = HR_TID; z < bx.nact; z += HR_STRIDE) {
    double gq[NPR], gX[NPR], gP[NPR], P[NPR];
    bool any = false;
#pragma unroll
    for (int q = 0; q < NPR; ++q) {
      gq[q] = a.gU[q * bx.nact + z];
      any = any || gq[q] != 0.0;
      if (s > 0) a.gUn[q * bx.nact + z] += A * gq[q];
      a.gX[q * bx.nact + z] = Bc * dt * gq[q];
      gq[q] *= Bc;
      gX[q] = dt * gq[q];
      gP[q] = 0.0;
    }
    // S* = A S^n + Bc (S(P_s) + dt X_S), S(P) = U_rho(P) s_gas(P)
    const double gs = a.gS[z];
    any = any || gs != 0.0;
    if (s > 0) a.gSn[z] += A * gs;
    a.gXS[z] = Bc * dt * gs;
    int i, j, k;
    zone_ijk(bx, z, i, j, k);
    const long long t = cell_index(bx, i, j, k);
    if (any) {
      MetricDeriv md{};
      const Geo<MET, double> g = centre_tables<MET>(p, bx, geo, i, j, &md);
#pragma unroll
      for (int q = 0; q < NPR; ++q) P[q] = Ps0[q * bx.ntot + t];
      cons_T<MET>(p, g, md, P, gq, gX, Bc * gs, gP);
    }
#pragma unroll
    for (int q = 0; q < NPR; ++q) a.gP[q * bx.ntot + t] = gP[q];
  }
}

// U^n = U(P^n): gP^n += (dU/dP)^T gU^n at the end of the sweep.
template <int MET>
__global__ void __launch_bounds__(128) ka_un(DevParams p, BoxGeo bx, AdjBufs a, const double* __restrict__ P0,
                                             const double* __restrict__ geo) {
  for (long long z = HR_TID; z < bx.nact; z += HR_STRIDE) {
    double gq[NPR], gX[NPR], gP[NPR], P[NPR];
    bool any = false;
#pragma unroll
    for (int q = 0; q < NPR; ++q) {
      gq[q] = a.gUn[q * bx.nact + z];
      any = any || gq[q] != 0.0;
      gX[q] = gP[q] = 0.0;
    }
    const double gs = a.gSn[z];  // S^n = U_rho(P^n) s_gas(P^n)
    any = any || gs != 0.0;
    if (!any) continue;
    int i, j, k;
    zone_ijk(bx, z, i, j, k);
    const long long t = cell_index(bx, i, j, k);
    MetricDeriv md{};
    const Geo<MET, double> g = centre_tables<MET>(p, bx, geo, i, j, &md);
#pragma unroll
    for (int q = 0; q < NPR; ++q) P[q] = P0[q * bx.ntot + t];
    cons_T<MET>(p, g, md, P, gq, gX, gs, gP);
#pragma unroll
    for (int q = 0; q < NPR; ++q) a.gN[q * bx.nact + z] += gP[q];
  }
}

// ------------------------------------------------ flux divergence (T)
// Face range of the face kernel of direction d; the flux at cell t is the
// flux through t's lower face: +1/dx in X of zone t, -1/dx in X of zone t-s_d.
template <int d>
__global__ void ka_fluxgrad(BoxGeo bx, const double* __restrict__ gX, double* __restrict__ gF,
                            const double* __restrict__ gXS, double* __restrict__ gFS) {
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
  const long long total = (long long)len[0] * len[1] * len[2];
  const double idx_ = 1.0 / bx.dx[d];
  for (long long id = HR_TID; id < total; id += HR_STRIDE) {
    long long r = id;
    int ii[3];
    ii[0] = (int)(r % len[0]) + off[0];
    r /= len[0];
    ii[1] = (int)(r % len[1]) + off[1];
    ii[2] = (int)(r / len[1]) + off[2];
    const long long t = cell_index(bx, ii[0], ii[1], ii[2]);
    bool trans = true;
    for (int e = 0; e < 3; ++e)
      if (e != d && (ii[e] < 0 || ii[e] >= bx.n[e])) trans = false;
    const int f = ii[d];
    const bool up = trans && f < bx.n[d];
    const bool dn = trans && f >= 1;
    int lo[3] = {ii[0], ii[1], ii[2]};
    lo[d] -= 1;
    const long long zu = up ? zone_of(bx, ii[0], ii[1], ii[2]) : 0;
    const long long zd = dn ? zone_of(bx, lo[0], lo[1], lo[2]) : 0;
    for (int q = 0; q < NPR; ++q) {
      double v = 0.0;
      if (up) v += gX[q * bx.nact + zu] * idx_;
      if (dn) v -= gX[q * bx.nact + zd] * idx_;
      gF[q * bx.ntot + t] = v;
    }
    if (gFS) {  // the entropy flux, X_S = -div F_S
      double v = 0.0;
      if (up) v += gXS[zu] * idx_;
      if (dn) v -= gXS[zd] * idx_;
      gFS[t] = v;
    }
  }
}

// ----------------------------------------------------------- flux-CT (T)
__device__ __forceinline__ bool in_range(const int ii[3], const int len[3]) {
  return ii[0] >= 0 && ii[0] < len[0] && ii[1] >= 0 && ii[1] < len[1] && ii[2] >= 0 && ii[2] < len[2];
}

// gEMF at every edge from the cotangents of the CT-replaced face fluxes.
static __global__ void ka_emf_T(DevParams p, BoxGeo bx, const double* __restrict__ gFab,
                                const double* __restrict__ gFba, double* __restrict__ gemf, int a, int b) {
  int len[3], la[3], lb[3];
  for (int e = 0; e < 3; ++e) {
    len[e] = bx.n[e] + ((e == a || e == b) ? 1 : 0);
    la[e] = bx.n[e] + (e == a ? 1 : 0);
    lb[e] = bx.n[e] + (e == b ? 1 : 0);
  }
  const long long total = (long long)len[0] * len[1] * len[2];
  const long long sa = bx.str[a], sb = bx.str[b];
  for (long long id = HR_TID; id < total; id += HR_STRIDE) {
    long long r = id;
    int ii[3];
    ii[0] = (int)(r % len[0]);
    r /= len[0];
    ii[1] = (int)(r % len[1]);
    ii[2] = (int)(r / len[1]);
    const long long t = cell_index(bx, ii[0], ii[1], ii[2]);
    const bool pole = p.metric == KS && (a == 1 || b == 1) &&
                      ((ii[1] == 0 && bx.bc[2] == 2) || (ii[1] == bx.n[1] && bx.bc[3] == 2));
    double v = 0.0;
    if (!pole) {
      int m[3] = {ii[0], ii[1], ii[2]};
      if (in_range(m, la)) v += 0.5 * gFab[t];
      m[b] -= 1;
      if (in_range(m, la)) v += 0.5 * gFab[t - sb];
      m[b] += 1;
      if (in_range(m, lb)) v -= 0.5 * gFba[t];
      m[a] -= 1;
      if (in_range(m, lb)) v -= 0.5 * gFba[t - sa];
    }
    gemf[t] = v;
  }
}

// Cotangents of the Godunov induction fluxes F_a[B_b] (and F_b[B_a]) over the
// face kernel's range: their only use is the edge EMFs.
template <int dd>
__global__ void ka_ct_T(BoxGeo bx, const double* __restrict__ gemf, double* __restrict__ gFq, int other,
                        double sign) {
  int len[3], off[3], le[3];
  for (int e = 0; e < 3; ++e) {
    if (e == dd) {
      len[e] = bx.n[e] + 1;
      off[e] = 0;
    } else if (bx.n[e] > 1) {
      len[e] = bx.n[e] + 2;
      off[e] = -1;
    } else {
      len[e] = 1;
      off[e] = 0;
    }
    le[e] = bx.n[e] + ((e == dd || e == other) ? 1 : 0);
  }
  const long long total = (long long)len[0] * len[1] * len[2];
  const long long so = bx.str[other];
  for (long long id = HR_TID; id < total; id += HR_STRIDE) {
    long long r = id;
    int ii[3];
    ii[0] = (int)(r % len[0]) + off[0];
    r /= len[0];
    ii[1] = (int)(r % len[1]) + off[1];
    ii[2] = (int)(r / len[1]) + off[2];
    const long long t = cell_index(bx, ii[0], ii[1], ii[2]);
    double v = 0.0;
    if (in_range(ii, le)) v += gemf[t];
    int m[3] = {ii[0], ii[1], ii[2]};
    m[other] += 1;
    if (in_range(m, le)) v += gemf[t + so];
    gFq[t] = sign * 0.25 * v;
  }
}

// ------------------------------------------------------ Riemann fluxes (T)
// Reverse sweep of face_flux64: the cotangents of the two states and of
// kappa_scale from those of the 12 fluxes and of the entropy flux, each
// operation of FaceSide transposed by hand.  About 1,500 FP64 instructions per
// face; 25 forward derivatives on dual numbers took fifteen times as many.

// Cotangents of one side's intermediates (names as in FaceSide).
struct SideCot {
  double u0, ud, u1, l0, l[3], bt, m0, m[3], iut, wb, pt, r0, rd, k0, k[3];
  double aF[2], aU[2];  // of the weights, gas and radiation
};

// FaceSide::add transposed: o the cotangents of out, oM that of the returned
// mass share.  Adds to gP what does not pass through the intermediates.
template <int MET, int d>
__device__ __forceinline__ void side_add_T(const FaceSide<MET, d>& s, const double P[NPR], const double aF[2],
                                           const double aU[2], const double o[NPR], double oM, double gP[NPR],
                                           SideCot& c) {
  const double ud = d == 1 ? s.u1 : P[U1 + d - 1], Bd = P[B1 + d - 1], iut = s.iut;
  const double V = fma(aU[0], s.u0, aF[0] * ud), bu = s.bt * s.u0, bd = fma(s.bt, ud, Bd);
  const double S = fma(aU[0], bu, aF[0] * bd), Y = -(iut * iut) * S, Z = fma(s.bt, Y, s.wb * V);
  double gZ = o[1] * s.l0, gY = o[1] * s.m0;
  c.l0 = o[1] * Z;
  c.m0 = o[1] * Y;
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    gZ = fma(o[2 + i], s.l[i], gZ);
    gY = fma(o[2 + i], s.m[i], gY);
    c.l[i] = o[2 + i] * Z;
    c.m[i] = o[2 + i] * Y;
  }
  c.pt = fma(o[1], aU[0], o[1 + d] * aF[0]);
  double gaU = o[1] * s.pt, gaF = o[1 + d] * s.pt;
  const double gM = o[0] + o[1] + oM;
  // induction rows
  const double vi = V * iut, Bi = aF[0] * Bd * iut;
  double gvi = 0.0, gBi = 0.0;
  c.u1 = 0.0;
#pragma unroll
  for (int i = 1; i <= 3; ++i) {
    if (i == d) continue;
    const double oi = o[4 + i];
    gvi = fma(oi, P[B1 + i - 1], gvi);
    gBi = fma(-oi, i == 1 ? s.u1 : P[U1 + i - 1], gBi);
    gP[B1 + i - 1] = fma(oi, vi, gP[B1 + i - 1]);
    if (i == 1) c.u1 = -oi * Bi;
    else gP[U1 + i - 1] = fma(-oi, Bi, gP[U1 + i - 1]);
  }
  double gV = gvi * iut, gBd = gBi * aF[0] * iut;
  c.iut = fma(gvi, V, gBi * aF[0] * Bd);
  gaF = fma(gBi, Bd * iut, gaF);
  // Z, M, Y
  c.bt = gZ * Y;
  gY = fma(gZ, s.bt, gY);
  c.wb = gZ * V;
  gV = fma(gZ, s.wb, fma(gM, P[RHO], gV));
  gP[RHO] = fma(gM, V, gP[RHO]);
  c.iut = fma(-2.0 * gY * iut, S, c.iut);
  const double gS = -(iut * iut) * gY, gbu = gS * aU[0], gbd = gS * aF[0];
  gaU = fma(gS, bu, gaU);
  gaF = fma(gS, bd, gaF);
  c.bt = fma(gbd, ud, fma(gbu, s.u0, c.bt));
  gBd += gbd;
  gP[B1 + d - 1] += gBd;
  c.u0 = fma(gbu, s.bt, gV * aU[0]);
  c.ud = fma(gbd, s.bt, gV * aF[0]);
  c.aU[0] = fma(gV, s.u0, gaU);
  c.aF[0] = fma(gV, ud, gaF);
  // radiation
  const double E = P[ER], e13 = E * (1.0 / 3.0), W = fma(aU[1], s.r0, aF[1] * s.rd), e43 = (4.0 / 3.0) * E, R = e43 * W;
  double gR = o[8] * s.k0;
  c.k0 = o[8] * R;
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    gR = fma(o[9 + i], s.k[i], gR);
    c.k[i] = o[9 + i] * R;
  }
  const double ge13 = fma(o[8], aU[1], o[8 + d] * aF[1]), gW = gR * e43;
  gP[ER] += fma(gR * (4.0 / 3.0), W, ge13 * (1.0 / 3.0));
  c.aU[1] = fma(gW, s.r0, o[8] * e13);
  c.aF[1] = fma(gW, s.rd, o[8 + d] * e13);
  c.r0 = gW * aU[1];
  c.rd = gW * aF[1];
}

// FaceSide::build transposed: gvp, gvm the cotangents of v_max and v_min (gas,
// radiation), c those of the other intermediates; adds to gP and *gks.
template <int MET, int d>
__device__ __forceinline__ void side_build_T(const DevParams& p, const Geo<MET, double>& g,
                                             const FaceGeo<MET, d>& f, const FaceSide<MET, d>& s, double dl,
                                             double kf, const double P[NPR], const double gvp[2],
                                             const double gvm[2], SideCot& c, double gP[NPR], double* gks) {
  double gc2[2];
#pragma unroll
  for (int w = 0; w < 2; ++w) {  // speeds
    const double ut = w ? s.r0 : s.u0, ud = w ? s.rd : (d == 1 ? s.u1 : P[U1 + d - 1]), c2 = s.c2[w], H = s.H[w];
    const double sum = gvp[w] + gvm[w], dif = gvp[w] - gvm[w], iq = s.iq[w];
    const double gBq = sum * iq, gqa = -(fma(sum, s.Bq[w], dif * s.sd[w])) * (iq * iq);
    const double gK = s.sd[w] > 0.0 ? 0.5 * dif * iq * rcp(s.sd[w]) : 0.0;
    const double AB = d == 1 ? g.Gt(1) : 0.0, u02 = ut * ut, mix = ut * ud;
    double gx = fma(gK, fma(c2, f.C0 - H, H) + c2 * (f.C0 - H), fma(-gBq, AB + mix, -gqa * (g.Gtt() + u02)));
    const double gH = gK * c2 * (1.0 - c2);
    const double gmix = fma(gBq, 1.0 - c2, -2.0 * AB * gH);
    const double gu02 = fma(gqa, 1.0 - c2, gH * g.Gdd(d));
    const double gu = fma(gmix, ud, 2.0 * ut * gu02), gd = fma(gmix, ut, 2.0 * ud * g.Gtt() * gH);
    if (w) {
      c.r0 += gu;
      c.rd += gd;
    } else {
      c.u0 += gu;
      c.ud += gd;
    }
    gc2[w] = gx;
  }
  const double rho = P[RHO], iwb = rcp(s.wb);
  double gpg = c.pt, gbsq = 0.5 * c.pt, gwb = c.wb;
  if (!(s.cd & 3u)) {  // c_ms^2 = (Gamma p + b^2) / (w + b^2), unclamped
    gpg = fma(gc2[0] * p.gam, iwb, gpg);
    gbsq = fma(gc2[0], iwb, gbsq);
    gwb = fma(-gc2[0] * s.c2[0], iwb, gwb);
  }
  if (s.cd & 4u) {  // (4 / (3 tau))^2: d/dtau = -2 c^2 / tau
    const double Tg = p.gm1 * P[UU] / rho;
    double ka, dr = 0.0, du = 0.0;  // absorption over kappa_scale and its derivatives
    if (p.opacity == 2) {
      ka = kf;
    } else if (p.opacity == 1) {
      const double Tc = Tg > p.Tmin ? Tg : p.Tmin, T2 = Tc * Tc;
      ka = p.kabs0 * rho * rho * rsqrt64(T2 * T2 * T2 * Tc);
      dr = (Tg > p.Tmin ? 5.5 : 2.0) * ka / rho;
      du = Tg > p.Tmin ? -3.5 * ka / P[UU] : 0.0;
    } else {
      ka = p.kabs0 * rho;
      dr = p.kabs0;
    }
    const double kt = fma(p.kes0, rho, ka);
    const double gk = -2.0 * s.c2[1] / (p.kscale * kt) * gc2[1];  // of kappa_scale kt
    *gks = fma(gk, kt, *gks);
    gP[RHO] = fma(gk * p.kscale, dr + p.kes0, gP[RHO]);
    gP[UU] = fma(gk * p.kscale, du, gP[UU]);
  }
  (void)dl;
  // w + b^2, p_tot
  gbsq += gwb;
  gP[RHO] += gwb;
  gP[UU] += fma(p.gm1, gpg, p.gam * gwb);
  // u^d, u_r^d
  if (d == 1) {
    c.u1 += c.ud;
  } else {
    gP[U1 + d - 1] += c.ud;
    gP[UR1 + d - 1] += c.rd;
  }
  frame_T<MET>(g, f.a01, f.b1, s, P, c.u0, c.u1, c.l0, c.l, c.m0, c.m, c.bt, c.iut, gbsq, c.r0, d == 1 ? c.rd : 0.0,
               c.k0, c.k, gP);
}

template <int MET, int d>
__global__ void __launch_bounds__(128) ka_face(DevParams p, BoxGeo bx, EdgeSet E, const double* __restrict__ K,
                                               const double* __restrict__ gF, double* __restrict__ gE,
                                               double* gk_out, const double* __restrict__ gFS,
                                               const double* __restrict__ geo) {
  constexpr int dd = d + 1;
  const bool weighted = (MET == KS) && (d != 1);
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
  const long long total = (long long)len[0] * len[1] * len[2], nt = bx.ntot;
  const long long st = bx.str[d];
  double gk = 0.0;
  for (long long id = HR_TID; id < total; id += HR_STRIDE) {
    long long r = id;
    int ii[3];
    ii[0] = (int)(r % len[0]) + off[0];
    r /= len[0];
    ii[1] = (int)(r % len[1]) + off[1];
    ii[2] = (int)(r / len[1]) + off[2];
    const long long t = cell_index(bx, ii[0], ii[1], ii[2]);
    const int fi = ii[d];
    if (MET == KS && d == 1 && ((fi == 0 && bx.bc[2] == 2) || (fi == bx.n[1] && bx.bc[3] == 2))) continue;
    double o[NPR];
    bool any = false;
#pragma unroll
    for (int q = 0; q < NPR; ++q) {
      o[q] = q == B1 + d ? 0.0 : gF[q * nt + t];
      any = any || o[q] != 0.0;
    }
    const double gfs = gFS ? gFS[t] : 0.0;
    any = any || gfs != 0.0;
    if (!any) continue;
    Geo<MET, double> g;
    double igf = 1.0, dl = bx.dx[d];
    if constexpr (MET == KS) {
      const GeoTab T = geotab(geo, bx);
      const double* tab = d == 0 ? T.F0 : (d == 1 ? T.F1 : T.C);
      const long long sz = d == 0 ? T.sF0 : (d == 1 ? T.sF1 : T.sC);
      const long long x = d == 0 ? gidx_f0(bx, ii[0], ii[1])
                                 : (d == 1 ? gidx_f1(bx, ii[0], ii[1]) : gidx_c(bx, ii[0], ii[1]));
      g = geo_load<MET>(tab, sz, x);
      if (weighted) igf = __ldg(tab + 16 * sz + x);
      dl *= __ldg(tab + (d == 2 ? 19 : 17) * sz + x);
    } else {
      g = make_geo<MET, double>(p, 0.0, 0.0);
    }
    double PL[NPR], PR[NPR];
#pragma unroll
    for (int q = 0; q < NPR; ++q) {
      const bool wq = weighted && ((q >= U1 && q <= B3) || q >= UR1);
      const double w = wq ? igf : 1.0;
      PL[q] = E.plane(1, q, nt)[t - st] * w;
      PR[q] = E.plane(0, q, nt)[t] * w;
    }
    const double kL = kfield(p, K, t - st), kR = kfield(p, K, t);
    const FaceGeo<MET, dd> f(g);
    FaceSide<MET, dd> L, R;
    L.build(p, g, f, dl, kL, PL, nullptr);
    R.build(p, g, f, dl, kR, PR, nullptr);
    double cp[2], cm[2], aFL[2], aFR[2], aUL[2], aUR[2], sc[2];
#pragma unroll
    for (int w = 0; w < 2; ++w) {
      cp[w] = fmax(0.0, fmax(L.vmax(w), R.vmax(w)));
      cm[w] = -fmin(0.0, fmin(L.vmin(w), R.vmin(w)));
      if (p.flux == 0) {
        aFL[w] = aFR[w] = 1.0;
        aUL[w] = cp[w] > cm[w] ? cp[w] : cm[w];
        aUR[w] = -aUL[w];
        sc[w] = 0.5 * g.gdet;
      } else {
        const double sum = cp[w] + cm[w];
        const bool ok = sum > 0.0;
        aFL[w] = ok ? cp[w] : 1.0;
        aFR[w] = ok ? cm[w] : 1.0;
        aUL[w] = ok ? cm[w] * cp[w] : 0.0;
        aUR[w] = -aUL[w];
        sc[w] = g.gdet * (ok ? 1.0 / sum : 0.5);
      }
    }
    // the entropy flux s_L M_L + s_R M_R (over the scale of the gas rows)
    double sL = 0.0, sR = 0.0;
    if (gfs != 0.0) {
      sL = entropy_per_baryon<double>(p, PL[RHO], PL[UU]);
      sR = entropy_per_baryon<double>(p, PR[RHO], PR[UU]);
    }
    double gsc[2] = {0.0, 0.0};  // cotangents of the scales (HLL)
    if (p.flux != 0) {
      double raw[NPR];
#pragma unroll
      for (int q = 0; q < NPR; ++q) raw[q] = 0.0;
      const double mL = L.template add<false>(g, PL, aFL[0], aUL[0], aFL[1], aUL[1], raw);
      const double mR = R.template add<false>(g, PR, aFR[0], aUR[0], aFR[1], aUR[1], raw);
#pragma unroll
      for (int q = 0; q < NPR; ++q)
        if (q != B1 + d) gsc[q < ER ? 0 : 1] = fma(o[q], raw[q], gsc[q < ER ? 0 : 1]);
      gsc[0] += gfs * (sL * mL + sR * mR);
    }
#pragma unroll
    for (int q = 0; q < NPR; ++q) o[q] *= sc[q < ER ? 0 : 1];
    double gL[NPR], gR[NPR];
#pragma unroll
    for (int q = 0; q < NPR; ++q) gL[q] = gR[q] = 0.0;
    SideCot cL, cR;
    side_add_T<MET, dd>(L, PL, aFL, aUL, o, gfs * sc[0] * sL, gL, cL);
    side_add_T<MET, dd>(R, PR, aFR, aUR, o, gfs * sc[0] * sR, gR, cR);
    if (gfs != 0.0) {  // d s = n d ug / ug - (n + 1) d rho / rho
      const double n = 1.0 / (p.gam - 1.0), ud1 = dd == 1 ? L.u1 : PL[U1 + d], ud2 = dd == 1 ? R.u1 : PR[U1 + d];
      const double gl = gfs * sc[0] * PL[RHO] * fma(aUL[0], L.u0, aFL[0] * ud1);
      const double gr = gfs * sc[0] * PR[RHO] * fma(aUR[0], R.u0, aFR[0] * ud2);
      gL[UU] += gl * n / PL[UU];
      gL[RHO] -= gl * (n + 1.0) / PL[RHO];
      gR[UU] += gr * n / PR[UU];
      gR[RHO] -= gr * (n + 1.0) / PR[RHO];
    }
    // weights -> v_max, v_min of the sides, by the branches the maxima took
    double vpL[2], vpR[2], vmL[2], vmR[2];
#pragma unroll
    for (int w = 0; w < 2; ++w) {
      double gp, gm;
      const double gU = cL.aU[w] - cR.aU[w];
      if (p.flux == 0) {
        gp = cp[w] > cm[w] ? gU : 0.0;
        gm = cp[w] > cm[w] ? 0.0 : gU;
      } else if (cp[w] + cm[w] > 0.0) {
        const double gs = -gsc[w] * sc[w] / (cp[w] + cm[w]);
        gp = cL.aF[w] + gU * cm[w] + gs;
        gm = cR.aF[w] + gU * cp[w] + gs;
      } else {
        gp = gm = 0.0;
      }
      const double a = L.vmax(w), b = R.vmax(w), e = L.vmin(w), h = R.vmin(w);
      if (!(cp[w] > 0.0)) gp = 0.0;
      if (!(cm[w] > 0.0)) gm = 0.0;
      vpL[w] = a >= b ? gp : 0.0;
      vpR[w] = a >= b ? 0.0 : gp;
      vmL[w] = e <= h ? -gm : 0.0;
      vmR[w] = e <= h ? 0.0 : -gm;
    }
    side_build_T<MET, dd>(p, g, f, L, dl, kL, PL, vpL, vmL, cL, gL, &gk);
    side_build_T<MET, dd>(p, g, f, R, dl, kR, PR, vpR, vmR, cR, gR, &gk);
#pragma unroll
    for (int q = 0; q < NPR; ++q) {
      const bool wq = weighted && ((q >= U1 && q <= B3) || q >= UR1);
      const double w = wq ? igf : 1.0;
      gE[(NPR + q) * nt + t - st] = gL[q] * w;  // upper edge of cell f-1
      gE[q * nt + t] = gR[q] * w;               // lower edge of cell f
    }
  }
  warp_atomic_add(gk_out, gk);
}

// ----------------------------------------------------- reconstruction (T)
// Per cell of the edge range: cotangents of the five stencil primitives of
// every variable (atomic, the stencils overlap) and of the cell's flattener,
// from the edge formulas of the reconstruction transposed by hand (twice the
// MC slope D, the interface values, flattening, monotonicity) along the
// branches they take.  Three directions of the 64x32x16 torus per step: 2.72 ms on
// dual numbers over the six inputs, 0.85 so.

// D = mc_twice(dm, dp) transposed.
__device__ __forceinline__ void mc_twice_T(double dm, double dp, double gD, double& gm, double& gp) {
  const unsigned c = mc_twice_code(dm, dp);
  gm = c == 1 ? gD : (c == 2 ? 4.0 * gD : 0.0);
  gp = c == 1 ? gD : (c == 3 ? 4.0 * gD : 0.0);
}

template <int MET, int d>
__global__ void ka_edges(DevParams p, BoxGeo bx, const double* __restrict__ P, const double* __restrict__ aux,
                         const double* __restrict__ flat, const double* __restrict__ gE, double* gP,
                         double* __restrict__ gchi) {
  const bool weighted = (MET == KS) && (d != 1);
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
  const long long total = (long long)len[0] * len[1] * len[2];
  const long long st = bx.str[d], nt = bx.ntot;
  for (long long id = HR_TID; id < total; id += HR_STRIDE) {
    long long r = id;
    int i = (int)(r % len[0]) + off[0];
    r /= len[0];
    int j = (int)(r % len[1]) + off[1];
    int k = (int)(r / len[1]) + off[2];
    const long long t = cell_index(bx, i, j, k);
    double gcg = 0.0, gcr = 0.0;
    const double chg = p.recon == 0 ? flat[t] : 0.0, chr = p.recon == 0 ? flat[nt + t] : 0.0;
    double gw[5];
#pragma unroll
    for (int m = 0; m < 5; ++m) gw[m] = weighted ? aux[t + (m - 2) * st] : 1.0;
#pragma unroll 2
    for (int q = 0; q < NPR; ++q) {
      double gl = gE[q * nt + t], gr = gE[(NPR + q) * nt + t];
      if (gl == 0.0 && gr == 0.0) continue;
      const bool wq = weighted && ((q >= U1 && q <= B3) || q >= UR1);
      double s[5], dd[4], gs[5] = {0.0, 0.0, 0.0, 0.0, 0.0}, gd[4] = {0.0, 0.0, 0.0, 0.0};
#pragma unroll
      for (int m = 0; m < 5; ++m) {
        const double v = P[q * nt + t + (m - 2) * st];
        s[m] = wq ? gw[m] * v : v;
      }
#pragma unroll
      for (int m = 0; m < 4; ++m) dd[m] = s[m + 1] - s[m];
      if (p.recon == 0) {
        const double chi = q < ER ? chg : chr, qc = s[2];
        const double D1 = mc_twice(dd[0], dd[1]), D2 = mc_twice(dd[1], dd[2]), D3 = mc_twice(dd[2], dd[3]);
        const double l0 = ppm_face(s[1], dd[1], D1, D2), r0 = ppm_face(s[2], dd[2], D2, D3);
        double l = l0, rr = r0;
        const unsigned code = ppm_limit(qc, chi, l, rr);
        if (code == 1) {
          gs[2] = gl + gr;
          gl = gr = 0.0;
        } else if (code == 2) {  // l = 3 q - 2 r
          gs[2] = 3.0 * gl;
          gr -= 2.0 * gl;
          gl = 0.0;
        } else if (code == 3) {  // r = 3 q - 2 l
          gs[2] = 3.0 * gr;
          gl -= 2.0 * gr;
          gr = 0.0;
        }
        const double gc = gl * (qc - l0) + gr * (qc - r0);
        if (q < ER) gcg += gc;
        else gcr += gc;
        gs[2] += chi * (gl + gr);
        gl *= 1.0 - chi;
        gr *= 1.0 - chi;
        // l0 = s1 + d1 / 2 + (D1 - D2) / 12, r0 = s2 + d2 / 2 + (D2 - D3) / 12
        gs[1] = gl;
        gs[2] += gr;
        double a, b;
        mc_twice_T(dd[0], dd[1], gl * (1.0 / 12.0), a, b);
        gd[0] = a;
        gd[1] = b + 0.5 * gl;
        mc_twice_T(dd[1], dd[2], (gr - gl) * (1.0 / 12.0), a, b);
        gd[1] += a;
        gd[2] = b + 0.5 * gr;
        mc_twice_T(dd[2], dd[3], gr * (-1.0 / 12.0), a, b);
        gd[2] += a;
        gd[3] = b;
      } else {  // s -+ D / 4
        gs[2] = gl + gr;
        mc_twice_T(dd[1], dd[2], 0.25 * (gr - gl), gd[1], gd[2]);
      }
#pragma unroll
      for (int m = 0; m < 5; ++m) {
        const double v = gs[m] + (m > 0 ? gd[m - 1] : 0.0) - (m < 4 ? gd[m] : 0.0);
        if (v != 0.0) atomicAdd(&gP[q * nt + t + (m - 2) * st], wq ? v * gw[m] : v);
      }
    }
    gchi[t] = gcg;
    gchi[nt + t] = gcr;
  }
}

// ---------------------------------------------------------- flattener (T)
// The flattener after sub-step s is max(previous, new); the cotangent goes to
// the new value where it won (strictly greater, as in the forward), else it
// is carried to the earlier sub-step.
template <int d>
__global__ void ka_flatten(DevParams p, BoxGeo bx, const double* __restrict__ P, const double* __restrict__ aux,
                           const double* __restrict__ prev, const double* __restrict__ gchi, double* carry,
                           double* gP, double* gaux) {
  typedef Dn<5> D5;
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
  const long long total = (long long)len[0] * len[1] * len[2];
  const long long st = bx.str[d];
  for (long long id = HR_TID; id < total; id += HR_STRIDE) {
    long long r = id;
    int i = (int)(r % len[0]) + off[0];
    r /= len[0];
    int j = (int)(r % len[1]) + off[1];
    int k = (int)(r / len[1]) + off[2];
    const long long t = cell_index(bx, i, j, k);
    double gg = gchi[t] + carry[t], gr = gchi[bx.ntot + t] + carry[bx.ntot + t];
    carry[t] = 0.0;
    carry[bx.ntot + t] = 0.0;
    if (gg == 0.0 && gr == 0.0) continue;
    FlatCell<double> c[7];
    for (int m = 0; m < 7; ++m) {
      const long long cm = t + (m - 3) * st;
      c[m].pg = (p.gam - 1.0) * P[UU * bx.ntot + cm];
      c[m].pr = P[ER * bx.ntot + cm] * (1.0 / 3.0);
      c[m].vg = aux[(1 + 3 * d) * bx.ntot + cm];
      c[m].vr = aux[(2 + 3 * d) * bx.ntot + cm];
      c[m].w = aux[(3 + 3 * d) * bx.ntot + cm];
    }
    double Fg, Fr;
    flatten_cell<double>(c, &Fg, &Fr);
    const double pg_prev = prev ? prev[t] : 0.0, pr_prev = prev ? prev[bx.ntot + t] : 0.0;
    if (!(Fg > pg_prev)) {
      carry[t] = gg;
      gg = 0.0;
    }
    if (!(Fr > pr_prev)) {
      carry[bx.ntot + t] = gr;
      gr = 0.0;
    }
    if (gg == 0.0 && gr == 0.0) continue;
    for (int m = 0; m < 7; ++m) {
      FlatCell<D5> cd[7];
      for (int n = 0; n < 7; ++n) {
        const int o = n == m ? 0 : -100;
        cd[n].pg = D5::seed(c[n].pg, o);
        cd[n].pr = D5::seed(c[n].pr, o + 1);
        cd[n].vg = D5::seed(c[n].vg, o + 2);
        cd[n].vr = D5::seed(c[n].vr, o + 3);
        cd[n].w = D5::seed(c[n].w, o + 4);
      }
      D5 Fgd, Frd;
      flatten_cell<D5>(cd, &Fgd, &Frd);
      double v[5];
      for (int c5 = 0; c5 < 5; ++c5) v[c5] = gg * Fgd.d[c5] + gr * Frd.d[c5];
      const long long cm = t + (m - 3) * st;
      if (v[0] != 0.0) atomicAdd(&gP[UU * bx.ntot + cm], (p.gam - 1.0) * v[0]);
      if (v[1] != 0.0) atomicAdd(&gP[ER * bx.ntot + cm], v[1] * (1.0 / 3.0));
      if (v[2] != 0.0) atomicAdd(&gaux[cm], v[2]);
      if (v[3] != 0.0) atomicAdd(&gaux[bx.ntot + cm], v[3]);
      if (v[4] != 0.0) atomicAdd(&gaux[2 * bx.ntot + cm], v[4]);
    }
  }
}

// Cell factors of direction d (T): sqrt(-g) u^d, sqrt(-g) u^d_rad and
// w_d = min(1, 2 tau_d) of every cell.
template <int MET, int d>
__global__ void ka_prep(DevParams p, BoxGeo bx, const double* __restrict__ P, const double* __restrict__ K,
                        const double* __restrict__ gaux, double* gP, double* gk_out) {
  typedef Dn<3> D3;
  double gk = 0.0;
  for (long long t = HR_TID; t < bx.ntot; t += HR_STRIDE) {
    const double gvg = gaux[t], gvr = gaux[bx.ntot + t], gw = gaux[2 * bx.ntot + t];
    if (gvg == 0.0 && gvr == 0.0 && gw == 0.0) continue;
    long long r = t;
    const int i = (int)(r % bx.N[0]) - bx.ng[0];
    r /= bx.N[0];
    const int j = (int)(r % bx.N[1]) - bx.ng[1];
    const Geo<MET, D3> g = geo_cast<D3>(make_geo<MET, double>(p, xcen(bx, 0, i), xcen(bx, 1, j)));
    if (gvg != 0.0) {
      D3 ucon[4], ucov[4], gm;
      fourvel<MET, D3>(g, D3::seed(P[U1 * bx.ntot + t], 0), D3::seed(P[U2 * bx.ntot + t], 1),
                       D3::seed(P[U3 * bx.ntot + t], 2), ucon, ucov, &gm);
      const D3 v = g.gdet * ucon[d + 1];
      for (int c = 0; c < 3; ++c) gP[(U1 + c) * bx.ntot + t] += gvg * v.d[c];
    }
    if (gvr != 0.0) {
      D3 ucon[4], ucov[4], gm;
      fourvel<MET, D3>(g, D3::seed(P[UR1 * bx.ntot + t], 0), D3::seed(P[UR2 * bx.ntot + t], 1),
                       D3::seed(P[UR3 * bx.ntot + t], 2), ucon, ucov, &gm);
      const D3 v = g.gdet * ucon[d + 1];
      for (int c = 0; c < 3; ++c) gP[(UR1 + c) * bx.ntot + t] += gvr * v.d[c];
    }
    if (gw != 0.0) {
      D3 kabs, ksca;
      opacity<D3>(p, D3::seed(P[RHO * bx.ntot + t], 0), D3::seed(P[UU * bx.ntot + t], 1), D3(kfield(p, K, t)),
                  &kabs, &ksca, D3::seed(p.kscale, 2));
      const D3 tau = (kabs + ksca) * sqrt(g.gdd(d + 1)) * D3(bx.dx[d]);
      const D3 w = D3(2.0) * tau;
      if (w < 1.0) {
        gP[RHO * bx.ntot + t] += gw * w.d[0];
        gP[UU * bx.ntot + t] += gw * w.d[1];
        gk += gw * w.d[2];
      }
    }
  }
  warp_atomic_add(gk_out, gk);
}

// --------------------------------------------------------- ghost fill (T)
// Launched for d = 2, 1, 0 (the reverse of the forward order): every ghost
// cell's cotangent goes to its source cell, with the polar sign flips and the
// outflow clamps (derivative 1 where the clamp let the value through).
static __global__ void ka_bc_T(BoxGeo bx, const double* __restrict__ P, double* gP, int d) {
  int lo[3], len[3];
  for (int e = 0; e < 3; ++e) {
    if (e == d) {
      lo[e] = 0;
      len[e] = bx.ng[d];
    } else if (e < d) {
      lo[e] = -bx.ng[e];
      len[e] = bx.n[e] + 2 * bx.ng[e];
    } else {
      lo[e] = 0;
      len[e] = bx.n[e];
    }
  }
  const long long total = 2LL * len[0] * len[1] * len[2];
  for (long long id = HR_TID; id < total; id += HR_STRIDE) {
    long long r = id;
    int a0 = (int)(r % len[0]);
    r /= len[0];
    int a1 = (int)(r % len[1]);
    r /= len[1];
    int a2 = (int)(r % len[2]);
    int side = (int)(r / len[2]);
    int c[3] = {a0 + lo[0], a1 + lo[1], a2 + lo[2]};
    int g = c[d];
    int dst[3] = {c[0], c[1], c[2]}, src[3] = {c[0], c[1], c[2]};
    int bc = bx.bc[2 * d + side];
    dst[d] = side == 0 ? -1 - g : bx.n[d] + g;
    double sgn = 1.0;
    int clamp = 0;
    if (bc == 0) {
      src[d] = side == 0 ? bx.n[d] - 1 - g : g;
    } else if (bc == 1 || bc == 3) {
      src[d] = side == 0 ? 0 : bx.n[d] - 1;
      clamp = bc == 3 ? 0 : (side == 0 ? -1 : 1);
    } else {
      src[d] = side == 0 ? g : bx.n[d] - 1 - g;
      if (bx.n[2] > 1) src[2] = (c[2] + bx.n[2] / 2) % bx.n[2];
      sgn = -1.0;
    }
    const long long s = cell_index(bx, src[0], src[1], src[2]);
    const long long t = cell_index(bx, dst[0], dst[1], dst[2]);
    for (int q = 0; q < NPR; ++q) {
      double gv = gP[q * bx.ntot + t];
      gP[q * bx.ntot + t] = 0.0;
      if (gv == 0.0) continue;
      if (q == U1 + d || q == B1 + d || q == UR1 + d) gv *= sgn;
      if (clamp != 0 && (q == U1 + d || q == UR1 + d)) {
        const double v = P[q * bx.ntot + s] * sgn;
        if (clamp < 0 ? !(v < 0.0) : !(v > 0.0)) gv = 0.0;
      }
      if (gv != 0.0) atomicAdd(&gP[q * bx.ntot + s], gv);
    }
  }
}

// Active cells of gP -> gN (the cotangent of the previous sub-step's output).
static __global__ void ka_gather(BoxGeo bx, const double* __restrict__ gP, double* __restrict__ gN) {
  for (long long z = HR_TID; z < bx.nact; z += HR_STRIDE) {
    int i, j, k;
    zone_ijk(bx, z, i, j, k);
    const long long t = cell_index(bx, i, j, k);
    for (int q = 0; q < NPR; ++q) gN[q * bx.nact + z] = gP[q * bx.ntot + t];
  }
}

}  // namespace hr

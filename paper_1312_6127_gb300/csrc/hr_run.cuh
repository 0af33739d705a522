// Launch sequences of one sub-step for a given metric (internal).
#pragma once
#include "hr_ctx.h"
#include "hr_kernels.cuh"
#include "hr_uct.cuh"

namespace hr {

inline Bufs make_bufs(harmrad_ctx* c) {
  Bufs b;
  b.P = c->P;
  b.K = c->K;
  b.Un = c->Un;
  b.Sn = c->Sn;
  for (int d = 0; d < 3; ++d) {
    b.F[d] = c->F[d];
    b.FS[d] = c->FS[d];
    b.ES[d] = c->ES[d];
    b.spd[d] = c->spd[d];
    b.flat[d] = c->flat[d];
  }
  b.aux = c->aux;
  b.emf = c->emf;
  b.dt = c->dt;
  b.status = c->status;
  b.iters = c->iters;
  b.failed = c->failed;
  b.qcount = c->qcount;
  b.ncont = (int)c->nact;
  b.qzone = c->qzone;
  b.qbox = c->qbox;
  b.qdata = c->qdata;
  b.fzone = c->fzone;
  b.fbox = c->fbox;
  b.ftmp = c->ftmp;
  b.czone = c->czone;
  b.cbox = c->cbox;
  b.cdata = c->cdata;
  b.stats = c->stats;
  b.dtmin = c->dtmin;
  b.geo = c->geotab;
  b.ust_rec = c->rec_ust;
  b.meth_rec = c->rec_meth;
  b.psol_rec = c->rec_psol;
  b.sst_rec = c->rec_sst;
  if (c->imex_M) {  // IMEX contexts record U* and the solutions for the stage sources
    b.ust_rec = c->imex_ust;
    b.psol_rec = c->imex_psol;
  }
  b.imexM = c->imex_M;
  for (int d = 0; d < 3; ++d) b.Bf[d] = c->dp.emf == 1 ? c->Bf[d] : nullptr;
  return b;
}

// Threads per block of a heavy kernel's launch: the tuned number, but at most
// `small` in a grid that does not fill one wave, whose blocks of one or two warps
// spread over all SMs and schedulers (per RK3 step with 32 and 128 threads, the
// reconstruction with 64 and 256: 32x32x32 box update 0.417, 0.458, reconstruction
// 0.079, 0.086 ms; 64x32x16 torus 0.567, 0.620 and 0.188, 0.217; 64 and 128 threads
// lie between, or within 7 % on either side).
inline int fit_block(const harmrad_ctx* c, int block, int small) {
  return small_grid(c->nact, c->sms) && block > small ? small : block;
}

// Largest per-grid count, and the work of all grids (the kernels deal the grids'
// items to the threads as one sequence, first_item), for sizing a launch.
template <typename Fn>
inline long long max_work(const harmrad_ctx* c, Fn work) {
  long long m = 1;
  for (int i = 0; i < c->nbox; ++i) {
    long long w = work(c->boxes[i]);
    if (w > m) m = w;
  }
  return m;
}
template <typename Fn>
inline long long all_work(const harmrad_ctx* c, Fn work) {
  long long m = 0;
  for (int i = 0; i < c->nbox; ++i) m += work(c->boxes[i]);
  return m;
}

inline FaceSet face_set(double* const f[3]) {
  FaceSet s;
  for (int d = 0; d < 3; ++d) s.f[d] = f[d];
  return s;
}

// Staggered field: the faces outside the evolved ranges (periodic images,
// else from the ghost cells' B; after the ghost fill of P).
template <int MET>
int face_ghosts(harmrad_ctx* c) {
  for (int d = 0; d < 3; ++d) {
    k_face_ghosts<MET><<<grid_for(c->ncell, c->sms, 256), 256, 0, c->stream>>>(c->dp, c->dboxes, c->nbox, c->P,
                                                                                 face_set(c->Bf), d, c->geotab);
    mark(c, HARMRAD_K_CT);
  }
  return 3;
}

// Ghost fill of P in every active direction.
inline int fill_ghost_cells(harmrad_ctx* c, double* P = nullptr) {
  const DevParams& p = c->dp;
  double* K = p.opacity == 2 ? c->K : nullptr;
  if (!P) P = c->P;
  int nk = 0;
  for (int d = 0; d < 3; ++d) {
    if (!p.act[d]) continue;
    const long long work = all_work(c, [d](const BoxGeo& b) {
      long long w = 2LL * b.ng[d];
      for (int e = 0; e < 3; ++e)
        if (e != d) w *= (e < d) ? b.N[e] : b.n[e];
      return w;
    });
    const bool one = c->nbox == 1;
    const dim3 g(grid_for(work, c->sms, 128), one ? NPR : 1);
    auto run = [&](auto kernel) { kernel<<<g, 128, 0, c->stream>>>(p, c->dboxes, c->nbox, P, K); };
    if (d == 0) one ? run(k_bc_fill<0, 1>) : run(k_bc_fill<0, NPR>);
    if (d == 1) one ? run(k_bc_fill<1, 1>) : run(k_bc_fill<1, NPR>);
    if (d == 2) one ? run(k_bc_fill<2, 1>) : run(k_bc_fill<2, NPR>);
    mark(c, HARMRAD_K_BC);
    ++nk;
  }
  return nk;
}

// Pieces a column of nd cells is cut into so that there are `slots` threads per
// SM, `least` cells or more each; the cells of a piece.
inline int column_chunk(const harmrad_ctx* c, long long columns, long long nd, int slots, int least,
                        long long* pieces) {
  long long n = ((long long)slots * c->sms + columns - 1) / columns;
  if (n > (nd + least - 1) / least) n = (nd + least - 1) / least;
  *pieces = n;
  return (int)((nd + n - 1) / n);
}

inline int range_width(const BoxGeo& b, int e) { return b.n[e] > 1 ? b.n[e] + 2 : 1; }

// Launches over directions take blockIdx.y for the direction, d0 + blockIdx.y.
// first_dir and dir_count: the range that holds the active ones (none in a grid
// of one zone, which launches nothing for them).
inline int first_dir(const DevParams& p) { return p.act[0] ? 0 : (p.act[1] ? 1 : 2); }
inline int dir_count(const DevParams& p) {
  return p.act[0] || p.act[1] || p.act[2] ? (p.act[2] ? 3 : (p.act[1] ? 2 : 1)) - first_dir(p) : 0;
}

// FP64 flattener of the active directions.
inline void flatten(harmrad_ctx* c, bool fresh) {
  const DevParams& p = c->dp;
  FlatSet fl;
  Chunks ch{};
  long long most = !p.act[0] ? 1 : all_work(c, [](const BoxGeo& b) {
    return 32LL * (((long long)range_width(b, 1) * range_width(b, 2) * b.N[0] + 25) / 26);
  });
  for (int d = 0; d < 3; ++d) {
    fl.f[d] = (double*)c->flat[d];
    if (d == 0 || !p.act[d]) continue;
    const long long cols =
        all_work(c, [d](const BoxGeo& b) { return (long long)range_width(b, 0) * range_width(b, 3 - d); });
    const long long nd = max_work(c, [d](const BoxGeo& b) { return b.n[d] + 2; });
    // a piece evaluates two cells more than it owns; 4 blocks of 128 fit an SM
    long long pieces;
    ch.c[d] = column_chunk(c, cols, nd, 1024, 4, &pieces);
    if (cols * pieces > most) most = cols * pieces;
  }
  const int d0 = first_dir(p);
  const dim3 g(grid_for(most, c->sms, 128), dir_count(p));
  const double* aux = (const double*)c->aux;
  if (p.sig) k_flat<true><<<g, 128, 0, c->stream>>>(p, c->dboxes, c->nbox, c->P, aux, fl, ch, fresh, d0);
  else k_flat<false><<<g, 128, 0, c->stream>>>(p, c->dboxes, c->nbox, c->P, aux, fl, ch, fresh, d0);
}

// FP64 reconstruction of the active directions d0 .. d0 + nd - 1: edge values of
// every cell of their face ranges.
template <int MET>
void recon(harmrad_ctx* c, int d0, int ndir, const double* P, const double* aux, const FlatSet& flat, int block,
           int per_sm) {
  const DevParams& p = c->dp;
  EdgeSets E;
  Chunks ch{};
  long long most = 1;
  for (int d = 0; d < 3; ++d) {
    E.d[d] = EdgeSet{(double*)c->edges[d], c->ES[d]};
    if (d < d0 || d >= d0 + ndir || !p.act[d]) continue;
    long long work;
    if (d == 0) {
      work = all_work(c, [](const BoxGeo& b) {
        return 12LL * 32 * (((long long)range_width(b, 1) * range_width(b, 2) * b.N[0] + 59) / 60);
      });
    } else {
      const long long cols =
          all_work(c, [d](const BoxGeo& b) { return (long long)range_width(b, 0) * range_width(b, 3 - d); });
      const long long nd = max_work(c, [d](const BoxGeo& b) { return b.n[d] + 2; });
      // a piece repeats about one cell's work: 16 cells or more, two threads per slot
      long long pieces;
      ch.c[d] = column_chunk(c, 12 * cols, nd, 4096, 16, &pieces);
      work = 12 * cols * pieces;
    }
    if (work > most) most = work;
  }
  const dim3 g(grid_for(most, c->sms, block, per_sm), ndir);
  auto run = [&](auto sig) {
    constexpr bool SIG = decltype(sig)::value;
    if (d0 == 0) k_recon_rows<MET, SIG><<<g, block, 0, c->stream>>>(p, c->dboxes, c->nbox, P, aux, flat.f[0], E.d[0]);
    else if (d0 == 1)
      k_recon_cols<MET, 1, SIG><<<g, block, 0, c->stream>>>(p, c->dboxes, c->nbox, P, aux, flat.f[1], E.d[1], ch.c[1]);
    else
      k_recon_cols<MET, 2, SIG><<<g, block, 0, c->stream>>>(p, c->dboxes, c->nbox, P, aux, flat.f[2], E.d[2], ch.c[2]);
  };
  if (ndir > 1) k_recon_all<MET><<<g, block, 0, c->stream>>>(p, c->dboxes, c->nbox, P, aux, flat, E, ch, d0);
  else if (p.sig) run(std::true_type{});
  else run(std::false_type{});
}

template <int MET, typename R>
int faces_impl(harmrad_ctx* c, bool fresh) {
  const DevParams& p = c->dp;
  cudaStream_t st = c->stream;
  const BoxGeo* bt = c->dboxes;
  const int nb = c->nbox;
  int nk = fill_ghost_cells(c);
  if (p.emf == 1) nk += face_ghosts<MET>(c);
  if constexpr (std::is_same<R, double>::value)
    k_prep64<MET><<<grid_for(c->ncell, c->sms, 256), 256, 0, st>>>(p, bt, nb, c->P, c->K, (double*)c->aux,
                                                                      c->geotab);
  else
    k_prep<MET, R><<<grid_for(c->ncell, c->sms, 256), 256, 0, st>>>(p, bt, nb, c->P, c->K, (R*)c->aux,
                                                                       c->geotab);
  mark(c, HARMRAD_K_PREP);
  ++nk;
  auto range_cells = [](const BoxGeo& b) {
    long long w = 1;
    for (int e = 0; e < 3; ++e) w *= b.n[e] > 1 ? b.n[e] + 2 : 1;
    return w;
  };
  if (p.recon == 0 && dir_count(p) > 0) {
    if constexpr (std::is_same<R, double>::value) {
      flatten(c, fresh);
      mark(c, HARMRAD_K_FLATTEN);
      ++nk;
    } else {
      for (int d = 0; d < 3; ++d) {
        if (!p.act[d]) continue;
        if (fresh) {
          if (cudaMemsetAsync(c->flat[d], 0, 2 * c->ncell * sizeof(R), st) != cudaSuccess) return HARMRAD_E_CUDA;
          mark(c, HARMRAD_K_OTHER);
        }
        k_flatten<R><<<grid_for(all_work(c, range_cells), c->sms, 256), 256, 0, st>>>(
            p, bt, nb, c->P, (const R*)c->aux, (R*)c->flat[d], d);
        mark(c, HARMRAD_K_FLATTEN);
        ++nk;
      }
    }
  }
  const harmrad_tuning& tu = c->tune;
  const int be = fit_block(c, tu.edge_block, 64), bf = fit_block(c, tu.face_block, 32);
  FlatSet fl;
  for (int d = 0; d < 3; ++d) fl.f[d] = (double*)c->flat[d];
  auto faces_of = [c](int d) {
    return all_work(c, [d](const BoxGeo& b) {
      long long w = 1;
      for (int e = 0; e < 3; ++e) w *= (e == d) ? b.n[e] + 1 : (b.n[e] > 1 ? b.n[e] + 2 : 1);
      return w;
    });
  };
  if (c->merged && !p.sig && dir_count(p) > 0) {  // FP64: all directions in one launch each
    FaceArgs fa;
    long long wf = 1;
    const int d0 = first_dir(p), nd = dir_count(p);
    for (int d = 0; d < 3; ++d) {
      fa.E.d[d] = EdgeSet{(double*)c->edges[d], c->ES[d]};
      fa.F[d] = (double*)c->F[d];
      fa.spd[d] = (double*)c->spd[d];
      fa.FS[d] = (double*)c->FS[d];
      fa.gsp[d] = (double*)c->gsp[d];
      if (p.act[d] && faces_of(d) > wf) wf = faces_of(d);
    }
    recon<MET>(c, d0, nd, c->P, (const double*)c->aux, fl, be, tu.edge_blocks_per_sm);
    mark(c, HARMRAD_K_EDGE);
    const dim3 g(grid_for(wf, c->sms, bf, tu.face_blocks_per_sm), nd);
    k_face_all<MET><<<g, bf, 0, st>>>(p, bt, nb, c->K, c->geotab, fa, d0);
    mark(c, HARMRAD_K_FACE);
    nk += 2;
  } else {
    for (int d = 0; d < 3; ++d) {
      if (!p.act[d]) continue;
      if constexpr (std::is_same<R, double>::value) {
        recon<MET>(c, d, 1, c->P, (const double*)c->aux, fl, be, tu.edge_blocks_per_sm);
      } else {
        const int ge = grid_for(all_work(c, range_cells), c->sms, be, tu.edge_blocks_per_sm);
        auto edge = [&](auto kernel) {
          kernel<<<ge, be, 0, st>>>(p, bt, nb, c->P, (const R*)c->aux, (const R*)c->flat[d], (R*)c->edges[d]);
        };
        d == 0 ? edge(k_edges<MET, 0>) : (d == 1 ? edge(k_edges<MET, 1>) : edge(k_edges<MET, 2>));
      }
      mark(c, HARMRAD_K_EDGE);
      const int gf = grid_for(faces_of(d), c->sms, bf, tu.face_blocks_per_sm);
      if constexpr (std::is_same<R, double>::value) {
        auto face = [&](auto kernel) {
          kernel<<<gf, bf, 0, st>>>(p, bt, nb, EdgeSet{(double*)c->edges[d], c->ES[d]}, c->K, (double*)c->F[d],
                                    (double*)c->spd[d], c->geotab, (double*)c->FS[d], (double*)c->gsp[d]);
        };
        d == 0 ? face(k_face<MET, 0>) : (d == 1 ? face(k_face<MET, 1>) : face(k_face<MET, 2>));
      } else {
        auto face = [&](auto kernel) {
          kernel<<<gf, bf, 0, st>>>(p, bt, nb, (const R*)c->edges[d], c->K, (R*)c->F[d], (R*)c->spd[d],
                                    (R*)c->FS[d], (R*)c->gsp[d]);
        };
        d == 0 ? face(k_face32<MET, 0>) : (d == 1 ? face(k_face32<MET, 1>) : face(k_face32<MET, 2>));
      }
      mark(c, HARMRAD_K_FACE);
      nk += 2;
    }
  }
  if (p.emf == 1) {  // staggered field: the 4-state upwind EMFs on the edges
    if constexpr (std::is_same<R, double>::value)
      k_vel64<MET><<<grid_for(c->ncell, c->sms, 256), 256, 0, st>>>(p, bt, nb, c->P, (double*)c->vel, c->geotab);
    else
      k_vel<MET, R><<<grid_for(c->ncell, c->sms, 256), 256, 0, st>>>(p, bt, nb, c->P, (R*)c->vel, c->geotab);
    mark(c, HARMRAD_K_CT);
    ++nk;
    for (int a = 0; a < 3; ++a)
      for (int b = a + 1; b < 3; ++b) {
        if (!p.act[a] && !p.act[b]) continue;
        long long we = all_work(c, [a, b](const BoxGeo& x) {
          long long w = 1;
          for (int e = 0; e < 3; ++e) w *= x.n[e] + (((e == a || e == b) && x.n[e] > 1) ? 1 : 0);
          return w;
        });
        k_uct_emf<MET, R><<<grid_for(we, c->sms, 128), 128, 0, st>>>(
            p, bt, nb, face_set(c->Bf), (const R*)c->vel, (const R*)c->gsp[a], (const R*)c->gsp[b],
            (R*)c->emf3[3 - a - b], a, b, c->geotab);
        mark(c, HARMRAD_K_CT);
        ++nk;
      }
    if (cudaGetLastError() != cudaSuccess) return HARMRAD_E_CUDA;
    return nk;
  }
  if (p.act[0] + p.act[1] + p.act[2] >= 2) {  // flux-CT of every pair of active directions
    const long long we = all_work(c, [](const BoxGeo& x) { return (x.n[0] + 1LL) * (x.n[1] + 1) * (x.n[2] + 1); });
    FluxSet<R> F;
    for (int d = 0; d < 3; ++d) F.f[d] = (R*)c->F[d];
    k_emf<R><<<dim3(grid_for(we, c->sms, 256), 3), 256, 0, st>>>(p, bt, nb, F, (R*)c->emf, c->ncell);
    mark(c, HARMRAD_K_CT);
    k_ct<R><<<dim3(grid_for(2 * we, c->sms, 256), 3), 256, 0, st>>>(p, bt, nb, (const R*)c->emf, F, c->ncell);
    mark(c, HARMRAD_K_CT);
    nk += 2;
  }
  if (cudaGetLastError() != cudaSuccess) return HARMRAD_E_CUDA;
  return nk;
}

template <int MET, typename R>
int cfl_impl(harmrad_ctx* c) {
  int nk = faces_impl<MET, R>(c, true);
  if (nk < 0) return nk;
  Bufs b = make_bufs(c);
  k_cfl_init<<<1, 128, 0, c->stream>>>(b, c->nbox);
  mark(c, HARMRAD_K_CFL);
  k_cfl<R><<<grid_for(c->nact, c->sms, 256), 256, 0, c->stream>>>(c->dp, c->dboxes, c->nbox, b);
  mark(c, HARMRAD_K_CFL);
  k_cfl_finish<<<1, 128, 0, c->stream>>>(c->dp, b, c->nbox);
  mark(c, HARMRAD_K_CFL);
  if (cudaGetLastError() != cudaSuccess) return HARMRAD_E_CUDA;
  return nk + 3;
}

template <int MET, typename R>
int solve_impl(harmrad_ctx* c, int stage, const ImexStage& im) {
  const DevParams& p = c->dp;
  cudaStream_t st = c->stream;
  if (cudaMemsetAsync(c->qcount, 0, 4 * sizeof(int), st) != cudaSuccess) return HARMRAD_E_CUDA;
  if (cudaMemsetAsync(c->failed, 0, c->nact, st) != cudaSuccess) return HARMRAD_E_CUDA;
  mark(c, HARMRAD_K_OTHER);
  Bufs b = make_bufs(c);
  const int bu = fit_block(c, c->tune.update_block, 32);
  const int gu = grid_for(c->nact, c->sms, bu, c->tune.update_blocks_per_sm);
  const int split = c->tune.newton_split;
  const bool one = c->nbox == 1;
  const BoxGeo& b0 = c->boxes[0];
  const BoxGeo* bt = c->dboxes;
  const int nb = c->nbox;
  int nf = 0;
  if (p.emf == 1) {  // the staggered field's stage, then its periodic images
    EmfSet es;
    for (int e = 0; e < 3; ++e) es.e[e] = c->emf3[e];
    const bool rhs = !im.on || im.d != 0.0;
    for (int d = 0; d < 3; ++d) {
      long long wf = all_work(c, [d](const BoxGeo& x) {
        long long w = 1;
        for (int e = 0; e < 3; ++e) w *= (e == d && x.n[e] > 1) ? x.n[e] + 1 : x.n[e];
        return w;
      });
      k_face_update<R><<<grid_for(wf, c->sms, 256), 256, 0, st>>>(p, bt, nb, face_set(c->Bf), face_set(c->Bfn), es,
                                                                  c->dt, stage, im, rhs, d);
      mark(c, HARMRAD_K_CT);
    }
    nf = 3 + face_ghosts<MET>(c);
  }
  if (!im.on) {
    if (one && split == 0)
      k_update<MET, R, true, false, false><<<gu, bu, 0, st>>>(p, b0, bt, 1, b, stage, 0, im);
    else if (one)
      k_update<MET, R, true, true, false><<<gu, bu, 0, st>>>(p, b0, bt, 1, b, stage, split, im);
    else if (split == 0)
      k_update<MET, R, false, false, false><<<gu, bu, 0, st>>>(p, b0, bt, nb, b, stage, 0, im);
    else
      k_update<MET, R, false, true, false><<<gu, bu, 0, st>>>(p, b0, bt, nb, b, stage, split, im);
  } else {
    if (one && split == 0)
      k_update<MET, R, true, false, true><<<gu, bu, 0, st>>>(p, b0, bt, 1, b, stage, 0, im);
    else if (one)
      k_update<MET, R, true, true, true><<<gu, bu, 0, st>>>(p, b0, bt, 1, b, stage, split, im);
    else if (split == 0)
      k_update<MET, R, false, false, true><<<gu, bu, 0, st>>>(p, b0, bt, nb, b, stage, 0, im);
    else
      k_update<MET, R, false, true, true><<<gu, bu, 0, st>>>(p, b0, bt, nb, b, stage, split, im);
  }
  mark(c, HARMRAD_K_UPDATE);
  int nk = 4 + nf;
  if (split > 0) {
    // the continuation queue, the retry queue and the back-up list are
    // short: one persistent wave of blocks each, of one warp so that a queue shorter
    // than the wave spreads over all SMs
    const double hfac = im.on ? im.g : (stage == 0 ? 1.0 : (stage == 1 ? 0.25 : 2.0 / 3.0));
    k_newton_cont<MET, std::is_same<R, double>::value><<<c->sms * 8, 32, 0, st>>>(p, c->dboxes, b, hfac);
    mark(c, HARMRAD_K_UPDATE);
    ++nk;
  }
  k_retry<MET, std::is_same<R, double>::value><<<c->sms * 8, 32, 0, st>>>(p, c->dboxes, b, stage);
  mark(c, HARMRAD_K_RETRY);
  if (im.on && im.g > 0.0) {
    k_imex_store<MET><<<grid_for(c->nact, c->sms, 256), 256, 0, st>>>(p, c->dboxes, c->nbox, b, stage, im.g);
    mark(c, HARMRAD_K_UPDATE);
    ++nk;
  }
  k_backup_avg<<<c->sms, 128, 0, st>>>(p, c->dboxes, b);
  mark(c, HARMRAD_K_BACKUP);
  k_backup_apply<MET><<<c->sms, 128, 0, st>>>(p, c->dboxes, b);
  mark(c, HARMRAD_K_BACKUP);
  if (cudaGetLastError() != cudaSuccess) return HARMRAD_E_CUDA;
  return nk;
}

// --------------------------------------------------- point-wise entry kernels
template <int MET>
__global__ void k_zone_physics(DevParams p, BoxGeo bg, int n, const double* __restrict__ x,
                               const double* __restrict__ P, double* U, double* SM, double* F,
                               double* speeds) {
  for (int z = blockIdx.x * blockDim.x + threadIdx.x; z < n; z += gridDim.x * blockDim.x) {
    double x1 = x[4 * z + 1], x2 = x[4 * z + 2];
    Geo<MET, double> g = make_geo<MET, double>(p, x1, x2);
    double Pz[NPR];
    for (int q = 0; q < NPR; ++q) Pz[q] = P[NPR * z + q];
    for (int d = 1; d <= 3; ++d) {
      double Uq[NPR], Fq[NPR], sp[4];
      face_state<MET, double>(p, g, d, bg.dx[d - 1], 1.0, Pz, Uq, Fq, sp);
      if (F)
        for (int q = 0; q < NPR; ++q) F[(3 * z + d - 1) * NPR + q] = Fq[q];
      if (speeds)
        for (int q = 0; q < 4; ++q) speeds[(3 * z + d - 1) * 4 + q] = sp[q];
      if (d == 1 && U)
        for (int q = 0; q < NPR; ++q) U[NPR * z + q] = Uq[q];
    }
    if (SM) {
      double S[NPR];
      for (int q = 0; q < NPR; ++q) S[q] = 0.0;
      if constexpr (MET == KS) {
        double ucon[4], ucov[4], gm, bcon[4], bcov[4], bsq, urc[4], urv[4], gr;
        fourvel<MET, double>(g, Pz[U1], Pz[U2], Pz[U3], ucon, ucov, &gm);
        bvec<MET, double>(g, ucon, ucov, Pz[B1], Pz[B2], Pz[B3], bcon, bcov, &bsq);
        fourvel<MET, double>(g, Pz[UR1], Pz[UR2], Pz[UR3], urc, urv, &gr);
        double pg = (p.gam - 1.0) * Pz[UU];
        double wb = Pz[RHO] + Pz[UU] + pg + bsq, pt = pg + 0.5 * bsq;
        double e43 = (4.0 / 3.0) * Pz[ER];
        MetricDeriv md = ks_derivs(p, x1, x2);
        for (int m = 0; m < 2; ++m) {
          S[2 + m] = 0.5 * g.gdet * (wb * qform(md, m, ucon) - qform(md, m, bcon)) + pt * md.sg[m];
          S[9 + m] = 0.5 * g.gdet * e43 * qform(md, m, urc) + Pz[ER] * (1.0 / 3.0) * md.sg[m];
        }
      }
      for (int q = 0; q < NPR; ++q) SM[NPR * z + q] = S[q];
    }
  }
}

template <int MET>
__global__ void k_zone_implicit(DevParams p, BoxGeo bg, int n, const double* __restrict__ x,
                                const double* __restrict__ Us, const double* __restrict__ Ps,
                                const double* __restrict__ hh, const double* __restrict__ Sst, double* Pout,
                                double* eTo, int* itso, unsigned char* meth) {
  for (int z = blockIdx.x * blockDim.x + threadIdx.x; z < n; z += gridDim.x * blockDim.x) {
    double x1 = x[4 * z + 1], x2 = x[4 * z + 2];
    Geo<MET, double> g = make_geo<MET, double>(p, x1, x2);
    double Ust[NPR], P0[NPR];
    for (int q = 0; q < NPR; ++q) {
      Ust[q] = Us[NPR * z + q];
      P0[q] = Ps[NPR * z + q];
    }
    // PMHD term by term: the outcome of a zone near a method's threshold (a whole
    // value) follows the last bits of the residual
    ImpSys<MET, false> s;
    build_sys<MET>(p, g, Ust, hh[z], 1.0, s);
    double x0[4] = {P0[UU], P0[U1], P0[U2], P0[U3]};
    double kabs, ksca;
    opacity<double>(p, P0[RHO], P0[UU], 1.0, &kabs, &ksca);
    double dl = 0.0;
    for (int d = 1; d <= 3; ++d)
      if (p.act[d - 1]) dl = fmax(dl, sqrt(g.gdd(d)) * bg.dx[d - 1]);
    if ((kabs + ksca) * dl < 2.0 / 3.0) {
      double go[5], T3[3] = {s.Ts[1], s.Ts[2], s.Ts[3]};
      if (gas_invert_ieee<MET>(p, g, s.Dlab, s.Ts[0], T3, s.B, P0, 1e-9, go) == 0) {
        x0[0] = go[1];
        x0[1] = go[2];
        x0[2] = go[3];
        x0[3] = go[4];
      }
    }
    double bx[4] = {0.0, 0.0, 0.0, 0.0}, beT = HUGE_VAL;
    // extremely sub-dominant radiation (Sec. 4.10): no PMHD attempt
    const bool subdom = radiation_subdominant<MET>(g, Ust, P0);
    int steps = subdom ? 0 : newton_pmhd<MET>(p, s, x0, bx, &beT);
    double Pn[NPR];
    int method = 0;
    double eT = beT;
    if (beT < 1e-9) {
      pmhd_final<MET>(p, s, bx, Pn);
    } else {
      int rs;
      const double tau = zone_tau<MET>(p, g, bg.dx, P0, 1.0);
      const double sz = Sst ? Sst[z] : NAN;
      ImpSys<MET> s;
      build_sys<MET>(p, g, Ust, hh[z], 1.0, s);
      method = retry_sequence<MET>(p, g, s, P0, bx, beT, tau, Pn, &eT, &rs, subdom, sz);
      steps += rs;
      if (method == ST_BACKUP) {  // the entropy (S* given), then the cold-MHD equations
        const int by = backup_equations<MET>(p, g, s, Ust, P0, sz, 1, tau, Pn, &eT, &steps);
        if (by) method = by == METH_COLD ? METH_COLD : METH_ENTROPY;
      }
    }
    for (int q = 0; q < NPR; ++q) Pout[NPR * z + q] = Pn[q];
    if (eTo) eTo[z] = eT;
    if (itso) itso[z] = steps;
    if (meth) meth[z] = (unsigned char)method;
  }
}

// One Newton method alone on each of n independent zones (test hook, the
// counterpart of the oracle's method hook): 0 PMHD from the gas of Ps, 1 URAD
// from R^t_nu of Ps, 2 PRAD from the radiation of Ps, 3 staged PMHD from the
// gas of Ps with u_g from the explicit entropy Sst (if given), 4 staged URAD,
// 5 staged PRAD (guesses as 1 and 2), 6, 7, 8 the entropy-based PMHD, URAD,
// PRAD (the entropy equation with the explicit entropy Sst; guesses as 0-2).  Writes the
// best iterate's primitives as its error function forms them (TYPE2
// radiation; Ps if none), its e_T (inf if none) and the Newton steps.
template <int MET>
__global__ void k_zone_method(DevParams p, BoxGeo bg, int n, const double* __restrict__ x,
                              const double* __restrict__ Us, const double* __restrict__ Ps,
                              const double* __restrict__ hh, const double* __restrict__ Sst, int method,
                              double* Pout, double* eTo, int* itso) {
  for (int z = blockIdx.x * blockDim.x + threadIdx.x; z < n; z += gridDim.x * blockDim.x) {
    const Geo<MET, double> g = make_geo<MET, double>(p, x[4 * z + 1], x[4 * z + 2]);
    double Ust[NPR], P0[NPR], Pn[NPR];
    for (int q = 0; q < NPR; ++q) {
      Ust[q] = Us[NPR * z + q];
      P0[q] = Pn[q] = Ps[NPR * z + q];
    }
    ImpSys<MET> s;
    build_sys<MET>(p, g, Ust, hh[z], 1.0, s);
    if (method >= 6) {  // the entropy-based PMHD, URAD, PRAD
      s.entropy = true;
      s.Sstar = Sst ? Sst[z] / g.gdet : 0.0;
      method -= 6;
    }
    double eT = HUGE_VAL;
    int steps = 0;
    if (method == 0 || method == 3) {
      double x0[4] = {P0[UU], P0[U1], P0[U2], P0[U3]}, bx[4];
      if (method == 3 && Sst) entropy_ug_guess(p, Sst[z], s.Dlab * g.gdet, P0[RHO], x0);
      steps = method == 0 ? newton_pmhd<MET>(p, s, x0, bx, &eT) : newton_pmhd_staged<MET>(p, s, x0, bx, &eT);
      if (isfinite(eT)) {
        ImpRes rr;
        ImpState st;
        pmhd_res<MET>(p, s, bx, rr, &st, false);
        Pn[RHO] = st.rho;
        for (int c = 0; c < 4; ++c) Pn[UU + c] = bx[c];
        for (int c = 0; c < 4; ++c) Pn[ER + c] = st.Pr[c];
        for (int c = 0; c < 3; ++c) Pn[B1 + c] = s.B[c];
      }
    } else {
      double gas[5] = {P0[RHO], P0[UU], P0[U1], P0[U2], P0[U3]}, bx[4], bgas[5];
      if (method == 1 || method == 4) {
        double urc[4], urv[4], gr;
        fourvel<MET, double>(g, P0[UR1], P0[UR2], P0[UR3], urc, urv, &gr);
        const double e43 = (4.0 / 3.0) * P0[ER];
        double xr[4];
        xr[0] = e43 * urc[0] * urv[0] + P0[ER] * (1.0 / 3.0);
        for (int c = 1; c < 4; ++c) xr[c] = e43 * urc[0] * urv[c];
        steps = method == 1 ? newton_urad<MET>(p, s, xr, gas, bx, bgas, &eT)
                            : newton_rad_staged<MET, false>(p, s, xr, gas, bx, bgas, &eT);
        if (isfinite(eT)) rad_invert<MET>(p, g, bx, 2, Pn + ER);
      } else {
        double xq[4] = {P0[ER], P0[UR1], P0[UR2], P0[UR3]};
        steps = method == 2 ? newton_rad<MET, true>(p, s, xq, gas, bx, bgas, &eT)
                            : newton_rad_staged<MET, true>(p, s, xq, gas, bx, bgas, &eT);
        if (isfinite(eT))
          for (int c = 0; c < 4; ++c) Pn[ER + c] = bx[c];
      }
      if (isfinite(eT)) {
        for (int c = 0; c < 5; ++c) Pn[c] = bgas[c];
        for (int c = 0; c < 3; ++c) Pn[B1 + c] = s.B[c];
      }
    }
    for (int q = 0; q < NPR; ++q) Pout[NPR * z + q] = Pn[q];
    eTo[z] = eT;
    itso[z] = steps;
  }
}

template <int MET>
int Run<MET>::zone_method(const DevParams& dp, const BoxGeo& bg, int n, const double* x, const double* Us,
                          const double* Ss, const double* Ps, const double* h, int method, double* Pout,
                          double* eT, int* iters, cudaStream_t st, int sms) {
  k_zone_method<MET><<<grid_for(n, sms, 128), 128, 0, st>>>(dp, bg, n, x, Us, Ps, h, Ss, method, Pout, eT, iters);
  return cudaGetLastError() == cudaSuccess ? 1 : HARMRAD_E_CUDA;
}

template <int MET>
int Run<MET>::init_faces(harmrad_ctx* c, bool from_centres) {
  fill_ghost_cells(c);
  if (from_centres)
    k_faces_from_centres<MET><<<grid_for(c->ncell, c->sms, 256), 256, 0, c->stream>>>(
        c->dp, c->dboxes, c->nbox, c->P, face_set(c->Bf), c->geotab);
  face_ghosts<MET>(c);
  k_centre_B<MET><<<grid_for(c->nact, c->sms, 256), 256, 0, c->stream>>>(c->dp, c->dboxes, c->nbox, c->P,
                                                                           face_set(c->Bf), c->geotab);
  return cudaGetLastError() == cudaSuccess ? 0 : HARMRAD_E_CUDA;
}
template <int MET>
int Run<MET>::faces(harmrad_ctx* c, bool fresh) {
  return c->real_size == 8 ? faces_impl<MET, double>(c, fresh) : faces_impl<MET, float>(c, fresh);
}
template <int MET>
int Run<MET>::cfl(harmrad_ctx* c) {
  return c->real_size == 8 ? cfl_impl<MET, double>(c) : cfl_impl<MET, float>(c);
}
template <int MET>
int Run<MET>::solve(harmrad_ctx* c, int stage, const ImexStage& im) {
  return c->real_size == 8 ? solve_impl<MET, double>(c, stage, im) : solve_impl<MET, float>(c, stage, im);
}
template <int MET>
int Run<MET>::zone_physics(const DevParams& dp, const BoxGeo& bg, int n, const double* x,
                           const double* P, double* U, double* SM, double* F, double* speeds,
                           cudaStream_t st, int sms) {
  k_zone_physics<MET><<<grid_for(n, sms, 128), 128, 0, st>>>(dp, bg, n, x, P, U, SM, F, speeds);
  return cudaGetLastError() == cudaSuccess ? 1 : HARMRAD_E_CUDA;
}
template <int MET>
int Run<MET>::zone_implicit(const DevParams& dp, const BoxGeo& bg, int n, const double* x,
                            const double* Us, const double* Ss, const double* Ps, const double* h,
                            double* Pout, double* eT, int* iters, unsigned char* method, cudaStream_t st,
                            int sms) {
  k_zone_implicit<MET><<<grid_for(n, sms, 128), 128, 0, st>>>(dp, bg, n, x, Us, Ps, h, Ss, Pout, eT, iters,
                                                              method);
  return cudaGetLastError() == cudaSuccess ? 1 : HARMRAD_E_CUDA;
}

}  // namespace hr

// kernels_fp64.cu -- FP64 stage of the explicit MHD scheme, one kernel per
// step of the paper's algorithm, with per-stage scratch in HBM.
//
//   k_prim        primitives + EOS at every cell the stencils touch, as
//                 deviations from the background (Sects. 2.2, 2.8); ghost
//                 cells are produced by mapping to their interior source cell
//                 (Table bcs) -- no ghost storage in the state.
//   k_flag_raw    shock indicator of Sect. 2.7 on interior cells, then its 5^d
//                 dilation (launch_flags).
//   k_flux_walk   van Leer PLM of the deviations (Sect. 2.5), background added
//                 at the face, LHLLD / HLL flux minus F_hat (Eqs. flux-hlld,
//                 pstar, wb1), several faces per thread; k_flux for the other
//                 reconstructions.
//   k_emf_all     Contact-CT edge EMFs (Sect. 2.4).
//   k_update_*    residual with sources (Eqs. fv, spatres, wb2) and the SSP-RK
//                 combination for cells and faces (Sect. 2.9).
//   k_dt          CFL condition (Eq. cfl) for phl_compute_dt; a step takes it
//                 from its first stage's k_prim.
//
// The FP64 pipe bounds the stage: 128 x 96 x 112 cells take 3.6 ms, 2.8 of
// them in the faces (6.5 and 5.1 ms with full-range divisions and roots,
// every slope formed twice, a CFL pass of its own and three launches for each
// of the EMFs and face updates).
#include <math.h>

#include "phl_internal.cuh"
#include "stage_common.cuh"

namespace phl {
using namespace stage;
namespace {

// Primitive deviations of interior cell (i, j, k) from the conserved state.
// Returns false (and sets the device flag) for rho <= 0, P <= 0 or NaN.
__device__ __forceinline__ bool cell_prims(const DevGeo &G, const double *__restrict__ U,
                                           const double *__restrict__ Bf, int i, int j, int k,
                                           double *w, int *dflag) {
  const long p = sidx(G, i, j, k);
  const long pl = G.plane;
  const double rho = U[p];
  const double ir = rcp_nr(rho);
  const double mx = U[pl + p], my = U[2 * pl + p], mz = U[3 * pl + p];
  const double vx = mx * ir, vy = my * ir, vz = mz * ir;
  const double bx = 0.5 * (Bf[p] + Bf[p + 1]);
  const double by = 0.5 * (Bf[pl + p] + Bf[pl + p + G.sy]);
  const double bz = 0.5 * (Bf[2 * pl + p] + Bf[2 * pl + p + G.sz]);
  const double P = (G.gamma - 1.0) * (U[4 * pl + p] - 0.5 * (mx * vx + my * vy + mz * vz) - 0.5 * (bx * bx + by * by + bz * bz));
  const Bg b = bg_cell(G, k);
  w[W_RHO] = rho - b.rho;
  w[W_VX] = vx; w[W_VY] = vy; w[W_VZ] = vz;
  w[W_BX] = bx; w[W_BY] = by; w[W_BZ] = bz;
  w[W_P] = P - b.p;
  w[W_GE] = G.gamma - b.ge;
  w[W_GC] = G.gamma - b.gc;
#pragma unroll
  for (int l = 0; l < PHL_NSPEC_MAX; ++l)
    if (l < G.nspec) w[W_X0 + l] = U[(U_X0 + l) * pl + p] * ir;
  bool ok = true;
  if (!(rho > 0.0) || !(P > 0.0)) { atomicOr(dflag, FLAG_NEG); ok = false; }
  if (!isfinite(P) || !isfinite(rho)) { atomicOr(dflag, FLAG_NAN); ok = false; }
  return ok;
}

// CFL sum of a cell from its deviations w at height k (Eq. cfl).
__device__ __forceinline__ double dt_rate(const DevGeo &G, const double *w, int k) {
  const Bg b = bg_cell(G, k);
  const double ir = rcp_nr(w[W_RHO] + b.rho), P = w[W_P] + b.p, gc = w[W_GC] + b.gc;
  const double a2 = gc * P * ir;
  const double ab = a2 + (w[W_BX] * w[W_BX] + w[W_BY] * w[W_BY] + w[W_BZ] * w[W_BZ]) * ir;
  double s = 0.0;
  for (int d = 0; d < 3; ++d) {
    if (!G.act[d]) continue;
    double disc = ab * ab - 4.0 * a2 * (w[W_BX + d] * w[W_BX + d] * ir);
    if (disc < 0.0) disc = 0.0;
    s += (fabs(w[W_VX + d]) + sqrt_nr(0.5 * (ab + sqrt_nr(disc)))) * G.idx[d];
  }
  return (s == s) ? s : INFINITY;
}

__device__ __forceinline__ void atomic_max_pos(unsigned long long *addr, double v) {
  // non-negative doubles order like their bit patterns
  atomicMax(addr, (unsigned long long)__double_as_longlong(v));
}
// Block maximum of m into *dmax (every thread of the block calls).
__device__ __forceinline__ void block_dmax(double m, unsigned long long *dmax) {
  for (int o = 16; o > 0; o >>= 1) m = fmax(m, __shfl_xor_sync(0xffffffffu, m, o));
  __shared__ double red[TPB / 32];
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = m;
  __syncthreads();
  if (threadIdx.x == 0) {
    double v = red[0];
    for (int w = 1; w < (int)(blockDim.x >> 5); ++w) v = fmax(v, red[w]);
    atomic_max_pos(dmax, v);
  }
}

// dmax (the step's first stage with the device CFL step; else null): the CFL
// maximum of the interior cells from the deviations just formed, instead of a
// second pass over the state.
__global__ void __launch_bounds__(256) k_prim(DevGeo G, Box box, const double *__restrict__ U,
                                              const double *__restrict__ Bf, double *__restrict__ W, int *dflag,
                                              unsigned long long *dmax, unsigned int *any) {
  int c[3], s[3];
  double rate = 0.0;
  if (blockIdx.x == 0 && threadIdx.x == 0) *any = 0u;   // the raw-flag kernel's vote, taken after this kernel
  if (cell3(box, c)) {
    bool fl[3], in = true;
    for (int d = 0; d < 3; ++d) {
      fl[d] = false;
      s[d] = G.act[d] ? cell_src(c[d], G.n[d], G.bc[d][0], G.bc[d][1], fl[d]) : 0;
      in = in && c[d] >= 0 && c[d] < G.n[d];
    }
    double w[NW_MAX];
    cell_prims(G, U, Bf, s[0], s[1], s[2], w, dflag);
    if (dmax && in) rate = dt_rate(G, w, c[2]);
    for (int d = 0; d < 3; ++d)
      if (fl[d]) { w[W_VX + d] = -w[W_VX + d]; w[W_BX + d] = -w[W_BX + d]; }
    const long q = widx(G, c[0], c[1], c[2]);
#pragma unroll
    for (int v = 0; v < NW_MAX; ++v)   // an ideal gas reconstructs no gamma deviations
      if (v < G.nw && v != W_GE && v != W_GC) W[v * G.wtot + q] = w[v];
  }
  if (dmax) block_dmax(rate, dmax);
}

__device__ __forceinline__ void update_cell(const DevGeo &G, const Box &box, long tl, const StageBufs &S) {
  const double dt = *S.dt;
  {
    int c[3];
    if (!cell_at(box, tl, c)) return;
    const long p = widx(G, c[0], c[1], c[2]);
    const long ps = sidx(G, c[0], c[1], c[2]);
    const long wt = G.wtot, pl = G.plane;
    double r[5 + PHL_NSPEC_MAX];
#pragma unroll
    for (int v = 0; v < 5 + PHL_NSPEC_MAX; ++v) {
      if (v >= G.nv) continue;
      const int fc = v < 5 ? v : F_X0 + (v - U_X0);
      double s = 0.0;
      for (int d = 0; d < 3; ++d) {
        if (!G.act[d]) continue;
        const double *f = S.F[d] + fc * wt;
        s += (f[p + wstride(G, d)] - f[p]) * G.idx[d];
      }
      r[v] = s;
    }
    const double rho = S.Uin[ps];
    const double rhohat = bg_cell(G, c[2]).rho;
    double se = 0.0;
    for (int d = 0; d < 3; ++d) {
      r[U_MX + d] -= (rho - rhohat) * G.g[d];
      se += S.Uin[(U_MX + d) * pl + ps] * G.g[d];
    }
    if (G.heat) se += G.heat[c[2]];
    r[U_E] -= se;
#pragma unroll
    for (int v = 0; v < 5 + PHL_NSPEC_MAX; ++v) {
      if (v >= G.nv) continue;
      const long q = v * pl + ps;
      S.Uout[q] = S.a * S.Ubase[q] + S.b * S.Uin[q] - S.b * dt * r[v];
    }
  }
}

__global__ void k_update_cells(DevGeo G, Box box, StageBufs S) {
  update_cell(G, box, blockIdx.x * (long)blockDim.x + threadIdx.x, S);
}

// Edge EMFs and the cell update in one launch (small grids): both need the
// faces only.  The first nemf blocks take the sites.
__global__ void __launch_bounds__(256) k_emf_cells(DevGeo G, Box bsite, Box bcell, unsigned nemf, StageBufs S) {
  if (blockIdx.x < nemf) {
    int c[3];
    if (cell3(bsite, c)) emf_sites<double>(G, c, S.W, S.F[0], S.F[1], S.F[2], S.E);
  } else {
    update_cell(G, bcell, (blockIdx.x - nemf) * (long)blockDim.x + threadIdx.x, S);
  }
}

template <int D>
__device__ __forceinline__ void face_update_fp64(const DevGeo &G, const int *c, const StageBufs &S, double dt) {
  constexpr int A = (D + 1) % 3, B = (D + 2) % 3;
  int e[3] = {c[0], c[1], c[2]};
  if (!G.act[D]) e[D] = 0;
  const long p = widx(G, e[0], e[1], e[2]);
  const long wt = G.wtot;
  double r = 0.0;
  if (G.act[A]) r += (S.E[(long)B * wt + p + wstride(G, A)] - S.E[(long)B * wt + p]) * G.idx[A];
  if (G.act[B]) r -= (S.E[(long)A * wt + p + wstride(G, B)] - S.E[(long)A * wt + p]) * G.idx[B];
  const long q = (long)D * G.plane + sidx(G, c[0], c[1], c[2]);
  S.Bout[q] = S.a * S.Bbase[q] + S.b * S.Bin[q] - S.b * dt * r;
}
// The three face components of a site (box: [0, n] along every axis).  Every
// face array is written: a field with no active curl direction still takes
// the RK combination a * base + b * in.
__global__ void k_update_faces(DevGeo G, Box box, StageBufs S) {
  int c[3];
  if (!cell3(box, c)) return;
  const double dt = *S.dt;
  const bool in[3] = {c[0] < G.n[0], c[1] < G.n[1], c[2] < G.n[2]};
  if (in[1] && in[2]) face_update_fp64<0>(G, c, S, dt);
  if (in[0] && in[2]) face_update_fp64<1>(G, c, S, dt);
  if (in[0] && in[1]) face_update_fp64<2>(G, c, S, dt);
}

__global__ void k_dt(DevGeo G, Box box, const double *__restrict__ U, const double *__restrict__ Bf,
                     unsigned long long *dmax, int *dflag) {
  double m = 0.0;
  for (long t = blockIdx.x * (long)blockDim.x + threadIdx.x; t < box.n; t += (long)gridDim.x * blockDim.x) {
    int c[3];
    unflat(box, t, c);
    double w[NW_MAX];
    cell_prims(G, U, Bf, c[0], c[1], c[2], w, dflag);
    const double r = dt_rate(G, w, c[2]);
    if (r > m) m = r;
  }
  block_dmax(m, dmax);
}

__global__ void k_dt_finalize(double cfl, unsigned long long *dmax, double *dt) {
  const double m = __longlong_as_double((long long)*dmax);
  *dt = cfl / m;
  *dmax = 0ull;
}

__global__ void k_set_scalar(double *p, double v) { *p = v; }

}  // namespace

void launch_set_scalar(double *p, double v, cudaStream_t s, Prof *prof) { PHL_LAUNCH(KC_SCALAR, prof, s, k_set_scalar<<<1, 1, 0, s>>>(p, v)); }

void launch_dt_fp64(const DevGeo &G, const double *U, const double *Bf, double *T, unsigned long long *dmax,
                    double *dt, int *dflag, cudaStream_t s, int *nlaunch, Prof *prof) {
  (void)T;
  Box b = make_box(0, G.n[0], 0, G.n[1], 0, G.n[2]);
  PHL_LAUNCH(KC_DT, prof, s, k_dt<<<nblocks(b.n), TPB, 0, s>>>(G, b, U, Bf, dmax, dflag));
  PHL_LAUNCH(KC_DT, prof, s, k_dt_finalize<<<1, 1, 0, s>>>(G.cfl, dmax, dt));
  if (nlaunch) *nlaunch += 2;
}

void launch_stage_fp64(const DevGeo &G, const StageBufs &S, cudaStream_t s, int *nlaunch, Prof *prof) {
  int nl = 0;
  auto rng = [&](int d, int lo_g, int hi_extra, int &lo, int &hi) {
    if (G.act[d]) { lo = -lo_g; hi = G.n[d] + hi_extra; }
    else { lo = 0; hi = 1; }
  };
  // (1) primitives on cells [-ge, n+ge) of every active dimension (ge: the work layout's ghost layers)
  {
    int l[3], h[3];
    for (int d = 0; d < 3; ++d) rng(d, G.ge[d], G.ge[d], l[d], h[d]);
    Box b = make_box(l[0], h[0], l[1], h[1], l[2], h[2]);
    if (G.eos == 1) {
      launch_eos_cells<double>(G, S.Uin, S.Bin, nullptr, nullptr, S.Tin, S.Tout, S.W, S.dflag, s, &nl, prof,
                               S.cfl_dmax, const_cast<double *>(S.dt));
    } else {
      const unsigned t = tpb_for(G, b.n);
      PHL_LAUNCH(KC_PRIM, prof, s, k_prim<<<gridt(b, t), t, 0, s>>>(G, b, S.Uin, S.Bin, S.W, S.dflag, S.cfl_dmax, S.any));
      if (S.cfl_dmax) {
        PHL_LAUNCH(KC_DT, prof, s, k_dt_finalize<<<1, 1, 0, s>>>(G.cfl, S.cfl_dmax, const_cast<double *>(S.dt)));
        ++nl;
      }
      ++nl;
    }
  }
  // (2) shock flags
  if (G.eps_sf > 0.0)
    nl += launch_flags<double>(G, S.W, S.raw, S.raw + (long)G.n[0] * G.n[1] * G.n[2], S.flag, S.any, s, prof,
                               G.eos != 1);
  // (3) fluxes: normal faces [0, n], one transverse ghost row each side
  Box bf[3];
  long most = 0;
  for (int D = 0; D < 3; ++D) {
    int l[3], h[3];
    for (int d = 0; d < 3; ++d) {
      if (d == D) { l[d] = 0; h[d] = G.n[d] + 1; }
      else rng(d, 1, 1, l[d], h[d]);
    }
    bf[D] = make_box(l[0], h[0], l[1], h[1], l[2], h[2]);
    if (G.act[D] && bf[D].n > most) most = bf[D].n;
  }
  // one launch for all directions, and one for the EMFs and the cell update,
  // where a direction's faces are fewer than the GPU's threads in a wave (128
  // x 128: 40 + 12 -> 28 + 8 us a stage, and two launches fewer; a step in
  // both forms: 128^2 177 and 236 us, 256^2 432 and 467, 32^3 442 and 466, and
  // above the line 288^2 574 and 644, 56^3 1614 and 1723)
  // (a grid without an active axis has no faces: nothing to launch for them)
  const bool small = most > 0 && most < G.sms * 512L && G.recon == PHL_RECON_VANLEER;
  if (small) {
    FaceSet<double> A{};
    const unsigned t = most < G.sms * 128L ? 32u : 64u;
    unsigned blocks = 0;
    for (int D = 0; D < 3; ++D) {
      A.first[D] = ~0u;
      if (!G.act[D]) continue;
      A.box[D] = bf[D];
      A.F[D] = S.F[D];
      A.Bf[D] = S.Bin;
      A.first[D] = blocks;
      blocks += (unsigned)((bf[D].n + t - 1) / t);
    }
    if (G.nspec == 0)
      PHL_LAUNCH(KC_FLUX_X, prof, s, (k_flux_all<double, 0><<<blocks, t, 0, s>>>(G, A, S.W, S.flag, S.dflag)));
    else
      PHL_LAUNCH(KC_FLUX_X, prof, s, (k_flux_all<double, PHL_NSPEC_MAX><<<blocks, t, 0, s>>>(G, A, S.W, S.flag, S.dflag)));
    ++nl;
  }
  for (int D = 0; D < 3 && !small; ++D) {
    if (!G.act[D]) continue;
    launch_flux<double>(D, G, bf[D], S.W, S.Bin, (const double *)nullptr, S.flag, S.F[D], S.dflag, s, prof);
    ++nl;
  }
  // (4) edge EMFs
  const Box bs = site_box(G), bc = make_box(0, G.n[0], 0, G.n[1], 0, G.n[2]);
  if (small) {
    const unsigned t = tpb_for(G, bs.n), nemf = gridt(bs, t).x;
    PHL_LAUNCH(KC_EMF, prof, s, k_emf_cells<<<nemf + gridt(bc, t).x, t, 0, s>>>(G, bs, bc, nemf, S));
    ++nl;
  } else {
    const unsigned t = tpb_for(G, bs.n);
    PHL_LAUNCH(KC_EMF, prof, s, k_emf_all<double><<<gridt(bs, t), t, 0, s>>>(G, bs, S.W, S.F[0], S.F[1], S.F[2], S.E));
    PHL_LAUNCH(KC_UPDATE_CELLS, prof, s, k_update_cells<<<gridt(bc, t), t, 0, s>>>(G, bc, S));
    nl += 2;
  }
  // (5) face updates
  {
    const Box bu = make_box(0, G.n[0] + 1, 0, G.n[1] + 1, 0, G.n[2] + 1);
    const unsigned t = tpb_for(G, bu.n);
    PHL_LAUNCH(KC_UPDATE_FACES, prof, s, k_update_faces<<<gridt(bu, t), t, 0, s>>>(G, bu, S));
    ++nl;
  }
  if (nlaunch) *nlaunch += nl;
}

}  // namespace phl

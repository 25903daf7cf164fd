// eos_stellar.cuh -- stellar equation of state on the device (Sect. 2.2, item ii).
//
// Ions (ideal gas), radiation (Eqs. prad, erad) and an electron-positron gas
// in pair equilibrium.  The e-/e+ part is a table of its Helmholtz
// free-energy density f over (x, y) = (ln n_e, ln T), n_e = rho Y_e N_A,
// holding at each node f and its derivatives f_x, f_y, f_xx, f_yy, f_xy,
// f_xxy, f_xyy, f_xxyy (eos_nodes.cuh), interpolated biquintically as the
// paper does with its Helmholtz table: the tensor product of quintic Hermite
// polynomials, which takes f and its derivatives up to second order in each
// variable from the nodes.  P = f_x - f, e = (f - f_y) / rho,
// c_v = (f_y - f_yy) / (rho T), dP/dT = (f_xy - f_y) / T,
// dP/drho = (f_xx - f_x) / rho all come from one interpolant, so the
// thermodynamic identities hold for the interpolated EOS, and c_v, gamma_c
// are continuous.
//
// Evaluation.  The interpolant on a table cell is one polynomial of degree 5
// in each of u, v (the position inside the cell along x and y, in cell
// units); its 36 coefficients c[r][p] (of u^p v^r) are formed once with the
// table.  The FP64 pipe bounds every inversion (1/64 of the FP32 rate on this
// GPU), so the evaluation is laid out for the fewest FP64 instructions:
// synthetic division (Horner's scheme carried on to the derivatives) gives
// value, first and half the second derivative of a degree-5 polynomial in
// 5 + 4 + 3 multiply-adds, so f, f_x, f_xx of the six rows take 72 and the six
// needed mixed derivatives 26 more.  The Hermite form it replaces (two bases
// of 62 operations, 108 + 36 multiply-adds) took 268.  With the shared
// subexpressions below and integer tests for compares and conversions, the
// recorded inversion of the stellar box went from 2.12 to 0.95 ms per launch on
// 128^3 cells, the shell's kernel from 2.40 to 0.95 ms on 2.36 million cells
// and the batch inversion from 4.63 to 1.99 ms for 10^6 far guesses; FP64 pipe
// bound as before.  The coefficients above
// the constant are the size of the cell's own differences, so no derivative
// cancels node values at evaluation; their set-up works on differences too.
#pragma once
#include <cuda_runtime.h>
#include <math.h>

#include "fp64_math.cuh"

namespace phl {
namespace eos {

// CODATA 2018 (CGS)
constexpr double KB = 1.380649e-16;
constexpr double MEC2 = 8.1871057769e-7;
constexpr double HPL = 6.62607015e-27;
constexpr double CL = 2.99792458e10;
constexpr double NAV = 6.02214076e23;
constexpr double ARAD = 7.565733250e-15;
constexpr double ARAD_QUARTER = 2.9492579329135276e-04;   // ARAD^(1/4)
constexpr double RGAS = KB * NAV;
constexpr double PI_D = 3.14159265358979323846;
constexpr int NQ = 9;          // node values: f, f_x, f_y, f_xx, f_yy, f_xy, f_xxy, f_xyy, f_xxyy
constexpr int NC1 = 6;         // coefficients of the quintic per direction
constexpr int NCF = NC1 * NC1; // coefficients of a table cell: [power of v][power of u]

// node slot of d^(p + r) f / dx^p dy^r
__host__ __device__ __forceinline__ int qslot(int p, int r) {
  return p == 0 ? 2 * r : (p == 1 ? (r == 0 ? 1 : 3 + 2 * r) : (r == 0 ? 3 : 4 + 2 * r));
}

struct Table {
  int nx, ny;
  double x0, dx, y0, dy;      // x = ln n_e, y = ln T
  const double *c;            // [ny-1][nx-1][NCF] polynomial coefficients in cell units
  const float *cf;            // FP32 copy
  float x0f, y0f;
  double idx, idy;            // 1/dx, 1/dy
  float idxf, idyf;
  double idxdy, idx2x2, idy2x2;   // idx idy, 2 idx^2, 2 idy^2 (the second derivatives come halved)
  float idxdyf, idx2x2f, idy2x2f;
  double Tlo, Thi;            // the table's temperature range, exp(y0) and
  float Tlof, Thif;           // exp(y0 + (ny - 1) dy), set with the table
};

// Position along x (x = ln n_e): table interval and fraction, fixed during
// an inversion.
template <typename R> struct XB {
  int i;
  bool ok;
  R u;
};

template <typename R>
__device__ __forceinline__ XB<R> xbasis(const Table &t, R x) {
  XB<R> X;
  const R x0 = sizeof(R) == 8 ? (R)t.x0 : (R)t.x0f, idx = sizeof(R) == 8 ? (R)t.idx : (R)t.idxf;
  X.i = 0;
  X.u = R(0);
  X.ok = interval((x - x0) * idx, t.nx - 1, X.i, X.u);
  return X;
}

// Value, first and half the second derivative (D = 0, 1, 2 selects how many)
// of the polynomial sum_k q[k] w^k by synthetic division.
template <typename R, int D>
__device__ __forceinline__ void horner5(const R *q, R w, R &h, R &d, R &e) {
  const R h4 = fma(q[5], w, q[4]), h3 = fma(h4, w, q[3]), h2 = fma(h3, w, q[2]), h1 = fma(h2, w, q[1]);
  h = fma(h1, w, q[0]);
  if (D >= 1) {
    const R d3 = fma(q[5], w, h4), d2 = fma(d3, w, h3), d1 = fma(d2, w, h2);
    d = fma(d1, w, h1);
    if (D >= 2) {
      const R e2 = fma(q[5], w, d3), e1 = fma(e2, w, d2);
      e = fma(e1, w, d1);
    }
  }
}

// The six coefficients of u^0 .. u^5 of row r (power of v) of a table cell.
template <typename R>
__device__ __forceinline__ void cell_row(const Table &t, long cell, int r, R *q) {
  if constexpr (sizeof(R) == 8) {   // 16-byte loads: a row is 48 bytes, a cell 288
    const double2 *p = reinterpret_cast<const double2 *>(t.c + cell * NCF) + 3 * r;
#pragma unroll
    for (int k = 0; k < 3; ++k) { const double2 w = __ldg(p + k); q[2 * k] = w.x; q[2 * k + 1] = w.y; }
  } else {
    const float2 *p = reinterpret_cast<const float2 *>(t.cf + cell * NCF) + 3 * r;
#pragma unroll
    for (int k = 0; k < 3; ++k) { const float2 w = __ldg(p + k); q[2 * k] = w.x; q[2 * k + 1] = w.y; }
  }
}

// f at fixed x on y-interval j as a polynomial in v, for the iterations that
// stay in one interval.
template <typename R> struct YC {
  int j;
  R a[NC1];
};

template <typename R>
__device__ __forceinline__ void contract(const Table &t, const XB<R> &X, int j, YC<R> &o) {
  o.j = j;
  const long cell = (long)j * (t.nx - 1) + X.i;
#pragma unroll
  for (int r = 0; r < NC1; ++r) {
    R q[NC1], d, e;
    cell_row<R>(t, cell, r, q);
    horner5<R, 0>(q, X.u, o.a[r], d, e);
  }
}

// f, f_y, f_yy / 2, f_x, f_xy, f_xx / 2 (in cell units) at (u, v): the rows
// from the highest power of v down, each folded into the synthetic divisions
// in v as it is formed, so no row is kept.
template <typename R> struct TV { R f, fy, fyy, fx, fxy, fxx; };

template <typename R>
__device__ __forceinline__ void cell_eval(const Table &t, int i, int j, R u, R v, TV<R> &o) {
  const long cell = (long)j * (t.nx - 1) + i;
  R h = R(0), d = R(0), e = R(0), bh = R(0), bd = R(0), ch = R(0);
#pragma unroll
  for (int r = NC1 - 1; r >= 0; --r) {
    R q[NC1], a0, a1, a2;
    cell_row<R>(t, cell, r, q);
    horner5<R, 2>(q, u, a0, a1, a2);
    if (r == NC1 - 1) { h = a0; bh = a1; ch = a2; continue; }
    if (r < NC1 - 3) e = fma(e, v, d);
    else if (r == NC1 - 3) e = d;
    if (r < NC1 - 2) { d = fma(d, v, h); bd = fma(bd, v, bh); }
    else { d = h; bd = bh; }
    h = fma(h, v, a0);
    bh = fma(bh, v, a1);
    ch = fma(ch, v, a2);
  }
  o.f = h; o.fy = d; o.fyy = e; o.fx = bh; o.fxy = bd; o.fxx = ch;
}

// Interval index of y and its fraction; false outside the table.
template <typename R>
__device__ __forceinline__ bool yloc(const Table &t, R y, int &j, R &v) {
  const R y0 = sizeof(R) == 8 ? (R)t.y0 : (R)t.y0f, idy = sizeof(R) == 8 ? (R)t.idy : (R)t.idyf;
  return interval((y - y0) * idy, t.ny - 1, j, v);
}

// icv: 1/c_v; er: de/drho at fixed T (the next inversion's first guess,
// eos_invert_rec)
template <typename R> struct EosOut { R P, e, icv, PT, ge, gc, er; };

// Full EOS at (rho, T): P, e, P_T, 1/c_v, de/drho|_T, c_s^2; each quantity
// shared between them formed once.
template <typename R> struct EosC { R P, e, PT, icv, er, cs2, iT; };

template <typename R>
__device__ __forceinline__ bool eos_rt_c(const Table &t, const XB<R> &X, R rho, R irho, R T, R lnT, R iT, R iab,
                                         EosC<R> &o) {
  int j;
  R v;
  if (!(X.ok && yloc<R>(t, lnT, j, v))) return false;
  TV<R> q;
  cell_eval<R>(t, X.i, j, X.u, v, q);
  constexpr bool dbl = sizeof(R) == 8;
  const R idx = dbl ? (R)t.idx : (R)t.idxf, idy = dbl ? (R)t.idy : (R)t.idyf;
  const R idxdy = dbl ? (R)t.idxdy : (R)t.idxdyf;
  const R idx2 = dbl ? (R)t.idx2x2 : (R)t.idx2x2f, idy2 = dbl ? (R)t.idy2x2 : (R)t.idy2x2f;
  const R f = q.f, fy = q.fy * idy, fx = q.fx * idx;
  R aT4, aT3;   // radiation a T^4 and a T^3
  if (dbl) {
    aT3 = (R(ARAD) * T) * (T * T);
    aT4 = aT3 * T;
  } else {   // T^4 overflows FP32 above 2^32 K: form (a^(1/4) T)^4 instead
    const R tt = R(ARAD_QUARTER) * T, t2 = tt * tt;
    aT4 = t2 * t2;
    aT3 = aT4 * iT;
  }
  const R Ra = R(RGAS) * iab, RT = Ra * T;
  const R w = (f - fy) + aT4;                    // rho e without the ions
  o.P = fma(aT4, R(1.0 / 3.0), fma(rho, RT, fx - f));
  o.e = fma(w, irho, R(1.5) * RT);
  // d/drho = (1/rho) d/dx at fixed T
  const R ir2 = irho * irho;
  o.er = (fma(-q.fxy, idxdy, fx) - w) * ir2;
  const R cv = fma(fma(fma(-q.fyy, idy2, fy), iT, R(4) * aT3), irho, R(1.5) * Ra);
  o.icv = rcp_nr(cv);
  o.PT = fma(fma(q.fxy, idxdy, -fy), iT, fma(rho, Ra, R(4.0 / 3.0) * aT3));
  const R Pr = fma(fma(q.fxx, idx2, -fx), irho, RT);
  // c_s^2 = P_rho + T P_T^2 / (rho^2 c_v), grouped so no product leaves the FP32 range
  const R pr = o.PT * irho;
  o.cs2 = fma((T * pr) * o.icv, pr, Pr);
  o.iT = iT;
  return true;
}

// auxiliary indices of Sect. 2.6: gamma_e = P / (rho e) + 1, gamma_c = rho c_s^2 / P
template <typename R>
__device__ __forceinline__ void gammas(R rho, R P, R e, R cs2, R &ge, R &gc) {
  if (sizeof(R) == 8) {   // one reciprocal for both
    const R re = rho * e, inv = rcp_nr(P * re);   // 1/(rho e) = P inv, 1/P = rho e inv
    ge = fma(P, P * inv, R(1));
    gc = rho * cs2 * (re * inv);
  } else {                // P rho e would leave the FP32 range
    ge = P / (rho * e) + R(1);
    gc = rho * cs2 / P;
  }
}

template <typename R>
__device__ __forceinline__ bool eos_rt_xy(const Table &t, const XB<R> &X, R rho, R irho, R T, R lnT, R iT, R iab,
                                          EosOut<R> &o) {
  EosC<R> f;
  if (!eos_rt_c<R>(t, X, rho, irho, T, lnT, iT, iab, f)) return false;
  o.P = f.P; o.e = f.e; o.icv = f.icv; o.PT = f.PT; o.er = f.er;
  gammas<R>(rho, f.P, f.e, f.cs2, o.ge, o.gc);
  return true;
}

template <typename R>
__device__ __forceinline__ bool eos_rt(const Table &t, R rho, R T, R abar, R ye, EosOut<R> &o) {
  return eos_rt_xy<R>(t, xbasis<R>(t, log(rho * ye * R(NAV))), rho, rcp_nr(rho), T, log(T), rcp_nr(T), R(1) / abar, o);
}

// Specific internal energy and c_v at (rho, T): what a Newton iteration needs.
// c holds the x-contraction of the current table interval and is redone when
// T has left it.
template <typename R>
__device__ __forceinline__ bool eos_ecv_xy(const Table &t, const XB<R> &X, YC<R> &c, R irho, R T, R lnT, R iT,
                                           R iab, R &e, R &cv) {
  int j;
  R v;
  if (!(X.ok && yloc<R>(t, lnT, j, v))) return false;
  if (j != c.j) contract<R>(t, X, j, c);
  const R idy = sizeof(R) == 8 ? (R)t.idy : (R)t.idyf, idy2 = sizeof(R) == 8 ? (R)t.idy2x2 : (R)t.idy2x2f;
  R f, a1, a2;
  horner5<R, 2>(c.a, v, f, a1, a2);
  const R fy = a1 * idy;
  R aT4, aT3;
  if (sizeof(R) == 8) {
    aT3 = (R(ARAD) * T) * (T * T);
    aT4 = aT3 * T;
  } else {
    const R tt = R(ARAD_QUARTER) * T, t2 = tt * tt;
    aT4 = t2 * t2;
    aT3 = aT4 * iT;
  }
  const R Ra = R(1.5) * R(RGAS) * iab;
  e = fma((f - fy) + aT4, irho, Ra * T);
  cv = fma(fma(fma(-a2, idy2, fy), iT, R(4) * aT3), irho, Ra);
  return true;
}

// ln Tn from ln T for a Newton step T -> Tn with d = (Tn - T) / T: below
// 2^-10, ln(1 + d) by its Taylor series to d^4 (truncation below d^5 / 5 <
// 2e-16, under the rounding of ln T ~ 16..23); otherwise the logarithm.
// Saves an FP64 logarithm per step once the iteration is close.
template <typename R>
__device__ __forceinline__ R next_lnT(R d, R lnT, R Tn) {
  if (!below_pow2<10>(d)) return log(Tn);
  return lnT + d * (R(1) - d * (R(0.5) - d * (R(1.0 / 3.0) - d * R(0.25))));
}

// Newton inversion e_int -> T (Sect. 2.2): T <- T + (e - e_EoS)/c_v until
// |de|/e < tol, then one more step; bracketed inside the table's T range.
// The iterations evaluate only e and c_v; the full EOS (P, gamma_e, gamma_c)
// is evaluated once, at the final T.  Returns the iteration count or -1.
template <typename R>
__device__ __forceinline__ int newton_loop(const Table &t, const XB<R> &X, YC<R> &c, R rho, R irho, R eint, R iab,
                                           R &T, R tol, int maxit, EosOut<R> &o, bool have, R e0, R cv0, R lnT0) {
  const R Tlo = sizeof(R) == 8 ? (R)t.Tlo : (R)t.Tlof, Thi = sizeof(R) == 8 ? (R)t.Thi : (R)t.Thif;
  R lo = Tlo, hi = Thi;
  if (!between_pos(T, Tlo, Thi)) { T = sqrt(Tlo * Thi); have = false; }
  R lnT = have ? lnT0 : log(T);   // e0, cv0 were evaluated at (T, lnT0), c may hold its interval
  for (int it = 1; it <= maxit; ++it) {
    const R iT = rcp_nr(T);
    R e = e0, cv = cv0;   // the first iteration may come evaluated
    if (!(have && it == 1) && !eos_ecv_xy<R>(t, X, c, irho, T, lnT, iT, iab, e, cv)) return -1;
    const R de = eint - e;
    const R step = de * rcp_nr(cv);
    if (fabs(de) < tol * fabs(eint)) {
      const R Tn = T + step;
      lnT = next_lnT<R>(step * iT, lnT, Tn);
      T = Tn;
      if (!eos_rt_xy<R>(t, X, rho, irho, T, lnT, rcp_nr(T), iab, o)) return -1;
      return it;
    }
    if (de > R(0)) lo = T; else hi = T;
    R Tn = T + step;
    if (!(Tn > lo && Tn < hi)) Tn = R(0.5) * (lo + hi);
    lnT = next_lnT<R>((Tn - T) * iT, lnT, Tn);
    T = Tn;
  }
  return -1;
}

// iab = 1/Abar
template <typename R>
__device__ __forceinline__ int eos_invert(const Table &t, R rho, R irho, R eint, R iab, R ye, R &T, R tol, int maxit,
                                          EosOut<R> &o) {
  const XB<R> X = xbasis<R>(t, log(rho * ye * R(NAV)));   // rho and Y_e fixed
  YC<R> c;
  c.j = -1;
  return newton_loop<R>(t, X, c, rho, irho, eint, iab, T, tol, maxit, o, false, R(0), R(0), R(0));
}

// The FP32 phase of the mixed inversion: Newton on e and c_v only, until
// |de|/e < tol or maxit; T keeps the last bracketed iterate.
__device__ __forceinline__ int newton_fp32(const Table &t, float rho, float eint, float iab, float ye, float &T,
                                           float tol, int maxit) {
  const float Tlo = t.Tlof, Thi = t.Thif;
  float lo = Tlo, hi = Thi;
  if (!(T > Tlo && T < Thi)) T = sqrtf(Tlo * Thi);
  const XB<float> X = xbasis<float>(t, logf(rho * ye * float(NAV)));
  const float irho = 1.0f / rho;
  YC<float> c;
  c.j = -1;
  for (int it = 1; it <= maxit; ++it) {
    float e, cv;
    if (!eos_ecv_xy<float>(t, X, c, irho, T, logf(T), 1.0f / T, iab, e, cv)) return -1;
    const float de = eint - e;
    if (de > 0.0f) lo = T; else hi = T;
    float Tn = T + de / cv;
    if (!(Tn > lo && Tn < hi)) Tn = 0.5f * (lo + hi);
    T = Tn;
    if (fabsf(de) < tol * fabsf(eint)) return it;
  }
  return -1;
}

// Mixed-precision inversion: from a guess farther than 1e-4 from the root,
// FP32 Newton iterations (e and c_v only) bring T within about 1e-5 of it (|de| / e; FP32 holds ln n_e ~ 70 and
// ln T ~ 20 only to ~1e-6, the floor of an FP32 table lookup); FP64 Newton
// then finishes with the FP64 path's stopping rule (|de|/e < tol, one more
// step, the full evaluation at the final T).  The low-Mach deviations need
// P to ~1e-12, so a single FP64 step from 1e-5 is not enough.  Returns the
// total iteration count, or -1 if the FP64 phase fails.
__device__ __forceinline__ int eos_invert_mixed(const Table &t, double rho, double irho, double eint, double iab,
                                                double ye, double &T, double tol, int maxit, EosOut<double> &o) {
  // a first guess already within 1e-4 of the root (the previous step's T in
  // a time step) goes straight to the FP64 iteration: the FP32 phase could
  // only degrade it to FP32's ~1e-6
  const XB<double> X = xbasis<double>(t, log(rho * ye * NAV));
  YC<double> c;
  c.j = -1;
  {
    double e, cv;
    if (T > t.Tlo && T < t.Thi) {
      const double lnT = log(T), iT = rcp_nr(T);
      if (eos_ecv_xy<double>(t, X, c, irho, T, lnT, iT, iab, e, cv) && fabs(eint - e) < 1e-4 * fabs(eint)) {
        const double de = eint - e;
        // From |de|/e < 2e-6 one Newton step lands within ~(de/e)^2 < 1e-11
        // of the root (quadratic convergence; d ln e / d ln T is 1..4 here):
        // the full evaluation at that T1, carried to the root T1 + dT, dT =
        // (e - e(T1)) / c_v(T1), to first order in dT -- P by P_T dT (error
        // ~ dT^2), gamma_e = P / (rho e) + 1 from that P and e; gamma_c keeps
        // its value at T1 (relative error ~ dT / T < 1e-11, wave speeds
        // only).  The plain iteration would evaluate e, c_v at T1 once more
        // and then the full EOS at T1 + dT.
        if (fabs(de) >= tol * fabs(eint) && fabs(de) < 2e-6 * fabs(eint)) {
          const double step = de * rcp_nr(cv), T1 = T + step;
          if (between_pos(T1, t.Tlo, t.Thi)) {
            EosC<double> f;
            if (!eos_rt_c<double>(t, X, rho, irho, T1, next_lnT<double>(step * iT, lnT, T1), rcp_nr(T1), iab, f))
              return -1;
            const double dT = (eint - f.e) * f.icv;
            o.P = fma(f.PT, dT, f.P);
            o.e = eint;
            o.icv = f.icv; o.PT = f.PT; o.er = f.er;
            double ge1;   // gamma_c from the pressure at T1, gamma_e from the carried one
            gammas<double>(rho, f.P, f.e, f.cs2, ge1, o.gc);
            o.ge = o.P * rcp_nr(rho * eint) + 1.0;
            T = T1 + dT;
            return 2;
          }
        }
        return newton_loop<double>(t, X, c, rho, irho, eint, iab, T, tol, maxit, o, true, e, cv, lnT);
      }
    }
  }
  float Tf = (float)T;
  const int it32 = newton_fp32(t, (float)rho, (float)eint, (float)iab, (float)ye, Tf, 1e-5f, maxit < 12 ? maxit : 12);
  if (isfinite(Tf) && Tf > 0.0f) T = (double)Tf;
  const int it64 = newton_loop<double>(t, X, c, rho, irho, eint, iab, T, tol, maxit, o, false, 0.0, 0.0, 0.0);
  return it64 < 0 ? -1 : it64 + (it32 > 0 ? it32 : 12);
}

// The last inversion of a cell, for the next one's first guess: its rho,
// e_int, 1/c_v and de/drho|_T there, ln T and 1/T of the result, and
// x = ln(n_e N_A) and 1/n_e with n_e = rho Y_e.
struct Pred {
  double rho, e, icv, er, lnT, iT, x, ine;
};

// 1/(a (1 + d)) from ia = 1/a: the series 1 - d + d^2 - d^3 + d^4 below
// |d| = 2^-10 (truncation below 2^-50), to d^2 below 2^-18 (truncation below
// 2^-54: the change of a low-Mach stage), else the reciprocal.
__device__ __forceinline__ double inv_step(double ia, double d, double a_new) {
  if (below_pow2<18>(d)) return ia * fma(-d, 1.0 - d, 1.0);
  if (!below_pow2<10>(d)) return rcp_nr(a_new);
  return ia * (1.0 - d * (1.0 - d * (1.0 - d * (1.0 - d))));
}

// ln(a) from ln(a_p) for a = a_p (1 + d): the series of ln(1 + d) to d^4
// below |d| = 2^-10 (as next_lnT), to d^2 below 2^-18 (d^3 / 3 < 2e-17), else
// fall back.
__device__ __forceinline__ double ln_step(double lnp, double d, double fallback_arg) {
  if (below_pow2<18>(d)) return fma(d, fma(d, -0.5, 1.0), lnp);
  if (!below_pow2<10>(d)) return log(fallback_arg);
  return lnp + d * (1.0 - d * (0.5 - d * (1.0 / 3.0 - d * 0.25)));
}

// The carry of a full evaluation c at T1 (within ~2e-6 of the root in e) to
// the root T1 + dT, dT = (e - e(T1)) / c_v, to first order: P + P_T dT;
// gamma_e = P / (rho e) + 1 from that P and e; gamma_c = rho c_s^2 / P
// (c_s^2 at T1: relative error ~dT/T, wave speeds only); one reciprocal for
// both.  |dT|/T < 2e-6, so ln(T1 + dT) takes two terms (the third is below
// 3e-18).  Writes the record of the inversion.
__device__ __forceinline__ void rec_carry(double rho, double eint, double ine, double x, double T1, double lnT1,
                                          const EosC<double> &c, EosOut<double> &o, double &T, Pred &pr) {
  const double dT = (eint - c.e) * c.icv;
  o.P = fma(c.PT, dT, c.P);
  o.e = eint;
  gammas<double>(rho, o.P, eint, c.cs2, o.ge, o.gc);
  o.icv = c.icv;
  o.PT = c.PT;
  o.er = c.er;
  T = T1 + dT;
  const double dd = dT * c.iT;
  pr = Pred{rho, eint, c.icv, c.er, fma(dd, fma(dd, -0.5, 1.0), lnT1), c.iT * (1.0 - dd), x, ine};
}

// Mixed-precision inversion with a per-cell record (rec: the record holds
// the cell's previous inversion).  With a record, the first-order guess
//   T1 = T + (e - e_p - (de/drho)_T (rho - rho_p)) / c_v
// lies within ~(relative change since then)^2 of the root: one full
// evaluation there and, where |e - e(T1)| / e < 2e-6, its carry to the root
// (rec_carry); ln(n_e N_A) and ln T1 follow from the record's by the series
// of ln(1 + d).  Without a record (or where the change was larger) the
// mixed inversion's own steps: e, c_v at T; from within 2e-6 one Newton
// step, the full evaluation and the carry; from within 1e-4 the FP64 Newton
// loop; else FP32 iterations first.  irho = 1/rho and iab = 1/Abar come
// with the arguments.  Writes the record; returns the count of evaluations
// at distinct temperatures (1 for the recorded path) or -1.
__device__ __forceinline__ int eos_invert_rec(const Table &t, double rho, double irho, double eint, double iab,
                                              double ye, double &T, double tol, int maxit, EosOut<double> &o, Pred &pr,
                                              bool rec) {
  const double ne = rho * ye;
  rec = rec && positive(pr.ine);
  const double dn = rec ? fma(ne, pr.ine, -1.0) : 0.0;   // n_e = n_e,p (1 + dn)
  const double x = rec ? ln_step(pr.x, dn, ne * NAV) : log(ne * NAV);
  const double ine = rec ? inv_step(pr.ine, dn, ne) : rcp_nr(ne);
  const XB<double> X = xbasis<double>(t, x);
  EosC<double> f;
  if (rec && positive(pr.icv) && between_pos(T, t.Tlo, t.Thi)) {
    const double T1 = T + (eint - pr.e - pr.er * (rho - pr.rho)) * pr.icv;
    if (between_pos(T1, t.Tlo, t.Thi)) {
      const double dT = (T1 - T) * pr.iT;   // T1 = T (1 + dT)
      const double lnT1 = ln_step(pr.lnT, dT, T1);
      if (!eos_rt_c<double>(t, X, rho, irho, T1, lnT1, inv_step(pr.iT, dT, T1), iab, f)) return -1;
      if (fabs(eint - f.e) < 2e-6 * fabs(eint)) {
        rec_carry(rho, eint, ine, x, T1, lnT1, f, o, T, pr);
        return 1;
      }
      T = T1;   // a larger change: the steps below from T1
    }
  }
  YC<double> c;
  c.j = -1;
  int it0 = -2;   // -2: a far guess, FP32 iterations first
  if (T > t.Tlo && T < t.Thi) {
    const double lnT = log(T), iT = rcp_nr(T);
    double e, cv;
    if (eos_ecv_xy<double>(t, X, c, irho, T, lnT, iT, iab, e, cv) && fabs(eint - e) < 1e-4 * fabs(eint)) {
      const double de = eint - e;
      if (fabs(de) < 2e-6 * fabs(eint)) {
        const double step = de * rcp_nr(cv), T1 = T + step;
        if (between_pos(T1, t.Tlo, t.Thi)) {
          const double lnT1 = next_lnT<double>(step * iT, lnT, T1);
          if (!eos_rt_c<double>(t, X, rho, irho, T1, lnT1, rcp_nr(T1), iab, f)) return -1;
          rec_carry(rho, eint, ine, x, T1, lnT1, f, o, T, pr);
          return 2;
        }
      }
      it0 = newton_loop<double>(t, X, c, rho, irho, eint, iab, T, tol, maxit, o, true, e, cv, lnT);
    }
  }
  if (it0 == -2) {
    float Tf = (float)T;
    const int it32 = newton_fp32(t, (float)rho, (float)eint, (float)iab, (float)ye, Tf, 1e-5f, maxit < 12 ? maxit : 12);
    if (isfinite(Tf) && Tf > 0.0f) T = (double)Tf;
    const int it64 = newton_loop<double>(t, X, c, rho, irho, eint, iab, T, tol, maxit, o, false, 0.0, 0.0, 0.0);
    it0 = it64 < 0 ? -1 : it64 + (it32 > 0 ? it32 : 12);
  }
  if (it0 > 0)   // the record of a Newton-loop result (the rare paths)
    pr = Pred{rho, eint, o.icv, o.er, log(T), rcp_nr(T), x, ine};
  return it0;
}

}  // namespace eos
}  // namespace phl

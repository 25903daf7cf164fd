// riemann_fp64.cuh -- the face flux of riemann.cuh in FP64, laid out for the
// fewest FP64 instructions (that pipe, 1/64 of the FP32 rate, bounds every
// FP64 form).  Same method and deviation form; what differs is which of the
// equal expressions for the flux inside the fan is evaluated (below), the
// reciprocals and roots (fp64_math.cuh) and that one-sided quantities are
// formed only for the side the flux is taken from.  Together with the walks of
// k_flux_walk: 1.70 -> 0.95 ms per direction on 128 x 96 x 112 cells.
// The FP32 solvers keep the difference form: where the flow is tangential a
// face's mass flux sits at rounding level, its sign picks Contact-CT's upwind
// side, and another rounding of the FP32 fluxes moves the field there by up to
// 1e-7 of its scale against earlier runs of the same state.
#pragma once
#include "fp64_math.cuh"
#include "riemann.cuh"

namespace phl {

// What both sides of a face need for the wave speeds and the intermediate
// states; the rest (enthalpy, u.B, the physical flux) is formed only for the
// side the flux is taken from.
struct SideD {
  double rho, un, ut1, ut2, bt1, bt2, p, ge;  // full rho, P, gamma_e
  double b2, u2;
  double dpt;    // p_T - P_hat
  double cf;
  double m2;     // |u|^2 / c_s^2
};

template <bool IDEAL>
__device__ __forceinline__ void side_init_d(SideD &s, const double *w, double bn, double rh, double ph, double geh, double gch, const GasK<double> &K) {
  s.rho = rh + w[RD_RHO];
  s.un = w[RD_UN]; s.ut1 = w[RD_UT1]; s.ut2 = w[RD_UT2];
  s.bt1 = w[RD_BT1]; s.bt2 = w[RD_BT2];
  const double dp = w[RD_P];
  s.p = ph + dp;
  const double irho = rcp_nr(s.rho);
  s.b2 = bn * bn + s.bt1 * s.bt1 + s.bt2 * s.bt2;
  s.u2 = s.un * s.un + s.ut1 * s.ut1 + s.ut2 * s.ut2;
  const double half = 0.5;
  s.dpt = dp + half * s.b2;
  s.ge = IDEAL ? K.g : geh + w[RD_GE];
  const double gc = IDEAL ? K.g : gch + w[RD_GC];
  const double a2 = gc * s.p * irho;
  const double bb = s.b2 * irho, bnn = bn * bn * irho;
  double disc = (a2 + bb) * (a2 + bb) - 4.0 * a2 * bnn;
  disc = not_below_zero(disc);
  s.cf = sqrt_nr(half * (a2 + bb + sqrt_nr(disc)));
  s.m2 = div_nr(s.u2, a2);
}

// E + p_T (full), u . B and the physical flux minus the background flux of a side.
struct SideFluxD { double enth, vb, F[7]; };
template <bool IDEAL>
__device__ __forceinline__ void side_flux(SideFluxD &o, const SideD &s, double bn, const GasK<double> &K) {
  const double kin = 0.5 * s.rho * s.u2;
  if (IDEAL) o.enth = K.ggm1 * s.p + kin + s.b2;
  else o.enth = div_nr(s.ge, s.ge - 1.0) * s.p + kin + s.b2;
  o.vb = s.un * bn + s.ut1 * s.bt1 + s.ut2 * s.bt2;
  o.F[RF_RHO] = s.rho * s.un;
  o.F[RF_MN] = s.rho * s.un * s.un + s.dpt - bn * bn;
  o.F[RF_MT1] = s.rho * s.un * s.ut1 - bn * s.bt1;
  o.F[RF_MT2] = s.rho * s.un * s.ut2 - bn * s.bt2;
  o.F[RF_E] = o.enth * s.un - bn * o.vb;
  o.F[RF_BT1] = s.un * s.bt1 - s.ut1 * bn;
  o.F[RF_BT2] = s.un * s.bt2 - s.ut2 * bn;
}

// E - E_hat of a side (the HLL flux's jump).
template <bool IDEAL>
__device__ __forceinline__ double side_de(const SideD &s, const double *w, double ph, double geh, const GasK<double> &K) {
  const double kin = 0.5 * s.rho * s.u2, dp = w[RD_P];
  // internal energy density P / (gamma_e - 1) relative to P_hat / (gamma_hat_e - 1)
  if (IDEAL) return dp * K.igm1 + kin + 0.5 * s.b2;
  const double gem1 = s.ge - 1.0;
  double deint;
  if (ph == 0.0) {
    deint = div_nr(s.p, gem1);
  } else {
    const double gehm1 = geh - 1.0;
    deint = div_nr(dp * gehm1 - ph * w[RD_GE], gem1 * gehm1);
  }
  return deint + kin + 0.5 * s.b2;
}

// One side's HLLD intermediate state: density, transverse velocity and field;
// 1/(S - S_M) and S_M - u for its energy.
struct StarD { double iq, smu, rhos, v1, v2, b1, b2; };
__device__ __forceinline__ void star_state(const SideD &s, double S, double SM, double bn, StarD &o) {
  const double su = S - s.un;           // S - u   (nonzero)
  const double q = S - SM;              // S - S_M (nonzero)
  const double rs = s.rho * su;
  o.iq = rcp_nr(q);
  o.smu = SM - s.un;
  o.rhos = rs * o.iq;
  const double den = rs * q - bn * bn;
  const double scale = rs * su + bn * bn;
  // degenerate case (den ~ 0): the transverse values stay those of the side;
  // selected rather than branched so that a warp's faces take one path
  const bool deg = fabs(den) < 1e-12 * scale;
  const double si = deg ? 0.0 : o.smu * rcp_nr(den);
  const double fv = bn * si, dbf = rs * si;   // (B*_t - B_t) / B_t
  o.v1 = s.ut1 - s.bt1 * fv;
  o.v2 = s.ut2 - s.bt2 * fv;
  o.b1 = s.bt1 + s.bt1 * dbf;
  o.b2 = s.bt2 + s.bt2 * dbf;
}

// sqrt(x) and a / sqrt(x)
__device__ __forceinline__ void root_and_quotient(double x, double a, double &s, double &q) {
  double r;
  sqrt_rsqrt_nr(x, s, r);
  q = a * r;
}
template <int NS, bool IDEAL>
__device__ __forceinline__ void riemann_fp64(const double *wl, const double *wr, double bn, double rh, double ph, double geh, double gch, int nspec,
                                            int solver, double mthr, double *f, int &up, const GasK<double> &K) {
  SideD L, R_;
  side_init_d<IDEAL>(L, wl, bn, rh, ph, geh, gch, K);
  side_init_d<IDEAL>(R_, wr, bn, rh, ph, geh, gch, K);
  const double SL = fmin(L.un - L.cf, R_.un - R_.cf);
  const double SR = fmax(L.un + L.cf, R_.un + R_.cf);
  double xl[NS > 0 ? NS : 1], xr[NS > 0 ? NS : 1];
  {
    double sl = 0.0, sr = 0.0;
#pragma unroll
    for (int l = 0; l < NS; ++l)
      if (l < nspec) { sl += wl[RD_X0 + l]; sr += wr[RD_X0 + l]; }
#pragma unroll
    for (int l = 0; l < NS; ++l)
      if (l < nspec) { xl[l] = div_nr(wl[RD_X0 + l], sl); xr[l] = div_nr(wr[RD_X0 + l], sr); }
  }

  if (solver == SOLVER_HLL) {
    SideFluxD fl, fr;
    side_flux<IDEAL>(fl, L, bn, K);
    side_flux<IDEAL>(fr, R_, bn, K);
    if (SL >= 0.0) {
      for (int q = 0; q < 7; ++q) f[q] = fl.F[q];
#pragma unroll
      for (int l = 0; l < NS; ++l)
        if (l < nspec) f[RF_X0 + l] = fl.F[RF_RHO] * xl[l];
    } else if (SR <= 0.0) {
      for (int q = 0; q < 7; ++q) f[q] = fr.F[q];
#pragma unroll
      for (int l = 0; l < NS; ++l)
        if (l < nspec) f[RF_X0 + l] = fr.F[RF_RHO] * xr[l];
    } else {
      double dU[7];
      dU[RF_RHO] = wr[RD_RHO] - wl[RD_RHO];
      dU[RF_MN] = R_.rho * R_.un - L.rho * L.un;
      dU[RF_MT1] = R_.rho * R_.ut1 - L.rho * L.ut1;
      dU[RF_MT2] = R_.rho * R_.ut2 - L.rho * L.ut2;
      dU[RF_E] = side_de<IDEAL>(R_, wr, ph, geh, K) - side_de<IDEAL>(L, wl, ph, geh, K);
      dU[RF_BT1] = R_.bt1 - L.bt1;
      dU[RF_BT2] = R_.bt2 - L.bt2;
      const double idn = rcp_nr(SR - SL);
      for (int q = 0; q < 7; ++q) f[q] = (SR * fl.F[q] - SL * fr.F[q] + SL * SR * dU[q]) * idn;
#pragma unroll
      for (int l = 0; l < NS; ++l)
        if (l < nspec)
          f[RF_X0 + l] = (SR * fl.F[RF_RHO] * xl[l] - SL * fr.F[RF_RHO] * xr[l] +
                          SL * SR * (R_.rho * xr[l] - L.rho * xl[l])) * idn;
    }
    up = contact_dir(f[RF_RHO], L.rho, R_.rho, SL, SR);
    return;
  }

  if (SL >= 0.0 || SR < 0.0) {   // supersonic: the physical flux of the upwind side
    const bool left = SL >= 0.0;
    SideFluxD fx;
    side_flux<IDEAL>(fx, left ? L : R_, bn, K);
    for (int q = 0; q < 7; ++q) f[q] = fx.F[q];
#pragma unroll
    for (int l = 0; l < NS; ++l)
      if (l < nspec) f[RF_X0 + l] = fx.F[RF_RHO] * (left ? xl[l] : xr[l]);
    up = contact_dir(f[RF_RHO], L.rho, R_.rho, SL, SR);
    return;
  }
  double xi = 1.0;
  if (solver == SOLVER_LHLLD) {   // xi = max(M_L, M_R) below the threshold, M = |u| / c_s
    const double m2 = L.m2 > R_.m2 ? L.m2 : R_.m2;
    xi = m2 < mthr * mthr ? sqrt_nr(m2) : 1.0;
  }
  const double sR = SR - R_.un, sL = SL - L.un;
  const double rsR = sR * R_.rho, rsL = sL * L.rho;
  const double iD = rcp_nr(rsR - rsL);
  const double SM = (rsR * R_.un - rsL * L.un - R_.dpt + L.dpt) * iD;
  const double pdis = rsR * rsL * ((R_.un - L.un) * iD);
  const double dpts = (rsR * L.dpt - rsL * R_.dpt) * iD + pdis;   // p_T* - P_hat

  // Inside the fan the face sits in one of the intermediate states of the side
  // X of the contact: the single star (S*_L >= 0 or S*_R < 0) or the double
  // star.  Both move with S_M and carry rho*, p_T*, so with (v, b) the state's
  // transverse velocity and field the flux is that state's own,
  //   F_rho = rho* S_M,  F_mn = F_rho S_M + p_T* - B_n^2,
  //   F_mt = F_rho v - B_n b,  F_bt = b S_M - B_n v,
  //   F_E = (E* + p_T*) S_M - B_n (u.B),
  // which the jump conditions make equal to F_X + S_X (U* - U_X) (+ S*_X (U** -
  // U*)).  It needs neither the side's flux nor the differences (about 60
  // operations fewer), and no term of it is larger than the flux itself,
  // where S_X (U* - U_X) subtracts products of the sound speed.
  StarD sL_, sR_;
  star_state(L, SL, SM, bn, sL_);
  star_state(R_, SR, SM, bn, sR_);
  const double abn = fabs(bn);
  double sqL, sqR, aL, aR;
  root_and_quotient(sL_.rhos, abn, sqL, aL);
  root_and_quotient(sR_.rhos, abn, sqR, aR);
  const bool starL = SM - aL >= 0.0, starR = !starL && SM + aR < 0.0, dbl = !starL && !starR;
  const bool left = starL || (!starR && SM >= 0.0);
  const double sgn = bn >= 0.0 ? 1.0 : -1.0;
  const double isum = rcp_nr(sqL + sqR);
  const double vss1 = (sqL * sL_.v1 + sqR * sR_.v1 + (sR_.b1 - sL_.b1) * sgn) * isum;
  const double vss2 = (sqL * sL_.v2 + sqR * sR_.v2 + (sR_.b2 - sL_.b2) * sgn) * isum;
  const double sqs2 = sqL * sqR * sgn;
  const double bss1 = (sqL * sR_.b1 + sqR * sL_.b1 + sqs2 * (sR_.v1 - sL_.v1)) * isum;
  const double bss2 = (sqL * sR_.b2 + sqR * sL_.b2 + sqs2 * (sR_.v2 - sL_.v2)) * isum;
  // X's quantities, selected so that the faces of a warp follow one path
  auto pick = [&](double a, double b) { return left ? a : b; };
  const double un = pick(L.un, R_.un), p = pick(L.p, R_.p), b2X = pick(L.b2, R_.b2), dptX = pick(L.dpt, R_.dpt);
  const double kin = 0.5 * pick(L.rho, R_.rho) * pick(L.u2, R_.u2);
  double enth;   // E + p_T
  if (IDEAL) {
    enth = K.ggm1 * p + kin + b2X;
  } else {
    const double ge = pick(L.ge, R_.ge);
    enth = div_nr(ge, ge - 1.0) * p + kin + b2X;
  }
  const double vb = un * bn + pick(L.ut1, R_.ut1) * pick(L.bt1, R_.bt1) + pick(L.ut2, R_.ut2) * pick(L.bt2, R_.bt2);
  const double iq = pick(sL_.iq, sR_.iq), smu = pick(sL_.smu, sR_.smu), rhos = pick(sL_.rhos, sR_.rhos);
  const double v1s = pick(sL_.v1, sR_.v1), v2s = pick(sL_.v2, sR_.v2), b1s = pick(sL_.b1, sR_.b1), b2s = pick(sL_.b2, sR_.b2);
  const double v1 = dbl ? vss1 : v1s, v2 = dbl ? vss2 : v2s, b1 = dbl ? bss1 : b1s, b2 = dbl ? bss2 : b2s;
  const double vbs = SM * bn + v1s * b1s + v2s * b2s;
  const double vbx = SM * bn + v1 * b1 + v2 * b2;
  // E* - E, then (double star) E** - E* = -+ sqrt(rho*) ((u.B)* - (u.B)**) sgn(B_n)
  const double dpt = dpts - dptX;
  const double dE = (smu * enth + dpt * SM + bn * (vb - vbs)) * iq;
  const double sqs = pick(-sqL, sqR) * sgn;
  // LHLLD: the dissipative part of p_T* is scaled by xi in the flux (the
  // states stay those of HLLD)
  const double corr = (xi != 1.0 && SR > 0.0) ? (xi - 1.0) * pdis : 0.0;
  const double hstar = enth + dE + (dbl ? sqs * (vbs - vbx) : 0.0) + (dpt + corr);
  f[RF_RHO] = rhos * SM;
  f[RF_MN] = f[RF_RHO] * SM + (dpts + corr - bn * bn);
  f[RF_MT1] = f[RF_RHO] * v1 - bn * b1;
  f[RF_MT2] = f[RF_RHO] * v2 - bn * b2;
  f[RF_E] = hstar * SM - bn * vbx;
  f[RF_BT1] = b1 * SM - bn * v1;
  f[RF_BT2] = b2 * SM - bn * v2;
#pragma unroll
  for (int l = 0; l < NS; ++l)
    if (l < nspec) f[RF_X0 + l] = f[RF_RHO] * (left ? xl[l] : xr[l]);
  up = contact_dir(f[RF_RHO], L.rho, R_.rho, SL, SR);
}

}  // namespace phl

// Device thermochemistry of one cell over one subcycle (Sec. 2.3.1, 4.1.1).
//
// State and update arithmetic are FP64 in both precision modes.  With
// FastRates the temperature-dependent rate coefficients (fits with exp/pow)
// are evaluated in FP32 with hardware intrinsics, as Sec. 6.2 proposes for
// the chemistry solver; the rate fits themselves carry percent-level
// uncertainty, far above FP32 rounding.
#pragma once
#include "rt_common.cuh"

namespace m1rt {

struct ChemParams {
  int B;
  int mode;          // 1 isothermal, 2 thermal energy evolves
  int flags;         // bit0 recombination, bit1 collisional ionisation, bit2 cooling, bit3 photoheating
  double c_red;
  double y_he;
  double f_s, f_max, x_floor;
  int max_sub;
  double sigma[kMaxBins][3];
  double eps[kMaxBins][3];
  int smask;         // bit 3b+s: sigma[b][s] != 0
  int emask;         // bit 3b+s: eps[b][s] != 0
  float heat_f[kMaxBins][3];   // mixed precision: eps sigma / kHeatScale in FP32
  // for the first attempts, whose length dt is the same for every cell:
  // c_red dt, c_red dt sigma, and the scaled factors of the heat and cooling
  double cdt, csig[kMaxBins][3];
  float cdt_heat, dt_cool;
};

// Scale of the FP32 photoheating products: eps sigma (~1e-29 erg cm^2) is
// carried as eps sigma / kHeatScale so that eps sigma n_s Nbar stays in the
// FP32 normal range.
constexpr double kHeatScale = 1e-30;

constexpr double kBoltzmann = 1.380649e-16;

// Rate coefficients at temperature T (cm^3/s), cooling (erg cm^-3 s^-1).
// Case-B recombination of HII and HeIII: Hui & Gnedin (1997); HeII case B
// plus dielectronic; collisional ionisation and cooling: Katz, Weinberg &
// Hernquist (1996).
struct Rates {
  double aHII, aHeII, aHeIII, bHI, bHeI, bHeII;
};

template <bool Fast> struct RateEval;

// Functions of T shared by the FP64 rate fits and the cooling rate: every
// power of T from one logarithm or from sqrt(T) and 1 / T, the Boltzmann
// factors that both use formed once (relative error ~1e-15 against the pow /
// exp of the definitions).
struct TFns {
  double T, iT, sT, tf, lnT, e94, e470, e157, e285, e631, T15, u407;   // T^-3/2, T^-0.407
};

// natural logarithms of the fits' scale constants, and 1 / ln 10
constexpr double kLnAH = 11.654317306519307;    // ln(2 x 157807 / 2.740)
constexpr double kLnAHe2 = 13.041066233619674;  // ln(2 x 631515 / 2.740)
constexpr double kLnLHe = 13.254566388120152;   // ln(2 x 285335)
constexpr double kLn1e3 = 6.907755278982137;
constexpr double kLn1e6 = 13.815510557964274;
constexpr double kInvLn10 = 0.43429448190325176;

__device__ __forceinline__ TFns tfns(double T) {
  TFns t;
  t.T = T;
  t.iT = rcp_nr<2>(T);
  t.sT = sqrt_nr(T);
  t.tf = rcp_nr<2>(fma(t.sT, 0.0031622776601683794, 1.0));   // 1 / (1 + sqrt(T / 1e5))
  t.lnT = log_series(T);
  t.e94 = exp(-94000.0 * t.iT);
  const double e2 = t.e94 * t.e94;
  t.e470 = e2 * e2 * t.e94;                                   // exp(-470000 / T)
  t.e157 = exp(-157809.1 * t.iT);
  t.e285 = exp(-285335.4 * t.iT);
  t.e631 = exp(-631515.0 * t.iT);
  t.T15 = t.iT * t.iT * t.sT;
  t.u407 = exp(-0.407 * t.lnT);
  return t;
}

// Constants of the fits' powers: 315614^1.5, 1263030^1.5 (lambda = 2 T_i / T of
// HII and HeIII), (315614 / 2.740)^0.407, (1263030 / 2.740)^0.407, 570670^0.75.
constexpr double kLam15H = 315614.0 * 561.7953363992976, kLam15He2 = 1263030.0 * 1123.8460748696862;
constexpr double kU407H = 114.81327852071512, kU407He2 = 201.88817541951113, kLam075He = 20762.93678880667;

template <> struct RateEval<false> {
  __device__ static Rates eval(const TFns& t) {
    Rates r;
    // Hui & Gnedin case B, lambda = 2 T_i / T: a lambda^1.5 / (1 + (lambda / 2.74)^0.407)^2.242
    r.aHII = (2.753e-14 * kLam15H) * t.T15 * exp(-2.242 * log_series(fma(kU407H, t.u407, 1.0)));
    r.aHeIII = (2.0 * 2.753e-14 * kLam15He2) * t.T15 * exp(-2.242 * log_series(fma(kU407He2, t.u407, 1.0)));
    const double die = 1.9e-3 * t.T15 * t.e470 * fma(0.3, t.e94, 1.0);
    const double rs = t.iT * t.sT;   // T^-1/2
    r.aHeII = fma(1.26e-14 * kLam075He, rs * sqrt_nr(rs), die);
    const double st = t.sT * t.tf;
    r.bHI = 5.85e-11 * st * t.e157;
    r.bHeI = 2.38e-11 * st * t.e285;
    r.bHeII = 5.68e-12 * st * t.e631;
    return r;
  }
  __device__ static Rates eval(double T) { return eval(tfns(T)); }
  // from the species' densities, grouped by species
  __device__ static double cooling(const TFns& t, double ne, double nHI, double nHII, double nHeI, double nHeII,
                                   double nHeIII) {
    const double st = t.sT * t.tf;
    const double kHI = fma(7.50e-19 * t.tf, exp(-118348.0 * t.iT), 1.27e-21 * st * t.e157);
    const double kHeI = 9.38e-22 * st * t.e285;
    const double t3 = t.sT * div_nr(exp(-0.2 * (t.lnT - kLn1e3)), 1.0 + exp(0.7 * (t.lnT - kLn1e6)));
    const double d = 5.5 - t.lnT * kInvLn10;
    const double br = 1.42e-27 * fma(0.34, exp(d * d * (-1.0 / 3.0)), 1.1) * t.sT;
    const double kHeII = fma(5.54e-17 * t.tf, exp(fma(-473638.0, t.iT, -0.397 * t.lnT)), 4.95e-22 * st * t.e631) +
                         fma(1.55e-26, exp(0.3647 * t.lnT), 1.24e-13 * t.T15 * t.e470 * fma(0.3, t.e94, 1.0));
    return ne * (kHI * nHI + kHeI * nHeI + (kHeII + br) * nHeII + fma(8.70e-27, t3, br) * nHII +
                 fma(3.48e-26, t3, 4.0 * br) * nHeIII);
  }
};

// FP32 intrinsics: x^p = 2^(p log2 x), e^x = 2^(x log2 e).
__device__ __forceinline__ float fpow(float x, float p) { return exp2f(p * __log2f(x)); }
__device__ __forceinline__ float fexp(float x) { return exp2f(x * 1.4426950408889634f); }

struct RatesF {
  float aHII, aHeII, aHeIII, bHI, bHeI, bHeII;
};

// Precision conversions of the mixed chemistry.  IntCvt: assembled on the
// integer pipe (d2f_int, f2d_int), for the first pass over every cell, where
// the FP64 pipe bounds the kernel; otherwise the hardware's conversions, for
// the worklist pass by threads, where a few stiff cells run long serial chains
// of attempts and an attempt's latency counts: one instruction instead of ten.
// The two round alike (to nearest) but for exact ties and subnormal values.
template <bool IntCvt> __device__ __forceinline__ float to_f(double x) {
  if constexpr (IntCvt) return d2f_int(x);
  else return __double2float_rn(x);
}
template <bool IntCvt> __device__ __forceinline__ double to_d(float x) {
  if constexpr (IntCvt) return f2d_int(x);
  else return (double)x;
}

template <> struct RateEval<true> {
  // the rate fits in FP32
  template <bool IntCvt = true>
  __device__ static RatesF eval_f(double Td) {
    const float T = to_f<IntCvt>(Td);
    const float iT = __frcp_rn(T);
    RatesF r;
    const float lH = 315614.0f * iT;
    r.aHII = 2.753e-14f * fpow(lH, 1.5f) / fpow(1.0f + fpow(lH * (1.0f / 2.740f), 0.407f), 2.242f);
    const float lHe = 570670.0f * iT;
    r.aHeII = 1.26e-14f * fpow(lHe, 0.750f) +
              1.9e-3f * fpow(T, -1.5f) * fexp(-470000.0f * iT) * (1.0f + 0.3f * fexp(-94000.0f * iT));
    const float lHe2 = 1263030.0f * iT;
    r.aHeIII = 2.0f * 2.753e-14f * fpow(lHe2, 1.5f) / fpow(1.0f + fpow(lHe2 * (1.0f / 2.740f), 0.407f), 2.242f);
    const float sT = sqrtf(T);
    const float tf = 1.0f / (1.0f + sqrtf(T * 1e-5f));
    r.bHI = 5.85e-11f * sT * fexp(-157809.1f * iT) * tf;
    r.bHeI = 2.38e-11f * sT * fexp(-285335.4f * iT) * tf;
    r.bHeII = 5.68e-12f * sT * fexp(-631515.0f * iT) * tf;
    return r;
  }
  // The same cooling rate divided by kCoolScale, entirely in FP32 from the
  // FP32 images of the densities (the coefficients, ~1e-27..1e-19, times
  // 1/kCoolScale lie in the FP32 normal range together with the densities'
  // products); it only enters the energy increment.
  template <bool IntCvt = true>
  __device__ static float cooling_scaled(double Td, float ne, float nHI, float nHII, float nHeI, float nHeII,
                                         float nHeIII) {
    const float T = to_f<IntCvt>(Td), iT = __frcp_rn(T);
    const float sT = sqrtf(T), tf = 1.0f / (1.0f + sqrtf(T * 1e-5f));
    const float ex1 = fexp(-157809.1f * iT), ex2 = fexp(-285335.4f * iT), ex3 = fexp(-631515.0f * iT);
    // coefficients of the KWH96 fits times 1/kCoolScale = 1e27
    const float kHI = (7.50e8f * fexp(-118348.0f * iT) + 1.27e6f * sT * ex1) * tf;
    const float t3 = fpow(T * 1e-3f, -0.2f) / (1.0f + fpow(T * 1e-6f, 0.7f));
    const float lg = __log10f(T);
    const float br = 1.42f * (1.1f + 0.34f * fexp(-(5.5f - lg) * (5.5f - lg) * (1.0f / 3.0f))) * sT;
    const float kHII = 8.70f * sT * t3;
    const float kHeI = 9.38e5f * sT * ex2 * tf;
    const float kHeII = (5.54e10f * fpow(T, -0.397f) * fexp(-473638.0f * iT) + 4.95e5f * sT * ex3) * tf +
                        15.5f * fpow(T, 0.3647f) +
                        1.24e14f * fpow(T, -1.5f) * fexp(-470000.0f * iT) * (1.0f + 0.3f * fexp(-94000.0f * iT));
    const float kHeIII = 34.8f * sT * t3;
    return ne * (kHI * nHI + (kHII + br) * nHII + kHeI * nHeI + (kHeII + br) * nHeII + (kHeIII + 4.0f * br) * nHeIII);
  }
};

// Scale of the FP32 cooling rate (see RateEval<true>::cooling_scaled).
constexpr double kCoolScale = 1e-27;

// Per-cell state of the photochemistry step.
struct CellState {
  double N[kMaxBins];
  double f[kMaxBins][3];   // reduced flux F / c_red
  double xHI, xHII, yI, yII, yIII, T;
};

__device__ __forceinline__ double rel_change(double a, double b, double fl) {
  double m = fabs(a) > fl ? fabs(a) : fl;
  return div_nr(fabs(b - a), m);
}

// The largest of n relative changes |b - a| / max(|a|, floor).  Each is formed
// in FP32 first (relative error below 1e-6: differences in FP64, cut to FP32,
// one quotient); a leader that is 4e-6 ahead of all others is the largest, and
// only its quotient is formed in FP64.  Otherwise (and with values outside
// the FP32 range or not finite) all of them are.
template <int n>
__device__ __forceinline__ double largest_change(const double a[n], const double b[n], const double fl[n], int use) {
  float m1 = 0.0f, m2 = 0.0f;
  double num = 0.0, den = 1.0;
  bool ok = true;
#pragma unroll
  for (int q = 0; q < n; ++q) {
    if (q >= use) continue;
    const double d = fabs(b[q] - a[q]);
    const double m = __double_as_longlong(fabs(a[q])) > __double_as_longlong(fl[q]) ? fabs(a[q]) : fl[q];
    const float df = d2f_int(d), mf = d2f_int(m);
    const float r = __fdividef(df, mf);
    ok = ok && mf > 1e-36f && r < 1e30f && (df > 0.0f || __double_as_longlong(d) == 0);
    if (r > m1) { num = d; den = m; }
    m2 = fmaxf(m2, fminf(m1, r));
    m1 = fmaxf(m1, r);
  }
  if (ok && m1 > 1e-30f && m1 - m2 > 4e-6f * m1) return div_nr(num, den);
  double f = 0.0;
#pragma unroll
  for (int q = 0; q < n; ++q)
    if (q < use) f = fmax(f, rel_change(a[q], b[q], fl[q]));
  return f;
}

// x, and 0 where it is negative (NaN stays), on the integer pipe (from the high
// word: a test on all the bits is compiled into an FP64 comparison).
__device__ __forceinline__ double clamp_neg(double x) {
  const unsigned h = (unsigned)__double2hiint(x) ^ 0x80000000u;   // of -x
  return h <= 0x7FF00000u ? 0.0 : x;
}

// |x| on the integer pipe.
__device__ __forceinline__ double no_sign(double x) {
  return __hiloint2double(__double2hiint(x) & 0x7FFFFFFF, __double2loint(x));
}

// x <= 0 (not NaN), on the integer pipe.  A bin that enters the attempts of the
// mixed path so leaves the first accepted one with N = 0 and without flux, and
// stays there; the others never come to N < 0.
__device__ __forceinline__ bool unlit(double x) {
  const unsigned h = (unsigned)__double2hiint(x);
  return (h ^ 0x80000000u) <= 0x7FF00000u || (h | (unsigned)__double2loint(x)) == 0u;
}

// One semi-implicit photochemistry attempt over dt from s into t; returns the
// largest relative change f of the substep rule.  Steps: radiation level
// over the step (implicit in N, absorbers at the start); photoionisation
// rates from it; backward Euler for H, then for He with the updated n_e;
// photons removed = photoionisations credited (absorbers at the end), F scaled
// alike; thermal energy explicit.  Arranged for the FP64 unit, which bounds it:
// one reciprocal per denominator, the photons' factor 1 - (c dt sum sigma n') /
// (1 + c dt sum sigma n) instead of a quotient by N, thirteen exponentials, one
// quotient for the measure.
__device__ double photochem_attempt(const ChemParams& P, double nH, double dt, const CellState& s, CellState& t) {
  const int B = P.B;
  const double cdt = P.c_red * dt;
  const double nHe = P.y_he * nH;
  const bool recomb = P.flags & 1, coll = P.flags & 2, cool = P.flags & 4, heat = P.flags & 8;
  const TFns tfn = tfns(s.T);
  const Rates r = RateEval<false>::eval(tfn);

  const double ns[3] = {nH * s.xHI, nHe * s.yI, nHe * s.yII};
  double inv[kMaxBins], Nbar[kMaxBins];
  double G[3] = {0.0, 0.0, 0.0};
#pragma unroll
  for (int b = 0; b < kMaxBins; ++b) {
    if (b < B) {
      double kap = 0.0;
#pragma unroll
      for (int q = 0; q < 3; ++q)
        if (P.smask & (1 << (3 * b + q))) kap = fma(P.sigma[b][q], ns[q], kap);
      inv[b] = rcp_nr<2>(fma(cdt, kap, 1.0));
      Nbar[b] = cdt * (s.N[b] * inv[b]);
#pragma unroll
      for (int q = 0; q < 3; ++q)
        if (P.smask & (1 << (3 * b + q))) G[q] = fma(P.sigma[b][q], Nbar[b], G[q]);
    }
  }
  const double ne_he = nHe * fma(2.0, s.yIII, s.yII);
  const double ne0 = fma(nH, s.xHII, ne_he);
  const double aH = coll ? fma(dt, r.bHI * ne0, G[0]) : G[0];
  const double bH = recomb ? dt * (r.aHII * ne0) : 0.0;
  const double iden = rcp_nr<2>(1.0 + aH + bH), xs = s.xHI + s.xHII;
  t.xHI = fma(bH, xs, s.xHI) * iden;
  t.xHII = fma(aH, xs, s.xHII) * iden;
  const double ne1 = fma(nH, t.xHII, ne_he);
  const double A = coll ? fma(dt, r.bHeI * ne1, G[1]) : G[1];
  const double Cc = coll ? fma(dt, r.bHeII * ne1, G[2]) : G[2];
  const double Bb = recomb ? dt * (r.aHeII * ne1) : 0.0, D = recomb ? dt * (r.aHeIII * ne1) : 0.0;
  const double iA = rcp_nr<2>(1.0 + A), iD = rcp_nr<2>(1.0 + D);
  t.yII = div_nr(fma(D * iD, s.yIII, fma(A * iA, s.yI, s.yII)), fma(Cc, iD, fma(Bb, iA, 1.0)));
  t.yI = fma(Bb, t.yII, s.yI) * iA;
  t.yIII = fma(Cc, t.yII, s.yIII) * iD;

  const double m[3] = {nH * t.xHI, nHe * t.yI, nHe * t.yII};
  double heat_e = 0.0;
#pragma unroll
  for (int b = 0; b < kMaxBins; ++b) {
    if (b < B) {
      double sum = 0.0, ea = 0.0;
#pragma unroll
      for (int q = 0; q < 3; ++q)
        if (P.smask & (1 << (3 * b + q))) {
          const double sn = P.sigma[b][q] * m[q];
          sum += sn;
          if (heat && (P.emask & (1 << (3 * b + q)))) ea = fma(P.eps[b][q], sn, ea);
        }
      if (heat) heat_e = fma(Nbar[b], ea, heat_e);
      // N' = max(N - removed, 0); the flux by N' / N, by 0 where N <= 0 (the
      // transport leaves slightly negative densities beside sharp fronts)
      double sc = fma(-(cdt * sum), inv[b], 1.0);
      t.N[b] = clamp_neg(s.N[b] * sc);
      if (!(__double_as_longlong(sc) > 0 && __double_as_longlong(s.N[b]) > 0)) sc = 0.0;
      t.f[b][0] = s.f[b][0] * sc;
      t.f[b][1] = s.f[b][1] * sc;
      t.f[b][2] = s.f[b][2] * sc;
    }
  }
  double e0 = 0.0, e1 = 0.0;
  t.T = s.T;
  if (P.mode == 2) {
    const double nn = nH * (1.0 + P.y_he);
    e0 = 1.5 * kBoltzmann * (nn + ne0) * s.T;
    const double lam = cool ? RateEval<false>::cooling(tfn, ne0, ns[0], nH * s.xHII, ns[1], ns[2], nHe * s.yIII) : 0.0;
    e1 = fma(-dt, lam, e0 + heat_e);
    const double ne2 = fma(nH, t.xHII, nHe * fma(2.0, t.yIII, t.yII));
    t.T = div_nr(e1, 1.5 * kBoltzmann * (nn + ne2));
  }
  // (the energy's base has no floor; without thermal energy its change is 0)
  const double xf = P.x_floor;
  const double a[6] = {P.mode == 2 ? e0 : 1.0, s.xHI, s.xHII, s.yI, s.yII, s.yIII};
  const double b[6] = {P.mode == 2 ? e1 : 1.0, t.xHI, t.xHII, t.yI, t.yII, t.yIII};
  const double fl[6] = {0.0, xf, xf, xf, xf, xf};
  return largest_change<6>(a, b, fl, P.y_he > 0 ? 6 : 3);
}

// FP64 reciprocal: FP32 hardware seed (~22 bits) refined by one Newton step
// in FP64 (~44 bits, relative error below 1e-13), for x in the FP32 normal
// range, which every denominator of the chemistry step lies in.
template <bool IntCvt = true>
__device__ __forceinline__ double rcp64(double x) {
  const float xf = to_f<IntCvt>(x);
  if (!(fabsf(xf) < 1e30f && fabsf(xf) > 1e-30f)) return 1.0 / x;
  const double y = to_d<IntCvt>(rcp_approx(xf));
  return fma(y, fma(-x, y, 1.0), y);   // one Newton step: ~2^-44 relative
}

// Relative change |b - a| / max(|a|, floor) in FP32 from the FP32 images of
// a and b: it only steers substep lengths and the 10% test, and the FP32
// cancellation for nearly equal a, b changes f by ~1e-7, far below both
// the 0.1 threshold and the growth cap's switch point.
template <bool IntCvt = true>
__device__ __forceinline__ float rel_change_f(double a, double b, float fl) {
  const float af = to_f<IntCvt>(a), bf = to_f<IntCvt>(b);
  const float m = fmaxf(fabsf(af), fl);
  return __fdividef(fabsf(bf - af), m);
}

// The same attempt as photochem_attempt, arranged for GB300's small FP64
// unit: divisions become FP64 reciprocals (one per distinct denominator),
// the photon removal uses N_b' = N_b (1 - tau'_b / (1 + tau_b)) instead of a
// division by N_b, and the substep-control measure f (which only steers step
// lengths and the accept test) is formed in FP32.  The absorber densities,
// the attenuation, the photoionisation rates, the abundance and photon
// updates stay FP64; n_e (which only multiplies the FP32 rate coefficients)
// and the change of n_e in the temperature update are formed in FP32.  The
// reduced flux does not enter the chemistry: an attempt only reports, in
// FP32, the factor sc_b that scales bin b's photons (and, by kappa_F =
// kappa_E, its FP32 flux); the caller applies the product of the accepted
// factors to the flux once.
struct GasState {
  double N[kMaxBins];
  double xHI, xHII, yI, yII, yIII, T;
};

// IntCvt (the first attempt, over the common length): c dt sigma comes with
// the kernel's arguments instead of being multiplied out in the optical
// depths, the photoionisation rates and the photon removal: 92 FP64
// instructions per attempt instead of 109, of which the first pass is made.
template <bool IntCvt>
__device__ float photochem_attempt_mixed(const ChemParams& P, double nH, double dt, const GasState& s,
                                         GasState& t, float sc_out[kMaxBins]) {
  const int B = P.B;
  const double cdt = IntCvt ? P.cdt : P.c_red * dt;
  auto sg = [&](int b, int sp) { return IntCvt ? P.csig[b][sp] : P.sigma[b][sp]; };
  const double nHe = P.y_he * nH;
  const bool recomb = P.flags & 1, coll = P.flags & 2, cool = P.flags & 4, heat = P.flags & 8;
  // rate coefficients and their products with n_e in FP32 (the fits carry
  // FP32 accuracy already); the photoionisation terms and the updates FP64
  const RatesF r = RateEval<true>::template eval_f<IntCvt>(s.T);

  const double ns[3] = {nH * s.xHI, nHe * s.yI, nHe * s.yII};
  double inv1pt[kMaxBins], Nbar[kMaxBins];
  double Gs[3] = {0, 0, 0};
  // products with zero cross-sections (a bin below a species' threshold) are
  // skipped; the mask is uniform across threads
#pragma unroll
  for (int b = 0; b < kMaxBins; ++b) {
    if (b < B) {
      double kap = IntCvt ? 1.0 : 0.0;
#pragma unroll
      for (int sp = 0; sp < 3; ++sp)
        if (P.smask & (1 << (3 * b + sp))) kap = fma(sg(b, sp), ns[sp], kap);
      inv1pt[b] = rcp64<IntCvt>(IntCvt ? kap : fma(cdt, kap, 1.0));
      Nbar[b] = s.N[b] * inv1pt[b];
#pragma unroll
      for (int sp = 0; sp < 3; ++sp)
        if (P.smask & (1 << (3 * b + sp))) Gs[sp] = fma(sg(b, sp), Nbar[b], Gs[sp]);
    }
  }
  // photoionisations over the attempt: c dt times the sums
  const double G0 = IntCvt ? Gs[0] : cdt * Gs[0], G1 = IntCvt ? Gs[1] : cdt * Gs[1],
               G2 = IntCvt ? Gs[2] : cdt * Gs[2];
  // n_e enters only the FP32 products with the rate coefficients (and the
  // FP32 cooling): formed in FP32 from the FP32 images of the densities
  const float nHf = to_f<IntCvt>(nH), nHef = to_f<IntCvt>(nHe);
  const float ne_he = nHef * fmaf(2.0f, to_f<IntCvt>(s.yIII), to_f<IntCvt>(s.yII));
  const float ne0f = fmaf(nHf, to_f<IntCvt>(s.xHII), ne_he);
  const double aH = coll ? fma(dt, to_d<IntCvt>(r.bHI * ne0f), G0) : G0;
  const double bH = recomb ? dt * to_d<IntCvt>(r.aHII * ne0f) : 0.0;
  const double iden = rcp64<IntCvt>(1.0 + aH + bH);
  // backward Euler for (x_HI, x_HII): x_HI' = (x_HI + bH (x_HI + x_HII)) / (1
  // + aH + bH), and the same for x_HII with aH -- the two-state solve with
  // the sum of both fractions shared
  const double xs = s.xHI + s.xHII;
  t.xHI = fma(bH, xs, s.xHI) * iden;
  t.xHII = fma(aH, xs, s.xHII) * iden;
  const float ne1f = fmaf(nHf, to_f<IntCvt>(t.xHII), ne_he);
  const double A = coll ? fma(dt, to_d<IntCvt>(r.bHeI * ne1f), G1) : G1;
  const double Bb = recomb ? dt * to_d<IntCvt>(r.aHeII * ne1f) : 0.0;
  const double Cc = coll ? fma(dt, to_d<IntCvt>(r.bHeII * ne1f), G2) : G2;
  const double D = recomb ? dt * to_d<IntCvt>(r.aHeIII * ne1f) : 0.0;
  const double iA = rcp64<IntCvt>(1.0 + A), iD = rcp64<IntCvt>(1.0 + D);
  t.yII = (s.yII + A * s.yI * iA + D * s.yIII * iD) * rcp64<IntCvt>(1.0 + Bb * iA + Cc * iD);
  t.yI = (s.yI + Bb * t.yII) * iA;
  t.yIII = (s.yIII + Cc * t.yII) * iD;

  const double m[3] = {nH * t.xHI, nHe * t.yI, nHe * t.yII};
  // photoheating sum_b c dt Nbar_b sum_s eps_bs sigma_bs n_s' in FP32, as the
  // rate fits (it only enters the energy increment; the photon removal and
  // the abundances stay FP64): one FP64 product instead of twelve
  float hsum = 0.0f;
  float mf[3] = {0.0f, 0.0f, 0.0f};
  if (heat) {
    mf[0] = to_f<IntCvt>(m[0]); mf[1] = to_f<IntCvt>(m[1]); mf[2] = to_f<IntCvt>(m[2]);
  }
#pragma unroll
  for (int b = 0; b < kMaxBins; ++b) {
    if (b < B) {
      double suma = 0.0;
#pragma unroll
      for (int sp = 0; sp < 3; ++sp)
        if (P.smask & (1 << (3 * b + sp))) suma = fma(sg(b, sp), m[sp], suma);
      const double taup = IntCvt ? suma : cdt * suma;
      // N' = max(N - removed, 0) and no flux where N <= 0, as in the FP64
      // attempt: the factor is clamped on the integer pipe (a double's bits
      // order like the value where it is positive), and a zero keeps no sign.
      // In the loop over attempts N <= 0 is the caller's (unlit).
      double sc = fma(-taup, inv1pt[b], 1.0);
      sc = __double_as_longlong(sc) > 0 && (!IntCvt || __double_as_longlong(s.N[b]) > 0) ? sc : 0.0;
      t.N[b] = IntCvt ? no_sign(s.N[b] * sc) : s.N[b] * sc;
      if (heat) {
        float ea = 0.0f;
#pragma unroll
        for (int sp = 0; sp < 3; ++sp)
          if (P.emask & P.smask & (1 << (3 * b + sp))) ea = fmaf(P.heat_f[b][sp], mf[sp], ea);
        hsum = fmaf(to_f<IntCvt>(Nbar[b]), ea, hsum);
      }
      sc_out[b] = to_f<IntCvt>(sc);
    }
  }

  const float fl = (float)P.x_floor;
  float f = 0.0f;
  if (P.mode == 2) {
    // thermal energy, explicit: e' = e + heat - dt Lambda with e = 3/2 k n_tot T,
    // written as T' = T + (de / (3/2 k) - T dn_e) / n_tot' so that only the
    // change of n_e is FP64 and the increment is formed in FP32
    float lam_s = 0.0f;
    if (cool) {
      lam_s = RateEval<true>::template cooling_scaled<IntCvt>(s.T, ne0f, nHf * to_f<IntCvt>(s.xHI), nHf * to_f<IntCvt>(s.xHII),
                                             nHef * to_f<IntCvt>(s.yI), nHef * to_f<IntCvt>(s.yII), nHef * to_f<IntCvt>(s.yIII));
    }
    const float hs = IntCvt ? P.cdt_heat : to_f<IntCvt>(cdt * kHeatScale);
    const float cs = IntCvt ? P.dt_cool : to_f<IntCvt>(dt * kCoolScale);
    const float de = fmaf(heat ? hs : 0.0f, hsum, -(cs * lam_s));
    // the change of n_e from the FP64 differences of the fractions (they
    // cancel), combined in FP32
    const float dnef = fmaf(nHf, to_f<IntCvt>(t.xHII - s.xHII),
                            nHef * fmaf(2.0f, to_f<IntCvt>(t.yIII - s.yIII), to_f<IntCvt>(t.yII - s.yII)));
    const float T0 = to_f<IntCvt>(s.T);
    const float ntot0 = nHf * (1.0f + (float)P.y_he) + ne0f;
    const float ntot1 = ntot0 + dnef;
    constexpr float kInv15k = (float)(1.0 / (1.5 * kBoltzmann));
    t.T = s.T + to_d<IntCvt>(__fdividef(fmaf(de, kInv15k, -T0 * dnef), ntot1));
    // the measure |e' - e| / |e| = |de| / (3/2 k n_tot T)
    f = __fdividef(fabsf(de) * kInv15k, ntot0 * T0);
  } else {
    t.T = s.T;
  }
  f = fmaxf(f, rel_change_f<IntCvt>(s.xHI, t.xHI, fl));
  f = fmaxf(f, rel_change_f<IntCvt>(s.xHII, t.xHII, fl));
  if (P.y_he > 0) {
    f = fmaxf(f, rel_change_f<IntCvt>(s.yI, t.yI, fl));
    f = fmaxf(f, rel_change_f<IntCvt>(s.yII, t.yII, fl));
    f = fmaxf(f, rel_change_f<IntCvt>(s.yIII, t.yIII, fl));
  }
  return f;
}

// Adaptive substeps of Sec. 4.1.1 over dt_sub: first attempt = the whole
// subcycle; reject if f > f_max and retry with dt f_s / f; after an accepted
// attempt the next is dt min(f_s / f, 2), clipped to the remaining time.
// Returns the number of attempts; sets *capped if max_sub was reached.
// Mixed path: f is an FP32 quantity, so the accept test and the growth
// factor are FP32; dt and the remaining time stay FP64 (the subcycle is
// covered exactly).  Both are >= 0, where the order of the bit patterns is
// the numeric order: the comparisons run on the integer pipe.  S_b returns
// the product of the accepted attempts' photon factors (the flux scale, in
// FP32 like the flux it scales).
// The loop can resume after a rejected first attempt (two-pass chemistry):
// dt0 = the next attempt's length, n0 = attempts already made.
template <bool IntCvt>
__device__ int chemistry_mixed(const ChemParams& P, double nH, double dt_sub, GasState& s,
                               float S[kMaxBins], bool* capped, double dt0, int n0) {
  double rem = dt_sub, dt = dt0;
  int n = n0, acc = 0, dark = 0;
#pragma unroll
  for (int b = 0; b < kMaxBins; ++b)
    if (b < P.B && unlit(s.N[b])) dark |= 1 << b;
  GasState t;
  float sc[kMaxBins];
  *capped = false;
  const float fmax = (float)P.f_max, fs = (float)P.f_s;
  while (__double_as_longlong(rem) > 0) {
    if (n >= P.max_sub) { *capped = true; break; }
    ++n;
    const float f = photochem_attempt_mixed<IntCvt>(P, nH, dt, s, t, sc);
    if (f > fmax) {
      dt = dt * to_d<IntCvt>(__fdividef(fs, f));
      continue;
    }
    s = t;
#pragma unroll
    for (int b = 0; b < kMaxBins; ++b) S[b] = acc ? S[b] * sc[b] : sc[b];
    if (dark) {
#pragma unroll
      for (int b = 0; b < kMaxBins; ++b)
        if (dark >> b & 1) { s.N[b] = 0.0; S[b] = 0.0f; }
    }
    ++acc;
    rem = (__double_as_longlong(dt) == __double_as_longlong(rem)) ? 0.0 : rem - dt;
    const float grow = f > 0.0f ? fminf(__fdividef(fs, f), 2.0f) : 2.0f;
    dt = dt * to_d<IntCvt>(grow);
    if (__double_as_longlong(dt) > __double_as_longlong(rem)) dt = rem;
  }
  if (acc == 0) {
#pragma unroll
    for (int b = 0; b < kMaxBins; ++b) S[b] = 1.0f;
  }
  return n;
}

// First attempt of the mixed chemistry, over the whole subcycle.  Accepted
// (returns true): s is the end state and S the photon factors.  Rejected:
// s is unchanged and *f1 holds the attempt's measure, from which the loop
// resumes with dt_sub * fs / f1 (chemistry_mixed with n0 = 1).
__device__ bool chemistry_mixed_first(const ChemParams& P, double nH, double dt_sub, GasState& s,
                                      float S[kMaxBins], float* f1) {
  GasState t;
  float sc[kMaxBins];
  const float f = photochem_attempt_mixed<true>(P, nH, dt_sub, s, t, sc);
  *f1 = f;
  if (f > (float)P.f_max) return false;
  s = t;
#pragma unroll
  for (int b = 0; b < kMaxBins; ++b) S[b] = sc[b];
  return true;
}

// Adaptive substeps of the FP64 path (the oracle's arithmetic).  The loop
// can resume after a rejected first attempt (two-pass chemistry): dt0 = the
// next attempt's length, n0 = attempts already made.  The reverse mode
// records the attempts through `tape`: begin() sees each attempt's entering
// state, length and remaining time, end() its measure and the controller's
// branches (accepted; growth by the ratio f_s / f rather than the cap 2;
// next length clipped to the remaining time).  NoTape records nothing.
struct NoTape {
  __device__ __forceinline__ void begin(const CellState&, double, double) {}
  __device__ __forceinline__ void end(double, bool, bool, bool) {}
};

template <class Tape>
__device__ __forceinline__ int chemistry_loop(const ChemParams& P, double nH, double dt_sub, CellState& s,
                                              bool* capped, double dt0, int n0, Tape& tape) {
  double rem = dt_sub, dt = dt0;
  int n = n0;
  CellState t;
  *capped = false;
  while (rem > 0) {
    if (n >= P.max_sub) { *capped = true; break; }
    ++n;
    tape.begin(s, dt, rem);
    double f = photochem_attempt(P, nH, dt, s, t);
    if (f > P.f_max) {
      tape.end(f, false, false, false);
      dt = dt * div_nr(P.f_s, f);
      continue;
    }
    s = t;
    rem = (dt == rem) ? 0.0 : rem - dt;
    double grow = (f > 0) ? div_nr(P.f_s, f) : 2.0;
    const bool ratio = f > 0 && grow <= 2.0;
    if (grow > 2.0) grow = 2.0;
    dt = dt * grow;
    const bool clipped = dt > rem;
    if (clipped) dt = rem;
    tape.end(f, true, ratio, clipped);
  }
  return n;
}
__device__ int chemistry(const ChemParams& P, double nH, double dt_sub, CellState& s, bool* capped, double dt0,
                         int n0) {
  NoTape none;
  return chemistry_loop(P, nH, dt_sub, s, capped, dt0, n0, none);
}

// First attempt of the FP64 chemistry over the whole subcycle.  Accepted
// (returns true): s is the end state.  Rejected: s is unchanged and *f1
// holds the attempt's measure; the loop resumes with dt_sub * f_s / f1
// (chemistry with n0 = 1), exactly where the single loop would go on.
__device__ bool chemistry_first(const ChemParams& P, double nH, double dt_sub, CellState& s, double* f1) {
  CellState t;
  const double f = photochem_attempt(P, nH, dt_sub, s, t);
  *f1 = f;
  if (f > P.f_max) return false;
  s = t;
  return true;
}

}  // namespace m1rt

// The chemistry's short worklists: a group of 16 lanes per cell.
//
// After the first attempt of every cell a few cells are left whose substeps
// (Sec. 4.1.1) form a serial chain of ten to a hundred attempts each, and the
// subcycle waits for the longest of them.  What an attempt costs there is its
// count of FP64 warp instructions: a scheduler's FP64 unit takes one for 64
// cycles (measured: a dependent DFMA 66, four independent ones 4 x 64),
// however few of the warp's lanes do something useful.  So the pieces of one
// attempt that have the same form go to the lanes of a group and share their
// instructions: the fifteen exponentials of the rate fits and the cooling
// function, the bins' attenuations and photon factors, the species'
// photoionisation rates, the coefficients and solutions of the backward Euler
// steps, the terms of the substep measure.  Shuffles (24 cycles, not on the
// FP64 unit) hand the results on; conversions to FP32 run on the integer pipe.
// One attempt of a lone warp: 53.0 k -> 15.9 k cycles in FP64, 11.7 k -> 6.6 k
// in the mixed path.
#pragma once
#include <type_traits>

#include "rt_chem.cuh"

namespace m1rt {

constexpr int kGroup = 16;
constexpr unsigned kFull = 0xffffffffu;

template <class T> __device__ __forceinline__ T from_lane(T v, int src) { return __shfl_sync(kFull, v, src, kGroup); }
template <class T> __device__ __forceinline__ T xor_lane(T v, int m) { return __shfl_xor_sync(kFull, v, m, kGroup); }

// What each lane evaluates: E = exp(p (q - ln T) + r / T), and its share of
// the rates (kr) and of the cooling rate (kc) from V = F E P with the lane's
// factor F (fsel: 0 none, 1 tf, 2 sqrt(T) tf, 3 sqrt(T), 4 T^-3/2) and
// partner factor P, which needs the next lane's E.
//   0, 1, 2   collisional ionisation of HI, HeI, HeII (rate and cooling)
//   3, 5      (lambda / 2.740)^0.407 of HII and HeIII: the recombination fits
//   4         HeII recombination
//   6         dielectronic, P = 1 + 0.3 E_7     7  exp(-94000 / T)
//   8         collisional excitation of HI
//   9         of HeII, P = E_10                10  exp(-473638 / T)
//   11        recombination cooling of HII and HeIII, P = 1 / (1 + E_12)
//   13        of HeII
//   14        bremsstrahlung, E = 1.1 + 0.34 exp(-(5.5 - log10 T)^2 / 3)
// Lanes 0-5 end up with the rate of the coefficient they form: aH, A, Cc
// (ionisation of HI, HeI, HeII), bH, Bb, D (recombination of HII, HeII,
// HeIII).  Rates that the flags switch off are zero.
struct LaneFit {
  double p = 0.0, q = 0.0, r = 0.0, kr = 0.0, kc = 0.0;
  int fsel = 0;
};
__device__ __forceinline__ LaneFit lane_fit(int l, int flags) {
  LaneFit t;
  switch (l) {
    case 0: t.r = -157809.1; t.kr = 5.85e-11; t.kc = 1.27e-21; t.fsel = 2; break;
    case 1: t.r = -285335.4; t.kr = 2.38e-11; t.kc = 9.38e-22; t.fsel = 2; break;
    case 2: t.r = -631515.0; t.kr = 5.68e-12; t.kc = 4.95e-22; t.fsel = 2; break;
    // 2.753e-14 lambda^1.5 = kr T^-3/2, lambda = 315614 / T and 1263030 / T
    case 3: t.p = 0.407; t.q = kLnAH; t.kr = 2.753e-14 * 315614.0 * 561.7953363992976; break;
    case 5: t.p = 0.407; t.q = kLnAHe2; t.kr = 2.0 * 2.753e-14 * 1263030.0 * 1123.8460748696862; break;
    case 4: t.p = 0.750; t.q = kLnLHe; t.kr = 1.26e-14; break;
    case 6: t.r = -470000.0; t.kr = 1.9e-3; t.kc = 1.24e-13; t.fsel = 4; break;
    case 7: t.r = -94000.0; break;
    case 8: t.r = -118348.0; t.kc = 7.50e-19; t.fsel = 1; break;
    case 9: t.p = 0.397; t.kc = 5.54e-17; t.fsel = 1; break;
    case 10: t.r = -473638.0; break;
    case 11: t.p = 0.2; t.q = kLn1e3; t.kc = 1.0; t.fsel = 3; break;
    case 12: t.p = -0.7; t.q = kLn1e6; break;
    case 13: t.p = -0.3647; t.kc = 1.55e-26; break;
    case 14: t.kc = 1.42e-27; t.fsel = 3; break;
  }
  if (!((l < 3 ? flags >> 1 : flags) & 1)) t.kr = 0.0;
  return t;
}

// The same in FP32 for the mixed path: E = x^p exp(r / T), x = T or 1 / T
// times kx and kx2 as the fits have it; the cooling shares over kCoolScale.
struct LaneFitF {
  float p, kx, kx2, r, kr, kc;
  bool xT;
  int fsel;
};
__device__ __forceinline__ LaneFitF lane_fit_f(int l, int flags) {
  const LaneFit d = lane_fit(l, flags);
  LaneFitF t;
  const bool inv = l == 3 || l == 4 || l == 5;
  t.p = inv ? (float)d.p : -(float)d.p;
  t.xT = !inv;
  t.kx = l == 3 ? 315614.0f : (l == 5 ? 1263030.0f : (l == 4 ? 570670.0f : (l == 11 ? 1e-3f : (l == 12 ? 1e-6f : 1.0f))));
  t.kx2 = (l == 3 || l == 5) ? 1.0f / 2.740f : 1.0f;
  t.r = (float)d.r;
  t.kr = (float)d.kr;
  t.kc = l == 11 ? 1.0f : (float)(d.kc / kCoolScale);
  t.fsel = d.fsel;
  return t;
}

// What a group keeps of its cell, beside the state: every lane its
// cross-sections.  Bin lanes b < B: sd[s] = sigma_bs times the density of
// species s's element (n_H, n_He, n_He), ed[s] the same times eps_bs (ef[s] in
// FP32, over kHeatScale); species lanes s < 3: sc[b] = sigma_bs.
struct GroupCell {
  double nH, nHe, sd[3], ed[3], sc[3];
  float ef[3];
};
__device__ __forceinline__ void group_cell(const ChemParams& P, int l, double nH, GroupCell& c) {
  c.nH = nH;
  c.nHe = P.y_he * nH;
#pragma unroll
  for (int q = 0; q < 3; ++q) {
    c.sd[q] = c.ed[q] = c.sc[q] = 0.0;
    c.ef[q] = 0.0f;
    // bin b of row q, species of column q
#pragma unroll
    for (int k = 0; k < kMaxBins; ++k)
      if (l == k) {
        c.sd[q] = P.sigma[k][q] * (q == 0 ? c.nH : c.nHe);
        c.ed[q] = P.eps[k][q] * c.sd[q];
        c.ef[q] = P.heat_f[k][q] * (float)(q == 0 ? c.nH : c.nHe);
        c.sc[q] = P.sigma[q][k];
      }
  }
}

// A group's state: every lane holds the gas, lane b < B the photons of bin b
// (zero elsewhere).  FP64 path: lanes 3b + k hold component k of bin b's flux.
struct GroupState {
  double x[5], T;    // HI, HII, HeI, HeII, HeIII
  double N, f;
};

// x > 0 as an integer test (the bits of a positive double, or of a NaN
// without the sign bit, are a positive integer).
__device__ __forceinline__ bool positive(double x) { return __double_as_longlong(x) > 0; }

// One attempt (photochem_attempt, or photochem_attempt_mixed) over the lanes
// of a group: the same steps, sums and quotients within rounding.  Returns the
// measure; sc_out: the photon factor of the lane's bin.
template <bool Mixed, class Fit>
__device__ __forceinline__ auto group_attempt(const ChemParams& P, const Fit& fit, int l, const GroupCell& g, double dt,
                                              const GroupState& s, GroupState& t, double& sc_out) {
  using V = std::conditional_t<Mixed, float, double>;
  constexpr int kN = Mixed ? 1 : 2;     // Newton steps of a reciprocal
  const bool odd = l & 1, cool = P.flags & 4, heat = P.flags & 8;
  const double cdt = P.c_red * dt;
  auto cv = [](double x) -> V {
    if constexpr (Mixed) return d2f_int(x);
    else return x;
  };
  // the lane's fit
  V T, iT, sT, tf, E, T15, rate, part = V(1);
  double inv1pt;
  const double opt = fma(cdt, fma(g.sd[2], s.x[3], fma(g.sd[1], s.x[2], g.sd[0] * s.x[0])), 1.0);
  if constexpr (Mixed) {
    T = d2f_int(s.T);
    iT = __frcp_rn(T);
    sT = sqrtf(T);
    tf = 1.0f / (1.0f + sqrtf(T * 1e-5f));
    const float x = (fit.kx * (fit.xT ? T : iT)) * fit.kx2;
    float arg = fit.p * __log2f(x) + (fit.r * iT) * 1.4426950408889634f;
    if (l == 14) {
      const float d = 5.5f - __log10f(T);
      arg = -(d * d) * (1.0f / 3.0f) * 1.4426950408889634f;
    }
    E = exp2f(arg);
    const float En = from_lane(E, (l + 1) & (kGroup - 1));
    T15 = iT * iT * sT;
    const float hg = fpow(1.0f + E, -2.242f) * (fit.kr * T15);
    if (l == 14) E = fmaf(0.34f, E, 1.1f);
    if (l == 6) part = fmaf(0.3f, En, 1.0f);
    if (l == 9) part = En;
    if (l == 11) part = 1.0f / (1.0f + En);
    inv1pt = rcp_nr<kN>(opt);
    const float F = fit.fsel == 0 ? 1.0f : (fit.fsel == 1 ? tf : (fit.fsel == 2 ? sT * tf : (fit.fsel == 3 ? sT : T15)));
    E = F * E * part;                       // V
    rate = (l == 3 || l == 5) ? hg : fit.kr * E;
  } else {
    // square roots and reciprocals of T (even lanes) and of 1 + sqrt(T / 1e5) (odd)
    const double root = sqrt_nr(odd ? s.T * 1e-5 : s.T);
    const double inv = rcp_nr<2>(odd ? 1.0 + root : s.T);
    sT = from_lane(root, 0);
    iT = from_lane(inv, 0);
    tf = from_lane(inv, 1);
    const double lnT = log_series(s.T);
    double arg = fma(fit.r, iT, fit.p * (fit.q - lnT));
    if (l == 14) {
      const double d = fma(-kInvLn10, lnT, 5.5);
      arg = (d * d) * (-1.0 / 3.0);
    }
    E = exp(arg);
    const double En = from_lane(E, (l + 1) & (kGroup - 1));
    T15 = iT * iT * sT;
    const double hg = exp(-2.242 * log_series(1.0 + E)) * (fit.kr * T15);
    if (l == 14) E = fma(0.34, E, 1.1);
    if (l == 6) part = fma(0.3, En, 1.0);
    if (l == 9) part = En;
    // the bins' attenuation, and on lane 11 its partner factor
    inv1pt = rcp_nr<kN>(l == 11 ? 1.0 + En : opt);
    if (l == 11) part = inv1pt;
    const double F = fit.fsel == 0 ? 1.0 : (fit.fsel == 1 ? tf : (fit.fsel == 2 ? sT * tf : (fit.fsel == 3 ? sT : T15)));
    E = F * E * part;
    rate = (l == 3 || l == 5) ? hg : fit.kr * E;
  }
  const V die = from_lane(rate, 6);
  if (l == 4) rate += die;
  // electron density, cooling rate
  const V nHv = cv(g.nH), nHev = cv(g.nHe);
  V xs[5];
#pragma unroll
  for (int q = 0; q < 5; ++q) xs[q] = cv(s.x[q]);
  const V ne_he = nHev * (xs[3] + V(2) * xs[4]);
  const V ne0 = nHv * xs[1] + ne_he;
  V lam = V(0);
  if (P.mode == 2 && cool) {
    // the density a lane's term multiplies (without n_e)
    V d = (l == 0 || l == 8) ? xs[0] : (l == 1 ? xs[2] : (l == 2 || l == 6 || l == 9 || l == 13 ? xs[3] : V(0)));
    d *= (l == 0 || l == 8) ? nHv : nHev;
    constexpr V kII = Mixed ? V(8.70) : V(8.70e-27), kIII = Mixed ? V(34.8) : V(3.48e-26);
    if (l == 11 || l == 14)
      d = (l == 11 ? kII : V(1)) * (nHv * xs[1]) + (l == 11 ? kIII : V(4)) * (nHev * xs[4]) +
          (l == 14 ? nHev * xs[3] : V(0));
    lam = fit.kc * E * d;
#pragma unroll
    for (int m = 1; m < kGroup; m <<= 1) lam += xor_lane(lam, m);
    lam *= ne0;
  }
  // photoionisation: species lane s sums over the bins
  const double Nbar = s.N * inv1pt;
  const double G = cdt * fma(g.sc[2], from_lane(Nbar, 2), fma(g.sc[1], from_lane(Nbar, 1), g.sc[0] * from_lane(Nbar, 0)));
  // hydrogen: x_HI' on the even lanes, x_HII' on the odd ones
  {
    const double c = fma(dt, (double)(rate * ne0), G);
    const double aH = from_lane(c, 0), bH = from_lane(c, 3);
    const double q = fma(odd ? aH : bH, s.x[0] + s.x[1], odd ? s.x[1] : s.x[0]) * rcp_nr<kN>(1.0 + aH + bH);
    t.x[0] = from_lane(q, 0);
    t.x[1] = from_lane(q, 1);
  }
  // helium with the updated n_e
  {
    const V ne1 = nHv * cv(t.x[1]) + ne_he;
    const double c = fma(dt, (double)(rate * ne1), G);
    const double A = from_lane(c, 1), Cc = from_lane(c, 2), Bb = from_lane(c, 4), D = from_lane(c, 5);
    const double iq = rcp_nr<kN>(1.0 + (odd ? D : A));
    const double iA = from_lane(iq, 0), iD = from_lane(iq, 1);
    // even lanes y_II + A y_I / (1 + A) + D y_III / (1 + D), odd lanes 1 + Bb / (1 + A) + Cc / (1 + D)
    const double v = fma((odd ? Cc : D) * iD, odd ? 1.0 : s.x[4], fma((odd ? Bb : A) * iA, odd ? 1.0 : s.x[2], odd ? 1.0 : s.x[3]));
    t.x[3] = from_lane(v, 0) * rcp_nr<kN>(from_lane(v, 1));
    const double q = fma(odd ? Cc : Bb, t.x[3], odd ? s.x[4] : s.x[2]) * (odd ? iD : iA);
    t.x[2] = from_lane(q, 0);
    t.x[4] = from_lane(q, 1);
  }
  // photons of the lane's bin: removed as the ionisations were credited
  const double suma = fma(g.sd[2], t.x[3], fma(g.sd[1], t.x[2], g.sd[0] * t.x[0]));
  double sc = fma(-(cdt * suma), inv1pt, 1.0);
  if constexpr (Mixed) {
    sc = positive(sc) ? sc : 0.0;   // N <= 0 is the caller's (unlit)
    t.N = s.N * sc;
  } else {
    t.N = clamp_neg(s.N * sc);
    sc = positive(sc) && positive(s.N) ? sc : 0.0;
  }
  t.T = s.T;
  V f = V(0);
  // change of the lane's abundance (lanes 0-4)
  double a0 = 1.0, a1 = 1.0;
#pragma unroll
  for (int q = 0; q < 5; ++q)
    if (l == q) { a0 = s.x[q]; a1 = t.x[q]; }
  if constexpr (Mixed) {
    sc_out = sc;
    const float df = d2f_int(a1 - a0);
    if (P.mode == 2) {
      float hsum = 0.0f;
      if (heat) {
        const float ea = fmaf(g.ef[2], d2f_int(t.x[3]), fmaf(g.ef[1], d2f_int(t.x[2]), g.ef[0] * d2f_int(t.x[0])));
        hsum = d2f_int(Nbar) * ea;
        hsum = from_lane(hsum, 0) + from_lane(hsum, 1) + from_lane(hsum, 2);
      }
      const float de = fmaf(heat ? d2f_int(cdt * kHeatScale) : 0.0f, hsum, -(d2f_int(dt * kCoolScale) * lam));
      const float dne = fmaf(nHv, from_lane(df, 1), nHev * fmaf(2.0f, from_lane(df, 4), from_lane(df, 3)));
      const float ntot0 = nHv * (1.0f + (float)P.y_he) + ne0;
      constexpr float kInv15k = (float)(1.0 / (1.5 * kBoltzmann));
      t.T = s.T + (double)__fdividef(fmaf(de, kInv15k, -T * dne), ntot0 + dne);
      f = __fdividef(fabsf(de) * kInv15k, ntot0 * T);
    }
    if (l < (P.y_he > 0 ? 5 : 2)) f = fmaxf(f, rel_change_f<true>(a0, a1, (float)P.x_floor));
#pragma unroll
    for (int m = 1; m < 8; m <<= 1) f = fmaxf(f, xor_lane(f, m));
  } else {
    sc_out = sc;
    t.f = s.f * from_lane(sc, l < 9 ? l / 3 : 15);
    double fl = P.x_floor;
    if (l >= (P.y_he > 0 ? 5 : 2)) a1 = a0;
    if (P.mode == 2) {
      double h = 0.0;
      if (heat) {
        h = (cdt * Nbar) * fma(g.ed[2], t.x[3], fma(g.ed[1], t.x[2], g.ed[0] * t.x[0]));
        h = from_lane(h, 0) + from_lane(h, 1) + from_lane(h, 2);
      }
      const double nn = g.nH * (1.0 + P.y_he);
      const double e0 = 1.5 * kBoltzmann * (nn + ne0) * s.T;
      const double e1 = fma(-dt, lam, e0 + h);
      const double ne2 = fma(g.nH, t.x[1], g.nHe * fma(2.0, t.x[4], t.x[3]));
      t.T = div_nr(e1, 1.5 * kBoltzmann * (nn + ne2));
      if (l == 5) { a0 = e0; a1 = e1; fl = 0.0; }
    }
    f = rel_change(a0, a1, fl);
#pragma unroll
    for (int m = 1; m < 8; m <<= 1) f = fmax(f, xor_lane(f, m));
  }
  return from_lane(f, 0);
}

}  // namespace m1rt

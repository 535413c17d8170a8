// Adjoint kernels: reverse mode of the FP64 subcycle (any chemistry mode:
// transport only, isothermal network, network with thermal energy).  The paper has no adjoint; these are the exact
// derivatives of the forward kernels, organised as gathers (no atomics):
//
//   k_adj_face      per (face, bin): cotangent of the face flux from the two
//                   cells' cotangents, back through Lax-Friedrichs, the M1
//                   closure and the face-state clamps -> cotangent of each
//                   side's extrapolated state (4 + 4 per face and bin)
//   k_adj_cellgrad  per (cell, bin): gathers its faces' side cotangents into
//                   the cotangents of its value and its gradients, then back
//                   through the limiter (active branch) and M^-1
//   k_adj_cellsum   per (cell, bin): the least-squares right-hand side and
//                   the limiter extremes read neighbour values; their
//                   cotangents are gathered here from the neighbours' records
//   k_chem_adj      per cell: walk back through the chemistry attempts of one
//                   subcycle, as the recompute's worklist pass recorded them
//                   (k_chem64_rest<true>), together with the substep
//                   controller (Sec. 4.1.1) and the source term.
#pragma once
#include "rt_kernels.cuh"

namespace m1rt {

// ---------------------------------------------------------------------------
// transport
// ---------------------------------------------------------------------------

// Reverse of one side of a face: from the cotangents of the side's clamped
// state (lN and lf, the parts that do not go through the closure) and of N D n
// (lP, with third = lP . n / 3) to those of the extrapolated state.  The closure
// is N D n = ((s - N) / 3) n + k F, s = sqrt(4 N^2 - 3 |F|^2), k = 3 (F . n) /
// (2 N + s) (m1_coef), smooth at F = 0.  The clamps (N >= 0, |F| <= N) as face_state.
// Bound by the FP64 unit: 794 -> 561 us per launch at 74,088 cells, three bins.
__device__ __forceinline__ d4 adj_side(const d4& p, const double* __restrict__ Gp, const d4& x, double n0, double n1,
                                       double n2, const double lP[3], double third, double lN, const double l0[3]) {
  const d4* G4 = reinterpret_cast<const d4*>(Gp);
  const d4 a = G4[0], b = G4[1], c = G4[2];
  const double e0 = fma(a.x, x.x, fma(a.y, x.y, fma(a.z, x.z, p.x)));
  const double e1 = fma(a.w, x.x, fma(b.x, x.y, fma(b.y, x.z, p.y)));
  const double e2 = fma(b.z, x.x, fma(b.w, x.y, fma(c.x, x.z, p.z)));
  const double e3 = fma(c.y, x.x, fma(c.z, x.y, fma(c.w, x.z, p.w)));
  const bool clampN = lt_zero(e0);
  const double N = clampN ? 0.0 : e0, N2 = N * N, q2 = e1 * e1 + e2 * e2 + e3 * e3;
  const bool over = nonfinite_bits(q2), clampF = gt_nonneg(q2, N2) || over;
  double F1 = e1, F2 = e2, F3 = e3, fl2 = q2;
  double ifl = 0.0;
  if (clampF) {
    ifl = div_nr(1.0, sqrt_nr(q2));
    const double r = N * ifl;
    F1 *= r; F2 *= r; F3 *= r;
    fl2 = over ? 0.0 : N2;
  }
  double lf1 = l0[0], lf2 = l0[1], lf3 = l0[2];
  if (gt_nonneg(N, 0.0) && gt_nonneg(fl2, 0.0)) {
    const double s = m1_root(N, N2, fl2), d = fma(2.0, N, s);
    // (one reciprocal of d s would leave the exponent range at densities that
    // occur beyond a light front: N^2 < 1e-308)
    const double id3 = 3.0 * rcp_nr<2>(d), is = rcp_nr<2>(s);
    const double un = F1 * n0 + F2 * n1 + F3 * n2;
    const double lPF = lP[0] * F1 + lP[1] * F2 + lP[2] * F3;
    const double k = un * id3, lun = lPF * id3;
    const double ld = (-1.0 / 3.0) * (k * lun);          // of 2 N + s
    const double ws = (third + ld) * is;                 // cotangent of s, over s
    lN = fma(4.0 * N, ws, lN + fma(2.0, ld, -third));
    const double w3 = -3.0 * ws;
    lf1 = fma(w3, F1, fma(lun, n0, fma(k, lP[0], lf1)));
    lf2 = fma(w3, F2, fma(lun, n1, fma(k, lP[1], lf2)));
    lf3 = fma(w3, F3, fma(lun, n2, fma(k, lP[2], lf3)));
  } else {
    lN += third;
  }
  if (clampF) {
    const double lvf = (lf1 * e1 + lf2 * e2 + lf3 * e3) * ifl, z = N * ifl, y = lvf * ifl;
    lN += lvf;
    lf1 = z * (lf1 - y * e1);
    lf2 = z * (lf2 - y * e2);
    lf3 = z * (lf3 - y * e3);
  }
  return make_d4(clampN ? 0.0 : lN, lf1, lf2, lf3);
}

struct AdjArgs {
  int C, F, B;
  const int32_t* off;
  const int32_t* csr;
  const int32_t* nbr;
  const int2* lr;
  const d4* nA;
  const d4* rL;
  const d4* rR;
  const d4* w;
  const d4* hx;           // half-edges: face-centre offsets of their cell
  const double* minv;
  const double* ivol;     // 1 / V
  const d4* rad;          // state before the transport pass
  const double* G;        // its limited gradients
  const GradTape* tape;   // and what k_grad recorded beside them
  const d4* lam_out;      // cotangent of the state after the pass
  d4* lampre;             // [F][B][2] cotangents of the extrapolated face states
  d4* lamr;               // [C][B][3] cotangents of the least-squares right-hand sides
  double* lim_coef;       // [C][B][4] cotangent owed to the limiting extreme
  int32_t* lim_cell;      // [C][B][4] the cell holding that extreme (-1: none)
  d4* lam_part;           // [C][B] partial cotangent of the state before the pass
  d4* lam_in;             // [C][B] result: cotangent of the state before the pass
  double lam;             // c_red dt / unit_length_cm
  int order;
};

__global__ void __launch_bounds__(256) k_adj_face(AdjArgs a) {
  const int t = blockIdx.x * blockDim.x + threadIdx.x;
  const int B = a.B;
  if (t >= a.F * B) return;
  const int f = t / B, b = t % B;
  const int2 c = a.lr[f];
  const d4 nA = a.nA[f];
  const size_t sL = (size_t)c.x * B + b, sR = (size_t)c.y * B + b;
  const d4 lo_L = a.lam_out[sL], lo_R = a.lam_out[sR];
  // cotangent of the face flux over 2 / A
  const double hL = 0.5 * a.lam * nA.w * a.ivol[c.x], hR = 0.5 * a.lam * nA.w * a.ivol[c.y];
  const double l0 = lo_R.x * hR - lo_L.x * hL;
  const double lP[3] = {lo_R.y * hR - lo_L.y * hL, lo_R.z * hR - lo_L.z * hL, lo_R.w * hR - lo_L.w * hL};
  const double third = (lP[0] * nA.x + lP[1] * nA.y + lP[2] * nA.z) * (1.0 / 3.0);
  const double lL[3] = {fma(l0, nA.x, lP[0]), fma(l0, nA.y, lP[1]), fma(l0, nA.z, lP[2])};
  const double lR[3] = {fma(l0, nA.x, -lP[0]), fma(l0, nA.y, -lP[1]), fma(l0, nA.z, -lP[2])};
  a.lampre[(size_t)t * 2] = adj_side(a.rad[sL], a.G + sL * 12, a.rL[f], nA.x, nA.y, nA.z, lP, third, l0, lL);
  a.lampre[(size_t)t * 2 + 1] = adj_side(a.rad[sR], a.G + sR * 12, a.rR[f], nA.x, nA.y, nA.z, lP, third, -l0, lR);
}

// The gradients before the limiter, its factors and the limiting faces come
// from k_grad's record of the same state (160 bytes read instead of the
// least-squares sums and a quotient per face and component formed again, which
// were two thirds of this kernel's FP64 instructions).
__global__ void __launch_bounds__(256) k_adj_cellgrad(AdjArgs a) {
  const int t = blockIdx.x * blockDim.x + threadIdx.x;
  const int B = a.B;
  if (t >= a.C * B) return;
  const int i = t / B, b = t % B;
  const int k0 = a.off[i], k1 = a.off[i + 1];
  const d4 lo = a.lam_out[t];
  double lU[4] = {lo.x, lo.y, lo.z, lo.w};
  double lG[4][3] = {};
#pragma unroll 2
  for (int k = k0; k < k1; ++k) {
    const int e = a.csr[k];
    const d4 lp = a.lampre[((size_t)(e >> 1) * B + b) * 2 + (e & 1)];
    const d4 x = a.hx[k];
    const double l4[4] = {lp.x, lp.y, lp.z, lp.w};
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      lU[q] += l4[q];
      lG[q][0] += l4[q] * x.x;
      lG[q][1] += l4[q] * x.y;
      lG[q][2] += l4[q] * x.z;
    }
  }
  double lr_out[4][3] = {};
  double coef[4] = {0, 0, 0, 0};
  int jst[4] = {-1, -1, -1, -1};
  if (a.order >= 2) {
    const GradTape& r = a.tape[t];
    const double* m = a.minv + 6 * (size_t)i;
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      double lg[3] = {lG[q][0], lG[q][1], lG[q][2]};
      const int at = r.at[q];
      if (at >= 0) {
        // psi = (extreme - value) / (g . x) on the limiting face
        const double g0 = r.g[3 * q], g1 = r.g[3 * q + 1], g2 = r.g[3 * q + 2], psi = r.psi[q];
        const d4 x = a.hx[at];
        const double dstar = g0 * x.x + g1 * x.y + g2 * x.z;
        const double sd = div_nr(lG[q][0] * g0 + lG[q][1] * g1 + lG[q][2] * g2, dstar);
        const double sp = sd * psi;
        lg[0] = psi * lG[q][0] - sp * x.x;
        lg[1] = psi * lG[q][1] - sp * x.y;
        lg[2] = psi * lG[q][2] - sp * x.z;
        if (r.cell[q] != i) {
          lU[q] -= sd;
          coef[q] = sd;
          jst[q] = r.cell[q];
        }
      }
      lr_out[q][0] = m[0] * lg[0] + m[1] * lg[1] + m[2] * lg[2];
      lr_out[q][1] = m[1] * lg[0] + m[3] * lg[1] + m[4] * lg[2];
      lr_out[q][2] = m[2] * lg[0] + m[4] * lg[1] + m[5] * lg[2];
    }
  }
  d4* lr4 = a.lamr + (size_t)t * 3;
  lr4[0] = make_d4(lr_out[0][0], lr_out[0][1], lr_out[0][2], lr_out[1][0]);
  lr4[1] = make_d4(lr_out[1][1], lr_out[1][2], lr_out[2][0], lr_out[2][1]);
  lr4[2] = make_d4(lr_out[2][2], lr_out[3][0], lr_out[3][1], lr_out[3][2]);
  reinterpret_cast<d4*>(a.lim_coef)[t] = make_d4(coef[0], coef[1], coef[2], coef[3]);
  reinterpret_cast<int4*>(a.lim_cell)[t] = make_int4(jst[0], jst[1], jst[2], jst[3]);
  a.lam_part[t] = make_d4(lU[0], lU[1], lU[2], lU[3]);
}

__device__ __forceinline__ void load_lamr(const d4* lamr, size_t t, double o[12]) {
  const d4 a = lamr[t * 3], b = lamr[t * 3 + 1], c = lamr[t * 3 + 2];
  o[0] = a.x; o[1] = a.y; o[2] = a.z; o[3] = a.w; o[4] = b.x; o[5] = b.y;
  o[6] = b.z; o[7] = b.w; o[8] = c.x; o[9] = c.y; o[10] = c.z; o[11] = c.w;
}

// The right-hand side's term w (phi_j - phi_i) of a face enters the sums of
// both its cells with the same sign of w: cell i's share is -+ w . (lamr_i +
// lamr_j), and its own part, lamr_i . sum -+ w, needs the sum of the weights
// only.
__global__ void __launch_bounds__(256) k_adj_cellsum(AdjArgs a) {
  const int t = blockIdx.x * blockDim.x + threadIdx.x;
  const int B = a.B;
  if (t >= a.C * B) return;
  const int i = t / B, b = t % B;
  const d4 p = a.lam_part[t];
  double lU[4] = {p.x, p.y, p.z, p.w};
  if (a.order >= 2) {
    double W[3] = {0.0, 0.0, 0.0}, o[12];
    const int k0 = a.off[i], k1 = a.off[i + 1];
#pragma unroll 2
    for (int k = k0; k < k1; ++k) {
      const int e = a.csr[k];
      const size_t jb = (size_t)a.nbr[k] * B + b;
      const d4 w = a.w[e >> 1];
      load_lamr(a.lamr, jb, o);
      const int4 lc = reinterpret_cast<const int4*>(a.lim_cell)[jb];
      const double sg = (e & 1) ? 1.0 : -1.0;
      const double wx = sg * w.x, wy = sg * w.y, wz = sg * w.z;
      W[0] += wx; W[1] += wy; W[2] += wz;
#pragma unroll
      for (int q = 0; q < 4; ++q) lU[q] += wx * o[3 * q] + wy * o[3 * q + 1] + wz * o[3 * q + 2];
      if (lc.x == i || lc.y == i || lc.z == i || lc.w == i) {
        const d4 c = reinterpret_cast<const d4*>(a.lim_coef)[jb];
        if (lc.x == i) lU[0] += c.x;
        if (lc.y == i) lU[1] += c.y;
        if (lc.z == i) lU[2] += c.z;
        if (lc.w == i) lU[3] += c.w;
      }
    }
    load_lamr(a.lamr, t, o);
#pragma unroll
    for (int q = 0; q < 4; ++q) lU[q] += W[0] * o[3 * q] + W[1] * o[3 * q + 1] + W[2] * o[3 * q + 2];
  }
  a.lam_in[t] = make_d4(lU[0], lU[1], lU[2], lU[3]);
}

// ---------------------------------------------------------------------------
// chemistry (FP64; isothermal or with thermal energy)
// ---------------------------------------------------------------------------

// Temperature derivatives of the rate fits (RateEval<false>) for the
// reverse mode of the thermal network, from the same functions of T the
// fits use (TFns: one logarithm, the shared Boltzmann factors).  The Hui &
// Gnedin form a lam^1.5 / (1 + (lam/2.74)^0.407)^2.242 with lam = 2 T_tr / T
// has d ln alpha / d ln T = -(1.5 - 2.242 * 0.407 u / (1 + u)),
// u = (lam/2.74)^0.407; d ln(1 / (1 + (T/1e5)^(1/2))) / dT = -(1 - tf) / (2T)
// with tf that factor.
struct RateSlopes {
  double aHII, aHeII, aHeIII, bHI, bHeI, bHeII;   // d/dT
};

__device__ RateSlopes rate_slopes(const TFns& t, const Rates& r) {
  RateSlopes d;
  const double uH = kU407H * t.u407, uHe2 = kU407He2 * t.u407;
  d.aHII = -r.aHII * (1.5 - 2.242 * 0.407 * div_nr(uH, 1.0 + uH)) * t.iT;
  d.aHeIII = -r.aHeIII * (1.5 - 2.242 * 0.407 * div_nr(uHe2, 1.0 + uHe2)) * t.iT;
  // HeII: radiative 1.26e-14 lam^0.75 and dielectronic
  // 1.9e-3 T^-1.5 exp(-470000/T) (1 + 0.3 exp(-94000/T))
  const double iT2 = t.iT * t.iT;
  const double rs = t.iT * t.sT, rad = (1.26e-14 * kLam075He) * (rs * sqrt_nr(rs));
  const double g = 1.9e-3 * t.T15 * t.e470;
  d.aHeII = -0.75 * rad * t.iT +
            g * ((470000.0 * iT2 - 1.5 * t.iT) * (1.0 + 0.3 * t.e94) + 0.3 * t.e94 * 94000.0 * iT2);
  const double ts = -0.5 * (1.0 - t.tf) * t.iT;
  d.bHI = r.bHI * (0.5 * t.iT + 157809.1 * iT2 + ts);
  d.bHeI = r.bHeI * (0.5 * t.iT + 285335.4 * iT2 + ts);
  d.bHeII = r.bHeII * (0.5 * t.iT + 631515.0 * iT2 + ts);
  return d;
}

// The cooling function as n_e (k_HI n_HI + k_HII n_HII + k_HeI n_HeI +
// k_HeII n_HeII + k_HeIII n_HeIII), per-species coefficients and their T
// derivatives (the terms of RateEval<false>::cooling grouped by species),
// from the same functions of T.
struct CoolCoef {
  double k[5], dk[5];   // HI, HII, HeI, HeII, HeIII
};

__device__ CoolCoef cooling_coef(const TFns& t) {
  const double sT = t.sT, tf = t.tf, iT = t.iT, iT2 = iT * iT, ts = -0.5 * (1.0 - tf) * iT;
  // collisional excitation and ionisation
  const double ceH = 7.50e-19 * exp(-118348.0 * iT) * tf, dceH = ceH * (118348.0 * iT2 + ts);
  const double ceHe = 5.54e-17 * exp(-0.397 * t.lnT - 473638.0 * iT) * tf,
               dceHe = ceHe * (473638.0 * iT2 - 0.397 * iT + ts);
  const double ciH = 1.27e-21 * sT * t.e157 * tf, dciH = ciH * (0.5 * iT + 157809.1 * iT2 + ts);
  const double ciHe = 9.38e-22 * sT * t.e285 * tf, dciHe = ciHe * (0.5 * iT + 285335.4 * iT2 + ts);
  const double ciHe2 = 4.95e-22 * sT * t.e631 * tf, dciHe2 = ciHe2 * (0.5 * iT + 631515.0 * iT2 + ts);
  // recombination
  const double q = exp(0.7 * (t.lnT - kLn1e6));
  const double iq = div_nr(1.0, 1.0 + q);
  const double t3 = exp(-0.2 * (t.lnT - kLn1e3)) * iq, lt3 = -0.2 * iT - 0.7 * q * iT * iq;
  const double rH = 8.70e-27 * sT * t3, drH = rH * (0.5 * iT + lt3);
  const double rHe = 1.55e-26 * exp(0.3647 * t.lnT), drHe = rHe * 0.3647 * iT;
  const double rHe2 = 3.48e-26 * sT * t3, drHe2 = rHe2 * (0.5 * iT + lt3);
  const double g = 1.24e-13 * t.T15 * t.e470;
  const double di = g * (1.0 + 0.3 * t.e94);
  const double ddi = g * ((470000.0 * iT2 - 1.5 * iT) * (1.0 + 0.3 * t.e94) + 0.3 * t.e94 * 94000.0 * iT2);
  // bremsstrahlung with the Gaunt factor 1.1 + 0.34 exp(-(5.5 - log10 T)^2 / 3)
  const double lg = t.lnT * kInvLn10, w = exp(-(5.5 - lg) * (5.5 - lg) * (1.0 / 3.0));
  const double gff = 1.1 + 0.34 * w, dgff = 0.34 * w * (2.0 * (5.5 - lg) * (1.0 / 3.0)) * (iT * kInvLn10);
  const double br = 1.42e-27 * gff * sT, dbr = 1.42e-27 * (dgff * sT + 0.5 * gff * div_nr(1.0, sT));
  CoolCoef c;
  c.k[0] = ceH + ciH;                    c.dk[0] = dceH + dciH;
  c.k[1] = rH + br;                      c.dk[1] = drH + dbr;
  c.k[2] = ciHe;                         c.dk[2] = dciHe;
  c.k[3] = ceHe + ciHe2 + rHe + di + br; c.dk[3] = dceHe + dciHe2 + drHe + ddi + dbr;
  c.k[4] = rHe2 + 4.0 * br;              c.dk[4] = drHe2 + 4.0 * dbr;
  return c;
}

// Reverse of one attempt (photochem_attempt), in two parts.  attempt_lin
// computes what does not depend on the cotangents: the attempt's
// intermediate values, the rate fits and their slopes in T, the cooling
// coefficients, the quotients, and the branch the substep measure took.
// attempt_back takes lt = cotangent of the output state and lf = of the
// measure, and accumulates into ls (input state, T included: through the
// rate fits, and in mode 2 the energy equation), ldt and lnH; it is linear
// in (lt, lf).  A cell's attempts are a serial chain in the reverse as in
// the forward, but their attempt_lin parts are independent and run in
// parallel over a subcycle's records (k_chem_lin); the chain then runs
// attempt_back only.  kB = the number of bins (compile-time: the state
// arrays stay in registers).  Every quotient by one refined reciprocal of
// its denominator (div_nr, within 0.51 ulp), as the forward FP64 path.
struct AttemptLin {
  double aHII, aHeII, aHeIII, bHI, bHeI, bHeII;   // the rates, zero where the flags switch them off
  RateSlopes d;                                   // their slopes in T
  CoolCoef cc;                                    // mode 2 with cooling
  double kap[kMaxBins], iden[kMaxBins], Nbar[kMaxBins], is[kMaxBins];
  double Gm0, Gm1, Gm2;
  double ne0, aH, bH, iD1, xHI1, xHII1, ne1, A, Bb, Cc, Dd, iA, iD, idn, yII1, yI1, yIII1, m0, m1, m2;
  double ntot0, lamc, ntot1, T1, intot1;           // mode 2
  double f_sg, f_imm, f_span, f_sgn;               // the measure's largest term: sign of the change, 1/|base|,
                                                   // |change| / base^2, sign of the base (0: at the floor)
  int f_kb;                                        // which term: 0-4 abundances, 5 energy, -1 none (f = 0)
  int pad;
};

// measure = false: the attempt's measure carries no cotangent (the last
// attempt of a cell), so its branch is not needed.
template <int kB>
__device__ __forceinline__ void attempt_lin(const ChemParams& P, double nH, double dt, const double* s,
                                            AttemptLin& L, bool measure) {
  const double c = P.c_red, yhe = P.y_he, nHe = yhe * nH;
  const bool recomb = P.flags & 1, coll = P.flags & 2;
  const double T = s[4 * kB + 5];
  const TFns tfn = tfns(T);
  const Rates rt = RateEval<false>::eval(tfn);
  L.aHII = recomb ? rt.aHII : 0.0; L.aHeII = recomb ? rt.aHeII : 0.0; L.aHeIII = recomb ? rt.aHeIII : 0.0;
  L.bHI = coll ? rt.bHI : 0.0; L.bHeI = coll ? rt.bHeI : 0.0; L.bHeII = coll ? rt.bHeII : 0.0;
  L.d = rate_slopes(tfn, rt);
  const double xHI = s[4 * kB], xHII = s[4 * kB + 1], yI = s[4 * kB + 2], yII = s[4 * kB + 3],
               yIII = s[4 * kB + 4];
  const double ns0 = nH * xHI, ns1 = nHe * yI, ns2 = nHe * yII;
  double Gm0 = 0, Gm1 = 0, Gm2 = 0;
#pragma unroll
  for (int b = 0; b < kB; ++b) {
    L.kap[b] = P.sigma[b][0] * ns0 + P.sigma[b][1] * ns1 + P.sigma[b][2] * ns2;
    L.iden[b] = div_nr(1.0, 1.0 + c * dt * L.kap[b]);
    L.Nbar[b] = s[b] * L.iden[b];
    Gm0 += c * P.sigma[b][0] * L.Nbar[b];
    Gm1 += c * P.sigma[b][1] * L.Nbar[b];
    Gm2 += c * P.sigma[b][2] * L.Nbar[b];
    L.is[b] = s[b] > 0 ? div_nr(1.0, s[b]) : 0.0;
  }
  L.Gm0 = Gm0; L.Gm1 = Gm1; L.Gm2 = Gm2;
  const double ne0 = nH * xHII + nHe * (yII + 2.0 * yIII);
  const double aH = dt * (Gm0 + L.bHI * ne0), bH = dt * L.aHII * ne0;
  const double iD1 = div_nr(1.0, 1.0 + aH + bH);
  const double xHI1 = (xHI * (1.0 + bH) + bH * xHII) * iD1;
  const double xHII1 = (xHII * (1.0 + aH) + aH * xHI) * iD1;
  const double ne1 = nH * xHII1 + nHe * (yII + 2.0 * yIII);
  const double A = dt * (Gm1 + L.bHeI * ne1), Bb = dt * L.aHeII * ne1, Cc = dt * (Gm2 + L.bHeII * ne1),
               Dd = dt * L.aHeIII * ne1;
  const double iA = div_nr(1.0, 1.0 + A), iD = div_nr(1.0, 1.0 + Dd);
  const double num = yII + A * yI * iA + Dd * yIII * iD;
  const double idn = div_nr(1.0, 1.0 + Bb * iA + Cc * iD);
  const double yII1 = num * idn;
  const double yI1 = (yI + Bb * yII1) * iA;
  const double yIII1 = (yIII + Cc * yII1) * iD;
  L.ne0 = ne0; L.aH = aH; L.bH = bH; L.iD1 = iD1; L.xHI1 = xHI1; L.xHII1 = xHII1; L.ne1 = ne1;
  L.A = A; L.Bb = Bb; L.Cc = Cc; L.Dd = Dd; L.iA = iA; L.iD = iD; L.idn = idn;
  L.yII1 = yII1; L.yI1 = yI1; L.yIII1 = yIII1;
  const double m0 = nH * xHI1, m1 = nHe * yI1, m2 = nHe * yII1;
  L.m0 = m0; L.m1 = m1; L.m2 = m2;
  // thermal energy (mode 2): e0 = 3/2 k n_tot0 T, e1 = e0 + heat - dt Lambda,
  // T1 = e1 / (3/2 k n_tot1)
  const bool thermal = P.mode == 2, cool = P.flags & 4, heat = P.flags & 8;
  double e0 = 0.0, e1 = 0.0;
  L.ntot0 = L.lamc = L.ntot1 = L.intot1 = 0.0;
  L.T1 = T;
  if (thermal) {
    const double nsp[5] = {nH * xHI, nH * xHII, nHe * yI, nHe * yII, nHe * yIII};
    L.ntot0 = nH * (1.0 + yhe) + ne0;
    e0 = 1.5 * kBoltzmann * L.ntot0 * T;
    if (cool) {
      L.cc = cooling_coef(tfn);
      L.lamc = ne0 * (L.cc.k[0] * nsp[0] + L.cc.k[1] * nsp[1] + L.cc.k[2] * nsp[2] + L.cc.k[3] * nsp[3] +
                      L.cc.k[4] * nsp[4]);
    }
    double heat_e = 0.0;
    if (heat)
#pragma unroll
      for (int b = 0; b < kB; ++b)
        heat_e += c * dt * L.Nbar[b] * (P.eps[b][0] * P.sigma[b][0] * m0 + P.eps[b][1] * P.sigma[b][1] * m1 +
                                        P.eps[b][2] * P.sigma[b][2] * m2);
    e1 = e0 + heat_e - dt * L.lamc;
    L.ntot1 = nH * (1.0 + yhe) + nH * xHII1 + nHe * (yII1 + 2.0 * yIII1);
    L.T1 = div_nr(e1, 1.5 * kBoltzmann * L.ntot1);
    L.intot1 = div_nr(1.0, L.ntot1);
  }
  // the largest term of the substep measure and its slope's factors
  L.f_sg = L.f_imm = L.f_span = L.f_sgn = 0.0;
  L.f_kb = -1;
  if (!measure) return;
  const double in_x[5] = {xHI, xHII, yI, yII, yIII};
  const double out_x[5] = {xHI1, xHII1, yI1, yII1, yIII1};
  const int nk = yhe > 0 ? 5 : 2;
  double best = -1.0;
  int kb = -1;
  if (thermal) {
    best = rel_change(e0, e1, 0.0);
    kb = 5;
  }
#pragma unroll
  for (int k = 0; k < 5; ++k) {
    if (k < nk) {
      const double r = rel_change(in_x[k], out_x[k], P.x_floor);
      if (r > best) { best = r; kb = k; }
    }
  }
  if (best > 0 && kb == 5) {
    const double imm = div_nr(1.0, fabs(e0));
    L.f_kb = 5;
    L.f_imm = imm;
    L.f_sg = e1 > e0 ? 1.0 : -1.0;
    L.f_span = fabs(e1 - e0) * imm * imm;
    L.f_sgn = e0 > 0 ? 1.0 : -1.0;
  } else if (best > 0) {
    double av = 0.0, bo = 0.0;
#pragma unroll
    for (int k = 0; k < 5; ++k)
      if (k == kb) { av = in_x[k]; bo = out_x[k]; }
    const double imm = div_nr(1.0, fabs(av) > P.x_floor ? fabs(av) : P.x_floor);
    L.f_kb = kb;
    L.f_imm = imm;
    L.f_sg = bo > av ? 1.0 : -1.0;
    L.f_span = fabs(bo - av) * imm * imm;
    L.f_sgn = fabs(av) > P.x_floor ? (av > 0 ? 1.0 : -1.0) : 0.0;
  }
}

// lt == nullptr: the output state carries no cotangent (a rejected
// attempt, whose result is discarded); only lf does.
template <int kB>
__device__ __forceinline__ void attempt_back(const ChemParams& P, double nH, double dt, const double* s,
                                             const AttemptLin& L, const double* lt, double lf, double* ls,
                                             double& ldt, double& lnH) {
  const double c = P.c_red, yhe = P.y_he, nHe = yhe * nH;
  const bool recomb = P.flags & 1, coll = P.flags & 2;
  const double T = s[4 * kB + 5];
  const double xHI = s[4 * kB], xHII = s[4 * kB + 1], yI = s[4 * kB + 2], yII = s[4 * kB + 3],
               yIII = s[4 * kB + 4];
  const double ne0 = L.ne0, aH = L.aH, bH = L.bH, iD1 = L.iD1, xHI1 = L.xHI1, xHII1 = L.xHII1, ne1 = L.ne1;
  const double A = L.A, Bb = L.Bb, Cc = L.Cc, Dd = L.Dd, iA = L.iA, iD = L.iD, idn = L.idn;
  const double yII1 = L.yII1, yI1 = L.yI1, yIII1 = L.yIII1, m0 = L.m0, m1 = L.m1, m2 = L.m2;
  const bool thermal = P.mode == 2, cool = P.flags & 4, heat = P.flags & 8;

  double lx1[5], lxin[5] = {0, 0, 0, 0, 0};
#pragma unroll
  for (int q = 0; q < 5; ++q) lx1[q] = lt ? lt[4 * kB + q] : 0.0;
  double lT0 = 0.0, le0 = 0.0, le1 = 0.0, lne0e = 0.0;
  const double lT1 = lt ? lt[4 * kB + 5] : 0.0;
  if (thermal) {
    le1 = lT1 * (1.0 / (1.5 * kBoltzmann)) * L.intot1;
    const double lnt1 = -lT1 * L.T1 * L.intot1;
    lx1[1] += lnt1 * nH;
    lx1[3] += lnt1 * nHe;
    lx1[4] += lnt1 * 2.0 * nHe;
    lnH += lnt1 * ((1.0 + yhe) + xHII1 + yhe * (yII1 + 2.0 * yIII1));
  } else {
    lT0 += lT1;
  }
  if (lf != 0.0 && L.f_kb >= 0) {
    if (L.f_kb == 5) {
      le1 += lf * L.f_sg * L.f_imm;
      le0 += -lf * L.f_sg * L.f_imm - lf * L.f_span * L.f_sgn;
    } else {
#pragma unroll
      for (int k = 0; k < 5; ++k)
        if (k == L.f_kb) {
          lx1[k] += lf * L.f_sg * L.f_imm;
          lxin[k] += -lf * L.f_sg * L.f_imm - lf * L.f_span * L.f_sgn;
        }
    }
  }
  double lNbar[kMaxBins] = {0, 0, 0}, lm0 = 0, lm1 = 0, lm2 = 0;
  if (thermal) {
    le0 += le1;
    ldt -= le1 * L.lamc;
    if (heat)
#pragma unroll
      for (int b = 0; b < kB; ++b) {
        const double e_0 = P.eps[b][0] * P.sigma[b][0], e_1 = P.eps[b][1] * P.sigma[b][1],
                     e_2 = P.eps[b][2] * P.sigma[b][2];
        const double ea = e_0 * m0 + e_1 * m1 + e_2 * m2;
        lNbar[b] += le1 * c * dt * ea;
        ldt += le1 * c * L.Nbar[b] * ea;
        const double w = le1 * c * dt * L.Nbar[b];
        lm0 += w * e_0;
        lm1 += w * e_1;
        lm2 += w * e_2;
      }
    if (cool) {
      const double nsp[5] = {nH * xHI, nH * xHII, nHe * yI, nHe * yII, nHe * yIII};
      const double ll = -le1 * dt;
      double dLdT = 0.0;
#pragma unroll
      for (int q = 0; q < 5; ++q) dLdT += L.cc.dk[q] * nsp[q];
      lT0 += ll * ne0 * dLdT;
      // Lambda is linear in n_e0: its slope needs no division (n_e0 = 0 in a
      // neutral cell)
      double kn = 0.0;
#pragma unroll
      for (int q = 0; q < 5; ++q) kn += L.cc.k[q] * nsp[q];
      lne0e += ll * kn;
      lxin[0] += ll * ne0 * L.cc.k[0] * nH;
      lxin[1] += ll * ne0 * L.cc.k[1] * nH;
      lxin[2] += ll * ne0 * L.cc.k[2] * nHe;
      lxin[3] += ll * ne0 * L.cc.k[3] * nHe;
      lxin[4] += ll * ne0 * L.cc.k[4] * nHe;
      lnH += ll * ne0 *
             (L.cc.k[0] * xHI + L.cc.k[1] * xHII + yhe * (L.cc.k[2] * yI + L.cc.k[3] * yII + L.cc.k[4] * yIII));
    }
    lT0 += le0 * 1.5 * kBoltzmann * L.ntot0;
    const double lnt0 = le0 * 1.5 * kBoltzmann * T;
    lne0e += lnt0;
    lnH += lnt0 * (1.0 + yhe);
  }
#pragma unroll
  for (int b = 0; b < kB; ++b) {
    const double sm = P.sigma[b][0] * m0 + P.sigma[b][1] * m1 + P.sigma[b][2] * m2;
    const double rem = c * dt * L.Nbar[b] * sm;
    double N1 = s[b] - rem;
    const bool clamped = N1 < 0;
    if (clamped) N1 = 0;
    const double is = L.is[b];
    const double scale = N1 * is;
    double lscale = 0.0;
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      const double lf3 = lt ? lt[kB + 3 * b + k] : 0.0;
      ls[kB + 3 * b + k] += lf3 * scale;
      lscale += lf3 * s[kB + 3 * b + k];
    }
    double lN1 = lt ? lt[b] : 0.0;
    if (s[b] > 0) {
      lN1 += lscale * is;
      ls[b] -= lscale * scale * is;
    }
    if (!clamped) {
      ls[b] += lN1;
      const double lrem = -lN1;
      lNbar[b] += lrem * c * dt * sm;
      ldt += lrem * c * L.Nbar[b] * sm;
      lm0 += lrem * c * dt * L.Nbar[b] * P.sigma[b][0];
      lm1 += lrem * c * dt * L.Nbar[b] * P.sigma[b][1];
      lm2 += lrem * c * dt * L.Nbar[b] * P.sigma[b][2];
    }
  }
  lx1[0] += lm0 * nH;
  lx1[2] += lm1 * nHe;
  lx1[3] += lm2 * nHe;
  lnH += lm0 * xHI1 + lm1 * yhe * yI1 + lm2 * yhe * yII1;
  double lyII1 = lx1[3];
  const double lyI1 = lx1[2], lyIII1 = lx1[4];
  double lCc = 0, lBb = 0, lA = 0, lDd = 0, lopA = 0, lopD = 0;
  lxin[4] += lyIII1 * iD;
  lCc += lyIII1 * yII1 * iD;
  lyII1 += lyIII1 * Cc * iD;
  lopD -= lyIII1 * yIII1 * iD;
  lxin[2] += lyI1 * iA;
  lBb += lyI1 * yII1 * iA;
  lyII1 += lyI1 * Bb * iA;
  lopA -= lyI1 * yI1 * iA;
  const double lnum = lyII1 * idn, ldn = -lyII1 * yII1 * idn;
  lBb += ldn * iA;
  lopA -= ldn * Bb * (iA * iA);
  lCc += ldn * iD;
  lopD -= ldn * Cc * (iD * iD);
  lxin[3] += lnum;
  lA += lnum * yI * iA;
  lxin[2] += lnum * A * iA;
  lopA -= lnum * A * yI * (iA * iA);
  lDd += lnum * yIII * iD;
  lxin[4] += lnum * Dd * iD;
  lopD -= lnum * Dd * yIII * (iD * iD);
  lA += lopA;
  lDd += lopD;
  ldt += lA * (L.Gm1 + L.bHeI * ne1) + lBb * L.aHeII * ne1 + lCc * (L.Gm2 + L.bHeII * ne1) + lDd * L.aHeIII * ne1;
  double lG0 = 0.0;
  const double lG1 = lA * dt, lG2 = lCc * dt;
  const double lne1 = lA * dt * L.bHeI + lBb * dt * L.aHeII + lCc * dt * L.bHeII + lDd * dt * L.aHeIII;
  const double lxHII1 = lx1[1] + lne1 * nH;
  const double lxHI1 = lx1[0];
  lnH += lne1 * (xHII1 + yhe * (yII + 2.0 * yIII));
  lxin[3] += lne1 * nHe;
  lxin[4] += lne1 * 2.0 * nHe;
  const double lD1 = -(lxHI1 * xHI1 + lxHII1 * xHII1) * iD1;
  lxin[1] += lxHII1 * (1.0 + aH) * iD1 + lxHI1 * bH * iD1;
  lxin[0] += lxHII1 * aH * iD1 + lxHI1 * (1.0 + bH) * iD1;
  const double laH = lxHII1 * (xHII + xHI) * iD1 + lD1;
  const double lbH = lxHI1 * (xHI + xHII) * iD1 + lD1;
  ldt += laH * (L.Gm0 + L.bHI * ne0) + lbH * L.aHII * ne0;
  lG0 += laH * dt;
  const double lne0 = laH * dt * L.bHI + lbH * dt * L.aHII;
  lxin[1] += lne0 * nH;
  lnH += lne0 * (xHII + yhe * (yII + 2.0 * yIII));
  lxin[3] += lne0 * nHe;
  lxin[4] += lne0 * 2.0 * nHe;
  if (coll) lT0 += laH * dt * L.d.bHI * ne0 + lA * dt * L.d.bHeI * ne1 + lCc * dt * L.d.bHeII * ne1;
  if (recomb) lT0 += lbH * dt * L.d.aHII * ne0 + lBb * dt * L.d.aHeII * ne1 + lDd * dt * L.d.aHeIII * ne1;
  lxin[1] += lne0e * nH;
  lxin[3] += lne0e * nHe;
  lxin[4] += lne0e * 2.0 * nHe;
  lnH += lne0e * (xHII + yhe * (yII + 2.0 * yIII));
  double lns0 = 0, lns1 = 0, lns2 = 0;
#pragma unroll
  for (int b = 0; b < kB; ++b) {
    lNbar[b] += c * (P.sigma[b][0] * lG0 + P.sigma[b][1] * lG1 + P.sigma[b][2] * lG2);
    ls[b] += lNbar[b] * L.iden[b];
    const double lden = -lNbar[b] * L.Nbar[b] * L.iden[b];
    ldt += lden * c * L.kap[b];
    const double lkap = lden * c * dt;
    lns0 += lkap * P.sigma[b][0];
    lns1 += lkap * P.sigma[b][1];
    lns2 += lkap * P.sigma[b][2];
  }
  lxin[0] += lns0 * nH;
  lxin[2] += lns1 * nHe;
  lxin[3] += lns2 * nHe;
  lnH += lns0 * xHI + lns1 * yhe * yI + lns2 * yhe * yII;
#pragma unroll
  for (int q = 0; q < 5; ++q) ls[4 * kB + q] += lxin[q];
  ls[4 * kB + 5] += lT0;
}

struct ChemAdjArgs {
  int C, B;
  const d4* rad;          // recorded radiation entering the subcycle's chemistry (before the source term)
  const double* x5;       // recorded abundances entering the chemistry
  const double* T;
  const double* nH;
  const double* vol;
  const ChemRec* rec;     // the segment's tape
  const int32_t* last;    // C: this subcycle's last record of each cell, -1 for one accepted attempt
  const AttemptLin* lin;  // attempt_lin of this subcycle's records [rec_lo, rec_hi)
  long long rec_lo, rec_hi;
  d4* lam_rad;            // in/out: cotangent of the cell's radiation
  double* lam_x5;         // in/out
  double* lam_T;          // in/out
  double* lam_nH;         // accumulated
  double* lam_S;          // [B][C] accumulated dL/dS
  int* status;
  const int32_t* src_idx; // C: index into src_rate or -1
  const double* src_rate; // [n][B] photons/s
  double dt;              // subcycle length
  double lu3;
  int do_inject, do_chem;
};

// The state entering the chemistry, packed: the recorded one plus the
// source term, exactly as in k_chem64_first.
template <int kB>
__device__ __forceinline__ void load_cell(const ChemAdjArgs& a, int i, double* s) {
  const size_t C = a.C;
#pragma unroll
  for (int b = 0; b < kB; ++b) {
    const d4 v = a.rad[(size_t)i * kB + b];
    s[b] = v.x; s[kB + 3 * b] = v.y; s[kB + 3 * b + 1] = v.z; s[kB + 3 * b + 2] = v.w;
  }
  s[4 * kB] = a.x5[i]; s[4 * kB + 1] = a.x5[C + i]; s[4 * kB + 2] = a.x5[2 * C + i];
  s[4 * kB + 3] = a.x5[3 * C + i]; s[4 * kB + 4] = a.x5[4 * C + i]; s[4 * kB + 5] = a.T[i];
  if (a.do_inject) {
    const int si = a.src_idx[i];
    if (si >= 0) {
      const double vcm3 = a.vol[i] * a.lu3;
#pragma unroll
      for (int b = 0; b < kB; ++b) s[b] += (a.src_rate[(size_t)si * kB + b] * a.dt) / vcm3;
    }
  }
}

// attempt_lin of every recorded attempt of one subcycle, one thread per
// record; the reverse chain then runs attempt_back only.
template <int kB>
__global__ void __launch_bounds__(128) k_chem_lin(ChemAdjArgs a, ChemParams P, AttemptLin* __restrict__ lin) {
  const long long j = a.rec_lo + (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (j >= a.rec_hi) return;
  const ChemRec& r = a.rec[j];
  AttemptLin L;
  attempt_lin<kB>(P, a.nH[r.cell], r.dt, r.s, L, true);
  lin[j - a.rec_lo] = L;
}

// Reverse over the attempts of one cell, last to first, then the source
// term.  Each attempt's cotangent flows to its entering state and, through
// the controller, to its length, which the previous attempt's measure set.
// A cell with one attempt (accepted, over the whole subcycle) has no record:
// its entering state is the recorded one, and no later attempt's length
// depends on its measure.
template <int kB>
__global__ void __launch_bounds__(128) k_chem_adj(ChemAdjArgs a, ChemParams P) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= a.C) return;
  constexpr int nv = 4 * kB + 6;
  const size_t C = a.C;
  double lt[nv], ls[nv];
#pragma unroll
  for (int b = 0; b < kB; ++b) {
    const d4 v = a.lam_rad[(size_t)i * kB + b];
    lt[b] = v.x; lt[kB + 3 * b] = v.y; lt[kB + 3 * b + 1] = v.z; lt[kB + 3 * b + 2] = v.w;
  }
#pragma unroll
  for (int q = 0; q < 5; ++q) lt[4 * kB + q] = a.lam_x5[q * C + i];
  lt[4 * kB + 5] = a.lam_T[i];
  const double nH = a.nH[i];
  double lnH = 0.0;
  int idx = a.do_chem ? a.last[i] : -1;
  if (a.do_chem && idx < 0) {
    double sv[nv];
    load_cell<kB>(a, i, sv);
    AttemptLin L;
    attempt_lin<kB>(P, nH, a.dt, sv, L, false);
#pragma unroll
    for (int q = 0; q < nv; ++q) ls[q] = 0.0;
    double cdt = 0.0;
    attempt_back<kB>(P, nH, a.dt, sv, L, lt, 0.0, ls, cdt, lnH);
#pragma unroll
    for (int q = 0; q < nv; ++q) lt[q] = ls[q];
  }
  double ldt = 0.0, lrem = 0.0;
  while (idx >= 0) {
    if (idx < a.rec_lo || idx >= a.rec_hi) {   // not reached: a cell's records lie in its subcycle's range
      atomicOr(a.status, kStNonFinite);
      break;
    }
    const ChemRec& r = a.rec[idx];
    const AttemptLin& L = a.lin[idx - a.rec_lo];
#pragma unroll
    for (int q = 0; q < nv; ++q) ls[q] = 0.0;
    double cdt = 0.0;
    if (r.flags & kRecAccepted) {
      const bool ratio = r.flags & kRecRatio;
      const double grow = ratio ? P.f_s / r.f : 2.0;
      double ldtg = 0.0;
      if (r.flags & kRecClipped) lrem += ldt;
      else ldtg = ldt;
      double ldtk = ldtg * grow;
      const double lg = ldtg * r.dt;
      const double lf = ratio ? -lg * P.f_s / (r.f * r.f) : 0.0;
      ldtk -= lrem;
      attempt_back<kB>(P, nH, r.dt, r.s, L, lt, lf, ls, cdt, lnH);
#pragma unroll
      for (int q = 0; q < nv; ++q) lt[q] = ls[q];
      ldt = ldtk + cdt;
    } else {
      const double ldtk = ldt * P.f_s / r.f;
      const double lf = -ldt * r.dt * P.f_s / (r.f * r.f);
      attempt_back<kB>(P, nH, r.dt, r.s, L, nullptr, lf, ls, cdt, lnH);
#pragma unroll
      for (int q = 0; q < nv; ++q) lt[q] += ls[q];
      ldt = ldtk + cdt;
    }
    idx = r.prev;
  }
#pragma unroll
  for (int b = 0; b < kB; ++b) {
    a.lam_rad[(size_t)i * kB + b] = make_d4(lt[b], lt[kB + 3 * b], lt[kB + 3 * b + 1], lt[kB + 3 * b + 2]);
    // source term N_b += S_b dt / (V lu^3)
    a.lam_S[(size_t)b * C + i] += lt[b] * a.dt / (a.vol[i] * a.lu3);
  }
#pragma unroll
  for (int q = 0; q < 5; ++q) a.lam_x5[q * C + i] = lt[4 * kB + q];
  a.lam_T[i] = lt[4 * kB + 5];
  a.lam_nH[i] += lnH;
}

}  // namespace m1rt

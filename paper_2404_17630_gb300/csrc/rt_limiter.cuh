// FP64 slope-limiter arithmetic shared by the gradient kernels: extremes as bit
// patterns on the integer pipe (the FP64 unit is what bounds those kernels) and
// the limiter's search for the faces that attain them.
#pragma once
#include "rt_common.cuh"

namespace m1rt {

// Running extremes of FP64 differences on the integer pipe.  The bits of a
// double x >= +0 order like x as signed 64-bit integers and those of x < 0
// are negative, so max(bits, bits(d)) keeps the largest d >= 0 (start: +0);
// the magnitude bits of d < 0 (0 for d >= 0) track the most negative d.
__device__ __forceinline__ long long max_bits_pos(long long b, double d) {
  const long long v = __double_as_longlong(d);
  return v > b ? v : b;
}
__device__ __forceinline__ long long max_bits_neg(long long m, double d) {
  const long long v = __double_as_longlong(d);
  const long long mag = (v & 0x7FFFFFFFFFFFFFFFLL) & (v >> 63);
  return mag > m ? mag : m;
}
// -magnitude from max_bits_neg, +0 where nothing was negative
__device__ __forceinline__ double neg_from_bits(long long m) {
  return __longlong_as_double(m ? (m | (long long)0x8000000000000000ULL) : 0LL);
}

// FP64 comparisons on the integer pipe, exact for the values they are used
// on: a > b for a, b >= +0 (the bit patterns order like the values), and
// x < 0 (negative, not -0, not NaN).
__device__ __forceinline__ bool gt_nonneg(double a, double b) {
  return __double_as_longlong(a) > __double_as_longlong(b);
}
__device__ __forceinline__ bool lt_zero(double x) {
  const long long b = __double_as_longlong(x), m = b & 0x7FFFFFFFFFFFFFFFLL;
  return b < 0 && m != 0 && m <= 0x7FF0000000000000LL;
}

// g scaled by a power of two so that its largest component lies in [1, 2),
// cut to FP32 on the integer pipe (relative error below 2^-23; components
// 2^-126 of the largest become zero).  false where the largest lies outside
// 2^-400 .. 2^400 (g = 0 or not finite among them): the squares of the
// regularisation test stay in the normal range only inside.
__device__ __forceinline__ bool scaled_f32(const double g[3], float o[3]) {
  unsigned hi[3], top = 0;
#pragma unroll
  for (int d = 0; d < 3; ++d) {
    hi[d] = (unsigned)__double2hiint(g[d]);
    const unsigned e = hi[d] & 0x7FF00000u;
    top = e > top ? e : top;
  }
#pragma unroll
  for (int d = 0; d < 3; ++d) {
    const int e = (int)((hi[d] & 0x7FF00000u) >> 20) - (int)(top >> 20) + 127;
    const unsigned m = ((hi[d] & 0xFFFFFu) << 3) | ((unsigned)__double2loint(g[d]) >> 29);
    o[d] = __uint_as_float((hi[d] & 0x80000000u) | (e > 0 ? ((unsigned)e << 23) | m : 0u));
  }
  return (top >> 20) - 623u < 800u;
}

// Limiter extremes of one (cell, bin) in FP64: dpos = max(0, max g.x_f) and
// dneg = min(0, min g.x_f) over the faces k0..k1-1 that pass the
// regularisation test (g.x_f)^2 > eps2 |g|^2 |x_f|^2 (X: the largest x.w =
// |x_f|^2), kept as bit patterns (integer compares; the FP64 pipe is the
// kernel's bound).  xf: the offsets in FP32, in any unit that is the same for the
// cell's faces, xm: the largest |x_f| in it (NaN: no search).  First a search in
// FP32 for the face that attains each extreme: |g| scaled to below 2 per
// component, the FP32 product g . x_f is within 6 2^-24 2 (|x| + |y| + |z|) <=
// 1.3e-6 |x_f| of the exact one (both operands rounded, three roundings of the
// sum), so a leader that is 2.6e-6 of the cell's largest |x_f| ahead of every
// other face and of zero is the FP64 leader, and its FP64 product is the
// extreme: eight FP64 products per (cell, bin) instead of four per face (with
// the matrix folded into the weights: 0.85 -> 0.52 ms per launch at 250,047
// cells, 142 -> 82 us at 262,144 cells of six faces and one bin).  A leader
// beyond the test's bound for the largest |x_f|, by the same margin, also passes
// its own test, and nothing more is to be tested: rounding is monotone.  Where a
// lead is smaller (faces that tie by symmetry; a leader within the band of zero)
// every face's product is formed in FP64 and, where an extreme does not clear the
// bound, tested.  A component without gradient has no extremes.  at[2q],
// at[2q + 1]: the first face that attains dpos[q], dneg[q].
__device__ __forceinline__ void lim_extremes(const d4* __restrict__ xs, const float4* __restrict__ xf, int k0, int k1,
                                             const double gr[4][3], double eps2, double X, float xm,
                                             double dpos[4], double dneg[4], int at[8]) {
  float gf[4][3], m1[8], m2[8];
  bool flat[4], sure = true;
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    flat[q] = ((__double_as_longlong(gr[q][0]) | __double_as_longlong(gr[q][1]) | __double_as_longlong(gr[q][2])) &
               0x7FFFFFFFFFFFFFFFLL) == 0;
    const bool ok = scaled_f32(gr[q], gf[q]);
    sure = sure && (ok || flat[q]);
    m1[2 * q] = m1[2 * q + 1] = m2[2 * q] = m2[2 * q + 1] = 0.0f;
    at[2 * q] = at[2 * q + 1] = k0;
  }
#pragma unroll 2
  for (int k = k0; k < k1; ++k) {
    const float4 x = xf[k];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const float v = gf[q][0] * x.x + gf[q][1] * x.y + gf[q][2] * x.z;
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const float u = h ? -v : v;
        m2[2 * q + h] = fmaxf(m2[2 * q + h], fminf(m1[2 * q + h], u));
        at[2 * q + h] = u > m1[2 * q + h] ? k : at[2 * q + h];
        m1[2 * q + h] = fmaxf(m1[2 * q + h], u);
      }
    }
  }
  const float ex = 1.0001f * sqrtf((float)eps2) * xm, lead = 2.6e-6f * xm;
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    const float clear = fmaf(ex, sqrtf(gf[q][0] * gf[q][0] + gf[q][1] * gf[q][1] + gf[q][2] * gf[q][2]), lead);
#pragma unroll
    for (int h = 0; h < 2; ++h)
      sure = sure && (flat[q] || (m1[2 * q + h] - m2[2 * q + h] > lead && m1[2 * q + h] > clear));
  }
  long long bpos[4], bneg[4];
#pragma unroll
  for (int q = 0; q < 4; ++q) bpos[q] = bneg[q] = 0;
  if (sure) {
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      if (flat[q]) continue;
      const d4 a = xs[at[2 * q]], c = xs[at[2 * q + 1]];
      bpos[q] = max_bits_pos(0, gr[q][0] * a.x + gr[q][1] * a.y + gr[q][2] * a.z);
      bneg[q] = max_bits_neg(0, gr[q][0] * c.x + gr[q][1] * c.y + gr[q][2] * c.z);
    }
  } else {
    bool exact = true;
    double thr[4];
#pragma unroll 1
    for (int k = k0; k < k1; ++k) {
      const d4 x = ld4<double>(xs + k);
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const double dphi = gr[q][0] * x.x + gr[q][1] * x.y + gr[q][2] * x.z;
        const long long p = max_bits_pos(bpos[q], dphi), n = max_bits_neg(bneg[q], dphi);
        at[2 * q] = p != bpos[q] ? k : at[2 * q];
        at[2 * q + 1] = n != bneg[q] ? k : at[2 * q + 1];
        bpos[q] = p;
        bneg[q] = n;
      }
    }
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      thr[q] = eps2 * (gr[q][0] * gr[q][0] + gr[q][1] * gr[q][1] + gr[q][2] * gr[q][2]);
      const long long t = __double_as_longlong(thr[q] * X);
      const double p = __longlong_as_double(bpos[q]), n = neg_from_bits(bneg[q]);
      exact = exact && (bpos[q] == 0 || __double_as_longlong(p * p) > t) &&
              (bneg[q] == 0 || __double_as_longlong(n * n) > t);
    }
    if (!exact) {
#pragma unroll
      for (int q = 0; q < 4; ++q) bpos[q] = bneg[q] = 0;
#pragma unroll 1
      for (int k = k0; k < k1; ++k) {
        const d4 x = ld4<double>(xs + k);
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          const double dphi = gr[q][0] * x.x + gr[q][1] * x.y + gr[q][2] * x.z;
          if (__double_as_longlong(dphi * dphi) > __double_as_longlong(thr[q] * x.w)) {
            const long long p = max_bits_pos(bpos[q], dphi), n = max_bits_neg(bneg[q], dphi);
            at[2 * q] = p != bpos[q] ? k : at[2 * q];
            at[2 * q + 1] = n != bneg[q] ? k : at[2 * q + 1];
            bpos[q] = p;
            bneg[q] = n;
          }
        }
      }
    }
  }
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    dpos[q] = __longlong_as_double(bpos[q]);
    dneg[q] = neg_from_bits(bneg[q]);
  }
}

// The limiter factor from the extremes: min(1, up / dpos, dn / dneg) with up, dn
// the largest and most negative difference to a neighbour.  The quotients are
// formed only where they are below 1 (tested on the integer pipe).
__device__ __forceinline__ bool limits_pos(double up, double dpos) { return gt_nonneg(dpos, up); }
__device__ __forceinline__ bool limits_neg(double dn, double dneg) { return gt_nonneg(-dneg, -dn); }

}  // namespace m1rt

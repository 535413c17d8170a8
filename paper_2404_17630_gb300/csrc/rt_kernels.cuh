// Kernels of the M1 RT subcycle.
//
//   k_mesh_*, k_scan_*  once per mesh: checks and per-cell face lists
//   k_geometry_*   once per mesh (Sec. 2.3.2: the least-squares matrix depends
//                  only on geometry and is inverted once)
//   k_grad<R>      least-squares gradients + slope limiter, one thread per
//                  (cell, bin)  (Sec. 2.3.2, 4.1.2)
//   k_flux<R>      face reconstruction, M1 closure, Lax-Friedrichs flux, one
//                  thread per (face, bin)  (Sec. 2.3.3, 4.1.3)
//   k_gather<R>    per (cell, bin): deterministic CSR gather of the stored
//                  face fluxes, FP64 update (Sec. 4.1.3)
//   k_chem_first,  source injection and thermochemistry (Eq. E, Sec. 2.3.1,
//   k_chem_rest    4.1.1) in two passes, mixed precision: the first attempt of
//                  every cell, then the rejected cells
//   k_chem64_*     the same in FP64
//
// R is the precision of the transport sweep (double, or float in the mixed
// mode of Sec. 6.2); the master state, the gather sums, the volume divisions
// and the chemistry are FP64 in both.
#pragma once
#include "rt_chem.cuh"
#include "rt_chem_coop.cuh"
#include "rt_limiter.cuh"

namespace m1rt {

// ---------------------------------------------------------------------------
// per-cell face lists, once per mesh
// ---------------------------------------------------------------------------
//
// A moving mesh comes anew with every step, so what a mesh costs counts: the
// checks, the degrees, their prefix sums and the lists are all built on the
// device (the host's passes over faces and cells took 4 ms of the 6.6 ms of a
// 64,000-cell mesh).

// What the checks found: the first bad face, volume and cell without faces
// (INT_MAX: none), the smallest volume's bits, the largest degree, the records
// of the largest block of cells.
struct MeshCheck {
  int bad_face, bad_volume, no_faces, max_deg, cap;
  int pad;
  long long min_volume;
};
constexpr int kNoIndex = 0x7fffffff;

__global__ void k_mesh_init(MeshCheck* r, double* x5, double* T, int32_t* deg, int C) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i == 0) *r = MeshCheck{kNoIndex, kNoIndex, kNoIndex, 0, 0, 0, 0x7FF0000000000000LL};
  if (i >= C) return;
  // neutral gas at 1e4 K
  x5[i] = x5[2 * (size_t)C + i] = 1.0;
  x5[(size_t)C + i] = x5[3 * (size_t)C + i] = x5[4 * (size_t)C + i] = 0.0;
  T[i] = 1e4;
  deg[i] = 0;
}

// Both ids of every face, checked; the cells' degrees.
__global__ void k_mesh_faces(int F, int C, const int32_t* __restrict__ left, const int32_t* __restrict__ right,
                             int2* __restrict__ lr, int32_t* __restrict__ deg, MeshCheck* r) {
  const int f = blockIdx.x * blockDim.x + threadIdx.x;
  if (f >= F) return;
  const int a = left[f], b = right[f];
  lr[f] = make_int2(a, b);
  if (a < 0 || a >= C || b < 0 || b >= C || a == b) {
    atomicMin(&r->bad_face, f);
    return;
  }
  atomicAdd(deg + a, 1);
  atomicAdd(deg + b, 1);
}

__global__ void k_mesh_cells(int C, const double* __restrict__ vol, const int32_t* __restrict__ deg, MeshCheck* r) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  long long v = 0x7FF0000000000000LL;
  int d = 0;
  if (i < C) {
    d = deg[i];
    if (!(vol[i] > 0.0) || !isfinite(vol[i])) atomicMin(&r->bad_volume, i);
    else v = __double_as_longlong(vol[i]);   // the bits of positive values order like them
    if (d == 0) atomicMin(&r->no_faces, i);
  }
#pragma unroll
  for (int m = 16; m > 0; m >>= 1) {
    const long long o = __shfl_xor_sync(0xffffffffu, v, m);
    v = o < v ? o : v;
  }
  d = __reduce_max_sync(0xffffffffu, d);
  if ((threadIdx.x & 31) == 0) {
    atomicMin(&r->min_volume, v);
    atomicMax(&r->max_deg, d);
  }
}

// Exclusive prefix sums in three steps: within blocks of kScan entries, over
// the blocks' sums (one block, kScan at a time), and the sums added.
constexpr int kScan = 1024;
__device__ __forceinline__ int block_scan(int v, int* warp_sums) {   // exclusive, kScan threads
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  int s = v;
#pragma unroll
  for (int d = 1; d < 32; d <<= 1) {
    const int o = __shfl_up_sync(0xffffffffu, s, d);
    if (lane >= d) s += o;
  }
  if (lane == 31) warp_sums[w] = s;
  __syncthreads();
  if (w == 0) {
    int t = warp_sums[lane];
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
      const int o = __shfl_up_sync(0xffffffffu, t, d);
      if (lane >= d) t += o;
    }
    warp_sums[lane] = t;   // inclusive over the warps
  }
  __syncthreads();
  const int r = s - v + (w > 0 ? warp_sums[w - 1] : 0);
  return r;
}
__global__ void __launch_bounds__(kScan) k_scan_blocks(int n, const int32_t* __restrict__ in, int32_t* __restrict__ out,
                                                       int32_t* __restrict__ sums) {
  __shared__ int ws[32];
  const long long i = (long long)blockIdx.x * kScan + threadIdx.x;
  const int v = i < n ? in[i] : 0;
  const int e = block_scan(v, ws);
  if (i < n) out[i] = e;
  if (threadIdx.x == kScan - 1) sums[blockIdx.x] = e + v;
}
// (sums holds n + 1 entries: the last one becomes the total)
__global__ void __launch_bounds__(kScan) k_scan_sums(int n, int32_t* __restrict__ sums) {
  __shared__ int ws[32];
  __shared__ int total;
  if (threadIdx.x == 0) total = 0;
  for (int c = 0; c < n; c += kScan) {
    const int i = c + threadIdx.x;
    const int v = i < n ? sums[i] : 0;
    __syncthreads();   // total of the earlier pieces, ws free again
    const int base = total;
    const int e = block_scan(v, ws);
    if (i < n) sums[i] = base + e;
    __syncthreads();
    if (threadIdx.x == kScan - 1) total = base + e + v;
  }
  __syncthreads();
  if (threadIdx.x == 0) sums[n] = total;
}
// off[i] += the sum of the blocks before; the last entry; next[i] = 0.
__global__ void k_scan_add(int n, int total, const int32_t* __restrict__ sums, int32_t* __restrict__ off,
                           int32_t* __restrict__ next) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i > n) return;
  if (i == n) {
    off[n] = total;
    return;
  }
  off[i] += sums[i / kScan];
  next[i] = 0;
}

// Every face into both its cells' lists, in any order.
__global__ void k_mesh_fill(int F, const int2* __restrict__ lr, const int32_t* __restrict__ off,
                            int32_t* __restrict__ next, int32_t* __restrict__ csr) {
  const int f = blockIdx.x * blockDim.x + threadIdx.x;
  if (f >= F) return;
  const int2 c = lr[f];
  csr[off[c.x] + atomicAdd(next + c.x, 1)] = f << 1;
  csr[off[c.y] + atomicAdd(next + c.y, 1)] = (f << 1) | 1;
}

// Each cell's list into ascending order (insertion for the usual handful of
// faces, a heap for long lists), its neighbours' ids, the records of its block
// of `per` cells.
__global__ void k_mesh_sort(int C, int per, const int32_t* __restrict__ off, int32_t* csr, const int2* __restrict__ lr,
                            int32_t* __restrict__ nbr, MeshCheck* r) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= C) return;
  const int k0 = off[i], n = off[i + 1] - k0;
  int32_t* a = csr + k0;
  if (n <= 64) {
    for (int k = 1; k < n; ++k) {
      const int32_t v = a[k];
      int j = k;
      for (; j > 0 && a[j - 1] > v; --j) a[j] = a[j - 1];
      a[j] = v;
    }
  } else {
    auto sift = [&](int root, int len) {
      const int32_t v = a[root];
      int c;
      while ((c = 2 * root + 1) < len) {
        if (c + 1 < len && a[c + 1] > a[c]) ++c;
        if (a[c] <= v) break;
        a[root] = a[c];
        root = c;
      }
      a[root] = v;
    };
    for (int k = n / 2 - 1; k >= 0; --k) sift(k, n);
    for (int k = n - 1; k > 0; --k) {
      const int32_t v = a[0];
      a[0] = a[k];
      a[k] = v;
      sift(0, k);
    }
  }
  for (int k = 0; k < n; ++k) {
    const int2 c = lr[a[k] >> 1];
    nbr[k0 + k] = (a[k] & 1) ? c.x : c.y;
  }
  if (i % per == 0) atomicMax(&r->cap, off[min(i + per, C)] - k0);
}

// Source k's index to its cell.
__global__ void k_mark_sources(int n, const int32_t* __restrict__ cell, int32_t* __restrict__ idx) {
  const int k = blockIdx.x * blockDim.x + threadIdx.x;
  if (k < n) idx[cell[k]] = k;
}

// ---------------------------------------------------------------------------
// geometry (FP64), once per mesh
// ---------------------------------------------------------------------------

// Per face: (n, A), x_f - s_L, x_f - s_R (minimum image), and w = A d / |d|^2
// with d = s_R - s_L (the face's weight in the right-hand side of the normal
// equation, the same for both of its cells), beside it |d|^2 / A (0 for a face
// without area, whose weight is 0 too).
__global__ void k_geometry_faces(int F, Box box, const int2* __restrict__ lr, const double* __restrict__ cx,
                                 const double* __restrict__ cy, const double* __restrict__ cz,
                                 const double* __restrict__ nx, const double* __restrict__ ny,
                                 const double* __restrict__ nz, const double* __restrict__ fx,
                                 const double* __restrict__ fy, const double* __restrict__ fz,
                                 const double* __restrict__ area, d4* __restrict__ nA, d4* __restrict__ rL,
                                 d4* __restrict__ rR, d4* __restrict__ w) {
  int f = blockIdx.x * blockDim.x + threadIdx.x;
  if (f >= F) return;
  const int2 c = lr[f];
  const double A = area[f];
  nA[f] = make_d4(nx[f], ny[f], nz[f], A);
  const double l0 = cx[c.x], l1 = cy[c.x], l2 = cz[c.x], r0 = cx[c.y], r1 = cy[c.y], r2 = cz[c.y];
  const double x0 = fx[f], x1 = fy[f], x2 = fz[f];
  rL[f] = make_d4(min_image(x0 - l0, box), min_image(x1 - l1, box), min_image(x2 - l2, box), 0.0);
  rR[f] = make_d4(min_image(x0 - r0, box), min_image(x1 - r1, box), min_image(x2 - r2, box), 0.0);
  const double d0 = min_image(r0 - l0, box), d1 = min_image(r1 - l1, box), d2 = min_image(r2 - l2, box);
  const double dd = d0 * d0 + d1 * d1 + d2 * d2;
  const double s = A / dd, q = dd / A;
  w[f] = make_d4(s * d0, s * d1, s * d2, isfinite(q) ? q : 0.0);
}

// Per cell: M = sum_f A n n^T with n = d / |d| towards the neighbour, which is
// (|d|^2 / A) w w^T of the face's weight, and its inverse (symmetric, 6
// entries).  Flags a singular matrix.  The geometry of a mesh of 64,000 cells,
// with the distances and minimum images formed once per face: 345 -> 70 us.
__global__ void k_geometry_cells(int C, const int32_t* __restrict__ off, const int32_t* __restrict__ csr,
                                 const d4* __restrict__ w, double* minv, int* status) {
  int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= C) return;
  double m00 = 0, m01 = 0, m02 = 0, m11 = 0, m12 = 0, m22 = 0;
  for (int k = off[i]; k < off[i + 1]; ++k) {
    const d4 v = w[csr[k] >> 1];
    const double a0 = v.w * v.x, a1 = v.w * v.y, a2 = v.w * v.z;
    m00 = fma(a0, v.x, m00); m01 = fma(a0, v.y, m01); m02 = fma(a0, v.z, m02);
    m11 = fma(a1, v.y, m11); m12 = fma(a1, v.z, m12); m22 = fma(a2, v.z, m22);
  }
  double c00 = m11 * m22 - m12 * m12, c01 = m12 * m02 - m01 * m22, c02 = m01 * m12 - m11 * m02;
  double det = m00 * c00 + m01 * c01 + m02 * c02;
  double* o = minv + 6 * (size_t)i;
  if (!(det != 0.0) || !isfinite(det)) {
    atomicOr(status, kStSingular);
    for (int q = 0; q < 6; ++q) o[q] = 0.0;
    return;
  }
  o[0] = c00 / det;
  o[1] = c01 / det;
  o[2] = c02 / det;
  o[3] = (m00 * m22 - m02 * m02) / det;
  o[4] = (m02 * m01 - m00 * m12) / det;
  o[5] = (m00 * m11 - m01 * m01) / det;
}

// Half-edge records in CSR order for the gradient kernel: u = +- M^-1 w of the
// face's least-squares weight w, with the sign that makes the cell's gradient
// sum_k u_k (phi_neighbour - phi_cell) (the matrix depends on the geometry
// only, so it is applied to the weights once per mesh instead of to every sum:
// 36 operations and six loads less per (cell, bin)), the neighbour id, and the
// face-centre offset x from this cell with, in the fourth lane, |x| (FP32
// sweep) or |x|^2 (FP64 sweep, summed in the order of the limiter's
// definition) for the limiter's regularisation test.
template <class R>
__global__ void k_build_halfedges(int n, const int32_t* __restrict__ csr, const int32_t* __restrict__ nbr,
                                  const int2* __restrict__ lr, const double* __restrict__ minv,
                                  const d4* __restrict__ w, const d4* __restrict__ rL, const d4* __restrict__ rR,
                                  R4<R>* hw, R4<R>* hx) {
  const int k = blockIdx.x * blockDim.x + threadIdx.x;
  if (k >= n) return;
  const int e = csr[k], f = e >> 1;
  const d4 wf = w[f];
  const double sg = (e & 1) ? -1.0 : 1.0;
  const double* m = minv + 6 * (size_t)((e & 1) ? lr[f].y : lr[f].x);
  R4<R> a;
  a.x = (R)(sg * (m[0] * wf.x + m[1] * wf.y + m[2] * wf.z));
  a.y = (R)(sg * (m[1] * wf.x + m[3] * wf.y + m[4] * wf.z));
  a.z = (R)(sg * (m[2] * wf.x + m[4] * wf.y + m[5] * wf.z));
  a.w = id_bits(nbr[k], R(0));
  hw[k] = a;
  const d4 x = (e & 1) ? rR[f] : rL[f];
  R4<R> b;
  const double xx = __dadd_rn(__dadd_rn(__dmul_rn(x.x, x.x), __dmul_rn(x.y, x.y)), __dmul_rn(x.z, x.z));
  b.x = (R)x.x; b.y = (R)x.y; b.z = (R)x.z;
  b.w = sizeof(R) == 4 ? (R)sqrt(xx) : (R)xx;
  hx[k] = b;
}

// Per cell, the largest hx.w over its half-edges (|x| in FP32, |x|^2 in FP64):
// the limiter's one-pass test (k_grad, k_grad_staged).
template <class R>
__global__ void k_cell_xmax(int C, const int32_t* __restrict__ off, const R4<R>* __restrict__ hx, R* xmax) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= C) return;
  R m = R(0);
  for (int k = off[i]; k < off[i + 1]; ++k) {
    const R w = hx[k].w;
    m = w > m ? w : m;
  }
  xmax[i] = m;
}

// FP64 sweep, per cell, for the limiter's search: the offsets in FP32, scaled by a
// power of two of the cell's own so that the largest |x_f| lies in [1, 2) whatever
// the unit of length (with cells of 1e20 cm unscaled offsets left FP32's range, and
// the search came on top of the scan it was to spare: 251 us a launch instead of
// 167 at 64,000 cells and three bins), and that largest |x_f|, NaN where |x_f|^2 is
// not a normal number.
__global__ void k_cell_search(int C, const int32_t* __restrict__ off, const d4* __restrict__ hx,
                              const double* __restrict__ xmax, float4* __restrict__ hx32, float* __restrict__ xm32) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= C) return;
  const double X = xmax[i];
  const int e = (__double2hiint(X) >> 20) - 1023;   // X > 0: in [-1022, 1023] where it is normal
  const bool ok = e >= -1022 && e <= 1023;
  const int k = ok ? e >> 1 : 0;
  const double s = __hiloint2double((1023 - k) << 20, 0);   // 2^-k
  for (int q = off[i]; q < off[i + 1]; ++q) {
    const d4 x = hx[q];
    hx32[q] = make_float4((float)(x.x * s), (float)(x.y * s), (float)(x.z * s), 0.f);
  }
  xm32[i] = ok ? sqrtf((float)(X * s * s)) : nanf("");
}

// Face records of the FP32 sweep: (n, A, x_f - s_L, left id) in 32 bytes
// and (x_f - s_R, right id) in 16 bytes.
__global__ void k_build_facerecs(int F, const int2* __restrict__ lr, const d4* __restrict__ nA,
                                 const d4* __restrict__ rL, const d4* __restrict__ rR, f8* fa, float4* fb) {
  const int f = blockIdx.x * blockDim.x + threadIdx.x;
  if (f >= F) return;
  const int2 c = lr[f];
  const d4 n = nA[f], a = rL[f], b = rR[f];
  f8 o;
  o.v[0] = (float)n.x; o.v[1] = (float)n.y; o.v[2] = (float)n.z; o.v[3] = (float)n.w;
  o.v[4] = (float)a.x; o.v[5] = (float)a.y; o.v[6] = (float)a.z; o.v[7] = __int_as_float(c.x);
  fa[f] = o;
  fb[f] = make_float4((float)b.x, (float)b.y, (float)b.z, __int_as_float(c.y));
}


// ---------------------------------------------------------------------------
// state packing: component-major caller arrays <-> per-cell interleaved records
// ---------------------------------------------------------------------------

// One thread per cell over its bins: the caller's component-major arrays are
// read and written a warp's 32 cells at a time (whole 256-byte runs), each
// cell's records as one contiguous piece.  The kernels work on the caller's
// device arrays themselves: no copy into a staging buffer and, in the mixed
// path, no pass through interleaved FP64 records.  Bound by memory: at 216,000
// cells and three bins setting and getting the radiation moved 280 MB in ten
// operations and moves 72 MB in two.

// rad[i*B + b] = (N, F_x / c, F_y / c, F_z / c) from N[b*C + i], F[(3b+k)*C + i].
__global__ void k_pack_rad(int C, int B, double inv_c, const double* __restrict__ N, const double* __restrict__ F,
                           d4* __restrict__ rad) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= C) return;
  for (int b = 0; b < B; ++b) {
    d4 v = make_d4(N[(size_t)b * C + i], 0.0, 0.0, 0.0);
    if (F) {
      v.y = F[(size_t)(3 * b) * C + i] * inv_c;
      v.z = F[(size_t)(3 * b + 1) * C + i] * inv_c;
      v.w = F[(size_t)(3 * b + 2) * C + i] * inv_c;
    }
    rad[(size_t)i * B + b] = v;
  }
}

__global__ void k_unpack_rad(int C, int B, double c, const d4* __restrict__ rad, double* __restrict__ N,
                             double* __restrict__ F) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= C) return;
  for (int b = 0; b < B; ++b) {
    const d4 v = rad[(size_t)i * B + b];
    if (N) N[(size_t)b * C + i] = v.x;
    if (F) {
      F[(size_t)(3 * b) * C + i] = v.y * c;
      F[(size_t)(3 * b + 1) * C + i] = v.z * c;
      F[(size_t)(3 * b + 2) * C + i] = v.w * c;
    }
  }
}

// Mixed precision keeps the photon density N of each (cell, bin) in FP64
// (radN) and the reduced flux in FP32, as lanes 1-3 of the FP32 sweep record
// (N rounded to FP32, f_x, f_y, f_z) that the gradient and flux kernels read.
__global__ void k_pack_mixed(int C, int B, double inv_c, const double* __restrict__ N, const double* __restrict__ F,
                             double* __restrict__ radN, float4* __restrict__ sh) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= C) return;
  for (int b = 0; b < B; ++b) {
    const double n = N[(size_t)b * C + i];
    float4 v = make_float4((float)n, 0.f, 0.f, 0.f);
    if (F) {
      v.y = (float)(F[(size_t)(3 * b) * C + i] * inv_c);
      v.z = (float)(F[(size_t)(3 * b + 1) * C + i] * inv_c);
      v.w = (float)(F[(size_t)(3 * b + 2) * C + i] * inv_c);
    }
    radN[(size_t)i * B + b] = n;
    sh[(size_t)i * B + b] = v;
  }
}
// The flux widened exactly, then times c.
__global__ void k_unpack_mixed(int C, int B, double c, const double* __restrict__ radN, const float4* __restrict__ sh,
                               double* __restrict__ N, double* __restrict__ F) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= C) return;
  for (int b = 0; b < B; ++b) {
    if (N) N[(size_t)b * C + i] = radN[(size_t)i * B + b];
    if (F) {
      const float4 v = sh[(size_t)i * B + b];
      F[(size_t)(3 * b) * C + i] = (double)v.y * c;
      F[(size_t)(3 * b + 1) * C + i] = (double)v.z * c;
      F[(size_t)(3 * b + 2) * C + i] = (double)v.w * c;
    }
  }
}

__global__ void k_widen(int n, const int32_t* __restrict__ in, double* __restrict__ out) {
  const int k = blockIdx.x * blockDim.x + threadIdx.x;
  if (k < n) out[k] = (double)in[k];
}

// ---------------------------------------------------------------------------
// active sets
// ---------------------------------------------------------------------------

// The masks of the active sets kept so far (null: none there).
struct KnownMasks {
  static constexpr int kMax = 8;
  const uint8_t* m[kMax];
};

// A new mask, normalised to 0 and 1 (padded with ones to whole 16-byte words),
// against the known ones: bit s of *out is set if it differs from mask s, bit
// kMax if some cell is inactive.  16 cells per thread; one pass over the mask
// and the known masks (0.12 MB each at 117,649 cells) in place of the host's
// hash and comparison, 150 us there.
__global__ void k_match_mask(int C, const uint8_t* __restrict__ in, uint8_t* __restrict__ norm, KnownMasks known,
                             unsigned* __restrict__ out) {
  const int w = blockIdx.x * blockDim.x + threadIdx.x;
  const long long i0 = 16LL * w;
  if (i0 >= C) return;
  unsigned v[4] = {0x01010101u, 0x01010101u, 0x01010101u, 0x01010101u};
#pragma unroll
  for (int k = 0; k < 16; ++k)
    if (i0 + k < C && in[i0 + k] == 0) v[k >> 2] &= ~(1u << (8 * (k & 3)));
  reinterpret_cast<uint4*>(norm)[w] = make_uint4(v[0], v[1], v[2], v[3]);
  unsigned r = (v[0] & v[1] & v[2] & v[3]) != 0x01010101u ? 1u << KnownMasks::kMax : 0u;
#pragma unroll
  for (int s = 0; s < KnownMasks::kMax; ++s)
    if (known.m[s]) {
      const uint4 q = reinterpret_cast<const uint4*>(known.m[s])[w];
      if (q.x != v[0] || q.y != v[1] || q.z != v[2] || q.w != v[3]) r |= 1u << s;
    }
  if (r & ~*(volatile unsigned*)out) atomicOr(out, r);
}

// The lists of a new active set, built on the device (the host's passes over
// cells and faces took 2.6 ms at 117,649 cells).  First the flags: a face is
// active if one of its cells is, a cell is touched if one of its faces is.
__global__ void k_set_faces(int F, const int2* __restrict__ lr, const uint8_t* __restrict__ mask,
                            uint8_t* __restrict__ face, uint8_t* __restrict__ touched) {
  const int f = blockIdx.x * blockDim.x + threadIdx.x;
  if (f >= F) return;
  const int2 c = lr[f];
  const uint8_t on = mask[c.x] | mask[c.y];
  face[f] = on;
  if (on) touched[c.x] = touched[c.y] = 1;   // whoever writes, writes 1
}
// A block of `per` cells holds a touched cell.
__global__ void k_set_blocks(int nb, int C, int per, const uint8_t* __restrict__ touched, uint8_t* __restrict__ block) {
  const int b = blockIdx.x * blockDim.x + threadIdx.x;
  if (b >= nb) return;
  uint8_t any = 0;
  for (int i = b * per; i < min(b * per + per, C); ++i) any |= touched[i];
  block[b] = any;
}
// The entries with a flag, in order: their number per kScan of them, then (the
// numbers summed up by k_scan_sums) their places.
__global__ void __launch_bounds__(kScan) k_flag_count(int n, const uint8_t* __restrict__ flag, int32_t* __restrict__ sums) {
  const long long i = (long long)blockIdx.x * kScan + threadIdx.x;
  const int c = __syncthreads_count(i < n && flag[i]);
  if (threadIdx.x == 0) sums[blockIdx.x] = c;
}
__global__ void __launch_bounds__(kScan) k_flag_list(int n, const uint8_t* __restrict__ flag,
                                                     const int32_t* __restrict__ sums, int32_t* __restrict__ list) {
  __shared__ int ws[32];
  const long long i = (long long)blockIdx.x * kScan + threadIdx.x;
  const int v = i < n && flag[i] ? 1 : 0;
  const int e = block_scan(v, ws);
  if (v) list[sums[blockIdx.x] + e] = (int)i;
}
// The face records of the largest run of `per` list entries.
__global__ void k_list_cap(int n, int per, const int32_t* __restrict__ list, const int32_t* __restrict__ off,
                           int* __restrict__ cap) {
  const long long j0 = (long long)per * (blockIdx.x * blockDim.x + threadIdx.x);
  if (j0 >= n) return;
  int sum = 0;
  for (long long j = j0; j < min(j0 + per, (long long)n); ++j) sum += off[list[j] + 1] - off[list[j]];
  atomicMax(cap, sum);
}

// ---------------------------------------------------------------------------
// gradients + limiter
// ---------------------------------------------------------------------------

template <class R> __device__ __forceinline__ R comp(const R4<R>& v, int q) {
  return q == 0 ? v.x : (q == 1 ? v.y : (q == 2 ? v.z : v.w));
}

// Limiter extremes of one (cell, bin) over its faces k0..k1-1: dpos =
// max(0, max g.x_f) and dneg = min(0, min g.x_f) over the faces that pass
// the regularisation test |g.x_f| > eps |g| |x_f|.  First one pass without
// the test.  Its extremes are those of the definition whenever each nonzero
// one clears the test bound of the cell's largest |x_f| (X): the face that
// attains it then passes its own test, since rounding is monotone.  Only
// otherwise (an extreme within the band; rare) the pass with the test runs.
// FP32: eg = eps |g|, X and x.w = |x_f|.
__device__ __forceinline__ void lim_extremes(const float4* __restrict__ xs, int k0, int k1, const float gr[4][3],
                                             const float eg[4], float X, float dpos[4], float dneg[4]) {
#pragma unroll
  for (int q = 0; q < 4; ++q) dpos[q] = dneg[q] = 0.0f;
#pragma unroll 4
  for (int k = k0; k < k1; ++k) {
    const float4 x = xs[k];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const float dphi = gr[q][0] * x.x + gr[q][1] * x.y + gr[q][2] * x.z;
      dpos[q] = fmaxf(dpos[q], dphi);
      dneg[q] = fminf(dneg[q], dphi);
    }
  }
  bool exact = true;
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    const float t = eg[q] * X;
    exact = exact && (dpos[q] == 0.0f || dpos[q] > t) && (dneg[q] == 0.0f || -dneg[q] > t);
  }
  if (exact) return;
#pragma unroll
  for (int q = 0; q < 4; ++q) dpos[q] = dneg[q] = 0.0f;
  for (int k = k0; k < k1; ++k) {
    const float4 x = xs[k];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const float dphi = gr[q][0] * x.x + gr[q][1] * x.y + gr[q][2] * x.z;
      const float dm = fabsf(dphi) > eg[q] * x.w ? dphi : 0.0f;
      dpos[q] = fmaxf(dpos[q], dm);
      dneg[q] = fminf(dneg[q], dm);
    }
  }
}

// max / min of two finite values: one FMNMX in FP32; the FP64 sweep keeps
// the comparison form of the limiter's definition.
template <class R> __device__ __forceinline__ R rmax(R a, R b) {
  if constexpr (sizeof(R) == 4) return fmaxf(a, b);
  else return b > a ? b : a;
}
template <class R> __device__ __forceinline__ R rmin(R a, R b) {
  if constexpr (sizeof(R) == 4) return fminf(a, b);
  else return b < a ? b : a;
}

// What the reverse mode needs of a (cell, bin)'s gradients beside the limited
// ones: the gradients before the limiter, the factors, the half-edge that
// limits each component (-1: none) and the cell that holds the extreme it is
// limited by.
struct GradTape {
  double g[12], psi[4];
  int32_t at[4], cell[4];
};

// G[(i*B + b)*12 + q*3 + d]: limited gradient of component q of bin b.
// kTape (FP64 sweep): the reverse mode's record too.
template <class R, bool kTape = false>
__global__ void __launch_bounds__(256) k_grad(Geo<R> g, const R4<R>* __restrict__ rad, R* __restrict__ G,
                                              int order, int limiter, R lim_eps2, GradTape* __restrict__ tape) {
  int t = blockIdx.x * blockDim.x + threadIdx.x;
  const int B = g.B;
  if (t >= (g.clist ? g.nc : g.C) * B) return;
  const int ii = divb(t, g.divB), b = t - ii * B;
  const int i = g.clist ? __ldg(g.clist + ii) : ii;
  t = i * B + b;
  const R4<R> pi = ld4<R>(rad + t);
  if (order < 2) {
    if constexpr (sizeof(R) == 4) {
      float4* G4 = reinterpret_cast<float4*>(G);
      for (int v = 0; v < 3; ++v) G4[grec(i, v, b, g.Bp)] = make_float4(0.f, 0.f, 0.f, 0.f);
      G4[grec(i, 3, b, g.Bp)] = pi;
    } else {
      R* Go = G + (size_t)t * 12;
#pragma unroll
      for (int k = 0; k < 12; ++k) Go[k] = R(0);
    }
    return;   // first order: the reverse mode reads no record either
  }
  R gr[4][3];
  R mx[4], mn[4];
  // FP64: the neighbour extremes as max_j (phi_j - phi_i) >= 0 and
  // min_j (phi_j - phi_i) <= 0, kept as bit patterns and compared on the
  // integer pipe (the FP64 pipe runs 1/64 of the FP32 rate on this part and
  // is what bounds this kernel).  Rounding is monotone, so max_j fl(phi_j -
  // phi_i) = fl(max_j phi_j - phi_i): the same values as the definition.
  long long dmx[4], dmn[4];   // bits of the largest difference, magnitude bits of the most negative
  int jmx[4], jmn[4];         // kTape: the cells they belong to
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    gr[q][0] = gr[q][1] = gr[q][2] = R(0);
    mx[q] = mn[q] = comp<R>(pi, q);
    dmx[q] = dmn[q] = 0;
    jmx[q] = jmn[q] = i;
  }
  const int k0 = g.off[i], k1 = g.off[i + 1];
  // half-edge k: u_k (phi_j - phi_i) is this face's term of the gradient
  auto acc_face = [&](const R4<R>& hw, const R4<R>& pj) {
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const R vj = comp<R>(pj, q), dphi = vj - comp<R>(pi, q);
      gr[q][0] += hw.x * dphi;
      gr[q][1] += hw.y * dphi;
      gr[q][2] += hw.z * dphi;
      if constexpr (sizeof(R) == 8) {
        const long long up = max_bits_pos(dmx[q], dphi), dn = max_bits_neg(dmn[q], dphi);
        if constexpr (kTape) {
          jmx[q] = up != dmx[q] ? bits_id(hw.w) : jmx[q];
          jmn[q] = dn != dmn[q] ? bits_id(hw.w) : jmn[q];
        }
        dmx[q] = up;
        dmn[q] = dn;
      } else {
        mx[q] = rmax<R>(mx[q], vj);
        mn[q] = rmin<R>(mn[q], vj);
      }
    }
  };
  int k = k0;
  // one face at a time, not unrolled (batches of four with a serial tail
  // were measured slower in the FP64 sweep)
#pragma unroll 1
  for (; k < k1; ++k) {
    const R4<R> hw = ld4<R>(g.hw + k);
    acc_face(hw, ld4<R>(rad + (size_t)bits_id(hw.w) * B + b));
  }
  R psi[4];
  int lim_at[4] = {-1, -1, -1, -1}, lim_cell[4] = {-1, -1, -1, -1};
#pragma unroll
  for (int q = 0; q < 4; ++q) psi[q] = R(1);
  if (limiter) {
    // psi = min over faces of (max - phi_i) / (g.x) for g.x > 0 and
    // (min - phi_i) / (g.x) for g.x < 0.  Rounded division is monotone in
    // the divisor, so each of these minima is the quotient by the largest
    // (most negative) g.x: two divisions per component instead of one per
    // face, with bitwise the same result.
    R dpos[4], dneg[4];
    int at[8];
    if constexpr (sizeof(R) == 4) {
      float eg[4];
#pragma unroll
      for (int q = 0; q < 4; ++q)
        eg[q] = sqrtf(lim_eps2 * (gr[q][0] * gr[q][0] + gr[q][1] * gr[q][1] + gr[q][2] * gr[q][2]));
      lim_extremes(g.hx, k0, k1, gr, eg, __ldg(g.xmax + i), dpos, dneg);
    } else {
      lim_extremes(g.hx, g.hx32, k0, k1, gr, lim_eps2, __ldg(g.xmax + i), __ldg(g.xm32 + i), dpos, dneg, at);
    }
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const R vi = comp<R>(pi, q);
      R up, dn;   // max_j phi_j - phi_i and min_j phi_j - phi_i
      if constexpr (sizeof(R) == 8) {
        up = __longlong_as_double(dmx[q]);
        dn = neg_from_bits(dmn[q]);
      } else {
        up = mx[q] - vi;
        dn = mn[q] - vi;
      }
      if constexpr (sizeof(R) == 8) {
        // dpos >= +0, dneg = -magnitude or +0, the factors >= +0: the
        // tests on the integer pipe
        if (limits_pos(up, dpos[q])) {
          const R lim = div_nr(up, dpos[q]);
          if (kTape && gt_nonneg(psi[q], lim)) { lim_at[q] = at[2 * q]; lim_cell[q] = jmx[q]; }
          psi[q] = gt_nonneg(psi[q], lim) ? lim : psi[q];
        }
        if (limits_neg(dn, dneg[q])) {
          const R lim = div_nr(dn, dneg[q]);
          // equal factors: the face that comes first
          if (kTape && (gt_nonneg(psi[q], lim) ||
                        (lim_at[q] > at[2 * q + 1] && __double_as_longlong(psi[q]) == __double_as_longlong(lim)))) {
            lim_at[q] = at[2 * q + 1];
            lim_cell[q] = jmn[q];
          }
          psi[q] = gt_nonneg(psi[q], lim) ? lim : psi[q];
        }
      } else {
        if (dpos[q] > R(0)) {
          const R lim = up / dpos[q];
          psi[q] = lim < psi[q] ? lim : psi[q];
        }
        if (dneg[q] < R(0)) {
          const R lim = dn / dneg[q];
          psi[q] = lim < psi[q] ? lim : psi[q];
        }
      }
    }
  }
  if constexpr (kTape) {
    GradTape& r = tape[t];
    d4* r4 = reinterpret_cast<d4*>(&r);
    r4[0] = make_d4(gr[0][0], gr[0][1], gr[0][2], gr[1][0]);
    r4[1] = make_d4(gr[1][1], gr[1][2], gr[2][0], gr[2][1]);
    r4[2] = make_d4(gr[2][2], gr[3][0], gr[3][1], gr[3][2]);
    r4[3] = make_d4(psi[0], psi[1], psi[2], psi[3]);
    reinterpret_cast<int4*>(r.at)[0] = make_int4(lim_at[0], lim_at[1], lim_at[2], lim_at[3]);
    reinterpret_cast<int4*>(r.cell)[0] = make_int4(lim_cell[0], lim_cell[1], lim_cell[2], lim_cell[3]);
  }
  R o[12];
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    o[3 * q + 0] = gr[q][0] * psi[q];
    o[3 * q + 1] = gr[q][1] * psi[q];
    o[3 * q + 2] = gr[q][2] * psi[q];
  }
  if constexpr (sizeof(R) == 4) {
    float4* G4 = reinterpret_cast<float4*>(G);
    G4[grec(i, 0, b, g.Bp)] = make_float4(o[0], o[1], o[2], o[3]);
    G4[grec(i, 1, b, g.Bp)] = make_float4(o[4], o[5], o[6], o[7]);
    G4[grec(i, 2, b, g.Bp)] = make_float4(o[8], o[9], o[10], o[11]);
    G4[grec(i, 3, b, g.Bp)] = pi;
  } else {
    R4<R>* G4 = reinterpret_cast<R4<R>*>(G + (size_t)t * 12);
#pragma unroll
    for (int v = 0; v < 3; ++v) {
      R4<R> w;
      w.x = o[4 * v]; w.y = o[4 * v + 1]; w.z = o[4 * v + 2]; w.w = o[4 * v + 3];
      G4[v] = w;
    }
  }
}

// Three-input FP32 maximum and minimum (one instruction on sm_100 and
// later); exact, like fmaxf / fminf of two.
__device__ __forceinline__ float max3f(float a, float b, float c) {
  float d;
  asm("max.f32 %0, %1, %2, %3;" : "=f"(d) : "f"(a), "f"(b), "f"(c));
  return d;
}
__device__ __forceinline__ float min3f(float a, float b, float c) {
  float d;
  asm("min.f32 %0, %1, %2, %3;" : "=f"(d) : "f"(a), "f"(b), "f"(c));
  return d;
}

// lim_extremes with the faces taken two at a time by three-input extremes:
// the same extremes (max and min are exact), half the compare instructions.
__device__ __forceinline__ void lim_extremes_pairs(const float4* __restrict__ xs, int k0, int k1,
                                                   const float gr[4][3], const float eg[4], float X, float dpos[4],
                                                   float dneg[4]) {
#pragma unroll
  for (int q = 0; q < 4; ++q) dpos[q] = dneg[q] = 0.0f;
  int k = k0;
#pragma unroll 2
  for (; k + 2 <= k1; k += 2) {
    const float4 xa = xs[k], xb = xs[k + 1];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const float da = gr[q][0] * xa.x + gr[q][1] * xa.y + gr[q][2] * xa.z;
      const float db = gr[q][0] * xb.x + gr[q][1] * xb.y + gr[q][2] * xb.z;
      dpos[q] = max3f(dpos[q], da, db);
      dneg[q] = min3f(dneg[q], da, db);
    }
  }
  if (k < k1) {
    const float4 x = xs[k];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const float dphi = gr[q][0] * x.x + gr[q][1] * x.y + gr[q][2] * x.z;
      dpos[q] = fmaxf(dpos[q], dphi);
      dneg[q] = fminf(dneg[q], dphi);
    }
  }
  bool exact = true;
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    const float t = eg[q] * X;
    exact = exact && (dpos[q] == 0.0f || dpos[q] > t) && (dneg[q] == 0.0f || -dneg[q] > t);
  }
  if (exact) return;
#pragma unroll
  for (int q = 0; q < 4; ++q) dpos[q] = dneg[q] = 0.0f;
  for (k = k0; k < k1; ++k) {
    const float4 x = xs[k];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const float dphi = gr[q][0] * x.x + gr[q][1] * x.y + gr[q][2] * x.z;
      const float dm = fabsf(dphi) > eg[q] * x.w ? dphi : 0.0f;
      dpos[q] = fmaxf(dpos[q], dm);
      dneg[q] = fminf(dneg[q], dm);
    }
  }
}

// The FP32 gradients' last part, from the gradients g and the neighbour
// extremes: the limiter factors (extremes of
// g . x_f over the offset records xs[k0, k1) by lim_extremes_pairs), and the
// record of (cell i, bin b) written as two 32-byte stores (groups 0-1 and
// 2-3).
__device__ __forceinline__ void grad_tail_fp32(const Geo<float>& g, float* __restrict__ G, int i, int b,
                                               const float4& pi, const float gr[4][3], const float mx[4],
                                               const float mn[4], float xm, const float4* __restrict__ shx,
                                               int k0, int k1, int limiter, float lim_eps2) {
  float psi[4], eg[4];
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    eg[q] = sqrtf(lim_eps2 * (gr[q][0] * gr[q][0] + gr[q][1] * gr[q][1] + gr[q][2] * gr[q][2]));
    psi[q] = 1.f;
  }
  if (limiter) {
    float dpos[4], dneg[4];
    lim_extremes_pairs(shx, k0, k1, gr, eg, xm, dpos, dneg);
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const float vi = comp<float>(pi, q);
      // approximate quotients (2 ulp): a limiter factor needs no
      // correctly rounded division
      if (dpos[q] > 0.f) psi[q] = fminf(psi[q], __fdividef(mx[q] - vi, dpos[q]));
      if (dneg[q] < 0.f) psi[q] = fminf(psi[q], __fdividef(mn[q] - vi, dneg[q]));
    }
  }
  // groups 0-1 and 2-3 as two 32-byte stores
  float4* G4 = reinterpret_cast<float4*>(G);
  st8(reinterpret_cast<f8*>(G4 + grec(i, 0, b, g.Bp)), gr[0][0] * psi[0], gr[0][1] * psi[0], gr[0][2] * psi[0],
      gr[1][0] * psi[1], gr[1][1] * psi[1], gr[1][2] * psi[1], gr[2][0] * psi[2], gr[2][1] * psi[2]);
  st8(reinterpret_cast<f8*>(G4 + grec(i, 2, b, g.Bp)), gr[2][2] * psi[2], gr[3][0] * psi[3], gr[3][1] * psi[3],
      gr[3][2] * psi[3], pi.x, pi.y, pi.z, pi.w);
}


// The same gradients and limiter for the FP32 sweep with the half-edge
// records staged in shared memory.  A block owns kGradCells cells: in block
// mode kGradCells consecutive cells, whose records are one contiguous range
// of the CSR arrays, copied by two bulk copies (TMA engine) from one thread;
// in list mode (list_mode != 0, an active set) kGradCells consecutive
// entries of the touched-cell list, each cell's records copied by its own
// two bulk copies to the prefix sums of the cells' face counts.  The copies
// complete on one mbarrier while every thread loads its own cell state;
// afterwards the only global loads left per face are the neighbour states,
// issued NB at a time.  `cap` is the largest record count of any block (the
// dynamic shared memory holds 2 cap records).
constexpr int kGradCells = 32;

template <int NB>
__global__ void __launch_bounds__(kGradCells* kMaxBins)
    k_grad_staged(Geo<float> g, const float4* __restrict__ rad, float* __restrict__ G, int limiter, float lim_eps2,
                  int cap, int* status, int list_mode) {
  extern __shared__ float4 sm[];  // [cap] weight records, then [cap] offset records
  __shared__ __align__(8) uint64_t bar;
  __shared__ int so[kGradCells];  // list mode: first record of each cell in shared memory
  static_assert(kGradCells == 32, "list mode scans one cell per lane of warp 0");
  const int B = g.B;
  const int lt = threadIdx.x;
  const int cl = divb(lt, g.divB), b = lt - cl * B;
  int i, k0 = 0, k1 = 0, kb0 = 0;
  bool active;
  if (lt == 0) mbar_init(&bar, 1);
  if (!list_mode) {
    // kGradCells consecutive cells: their records are one contiguous range
    const int c0 = (g.blist ? __ldg(g.blist + blockIdx.x) : (int)blockIdx.x) * kGradCells;
    const int c1 = min(c0 + kGradCells, g.C);
    kb0 = __ldg(g.off + c0);
    const int kb1 = __ldg(g.off + c1);
    i = c0 + cl;
    active = i < c1 && (!g.touched || __ldg(g.touched + i));
    __syncthreads();
    if (lt == 0) {
      const uint32_t bytes = (uint32_t)(kb1 - kb0) * (uint32_t)sizeof(float4);
      mbar_arrive_expect_tx(&bar, 2 * bytes);
      bulk_g2s(sm, g.hw + kb0, bytes, &bar);
      bulk_g2s(sm + cap, g.hx + kb0, bytes, &bar);
    }
  } else {
    // kGradCells entries of the touched-cell list: one contiguous range of
    // records per cell, packed in shared memory at the prefix sums of the
    // cells' face counts (warp 0, one cell per lane), one bulk copy per cell
    // and array, all counted on the one mbarrier
    const int l0 = blockIdx.x * kGradCells;
    int ci = 0, o0 = 0, deg = 0, total = 0;
    if (lt < 32) {
      if (l0 + lt < g.nc) {
        ci = __ldg(g.clist + l0 + lt);
        o0 = __ldg(g.off + ci);
        deg = __ldg(g.off + ci + 1) - o0;
      }
      int sc = deg;
#pragma unroll
      for (int d = 1; d < 32; d <<= 1) {
        const int v = __shfl_up_sync(0xffffffffu, sc, d);
        if (lt >= d) sc += v;
      }
      total = __shfl_sync(0xffffffffu, sc, 31);
      so[lt] = sc - deg;
    }
    __syncthreads();
    if (lt < 32) {
      if (lt == 0) mbar_arrive_expect_tx(&bar, 2u * (uint32_t)total * (uint32_t)sizeof(float4));
      if (deg > 0) {
        const uint32_t bytes = (uint32_t)deg * (uint32_t)sizeof(float4);
        bulk_g2s(sm + so[lt], g.hw + o0, bytes, &bar);
        bulk_g2s(sm + cap + so[lt], g.hx + o0, bytes, &bar);
      }
    }
    active = l0 + cl < g.nc;
    i = active ? __ldg(g.clist + l0 + cl) : 0;
  }
  float4 pi = make_float4(0.f, 0.f, 0.f, 0.f);
  float xm = 0.f;
  if (active) {
    pi = __ldg(rad + (size_t)i * B + b);
    if (!list_mode) {
      k0 = __ldg(g.off + i) - kb0;
      k1 = __ldg(g.off + i + 1) - kb0;
    } else {
      k0 = so[cl];
      k1 = k0 + (__ldg(g.off + i + 1) - __ldg(g.off + i));
    }
    xm = __ldg(g.xmax + i);
  }
  if (!mbar_wait(&bar, 0)) {
    // record the timeout, give the copies in flight a second bounded wait
    // to land before the block's shared memory goes away, and give up
    if (lt == 0) atomicOr(status, kStTimeout);
    mbar_wait(&bar, 0);
    return;
  }
  if (!active) return;
  const float4* shw = sm;
  const float4* shx = sm + cap;
  float r[4][3], mx[4], mn[4];
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    r[q][0] = r[q][1] = r[q][2] = 0.f;
    mx[q] = mn[q] = comp<float>(pi, q);
  }
  auto acc_rhs = [&](const float4& hw, const float4& pj) {
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const float dphi = comp<float>(pj, q) - comp<float>(pi, q);
      r[q][0] += hw.x * dphi;
      r[q][1] += hw.y * dphi;
      r[q][2] += hw.z * dphi;
    }
  };
  // neighbour states NB at a time, the last batch predicated (no serial
  // tail of single loads); the sums still run in CSR order.  The extremes
  // take the batch by three-input max / min, the entries past the cell's
  // last face filled with its own state (the extremes start from it).
  static_assert(NB % 2 == 0, "neighbour batches in pairs");
  for (int k = k0; k < k1; k += NB) {
    float4 pj[NB];
#pragma unroll
    for (int u = 0; u < NB; ++u)
      pj[u] = k + u < k1 ? __ldg(rad + (size_t)bits_id(shw[k + u].w) * B + b) : pi;
#pragma unroll
    for (int u = 0; u < NB; ++u)
      if (k + u < k1) acc_rhs(shw[k + u], pj[u]);
#pragma unroll
    for (int u = 0; u < NB; u += 2)
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        mx[q] = max3f(mx[q], comp<float>(pj[u], q), comp<float>(pj[u + 1], q));
        mn[q] = min3f(mn[q], comp<float>(pj[u], q), comp<float>(pj[u + 1], q));
      }
  }
  grad_tail_fp32(g, G, i, b, pi, r, mx, mn, xm, shx, k0, k1, limiter, lim_eps2);
}

// ---------------------------------------------------------------------------
// face flux
// ---------------------------------------------------------------------------

// FP64: linear extrapolation of the cell state to the face centre, summed onto
// the state by fused multiply-adds, clamped to N >= 0 and |F| <= c N (tested on
// squares on the integer pipe; the square root only where it clamps).  Also the
// squares N2 = N^2 and fl2 = |F|^2 that the closure needs.
__device__ __forceinline__ void face_state(const d4& p, const double* __restrict__ Gp, const d4& x, double v[4],
                                           double& N2, double& fl2) {
  // the 12 gradient words of one (cell, bin) as three aligned 4-vectors
  const d4* G4 = reinterpret_cast<const d4*>(Gp);
  const d4 a = G4[0], b = G4[1], c = G4[2];
  const double Gc[12] = {a.x, a.y, a.z, a.w, b.x, b.y, b.z, b.w, c.x, c.y, c.z, c.w};
#pragma unroll
  for (int q = 0; q < 4; ++q)
    v[q] = fma(Gc[3 * q], x.x, fma(Gc[3 * q + 1], x.y, fma(Gc[3 * q + 2], x.z, comp<double>(p, q))));
  if (lt_zero(v[0])) v[0] = 0.0;
  N2 = v[0] * v[0];
  fl2 = v[1] * v[1] + v[2] * v[2] + v[3] * v[3];
  const bool over = nonfinite_bits(fl2);   // |F| beyond 1e154: F = 0, as by the definition's own squares
  if (gt_nonneg(fl2, N2) || over) {
    const double s = div_nr(v[0], sqrt_nr(fl2));
    v[1] *= s; v[2] *= s; v[3] *= s;
    fl2 = over ? 0.0 : N2;
  }
}

// s = sqrt(4 N^2 - 3 |F|^2) >= N within rounding (f <= 1), from the squares; where
// N^2 is near an end of the exponent range (densities beyond 1e150 or below
// 1e-150), from squares scaled by a power of two.
__device__ __forceinline__ double m1_root(double N, double N2, double fl2) {
  const unsigned e = (unsigned)__double2hiint(N2) & 0x7FF00000u;
  if (e - (23u << 20) < (2000u << 20)) {   // 2^-1000 <= N^2 < 2^1000
    const double t = fma(-3.0, fl2, 4.0 * N2);
    return sqrt_nr(gt_nonneg(N2, t) ? N2 : t);
  }
  const bool big = e >= 0x40000000u;
  const double c = big ? 0x1p-600 : 0x1p600, n = N * c, n2 = n * n;
  const double t = fma(-3.0, fl2 * c * c, 4.0 * n2);
  return sqrt_nr(gt_nonneg(n2, t) ? n2 : t) * (big ? 0x1p600 : 0x1p-600);
}

// The same extrapolation from the four groups of an FP32 gradient record:
// component q's gradient at words 3q..3q+2, the cell state at words 12..15.
__device__ __forceinline__ void face_state_rec(const float4 r[4], float x0, float x1, float x2, float v[4]) {
  const float w[16] = {r[0].x, r[0].y, r[0].z, r[0].w, r[1].x, r[1].y, r[1].z, r[1].w,
                       r[2].x, r[2].y, r[2].z, r[2].w, r[3].x, r[3].y, r[3].z, r[3].w};
#pragma unroll
  for (int q = 0; q < 4; ++q) v[q] = w[12 + q] + (w[3 * q] * x0 + w[3 * q + 1] * x1 + w[3 * q + 2] * x2);
  if (v[0] < 0.0f) v[0] = 0.0f;
  const float fl2 = v[1] * v[1] + v[2] * v[2] + v[3] * v[3];
  if (fl2 > v[0] * v[0]) {
    const float s = v[0] * rsqrtf(fl2);
    v[1] *= s; v[2] *= s; v[3] *= s;
  }
}

// N D n with the Levermore M1 Eddington tensor, FP32 sweep.
__device__ __forceinline__ void m1_normal(const float v[4], float n0, float n1, float n2, float P[3]) {
  // FP32 sweep, without branches, from hardware approximations (rsqrt,
  // reciprocal; sqrt(t) = t rsqrt(t) on t in [1, 4]).  Where F = 0 (which
  // the face-state clamp also makes of N = 0), f = 0 and u = 0 give
  // chi = 1/3 and D n = n / 3: the isotropic case needs no branch.
  const float fl2 = v[1] * v[1] + v[2] * v[2] + v[3] * v[3];
  const bool has_f = fl2 > 0.0f;
  const float ifl = has_f ? rsqrtf(fl2) : 0.0f;
  const float f = has_f ? fminf(fl2 * ifl * rcp_approx(v[0]), 1.0f) : 0.0f;
  const float f2 = f * f;
  const float t = 4.0f - 3.0f * f2;
  const float chi = (3.0f + 4.0f * f2) * rcp_approx(5.0f + 2.0f * (t * rsqrtf(t)));
  const float u0 = v[1] * ifl, u1 = v[2] * ifl, u2 = v[3] * ifl;
  const float un = u0 * n0 + u1 * n1 + u2 * n2;
  const float a = 0.5f * (1.0f - chi), bb = 0.5f * (3.0f * chi - 1.0f) * un;
  P[0] = v[0] * (a * n0 + bb * u0);
  P[1] = v[0] * (a * n1 + bb * u1);
  P[2] = v[0] * (a * n2 + bb * u2);
}

// FP64: N D n, D = (1 - chi)/2 I + (3 chi - 1)/2 u u, chi = (3 + 4 f^2) /
// (5 + 2 r) with r = sqrt(4 - 3 f^2), f = |F| / N and u = F / |F|.
// Multiplying chi's numerator and denominator by 5 - 2 r makes the denominator
// 9 + 12 f^2, so chi = (5 - 2 r) / 3 and
//   N D n = ((s - N) / 3) n + 3 (F . n) / (2 N + s) F,   s = N r = sqrt(4 N^2 - 3 |F|^2)
// (2 - r = 3 f^2 / (2 + r) takes the division by |F|^2 away): one square
// root and one quotient per face state instead of three quotients and a root,
// no case for F = 0, and no divisor that leaves the range of a fast quotient
// where N is small.  The kernel is bound by the FP64 unit: 1.67 -> 0.96 ms per
// launch at 250,047 cells, 234 -> 138 us at 262,144 cells with one bin (1.06 and
// 0.152 with the squares formed twice).
// Here: the two coefficients of 3 N D n = a n + 9 k F, and F . n.
__device__ __forceinline__ void m1_coef(const double v[4], double N2, double fl2, double n0, double n1, double n2,
                                        double& a, double& k, double& un) {
  un = v[1] * n0 + v[2] * n1 + v[3] * n2;
  a = v[0];
  k = 0.0;
  // the tests on the integer pipe (v[0] >= 0 after the face-state clamp)
  if (gt_nonneg(v[0], 0.0) && gt_nonneg(fl2, 0.0)) {
    const double s = m1_root(v[0], N2, fl2);
    a = s - v[0];
    k = div_nr(un, fma(2.0, v[0], s));
  }
}

// flux[f*B + b] = A (Phi_N, Phi_F) / c_red, global Lax-Friedrichs at c_red.
template <class R>
__global__ void __launch_bounds__(256, sizeof(R) == 4 ? 6 : 1) k_flux(Geo<R> g, const R4<R>* __restrict__ rad, const R* __restrict__ G,
                                              R4<R>* __restrict__ flux) {
  int t = blockIdx.x * blockDim.x + threadIdx.x;
  const int B = g.B;
  if (t >= (g.flist ? g.nf : g.F) * B) return;
  const int fi = divb(t, g.divB), b = t - fi * B;
  const int f = g.flist ? __ldg(g.flist + fi) : fi;
  t = f * B + b;
  if constexpr (sizeof(R) == 4) {
    // FP32 sweep: one 32-byte and one 16-byte face record, then the four
    // groups (gradients, state) of each side's cell-major record as two
    // 32-byte loads (groups 0-1 and 2-3 are adjacent in the paired layout);
    // with the registers of 6 blocks per SM, 6 % faster than four 16-byte
    // loads at 2e5 cells and 4 % at 2.1M (8 blocks: 3 % and 6 %)
    const f8 a = ld8(g.fa + f);
    const float4 xr = __ldg(g.fb + f);
    const float4* G4 = reinterpret_cast<const float4*>(G);
    const int cL = __float_as_int(a.v[7]), cR = __float_as_int(xr.w), Bp = g.Bp;
    float4 l[4], r[4];
    {
      const f8* G8 = reinterpret_cast<const f8*>(G4);
      const f8 l01 = ld8(G8 + (size_t)cL * 2 * Bp + b), l23 = ld8(G8 + (size_t)cL * 2 * Bp + Bp + b);
      const f8 r01 = ld8(G8 + (size_t)cR * 2 * Bp + b), r23 = ld8(G8 + (size_t)cR * 2 * Bp + Bp + b);
      l[0] = make_float4(l01.v[0], l01.v[1], l01.v[2], l01.v[3]);
      l[1] = make_float4(l01.v[4], l01.v[5], l01.v[6], l01.v[7]);
      l[2] = make_float4(l23.v[0], l23.v[1], l23.v[2], l23.v[3]);
      l[3] = make_float4(l23.v[4], l23.v[5], l23.v[6], l23.v[7]);
      r[0] = make_float4(r01.v[0], r01.v[1], r01.v[2], r01.v[3]);
      r[1] = make_float4(r01.v[4], r01.v[5], r01.v[6], r01.v[7]);
      r[2] = make_float4(r23.v[0], r23.v[1], r23.v[2], r23.v[3]);
      r[3] = make_float4(r23.v[4], r23.v[5], r23.v[6], r23.v[7]);
    }
    float vL[4], vR[4], PL[3], PR[3];
    face_state_rec(l, a.v[4], a.v[5], a.v[6], vL);
    face_state_rec(r, xr.x, xr.y, xr.z, vR);
    const float n0 = a.v[0], n1 = a.v[1], n2 = a.v[2], A = a.v[3];
    m1_normal(vL, n0, n1, n2, PL);
    m1_normal(vR, n0, n1, n2, PR);
    const float h = 0.5f;
    const float fn = h * ((vL[1] + vR[1]) * n0 + (vL[2] + vR[2]) * n1 + (vL[3] + vR[3]) * n2);
    float4 o;
    o.x = A * (fn - h * (vR[0] - vL[0]));
    o.y = A * (h * (PL[0] + PR[0]) - h * (vR[1] - vL[1]));
    o.z = A * (h * (PL[1] + PR[1]) - h * (vR[2] - vL[2]));
    o.w = A * (h * (PL[2] + PR[2]) - h * (vR[3] - vL[3]));
    flux[t] = o;
    return;
  }
  if constexpr (sizeof(R) == 8) {
    const int2 c = __ldg(g.lr + f);
    const d4 nA = g.nA[f];
    double vL[4], vR[4], N2L, N2R, f2L, f2R, aL, aR, kL, kR, uL, uR;
    const size_t sL = (size_t)c.x * B + b, sR = (size_t)c.y * B + b;
    face_state(rad[sL], G + sL * 12, g.rL[f], vL, N2L, f2L);
    face_state(rad[sR], G + sR * 12, g.rR[f], vR, N2R, f2R);
    m1_coef(vL, N2L, f2L, nA.x, nA.y, nA.z, aL, kL, uL);
    m1_coef(vR, N2R, f2R, nA.x, nA.y, nA.z, aR, kR, uR);
    const double hA = 0.5 * nA.w, h3 = 1.5 * nA.w, a9 = (aL + aR) * (1.0 / 9.0);
    d4 o;
    o.x = hA * ((uL + uR) - (vR[0] - vL[0]));
    o.y = fma(h3, fma(kR, vR[1], fma(kL, vL[1], a9 * nA.x)), hA * (vL[1] - vR[1]));
    o.z = fma(h3, fma(kR, vR[2], fma(kL, vL[2], a9 * nA.y)), hA * (vL[2] - vR[2]));
    o.w = fma(h3, fma(kR, vR[3], fma(kL, vL[3], a9 * nA.z)), hA * (vL[3] - vR[3]));
    flux[t] = o;
  }
}

// ---------------------------------------------------------------------------
// per cell: gather + sources + chemistry
// ---------------------------------------------------------------------------

struct CellArgs {
  int C, B;
  DivB divB;               // division by B
  const int32_t* list;     // individual time steps: the n cells to work on (null = all C)
  int n;
  const int32_t* off;
  const int32_t* csr;
  const double* vol;       // V_i (L_u^3)
  const double* ivol;      // 1 / V_i (mixed precision only)
  d4* rad;                 // FP64 sweep: radiation records (N, f) per (cell, bin)
  double* radN;            // mixed precision: N per (cell, bin) in FP64 (the flux is in the FP32 sweep records)
  double* nH;
  double* x5;              // 5*C
  double* T;
  const int32_t* src_idx;  // C: index into src_rate or -1
  const double* src_rate;  // [n_src_cells][B] photons/s
  int32_t* nsub;           // C
  int* status;
  d4* rad0;                // Heun: the state at the start of the transport step
  int heun;                // 0 plain; 1 keep the input in rad0; 2 write rad0/2 + (updated)/2
  double lam;              // c_red dt / unit_length_cm
  double dt;
  double lu3;              // unit_length_cm^3
  int do_gather, do_inject, do_chem;
};

// Error-free sum of two floats (Knuth): s + e == a + b exactly.
__device__ __forceinline__ void two_sum(float a, float b, float& s, float& e) {
  s = a + b;
  float bb = s - a;
  e = (a - (s - bb)) + (b - bb);
}

// The flux application's sum for (cell i, bin b): the cell's stored face
// fluxes in CSR order, + where the cell is the left cell, - where it is the
// right cell.  flux_sum_pair (mixed precision): the FP32 terms summed as an
// unevaluated FP32 pair hi + lo (error-free two_sum).  flux_sum: each term
// widened and summed in FP64.  Pred: the face loads in batches of four with
// a predicated last batch (no serial tail of single loads) -- faster where
// the flux array is held in L2, slower where the loads go to HBM and the
// extra registers cost occupancy.
template <bool Pred>
__device__ __forceinline__ void flux_sum_pair(const CellArgs& a, const float4* __restrict__ flux, int i, int b,
                                              float hi[4], float lo[4]) {
  const int B = a.B;
  const int k0 = a.off[i], k1 = a.off[i + 1];
#pragma unroll
  for (int q = 0; q < 4; ++q) hi[q] = lo[q] = 0.f;
  auto add = [&](int e, const float4& v) {
    const float sg = (e & 1) ? -1.0f : 1.0f;
    const float tv[4] = {sg * v.x, sg * v.y, sg * v.z, sg * v.w};
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      float sum, err;
      two_sum(hi[q], tv[q], sum, err);
      hi[q] = sum;
      lo[q] += err;
    }
  };
  if constexpr (Pred) {
    // the next batch's CSR entries are loaded while this batch's fluxes are
    // in flight (one round trip less per batch)
    int e[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) e[u] = k0 + u < k1 ? __ldg(a.csr + k0 + u) : 0;
    for (int k = k0; k < k1; k += 4) {
      float4 v[4];
#pragma unroll
      for (int u = 0; u < 4; ++u)
        if (k + u < k1) v[u] = __ldg(flux + (size_t)(e[u] >> 1) * B + b);
      int en[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) en[u] = k + 4 + u < k1 ? __ldg(a.csr + k + 4 + u) : 0;
#pragma unroll
      for (int u = 0; u < 4; ++u)
        if (k + u < k1) add(e[u], v[u]);
#pragma unroll
      for (int u = 0; u < 4; ++u) e[u] = en[u];
    }
  } else {
    int k = k0;
    // batches of four faces: all index and flux loads issued before use;
    // the terms are still added in CSR order
    for (; k + 4 <= k1; k += 4) {
      const int e0 = __ldg(a.csr + k), e1 = __ldg(a.csr + k + 1), e2 = __ldg(a.csr + k + 2),
                e3 = __ldg(a.csr + k + 3);
      const float4 v0 = __ldg(flux + (size_t)(e0 >> 1) * B + b), v1 = __ldg(flux + (size_t)(e1 >> 1) * B + b),
                   v2 = __ldg(flux + (size_t)(e2 >> 1) * B + b), v3 = __ldg(flux + (size_t)(e3 >> 1) * B + b);
      add(e0, v0); add(e1, v1); add(e2, v2); add(e3, v3);
    }
    for (; k < k1; ++k) {
      const int e = __ldg(a.csr + k);
      add(e, __ldg(flux + (size_t)(e >> 1) * B + b));
    }
  }
}

template <class R>
__device__ __forceinline__ void flux_sum(const CellArgs& a, const R4<R>* __restrict__ flux, int i, int b,
                                         double acc[4]) {
  const int B = a.B;
  const int k0 = a.off[i], k1 = a.off[i + 1];
  acc[0] = acc[1] = acc[2] = acc[3] = 0.0;
  // FP64 terms: acc +- v as one fused multiply-add by +-1 (exact product, one
  // rounding: the same sum as the add or subtract, without predicated copies
  // of both).  FP32 terms: the sign set and the term widened on the integer
  // pipe (the FP64 unit, which bounds this sum, also executes the hardware's
  // conversion: 66 -> 42 us at 64,000 cells and three bins), subnormal terms
  // included: with N near 1e-37 many are.
  auto add = [&](int e, const R4<R>& v) {
    if constexpr (sizeof(R) == 8) {
      const double sg = (e & 1) ? -1.0 : 1.0;
      acc[0] = fma(sg, v.x, acc[0]);
      acc[1] = fma(sg, v.y, acc[1]);
      acc[2] = fma(sg, v.z, acc[2]);
      acc[3] = fma(sg, v.w, acc[3]);
    } else {
      const unsigned sg = (unsigned)(e & 1) << 31;
      acc[0] += f2d_all(__uint_as_float(__float_as_uint(v.x) ^ sg));
      acc[1] += f2d_all(__uint_as_float(__float_as_uint(v.y) ^ sg));
      acc[2] += f2d_all(__uint_as_float(__float_as_uint(v.z) ^ sg));
      acc[3] += f2d_all(__uint_as_float(__float_as_uint(v.w) ^ sg));
    }
  };
  int k = k0;
  for (; k + 4 <= k1; k += 4) {
    const int e0 = __ldg(a.csr + k), e1 = __ldg(a.csr + k + 1), e2 = __ldg(a.csr + k + 2),
              e3 = __ldg(a.csr + k + 3);
    const R4<R> v0 = ld4<R>(flux + (size_t)(e0 >> 1) * B + b), v1 = ld4<R>(flux + (size_t)(e1 >> 1) * B + b),
                v2 = ld4<R>(flux + (size_t)(e2 >> 1) * B + b), v3 = ld4<R>(flux + (size_t)(e3 >> 1) * B + b);
    add(e0, v0); add(e1, v1); add(e2, v2); add(e3, v3);
  }
  for (; k < k1; ++k) {
    const int e = __ldg(a.csr + k);
    add(e, ld4<R>(flux + (size_t)(e >> 1) * B + b));
  }
}

// Flux application, one thread per (cell, bin): U <- U - c dt / V * sum of
// the cell's stored face fluxes.  Heun: the kernel handles Heun's stages
// (a.heun); the plain update is its own instantiation, without the stages'
// code (which the compiler would otherwise issue as predicated FP64
// instructions on every launch).
//
// FP64 sweep (R = double): the interleaved FP64 records, c dt / V divided
// as defined.  Mixed precision (R = float): c dt (1/V) with 1/V formed once
// per mesh (one FP64 multiply instead of a division per subcycle); N is
// updated in FP64 (radN) and the reduced flux in FP32 in the sweep record,
// whose N lane is then refreshed.  Comp: the face terms summed as an FP32
// pair (flux_sum_pair) and widened to FP64 once for N; otherwise summed in
// FP64 (flux_sum).
template <class R, bool Comp, bool Pred = false, bool Heun = false>
__global__ void __launch_bounds__(256) k_gather(CellArgs a, const R4<R>* __restrict__ flux,
                                                float4* __restrict__ shadow) {
  int t = blockIdx.x * blockDim.x + threadIdx.x;
  const int B = a.B;
  if (t >= (a.list ? a.n : a.C) * B) return;
  const int ii = divb(t, a.divB), b = t - ii * B;
  const int i = a.list ? __ldg(a.list + ii) : ii;
  t = i * B + b;
  if constexpr (sizeof(R) == 4) {
    // the state is loaded after the face sum (fewer registers live across
    // the loop)
    double N;
    float4 u;
    if constexpr (Comp) {
      float hi[4], lo[4];
      flux_sum_pair<Pred>(a, flux, i, b, hi, lo);
      const double kfac = a.lam * __ldg(a.ivol + i);
      N = a.radN[t];
      u = shadow[t];
      if (Heun && a.heun == 1) a.rad0[t] = make_d4(N, f2d_int(u.y), f2d_int(u.z), f2d_int(u.w));
      N -= kfac * (f2d_int(hi[0]) + f2d_int(lo[0]));
      const float kf = d2f_int(kfac);
      u.y = fmaf(-kf, hi[1], fmaf(-kf, lo[1], u.y));
      u.z = fmaf(-kf, hi[2], fmaf(-kf, lo[2], u.z));
      u.w = fmaf(-kf, hi[3], fmaf(-kf, lo[3], u.w));
    } else {
      double acc[4];
      flux_sum<float>(a, flux, i, b, acc);
      const double kfac = a.lam * __ldg(a.ivol + i);
      N = a.radN[t];
      u = shadow[t];
      if (Heun && a.heun == 1) a.rad0[t] = make_d4(N, f2d_int(u.y), f2d_int(u.z), f2d_int(u.w));
      N -= kfac * acc[0];
      u.y = d2f_int(f2d_int(u.y) - kfac * acc[1]);
      u.z = d2f_int(f2d_int(u.z) - kfac * acc[2]);
      u.w = d2f_int(f2d_int(u.w) - kfac * acc[3]);
    }
    if (Heun && a.heun == 2) {
      const d4 u0 = a.rad0[t];
      N = 0.5 * u0.x + 0.5 * N;
      u.y = d2f_int(0.5 * u0.y + 0.5 * f2d_int(u.y));
      u.z = d2f_int(0.5 * u0.z + 0.5 * f2d_int(u.z));
      u.w = d2f_int(0.5 * u0.w + 0.5 * f2d_int(u.w));
    }
    a.radN[t] = N;
    if (nonfinite_bits(N)) atomicOr(a.status, kStNonFinite);
    u.x = d2f_int(N);
    shadow[t] = u;
    return;
  } else {
    double acc[4];
    flux_sum<R>(a, flux, i, b, acc);
    const double kfac = a.lam / a.vol[i];
    d4 u = a.rad[t];
    if (Heun && a.heun == 1) a.rad0[t] = u;
    u.x -= kfac * acc[0];
    u.y -= kfac * acc[1];
    u.z -= kfac * acc[2];
    u.w -= kfac * acc[3];
    if (Heun && a.heun == 2) {
      const d4 u0 = a.rad0[t];
      u.x = 0.5 * u0.x + 0.5 * u.x;
      u.y = 0.5 * u0.y + 0.5 * u.y;
      u.z = 0.5 * u0.z + 0.5 * u.z;
      u.w = 0.5 * u0.w + 0.5 * u.w;
    }
    a.rad[t] = u;
    if (!isfinite(u.x)) atomicOr(a.status, kStNonFinite);
  }
}

__global__ void k_reciprocal(int n, const double* __restrict__ in, double* out) {
  const int k = blockIdx.x * blockDim.x + threadIdx.x;
  if (k < n) out[k] = 1.0 / in[k];
}

// Sources and thermochemistry, one thread per cell (Eq. E source term,
// Sec. 2.3.1, 4.1.1).  FP64 sweep: one kernel, the oracle's arithmetic.
// Mixed precision: two passes (the remedy Sec. 6.2 proposes for the
// divergence of the substep loop): k_chem_first makes the first attempt of
// every cell over the whole subcycle -- one attempt per lane, no divergence
// -- and finishes the cells it accepts; the cells it rejects go to a
// worklist that k_chem_rest works through with the adaptive loop.  Each
// cell makes the attempts one pass would make: the first pass converts
// between FP32 and FP64 on the integer pipe (it is bound by the FP64 pipe), as
// do the worklist's groups of lanes, its threads with the hardware's
// conversions (a few stiff cells run long serial chains of attempts there,
// bound by an attempt's latency); the two round alike but for exact ties and
// subnormal values.  The attempts
// carry N and the gas only; the flux is read at the end and scaled by the
// product of the accepted photon factors.

// The worklist's rule.  A group of lanes (rest_groups) makes an attempt in half
// the latency of a thread (rest_threads): 17 k against 35 k cycles in FP64.  But
// it costs the FP64 unit six times as much per cell, 6.4 k cycles against 1.1 k
// in a full warp.  Groups therefore win while the longest chain of attempts
// decides and lose where the list's whole work does: the line lies at a number
// of chains side by side, (attempts of all cells) / (attempts of the longest),
// of 2,700 in FP64 and 2,000 in the mixed path.  The chains are foretold by
// their first attempts: a quantity that has to change by the measure f in steps
// of f_s takes about ln(1 + f) / f_s of them.  The first pass adds these up and
// keeps the largest (rest_entry), in integers, so that the choice does not
// depend on the order of the list.  Foretold so, the line lies at 2,000 and
// 1,500.  ms by threads / by groups at (cells; foretold chains side by side):
// FP64 4.06 / 2.54 (12,074; 1,186), 10.6 / 11.8 (12,147; 1,853), 4.38 / 4.43
// (34,535; 2,575), 9.04 / 20.6 (21,511; 10,121), and for even chains 0.135 /
// 0.41 (12,167; 11,701); mixed 1.22 / 0.96, 3.16 / 3.62, 1.26 / 1.39, 2.53 / 5.75,
// 0.047 / 0.137.  Beyond the lengths below the sums are not looked at.
constexpr int kGroupMax64 = 49152, kGroupMaxMixed = 24576;
constexpr int kGroupSide64 = 2000, kGroupSideMixed = 1500;

// Entry of a rejected cell with measure f1 in the worklist whose counters are
// ctl: its place.  One addition per warp and counter.
__device__ __forceinline__ int rest_entry(int* ctl, float f1) {
  const int k = atomicAdd(ctl, 1);
  const int w = 1 + (int)(1000.0f * fminf(__log2f(1.0f + f1), 32.0f));   // 49,152 of them fit the sum
  const unsigned m = __activemask();
  const int sum = __reduce_add_sync(m, w), top = __reduce_max_sync(m, w);
  if ((int)(threadIdx.x & 31) == __ffs(m) - 1) {
    atomicAdd(ctl + 1, sum);
    atomicMax(ctl + 2, top);
  }
  return k;
}
__device__ __forceinline__ bool rest_by_groups(const int4& c, int most, int side) {
  return c.x <= most && c.y <= side * c.z;
}

// Worklist of the cells whose first attempt was rejected, and its counters:
// entries, sum and largest of the foretold chains (read together, as one
// 16-byte word), next entry to hand out, finished warps.
constexpr int kRestCtl = 5, kRestNext = 3, kRestDone = 4;
struct ChemWork {
  int32_t* cell;   // C
  float* f1;       // C: the rejected first attempt's measure
  int* ctl;        // kRestCtl counters
};

// Source term of Eq. (E) over the subcycle: the photons of the cell's
// sources (rates summed in source order) added to N.
__device__ __forceinline__ void inject_cell(const CellArgs& a, int i, int si, double N[kMaxBins]) {
  const double vcm3 = a.vol[i] * a.lu3;
#pragma unroll
  for (int b = 0; b < kMaxBins; ++b)
    if (b < a.B) N[b] += (a.src_rate[(size_t)si * a.B + b] * a.dt) / vcm3;
}

__device__ __forceinline__ void chem_load_mixed(const CellArgs& a, int i, GasState& s, bool inject) {
  const int B = a.B;
#pragma unroll
  for (int b = 0; b < kMaxBins; ++b)
    if (b < B) s.N[b] = a.radN[(size_t)i * B + b];
  if (inject) {
    const int si = a.src_idx[i];
    if (si >= 0) inject_cell(a, i, si, s.N);
  }
  const size_t C = a.C;
  s.xHI = a.x5[i]; s.xHII = a.x5[C + i]; s.yI = a.x5[2 * C + i]; s.yII = a.x5[3 * C + i];
  s.yIII = a.x5[4 * C + i]; s.T = a.T[i];
}

// Final state of a cell: N (FP64), the FP32 sweep record (N rounded, the
// reduced flux scaled by S in FP32), gas, attempt count.
__device__ __forceinline__ void chem_store_mixed(const CellArgs& a, int i, const GasState& s,
                                                 const float S[kMaxBins], int n, bool gas,
                                                 float4* __restrict__ shadow) {
  const int B = a.B;
  bool bad = false;
#pragma unroll
  for (int b = 0; b < kMaxBins; ++b) {
    if (b < B) {
      const size_t t = (size_t)i * B + b;
      a.radN[t] = s.N[b];
      float4 u = shadow[t];
      u.x = d2f_int(s.N[b]);
      u.y *= S[b]; u.z *= S[b]; u.w *= S[b];
      shadow[t] = u;
      if (nonfinite_bits(s.N[b])) bad = true;
    }
  }
  if (bad) atomicOr(a.status, kStNonFinite);
  if (gas) {
    const size_t C = a.C;
    a.nsub[i] = n;
    a.x5[i] = s.xHI; a.x5[C + i] = s.xHII; a.x5[2 * C + i] = s.yI; a.x5[3 * C + i] = s.yII;
    a.x5[4 * C + i] = s.yIII; a.T[i] = s.T;
  }
}

__global__ void __launch_bounds__(128, 6) k_chem_first(CellArgs a, ChemParams P, float4* __restrict__ shadow,
                                                    ChemWork w) {
  const int ii = blockIdx.x * blockDim.x + threadIdx.x;
  if (ii >= (a.list ? a.n : a.C)) return;
  const int i = a.list ? __ldg(a.list + ii) : ii;
  GasState s;
  float S[kMaxBins];
#pragma unroll
  for (int b = 0; b < kMaxBins; ++b) S[b] = 1.0f;
  chem_load_mixed(a, i, s, a.do_inject);
  if (!a.do_chem) {
    chem_store_mixed(a, i, s, S, 0, false, shadow);
    return;
  }
  float f1;
  if (chemistry_mixed_first(P, a.nH[i], a.dt, s, S, &f1)) {
    chem_store_mixed(a, i, s, S, 1, true, shadow);
    return;
  }
  // rejected: keep the injected photons, hand the cell to the second pass
#pragma unroll
  for (int b = 0; b < kMaxBins; ++b)
    if (b < a.B) a.radN[(size_t)i * a.B + b] = s.N[b];
  const int k = rest_entry(w.ctl, f1);
  w.cell[k] = i;
  w.f1[k] = f1;
}

// The last warp to finish resets the worklist's counters for the next
// subcycle.
__device__ __forceinline__ void rest_done(int* ctl) {
  __syncwarp();
  if ((threadIdx.x & 31) == 0) {
    __threadfence();
    if (atomicAdd(ctl + kRestDone, 1) == (int)(gridDim.x * (blockDim.x >> 5)) - 1) {
      for (int q = 0; q < kRestCtl; ++q) ctl[q] = 0;
      __threadfence();
    }
  }
}

// The next entry of the worklist for every group with need: its leader takes
// one.  The first entries are dealt out so that consecutive ones lie on
// different SMs.
__device__ __forceinline__ int group_first() {
  return (int)((threadIdx.x / kGroup) * gridDim.x + blockIdx.x);
}
__device__ __forceinline__ int group_next(int* ctl, bool need, int l) {
  int k = 0;
  if (need && l == 0) k = (int)(gridDim.x * (blockDim.x / kGroup)) + atomicAdd(ctl + kRestNext, 1);
  return from_lane(k, 0);
}

// A short worklist in the mixed path, one group of lanes per cell (the
// adaptive loop of chemistry_mixed, resumed after the rejected first attempt;
// both groups of a warp stay in step, an idle one repeating its last
// attempt).
__device__ __forceinline__ void rest_groups(const CellArgs& a, const ChemParams& P, float4* __restrict__ shadow,
                                            const ChemWork& w, int total) {
  const int l = threadIdx.x & (kGroup - 1), B = a.B;
  const size_t C = a.C;
  const LaneFitF fit = lane_fit_f(l, P.flags);
  GroupState s{{1.0, 0.0, 1.0, 0.0, 0.0}, 1e4, 0.0, 0.0}, t;
  GroupCell g;
  group_cell(P, l, 1.0, g);
  double rem = 0.0, dt = 0.0;
  float S = 1.0f;
  bool dark = false;   // the lane's bin came with N <= 0
  int i = 0, n = 0;
  const float fmx = (float)P.f_max, fs = (float)P.f_s;
  auto load = [&](int k) {
    i = w.cell[k];
    group_cell(P, l, a.nH[i], g);
#pragma unroll
    for (int q = 0; q < 5; ++q) s.x[q] = a.x5[q * C + i];
    s.T = a.T[i];
    s.N = l < B ? a.radN[(size_t)i * B + l] : 0.0;
    dark = unlit(s.N);
    rem = a.dt;
    dt = a.dt * f2d_int(__fdividef(fs, w.f1[k]));
    S = dark ? 0.0f : 1.0f;
    n = 1;
  };
  auto store = [&]() {
    if (__double_as_longlong(rem) == __double_as_longlong(a.dt)) S = 1.0f;   // nothing was accepted
    if (l < B) {
      const size_t r = (size_t)i * B + l;
      a.radN[r] = s.N;
      float4 u = shadow[r];
      u.x = d2f_int(s.N);
      u.y *= S; u.z *= S; u.w *= S;
      shadow[r] = u;
      if (nonfinite_bits(s.N)) atomicOr(a.status, kStNonFinite);
    }
#pragma unroll
    for (int q = 0; q < 5; ++q)
      if (l == q) a.x5[q * C + i] = s.x[q];
    if (l == 5) a.T[i] = s.T;
    if (l == 6) a.nsub[i] = n;
    if (l == 7 && rem > 0) atomicOr(a.status, kStChemSubsteps);
  };
  int k = group_first();
  bool have = k < total;
  if (have) load(k);
  for (;;) {
    const bool done = have && (!positive(rem) || n >= P.max_sub);
    if (__any_sync(kFull, done)) {
      if (done) store();
      k = group_next(w.ctl, done, l);
      if (done) {
        have = k < total;
        if (have) load(k);
      }
    } else {
      if (!__any_sync(kFull, have)) break;
      double sc;
      const float f = group_attempt<true>(P, fit, l, g, dt, s, t, sc);
      if (have) {
        ++n;
        if (f > fmx) {
          dt = dt * (double)__fdividef(fs, f);
        } else {
          s = t;
          s.N = dark ? 0.0 : t.N;
          S *= d2f_int(sc);
          rem = __double_as_longlong(dt) == __double_as_longlong(rem) ? 0.0 : rem - dt;
          dt = dt * (double)(f > 0.0f ? fminf(__fdividef(fs, f), 2.0f) : 2.0f);
          if (__double_as_longlong(dt) > __double_as_longlong(rem)) dt = rem;
        }
      }
    }
    __syncwarp();
  }
}

// The worklist's cells, one per thread, handed out 32 at a time to warps.
// The cells left after the first pass are few and stiff (each runs its own
// serial chain of attempts, and a warp runs as long as its slowest cell), so
// the first chunks go to warp 0 of every block -- one warp per SM, each with
// the SM's FP64 unit to itself -- then to warp 1 of every block, and so on;
// later chunks go to whichever warp is free.
__device__ __forceinline__ void rest_threads(const CellArgs& a, const ChemParams& P, float4* __restrict__ shadow,
                                             const ChemWork& w, int total) {
  const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
  const int n_warps = gridDim.x * (blockDim.x >> 5);
  // static first chunk: warp-in-block major, so that consecutive chunks lie
  // on different SMs; then dynamic chunks after all the static ones
  int chunk = wib * gridDim.x + blockIdx.x;
  for (;;) {
    const int k = chunk * 32 + lane;
    if (chunk * 32 >= total) break;
    if (k < total) {
      const int i = w.cell[k];
      GasState s;
      float S[kMaxBins];
      chem_load_mixed(a, i, s, false);
      bool capped;
      const double dt0 = a.dt * f2d_int(__fdividef((float)P.f_s, w.f1[k]));
      const int n = chemistry_mixed<false>(P, a.nH[i], a.dt, s, S, &capped, dt0, 1);
      if (capped) atomicOr(a.status, kStChemSubsteps);
      chem_store_mixed(a, i, s, S, n, true, shadow);
    }
    int next = 0;
    if (lane == 0) next = n_warps + atomicAdd(w.ctl + kRestNext, 1);
    chunk = __shfl_sync(0xffffffffu, next, 0);
  }
}

__global__ void __launch_bounds__(128) k_chem_rest(CellArgs a, ChemParams P, float4* __restrict__ shadow,
                                                   ChemWork w) {
  const int4 c = *reinterpret_cast<const int4*>(w.ctl);
  if (c.x == 0) return;   // nothing was rejected: the worklist's counters are all zero already
  if (rest_by_groups(c, kGroupMaxMixed, kGroupSideMixed)) rest_groups(a, P, shadow, w, c.x);
  else rest_threads(a, P, shadow, w, c.x);
  rest_done(w.ctl);
}

// FP64 path: a cell's state (radiation of every bin and gas) in and out.
__device__ __forceinline__ void chem_load64(const CellArgs& a, int i, CellState& s, bool inject) {
  const int B = a.B;
  const size_t C = a.C;
#pragma unroll
  for (int b = 0; b < kMaxBins; ++b) {
    if (b < B) {
      d4 v = a.rad[(size_t)i * B + b];
      s.N[b] = v.x; s.f[b][0] = v.y; s.f[b][1] = v.z; s.f[b][2] = v.w;
    }
  }
  if (inject) {
    const int si = a.src_idx[i];
    if (si >= 0) inject_cell(a, i, si, s.N);
  }
  s.xHI = a.x5[i]; s.xHII = a.x5[C + i]; s.yI = a.x5[2 * C + i]; s.yII = a.x5[3 * C + i];
  s.yIII = a.x5[4 * C + i]; s.T = a.T[i];
}
__device__ __forceinline__ void chem_store64(const CellArgs& a, int i, const CellState& s, bool gas) {
  const int B = a.B;
  const size_t C = a.C;
  if (gas) {
    a.x5[i] = s.xHI; a.x5[C + i] = s.xHII; a.x5[2 * C + i] = s.yI; a.x5[3 * C + i] = s.yII;
    a.x5[4 * C + i] = s.yIII; a.T[i] = s.T;
  }
  bool bad = false;
#pragma unroll
  for (int b = 0; b < kMaxBins; ++b) {
    if (b < B) {
      a.rad[(size_t)i * B + b] = make_d4(s.N[b], s.f[b][0], s.f[b][1], s.f[b][2]);
      if (!isfinite(s.N[b])) bad = true;
    }
  }
  if (bad) atomicOr(a.status, kStNonFinite);
}

// Tape of the reverse mode: one record per chemistry attempt of the cells
// whose first attempt was rejected (the worklist's cells), written by the
// forward's own worklist pass while the reverse mode recomputes a segment.
// A cell's records are linked backwards (prev); last[i] is the index of its
// last record, or -1 for a cell whose one attempt was accepted over the
// whole subcycle (its entering state is the recorded pre-chemistry state,
// and nothing downstream depends on its measure).  Records are handed out
// by one counter, so a subcycle's records are one contiguous range; past
// the capacity nothing is written, and the host, which reads the counter
// after each subcycle's chemistry, grows the tape and records that
// subcycle's chemistry again.
constexpr int kNv = 4 * kMaxBins + 6;

struct ChemRec {
  double s[kNv];     // state entering the attempt (N[B], f[3B], xHI, xHII, yI, yII, yIII, T)
  double dt, f;      // its length and measure
  int cell;
  int flags;         // kRecAccepted | kRecRatio (growth by f_s / f, not the cap) | kRecClipped (next length cut)
  int prev;          // the cell's previous record, -1 for its first
  int pad;
};
constexpr int kRecAccepted = 1, kRecRatio = 2, kRecClipped = 4;

struct ChemTape {
  ChemRec* rec;
  long long cap;
  unsigned long long* used;   // records handed out (may pass cap)
  int32_t* last;              // C, this subcycle's
};

__device__ __forceinline__ void pack_state(const CellState& c, int B, double* s) {
  for (int b = 0; b < B; ++b) {
    s[b] = c.N[b];
    s[B + 3 * b] = c.f[b][0]; s[B + 3 * b + 1] = c.f[b][1]; s[B + 3 * b + 2] = c.f[b][2];
  }
  s[4 * B] = c.xHI; s[4 * B + 1] = c.xHII; s[4 * B + 2] = c.yI; s[4 * B + 3] = c.yII; s[4 * B + 4] = c.yIII;
  s[4 * B + 5] = c.T;
}

// Records the attempts of one cell (the Tape of chemistry_loop).
struct TapeWriter {
  ChemTape t;
  int B, cell;
  int prev = -1;
  long long cur = 0;
  __device__ __forceinline__ void begin(const CellState& s, double dt, double) {
    cur = (long long)atomicAdd(t.used, 1ull);
    if (cur < t.cap) {
      ChemRec& r = t.rec[cur];
      pack_state(s, B, r.s);
      r.dt = dt;
    }
  }
  __device__ __forceinline__ void end(double f, bool accepted, bool ratio, bool clipped) {
    if (cur < t.cap) {
      ChemRec& r = t.rec[cur];
      r.f = f;
      r.cell = cell;
      r.flags = (accepted ? kRecAccepted : 0) | (ratio ? kRecRatio : 0) | (clipped ? kRecClipped : 0);
      r.prev = prev;
    }
    prev = cur < t.cap ? (int)cur : -1;
  }
};

// Sources and thermochemistry of the FP64 path in two passes, as the mixed
// path (Sec. 6.2's remedy for the divergence of the substep loop): the first
// attempt of every cell, then the rejected cells from a worklist.  The
// attempts of every cell are those of the single loop.
__global__ void __launch_bounds__(128) k_chem64_first(CellArgs a, ChemParams P, int32_t* __restrict__ work_cell,
                                                      double* __restrict__ work_f1, int* __restrict__ work_ctl) {
  const int ii = blockIdx.x * blockDim.x + threadIdx.x;
  if (ii >= (a.list ? a.n : a.C)) return;
  const int i = a.list ? __ldg(a.list + ii) : ii;
  CellState s;
  chem_load64(a, i, s, a.do_inject);
  if (!a.do_chem) {
    chem_store64(a, i, s, false);
    return;
  }
  double f1;
  if (chemistry_first(P, a.nH[i], a.dt, s, &f1)) {
    a.nsub[i] = 1;
    chem_store64(a, i, s, true);
    return;
  }
  // rejected: keep the injected photons, hand the cell to the second pass
#pragma unroll
  for (int b = 0; b < kMaxBins; ++b)
    if (b < a.B) a.rad[(size_t)i * a.B + b].x = s.N[b];
  const int k = rest_entry(work_ctl, (float)f1);
  work_cell[k] = i;
  work_f1[k] = f1;
}

// A short worklist in the FP64 path, one group of lanes per cell, as
// rest_groups.  kTape: also record every attempt, as rest_threads64.
template <bool kTape>
__device__ __forceinline__ void rest_groups64(const CellArgs& a, const ChemParams& P,
                                              const int32_t* __restrict__ work_cell,
                                              const double* __restrict__ work_f1, int* work_ctl, const ChemTape& tape,
                                              int total) {
  const int l = threadIdx.x & (kGroup - 1), B = a.B;
  const size_t C = a.C;
  const LaneFit fit = lane_fit(l, P.flags);
  GroupState s{{1.0, 0.0, 1.0, 0.0, 0.0}, 1e4, 0.0, 0.0}, t;
  GroupCell g;
  group_cell(P, l, 1.0, g);
  double rem = 0.0, dt = 0.0;
  double* rad = reinterpret_cast<double*>(a.rad);   // (N, f_x, f_y, f_z) per (cell, bin)
  int i = 0, n = 0;
  int prev = -1;            // kTape: the cell's last record (the leader's)
  auto load = [&](int k) {
    i = work_cell[k];
    group_cell(P, l, a.nH[i], g);
#pragma unroll
    for (int q = 0; q < 5; ++q) s.x[q] = a.x5[q * C + i];
    s.T = a.T[i];
    const double* r = rad + (size_t)i * B * 4;
    s.N = l < B ? r[4 * l] : 0.0;
    s.f = l < 3 * B ? r[4 * (l / 3) + 1 + l % 3] : 0.0;
    rem = a.dt;
    n = 1;
  };
  auto store = [&]() {
    double* r = rad + (size_t)i * B * 4;
    if (l < B) {
      r[4 * l] = s.N;
      if (!isfinite(s.N)) atomicOr(a.status, kStNonFinite);
    }
    if (l < 3 * B) r[4 * (l / 3) + 1 + l % 3] = s.f;
#pragma unroll
    for (int q = 0; q < 5; ++q)
      if (l == q) a.x5[q * C + i] = s.x[q];
    if (l == 5) a.T[i] = s.T;
    if (l == 6) a.nsub[i] = n;
    if (l == 7 && rem > 0) atomicOr(a.status, kStChemSubsteps);
    if (kTape && l == 0) tape.last[i] = prev;
  };
  // one record of the attempts of each group with rec (past the capacity
  // nothing is written, the counter still runs): the leader hands it out, the
  // lanes write the entering state
  auto begin = [&](bool rec) -> long long {
    long long cur = 0;
    if (rec && l == 0) cur = (long long)atomicAdd(tape.used, 1ull);
    cur = from_lane(cur, 0);
    if (rec && cur < tape.cap) {
      ChemRec& r = tape.rec[cur];
      if (l < B) r.s[l] = s.N;
      if (l < 3 * B) r.s[B + l] = s.f;
#pragma unroll
      for (int q = 0; q < 5; ++q)
        if (l == q) r.s[4 * B + q] = s.x[q];
      if (l == 5) r.s[4 * B + 5] = s.T;
    }
    return cur;
  };
  auto end = [&](long long cur, double len, double f, int flags) {
    if (l == 0 && cur < tape.cap) {
      ChemRec& r = tape.rec[cur];
      r.dt = len; r.f = f; r.cell = i; r.flags = flags; r.prev = prev;
    }
    prev = cur < tape.cap ? (int)cur : -1;
  };
  // a new cell: its rejected first attempt is recorded too
  auto take = [&](bool fresh, int k) {
    if (fresh) load(k);
    if constexpr (kTape) {
      const long long cur = begin(fresh);
      if (fresh) {
        prev = -1;
        end(cur, a.dt, work_f1[k], 0);
      }
    }
    if (fresh) dt = a.dt * div_nr(P.f_s, work_f1[k]);
  };
  int k = group_first();
  bool have = k < total;
  take(have, k);
  for (;;) {
    const bool done = have && (!(rem > 0) || n >= P.max_sub);
    if (__any_sync(kFull, done)) {
      if (done) store();
      k = group_next(work_ctl, done, l);
      if (done) have = k < total;
      take(done && have, k);
    } else {
      if (!__any_sync(kFull, have)) break;
      long long cur = 0;
      if constexpr (kTape) cur = begin(have);
      double sc;
      const double f = group_attempt<false>(P, fit, l, g, dt, s, t, sc);
      if (have) {
        ++n;
        if (f > P.f_max) {
          if constexpr (kTape) end(cur, dt, f, 0);
          dt = dt * div_nr(P.f_s, f);
        } else {
          s = t;
          const double len = dt;
          rem = (dt == rem) ? 0.0 : rem - dt;
          double grow = (f > 0) ? div_nr(P.f_s, f) : 2.0;
          const bool ratio = f > 0 && grow <= 2.0;
          if (grow > 2.0) grow = 2.0;
          dt = dt * grow;
          const bool clipped = dt > rem;
          if (clipped) dt = rem;
          if constexpr (kTape)
            end(cur, len, f, kRecAccepted | (ratio ? kRecRatio : 0) | (clipped ? kRecClipped : 0));
        }
      }
    }
    __syncwarp();
  }
}

// The FP64 worklist, one cell per thread, handed out as rest_threads.
// kTape: also record every attempt of these cells, the rejected first one
// included, for the reverse mode.
template <bool kTape>
__device__ __forceinline__ void rest_threads64(const CellArgs& a, const ChemParams& P,
                                               const int32_t* __restrict__ work_cell,
                                               const double* __restrict__ work_f1, int* work_ctl,
                                               const ChemTape& tape, int total) {
  const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
  const int n_warps = gridDim.x * (blockDim.x >> 5);
  int chunk = wib * gridDim.x + blockIdx.x;
  for (;;) {
    const int k = chunk * 32 + lane;
    if (chunk * 32 >= total) break;
    if (k < total) {
      const int i = work_cell[k];
      CellState s;
      chem_load64(a, i, s, false);
      bool capped;
      const double dt0 = a.dt * div_nr(P.f_s, work_f1[k]);
      int n;
      if constexpr (kTape) {
        TapeWriter tw{tape, a.B, i};
        tw.begin(s, a.dt, a.dt);   // the first attempt, made and rejected by k_chem64_first
        tw.end(work_f1[k], false, false, false);
        n = chemistry_loop(P, a.nH[i], a.dt, s, &capped, dt0, 1, tw);
        tape.last[i] = tw.prev;
      } else {
        n = chemistry(P, a.nH[i], a.dt, s, &capped, dt0, 1);
      }
      a.nsub[i] = n;
      if (capped) atomicOr(a.status, kStChemSubsteps);
      chem_store64(a, i, s, true);
    }
    int next = 0;
    if (lane == 0) next = n_warps + atomicAdd(work_ctl + kRestNext, 1);
    chunk = __shfl_sync(0xffffffffu, next, 0);
  }
}

template <bool kTape>
__global__ void __launch_bounds__(128) k_chem64_rest(CellArgs a, ChemParams P, const int32_t* __restrict__ work_cell,
                                                     const double* __restrict__ work_f1, int* work_ctl,
                                                     ChemTape tape) {
  const int4 c = *reinterpret_cast<const int4*>(work_ctl);
  if (c.x == 0) return;   // nothing was rejected: the worklist's counters are all zero already
  if (rest_by_groups(c, kGroupMax64, kGroupSide64))
    rest_groups64<kTape>(a, P, work_cell, work_f1, work_ctl, tape, c.x);
  else rest_threads64<kTape>(a, P, work_cell, work_f1, work_ctl, tape, c.x);
  rest_done(work_ctl);
}

}  // namespace m1rt

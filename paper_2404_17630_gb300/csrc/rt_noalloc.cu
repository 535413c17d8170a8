// rt_gradients_noalloc: limited least-squares gradients for callers that
// cannot allocate device memory.
//
// Who needs it: code that runs where cudaMalloc is not available or not
// allowed -- inside a host framework that owns all device memory through its
// own pool, in a real-time loop that must not allocate, or in a plug-in that
// only receives device pointers.  Such a caller cannot create an rt_ctx
// (rt_init_mesh allocates), so this entry point takes the whole mesh and state
// as caller-owned device arrays and needs no device memory of its own: a block
// keeps its cells' geometry in shared memory.
#include <cstdint>
#include <cstdio>

#include <cuda_runtime.h>

#include "../../include/rt.h"
#include "rt_limiter.cuh"

namespace {

// The interface's limit on the mesh (what the entry point has always refused).
constexpr int64_t kNoallocMaxCells = 262144;

// Kernel launch that returns this launch's own status (a triple-chevron
// launch only leaves it in the thread's last-error slot, where an error the
// caller left pending is indistinguishable from it).
template <class T> struct ident { using type = T; };
template <class... KA>
cudaError_t launch(void (*k)(KA...), dim3 grid, dim3 block, size_t smem, cudaStream_t s,
                   typename ident<KA>::type... args) {
  void* p[] = {(void*)&args...};
  return cudaLaunchKernel((const void*)k, grid, block, p, smem, s);
}

thread_local char g_err[256];

rt_status set_err(rt_status st, const char* msg) {
  snprintf(g_err, sizeof g_err, "%s", msg);
  return st;
}

using namespace m1rt;

struct NoallocArgs {
  int C, B;
  Box box;
  int limiter;
  double lim_eps2;
  const int32_t *off, *csr, *left, *right;
  const double *cx, *cy, *cz, *area, *fx, *fy, *fz, *N, *F;
  double* G;
  int* bad;
};

// Half-edge k of cell i: the weight w = A d / |d|^2 towards the neighbour j and
// the face-centre offset x with |x|^2.
struct HalfEdge {
  d4 w, x;   // w.w: the neighbour id's bits
};
__device__ __forceinline__ HalfEdge half_edge(const NoallocArgs& a, int i, int k, double d[3]) {
  const int e = a.csr[k], f = e >> 1;
  const int j = (e & 1) ? a.left[f] : a.right[f];
  const double c0 = a.cx[i], c1 = a.cy[i], c2 = a.cz[i];
  d[0] = min_image(a.cx[j] - c0, a.box);
  d[1] = min_image(a.cy[j] - c1, a.box);
  d[2] = min_image(a.cz[j] - c2, a.box);
  const double s = div_nr(a.area[f], d[0] * d[0] + d[1] * d[1] + d[2] * d[2]);
  HalfEdge h;
  h.w = make_d4(s * d[0], s * d[1], s * d[2], id_bits(j, 0.0));
  const double x0 = min_image(a.fx[f] - c0, a.box), x1 = min_image(a.fy[f] - c1, a.box), x2 = min_image(a.fz[f] - c2, a.box);
  h.x = make_d4(x0, x1, x2, x0 * x0 + x1 * x1 + x2 * x2);
  return h;
}

__device__ __forceinline__ void add_matrix(const HalfEdge& h, const double d[3], double m[6]) {
  // A n n^T = w d^T with n = d / |d|
  m[0] += h.w.x * d[0]; m[1] += h.w.x * d[1]; m[2] += h.w.x * d[2];
  m[3] += h.w.y * d[1]; m[4] += h.w.y * d[2]; m[5] += h.w.z * d[2];
}

// A block's cells, and the half-edges it can hold in shared memory: the weight
// and offset records, the offsets in FP32 and the partial matrices.
constexpr int kNaCells = 32, kNaCap = 640;
constexpr size_t kNaSmem = kNaCap * (2 * sizeof(d4) + sizeof(float4)) + kNaCells * 3 * 6 * sizeof(double);

// Least-squares sums and slope limiter, one thread per (cell, bin).  The
// geometry is formed once per half-edge: the threads of a cell take its
// half-edges in turn, leave their records in shared memory and add up M =
// sum A n n^T; each bin then reads the records.  The kernel is bound by the
// FP64 unit (about 1.7 k FP64 instructions per cell of 15.4 faces and three
// bins; with the geometry formed per bin and per pass, its divisions and the
// limiter's quotient per face and component 13 k): 3.22 -> 0.39 ms at 91,125
// cells.  With lengths beyond 1e18 or below 1e-18 the limiter does without its
// FP32 search: 281 -> 371 us at 64,000 cells.  A block whose cells have more
// than kNaCap half-edges forms them anew at each use.
__global__ void __launch_bounds__(kNaCells * 3) k_noalloc_grad(NoallocArgs a) {
  extern __shared__ __align__(32) unsigned char smem[];
  d4* sw = reinterpret_cast<d4*>(smem);
  d4* sx = sw + kNaCap;
  float4* sf = reinterpret_cast<float4*>(sx + kNaCap);
  double* sm = reinterpret_cast<double*>(sf + kNaCap);
  const int B = a.B, C = a.C;
  const int cl = threadIdx.x / B, b = threadIdx.x - cl * B;
  const int c0 = blockIdx.x * kNaCells, c1 = min(c0 + kNaCells, C), i = c0 + cl;
  const int kb = a.off[c0], n = a.off[c1] - kb;
  const bool act = i < c1, staged = n <= kNaCap;
  const int k0 = act ? a.off[i] : 0, k1 = act ? a.off[i + 1] : 0;
  double m[6] = {0.0, 0.0, 0.0, 0.0, 0.0, 0.0}, d[3];
  if (staged) {
    for (int k = k0 + b; k < k1; k += B) {
      const HalfEdge h = half_edge(a, i, k, d);
      add_matrix(h, d, m);
      sw[k - kb] = h.w;
      sx[k - kb] = h.x;
      sf[k - kb] = make_float4((float)h.x.x, (float)h.x.y, (float)h.x.z, 0.f);
    }
#pragma unroll
    for (int q = 0; q < 6; ++q) sm[threadIdx.x * 6 + q] = m[q];
    __syncthreads();
    if (!act) return;
#pragma unroll
    for (int q = 0; q < 6; ++q) {
      m[q] = sm[cl * B * 6 + q];
      for (int p = 1; p < B; ++p) m[q] += sm[(cl * B + p) * 6 + q];
    }
  } else {
    if (!act) return;
    for (int k = k0; k < k1; ++k) {
      const HalfEdge h = half_edge(a, i, k, d);
      add_matrix(h, d, m);
    }
  }
  // inverse of M
  const double v00 = m[3] * m[5] - m[4] * m[4], v01 = m[4] * m[2] - m[1] * m[5], v02 = m[1] * m[4] - m[3] * m[2];
  const double det = m[0] * v00 + m[1] * v01 + m[2] * v02;
  double* Go = a.G + ((size_t)i * B + b) * 12;
  if (!(det != 0.0) || !isfinite(det)) {
    atomicExch(a.bad, 1);
#pragma unroll
    for (int q = 0; q < 12; ++q) Go[q] = 0.0;
    return;
  }
  const double idet = 1.0 / det;
  const double i00 = v00 * idet, i01 = v01 * idet, i02 = v02 * idet, i11 = (m[0] * m[5] - m[2] * m[2]) * idet,
               i12 = (m[2] * m[1] - m[0] * m[4]) * idet, i22 = (m[0] * m[3] - m[1] * m[1]) * idet;
  const double* f[4] = {a.N + (size_t)b * C, a.F + (size_t)(3 * b) * C, a.F + (size_t)(3 * b + 1) * C,
                        a.F + (size_t)(3 * b + 2) * C};
  double pi[4], r[4][3];
  long long up[4], dn[4];   // largest and most negative difference to a neighbour, as bits
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    pi[q] = f[q][i];
    r[q][0] = r[q][1] = r[q][2] = 0.0;
    up[q] = dn[q] = 0;
  }
  long long X = 0;          // largest |x_f|^2
  for (int k = k0; k < k1; ++k) {
    HalfEdge h;
    if (staged) {
      h.w = sw[k - kb];
      h.x = sx[k - kb];
    } else {
      h = half_edge(a, i, k, d);
    }
    const int j = bits_id(h.w.w);
    X = __double_as_longlong(h.x.w) > X ? __double_as_longlong(h.x.w) : X;
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const double dphi = f[q][j] - pi[q];
      r[q][0] += h.w.x * dphi;
      r[q][1] += h.w.y * dphi;
      r[q][2] += h.w.z * dphi;
      up[q] = max_bits_pos(up[q], dphi);
      dn[q] = max_bits_neg(dn[q], dphi);
    }
  }
  double g[4][3], psi[4];
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    g[q][0] = i00 * r[q][0] + i01 * r[q][1] + i02 * r[q][2];
    g[q][1] = i01 * r[q][0] + i11 * r[q][1] + i12 * r[q][2];
    g[q][2] = i02 * r[q][0] + i12 * r[q][1] + i22 * r[q][2];
    psi[q] = 1.0;
  }
  if (a.limiter) {
    double dpos[4], dneg[4];
    if (staged) {
      int at[8];
      // offsets that FP32 holds, with their squares (in cm a cell of 1e19 does not: every face's product in FP64)
      float xm = sqrtf((float)__longlong_as_double(X));
      if (!(xm > 1e-18f && xm < 1e18f)) xm = nanf("");
      lim_extremes(sx, sf, k0 - kb, k1 - kb, g, a.lim_eps2, __longlong_as_double(X), xm, dpos, dneg, at);
    } else {
      long long p[4] = {0, 0, 0, 0}, q4[4] = {0, 0, 0, 0};
      double thr[4];
#pragma unroll
      for (int q = 0; q < 4; ++q)
        thr[q] = a.lim_eps2 * (g[q][0] * g[q][0] + g[q][1] * g[q][1] + g[q][2] * g[q][2]);
      for (int k = k0; k < k1; ++k) {
        const d4 x = half_edge(a, i, k, d).x;
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          const double dphi = g[q][0] * x.x + g[q][1] * x.y + g[q][2] * x.z;
          if (__double_as_longlong(dphi * dphi) > __double_as_longlong(thr[q] * x.w)) {
            p[q] = max_bits_pos(p[q], dphi);
            q4[q] = max_bits_neg(q4[q], dphi);
          }
        }
      }
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        dpos[q] = __longlong_as_double(p[q]);
        dneg[q] = neg_from_bits(q4[q]);
      }
    }
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      // the smallest quotient is the one by the largest g . x: rounded division
      // is monotone in the divisor
      if (limits_pos(__longlong_as_double(up[q]), dpos[q])) {
        const double lim = div_nr(__longlong_as_double(up[q]), dpos[q]);
        psi[q] = gt_nonneg(psi[q], lim) ? lim : psi[q];
      }
      if (limits_neg(neg_from_bits(dn[q]), dneg[q])) {
        const double lim = div_nr(neg_from_bits(dn[q]), dneg[q]);
        psi[q] = gt_nonneg(psi[q], lim) ? lim : psi[q];
      }
    }
  }
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    Go[3 * q + 0] = g[q][0] * psi[q];
    Go[3 * q + 1] = g[q][1] * psi[q];
    Go[3 * q + 2] = g[q][2] * psi[q];
  }
}

// Device memory of the current device `dev`, or managed memory.  Device memory
// of another GPU is refused: the kernels run on `dev` and would otherwise read
// another GPU's memory (a fault, or peer traffic where peer access is on).
bool on_device(const void* p, int dev) {
  cudaPointerAttributes a;
  if (cudaPointerGetAttributes(&a, p) != cudaSuccess) {
    cudaGetLastError();
    return false;
  }
  if (a.type == cudaMemoryTypeManaged) return true;
  return a.type == cudaMemoryTypeDevice && a.device == dev;
}

}  // namespace

extern "C" {

rt_status rt_gradients_noalloc(const rt_cells* cells, const rt_faces* faces, const int32_t* cell_off,
                               const int32_t* cell_faces, int n_bins, int order, int limiter, double lim_eps,
                               double box, const double* N, const double* F_red, double* G, int* bad_cell,
                               void* stream) {
  if (!cells || !faces || !cell_off || !cell_faces || !N || !F_red || !G || !bad_cell)
    return set_err(RT_INVALID_ARG, "rt_gradients_noalloc: NULL argument");
  if (n_bins < 1 || n_bins > 3 || order < 1 || order > 2 || lim_eps < 0 || box < 0)
    return set_err(RT_INVALID_ARG, "rt_gradients_noalloc: bad n_bins, order, lim_eps or box");
  const int64_t C = cells->n, F = faces->n;
  if (C <= 0 || F <= 0) return set_err(RT_INVALID_ARG, "rt_gradients_noalloc: empty mesh");
  if (C > kNoallocMaxCells)
    return set_err(RT_INVALID_ARG, "rt_gradients_noalloc: more than 262144 cells (larger meshes through a context)");
  if (F > (1LL << 29)) return set_err(RT_INVALID_ARG, "rt_gradients_noalloc: too many faces");
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) {
    cudaGetLastError();
    return set_err(RT_CUDA, "rt_gradients_noalloc: no current device");
  }
  const void* dev_ptrs[] = {cells->cx, cells->cy, cells->cz, faces->left, faces->right, faces->area, faces->fx,
                            faces->fy, faces->fz, cell_off, cell_faces, N, F_red, G, bad_cell};
  for (const void* p : dev_ptrs)
    if (!p || !on_device(p, dev))
      return set_err(RT_INVALID_ARG, "rt_gradients_noalloc: every array must be device memory of the current device");
  cudaStream_t s = (cudaStream_t)stream;
  const int Ci = (int)C;
  if (order < 2) {
    if (cudaMemsetAsync(G, 0, (size_t)C * n_bins * 12 * sizeof(double), s) != cudaSuccess ||
        cudaMemsetAsync(bad_cell, 0, sizeof(int), s) != cudaSuccess) {
      cudaGetLastError();
      return set_err(RT_CUDA, "rt_gradients_noalloc: memset failed");
    }
    return RT_OK;
  }
  if (cudaMemsetAsync(bad_cell, 0, sizeof(int), s) != cudaSuccess) {
    cudaGetLastError();
    return set_err(RT_CUDA, "rt_gradients_noalloc: memset failed");
  }
  NoallocArgs a{};
  a.C = Ci; a.B = n_bins; a.box = make_box(box);
  a.limiter = limiter; a.lim_eps2 = lim_eps * lim_eps;
  a.off = cell_off; a.csr = cell_faces; a.left = faces->left; a.right = faces->right;
  a.cx = cells->cx; a.cy = cells->cy; a.cz = cells->cz; a.area = faces->area;
  a.fx = faces->fx; a.fy = faces->fy; a.fz = faces->fz; a.N = N; a.F = F_red; a.G = G; a.bad = bad_cell;
  cudaError_t e = cudaFuncSetAttribute(k_noalloc_grad, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kNaSmem);
  if (e == cudaSuccess)
    e = launch(k_noalloc_grad, dim3((unsigned)((Ci + kNaCells - 1) / kNaCells)), dim3(kNaCells * n_bins), kNaSmem,
               s, a);
  if (e != cudaSuccess) {
    cudaGetLastError();   // the failed launch's own error
    return set_err(RT_CUDA, cudaGetErrorString(e));
  }
  return RT_OK;
}

const char* rt_noalloc_last_error(void) { return g_err; }

}  // extern "C"

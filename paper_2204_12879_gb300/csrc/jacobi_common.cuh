// jacobi_common.cuh -- device helpers of the one-sided Jacobi SVT shared by
// the blocked kernel (jacobi_blk.cu) and the per-slice kernels (svt.cu).
#pragma once
#include "lrstv_internal.cuh"

namespace lrstv {
namespace {

__device__ __forceinline__ void pair_of(int r, int i, int np, int &p, int &q) {
  if (i == 0) {
    p = r;
    q = np - 1;
  } else {
    p = (r + i) % (np - 1);
    q = (r - i + np - 1) % (np - 1);
  }
}

__device__ __forceinline__ float warp_sum(float v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// 1/sqrt(x) to about an ulp: the MUFU estimate refined by one Newton step.
__device__ __forceinline__ float rsqrt_nr(float x) {
  const float y = rsqrtf(x);
  return y * fmaf(-0.5f * x * y, y, 1.5f);
}

// Loads of W and V that another SM may have written during the same launch
// (the blocked kernel's tasks) bypass L1, which is not coherent across SMs.
template <bool CG>
__device__ __forceinline__ float2 ldw(const float2 *p) {
  return CG ? __ldcg(p) : *p;
}

// This thread's share of sum |x_e|^2 over n complex values (e = thread,
// thread + blockDim.x, ...), in four chains so that four loads are in flight.
__device__ __forceinline__ float sumsq4(const float2 *x, size_t n) {
  const size_t T = blockDim.x;
  float p0 = 0.0f, p1 = 0.0f, p2 = 0.0f, p3 = 0.0f;
  size_t e = threadIdx.x;
  for (; e + 3 * T < n; e += 4 * T) {
    const float2 a = x[e], b = x[e + T], c = x[e + 2 * T],
                 d = x[e + 3 * T];
    p0 = fmaf(a.x, a.x, fmaf(a.y, a.y, p0));
    p1 = fmaf(b.x, b.x, fmaf(b.y, b.y, p1));
    p2 = fmaf(c.x, c.x, fmaf(c.y, c.y, p2));
    p3 = fmaf(d.x, d.x, fmaf(d.y, d.y, p3));
  }
  for (; e < n; e += T) {
    const float2 a = x[e];
    p0 = fmaf(a.x, a.x, fmaf(a.y, a.y, p0));
  }
  return (p0 + p1) + (p2 + p3);
}

// Per-slice set-up of a packed Jacobi run by the whole CTA: V := I unless warm
// (warm: V holds the basis W was multiplied by), then ||W||_F^2, returned to
// every thread (s_red: 32 floats of shared memory).
__device__ __forceinline__ float pk_setup(int nr, int nc, const float2 *W, float2 *V, int warm,
                                          float *s_red) {
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  if (!warm)
    for (int e = tid; e < nc * nc; e += blockDim.x)
      V[e] = make_float2((e % nc) == (e / nc) ? 1.0f : 0.0f, 0.0f);
  float part = sumsq4(W, (size_t)nr * nc);
  part = warp_sum(part);
  if (lane == 0) s_red[warp] = part;
  __syncthreads();
  if (warp == 0) {
    float v = lane < (int)(blockDim.x >> 5) ? s_red[lane] : 0.0f;
    v = warp_sum(v);
    if (lane == 0) s_red[0] = v;
  }
  __syncthreads();
  const float fro2 = s_red[0];
  __syncthreads();
  return fro2;
}

// A pair left with relative inner product g moves the SVT result by at most
// about t g (both values kept: t g s_p / (s_p + s_q); one kept: g s_cut <= t g;
// both cut: nothing), so with the threshold t below the columns' RMS norm the
// relative tolerance is raised to tol rms / t: the absolute error stays at
// the level tol rms that a threshold near the RMS norm already allows.  The
// RMS norm is the largest over the slices of one tensor when it is given
// (ms2 >= 0): the inverse DFT mixes the slices, so all of them are resolved to
// the same absolute precision.
__device__ __forceinline__ float pk_tolerance(float tol, float fro2, int nc, float skip_t,
                                              float gms2) {
  if (skip_t > 0.0f && nc > 0) {
    const float ms2 = gms2 >= 0.0f ? gms2 : fro2 / (float)nc;
    tol = fmaxf(tol, tol * (sqrtf(ms2) / skip_t));
  }
  return tol;
}

// |w|^2 of a column by one warp, in the order of every epilogue
template <bool CG>
__device__ __forceinline__ float column_norm2(int nr, const float2 *w) {
  float n2 = 0.f;
  for (int row = threadIdx.x & 31; row < nr; row += 32) {
    const float2 x = ldw<CG>(w + row);
    n2 = fmaf(x.x, x.x, fmaf(x.y, x.y, n2));
  }
  return warp_sum(n2);
}

// g = max(1 - t / sigma, 0) of a column of squared norm n2; the sigma-vs-t decision
// is taken in FP64.
__device__ __forceinline__ float gain(float n2, float t) {
  const double sigma = sqrt((double)n2);
  return sigma > (double)t ? (float)(1.0 - (double)t / sigma) : 0.0f;
}

// g_i = max(1 - t / sigma_i, 0) applied to V's columns (t < 0: V unscaled).
template <bool CG>
__device__ __forceinline__ void pk_epilogue(int nr, int nc, const float2 *W, float2 *V, float t) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  if (t < 0.0f) return;
  for (int i = warp; i < nc; i += (int)(blockDim.x >> 5)) {
    const float g = gain(column_norm2<CG>(nr, W + (size_t)nr * i), t);
    float2 *vi = V + (size_t)nc * i;
    for (int row = lane; row < nc; row += 32) {
      const float2 v = ldw<CG>(vi + row);
      vi[row] = make_float2(v.x * g, v.y * g);
    }
  }
}

// The order of a slice's columns for its next sweep, by the whole CTA: by
// decreasing squared norm, ties by index (the norm-sorted ordering that de
// Rijk proposed for one-sided Jacobi, 1989: sweeps that pair the large
// columns first converge in fewer sweeps).  key: nc squared norms in shared
// memory (a NaN or a negative value sorts as 0); perm[rank] = column.  The
// ranks are counted, not sorted, so ties and the result are deterministic.
__device__ void order_columns(int nc, float *key, int *perm) {
  for (int i = threadIdx.x; i < nc; i += blockDim.x) {
    const float v = key[i];
    key[i] = v > 0.0f ? v : 0.0f;
  }
  __syncthreads();
  for (int i = threadIdx.x; i < nc; i += blockDim.x) {
    const float ki = key[i];
    int rank = 0;
    for (int j = 0; j < nc; ++j) {
      const float kj = key[j];
      rank += (kj > ki) || (kj == ki && j < i);
    }
    perm[rank] = i;
  }
}

}  // namespace
}  // namespace lrstv

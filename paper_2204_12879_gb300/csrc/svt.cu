// svt.cu -- the small kernels around the t-SVT's Jacobi (arXiv 2204.12879, eq.
// E_solution; the slice-wise form follows Theorem 4.2's t-SVD): the RMS norms,
// the Gram pre-check, sigma and V diag g; and the FP32 one-sided Jacobi of slices
// with few columns, of the calls without a task queue's scratch (slices of up to 256
// rows) and of the Tucker L-update's eigen-solves, one CTA each.
//
// The FP32 Jacobi orthogonalises a working matrix W (nr x nc complex, nr >= nc)
// by one-sided (Hestenes) rotations of column pairs (p, q) until
// |w_p^H w_q| <= tol |w_p| |w_q|.  The rotations accumulate in V, so W = A V
// has orthogonal columns sigma_i u_i.  One CTA per matrix; the sweep loop is
// capped and a matrix that reaches the cap reports it.  Two kernels share the
// rotation formula and differ in how columns move:
//  - k_jacobi_pk (nr <= 256): 32-column panels staged in
//    shared memory, a panel's W and V columns held in registers while later
//    panels stream past, one column pair per half-warp, paired FP32
//    instructions (__ffma2_rn) on a split row-pair layout;
//  - k_jacobi (257 to 512 rows): round-robin over all columns in global memory
//    (L2-resident), one pair per warp.
// The other Fourier slices' SVDs are jacobi_blk.cu's.
#include <float.h>

#include "jacobi_common.cuh"

namespace lrstv {

namespace {

// Whether a slice needs no sweep, with the sweeps to report: every singular value
// is at most ||W||_F, so at or below the threshold the SVT is zero whatever the
// sweeps would find (0); or the Gram check showed that one would rotate no pair (1).
__device__ __forceinline__ bool slice_known(float fro2, const JacOpt &o, int slice, int &sweeps) {
  if (o.t_svt >= 0.0f && fro2 <= o.t_svt * o.t_svt) {
    sweeps = 0;
    return true;
  }
  if (o.conv && o.conv[slice]) {
    sweeps = 1;
    return true;
  }
  return false;
}

__global__ void __launch_bounds__(512)
    k_jacobi(int nr, int nc, size_t wstride, size_t vstride, float2 *W_all, float2 *V_all,
             float t, int max_sweeps, float tol, float negl_rel, int *__restrict__ sweeps_out,
             unsigned long long *__restrict__ work, JacOpt o) {
  constexpr int R = 16;  // rows a lane
  const int warm = o.warm;
  float2 *W = W_all + (size_t)blockIdx.x * wstride;
  float2 *V = V_all + (size_t)blockIdx.x * vstride;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nwarps = blockDim.x >> 5;
  __shared__ float s_red[32];
  __shared__ int s_rot;

  if (!warm)  // warm: V holds the basis W was multiplied by
    for (int e = tid; e < nc * nc; e += blockDim.x)
      V[e] = make_float2((e % nc) == (e / nc) ? 1.0f : 0.0f, 0.0f);

  // ||W||_F^2: columns whose squared norm is below negl_rel ||W||_F^2 are
  // rounding residue and take part in no rotation.
  float part = 0.0f;
  for (size_t e = tid; e < (size_t)nr * nc; e += blockDim.x) {
    const float2 x = W[e];
    part = fmaf(x.x, x.x, fmaf(x.y, x.y, part));
  }
  part = warp_sum(part);
  if (lane == 0) s_red[warp] = part;
  __syncthreads();
  if (warp == 0) {
    float v = lane < nwarps ? s_red[lane] : 0.0f;
    v = warp_sum(v);
    if (lane == 0) s_red[0] = v;
  }
  __syncthreads();
  const float fro2 = s_red[0], negl = negl_rel * fro2;

  const int np = nc + (nc & 1);
  unsigned long long n_pairs = 0, n_rot = 0;  // counted by lane 0 of each warp
  // a slice with fewer than two columns is diagonal already: one empty sweep
  int sweeps = (nc < 2) ? 1 : 0;
  bool converged = slice_known(fro2, o, blockIdx.x, sweeps) || nc < 2;
  tol = pk_tolerance(tol, fro2, nc, o.t_svt, o.ms2 ? o.ms2[blockIdx.x / o.group] : -1.0f);
  for (int sweep = 1; sweep <= max_sweeps && !converged; ++sweep) {
    if (tid == 0) s_rot = 0;
    __syncthreads();
    for (int r = 0; r < np - 1; ++r) {
      for (int pr = warp; pr < np / 2; pr += nwarps) {
        int p, q;
        pair_of(r, pr, np, p, q);
        if (p >= nc || q >= nc) continue;
        n_pairs += 1;
        float2 *wp = W + (size_t)nr * p, *wq = W + (size_t)nr * q;
        float2 a[R], b[R];
        float al = 0.f, be = 0.f, gr = 0.f, gi = 0.f;
#pragma unroll
        for (int k = 0; k < R; ++k) {
          const int row = lane + 32 * k;
          if (row < nr) {
            a[k] = wp[row];
            b[k] = wq[row];
          } else {
            a[k] = make_float2(0.f, 0.f);
            b[k] = make_float2(0.f, 0.f);
          }
          al = fmaf(a[k].x, a[k].x, fmaf(a[k].y, a[k].y, al));
          be = fmaf(b[k].x, b[k].x, fmaf(b[k].y, b[k].y, be));
          // conj(a) * b
          gr = fmaf(a[k].x, b[k].x, fmaf(a[k].y, b[k].y, gr));
          gi = fmaf(a[k].x, b[k].y, fmaf(-a[k].y, b[k].x, gi));
        }
        al = warp_sum(al);
        be = warp_sum(be);
        gr = warp_sum(gr);
        gi = warp_sum(gi);
        const float ag = hypotf(gr, gi);
        if (!(al > negl && be > negl)) continue;
        if (!(ag > tol * sqrtf(al) * sqrtf(be))) continue;
        // 2x2 Hermitian [[al, g], [conj g, be]]: remove the phase of g, then
        // the real symmetric Schur rotation tan = sign(z) / (|z| + sqrt(1+z^2)).
        const float zeta = (be - al) / (2.0f * ag);
        const float az = fabsf(zeta);
        const float tn = (az > 1e18f ? 0.5f / az : 1.0f / (az + sqrtf(fmaf(az, az, 1.0f))));
        const float tt = zeta >= 0.0f ? tn : -tn;
        const float c = 1.0f / sqrtf(fmaf(tt, tt, 1.0f));
        const float s = c * tt;
        const float er = gr / ag, ei = -gi / ag;  // conj(g) / |g|
#pragma unroll
        for (int k = 0; k < R; ++k) {
          const int row = lane + 32 * k;
          if (row < nr) {
            const float2 bb = make_float2(er * b[k].x - ei * b[k].y, er * b[k].y + ei * b[k].x);
            wp[row] = make_float2(c * a[k].x - s * bb.x, c * a[k].y - s * bb.y);
            wq[row] = make_float2(s * a[k].x + c * bb.x, s * a[k].y + c * bb.y);
          }
        }
        float2 *vp = V + (size_t)nc * p, *vq = V + (size_t)nc * q;
#pragma unroll
        for (int k = 0; k < R; ++k) {
          const int row = lane + 32 * k;
          if (row < nc) {
            const float2 x = vp[row], y = vq[row];
            const float2 yy = make_float2(er * y.x - ei * y.y, er * y.y + ei * y.x);
            vp[row] = make_float2(c * x.x - s * yy.x, c * x.y - s * yy.y);
            vq[row] = make_float2(s * x.x + c * yy.x, s * x.y + c * yy.y);
          }
        }
        n_rot += 1;
        if (lane == 0) s_rot = 1;
      }
      __syncthreads();
    }
    sweeps = sweep;
    converged = (s_rot == 0);
    __syncthreads();
  }

  pk_epilogue<false>(nr, nc, W, V, t);
  if (tid == 0) sweeps_out[blockIdx.x] = converged ? sweeps : -max_sweeps;
  if (work && lane == 0) {
    atomicAdd(work + 0, n_pairs);
    atomicAdd(work + 1, n_rot);
  }
}

// ---------------------------------------------------------------------------
// Shared pieces of the packed kernel: panel width (columns; a warp per pair of
// them), rotation formula.
constexpr int kPW = 32;

struct Rot {
  float c, s, er, ei;
  float d;  // |a'|^2 = |a|^2 - d and |b'|^2 = |b|^2 + d (d = t |g|, the 2x2 Schur rotation's shift)
};

// Rotation of the 2x2 Hermitian [[al, g], [conj g, be]], or false when the
// pair is orthogonal to tolerance (|g|^2 <= tol^2 al be) or a column is
// negligible.  Unitarity rests on c = 1/sqrt(1 + t^2), s = c t and |e| = 1,
// which take the Newton-refined reciprocal square root; the angle itself
// (zeta, t) may carry a few ulps of error without affecting unitarity.
__device__ __forceinline__ bool make_rot(float al, float be, float gr, float gi, float tol,
                                         float negl, Rot &r) {
  if (!(al > negl && be > negl)) return false;
  const float g2 = fmaf(gr, gr, gi * gi);
  if (!(g2 > (tol * tol) * (al * be))) return false;
  const float inv_ag = rsqrt_nr(g2);
  const float zeta = 0.5f * (be - al) * inv_ag;
  const float az = fabsf(zeta);
  const float q = fmaf(az, az, 1.0f);
  const float tn = az > 1e18f ? __fdividef(0.5f, az) : __fdividef(1.0f, az + q * rsqrtf(q));
  const float tt = zeta >= 0.0f ? tn : -tn;
  r.c = rsqrt_nr(fmaf(tt, tt, 1.0f));
  r.s = r.c * tt;
  r.er = gr * inv_ag;
  r.ei = -gi * inv_ag;
  r.d = tt * (g2 * inv_ag);
  return true;
}

constexpr int kHW = kPW / 2;  // warps per CTA

__device__ __forceinline__ float half_sum(float v) {
#pragma unroll
  for (int o = 8; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// ---------------------------------------------------------------------------
// Packed kernel (nr <= 256): the half-warp panel scheme with Blackwell's
// paired FP32 instructions (__ffma2_rn / __fmul2_rn: two FP32 FMAs per lane
// per instruction).  Staged columns use a split row-pair layout: row pair m is
// one float4 (re_2m, re_2m+1, im_2m, im_2m+1), so a 128-bit load gives the two
// packed operands (re, re) and (im, im) directly and complex arithmetic needs
// no register shuffles: a dot-product step costs 4 paired instructions per two
// rows and a rotation 12 (against 16 and 24 scalar FMAs).  Panel a's W columns
// live in registers (one per half-warp); V columns of panel a and of the
// streamed panel b stay in shared memory.
__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }
__device__ __forceinline__ float2 mul2(float2 a, float2 b) { return __fmul2_rn(a, b); }
__device__ __forceinline__ float2 dup(float x) { return make_float2(x, x); }
__device__ __forceinline__ float2 lo2(const float4 &v) { return make_float2(v.x, v.y); }
__device__ __forceinline__ float2 hi2(const float4 &v) { return make_float2(v.z, v.w); }

// A rotation as broadcast pairs: a' = c a - (s e) b, b' = s a + (c e) b.
struct PRot {
  float2 C, S, NSEX, SEY, NSEY, CEX, CEY, NCEY;
};

__device__ __forceinline__ PRot packed(const Rot &r) {
  const float sex = r.s * r.er, sey = r.s * r.ei, cex = r.c * r.er, cey = r.c * r.ei;
  PRot q;
  q.C = dup(r.c);
  q.S = dup(r.s);
  q.NSEX = dup(-sex);
  q.SEY = dup(sey);
  q.NSEY = dup(-sey);
  q.CEX = dup(cex);
  q.CEY = dup(cey);
  q.NCEY = dup(-cey);
  return q;
}

__device__ __forceinline__ void pk_rot(float4 &a, float4 &b, const PRot &q) {
  const float2 Ra = lo2(a), Ia = hi2(a), Rb = lo2(b), Ib = hi2(b);
  const float2 aR = fma2(q.SEY, Ib, fma2(q.NSEX, Rb, mul2(q.C, Ra)));
  const float2 aI = fma2(q.NSEY, Rb, fma2(q.NSEX, Ib, mul2(q.C, Ia)));
  const float2 bR = fma2(q.NCEY, Ib, fma2(q.CEX, Rb, mul2(q.S, Ra)));
  const float2 bI = fma2(q.CEY, Rb, fma2(q.CEX, Ib, mul2(q.S, Ia)));
  a = make_float4(aR.x, aR.y, aI.x, aI.y);
  b = make_float4(bR.x, bR.y, bI.x, bI.y);
}

// lane partial sums of |a|^2, |b|^2, re(a^H b), im(a^H b) over K row pairs,
// in two interleaved chains (even / odd k) to halve the dependent FMA depth
template <int K>
__device__ __forceinline__ void pk_dots(const float4 (&a)[K], const float4 (&b)[K], float &al,
                                        float &be, float &gr, float &gi) {
  const float2 z = make_float2(0.f, 0.f);
  float2 aa[2] = {z, z}, bb[2] = {z, z}, rr[2] = {z, z}, i1[2] = {z, z}, i2[2] = {z, z};
#pragma unroll
  for (int k = 0; k < K; ++k) {
    const int c = k & 1;
    const float2 Ra = lo2(a[k]), Ia = hi2(a[k]), Rb = lo2(b[k]), Ib = hi2(b[k]);
    aa[c] = fma2(Ia, Ia, fma2(Ra, Ra, aa[c]));
    bb[c] = fma2(Ib, Ib, fma2(Rb, Rb, bb[c]));
    rr[c] = fma2(Ia, Ib, fma2(Ra, Rb, rr[c]));
    i1[c] = fma2(Ra, Ib, i1[c]);
    i2[c] = fma2(Ia, Rb, i2[c]);
  }
  al = (aa[0].x + aa[1].x) + (aa[0].y + aa[1].y);
  be = (bb[0].x + bb[1].x) + (bb[0].y + bb[1].y);
  gr = (rr[0].x + rr[1].x) + (rr[0].y + rr[1].y);
  gi = ((i1[0].x + i1[1].x) + (i1[0].y + i1[1].y)) - ((i2[0].x + i2[1].x) + (i2[0].y + i2[1].y));
}

// lane partial sums of re(a^H b), im(a^H b) only (pk_dots without the norms,
// in the same order, so the inner product is bit-identical to pk_dots')
template <int K>
__device__ __forceinline__ void pk_cross(const float4 (&a)[K], const float4 (&b)[K], float &gr,
                                         float &gi) {
  const float2 z = make_float2(0.f, 0.f);
  float2 rr[2] = {z, z}, i1[2] = {z, z}, i2[2] = {z, z};
#pragma unroll
  for (int k = 0; k < K; ++k) {
    const int c = k & 1;
    const float2 Ra = lo2(a[k]), Ia = hi2(a[k]), Rb = lo2(b[k]), Ib = hi2(b[k]);
    rr[c] = fma2(Ia, Ib, fma2(Ra, Rb, rr[c]));
    i1[c] = fma2(Ra, Ib, i1[c]);
    i2[c] = fma2(Ia, Rb, i2[c]);
  }
  gr = (rr[0].x + rr[1].x) + (rr[0].y + rr[1].y);
  gi = ((i1[0].x + i1[1].x) + (i1[0].y + i1[1].y)) - ((i2[0].x + i2[1].x) + (i2[0].y + i2[1].y));
}

// lane partial sum of |a|^2 over K row pairs
template <int K>
__device__ __forceinline__ float pk_norm(const float4 (&a)[K]) {
  const float2 z = make_float2(0.f, 0.f);
  float2 aa[2] = {z, z};
#pragma unroll
  for (int k = 0; k < K; ++k) {
    const int c = k & 1;
    const float2 Ra = lo2(a[k]), Ia = hi2(a[k]);
    aa[c] = fma2(Ia, Ia, fma2(Ra, Ra, aa[c]));
  }
  return (aa[0].x + aa[1].x) + (aa[0].y + aa[1].y);
}

// A tracked squared norm that fell below this fraction of its value before
// the rotation is marked for recomputation from the column itself (when the
// column is next read): the update |a|^2 - d cancels there, and its absolute
// rounding (about eps |a|^2) would become a large relative error.
constexpr float kNormDrop = 0.0625f;

// rotates two shared-memory columns (row-pair layout), lane stride `step`
template <int K, int STEP>
__device__ __forceinline__ void pk_rot_smem(float4 *ca, float4 *cb, const PRot &q, int l) {
#pragma unroll
  for (int k = 0; k < K; k += 2) {
    float4 x0 = ca[l + STEP * k], y0 = cb[l + STEP * k];
    float4 x1, y1;
    if (k + 1 < K) {
      x1 = ca[l + STEP * (k + 1)];
      y1 = cb[l + STEP * (k + 1)];
    }
    pk_rot(x0, y0, q);
    ca[l + STEP * k] = x0;
    cb[l + STEP * k] = y0;
    if (k + 1 < K) {
      pk_rot(x1, y1, q);
      ca[l + STEP * (k + 1)] = x1;
      cb[l + STEP * (k + 1)] = y1;
    }
  }
}

// rotates the register column a against shared-memory column col (row-pair
// layout, half-warp lane stride), two row pairs at a time
template <int K>
__device__ __forceinline__ void pk_rot_stream(float4 (&a)[K], float4 *col, const PRot &q, int ul) {
  // loads run one row pair ahead of the rotate-and-store
  float4 y = col[ul];
#pragma unroll
  for (int k = 0; k < K; ++k) {
    float4 ynext;
    if (k + 1 < K) ynext = col[ul + 16 * (k + 1)];
    pk_rot(a[k], y, q);
    col[ul + 16 * k] = y;
    if (k + 1 < K) y = ynext;
  }
}

// Staging of panels into shared memory: a shared panel holds ld2 row pairs
// per column in the split layout, zero padded, of wcols columns of n rows;
// warp w copies columns w, w + kHW.  A lane's row pairs of one column:
// ld2 <= kStageIt * 32 for every packed shape (PkShape: at most 128).
constexpr int kStageIt = 4;

// One column of n rows into registers (the lane's row pairs m = lane + 32 it,
// zeros past n or for a padding column), and from there into a shared panel
// column in the split row-pair layout, returning the lane's part of its
// squared norm.
__device__ __forceinline__ void col_load(float2 (&x0)[kStageIt], float2 (&x1)[kStageIt],
                                         const float2 *s, int n, int ld2, bool real) {
  const int lane = threadIdx.x & 31;
#pragma unroll
  for (int it = 0; it < kStageIt; ++it) {
    const int m = lane + 32 * it, r0 = 2 * m, r1 = 2 * m + 1;
    x0[it] = (real && m < ld2 && r0 < n) ? s[r0] : make_float2(0.f, 0.f);
    x1[it] = (real && m < ld2 && r1 < n) ? s[r1] : make_float2(0.f, 0.f);
  }
}

__device__ __forceinline__ float col_store(float4 *d, const float2 (&x0)[kStageIt],
                                           const float2 (&x1)[kStageIt], int ld2) {
  const int lane = threadIdx.x & 31;
  float part = 0.0f;
#pragma unroll
  for (int it = 0; it < kStageIt; ++it) {
    const int m = lane + 32 * it;
    if (m < ld2) {
      d[m] = make_float4(x0[it].x, x1[it].x, x0[it].y, x1[it].y);
      part = fmaf(x0[it].x, x0[it].x,
                  fmaf(x0[it].y, x0[it].y, fmaf(x1[it].x, x1[it].x, fmaf(x1[it].y, x1[it].y, part))));
    }
  }
  return part;
}

// A panel's W (nr rows, squared column norms into nrm) and V (nc rows)
// staged together: a warp issues the loads of its W and V columns (NCOL of
// each) before its first shared store, so that 16 NCOL loads a lane are in
// flight.  NCOL = 2 holds 32 float2 a lane, for stagings with no register
// panel live.
// sW and sV are the slice's first columns; panel column c is column cols[c]
// (shared memory: the panel's wcols column indices).
template <int NCOL>
__device__ __forceinline__ void pk_stage_wv(float4 *dW, const float2 *sW, int nr, float *nrm,
                                            float4 *dV, const float2 *sV, int nc, int ld2,
                                            int wcols, const int *cols) {
  const int lane = threadIdx.x & 31;
  for (int c0 = threadIdx.x >> 5; c0 < kPW; c0 += NCOL * kHW) {
    float2 w0[NCOL][kStageIt], w1[NCOL][kStageIt], v0[NCOL][kStageIt], v1[NCOL][kStageIt];
#pragma unroll
    for (int k = 0; k < NCOL; ++k) {
      const int c = c0 + k * kHW;
      const bool real = c < kPW && c < wcols;
      const int g = real ? cols[c] : 0;
      col_load(w0[k], w1[k], sW + (size_t)nr * g, nr, ld2, real);
      col_load(v0[k], v1[k], sV + (size_t)nc * g, nc, ld2, real);
    }
#pragma unroll
    for (int k = 0; k < NCOL; ++k) {
      const int c = c0 + k * kHW;
      if (c >= kPW) break;
      const float part = warp_sum(col_store(dW + ld2 * c, w0[k], w1[k], ld2));
      if (lane == 0) nrm[c] = part;
      col_store(dV + ld2 * c, v0[k], v1[k], ld2);
    }
  }
}

__device__ __forceinline__ void pk_stage_out(float2 *dst, const float4 *src, int ld2, int n,
                                             int wcols, const int *cols) {
  const int lane = threadIdx.x & 31;
  for (int c = threadIdx.x >> 5; c < wcols; c += kHW) {
    float2 *d = dst + (size_t)n * cols[c];
    const float4 *s = src + ld2 * c;
    for (int m = lane; 2 * m < n; m += 32) {
      const float4 v = s[m];
      d[2 * m] = make_float2(v.x, v.z);
      if (2 * m + 1 < n) d[2 * m + 1] = make_float2(v.y, v.w);
    }
  }
}

template <int KP>
struct PkShape {
  static constexpr int KPF = (KP + 1) / 2;  // row pairs per lane, full warp
  static constexpr int LD2 = (16 * KP > 32 * KPF) ? 16 * KP : 32 * KPF;  // row pairs per column
  static_assert(LD2 <= 32 * kStageIt, "col_load covers a column in kStageIt loads a lane");
};

// The pairs inside one staged panel (W in sW with squared norms s_na, V in
// sVa; wa real columns): 31 rounds of 16 disjoint pairs, one per warp.
template <int KP>
__device__ __forceinline__ void pk_intra(float4 *sW, float4 *sVa, float *s_na, int wa, float tol,
                                         float negl, unsigned &n_pairs, unsigned &n_rot,
                                         int &rotated) {
  constexpr int KPF = PkShape<KP>::KPF;
  constexpr int LD2 = PkShape<KP>::LD2;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  for (int r = 0; r < kPW - 1; ++r) {
    int p, q;
    pair_of(r, warp, kPW, p, q);
    if (p < wa && q < wa) {
      float4 xa[KPF], xb[KPF];
#pragma unroll
      for (int k = 0; k < KPF; ++k) {
        xa[k] = sW[LD2 * p + lane + 32 * k];
        xb[k] = sW[LD2 * q + lane + 32 * k];
      }
      float gr, gi;
      pk_cross<KPF>(xa, xb, gr, gi);
      gr = warp_sum(gr);
      gi = warp_sum(gi);
      // a norm marked negative after a rotation that cancelled it is
      // recomputed from the column (warp-uniform: p, q are the warp's)
      float al = s_na[p], be = s_na[q];
      if (al < 0.0f) al = warp_sum(pk_norm<KPF>(xa));
      if (be < 0.0f) be = warp_sum(pk_norm<KPF>(xb));
      if (lane == 0) n_pairs += 1;
      Rot rt;
      if (make_rot(al, be, gr, gi, tol, negl, rt)) {
        const PRot pq = packed(rt);
#pragma unroll
        for (int k = 0; k < KPF; ++k) {
          pk_rot(xa[k], xb[k], pq);
          sW[LD2 * p + lane + 32 * k] = xa[k];
          sW[LD2 * q + lane + 32 * k] = xb[k];
        }
        pk_rot_smem<KPF, 32>(sVa + LD2 * p, sVa + LD2 * q, pq, lane);
        const float na = al - rt.d, nb = be + rt.d;
        if (lane == 0) {
          s_na[p] = na < kNormDrop * al ? -1.0f : na;
          s_na[q] = nb < kNormDrop * be ? -1.0f : nb;
          n_rot += 1;
        }
        rotated = 1;
      }
    }
    __syncthreads();
  }
}

// Panel a's columns (one per half-warp, `unit`; W in aW, V in aV, both in
// registers; mine = the column is real) against the streamed panel b (W in
// sW with squared norms s_nb, V in sVb; wb real columns): 16 double rounds in
// which warp w owns streamed columns 2c, 2c+1 (c = (w + R) mod 16) and its
// half-warps rotate them in swapped order, so only the warp synchronises
// between the two sub-steps and the block once per double round.
template <int KP>
__device__ __forceinline__ void pk_cross_pass(float4 (&aW)[KP], float4 (&aV)[KP], bool mine,
                                              float4 *sW, float4 *sVb, float *s_nb, int wb,
                                              float tol, float negl, unsigned &n_pairs,
                                              unsigned &n_rot, int &rotated,
                                              float *al_out = nullptr) {
  constexpr int LD2 = PkShape<KP>::LD2;
  const int tid = threadIdx.x, warp = tid >> 5;
  const int unit = tid >> 4, ul = tid & 15;
  float4 bW[KP];
  // the register column's squared norm, exact at the start of each streamed
  // panel (the whole warp shuffles: both halves compute theirs)
  float al_reg = half_sum(pk_norm<KP>(aW));
  __syncthreads();
  for (int r = 0; r < kPW; ++r) {
    const int sub = r & 1;
    const int cpi = (warp + (r >> 1)) & (kHW - 1);
    const int j = 2 * cpi + ((unit & 1) ^ sub);
    const bool real = mine && j < wb;
#pragma unroll
    for (int k = 0; k < KP; ++k) bW[k] = sW[LD2 * j + ul + 16 * k];
    float gr, gi;
    pk_cross<KP>(aW, bW, gr, gi);
    gr = half_sum(gr);
    gi = half_sum(gi);
    // norms marked negative after a rotation that cancelled them are
    // recomputed here, where both columns are in registers; the decision is
    // made per warp so that both halves take part in the shuffles
    float be = s_nb[j];
    if (__any_sync(0xffffffffu, be < 0.0f || al_reg < 0.0f)) {
      const float xa = half_sum(pk_norm<KP>(aW));
      const float xb = half_sum(pk_norm<KP>(bW));
      if (al_reg < 0.0f) al_reg = xa;
      if (be < 0.0f) be = xb;
    }
    Rot rt;
    const bool go = real && make_rot(al_reg, be, gr, gi, tol, negl, rt);
    if (ul == 0 && real) n_pairs += 1;
    if (__any_sync(0xffffffffu, go)) {
      // the other half-warp may rotate: this half applies the identity, which
      // rewrites its columns unchanged
      if (!go) {
        rt.c = 1.0f;
        rt.s = 0.0f;
        rt.er = 1.0f;
        rt.ei = 0.0f;
        rt.d = 0.0f;
      }
      const PRot pq = packed(rt);
#pragma unroll
      for (int k = 0; k < KP; ++k) {
        pk_rot(aW[k], bW[k], pq);
        sW[LD2 * j + ul + 16 * k] = bW[k];
      }
      pk_rot_stream<KP>(aV, sVb + LD2 * j, pq, ul);
      if (go) {
        const float na = al_reg - rt.d, nb = be + rt.d;
        al_reg = na < kNormDrop * al_reg ? -1.0f : na;
        if (ul == 0) {
          s_nb[j] = nb < kNormDrop * be ? -1.0f : nb;
          n_rot += 1;
        }
        rotated = 1;
      }
    }
    if (sub == 0)
      __syncwarp();
    else
      __syncthreads();
  }
  if (al_out) *al_out = al_reg;
}

// Panel a's W column `unit` of the staged panel moves to registers, with its V.
template <int KP>
__device__ __forceinline__ void pk_to_registers(const float4 *sW, const float4 *sVa,
                                                float4 (&aW)[KP], float4 (&aV)[KP]) {
  constexpr int LD2 = PkShape<KP>::LD2;
  const int unit = threadIdx.x >> 4, ul = threadIdx.x & 15;
#pragma unroll
  for (int k = 0; k < KP; ++k) {
    aW[k] = sW[LD2 * unit + ul + 16 * k];
    aV[k] = sVa[LD2 * unit + ul + 16 * k];
  }
}

// Panel a back to global memory from the registers (W) and, through sVa, V.
template <int KP>
__device__ __forceinline__ void pk_from_registers(const float4 (&aW)[KP], const float4 (&aV)[KP],
                                                  bool mine, float4 *sVa, float2 *Wa,
                                                  float2 *Va, int nr, int nc, int wa,
                                                  const int *cols) {
  constexpr int LD2 = PkShape<KP>::LD2;
  const int unit = threadIdx.x >> 4, ul = threadIdx.x & 15;
#pragma unroll
  for (int k = 0; k < KP; ++k) sVa[LD2 * unit + ul + 16 * k] = aV[k];
  __syncthreads();
  if (mine) {
    float2 *wcol = Wa + (size_t)nr * cols[unit];
#pragma unroll
    for (int k = 0; k < KP; ++k) {
      const int m = ul + 16 * k;
      if (2 * m < nr) wcol[2 * m] = make_float2(aW[k].x, aW[k].z);
      if (2 * m + 1 < nr) wcol[2 * m + 1] = make_float2(aW[k].y, aW[k].w);
    }
  }
  pk_stage_out(Va, sVa, LD2, nc, wa, cols);
}

// Columns of a slice of the packed kernels at most (nc <= nr <= 256).
constexpr int kSortCols = 256;

// Squared norms of a slice's nc columns of nr <= 256 rows into key (shared
// memory), by the whole CTA: two columns a warp at a time, every lane's loads
// of both issued together.  W was written by an earlier launch.
__device__ void col_norms(int nr, int nc, const float2 *W, float *key) {
  const int lane = threadIdx.x & 31, nwarp = blockDim.x >> 5;
  for (int c = threadIdx.x >> 5; c < nc; c += 2 * nwarp) {
    const int c2 = c + nwarp;
    const float2 *w0 = W + (size_t)nr * c, *w1 = W + (size_t)nr * (c2 < nc ? c2 : c);
    float2 x[8], y[8];
#pragma unroll
    for (int k = 0; k < 8; ++k) {
      const int r = lane + 32 * k;
      x[k] = r < nr ? w0[r] : make_float2(0.f, 0.f);
      y[k] = r < nr ? w1[r] : make_float2(0.f, 0.f);
    }
    float a = 0.f, b = 0.f;
#pragma unroll
    for (int k = 0; k < 8; ++k) {
      a = fmaf(x[k].x, x[k].x, fmaf(x[k].y, x[k].y, a));
      b = fmaf(y[k].x, y[k].x, fmaf(y[k].y, y[k].y, b));
    }
    a = warp_sum(a);
    b = warp_sum(b);
    if (lane == 0) {
      key[c] = a;
      if (c2 < nc) key[c2] = b;
    }
  }
}

// The packed Jacobi SVT of one matrix by the whole CTA (kHW warps): W (nr x
// nc) and V (nc x nc) in global memory, `smem` the CTA's dynamic shared memory
// (3 kPW LD2 float4).  Panel by panel: panel a's own pairs, then panel a (in
// registers) against every later panel b streamed through shared memory.
// Writes the sweep count (negative at the cap) to *sweeps_slot.
template <int KP>
__device__ __forceinline__ void jacobi_pk_slice(int nr, int nc, float2 *W, float2 *V, float t,
                                                int max_sweeps, float tol, float negl_rel,
                                                int *sweeps_slot, unsigned long long *work,
                                                float4 *smem, const JacOpt &o, int slice) {
  constexpr int LD2 = PkShape<KP>::LD2;
  float4 *sW = smem;              // panel a (own pairs), then panel b: W
  float4 *sVa = sW + kPW * LD2;    // panel a: V
  float4 *sVb = sVa + kPW * LD2;   // panel b: V
  const int tid = threadIdx.x, ul = tid & 15, unit = tid >> 4;
  __shared__ float s_red[32];
  __shared__ int s_rot;
  // squared column norms of panel a and of the streamed panel b: exact when
  // a panel is staged, then carried through each rotation by the 2x2 update
  // (|a|^2 - d, |b|^2 + d), so that a pair's test needs only its inner product
  __shared__ float s_na[kPW], s_nb[kPW];
  // the sweep's column order (position -> column; panel a holds positions
  // a kPW ...) and each column's squared norm as the sweep left it
  __shared__ int s_perm[kSortCols];
  __shared__ float s_key[kSortCols];

  const float fro2 = pk_setup(nr, nc, W, V, o.warm, s_red);
  const float negl = negl_rel * fro2;
  const int npan = (nc + kPW - 1) / kPW;
  unsigned n_pairs = 0, n_rot = 0;  // lane 0 (own pairs) and ul 0 (cross pairs) count
  int sweeps = (nc < 2) ? 1 : 0;
  bool converged = slice_known(fro2, o, slice, sweeps) || nc < 2;
  tol = pk_tolerance(tol, fro2, nc, o.t_svt, o.ms2 ? o.ms2[slice / o.group] : -1.0f);
  float4 aW[KP], aV[KP];
  if (!converged) {  // the first sweep's order: by the columns' norms, or as stored
    if (o.sort) {
      col_norms(nr, nc, W, s_key);
      __syncthreads();
      order_columns(nc, s_key, s_perm);
    } else {
      for (int c = tid; c < nc; c += blockDim.x) s_perm[c] = c;
    }
  }
  for (int sweep = 1; sweep <= max_sweeps && !converged; ++sweep) {
    if (tid == 0) s_rot = 0;
    int rotated = 0;
    for (int a = 0; a < npan; ++a) {
      const int ca = a * kPW, wa = min(kPW, nc - ca);
      const int *cola = s_perm + ca;  // panel a: positions ca ... of the sweep's order
      __syncthreads();
      pk_stage_wv<2>(sW, W, nr, s_na, sVa, V, nc, LD2, wa, cola);
      __syncthreads();
      pk_intra<KP>(sW, sVa, s_na, wa, tol, negl, n_pairs, n_rot, rotated);
      if (tid < wa) s_key[cola[tid]] = s_na[tid];
      const bool mine = unit < wa;
      pk_to_registers<KP>(sW, sVa, aW, aV);
      for (int b = a + 1; b < npan; ++b) {
        const int cb = b * kPW, wb = min(kPW, nc - cb);
        const int *colb = s_perm + cb;
        __syncthreads();
        pk_stage_wv<1>(sW, W, nr, s_nb, sVb, V, nc, LD2, wb, colb);
        float al = 0.0f;
        pk_cross_pass<KP>(aW, aV, mine, sW, sVb, s_nb, wb, tol, negl, n_pairs, n_rot, rotated,
                              &al);
        if (mine && ul == 0) s_key[cola[unit]] = al;
        if (tid < wb) s_key[colb[tid]] = s_nb[tid];
        pk_stage_out(W, sW, LD2, nr, wb, colb);
        pk_stage_out(V, sVb, LD2, nc, wb, colb);
      }
      pk_from_registers<KP>(aW, aV, mine, sVa, W, V, nr, nc, wa, cola);
    }
    if (rotated) s_rot = 1;
    __syncthreads();
    sweeps = sweep;
    converged = (s_rot == 0);
    // the next sweep's order, from the norms this one left
    if (o.sort && !converged) order_columns(nc, s_key, s_perm);
    __syncthreads();
  }
  pk_epilogue<false>(nr, nc, W, V, t);
  if (tid == 0) *sweeps_slot = converged ? sweeps : -max_sweeps;
  if (work && ul == 0) {
    atomicAdd(work + 0, (unsigned long long)n_pairs);
    atomicAdd(work + 1, (unsigned long long)n_rot);
  }
}

// Slices of up to 64 rows fit in 64 registers a thread: two CTAs share an SM.
template <int KP>
__global__ void __launch_bounds__(kPW * 16, KP <= 2 ? 2 : 1)
    k_jacobi_pk(int nr, int nc, size_t wstride, size_t vstride, float2 *W_all, float2 *V_all,
                float t, int max_sweeps, float tol, float negl_rel, int *__restrict__ sweeps_out,
                unsigned long long *__restrict__ work, JacOpt o) {
  extern __shared__ float4 smem_f4[];
  const int s = blockIdx.x;
  jacobi_pk_slice<KP>(nr, nc, W_all + (size_t)s * wstride, V_all + (size_t)s * vstride, t,
                          max_sweeps, tol, negl_rel, sweeps_out + s, work, smem_f4, o, s);
}

template <int KP>
cudaError_t launch_pk(int nslices, int nr, int nc, size_t ws, size_t vs, float2 *W, float2 *V,
                      float t, int max_sweeps, float tol, float negl, int *sweeps,
                      unsigned long long *work, const JacOpt &o, cudaStream_t st) {
  const size_t smem = sizeof(float4) * 3 * (size_t)kPW * PkShape<KP>::LD2;
  cudaError_t e = cudaFuncSetAttribute(k_jacobi_pk<KP>,
                                       cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  k_jacobi_pk<KP><<<nslices, kPW * 16, smem, st>>>(nr, nc, ws, vs, W, V, t, max_sweeps, tol,
                                                        negl, sweeps, work, o);
  return cudaGetLastError();
}

// sigma_i = |w_i| and V_s = V diag(g), g = max(1 - t / sigma, 0), with the same
// arithmetic and summation order as the Jacobi kernels' epilogue (so a Jacobi
// run with t < 0 followed by this kernel equals a run with threshold t).
__global__ void __launch_bounds__(512)
    k_sigma_scale(int nr, int nc, size_t wstride, const float2 *__restrict__ W,
                  const float2 *__restrict__ V, float t, double *__restrict__ sig,
                  float2 *__restrict__ Vs) {
  // slice blockIdx.x, one column a warp: blockIdx.y takes columns
  // blockDim.x / 32 blockIdx.y .. + blockDim.x / 32 - 1
  const int s = blockIdx.x, warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int nwarps = blockDim.x >> 5;
  const float2 *Ws = W + (size_t)s * wstride;
  const size_t vs = (size_t)nc * nc;
  const int i = blockIdx.y * nwarps + warp;
  if (i < nc) {
    const float2 *wi = Ws + (size_t)nr * i;
    float n2 = 0.f;
#pragma unroll 4
    for (int row = lane; row < nr; row += 32)
      n2 = fmaf(wi[row].x, wi[row].x, fmaf(wi[row].y, wi[row].y, n2));
    n2 = warp_sum(n2);
    const double sigma = sqrt((double)n2);
    const float g = sigma > (double)t ? (float)(1.0 - (double)t / sigma) : 0.0f;
    if (sig && lane == 0) sig[(size_t)s * nc + i] = sigma;
    const float2 *vi = V + s * vs + (size_t)nc * i;
    float2 *oi = Vs + s * vs + (size_t)nc * i;
#pragma unroll 4
    for (int row = lane; row < nc; row += 32) oi[row] = make_float2(vi[row].x * g, vi[row].y * g);
  }
}

// Mean-square column norm ||W_s||_F^2 / nc of every slice, reduced to the
// largest over each group of `group` consecutive slices (atomic max on the
// bits of non-negative floats; the group slots start at zero).
__global__ void __launch_bounds__(1024)
    k_group_ms2(int nr, int nc, size_t wstride, const float2 *__restrict__ W, int group,
                unsigned *__restrict__ gmax) {
  __shared__ float s_red[32];
  const float2 *Ws = W + (size_t)blockIdx.x * wstride;
  float part = sumsq4(Ws, (size_t)nr * nc);
  part = warp_sum(part);
  if ((threadIdx.x & 31) == 0) s_red[threadIdx.x >> 5] = part;
  __syncthreads();
  if (threadIdx.x == 0) {
    float v = 0.0f;
    for (int w = 0; w < (int)(blockDim.x >> 5); ++w) v += s_red[w];
    atomicMax(gmax + blockIdx.x / group, __float_as_uint(v / (float)nc));
  }
}

// cand[s] = 1 when slice s's previous Jacobi run took one sweep (not none:
// a slice whose singular values were all cut, or that has not run yet, is
// left to the Jacobi's own cheap all-cut test or to its sweeps).
__global__ void k_gram_gate(const int *__restrict__ sweeps, int n, int *__restrict__ cand) {
  const int s = blockIdx.x * blockDim.x + threadIdx.x;
  if (s < n) cand[s] = sweeps[s] == 1 ? 1 : 0;
}

// conv[s] for the Gram matrix G_s (nc x nc, column-major) of a candidate slice:
// 1 when every pair p < q passes |G_pq| <= (tol (1 - 1e-3) - kappa) sqrt(G_pp G_qq).
// The sweep rotates a pair when |g|^2 > tol^2 |w_p|^2 |w_q|^2 with g the inner
// product of its own Gram.  G_pq carries at most about (nr eps + 2^-20) |w_p| |w_q|
// of rounding (3xTF32 products, FP32 sums); g carries the 22-bit halves' 2^-22
// and the tensor core's truncation, one ulp (2 eps) of at most |w_p| |w_q| for each
// 16 rows and each of the four split products, of which hi*hi alone is full-size:
// nr eps / 8 and a little.  kappa = 4 nr eps + 4e-6 keeps every passing pair below
// the sweep's test, and the (1 - 1e-3) covers the sweep's own squared norms and
// this test's FP32 squares.  tol: the Jacobi's threshold-aware tolerance (pk_tolerance with the
// tensor's ms2).  One CTA a slice.
__global__ void __launch_bounds__(256)
    k_gram_check(const float2 *__restrict__ G, int nr, int nc, const int *__restrict__ cand,
                 float tol0, float skip_t, const float *__restrict__ ms2, int group,
                 int *__restrict__ conv) {
  const int s = blockIdx.x;
  if (!cand[s]) {
    if (threadIdx.x == 0) conv[s] = 0;
    return;
  }
  const float2 *Gs = G + (size_t)s * nc * nc;
  __shared__ float s_d[512];
  __shared__ float s_red[8];
  float part = 0.0f;
  for (int i = threadIdx.x; i < nc; i += blockDim.x) {
    const float di = Gs[(size_t)i * nc + i].x;
    s_d[i] = fmaxf(di, 0.0f);
    part += di;
  }
  part = warp_sum(part);
  if ((threadIdx.x & 31) == 0) s_red[threadIdx.x >> 5] = part;
  __syncthreads();
  float fro2 = 0.0f;
  for (int w = 0; w < (int)(blockDim.x >> 5); ++w) fro2 += s_red[w];
  const float tol = pk_tolerance(tol0, fro2, nc, skip_t, ms2 ? ms2[s / group] : -1.0f);
  const double eps = (double)FLT_EPSILON * 0.5;
  const double lim = (double)tol * (1.0 - 1e-3) - (4.0 * nr * eps + 4e-6);
  const float lim2 = (float)(lim * lim);
  int ok = lim > 0.0;
  for (size_t e = threadIdx.x; ok && e < (size_t)nc * nc; e += blockDim.x) {
    const int p = (int)(e % nc), q = (int)(e / nc);
    if (p >= q) continue;
    const float2 g = Gs[e];
    if (!(fmaf(g.x, g.x, g.y * g.y) <= lim2 * (s_d[p] * s_d[q]))) ok = 0;
  }
  ok = __syncthreads_and(ok);
  if (threadIdx.x == 0) conv[s] = ok;
}

// One Newton-Schulz step towards the nearest unitary matrix:
// V := V (3 I - V^H V) / 2 = 1.5 V - 0.5 D with D = (V V^H) V given.
__global__ void k_ns_update(int nc, int nslices, size_t dstride, float2 *__restrict__ V,
                            const float2 *__restrict__ D) {
  const size_t per = (size_t)nc * nc, total = per * nslices;
  for (size_t e = blockIdx.x * (size_t)blockDim.x + threadIdx.x; e < total;
       e += (size_t)gridDim.x * blockDim.x) {
    const size_t s = e / per, r = e - s * per;
    const float2 v = V[e], d = D[s * dstride + r];
    V[e] = make_float2(1.5f * v.x - 0.5f * d.x, 1.5f * v.y - 0.5f * d.y);
  }
}

}  // namespace

cudaError_t launch_sigma_scale(const Dims &d, int nslices, const float2 *W, const float2 *V,
                               float t, double *sig, float2 *Vs, cudaStream_t st) {
  if (nslices <= 0) return cudaSuccess;
  // 16 columns a CTA: about a dozen CTAs a slice, so every SM streams
  k_sigma_scale<<<dim3(nslices, (d.nc + 15) / 16), 512, 0, st>>>(d.nr, d.nc, d.P, W, V, t, sig,
                                                                   Vs);
  return cudaGetLastError();
}

cudaError_t launch_group_ms2(const Dims &d, int nslices, const float2 *W, int group, float *ms2,
                             cudaStream_t st) {
  if (nslices <= 0) return cudaSuccess;
  const int ngroups = (nslices + group - 1) / group;
  cudaError_t e = cudaMemsetAsync(ms2, 0, sizeof(float) * ngroups, st);
  if (e != cudaSuccess) return e;
  k_group_ms2<<<nslices, 1024, 0, st>>>(d.nr, d.nc, d.P, W, group, (unsigned *)ms2);
  return cudaGetLastError();
}

// A slice of one panel of 16 columns, or little more than half of one, is a chain of
// single tasks, a set-up and a closing launch that the FP32 kernels do in one.  t-SVT
// with the blocked / the FP32 kernel, us: 20 x 4 x 4 111 / 62, 64 x 12 x 64 156 / 121,
// 256 x 8 x 64 170 / 121, 512 x 4 x 4 131 / 53.  The ratio at the line, with 4, 31 and
// 128 bands: 48 x 16 1.15, 0.99, 1.10; 128 x 14 1.08, 1.20, 1.01; 230 x 12 1.02, 1.05,
// 0.97; beyond it 128 x 16 0.90, 0.90, 1.01; 230 x 13 0.89, 0.96, 0.99.
bool jacobi_few(int nr, int nc) { return nr > 256 ? nc <= 12 : 48 * nc <= 816 - nr; }

float jacobi_tol0(int nr) { return 8.0f * sqrtf((float)nr) * (FLT_EPSILON * 0.5f); }

cudaError_t launch_gram_check(const Dims &d, int nslices, const float2 *W, float2 *G,
                              const int *sweeps, int *cand, int *conv, float t_svt,
                              const float *ms2, int group, int *gemm_err, cudaStream_t st) {
  if (nslices <= 0) return cudaSuccess;
  if (d.nc > 512) return cudaErrorInvalidValue;  // s_d holds the diagonal
  k_gram_gate<<<(nslices + 255) / 256, 256, 0, st>>>(sweeps, nslices, cand);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  CGemm g{};
  g.A = W; g.sA = (long long)d.P; g.lda = d.nr; g.opA = 1;
  g.B = W; g.sB = (long long)d.P; g.ldb = d.nr; g.opB = 0;
  g.C = G; g.sC = (long long)d.nc * d.nc; g.ldc = d.nc;
  g.M = d.nc; g.N = d.nc; g.K = d.nr; g.batch = nslices;
  g.gate = cand;
  if ((e = launch_cgemm_tc(g, gemm_err, st, 0)) != cudaSuccess) return e;
  k_gram_check<<<nslices, 256, 0, st>>>(G, d.nr, d.nc, cand, jacobi_tol0(d.nr), t_svt, ms2, group,
                                        conv);
  return cudaGetLastError();
}

cudaError_t launch_ns_update(int nc, int nslices, size_t dstride, float2 *V, const float2 *D,
                             cudaStream_t st) {
  const size_t total = (size_t)nc * nc * nslices;
  if (total == 0) return cudaSuccess;
  size_t blocks = (total + 255) / 256;
  if (blocks > 152 * 16) blocks = 152 * 16;
  k_ns_update<<<(unsigned)blocks, 256, 0, st>>>(nc, nslices, dstride, V, D);
  return cudaGetLastError();
}

cudaError_t launch_jacobi(const Dims &d, int nslices, float2 *W, float2 *V, float t,
                          int max_sweeps, int *sweeps, unsigned long long *work,
                          cudaStream_t st, const JacOpt &o) {
  const int nr = d.nr, nc = d.nc;
  if (nslices <= 0) return cudaSuccess;
  // Few columns, or no queue's scratch: one CTA runs a slice.  Without scratch, up to 256 rows the FP32 kernel,
  // which keeps a panel in registers while the others stream past (200 x 200 x 80:
  // 10.5 ms a t-SVT against 23.3 with the blocked kernel's tasks one after another,
  // 64 x 64 x 31: 0.68 against 0.82, 32 x 32 x 16: 0.23 against 0.21); above, the
  // blocked one (280 x 300 x 31: 53 ms against k_jacobi's 84).
  const bool eig = o.negl_rel >= 0.0f;
  if (!eig && !jacobi_few(nr, nc) && (o.sched || nr > 256))
    return launch_jacobi_blk(d, nslices, W, V, t, max_sweeps, sweeps, work, st, o);
  const int pairs = (nc + 1) / 2, nw = pairs < 16 ? pairs : 16;  // k_jacobi's warps
  const float eps = FLT_EPSILON * 0.5f;
  const float tol = jacobi_tol0(nr), negl = eig ? o.negl_rel : ((float)nr * eps) * ((float)nr * eps);
  const size_t ws = d.P, vs = (size_t)nc * nc;
  if (nr <= 256) {
    const int KP = (nr + 31) / 32;
#define LRSTV_PK(K) \
  return launch_pk<K>(nslices, nr, nc, ws, vs, W, V, t, max_sweeps, tol, negl, sweeps, work, o, st)
    if (KP <= 1) LRSTV_PK(1);
    if (KP <= 2) LRSTV_PK(2);
    if (KP <= 4) LRSTV_PK(4);
    if (KP <= 5) LRSTV_PK(5);
    if (KP <= 7) LRSTV_PK(7);
    LRSTV_PK(8);
#undef LRSTV_PK
  }
  if (nr > 512) return cudaErrorInvalidValue;
  k_jacobi<<<nslices, 32 * nw, 0, st>>>(nr, nc, ws, vs, W, V, t, max_sweeps, tol, negl, sweeps, work, o);
  return cudaGetLastError();
}

}  // namespace lrstv

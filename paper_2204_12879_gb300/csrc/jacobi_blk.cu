// jacobi_blk.cu -- the blocked one-sided Jacobi SVD of the Fourier frontal
// slices in the t-SVT of the E-update (arXiv 2204.12879, eq. E_solution with
// Theorem 4.2's slice-wise t-SVD), with its dense products on the tensor cores.
//
// A slice's columns, ordered by norm (largest first), form panels of 16.  One
// task makes the 32 columns of a pair of panels mutually orthogonal:
//   1. Gram: G = P^H P of the pair's columns (tcgen05).  When no pair of them
//      needs a rotation the task ends here, with nothing else read or written.
//   2. Rotations: the usual cyclic Jacobi sweep over the pair's column pairs,
//      but two-sided on the 32 x 32 G and on the accumulated unitary Q, in
//      shared memory: a rotation touches some 100 values instead of the 800 of
//      two columns of W and V, and its test costs no inner product.
//   3. Update: W := W + W (Q - I), then V alike (tcgen05).
// G is formed afresh from W in every task, so the rounding of the two-sided
// updates does not accumulate: the method keeps one-sided Jacobi's accuracy.
// In a sweep the panels play a round-robin tournament: every round pairs them
// disjointly, and the first round's tasks also visit the pairs inside each
// panel, so that every column pair is visited once a sweep.  The order is set
// once, at the start: sorting again before every sweep took more sweeps and
// 10-15% more rotations (FP32 emulation, warm-started 64- and 200-column
// slices of iterations 5 to 20).
//
// Precision.  The products split their operands into two FP16 halves (22 bits)
// and form hi*hi + hi*lo + lo*hi with FP32 accumulation (the Gram adds lo*lo).
// W is scaled by a power of two that puts ||W||_F into [2^14, 2^15), V by 2^13
// and Q - I by 2^14, so that no half overflows and the low halves of every
// column that is not negligible stay above FP16's smallest step.  Between two
// tasks W and V are held in these halves alone: 22 bits, down to 2^-39 of ||W||_F
// (2^-38 in V), rounded once for each task that rotates the column, where FP32
// rotations on the columns round at each of their 16 to 31.  The t-SVT's error
// against FP64 is 0.60 to 0.90 of what such rotations left (22 cubes of 27 to 91
// pixels).  A slice that rotates nothing keeps its FP32 values.  The tensor
// core truncates its sums; the identity is added outside of it, in FP32, so
// that the truncation is relative to a task's change and does not shorten the
// columns task after task.  A rotation is applied as a' = a + m a - sigma b,
// b' = b + m b + conj(sigma) a with m = c - 1 = -s^2 / (1 + c) and sigma =
// s e^{i phase}: for small angles the rounding of c itself would make every
// rotation lengthen the columns by up to 3e-8 (4e-5 over the 1,500 rotations a
// column takes in a cold 200-column run); with m it does not.
//
// Layout.  During a run W and V live in scratch, as the MMA operands that the
// tasks read: a panel is 8 groups (Re hi of its columns 0-7 and 8-15, Re lo,
// then Im alike), a group holds 16 bytes (8 columns) of every row,
// rows contiguous.  A task's panels then arrive by two bulk copies with no
// instruction spent on them, and serve the update as the K-major A operand
// and the Gram as both MN-major operands.
//
// Schedules.  Tasks: every CTA takes tasks of any slice from a queue in global
// memory; a scheduler warp claims tasks, counts them off and queues the next
// round while the eight worker warps run.  Per slice: one CTA runs a slice's
// tasks one after another on W and V in place (for calls that have no scratch,
// slices above 256 rows; smaller ones are faster in FP32, svt.cu).  The pairs of
// a round touch disjoint columns and both schedules do the same arithmetic, so a
// slice's result is the same on either up to rounding: a value kept in FP32
// between two tasks and split again may get other halves of the same sum.
//
// What bounds it: the latency of a task's chain (16 rotation rounds of two
// barriers each, two loads, three MMA waits); 72 registers and one region of
// shared memory for W and then V let three CTAs share an SM up to 256 rows.
#include <cuda_fp16.h>
#include <float.h>

#include "jacobi_common.cuh"
#include "tc_ptx.cuh"

namespace lrstv {

namespace {

constexpr int kB = 16;              // panel width
constexpr int kW = 256;             // worker threads
constexpr int kT = kW + 32;         // and the ninth warp: rotations, scheduling
constexpr int kMaxTasks = 16;       // tasks of a round: 512 columns in 32 panels
constexpr int kMaxRounds = 32;
// The scratch holds the Gram's dump, then G, then Q as an operand.  In 10 KB the
// dump takes two passes and Q's lo has no -Im Q of its own; in 16 KB (kWide)
// neither holds, which is 1.5% faster in whole runs (sixteen cubes of 64 to 200
// columns, 12 iterations: 464 ms against 471) and is taken unless it costs an SM
// a CTA: with 10 KB three CTAs of 256 rows fit instead of two (256 x 256 x 191,
// 16 iterations with BF16X3: 250.9 -> 223.5 ms).
template <bool kWide>
constexpr size_t kScratch = kWide ? 16384 : 10240;
constexpr uint32_t kLoQ = 6144;  // Q's lo in the operand
constexpr float kScaleV = 8192.0f, kScaleQ = 16384.0f;
// A pair is left alone when the component of the smaller column along the
// larger is below kAbsTol ||W||_F: 1e-3 of an FP32 rounding of ||W||_F, and
// above the FP16 low halves' floor for columns near the negligible level.
constexpr float kAbsTol = 1e-3f * 0.5f * FLT_EPSILON;
constexpr unsigned long long kTaskWaitNs = 2000000000ull;  // a wait for work gives up after 2 s
constexpr long long kWorkerWait = 2000000;  // tries of a worker's wait for its scheduler (about 8 s)

// f16 operands, F32 accumulator, M = 128: the update (K-major operands; N = 64 or
// 32, bit 13: A negated) and the Gram (N = 128, MN-major operands: transpose bits
// 15, 16)
constexpr uint32_t kIdescUpd = (1u << 4) | ((64u >> 3) << 17) | ((128u >> 4) << 24);
constexpr uint32_t kIdescUpdIm = (1u << 4) | ((32u >> 3) << 17) | ((128u >> 4) << 24);
constexpr uint32_t kIdescUpdRe = kIdescUpdIm | (1u << 13);
constexpr uint32_t kIdescGram =
    (1u << 4) | (1u << 15) | (1u << 16) | ((128u >> 3) << 17) | ((128u >> 4) << 24);

__device__ __forceinline__ unsigned long long gtimer() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}
// barrier of the eight worker warps
__device__ __forceinline__ void wsync() { asm volatile("bar.sync 1, 256;" ::: "memory"); }
__device__ __forceinline__ bool wsync_and(bool v) {
  uint32_t r;
  asm volatile(
      "{\n .reg .pred p, q;\n setp.ne.u32 p, %1, 0;\n bar.red.and.pred q, 1, 256, p;\n"
      " selp.u32 %0, 1, 0, q;\n}\n"
      : "=r"(r)
      : "r"((uint32_t)v)
      : "memory");
  return r != 0;
}
// barriers of the whole CTA: workers and the ninth warp
__device__ __forceinline__ void csync() { asm volatile("bar.sync 2, 288;" ::: "memory"); }
// ... and of a rotation round's copy c, where one side arrives without waiting:
// its state is published (the ninth warp waits), its rotations are formed (the
// workers wait)
__device__ __forceinline__ void state_arrive(int c) {
  if (c)
    asm volatile("bar.arrive 4, 288;" ::: "memory");
  else
    asm volatile("bar.arrive 3, 288;" ::: "memory");
}
__device__ __forceinline__ void state_sync(int c) {
  if (c)
    asm volatile("bar.sync 4, 288;" ::: "memory");
  else
    asm volatile("bar.sync 3, 288;" ::: "memory");
}
__device__ __forceinline__ void formed_arrive(int c) {
  if (c)
    asm volatile("bar.arrive 6, 288;" ::: "memory");
  else
    asm volatile("bar.arrive 5, 288;" ::: "memory");
}
__device__ __forceinline__ void formed_sync(int c) {
  if (c)
    asm volatile("bar.sync 6, 288;" ::: "memory");
  else
    asm volatile("bar.sync 5, 288;" ::: "memory");
}
// ... and where one state of G has one copy: it has been read by all (the ninth
// warp does not wait)
__device__ __forceinline__ void state_read() { asm volatile("bar.sync 7, 288;" ::: "memory"); }
__device__ __forceinline__ void state_read_arrive() {
  asm volatile("bar.arrive 7, 288;" ::: "memory");
}

__host__ __device__ inline int panels_of(int nc) { return (nc + kB - 1) / kB; }
// with an empty panel that makes an odd number even
__host__ __device__ inline int players_of(int npan) { return npan + (npan & 1); }
__host__ __device__ inline int rows16(int n) { return (n + 15) & ~15; }
// scratch bytes of one slice's W and V
__host__ __device__ inline size_t op_bytes(int nr, int nc) {
  return (size_t)players_of(panels_of(nc)) * (rows16(nr) + rows16(nc)) * 128;
}
// rounds of a sweep
__host__ __device__ inline int rounds_of(int npan) { return players_of(npan) - 1; }
// pair i of round r: panels p < q; false: no such task.  The panel that meets
// the empty one has a task in round 0 only (its own pairs).
__device__ __forceinline__ bool round_pair(int npan, int r, int i, int &p, int &q) {
  const int np = players_of(npan);
  if (i >= np / 2) return false;
  pair_of(r, i, np, p, q);
  if (p > q) {
    const int x = p;
    p = q;
    q = x;
  }
  return q < npan || r == 0;
}

int queue_cap(int nslices) {
  // a slot is reused only after the ring has wrapped: queued-but-untaken
  // tasks stay below one round per live slice and claimed-but-unfilled slots
  // below one per worker CTA, under the capacity
  int cap = 4096;
  while (cap < kMaxTasks * nslices + 4096) cap <<= 1;
  return cap;
}

// pair index of panel p in round r
__device__ __forceinline__ int pair_index(int np, int r, int p) {
  if (p == np - 1 || p == r) return 0;
  const int d = p > r ? p - r : p - r + np - 1;
  return d <= (np - 2) / 2 ? d : np - 1 - d;
}

// Scratch of the task queue (ints; jacobi_task_ints): the header, the queue and
// per-slice state, zeroed before each launch, then per slice the column order
// and, 256-byte aligned, the operands.  A task of round r > 0 is ready when
// both of its panels have had their task of the round before (an arrival
// each, counted from one sweep to the next: ready on every second one); a sweep's
// round 0 starts when every task of the sweep before is done.  A task is done
// for this when W is and the panels' V of the tasks before (vdone): V, which
// nothing but the panels' next V update reads, follows a round behind, and is
// waited for only when a round's W overtakes the V of the round before.
struct Sched {
  int *head, *tail, *finished, *err, *npend, *pend_head, *live;
  int *sweep, *left, *pend, *packed;
  int *vdone;                // per slice, `pan`: stamp of the panel's last task whose V is done
  float4 *lim;               // tol^2, negligible squared norm, kAbsTol^2 ||W||_F^2 (all scaled), 1 / scale
  unsigned long long *slot;  // (mark << 32) | task; the i-th task's mark is i + 1
  int *arrive;               // per slice, `per` (rounds x pairs): arrivals
  int *perm;                 // per slice, `cols`: position -> column
  int cap, cols, per, pan;
  __host__ __device__ Sched(int *s, int ns, int cap_, int cols_)
      : cap(cap_), cols(cols_), per(pairs_of(cols_)), pan(players_of(panels_of(cols_))) {
    head = s;
    tail = s + 1;
    finished = s + 2;
    err = s + 3;
    npend = s + 4;
    pend_head = s + 5;
    live = s + 6;
    slot = (unsigned long long *)(s + 8);
    lim = (float4 *)(slot + cap);
    sweep = (int *)(lim + ns);
    left = sweep + ns;
    pend = left + ns;
    packed = pend + ns;
    arrive = packed + ns;
    vdone = arrive + (size_t)per * ns;
    perm = vdone + (size_t)pan * ns;
  }
  __host__ __device__ static int pairs_of(int nc) {  // rounds x pairs of a round
    const int np = players_of(panels_of(nc));
    return (np - 1) * (np / 2);
  }
  static size_t zeroed(int ns, int cap_, int cols_) {  // ints zeroed before a launch
    return 8 + 2 * (size_t)cap_ + (8 + (size_t)pairs_of(cols_) + players_of(panels_of(cols_))) * ns;
  }
  static size_t ints(int ns, int cap_, int cols_) {  // ints before the operands
    return (zeroed(ns, cap_, cols_) + (size_t)cols_ * ns + 63) / 64 * 64;
  }
  // the stamp of panel p's task before the one of round r in sweep sw (0: none)
  __device__ static int stamp_before(int npan, int sw, int r, int p) {
    const int np = players_of(npan), n = np - 1;
    for (;;) {
      if (--r < 0) {
        r = n - 1;
        if (--sw < 0) return 0;
      }
      int x, y;
      if (round_pair(npan, r, pair_index(np, r, p), x, y)) return sw * n + r + 1;
    }
  }
  // a task: (s kMaxRounds + r) kMaxTasks + its pair index in the round
  __device__ static int task_of(int s, int r, int i) {
    return (s * kMaxRounds + r) * kMaxTasks + i;
  }
  // queues n tasks; what they read was written before (one thread)
  __device__ void push(const int *task, int n) {
    if (n <= 0) return;
    __threadfence();
    const int idx = atomicAdd(tail, n);
    for (int k = 0; k < n; ++k)
      *(volatile unsigned long long *)(slot + ((idx + k) & (cap - 1))) =
          ((unsigned long long)(unsigned)(idx + k + 1) << 32) | (unsigned)task[k];
  }
  // starts a sweep of slice s: its first round's tasks; returns their number
  __device__ int begin_sweep(int s, int npan, int *task) {
    const int np = players_of(npan);
    // an odd number of panels: one has no partner in the rounds after the first
    left[s] = (np - 1) * (np / 2) - (npan & 1) * (np - 2);
    for (int i = 0; i < np / 2; ++i) task[i] = task_of(s, 0, i);
    return np / 2;
  }
};

struct Run {
  int nslices, nr, nc;      // one shape: slice s at W + s ws, V + s vs
  size_t ws, vs;
  float2 *W, *V;
  float t, tol0, negl_rel;
  int max_sweeps;
  int *sweeps;
  unsigned long long *work;
  JacOpt o;
  const SliceTask *list;    // or a list of slices of any shapes (threshold alpha / mu)
  double mu;
  int keep;
  int *sched;
  char *op;                 // one shape: the operands, slice s at op + s op_bytes
  int cap, cols;
  int live_max;             // slices in flight at most (task schedule)
  int rows;                 // rows of the tallest slice, rounded up to 16
};

struct Slice {
  int nr, nc, warm;
  float2 *W, *V;
  char *op;
  float t, skip_t, tol0, negl_rel, gms2;
  int *sweeps;
  bool pre;
};

__device__ __forceinline__ Slice slice_of(const Run &a, int s) {
  Slice x;
  x.warm = a.o.warm;
  if (a.list) {
    const SliceTask tk = a.list[s];
    const float eps = FLT_EPSILON * 0.5f;
    x.nr = tk.nr;
    x.nc = tk.nc;
    x.W = tk.W;
    x.V = tk.V;
    x.op = tk.op;
    x.skip_t = (float)((double)tk.alpha / a.mu);
    x.t = a.keep ? -1.0f : x.skip_t;
    x.tol0 = 8.0f * sqrtf((float)tk.nr) * eps;
    x.negl_rel = ((float)tk.nr * eps) * ((float)tk.nr * eps);
    x.gms2 = tk.ms2 ? *tk.ms2 : -1.0f;
    x.sweeps = tk.sweeps;
    x.pre = tk.conv && *tk.conv != 0;
  } else {
    x.nr = a.nr;
    x.nc = a.nc;
    x.W = a.W + (size_t)s * a.ws;
    x.V = a.V + (size_t)s * a.vs;
    x.op = a.op + (size_t)s * op_bytes(a.nr, a.nc);
    x.skip_t = a.o.t_svt;
    x.t = a.t;
    x.tol0 = a.tol0;
    x.negl_rel = a.negl_rel;
    x.gms2 = a.o.ms2 ? a.o.ms2[s / a.o.group] : -1.0f;
    x.sweeps = a.sweeps + s;
    x.pre = a.o.conv && a.o.conv[s] != 0;
  }
  return x;
}

// Squared column norms of a slice into key[0..nc) and their sum, by the whole
// CTA (a warp per column); s_red: 32 floats.  W was written by an earlier launch.
__device__ float norms_and_sum(int nr, int nc, const float2 *W, float *key, float *s_red) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
  for (int c = warp; c < nc; c += nw) {
    const float2 *w = W + (size_t)nr * c;
    float p0 = 0.f, p1 = 0.f;
    int r = lane;
    for (; r + 96 < nr; r += 128) {
      const float2 x = w[r], y = w[r + 32], z = w[r + 64], u = w[r + 96];
      p0 = fmaf(x.x, x.x, fmaf(x.y, x.y, p0));
      p1 = fmaf(y.x, y.x, fmaf(y.y, y.y, p1));
      p0 = fmaf(z.x, z.x, fmaf(z.y, z.y, p0));
      p1 = fmaf(u.x, u.x, fmaf(u.y, u.y, p1));
    }
    for (; r < nr; r += 32) {
      const float2 x = w[r];
      p0 = fmaf(x.x, x.x, fmaf(x.y, x.y, p0));
    }
    p0 = warp_sum(p0 + p1);
    if (lane == 0) key[c] = p0;
  }
  __syncthreads();
  float part = 0.f;
  for (int c = threadIdx.x; c < nc; c += blockDim.x) part += key[c];
  part = warp_sum(part);
  if (lane == 0) s_red[warp] = part;
  __syncthreads();
  float sum = 0.f;
  for (int w = 0; w < nw; ++w) sum += s_red[w];
  __syncthreads();
  return sum;
}

// The power of two that scales W for the FP16 split: ||W||_F s in [2^14, 2^15),
// for every finite ||W||_F^2 (slice_start lets no other slice run).
__device__ __forceinline__ float w_scale(float fro2) {
  if (!(fro2 > 0.0f) || !(fro2 <= FLT_MAX)) return 1.0f;
  int e = ilogbf(sqrtf(fro2));
  e = e < -100 ? -100 : (e > 100 ? 100 : e);
  return ldexpf(1.0f, 14 - e);
}

// The limits of a slice's rotations, in the scaled units of its operands.
__device__ __forceinline__ float4 limits(const Slice &x, float fro2) {
  const float tol = pk_tolerance(x.tol0, fro2, x.nc, x.skip_t, x.gms2);
  const float sc = w_scale(fro2), f = fro2 * sc * sc;
  return make_float4(tol * tol, x.negl_rel * f, kAbsTol * kAbsTol * f, 1.0f / sc);
}

// FP16 + FP32 and FP16 - FP32 in one instruction (no conversion first)
__device__ __forceinline__ float add_h(__half h, float x) {
  float r;
  asm("add.f32.f16 %0, %1, %2;" : "=f"(r) : "h"(__half_as_ushort(h)), "f"(x));
  return r;
}
__device__ __forceinline__ float sub_h(__half h, float x) {
  float r;
  asm("sub.f32.f16 %0, %1, %2;" : "=f"(r) : "h"(__half_as_ushort(h)), "f"(x));
  return r;
}
__device__ __forceinline__ __half2 pair_of_halves(uint32_t v) { return *(const __half2 *)&v; }

// eight values split into FP16 halves: 16 bytes of hi, 16 of lo
__device__ __forceinline__ void split8(const float (&x)[8], uint4 &hi, uint4 &lo) {
  uint32_t h[4], l[4];
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    const __half2 a = __floats2half2_rn(x[2 * j], x[2 * j + 1]);
    const __half2 b = __floats2half2_rn(-sub_h(__low2half(a), x[2 * j]),
                                        -sub_h(__high2half(a), x[2 * j + 1]));
    h[j] = *(const uint32_t *)&a;
    l[j] = *(const uint32_t *)&b;
  }
  hi = make_uint4(h[0], h[1], h[2], h[3]);
  lo = make_uint4(l[0], l[1], l[2], l[3]);
}
// ... and joined again, added to x
__device__ __forceinline__ void join8(const uint4 &hi, const uint4 &lo, float (&x)[8]) {
  const uint32_t h[4] = {hi.x, hi.y, hi.z, hi.w}, l[4] = {lo.x, lo.y, lo.z, lo.w};
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    const __half2 a = pair_of_halves(h[j]), b = pair_of_halves(l[j]);
    x[2 * j] = add_h(__low2half(a), add_h(__low2half(b), x[2 * j]));
    x[2 * j + 1] = add_h(__high2half(a), add_h(__high2half(b), x[2 * j + 1]));
  }
}

// Group `g` of a panel (0: columns 0-7, 1: columns 8-15) of one row as operand
// rows: dst + 16 row, groups of `rows` rows.
__device__ __forceinline__ void put_row(char *dst, int rows, int row, int g, const float2 (&x)[8],
                                        float scale) {
  float re[8], im[8];
#pragma unroll
  for (int j = 0; j < 8; ++j) {
    re[j] = x[j].x * scale;
    im[j] = x[j].y * scale;
  }
  const size_t step = (size_t)rows * 32;  // Re hi, Re lo, Im hi, Im lo: two groups each
  char *d = dst + ((size_t)g * rows + row) * 16;
  uint4 hi, lo;
  split8(re, hi, lo);
  *(uint4 *)d = hi;
  *(uint4 *)(d + step) = lo;
  split8(im, hi, lo);
  *(uint4 *)(d + 2 * step) = hi;
  *(uint4 *)(d + 3 * step) = lo;
}

// `np` panels of columns cols[16 p ..] (-1: zero) of M (n rows) into dst as
// operands of `rows` rows, zero past n; thread `tid` of `nt`.  M null: the
// identity.  The loads bypass L1 (the per-slice schedule reads what the CTA
// wrote).
__device__ __forceinline__ void pack_panels(char *dst, const float2 *M, int n, int rows, int np,
                                            const int *cols, float scale, int tid, int nt) {
  for (int u = tid; u < 2 * rows * np; u += nt) {
    const int pg = u / rows, r = u - pg * rows;  // panel and group, row
    float2 x[8];
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      const int c = cols[8 * pg + j];
      x[j] = make_float2(0.f, 0.f);
      if (M) {
        if (c >= 0 && r < n) x[j] = __ldcg(M + (size_t)n * c + r);
      } else if (c == r) {
        x[j].x = 1.0f;
      }
    }
    put_row(dst + (size_t)(pg >> 1) * rows * 128, rows, r, pg & 1, x, scale);
  }
}

// Shared memory of one CTA: the pair's columns of W, then of V, as operands
// (`A`: panel a's 8 groups, then panel b's), and the scratch (`S`).
struct Smem {
  char *A, *S;
  uint32_t bar[2], bar_w, bar_v, bar_task, bar_done, bar_vdone;
  uint32_t tmem;     // 128 columns: the Gram, then two 64-column update tiles
  float4 *par;       // 2 x 16: a round's rotations (m, sigma)
  float2 *piv;       // 16: the first round's G(p, q)
  float *diag;       // 32: G's diagonal at first
  unsigned *rounds;  // the rounds that rotate a pair
};

struct Rot2 {
  float m, sr, si;  // c - 1, Re and Im of s e^{i phase}
};

// whether a pair is rotated: beyond the tolerance, no column negligible
__device__ __forceinline__ bool rotates(float al, float be, float g2, const float4 &lim) {
  return (al > lim.y) & (be > lim.y) & (g2 > lim.x * (al * be)) & (g2 > lim.z * fmaxf(al, be));
}

__device__ __forceinline__ float rsqrt_ftz(float x) {
  float r;
  asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
}
__device__ __forceinline__ float rcp_ftz(float x) {
  float r;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
}

// Rotation of the Hermitian [[al, g], [conj g, be]], g2 = |g|^2, by the smaller
// angle: with d = (be - al) / 2 and h = sqrt(d^2 + g2), cos^2 = (1 + |d| / h) / 2
// and sin = |g| / (2 h cos), so that the phase conj(g) / |g| needs no division.
// The diagonal becomes al - shift, be + shift (shift = tan |g|).  An error of
// either reciprocal root turns the angle, not the columns' lengths: m follows
// from the sigma that is applied.
__device__ __forceinline__ Rot2 make_rot2(float al, float be, float2 g, float g2, float &shift) {
  const float d = 0.5f * (be - al);
  const float ih = rsqrt_ftz(fmaf(d, d, g2));
  const float c2 = fmaf(0.5f * fabsf(d), ih, 0.5f);
  const float ic = rsqrt_ftz(c2);
  const float f = copysignf(0.5f * ih * ic, d);  // sin / |g|
  Rot2 r;
  r.sr = f * g.x;
  r.si = -f * g.y;
  r.m = -(f * f) * g2 * rcp_ftz(fmaf(c2, ic, 1.0f));
  shift = f * g2 * ic;
  return r;
}

// a' = a + m a - sigma b, b' = b + m b + conj(sigma) a
__device__ __forceinline__ void rot_cols(float2 &a, float2 &b, const Rot2 &r) {
  const float2 x = a, y = b;
  a.x = fmaf(-r.sr, y.x, fmaf(r.si, y.y, fmaf(r.m, x.x, x.x)));
  a.y = fmaf(-r.sr, y.y, fmaf(-r.si, y.x, fmaf(r.m, x.y, x.y)));
  b.x = fmaf(r.sr, x.x, fmaf(r.si, x.y, fmaf(r.m, y.x, y.x)));
  b.y = fmaf(r.sr, x.y, fmaf(-r.si, x.x, fmaf(r.m, y.y, y.y)));
}
// the same for two rows of J^H G: a' = a + m a - conj(sigma) b, b' = b + m b + sigma a
__device__ __forceinline__ void rot_rows(float2 &a, float2 &b, const Rot2 &r) {
  Rot2 q = r;
  q.si = -r.si;
  rot_cols(a, b, q);
}
// The MMAs of G's real products: D (128 x 128) = P^T P of the pair's 128 operand
// columns (one thread).
__device__ __forceinline__ void issue_gram(uint32_t d, uint32_t a, int rows, uint32_t bar) {
  tc_fence_after();
  uint64_t x = tc_desc(a, 128, (uint32_t)rows * 16);
  for (int k = 0; k < rows / 16; ++k, x += 16)  // 256 bytes on
    tc_mma_f16(d, x, x, kIdescGram, k > 0 ? 1u : 0u);
  tc_commit(bar);
}

// The MMAs of one 128-row tile of an update: D (128 x 64: Re, then Im, of both
// panels' columns) = tile (Q - I), the small split products first (one thread).
// The columns' real parts meet [Re Q, Im Q], their imaginary parts [-Im Q, Re Q]:
// two windows of Q's hi, which holds -Im Q, Re Q and Im Q; where the lo has no
// -Im Q, two MMAs with N = 32, one with A negated, take its place.
template <bool kWide>
__device__ __forceinline__ void issue_update(uint32_t d, uint32_t a, int rows, uint32_t q,
                                             uint32_t bar) {
  const uint64_t x = tc_desc(a, (uint32_t)rows * 16, 128), y = tc_desc(q, 1536, 128),
                 z = tc_desc(q + kLoQ, kWide ? 1536 : 1024, 128);
  const uint32_t lo = (uint32_t)(2 * rows);
#pragma unroll
  for (int k = 0; k < 4; ++k) {  // Re a, Im a, Re b, Im b
    const uint64_t xk = x + (uint32_t)(4 * k * rows);
    const uint32_t at = 192 * (k >> 1) + ((k & 1) ? 0 : 32);
    const uint64_t yk = y + at, zk = z + (kWide ? at : 128 * (k >> 1));
    if (!kWide && (k & 1)) {
      tc_mma_f16(d, xk, zk + 32, kIdescUpdRe, 1u);
      tc_mma_f16(d + 32, xk, zk, kIdescUpdIm, 1u);
    } else {
      tc_mma_f16(d, xk, zk, kIdescUpd, k > 0 ? 1u : 0u);
    }
    tc_mma_f16(d, xk + lo, yk, kIdescUpd, 1u);
  }
#pragma unroll
  for (int k = 0; k < 4; ++k)
    tc_mma_f16(d, x + (uint32_t)(4 * k * rows),
               y + 192 * (k >> 1) + ((k & 1) ? 0 : 32), kIdescUpd, 1u);
  tc_commit(bar);
}

// Waits of one CTA's accumulators: the parity of each barrier's next commit
// (bits 0, 1) and, in warp 0, the commits not yet seen complete.  Only warp 0
// polls, the other warps wait at the worker barrier: eight polling warps took a
// quarter of the SM's issue slots from the CTAs beside them.
struct Waits {
  unsigned ph = 0, out = 0;
  __device__ __forceinline__ bool mma(const Smem &sm, int i, bool ok) {
    if (threadIdx.x < 32 && ok) {
      ok = mbar_wait(sm.bar[i], (ph >> i) & 1u);
      if (ok) out &= ~(1u << i);
    }
    ph ^= 1u << i;
    tc_fence_before();
    ok = wsync_and(ok);
    tc_fence_after();
    return ok;
  }
};

// The rotations' shared state (sm.S and sm.par): a round's rotations, its
// state of G, and the blocks that the next round's rotations come from, in two
// copies.  A worker that has rotated G publishes state r + 1 without waiting,
// rotates Q, and then waits for round r + 1's rotations (and so for the other
// workers' states); the ninth warp forms them from state r meanwhile.  With one
// barrier of all a round, both chains had to end before either went on: 600
// cycles a round; with mbarriers in place of the hardware's named ones, 900.
// Across the panels, round r pairs a_k with b_(k + r); only the rounds in which
// some pair is beyond the tolerance at first are run (a pair that other
// rotations push beyond it waits for the next sweep; about a third of the
// rounds fall away, with the same sweeps and rotations in emulation).  From a
// round to the next, d rounds on, thread (i, k)'s b-row values come from the
// threads of row i + d, through BA and BB; the blocks (i, i + d') that hold the
// round after's pairs are published in AX (aa) and AB (ab).
// All 32 columns (the first round's tasks): a tournament of 31 rounds in which
// pair k is (a_k, b_k) and after a round a_0 stays, a_1 := b_0, a_k := a_(k-1),
// b_k := b_(k+1), b_15 := a_15; G moves through shared memory, in one copy that
// is rewritten when all workers and the ninth warp have read it.
__device__ __forceinline__ int from_a(int j) { return j == 0 ? 0 : (j == 1 ? 16 : j - 1); }
__device__ __forceinline__ int from_b(int j) { return j == 15 ? 15 : 17 + j; }
// the round after round r in the mask of those left (0: none)
__device__ __forceinline__ int after(unsigned left, int r) { return left ? __ffs(left) - 1 - r : 0; }
struct Cross {
  float2 BA[2][256], BB[2][256], AX[2][16], AB[2][16];
};
struct Whole {
  float2 G[1024];
};
static_assert(sizeof(Cross) <= kScratch<false> && sizeof(Whole) <= kScratch<false>, "the scratch holds them");

// Steps 1 and 2 of a task by the worker warps, W's operands being in sm.A
// (`rows` rows; ok: warp 0 saw them arrive): G, the rotations, and Q - I as an operand in
// sm.S.  Returns 1 (rotated), 0 (no pair needed it) or -1 (a wait ran out).
// The ninth warp runs form_rotations beside it.
template <bool kWide>
__device__ int gram_rotate(const Smem &sm, int rows, bool own, const float4 &lim, Waits &wt,
                           bool ok) {
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  if (tid == 0) {
    *sm.rounds = 0;
    if (ok) issue_gram(sm.tmem, smem_u32(sm.A), rows, sm.bar[0]);
  }
  if (ok) wt.out |= 1u;
  if (!wt.mma(sm, 0, ok)) {
    csync();
    return -1;
  }
  // Thread (i, k) holds the 2 x 2 block of G's rows a_i, b_i and columns a_k, b_k
  // (a_j, b_j: column j of panel a, of panel b) and Q's rows 2i, 2i + 1 there.
  // D's rows and columns: panel, Re/Im, hi/lo, column (1, 1, 1, 4 bits).  A lane
  // adds hi and lo of its row's columns, then the lanes l and l + 16 (a row's hi
  // and lo) exchange halves: l keeps the sums of the columns' Re (h = 0), l + 16
  // of their Im.  The rows that are Re, then those that are Im, go to
  // S[h][column][row], the row XOR-ed so that the two i of a warp read different
  // banks.
  // G(p, q) = conj(w_p) . w_q is read as conj(G(q, p)): the lanes' q are D's rows.
  const int i = tid >> 4, k = tid & 15;
  float *S = (float *)sm.S;
  float2 aa, ab, ba, bb;
  {
    const uint32_t at = sm.tmem + ((uint32_t)(32 * (warp & 3)) << 16) + 64 * (warp >> 2);
    float x[16];
    {
      uint32_t v[16], w[16];
      tc_ld16(at, v);
      tc_ld16(at + 16, w);
      tc_wait_ld();
#pragma unroll
      for (int j = 0; j < 16; ++j) x[j] = __uint_as_float(v[j]) + __uint_as_float(w[j]);
      tc_ld16(at + 32, v);
      tc_ld16(at + 48, w);
      tc_wait_ld();
      const bool up = lane > 15;
#pragma unroll
      for (int j = 0; j < 16; ++j) {
        const float y = __uint_as_float(v[j]) + __uint_as_float(w[j]);
        x[j] = (up ? y : x[j]) + __shfl_xor_sync(0xffffffffu, up ? x[j] : y, 16);
      }
    }
    float *d = S + (kWide ? 2048 * (warp & 1) : 0) + 1024 * (lane >> 4) + 512 * (warp >> 2) + k;
    const int f = 16 * (((warp >> 1) ^ (lane >> 4)) & 1);
    auto store = [&]() {
#pragma unroll
      for (int j = 0; j < 16; ++j) d[32 * j + (f ^ (16 * (j & 1)))] = x[j];
    };
    if (kWide || !(warp & 1)) store();
    wsync();
    auto part = [&](int n, int q, float &re, float &im) {  // q . Re p, q . Im p
      const float *y = S + 32 * n + k;
      const int e = 16 * ((q ^ i) & 1);
      re = y[e];
      im = y[1024 + 16 - e];
    };
    part(i, 0, aa.x, aa.y);
    part(i, 1, ab.x, ab.y);
    part(16 + i, 0, ba.x, ba.y);
    part(16 + i, 1, bb.x, bb.y);
    if (kWide) {
      S += 2048;
    } else {
      wsync();
      if (warp & 1) store();
      wsync();
    }
    auto second = [&](int n, int q, float2 &g) {
      float re, im;
      part(n, q, re, im);
      g = make_float2(g.x + im, re - g.y);
    };
    second(i, 0, aa);
    second(i, 1, ab);
    second(16 + i, 0, ba);
    second(16 + i, 1, bb);
    wsync();
  }
  // the diagonal, and the rounds in which a pair needs a rotation
  Cross *X = (Cross *)sm.S;
  Whole *A = (Whole *)sm.S;
  const int ga = 32 * from_a(i), gb = 32 * from_b(i), ca = from_a(k), cb = from_b(k);
  if (i == k) {
    sm.diag[k] = aa.x;
    sm.diag[16 + k] = bb.x;
    if (own) sm.piv[k] = ab;
  }
  if (own) {
    A->G[ga + ca] = aa;
    A->G[ga + cb] = ab;
    A->G[gb + ca] = ba;
    A->G[gb + cb] = bb;
  }
  wsync();
  {
    const float dai = sm.diag[i], dbi = sm.diag[16 + i], dak = sm.diag[k], dbk = sm.diag[16 + k];
    auto test = [&](float al, float be, float2 g) {
      return rotates(al, be, fmaf(g.x, g.x, g.y * g.y), lim);
    };
    bool need = test(dai, dbk, ab);
    if (own && i < k) need = need || test(dai, dak, aa) || test(dbi, dbk, bb);
    // bit k of half h: the pair (a_i, b_k), i = 2 warp + h, of round k - i
    const unsigned b = __ballot_sync(0xffffffffu, need);
    const unsigned lo = (b & 0xffffu) * 0x10001u, hi = (b >> 16) * 0x10001u;
    const unsigned m = ((lo >> (2 * warp)) | (hi >> (2 * warp + 1))) & 0xffffu;
    if (lane == 0 && m) atomicOr(sm.rounds, m);
  }
  csync();
  const unsigned rounds = *sm.rounds;
  if (!rounds) return 0;

  float4 qa = make_float4(k == 2 * i ? 1.f : 0.f, k == 2 * i + 1 ? 1.f : 0.f, 0.f, 0.f);
  float4 qb = make_float4(16 + k == 2 * i ? 1.f : 0.f, 16 + k == 2 * i + 1 ? 1.f : 0.f, 0.f, 0.f);
  auto apply_g = [&](const Rot2 &rk, const Rot2 &ri) {  // its columns' rotations, its rows'
    rot_cols(aa, ab, rk);
    rot_cols(ba, bb, rk);
    rot_rows(aa, ba, ri);
    rot_rows(ab, bb, ri);
  };
  auto apply_q = [&](const Rot2 &rk) {
    float2 x = make_float2(qa.x, qa.z), y = make_float2(qb.x, qb.z);
    rot_cols(x, y, rk);
    float2 z = make_float2(qa.y, qa.w), w = make_float2(qb.y, qb.w);
    rot_cols(z, w, rk);
    qa = make_float4(x.x, z.x, x.y, z.y);
    qb = make_float4(y.x, w.x, y.y, w.y);
  };
  auto shfl4 = [](float4 v, int src) {
    return make_float4(__shfl_sync(0xffffffffu, v.x, src), __shfl_sync(0xffffffffu, v.y, src),
                       __shfl_sync(0xffffffffu, v.z, src), __shfl_sync(0xffffffffu, v.w, src));
  };
  if (own) {
    const int w = 32 * i + k;
    state_arrive(0);
    for (int r = 0; r < 31; ++r) {
      formed_sync(r & 1);
      float2 *G = A->G;
      const float4 u = sm.par[16 * (r & 1) + k], v = sm.par[16 * (r & 1) + i];
      const Rot2 rk = {u.x, u.y, u.z}, ri = {v.x, v.y, v.z};
      aa = G[ga + ca];
      ab = G[ga + cb];
      ba = G[gb + ca];
      bb = G[gb + cb];
      apply_g(rk, ri);
      if (r < 30) {
        state_read();
        G[w] = aa;
        G[w + 16] = ab;
        G[w + 512] = ba;
        G[w + 528] = bb;
        state_arrive((r + 1) & 1);
      }
      apply_q(rk);
      const float4 t = shfl4(k == 0 ? qb : qa, (lane & 16) | ((k + 15) & 15));
      const float4 z = shfl4(qb, (lane & 16) | ((k + 1) & 15));
      qb = k == 15 ? qa : z;
      qa = k == 0 ? qa : t;
    }
  } else {
    // to the first round, whose pairs the ninth warp takes from piv
    unsigned left = rounds & (rounds - 1);
    int r = __ffs(rounds) - 1, d = r, d2 = after(left, r);
    if (k == ((i + d) & 15)) sm.piv[i] = ab;
    // G into copy n for a state d rounds on, d2 the move after that (block (i, i + d2)
    // of that state: its ab is still d columns on here), then the columns
    auto move = [&](int n, bool pa, bool pb) {
      X->BA[n][tid] = ba;
      X->BB[n][tid] = bb;
      if (pa) X->AX[n][i] = aa;
      if (pb) X->AB[n][i] = ab;
      state_arrive(n);
    };
    auto columns = [&](int from) {
      ab.x = __shfl_sync(0xffffffffu, ab.x, from);
      ab.y = __shfl_sync(0xffffffffu, ab.y, from);
      qb = shfl4(qb, from);
    };
    move(0, k == ((i + d2) & 15), k == ((i + d + d2) & 15));
    columns((lane & 16) | ((k + d) & 15));
    auto step = [&](int c) -> bool {  // a round on copy c; true after the last
      // what does not wait for the round comes before it
      const int row = (tid + 16 * d) & 0xff;
      const float2 *pa = X->BA[c] + row, *pb = X->BB[c] + ((row & 0xf0) | ((k + d) & 15));
      const bool last = !left;
      d = d2;
      r += d;
      left &= left - 1;
      d2 = after(left, r);
      const int from = (lane & 16) | ((k + d) & 15);
      const bool ea = k == ((i + d2) & 15), eb = k == ((i + d + d2) & 15);
      formed_sync(c);
      const float4 u = sm.par[16 * c + k], v = sm.par[16 * c + i];
      const Rot2 rk = {u.x, u.y, u.z}, ri = {v.x, v.y, v.z};
      ba = *pa;
      bb = *pb;
      apply_g(rk, ri);
      if (!last) move(c ^ 1, ea, eb);
      apply_q(rk);
      if (!last) columns(from);
      return last;
    };
    while (!step(0) && !step(1)) {
    }
    qb = shfl4(qb, (lane & 16) | ((k + 16 - r) & 15));  // home
  }
  // Q - I as the K-major operand: output n = -Im (see issue_update), Re, Im times panel
  // and column; input = panel, column.  This thread: inputs 2i and 2i + 1 (one
  // 4-byte word), outputs a_k and b_k.
  wsync();
  {
    const int d = k - 2 * i;  // 0, 1: the diagonal is in a_k; 16, 17 below: in b_k
    qa.x -= d == 0 ? 1.f : 0.f;
    qa.y -= d == 1 ? 1.f : 0.f;
    qb.x -= d + 16 == 0 ? 1.f : 0.f;
    qb.y -= d + 16 == 1 ? 1.f : 0.f;
    // inputs 2i, 2i + 1: k-group i >> 2
    char *hi = sm.S + (i >> 2) * 1536 + 512 + (i & 3) * 4 + k * 16;
    char *lo = kWide ? hi + kLoQ : sm.S + kLoQ + (i >> 2) * 1024 + (i & 3) * 4 + k * 16;
    auto put = [&](int at, float x, float y, bool im) {
      const __half2 h = __floats2half2_rn(x * kScaleQ, y * kScaleQ);
      const float2 f = __half22float2(h);
      const __half2 l = __floats2half2_rn(fmaf(x, kScaleQ, -f.x), fmaf(y, kScaleQ, -f.y));
      *(__half2 *)(hi + at) = h;
      *(__half2 *)(lo + at) = l;
      if (im) *(__half2 *)(hi + at - 1024) = __hneg2(h);
      if (im && kWide) *(__half2 *)(lo + at - 1024) = __hneg2(l);
    };
    put(0, qa.x, qa.y, false);
    put(256, qb.x, qb.y, false);
    put(512, qa.z, qa.w, true);
    put(768, qb.z, qb.w, true);
  }
  tc_fence_smem();
  tc_fence_before();
  wsync();
  return 1;
}

// base + m base + coef other: one column (or row) of a rotated pair
__device__ __forceinline__ float2 rot_one(float2 base, float2 other, float m, float cr, float ci) {
  return make_float2(fmaf(-ci, other.y, fmaf(cr, other.x, fmaf(m, base.x, base.x))),
                     fmaf(ci, other.x, fmaf(cr, other.y, fmaf(m, base.y, base.y))));
}

// The ninth warp's part of a task: the rotations of every round, one round
// ahead of the workers.  Lane k (and k + 16) owns pair k.  While the workers
// apply round r, it forms from the same state the entries that round r + 1
// pairs (a 2 x 2 block, rotated from both sides; the diagonal by the 2 x 2
// Schur shift), and from them the next rotations, so that this chain is not in
// series with theirs.  Returns the number of rotations: it decides whether the
// sweep rotated anything (the workers' first look at a pair may differ from the
// look here by a rounding).
__device__ unsigned form_rotations(const Smem &sm, bool own, const float4 &lim) {
  const int lane = threadIdx.x & 31, k = lane & 15;
  csync();
  unsigned left = *sm.rounds;
  if (!left) return 0;
  unsigned n_rot = 0;
  const Cross *X = (const Cross *)sm.S;
  const Whole *A = (const Whole *)sm.S;
  int r = own ? 0 : __ffs(left) - 1, d = r;
  left &= left - 1;
  state_sync(0);
  float al = sm.diag[k], be = sm.diag[16 + ((k + r) & 15)];
  float2 g = sm.piv[k];
  Rot2 t;
  float shift;
  auto form = [&](int c) {
    const float g2 = fmaf(g.x, g.x, g.y * g.y);
    const bool go = rotates(al, be, g2, lim);
    t = make_rot2(al, be, g, g2, shift);
    if (!go) t.m = t.sr = t.si = shift = 0.f;
    if (lane < 16) sm.par[16 * c + lane] = make_float4(t.m, t.sr, t.si, 0.f);
    formed_arrive(c);
    n_rot += __popc(__ballot_sync(0xffffffffu, go) & 0xffffu);
  };
  form(0);
  if (own) {
    // pair k of the next round: x and y of this one (slots 0-15: a, 16-31: b)
    const int x = from_a(k), y = from_b(k), ix = x & 15, ky = y & 15;
    const bool xb = x > 15, yb = y > 15;
    const int rt = 32 * from_a(ix), ru = 32 * from_b(ix), ct = from_a(ky), cu = from_b(ky);
    for (r = 0; r < 31; ++r) {
      const float my = __shfl_sync(0xffffffffu, t.m, ky), sry = __shfl_sync(0xffffffffu, t.sr, ky),
                  siy = __shfl_sync(0xffffffffu, t.si, ky);
      const float mx = __shfl_sync(0xffffffffu, t.m, ix), srx = __shfl_sync(0xffffffffu, t.sr, ix),
                  six = __shfl_sync(0xffffffffu, t.si, ix);
      const float a1 = al - shift, b1 = be + shift;
      const float ax = __shfl_sync(0xffffffffu, a1, ix), bx = __shfl_sync(0xffffffffu, b1, ix);
      const float ay = __shfl_sync(0xffffffffu, a1, ky), by = __shfl_sync(0xffffffffu, b1, ky);
      al = xb ? bx : ax;
      be = yb ? by : ay;
      if (r > 0) state_sync(r & 1);
      if (r == 30) break;
      const float2 *G = A->G;
      const float2 tt = G[rt + ct], tu = G[rt + cu], ut = G[ru + ct], uu = G[ru + cu];
      state_read_arrive();
      // column y: a' = a + m a - sigma b, b' = b + m b + conj(sigma) a
      const float cr = yb ? sry : -sry;
      const float2 vt = rot_one(yb ? tu : tt, yb ? tt : tu, my, cr, -siy);
      const float2 vu = rot_one(yb ? uu : ut, yb ? ut : uu, my, cr, -siy);
      // row x: a' = a + m a - conj(sigma) b, b' = b + m b + sigma a
      g = rot_one(xb ? vu : vt, xb ? vt : vu, mx, xb ? srx : -srx, six);
      form((r + 1) & 1);
    }
  } else {
    int d2 = after(left, r);
    bool first = true;  // the first state has been waited for
    for (int c = 0;; c ^= 1) {
      // what does not wait for the workers comes before the barrier
      const int k2 = (k + d2) & 15, row = ((k + d) & 15) * 16;
      const float2 *pa = X->BA[c] + row + k2, *pb = X->BB[c] + row + ((k2 + d) & 15);
      const float m1 = __shfl_sync(0xffffffffu, t.m, k2), sr1 = __shfl_sync(0xffffffffu, t.sr, k2),
                  si1 = __shfl_sync(0xffffffffu, t.si, k2);
      al -= shift;
      be = __shfl_sync(0xffffffffu, be + shift, k2);
      if (!first) state_sync(c);
      first = false;
      if (!left) break;
      const float2 aa = X->AX[c][k], ab = X->AB[c][k], ba = *pa, bb = *pb;
      const float2 va = rot_one(ab, aa, m1, sr1, -si1), vb = rot_one(bb, ba, m1, sr1, -si1);
      g = rot_one(va, vb, t.m, -t.sr, t.si);
      form(c ^ 1);
      d = d2;
      r += d;
      left &= left - 1;
      d2 = after(left, r);
    }
  }
  return n_rot;
}

// Step 3 for the operands in sm.A (`rows` rows): every 128-row tile's product
// with Q - I is added to it and handed, eight columns at a time, to
// put(panel, Re (0) or Im (1), its group 0..1, row, values).
template <bool kWide, class Put>
__device__ bool update(const Smem &sm, int rows, Waits &wt, Put put) {
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, pan = warp >> 2;
  const int tiles = (rows + 127) / 128;
  const uint32_t grp = (uint32_t)rows * 16;
  for (int t0 = 0; t0 < tiles; t0 += 2) {
    const int n = tiles - t0 < 2 ? 1 : 2;
    if (tid == 0) {
      tc_fence_after();
      for (int i = 0; i < n; ++i)
        issue_update<kWide>(sm.tmem + 64 * i, smem_u32(sm.A) + (t0 + i) * 2048, rows,
                            smem_u32(sm.S), sm.bar[i]);
    }
    wt.out |= (1u << n) - 1u;
    for (int i = 0; i < n; ++i) {
      if (!wt.mma(sm, i, true)) return false;
      const int row = 128 * (t0 + i) + 32 * (warp & 3) + lane;
      const uint32_t at = sm.tmem + 64 * i + ((uint32_t)(32 * (warp & 3)) << 16) + 16 * pan;
      const char *src = sm.A + 8 * pan * grp + row * 16;
#pragma unroll
      for (int part = 0; part < 2; ++part) {
        uint32_t acc[16];
        tc_ld16(at + 32 * part, acc);
        tc_wait_ld();
        if (row < rows) {
#pragma unroll
          for (int g = 0; g < 2; ++g) {
            const char *p = src + (4 * part + g) * grp;
            float x[8];
#pragma unroll
            for (int j = 0; j < 8; ++j) x[j] = __uint_as_float(acc[8 * g + j]) * (1.0f / kScaleQ);
            join8(*(const uint4 *)p, *(const uint4 *)(p + 2 * grp), x);
            put(pan, part, g, row, x);
          }
        }
      }
    }
    tc_fence_before();
    wsync();
  }
  return true;
}

// two panels' operands (bytes each) into sm.A; arrives at `bar` (one thread)
__device__ __forceinline__ void load_pair(const Smem &sm, const char *a, const char *b,
                                          uint32_t bytes, uint32_t bar) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar),
               "r"(2 * bytes)
               : "memory");
  const uint32_t dst = smem_u32(sm.A);
  asm volatile(
      "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::
          "r"(dst),
      "l"(a), "r"(bytes), "r"(bar)
      : "memory");
  asm volatile(
      "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::
          "r"(dst + bytes),
      "l"(b), "r"(bytes), "r"(bar)
      : "memory");
}
__device__ __forceinline__ void fence_async() {
  asm volatile("fence.proxy.async;" ::: "memory");
}
__device__ __forceinline__ void mbar_arrive(uint32_t bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}

// A slice's start by the whole CTA: the columns' squared norms (key) and
// ||W||_F^2.  Returns 0 when sweeps are to run, 1 when every singular value is
// cut (||W||_F <= skip_t: the SVT is zero whatever the sweeps would find), 2
// when there is no pair, the Gram check showed that a sweep would rotate
// nothing, or ||W||_F^2 is not finite (no column then counts as negligible or
// not, and nothing can be rotated).
__device__ int slice_start(const Slice &x, float *key, float *s_red, float &fro2) {
  fro2 = norms_and_sum(x.nr, x.nc, x.W, key, s_red);
  if (x.skip_t >= 0.0f && fro2 <= x.skip_t * x.skip_t) return 1;
  return x.pre || x.nc < 2 || !(fro2 <= FLT_MAX) ? 2 : 0;
}
// a slice that runs no sweep: V := I unless warm, and the epilogue
__device__ void slice_skip(const Slice &x) {
  if (!x.warm)
    for (int e = threadIdx.x; e < x.nc * x.nc; e += blockDim.x)
      x.V[e] = make_float2((e % x.nc) == (e / x.nc) ? 1.0f : 0.0f, 0.0f);
  __syncthreads();
  pk_epilogue<true>(x.nr, x.nc, x.W, x.V, x.t);
}
__device__ void slice_order(const Run &a, const Slice &x, float *key, int *perm) {
  if (a.o.sort) {
    order_columns(x.nc, key, perm);
  } else {
    for (int c = threadIdx.x; c < x.nc; c += blockDim.x) perm[c] = c;
  }
}

// Set-up launch of the task schedule, one CTA a slice: the order, the limits,
// the operands, and the slice's first round in the queue.
__global__ void __launch_bounds__(1024) k_blk_setup(Run a) {
  __shared__ float s_red[32];
  __shared__ float s_key[kMaxSpatial];
  __shared__ int s_perm[kMaxSpatial + 2 * kB];
  const int s = blockIdx.x;
  Sched q(a.sched, a.nslices, a.cap, a.cols);
  const Slice x = slice_of(a, s);
  float fro2;
  const int done = slice_start(x, s_key, s_red, fro2);
  if (done) {
    slice_skip(x);
    if (threadIdx.x == 0) {
      *x.sweeps = done == 1 ? 0 : 1;
      __threadfence();
      atomicAdd(q.finished, 1);
    }
    return;
  }
  for (int c = threadIdx.x; c < kMaxSpatial + 2 * kB; c += blockDim.x) s_perm[c] = -1;
  __syncthreads();
  slice_order(a, x, s_key, s_perm);
  __syncthreads();
  int *perm = q.perm + (size_t)a.cols * s;
  for (int c = threadIdx.x; c < x.nc; c += blockDim.x) perm[c] = s_perm[c];
  const float4 lim = limits(x, fro2);
  const int np = players_of(panels_of(x.nc)), rw = rows16(x.nr), rv = rows16(x.nc);
  char *ov = x.op + (size_t)np * rw * 128;
  pack_panels(x.op, x.W, x.nr, rw, np, s_perm, 1.0f / lim.w, threadIdx.x, blockDim.x);
  pack_panels(ov, x.warm ? x.V : nullptr, x.nc, rv, np, s_perm, kScaleV, threadIdx.x, blockDim.x);
  __threadfence();
  __syncthreads();
  if (threadIdx.x == 0) {
    q.lim[s] = lim;
    q.packed[s] = 1;
    *x.sweeps = -a.max_sweeps;  // until the slice ends: a run that stops early reports it
    if (atomicAdd(q.live, 1) < a.live_max) {
      int task[kMaxTasks];
      q.push(task, q.begin_sweep(s, panels_of(x.nc), task));
    } else {
      q.pend[atomicAdd(q.npend, 1)] = s;
    }
  }
}

// Closing launch of the task schedule: a slice's operands back to W and V, and
// g_i = max(1 - t / sigma_i, 0) applied to V (t >= 0), summed in the order of the
// other kernels' epilogues.  A slice whose first sweep rotated nothing keeps the W
// and V it came with, not their 22-bit halves: as if the sweep had not run.  One
// CTA a panel, a warp a column.
__global__ void __launch_bounds__(32 * kB) k_blk_close(Run a) {
  __shared__ float s_g[kB];
  __shared__ int s_col[kB];
  const int s = blockIdx.x, p = blockIdx.y;
  Sched q(a.sched, a.nslices, a.cap, a.cols);
  if (!q.packed[s]) return;
  const Slice x = slice_of(a, s);
  const int npan = panels_of(x.nc);
  const bool still = *x.sweeps == 1;
  if (p >= npan || (still && x.warm && x.t < 0.0f)) return;
  if (threadIdx.x < kB) {
    const int at = p * kB + threadIdx.x;
    s_col[threadIdx.x] = at < x.nc ? q.perm[(size_t)a.cols * s + at] : -1;
    s_g[threadIdx.x] = 1.0f;
  }
  __syncthreads();
  const int np = players_of(npan), rw = rows16(x.nr), rv = rows16(x.nc);
  auto unpack = [&](const char *src, int rows, int n, float2 *M, float inv, bool isv) {
    for (int u = threadIdx.x; u < 2 * n; u += 32 * kB) {
      const int g = u >= n, r = u - g * n;
      const char *b = src + ((size_t)g * rows + r) * 16;
      const size_t st = (size_t)rows * 32;
      float re[8] = {}, im[8] = {};
      join8(*(const uint4 *)b, *(const uint4 *)(b + st), re);
      join8(*(const uint4 *)(b + 2 * st), *(const uint4 *)(b + 3 * st), im);
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        const int c = s_col[8 * g + j];
        float2 v = make_float2(re[j] * inv, im[j] * inv);
        if (isv) {
          v.x *= s_g[8 * g + j];
          v.y *= s_g[8 * g + j];
        }
        if (c >= 0) M[(size_t)n * c + r] = v;
      }
    }
  };
  if (!still) unpack(x.op + (size_t)p * rw * 128, rw, x.nr, x.W, q.lim[s].w, false);
  if (x.t >= 0.0f) {
    __syncthreads();
    const int j = threadIdx.x >> 5;
    if (s_col[j] >= 0) {
      const float n2 = column_norm2<false>(x.nr, x.W + (size_t)x.nr * s_col[j]);
      if ((threadIdx.x & 31) == 0) s_g[j] = n2;
    }
    __syncthreads();
    // FP64 by sixteen threads: with every lane of the warps the kernel took 16.4 us at
    // 75 x 91 x 220, so 10.8
    if (threadIdx.x < kB && s_col[threadIdx.x] >= 0) s_g[threadIdx.x] = gain(s_g[threadIdx.x], x.t);
    __syncthreads();
  }
  if (!still) {
    unpack(x.op + ((size_t)np * rw + (size_t)p * rv) * 128, rv, x.nc, x.V, 1.0f / kScaleV, true);
    return;
  }
  for (int e = threadIdx.x; e < kB * x.nc; e += 32 * kB) {
    const int j = e / x.nc, r = e - j * x.nc, c = s_col[j];
    if (c < 0) continue;
    float2 *v = x.V + (size_t)x.nc * c + r;
    const float2 u = x.warm ? *v : make_float2(c == r ? 1.0f : 0.0f, 0.0f);
    *v = make_float2(u.x * s_g[j], u.y * s_g[j]);
  }
}

// TMEM and barriers of a CTA (every thread); `tasks`: those of the task schedule too
__device__ __forceinline__ void cta_begin(Smem &sm, uint64_t *bars, uint32_t *slot) {
  for (int j = 0; j < 2; ++j) sm.bar[j] = smem_u32(bars + j);
  sm.bar_w = smem_u32(bars + 2);
  sm.bar_v = smem_u32(bars + 3);
  sm.bar_task = smem_u32(bars + 4);
  sm.bar_done = smem_u32(bars + 5);
  sm.bar_vdone = smem_u32(bars + 6);
  if (threadIdx.x == 0) {
    for (int j = 0; j < 5; ++j) mbar_init1(smem_u32(bars + j));
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 8;" ::"r"(sm.bar_done) : "memory");
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 8;" ::"r"(sm.bar_vdone) : "memory");
    asm volatile("fence.mbarrier_init.release.cluster;");
  }
  if (threadIdx.x < 32) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], 128;" ::"r"(
        smem_u32(slot)));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  sm.tmem = *slot;
}
__device__ __forceinline__ void cta_end(const Smem &sm, const Waits &wt) {
  // MMAs whose wait ran out get a last bounded chance to land
  for (int j = 0; j < 2; ++j)
    if (threadIdx.x < 32 && ((wt.out >> j) & 1u)) mbar_wait(sm.bar[j], (wt.ph >> j) & 1u);
  tc_fence_before();
  __syncthreads();
  if (threadIdx.x < 32)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, 128;" ::"r"(sm.tmem));
}

struct TaskInfo {
  char *wa, *wb, *va, *vb;  // the panels' operands
  int rw, rv;               // their rows; rw < 0: no task, the run is over
  int own;
  float4 lim;
};

// The task schedule: a persistent grid whose CTAs take tasks of any slice until
// every slice has ended (or a wait runs out; slices still open then stay
// reported as capped).
template <bool kWide>
__global__ void __launch_bounds__(kT, 3) k_jacobi_tasks(Run a) {
  extern __shared__ __align__(128) char smem[];
  __shared__ __align__(8) uint64_t s_bar[7];
  __shared__ float4 s_par[32];
  __shared__ float2 s_piv[16];
  __shared__ float s_diag[32];
  __shared__ unsigned s_rounds;
  __shared__ uint32_t s_tmem;
  __shared__ TaskInfo s_info;
  __shared__ volatile int s_rot, s_vrot;  // the task rotated (-1: failed), after W and after V
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  Smem sm;
  sm.A = smem;
  sm.S = smem + (size_t)a.rows * 256;
  sm.par = s_par;
  sm.piv = s_piv;
  sm.diag = s_diag;
  sm.rounds = &s_rounds;
  cta_begin(sm, s_bar, &s_tmem);
  Waits wt;

  if (warp < kW / 32) {
    unsigned v_ph = 0;
    for (unsigned k = 0;; ++k) {
      if (!wsync_and(warp != 0 || mbar_wait(sm.bar_task, k & 1u, kWorkerWait))) break;
      const TaskInfo ti = s_info;
      if (ti.rw < 0) break;
      int rot = gram_rotate<kWide>(sm, ti.rw, ti.own, ti.lim, wt,
                            warp != 0 || mbar_wait(sm.bar_w, k & 1u));
      if (rot > 0) {
        auto put_to = [&](char *pa, char *pb, int rows) {
          return [=](int pan, int part, int g, int row, const float (&x)[8]) {
            uint4 hi, lo;
            split8(x, hi, lo);
            char *d = (pan ? pb : pa) + ((4 * part + g) * rows + row) * 16;
            __stcg((uint4 *)d, hi);
            __stcg((uint4 *)(d + rows * 32), lo);
          };
        };
        if (!update<kWide>(sm, ti.rw, wt, put_to(ti.wa, ti.wb, ti.rw))) rot = -1;
        fence_async();  // the columns' next readers are bulk copies
        // every thread has read W's operands: the ninth warp lets V's take their place
        if (tid == 0) s_rot = rot;
        __syncwarp();
        if (lane == 0) mbar_arrive(sm.bar_done);
        if (rot > 0) {
          const bool here = wsync_and(warp != 0 || mbar_wait(sm.bar_v, v_ph, kWorkerWait));
          v_ph ^= 1u;
          if (!here || !update<kWide>(sm, ti.rv, wt, put_to(ti.va, ti.vb, ti.rv))) rot = -1;
          fence_async();
        }
      } else {
        if (tid == 0) s_rot = rot;
        __syncwarp();
        if (lane == 0) mbar_arrive(sm.bar_done);
      }
      if (tid == 0) s_vrot = rot;
      __syncwarp();
      if (lane == 0) mbar_arrive(sm.bar_vdone);
    }
  } else {
    Sched q(a.sched, a.nslices, a.cap, a.cols);
    unsigned n_pairs = 0, n_rot = 0, done_ph = 0;
    int claim = -1, task = -1;  // lane 0: a queue slot taken, the next task
    auto panels = [&](int s) { return panels_of(a.list ? a.list[s].nc : a.nc); };
    // lane 0: counts a task whose W is done off; those that became ready go to
    // the queue
    auto finish = [&](int done, bool rot) {
      const int s = done / (kMaxTasks * kMaxRounds), r = (done / kMaxTasks) % kMaxRounds;
      const int npan = panels(s), np = players_of(npan);
      int ready[kMaxTasks + 2], n = 0, pan[2];
      round_pair(npan, r, done % kMaxTasks, pan[0], pan[1]);
      __threadfence();
      const int was = atomicAdd(q.left + s, (rot ? 0x10000 : 0) - 1);
      int next[2] = {-1, -1}, old[2];
      for (int j = 0; j < 2; ++j) {
        if (pan[j] >= npan) continue;
        for (int r1 = r + 1; r1 < np - 1; ++r1) {
          int p, p2;
          const int i = pair_index(np, r1, pan[j]);
          if (!round_pair(npan, r1, i, p, p2)) continue;  // it has no partner there
          next[j] = Sched::task_of(s, r1, i);
          old[j] = atomicAdd(q.arrive + (size_t)q.per * s + r1 * (np / 2) + i, 1);
          break;
        }
      }
      for (int j = 0; j < 2; ++j)
        if (next[j] >= 0 && (old[j] & 1)) ready[n++] = next[j];
      if ((was & 0xffff) == 1) {  // the sweep is complete
        __threadfence();
        const int sw = *(volatile int *)(q.sweep + s) + 1;
        int end = 0;
        if (!(was >> 16) && !rot) end = sw;  // converged: a sweep without a rotation
        else if (sw >= a.max_sweeps) end = -a.max_sweeps;
        if (!end) {
          *(volatile int *)(q.sweep + s) = sw;
          n = q.begin_sweep(s, npan, ready);
        } else {
          *(a.list ? a.list[s].sweeps : a.sweeps + s) = end;
          const int w = atomicAdd(q.pend_head, 1);  // a waiting slice may start
          if (w < *(volatile int *)q.npend) {
            const int s1 = q.pend[w];
            n = q.begin_sweep(s1, panels(s1), ready);
          }
        }
        q.push(ready, n);
        if (end) {
          __threadfence();
          atomicAdd(q.finished, 1);
        }
      } else {
        q.push(ready, n);
      }
    };
    auto test = [&](uint32_t bar, unsigned parity) {
      uint32_t done;
      asm volatile(
          "{\n .reg .pred p;\n mbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\n"
          " selp.u32 %0, 1, 0, p;\n}\n"
          : "=r"(done)
          : "r"(bar), "r"(parity)
          : "memory");
      return done != 0;
    };
    // lane 0: looks once at the queue; a task, or -1
    auto look = [&]() -> int {
      if (claim < 0) claim = atomicAdd(q.head, 1);
      const unsigned long long v =
          *(volatile unsigned long long *)(q.slot + (claim & (q.cap - 1)));
      if ((unsigned)(v >> 32) != (unsigned)(claim + 1)) return -1;
      __threadfence();
      claim = -1;
      return (int)(unsigned)v;
    };
    for (;;) {
      int s = 0, r = 0, pa = 0, pb = 0, npan = 1, nr = 1, nc = 1, sw = 0;
      if (lane == 0) {
        // the next task, unless it was found while the last one's V was updated
        const unsigned long long t0 = gtimer();
        while (task < 0) {
          if ((task = look()) >= 0) break;
          if (*(volatile int *)q.finished >= a.nslices) break;
          if (gtimer() - t0 > kTaskWaitNs) {
            atomicExch(q.err, 1);
            break;
          }
          __nanosleep(32);
        }
        if (task < 0) {
          s_info.rw = -1;
        } else {
          s = task / (kMaxTasks * kMaxRounds);
          r = (task / kMaxTasks) % kMaxRounds;
          nr = a.list ? a.list[s].nr : a.nr;
          nc = a.list ? a.list[s].nc : a.nc;
          char *op = a.list ? a.list[s].op : a.op + (size_t)s * op_bytes(nr, nc);
          npan = panels_of(nc);
          const int rw = rows16(nr), rv = rows16(nc);
          round_pair(npan, r, task % kMaxTasks, pa, pb);
          char *ov = op + (size_t)players_of(npan) * rw * 128;
          s_info.wa = op + (size_t)pa * rw * 128;
          s_info.wb = op + (size_t)pb * rw * 128;
          fence_async();
          load_pair(sm, s_info.wa, s_info.wb, (uint32_t)rw * 128, sm.bar_w);
          s_info.va = ov + (size_t)pa * rv * 128;
          s_info.vb = ov + (size_t)pb * rv * 128;
          s_info.rw = rw;
          s_info.rv = rv;
          s_info.own = r == 0;
          s_info.lim = q.lim[s];
          sw = *(volatile int *)(q.sweep + s);
          const int wa = min(kB, nc - pa * kB), wb = max(0, min(kB, nc - pb * kB));
          n_pairs += wa * wb + (r == 0 ? (wa * (wa - 1) + wb * (wb - 1)) / 2 : 0);
        }
        mbar_arrive(sm.bar_task);
      }
      __syncwarp();
      if (s_info.rw < 0) break;
      const unsigned made = form_rotations(sm, s_info.own, s_info.lim);
      n_rot += made;
      int go = 1;
      if (lane == 0) {
        // the panels' V as their tasks before left it
        volatile int *va = q.vdone + (size_t)q.pan * s + pa, *vb = q.vdone + (size_t)q.pan * s + pb;
        const int na = Sched::stamp_before(npan, sw, r, pa);
        const int nb = pb < npan ? Sched::stamp_before(npan, sw, r, pb) : 0;
        const unsigned long long t0 = gtimer();
        bool ok = true;
        for (;;) {
          const int x = *va, y = *vb;
          if (x >= na && y >= nb) break;
          if (gtimer() - t0 > kTaskWaitNs) {
            ok = false;
            break;
          }
        }
        // the workers' waits are bounded, so these end
        ok = mbar_wait(sm.bar_done, done_ph, kWorkerWait) && ok && s_rot >= 0;
        const int done = task;
        task = -1;
        if (ok) {
          const int rot = s_rot;
          __threadfence();
          if (rot) {
            fence_async();
            load_pair(sm, s_info.va, s_info.vb, (uint32_t)s_info.rv * 128, sm.bar_v);
          }
          finish(done, made != 0);
          for (long long n = 0; !test(sm.bar_vdone, done_ph); ++n) {
            if (task < 0)
              task = look();
            else
              __nanosleep(64);
            if (n > kWorkerWait) {
              ok = false;
              break;
            }
          }
          ok = ok && s_vrot >= 0;
        }
        if (ok) {
          const int stamp = sw * (players_of(npan) - 1) + r + 1;
          __threadfence();
          *va = stamp;
          *vb = stamp;
        } else {
          atomicExch(q.err, 1);
          go = 0;
          s_info.rw = -1;
          mbar_arrive(sm.bar_task);
        }
      }
      done_ph ^= 1u;
      if (!__shfl_sync(0xffffffffu, go, 0)) break;
    }
    if (a.work && lane == 0) {
      atomicAdd(a.work + 0, (unsigned long long)n_pairs);
      atomicAdd(a.work + 1, (unsigned long long)n_rot);
    }
  }
  __syncwarp();
  cta_end(sm, wt);
}

// The per-slice schedule: CTA b runs the tasks of slice b one after another on
// W and V in place.  Gathering and splitting a task's columns every time makes it
// slower than the FP32 kernel where that holds a panel in registers (up to 256
// rows, see launch_jacobi).
__global__ void __launch_bounds__(kT, 2) k_jacobi_slices(Run a) {
  extern __shared__ __align__(128) char smem[];
  __shared__ __align__(8) uint64_t s_bar[7];
  __shared__ float4 s_par[32];
  __shared__ float2 s_piv[16];
  __shared__ float s_diag[32];
  __shared__ unsigned s_rounds;
  __shared__ uint32_t s_tmem;
  __shared__ float s_red[32];
  __shared__ int s_cols[2 * kB];
  __shared__ int s_any, s_made;
  const int tid = threadIdx.x, s = blockIdx.x;
  Smem sm;
  sm.A = smem;
  sm.S = smem + (size_t)a.rows * 256;
  sm.par = s_par;
  sm.diag = s_diag;
  sm.rounds = &s_rounds;
  sm.piv = s_piv;
  int *perm = (int *)(sm.S + kScratch<false>);
  cta_begin(sm, s_bar, &s_tmem);
  Waits wt;
  unsigned n_pairs = 0, n_rot = 0;
  const Slice x = slice_of(a, s);
  float *key = (float *)sm.S;
  float fro2;
  const int done = slice_start(x, key, s_red, fro2);
  if (done) {
    slice_skip(x);
    if (tid == 0) *x.sweeps = done == 1 ? 0 : 1;
  } else {
    if (!x.warm)
      for (int e = tid; e < x.nc * x.nc; e += kT)
        x.V[e] = make_float2((e % x.nc) == (e / x.nc) ? 1.0f : 0.0f, 0.0f);
    slice_order(a, x, key, perm);
    __syncthreads();
    const float4 lim = limits(x, fro2);
    const int npan = panels_of(x.nc), rw = rows16(x.nr), rv = rows16(x.nc);
    const bool worker = tid < kW;
    auto load = [&](const float2 *M, int n, int rows, float scale) {
      pack_panels(sm.A, M, n, rows, 2, s_cols, scale, tid, kW);
      tc_fence_smem();
      tc_fence_before();
      wsync();
    };
    // both parts of a value meet here: Re is written first, then Im
    auto put_to = [&](float2 *M, int n, float inv) {
      return [=](int pan, int part, int g, int row, const float (&v)[8]) {
        uint4 hi, lo;
        float f[8] = {};
        split8(v, hi, lo);
        join8(hi, lo, f);
        if (row >= n) return;
#pragma unroll
        for (int j = 0; j < 8; ++j) {
          const int c = s_cols[kB * pan + 8 * g + j];
          if (c >= 0) ((float *)(M + (size_t)n * c + row))[part] = f[j] * inv;
        }
      };
    };
    int result = -a.max_sweeps, any = 1;
    for (int sweep = 1; sweep <= a.max_sweeps && any > 0; ++sweep) {
      any = 0;
      for (int r = 0; r < rounds_of(npan) && any >= 0; ++r)
        for (int i = 0; i < kMaxTasks; ++i) {
          int pa, pb;
          if (!round_pair(npan, r, i, pa, pb)) continue;
          if (tid < 2 * kB) {
            const int at = (tid < kB ? pa : pb) * kB + (tid & (kB - 1));
            s_cols[tid] = at < x.nc ? perm[at] : -1;
          }
          __syncthreads();
          const int wa = min(kB, x.nc - pa * kB), wb = max(0, min(kB, x.nc - pb * kB));
          n_pairs += wa * wb + (r == 0 ? (wa * (wa - 1) + wb * (wb - 1)) / 2 : 0);
          if (worker) {
            load(x.W, x.nr, rw, 1.0f / lim.w);
            int rot = gram_rotate<false>(sm, rw, r == 0, lim, wt, true);
            if (rot > 0) {
              bool ok = update<false>(sm, rw, wt, put_to(x.W, x.nr, lim.w));
              if (ok) {
                load(x.V, x.nc, rv, kScaleV);
                ok = update<false>(sm, rv, wt, put_to(x.V, x.nc, 1.0f / kScaleV));
              }
              if (!ok) rot = -1;
            }
            if (tid == 0) s_any = rot;
          } else {
            const unsigned made = form_rotations(sm, r == 0, lim);
            n_rot += made;
            if (tid == kW) s_made = made != 0;
          }
          __syncthreads();
          const int rot = s_any;
          if (rot < 0) {
            any = -1;
            break;
          }
          any |= s_made;
        }
      if (any == 0) result = sweep;
    }
    pk_epilogue<true>(x.nr, x.nc, x.W, x.V, x.t);
    if (tid == 0) *x.sweeps = result;
  }
  if (a.work && tid == kW) {
    atomicAdd(a.work + 0, (unsigned long long)n_pairs);
    atomicAdd(a.work + 1, (unsigned long long)n_rot);
  }
  cta_end(sm, wt);
}

cudaError_t blk_launch(Run a, cudaStream_t st) {
  int dev = 0, nsm = 0, sm_smem = 0, cta_smem = 0;
  cudaError_t e;
  if ((e = cudaGetDevice(&dev)) != cudaSuccess) return e;
  if ((e = cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess ||
      (e = cudaDeviceGetAttribute(&sm_smem, cudaDevAttrMaxSharedMemoryPerMultiprocessor, dev)) !=
          cudaSuccess ||
      (e = cudaDeviceGetAttribute(&cta_smem, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev)) !=
          cudaSuccess)
    return e;
  const size_t ops = (size_t)a.rows * 256;
  // resident CTAs of an SM, by shared memory (1 KB a CTA is the system's),
  // registers (three by the launch bounds) and TMEM (128 of 512 columns a CTA);
  // cudaOccupancyMaxActiveBlocksPerMultiprocessor says 1 of this kernel.  The
  // dynamic limit is the same for every size: threads may launch at once.
  auto prepare = [&](const void *f, size_t smem, int &per_sm) -> cudaError_t {
    cudaFuncAttributes at;
    cudaError_t r = cudaFuncGetAttributes(&at, f);
    if (r != cudaSuccess) return r;
    const int fit = (int)((size_t)sm_smem / (smem + at.sharedSizeBytes + 1024));
    per_sm = fit < 1 ? 1 : (fit > 3 ? 3 : fit);
    return cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                cta_smem - (int)at.sharedSizeBytes);
  };
  int per_sm = 0, per_sm_wide = 0;
  if (!a.sched) {
    const size_t smem = ops + kScratch<false> + sizeof(int) * (size_t)a.cols;
    if ((e = prepare((const void *)k_jacobi_slices, smem, per_sm)) != cudaSuccess) return e;
    k_jacobi_slices<<<a.nslices, kT, smem, st>>>(a);
    return cudaGetLastError();
  }
  a.cap = queue_cap(a.nslices);
  a.op = (char *)(a.sched + Sched::ints(a.nslices, a.cap, a.cols));
  if ((e = prepare((const void *)k_jacobi_tasks<false>, ops + kScratch<false>, per_sm)) !=
          cudaSuccess ||
      (e = prepare((const void *)k_jacobi_tasks<true>, ops + kScratch<true>, per_sm_wide)) !=
          cudaSuccess)
    return e;
  // workers: the resident CTAs, and no more than twice the tasks a round offers
  // (a CTA that updates V leaves the next round's W to another)
  const int width = players_of(panels_of(a.cols)) / 2;
  long long grid = (long long)per_sm * nsm;
  if (grid > 2ll * a.nslices * width) grid = 2ll * a.nslices * width;
  // slices in flight: their operands within about 96 MB of the 129 MB L2, and
  // enough of them to give every worker two tasks (1.5 tasks: 200 x 200 x 80, 50
  // iterations, 115 -> 134 ms; three, four or all slices: within 1%)
  const long long bytes = (long long)op_bytes(a.nr, a.nc);
  long long live = (96ll << 20) / bytes;
  const long long least = (2 * grid + width - 1) / width;
  if (live < least) live = least;
  a.live_max = live > a.nslices ? a.nslices : (int)live;
  e = cudaMemsetAsync(a.sched, 0, sizeof(int) * Sched::zeroed(a.nslices, a.cap, a.cols), st);
  if (e != cudaSuccess) return e;
  k_blk_setup<<<a.nslices, 1024, 0, st>>>(a);
  if ((e = cudaGetLastError()) != cudaSuccess) return e;
  if (per_sm_wide == per_sm)
    k_jacobi_tasks<true><<<(unsigned)grid, kT, ops + kScratch<true>, st>>>(a);
  else
    k_jacobi_tasks<false><<<(unsigned)grid, kT, ops + kScratch<false>, st>>>(a);
  if ((e = cudaGetLastError()) != cudaSuccess) return e;
  k_blk_close<<<dim3(a.nslices, panels_of(a.cols)), 32 * kB, 0, st>>>(a);
  return cudaGetLastError();
}

}  // namespace

size_t jacobi_op_bytes(int nr, int nc) { return op_bytes(nr, nc); }

size_t jacobi_task_ints(int nslices, int nc, size_t op_total) {
  return Sched::ints(nslices, queue_cap(nslices), nc) + op_total / sizeof(int);
}

cudaError_t launch_jacobi_blk(const Dims &d, int nslices, float2 *W, float2 *V, float t,
                              int max_sweeps, int *sweeps, unsigned long long *work,
                              cudaStream_t st, const JacOpt &o) {
  if (nslices <= 0) return cudaSuccess;
  Run a{};
  a.nslices = nslices;
  a.nr = d.nr;
  a.nc = d.nc;
  a.ws = d.P;
  a.vs = (size_t)d.nc * d.nc;
  a.W = W;
  a.V = V;
  a.t = t;
  a.tol0 = jacobi_tol0(d.nr);
  const float eps = FLT_EPSILON * 0.5f;
  a.negl_rel = ((float)d.nr * eps) * ((float)d.nr * eps);
  a.max_sweeps = max_sweeps;
  a.sweeps = sweeps;
  a.work = work;
  a.o = o;
  a.sched = o.sched;
  a.cols = d.nc;
  a.rows = rows16(d.nr);
  return blk_launch(a, st);
}

cudaError_t launch_jacobi_list(const SliceTask *list, int nslices, int max_nr, int max_nc,
                               double mu, int max_sweeps, unsigned long long *work,
                               cudaStream_t st, int warm, int keep, int sort, int *sched) {
  if (nslices <= 0) return cudaSuccess;
  Run a{};
  a.nslices = nslices;
  a.nr = max_nr;
  a.nc = max_nc;
  a.list = list;
  a.mu = mu;
  a.keep = keep;
  a.max_sweeps = max_sweeps;
  a.work = work;
  a.o.warm = warm;
  a.o.sort = sort;
  a.sched = sched;
  a.cols = max_nc;
  a.rows = rows16(max_nr);
  return blk_launch(a, st);
}

}  // namespace lrstv

// tcgemm.cu -- batched complex GEMM on the 5th-generation tensor cores
// (tcgen05.mma, accumulators in tensor memory) for the dense contractions of
// the iteration: the spatial DFT passes of the Z-solve (eq. Z_solution) and
// the SVT reconstruction W (V diag g)^H of the E-update (eq. E_solution).
//
// Same contract as k_cgemm (dft.cu): C_b = A_b op(B_b), column-major complex,
// op(B) = B or B^H, optional spectral-division epilogue.
//
// Precision: FP32-accurate "3xTF32".  Each FP32 operand x is split into
// x_hi = tf32(x) and x_lo = x - x_hi, and a product is formed as
// hi*hi + hi*lo + lo*hi with FP32 accumulation (the lo*lo term is below FP32
// resolution), so the result carries about 2^-21 relative error per term
// instead of TF32's 2^-11.  The tensor core accumulates with truncation, so
// each K chunk (16 real terms) goes into a fresh TMEM tile that the threads
// drain into FP32 register accumulators: accumulation error then grows over
// 16 terms, not over the whole K.
//
// The tensor core's truncation is then that of the hi*hi sums at each of the six
// products.  prec = 2 forms a chunk's four small products first, so that only the
// two hi*hi are added to a full-size sum: for the single operators, whose error
// against FP64 this keeps below that of FP32 sums (Z-solve of 145 x 145 x 220:
// 4.4e-7 relative, 8.9e-7 with prec = 0, 1.12e-6 with FP32 FMAs; 857 -> 281 us).  The iterations keep prec =
// 0, whose rounding their runs' results have always had.
//
// Complex arithmetic as real GEMMs with K doubled: for a K chunk,
//   Re C += [Re A | Im A] . [Re B | -Im B]^T,   Im C += [Re A | Im A] . [Im B | Re B]^T.
//
// Mixed precision (prec = 1, "3xBF16"): the same split with bf16 halves,
// x_hi = bf16(x), x_lo = bf16(x - x_hi), and the three products on the BF16
// tensor-core path (kind::f16, both operands bf16, FP32 accumulation): about
// 2^-17 relative error per term, half the shared-memory bytes and half the
// MMA instructions of 3xTF32 (K = 16 per instruction instead of 8).
//
// Tile: 128 rows of C (M = 128 MMA), 64 complex columns (one N = 128 MMA over
// adjacent Re and Im B blocks into 128 TMEM columns, which reads the A tile
// once for both parts), 8 (3xTF32) or 16 (3xBF16) complex K per chunk: the
// chunk's real parts are one MMA's K, its imaginary parts the other's; 28 KB a
// stage.  Operands are staged by the CTA's threads into shared memory in the
// canonical K-major layout without swizzle: 8-row x 16-byte core matrices, the
// two of an MMA's K 128 B apart (LBO), 8-row groups 256 B apart (SBO).  B is
// held as the blocks -Im, Re, Im: [Re | Im] meets A's real parts, [-Im | Re] its
// imaginary ones.
//
// What bounds it: the instructions that stage the operands; the tensor core's
// part of a chunk is a third.  A thread therefore owns one row of A and a run of
// consecutive k, a whole 16-byte row of a core matrix (B: half of one): its
// bounds and addresses are worked out once, a chunk's loads walk along K, and a
// run goes to shared memory in one store.  With an element's position worked
// out at a time and 4-byte stores, 123 slices of 200 x 200 took 114 us instead
// of 105 (3xTF32; 288 of 256 x 256 with 3xBF16 249 instead of 200), and the
// forward DFT of three 200 x 200 x 80 cubes 71 instead of 41; sums in pairs and
// TF32 by integers made the 105 95.  More chunks under way (asynchronous copies
// into shared memory, read back) were slower: 110-123.
// Two stages and two TMEM tiles pipeline the chunks: chunk k is loaded and
// staged while chunk k - 1's MMAs run, and chunk k - 1's tile is drained while
// chunk k's MMAs run.
// One thread issues the MMAs and commits them to the stage's mbarrier; every
// wait on a barrier is bounded and, if it runs out, the CTA records an error
// flag, skips its epilogue and still frees its tensor memory.
#include <cuda_bf16.h>
#include <stdint.h>

#include "lrstv_internal.cuh"
#include "tc_ptx.cuh"

namespace lrstv {

namespace {

constexpr int TM = 128;       // rows of C per CTA
constexpr int TN = 64;        // complex columns of C per CTA
// eight warps: warp w reads TMEM lanes 32 (w mod 4) .. + 31 (rows of the tile)
// and, by warpgroup, columns 0..31 or 32..63 of each Re / Im tile
constexpr int kThreads = 256;
constexpr uint32_t kLBO = 128, kSBO = 256;  // bytes
// Per precision: element bytes, the K of one MMA (two core matrices, 32 bytes of a
// row), the elements of a core matrix's row and the instruction descriptor's operand
// format (kind::tf32: TF32 = 2; kind::f16: BF16 = 1).
template <int PREC>
struct Prec {
  static constexpr int kBytes = PREC == 1 ? 2 : 4;
  static constexpr int kTK = 32 / kBytes;   // complex K per chunk: 16 real terms per TMEM
  static constexpr int kKR = 2 * kTK;       // tile with 3xTF32
  static constexpr int kRun = 16 / kBytes;
  static constexpr uint32_t kFmt = PREC == 1 ? 1u : 2u;
};
constexpr uint32_t kHalfA = TM * 32;   // A's real (imaginary) parts of a chunk, one split
constexpr uint32_t kBlockB = TN * 32;  // a block of B, one split
// blocks of B (KIND 0: -Im, Re, Im; 1: Re and Im of each half's bands; 2: Re, -Im)
__host__ __device__ constexpr uint32_t blocks_b(int kind) {
  return kind == 0 ? 3 : (kind == 1 ? 4 : 2);
}
__host__ __device__ constexpr uint32_t stage_bytes(int kind) {
  return 4 * kHalfA + 2 * blocks_b(kind) * kBlockB;
}

__device__ __forceinline__ uint64_t sdesc(uint32_t addr) { return tc_desc(addr, kLBO, kSBO); }

// x to TF32, to nearest, ties away from zero: the value of cvt.rna.tf32.f32, which
// takes five instructions here (a NaN may become an infinity: x - hi is NaN then)
__device__ __forceinline__ float tf32_hi(float x) {
  return __uint_as_float((__float_as_uint(x) + 0x1000u) & 0xffffe000u);
}

// two FP32 sums in one instruction, each rounded as alone
__device__ __forceinline__ void add2(float &a0, float &a1, float b0, float b1) {
  asm("{\n .reg .b64 a, b;\n mov.b64 a, {%0, %1};\n mov.b64 b, {%2, %3};\n"
      " add.rn.f32x2 a, a, b;\n mov.b64 {%0, %1}, a;\n}\n"
      : "+f"(a0), "+f"(a1)
      : "f"(b0), "f"(b1));
}

// N consecutive k of a row, split into hi and lo words
template <int PREC, int N>
struct Run {
  static constexpr int kWords = PREC == 1 ? N / 2 : N;
  uint32_t hi[kWords], lo[kWords];
  __device__ __forceinline__ explicit Run(const float (&x)[N]) {
#pragma unroll
    for (int j = 0; j < kWords; ++j) {
      if constexpr (PREC != 1) {
        const float h = tf32_hi(x[j]);
        hi[j] = __float_as_uint(h);
        lo[j] = __float_as_uint(x[j] - h);
      } else {
        const __nv_bfloat162 h = __floats2bfloat162_rn(x[2 * j], x[2 * j + 1]);
        const float2 f = __bfloat1622float2(h);
        const __nv_bfloat162 l = __floats2bfloat162_rn(x[2 * j] - f.x, x[2 * j + 1] - f.y);
        hi[j] = *(const uint32_t *)&h;
        lo[j] = *(const uint32_t *)&l;
      }
    }
  }
  __device__ __forceinline__ void negate() {
    constexpr uint32_t sign = PREC == 1 ? 0x80008000u : 0x80000000u;
#pragma unroll
    for (int j = 0; j < kWords; ++j) {
      hi[j] ^= sign;
      lo[j] ^= sign;
    }
  }
  // a run is 16 (A) or 8 (B) bytes
  __device__ __forceinline__ void put(char *at_hi, char *at_lo) const {
    if constexpr (kWords == 4) {
      *(uint4 *)at_hi = make_uint4(hi[0], hi[1], hi[2], hi[3]);
      *(uint4 *)at_lo = make_uint4(lo[0], lo[1], lo[2], lo[3]);
    } else {
      *(uint2 *)at_hi = make_uint2(hi[0], hi[1]);
      *(uint2 *)at_lo = make_uint2(lo[0], lo[1]);
    }
  }
};

template <int PREC>
__device__ __forceinline__ void mma(uint32_t d, uint64_t a, uint64_t b, uint32_t idesc,
                                    uint32_t accumulate) {
  if (PREC != 1)
    asm volatile(
        "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
        " tcgen05.mma.cta_group::1.kind::tf32 [%0], %1, %2, %3, p;\n}\n" ::"r"(d),
        "l"(a), "l"(b), "r"(idesc), "r"(accumulate));
  else
    asm volatile(
        "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
        " tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(d),
        "l"(a), "l"(b), "r"(idesc), "r"(accumulate));
}

// KIND 0: the complex GEMM C = A op(B) of CGemm (OPB 0: B, 1: B^H), or, with
// OPB 2, C = A^H B (the Gram products W^H W).  KIND 1 and 2: the mode-3
// DFTs of the cubes of Dft3 as GEMMs over the pixels (M = n1 n2):
//  KIND 1 (real -> half spectrum): C(p, k) = sum_c x(p, c) exp(-2 pi i k c / n3),
//    k < h, a real A (x, or x - ycoef y) against the twiddles; a K chunk holds
//    KR real bands in the A tile, and the B tiles hold the real and the
//    imaginary twiddle parts of those bands, so that the MMAs form Re C and
//    Im C directly.  Written at the working orientation's pixel (conjugated
//    when transposed).
//  KIND 2 (half spectrum -> real): x(p, c) = (1/n3) sum_{k<h} w_k Re(X_k(p)
//    exp(2 pi i k c / n3)) with w_k = 1 at k = 0 and k = n3/2, else 2: the
//    complex GEMM's Re C alone, B(k, c) = w_k exp(2 pi i k c / n3); the
//    epilogue scales by 1/n3 and, in mode 1, updates Gamma4 += mu (x - F).
// The DFT kinds take their tile indices from blockIdx.x with the N tiles of
// one M tile adjacent in launch order, so the M tile's inputs come from DRAM
// once and from L2 for the other N tiles.
//
// Where A or B is one matrix for the whole batch (the spatial DFTs), the other
// side's slices are one tall (fold: row m is row m mod slice_m of slice
// m / slice_m) or, being contiguous, one wide matrix: tiles then cross slices, and
// only the last one is padded.
template <int OPB, int EPI, int PREC, int KIND = 0>
__global__ void __launch_bounds__(kThreads, 2) k_cgemm_tc(CGemm g, Dft3 f, int *err) {
  extern __shared__ __align__(1024) char smem[];
  using P = Prec<PREC>;
  // two shared-memory stages, so that a chunk is staged while the previous
  // chunk's MMAs run, and two TMEM tiles (one per stage)
  constexpr uint32_t kCols = 256;
  constexpr bool kTwo = KIND == 1 && PREC != 2;  // x - ycoef y; the operators' DFTs take one cube
  constexpr uint32_t kStageBytes = stage_bytes(KIND), kLoB = blocks_b(KIND) * kBlockB;
  __shared__ __align__(8) uint64_t mbar[2];
  __shared__ uint32_t tslot;

  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int b = blockIdx.z;
  if (KIND == 0 && g.gate && !g.gate[b]) return;  // a gated-off batch entry (CTA-uniform)
  int m0 = blockIdx.x * TM, n0 = blockIdx.y * TN;
  // the DFT kinds: problem size, this batch entry's cubes
  int gM = g.M, gN = g.N, gK = g.K;
  const float *xb = nullptr, *yb = nullptr;
  const float2 *specb = nullptr;
  if (KIND != 0 || g.fold) {
    const int nt = ((KIND == 0 ? g.N : (KIND == 1 ? f.h : f.n3)) + TN - 1) / TN;
    m0 = (blockIdx.x / nt) * TM;
    n0 = (blockIdx.x % nt) * TN;
  }
  if (KIND != 0) {
    gM = (int)f.P;
    gN = KIND == 1 ? f.h : f.n3;
    gK = KIND == 1 ? f.n3 : f.h;
    if (KIND == 1) {
      xb = f.x + (size_t)b * f.N;
      if (kTwo && f.y) yb = f.y + (size_t)b * f.N;
    } else {
      specb = f.spec + (size_t)b * f.h * f.P;
    }
  }
  // pixel p of the cube -> its index in the working orientation's slice
  auto wpos = [&](int p) -> size_t {
    if (!f.trans) return (size_t)p;
    const int i = p % f.n1, j = p / f.n1;
    return (size_t)j + (size_t)f.n2 * i;
  };

  if (tid == 0) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_u32(&mbar[0])));
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_u32(&mbar[1])));
    asm volatile("fence.mbarrier_init.release.cluster;");
  }
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                     smem_u32(&tslot)),
                 "n"(kCols));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
  }
  asm volatile("tcgen05.fence::before_thread_sync;");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;");
  const uint32_t tmem = tslot;
  // D format F32, A and B in the precision's format, both K-major, N, M
  const uint32_t idesc = (1u << 4) | (P::kFmt << 7) | (P::kFmt << 10) |
                         ((uint32_t)(TN >> 3) << 17) | ((uint32_t)(TM >> 4) << 24);
  const uint32_t idesc2 = (1u << 4) | (P::kFmt << 7) | (P::kFmt << 10) |
                          ((uint32_t)((2 * TN) >> 3) << 17) | ((uint32_t)(TM >> 4) << 24);
  const uint32_t bar0 = smem_u32(&mbar[0]), bar1 = smem_u32(&mbar[1]);
  // per stage: the parity of its next MMA commit, and whether a commit is
  // outstanding (issued, not yet seen complete)
  uint32_t ph0 = 0u, ph1 = 0u;
  bool out0 = false, out1 = false;
  bool ok = true;
  const int row = 32 * (warp & 3) + lane;  // TMEM lane = row of the tile this thread drains
  const int colh = (warp >> 2) * (TN / 2);  // first of the 32 columns it drains
  const uint32_t tl = tmem + ((uint32_t)(32 * (warp & 3)) << 16) + (uint32_t)colh;
  float accRe[TN / 2], accIm[TN / 2];
#pragma unroll
  for (int c = 0; c < TN / 2; ++c) {
    accRe[c] = 0.f;
    accIm[c] = 0.f;
  }
  constexpr int TK = P::kTK, KR = P::kKR, kRun = P::kRun, kHalf = kRun / 2;
  // a chunk is TK complex K (KIND 0, 2) or KR real bands (KIND 1)
  constexpr int kStep = KIND == 1 ? KR : TK;
  const int nchunks = (gK + kStep - 1) / kStep;
  // Staging is software-pipelined: chunk ch + 1's operands are loaded from
  // global memory into registers while chunk ch's MMAs run, then split and
  // stored to shared memory once those MMAs are done with the tiles.
  // A: this thread's row and its run of kRun k (KIND 1: of two runs of bands, TK
  // apart, the halves of a chunk).  A warp loads 32 rows of one k and stores four
  // contiguous core matrices.
  const int ar = tid & (TM - 1), ak = (tid / TM) * kRun, am = m0 + ar;
  const uint32_t aoff = (ar >> 3) * kSBO + (tid / TM) * kLBO + (ar & 7) * 16;
  // B: its column n and its half run of k; a warp loads 8 columns by the chunk's
  // K (whole sectors in either order), and half a warp stores one core matrix
  const int bp = (lane & 1) | ((lane >> 4) << 1), br = 8 * warp + ((lane >> 1) & 7);
  const int bk = bp * kHalf, bn = n0 + br;
  const uint32_t boff = (br >> 3) * kSBO + (bp >> 1) * kLBO + (br & 7) * 16 + (bp & 1) * 8;
  // the slice and the row in it of row m (KIND 0)
  auto slice_of = [&](int m) -> int { return g.fold ? m / g.slice_m : b; };
  auto row_of = [&](int m) -> int { return g.fold ? m % g.slice_m : m; };
  // where the row's and the column's k = 0 are, the step along k, and the end of k
  // (0: a row or column outside); 32-bit element steps, 64-bit addresses
  const float2 *ap = nullptr, *bq = nullptr;
  const float *xp = nullptr, *yp = nullptr;
  size_t as = 1, bs = 1;
  const int aend = am < gM ? gK : 0;
  int bend = bn < gN ? gK : 0;
  if (KIND == 0) {
    const int m = am < gM ? am : 0, n = bn < gN ? bn : 0;
    const float2 *A = g.A + (size_t)slice_of(m) * g.sA, *B = g.B + (size_t)b * g.sB;
    as = OPB == 2 ? 1 : (size_t)g.lda;
    ap = A + (OPB == 2 ? (size_t)g.lda * row_of(m) : (size_t)row_of(m)) + as * ak;
    bs = OPB == 1 ? (size_t)g.ldb : 1;
    bq = B + (OPB == 1 ? (size_t)n : (size_t)g.ldb * n) + bs * bk;
  } else {
    as = f.P;
    const int m = am < gM ? am : 0;
    if (KIND == 1) {
      xp = xb + m + as * ak;
      if (kTwo && yb) yp = yb + m + as * ak;
    } else {
      ap = specb + wpos(m) + as * ak;
    }
  }
  // The DFT kinds' B operand, twiddles exp(-2 pi i j / n3) from a table that stays
  // in L1, is read when the chunk is stored.  Entry k of column n is j = n k mod n3:
  // ti is this thread's first of the chunk, and j goes on by n, ti by n kStep.
  unsigned ti = 0, tstep = 0, thalf = 0;
  if (KIND != 0) {
    const unsigned n3 = (unsigned)f.n3, n = (unsigned)bn;
    ti = n * (unsigned)bk % n3;
    tstep = n * (unsigned)kStep % n3;
    thalf = n * (unsigned)TK % n3;
  }
  auto on = [&](unsigned j, unsigned by) -> unsigned {  // (j + by) mod n3, both below n3
    j += by;
    return j >= (unsigned)f.n3 ? j - (unsigned)f.n3 : j;
  };
  float2 ra[kRun], rb[KIND == 0 ? kHalf : 1];
  // KIND 1 with a second cube: its raw values, combined (x - ycoef y) only when
  // the chunk is stored, so that the loads stay in flight meanwhile
  float2 ry[kTwo ? kRun : 1];
  auto load_chunk = [&](int k0) {
    if constexpr (KIND == 1) {
      auto pair = [&](const float *q, int i) -> float2 {
        const int k = k0 + ak + i;
        return make_float2(k < aend ? q[as * (k0 + i)] : 0.f,
                           k + TK < aend ? q[as * (k0 + TK + i)] : 0.f);
      };
#pragma unroll
      for (int i = 0; i < kRun; ++i) {
        ra[i] = pair(xp, i);
        if (kTwo && yp) ry[kTwo ? i : 0] = pair(yp, i);
      }
    } else {
      const float2 *q = ap + as * k0;
#pragma unroll
      for (int i = 0; i < kRun; ++i)  // raw: conjugated (OPB 2, transposed slices) when stored
        ra[i] = k0 + ak + i < aend ? q[as * i] : make_float2(0.f, 0.f);
      if constexpr (KIND == 0) {
        const float2 *p = bq + bs * k0;
#pragma unroll
        for (int i = 0; i < kHalf; ++i)  // raw (OPB 1: conjugated when stored): combining a
          // value where it is loaded makes the thread wait for it there
          rb[i] = k0 + bk + i < bend ? p[bs * i] : make_float2(0.f, 0.f);
      }
    }
  };
  // split the registers' chunk into the hi / lo tiles of stage `st`
  auto store_chunk = [&](int st, int k0) {
    char *a = smem + st * kStageBytes + aoff, *q = smem + st * kStageBytes + 4 * kHalfA + boff;
    float re[kRun], im[kRun];
#pragma unroll
    for (int i = 0; i < kRun; ++i) {
      float2 v = ra[i];
      if (kTwo && yp) {
        const float2 w = ry[kTwo ? i : 0];
        v = make_float2(v.x - f.ycoef * w.x, v.y - f.ycoef * w.y);
      }
      if ((KIND == 2 && f.trans) || (KIND == 0 && OPB == 2)) v.y = -v.y;
      re[i] = v.x;
      im[i] = v.y;
    }
    Run<PREC, kRun>(re).put(a, a + 2 * kHalfA);
    Run<PREC, kRun>(im).put(a + kHalfA, a + 3 * kHalfA);
    auto block = [&](int i, const Run<PREC, kHalf> &x) {
      x.put(q + i * kBlockB, q + kLoB + i * kBlockB);
    };
    float u[kHalf], v[kHalf];
    if constexpr (KIND == 0) {
#pragma unroll
      for (int i = 0; i < kHalf; ++i) {
        u[i] = rb[i].x;
        v[i] = OPB == 1 ? -rb[i].y : rb[i].y;
      }
      block(1, Run<PREC, kHalf>(u));
      Run<PREC, kHalf> y(v);
      block(2, y);
      y.negate();
      block(0, y);
    } else if constexpr (KIND == 1) {
      // the twiddles of the chunk's bands, half by half
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        unsigned j = h ? on(ti, thalf) : ti;
#pragma unroll
        for (int i = 0; i < kHalf; ++i) {
          const float2 t = k0 + bk + h * TK + i < bend ? f.tw3[j] : make_float2(0.f, 0.f);
          u[i] = t.x;
          v[i] = t.y;
          j = on(j, (unsigned)bn);
        }
        block(2 * h, Run<PREC, kHalf>(u));
        block(2 * h + 1, Run<PREC, kHalf>(v));
      }
      ti = on(ti, tstep);
    } else {
      // w_k exp(+2 pi i k c / n3) of the chunk's frequencies, its imaginary part
      // negated: the table's, as it is
      unsigned j = ti;
#pragma unroll
      for (int i = 0; i < kHalf; ++i) {
        const int k = k0 + bk + i;
        const float2 t = k < bend ? f.tw3[j] : make_float2(0.f, 0.f);
        const float wk = (k == 0 || 2 * k == f.n3) ? 1.0f : 2.0f;
        u[i] = wk * t.x;
        v[i] = wk * t.y;
        j = on(j, (unsigned)bn);
      }
      block(0, Run<PREC, kHalf>(u));
      block(1, Run<PREC, kHalf>(v));
      ti = on(ti, tstep);
    }
  };
  // one thread: the chunk's MMAs on stage `st` into a fresh TMEM tile `st`,
  // committed to barrier `st`
  auto issue = [&](int st) {
    const uint32_t a = smem_u32(smem + st * kStageBytes), q = a + 4 * kHalfA;
    const uint32_t dt = tmem + (uint32_t)st * (2 * TN);
    // Re C (tile columns 0..63) and Im C (64..127) from one N = 128 MMA over two
    // adjacent blocks, so that A is read once for both; the real part alone (KIND 2)
    // from N = 64.  j: A's real parts (KIND 1: the first bands), then the others.
    // Three split products each, into a fresh tile per chunk.
    const uint32_t id = KIND == 2 ? idesc : idesc2;
#pragma unroll
    for (int j = 0; j < 2; ++j) {
      const uint32_t acc0 = j > 0 ? 1u : 0u;
      const uint64_t ah = sdesc(a + j * kHalfA), al = sdesc(a + (2 + j) * kHalfA);
      const int blk = KIND == 0 ? 1 - j : (KIND == 1 ? 2 * j : j);
      const uint64_t bh = sdesc(q + blk * kBlockB), bl = sdesc(q + kLoB + blk * kBlockB);
      if (PREC != 2) mma<PREC>(dt, ah, bh, id, acc0);
      mma<PREC>(dt, ah, bl, id, PREC != 2 ? 1u : acc0);
      mma<PREC>(dt, al, bh, id, 1u);
    }
    if (PREC == 2) {
#pragma unroll
      for (int j = 0; j < 2; ++j) {
        const int blk = KIND == 0 ? 1 - j : (KIND == 1 ? 2 * j : j);
        mma<PREC>(dt, sdesc(a + j * kHalfA), sdesc(q + blk * kBlockB), id, 1u);
      }
    }
    asm volatile(
        "tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(
            st ? bar1 : bar0));
  };
  auto mark_issued = [&](int st) {
    if (st) out1 = true;
    else out0 = true;
  };
  // add TMEM tile `st` into the FP32 register accumulators
  auto drain = [&](int st) {
    const uint32_t tile = (uint32_t)st * (2 * TN);
#pragma unroll
    for (int c0 = 0; c0 < TN / 2; c0 += 16) {
      uint32_t re[16], im[16];
      asm volatile(
          "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
          : "=r"(re[0]), "=r"(re[1]), "=r"(re[2]), "=r"(re[3]), "=r"(re[4]), "=r"(re[5]),
            "=r"(re[6]), "=r"(re[7]), "=r"(re[8]), "=r"(re[9]), "=r"(re[10]), "=r"(re[11]),
            "=r"(re[12]), "=r"(re[13]), "=r"(re[14]), "=r"(re[15])
          : "r"(tl + tile + c0));
      if (KIND == 1) {
        // the real parts first: half the destination registers live at once,
        // which leaves room for the next chunk's loads of both cubes
        asm volatile("tcgen05.wait::ld.sync.aligned;");
#pragma unroll
        for (int c = 0; c < 16; ++c) accRe[c0 + c] += __uint_as_float(re[c]);
      }
      if (KIND != 2)
        asm volatile(
            "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
            : "=r"(im[0]), "=r"(im[1]), "=r"(im[2]), "=r"(im[3]), "=r"(im[4]), "=r"(im[5]),
              "=r"(im[6]), "=r"(im[7]), "=r"(im[8]), "=r"(im[9]), "=r"(im[10]), "=r"(im[11]),
              "=r"(im[12]), "=r"(im[13]), "=r"(im[14]), "=r"(im[15])
            : "r"(tl + tile + TN + c0));
      asm volatile("tcgen05.wait::ld.sync.aligned;");
#pragma unroll
      for (int c = 0; c < 16; c += 2) {
        if (KIND != 1)
          add2(accRe[c0 + c], accRe[c0 + c + 1], __uint_as_float(re[c]),
               __uint_as_float(re[c + 1]));
        if (KIND == 1) {  // no packed pairs among this kind's live registers
          accIm[c0 + c] += __uint_as_float(im[c]);
          accIm[c0 + c + 1] += __uint_as_float(im[c + 1]);
        } else if (KIND == 0) {
          add2(accIm[c0 + c], accIm[c0 + c + 1], __uint_as_float(im[c]),
               __uint_as_float(im[c + 1]));
        }
      }
    }
    // the tile is rewritten only after every thread's reads
    asm volatile("tcgen05.fence::before_thread_sync;");
  };
  // every thread waits for the MMAs committed to barrier `st`; on a timeout
  // the commit stays outstanding for the last bounded wait before the free
  auto wait_mmas = [&](int st) {
    const bool done = mbar_wait(st ? bar1 : bar0, st ? ph1 : ph0);
    if (done) {
      if (st) {
        ph1 ^= 1u;
        out1 = false;
      } else {
        ph0 ^= 1u;
        out0 = false;
      }
    } else {
      ok = false;
    }
    asm volatile("tcgen05.fence::after_thread_sync;");
  };
  // the stage is written and the tile drained by all; whether no wait ran out
  auto stage_barrier = [&]() {
    asm volatile("fence.proxy.async.shared::cta;");
    asm volatile("tcgen05.fence::before_thread_sync;");
    ok = __syncthreads_and(ok) != 0;
    asm volatile("tcgen05.fence::after_thread_sync;");
  };
  if (nchunks > 0) load_chunk(0);
  // chunk ch: stage s = ch & 1 is written while chunk ch - 1's MMAs (stage
  // s ^ 1) run; chunk ch's are queued behind them, and chunk ch - 1's tile is
  // drained while they run
  for (int ch = 0; ch < nchunks; ++ch) {
    const int st = ch & 1;
    store_chunk(st, ch * kStep);  // stage st was last read by chunk ch - 2
    if (ch + 1 < nchunks) load_chunk((ch + 1) * kStep);
    stage_barrier();
    if (!ok) break;
    if (tid == 0) issue(st);
    mark_issued(st);
    if (ch > 0) {
      wait_mmas(st ^ 1);
      if (ok) drain(st ^ 1);
    }
  }
  if (nchunks > 0) {
    const int last = (nchunks - 1) & 1;
    if (ok) wait_mmas(last);
    ok = __syncthreads_and(ok) != 0;
    if (ok) drain(last);
  }
  if constexpr (PREC == 2) {
    // Below about 2^-102 the low halves leave FP32's normal range and a value's
    // digits are lost (2.6e-6 of a cube at 1e-34).  The single operators take any
    // magnitude: a warp whose part of the tile lies all below what K such terms can
    // sum to forms it again with FP32 FMAs, eight terms at a time, unless an operand
    // is zero.  One accumulator decides for most warps: a Z-solve of 145 x 145 x 220
    // takes 261 us without it and 262 with it (cubes below 1e-30: 2.7 ms, of zeros 390
    // us); collecting the operands' magnitudes where they are split took 312.
    constexpr float limit = KIND == 0 ? 0x1p-93f : 0x1p-90f;  // K up to 512, 4096
    float most = fabsf(accRe[0]);
    bool low = ok && m0 + row - lane < gM && n0 + colh < gN &&
               !__any_sync(0xffffffffu, !(most < limit));
    if (low) {
#pragma unroll
      for (int c = 0; c < TN / 2; ++c)
        most = fmaxf(most, fmaxf(fabsf(accRe[c]), fabsf(accIm[c])));
      low = !__any_sync(0xffffffffu, !(most < limit));
    }
    if (low) {
      const int gm = m0 + row < gM ? m0 + row : 0, sl = KIND == 0 ? slice_of(gm) : 0;
      auto at = [&](int k) -> float2 {  // A(gm, k)
        if constexpr (KIND == 0) {
          static_assert(OPB == 0, "of the operators' products");
          return g.A[(size_t)sl * g.sA + row_of(gm) + (size_t)g.lda * k];
        } else if constexpr (KIND == 1) {
          return make_float2(f.x[(size_t)blockIdx.z * f.N + gm + f.P * k], 0.f);
        } else {
          const float2 v = f.spec[((size_t)blockIdx.z * f.h + k) * f.P + wpos(gm)];
          return make_float2(v.x, f.trans ? -v.y : v.y);
        }
      };
      auto with = [&](int k, int n) -> float2 {  // op(B)(k, n)
        if constexpr (KIND == 0) {
          return g.B[(size_t)b * g.sB + (size_t)g.ldb * n + k];
        } else {
          const float2 v = f.tw3[(unsigned)n * (unsigned)k % (unsigned)f.n3];
          if (KIND == 1) return v;
          const float w = (k == 0 || 2 * k == f.n3) ? 1.0f : 2.0f;
          return make_float2(w * v.x, -w * v.y);
        }
      };
      bool a_any = false, b_any = KIND != 0;
      for (int k = 0; k < gK; ++k) {
        const float2 v = at(k);
        a_any |= v.x != 0.f || v.y != 0.f;
        if (KIND == 0 && n0 + colh + lane < gN) {
          const float2 w = with(k, n0 + colh + lane);
          b_any |= w.x != 0.f || w.y != 0.f;
        }
      }
      if (__any_sync(0xffffffffu, a_any) && __any_sync(0xffffffffu, b_any)) {
#pragma unroll
        for (int c0 = 0; c0 < TN / 2; c0 += 4) {
          float re[4] = {}, im[4] = {};
          for (int k0 = 0; k0 < gK; k0 += 8) {
            float pr[4] = {}, pi[4] = {};
            for (int k = k0; k < k0 + 8 && k < gK; ++k) {
              const float2 a = at(k);
#pragma unroll
              for (int c = 0; c < 4; ++c) {
                const int n = n0 + colh + c0 + c;
                const float2 v = with(k, n < gN ? n : 0);
                pr[c] = fmaf(a.x, v.x, fmaf(-a.y, v.y, pr[c]));
                pi[c] = fmaf(a.x, v.y, fmaf(a.y, v.x, pi[c]));
              }
            }
#pragma unroll
            for (int c = 0; c < 4; ++c) {
              re[c] += pr[c];
              im[c] += pi[c];
            }
          }
#pragma unroll
          for (int c = 0; c < 4; ++c) {
            accRe[c0 + c] = re[c];
            accIm[c0 + c] = im[c];
          }
        }
      }
    }
  }
  // give MMAs still in flight a last bounded chance to land before the free
  auto last_wait = [&]() {
    if (out0) mbar_wait(bar0, ph0);
    if (out1) mbar_wait(bar1, ph1);
  };
  if (PREC == 2 && !ok) {  // the single operators have no flag to set: the tile is not a number
    last_wait();
#pragma unroll
    for (int c = 0; c < TN / 2; ++c) accRe[c] = accIm[c] = __int_as_float(0x7fffffff);
  }
  if (PREC != 2 && !ok) {
    if (tid == 0 && err) atomicExch(err, 1);
    last_wait();
  } else if (nchunks > 0) {
    // epilogue: thread (warp w, lane l) owns row m0 + 32 (w mod 4) + l of the
    // tile, columns colh .. colh + 31
    const int gm = m0 + row;
    if (KIND == 1 && gm < gM) {
      float2 *ob = f.spec_out + (size_t)b * f.h * f.P + wpos(gm);
#pragma unroll
      for (int c = 0; c < TN / 2; ++c) {
        const int n = n0 + colh + c;
        if (n >= gN) break;
        ob[f.P * n] = make_float2(accRe[c], f.trans ? -accIm[c] : accIm[c]);
      }
    } else if (KIND == 2 && gm < gM) {
      const float inv = 1.0f / (float)f.n3;
      const size_t base = (size_t)b * f.N + gm;
      const bool g4 = f.mode == 1 && f.gamma4;
      // eight columns at a time: their Gamma4 and F loads are issued together
      // before any is used
#pragma unroll
      for (int c0 = 0; c0 < TN / 2; c0 += 8) {
        float g[8], fv[8];
        if (g4) {
#pragma unroll
          for (int c = 0; c < 8; ++c) {
            const int n = n0 + colh + c0 + c;
            const bool in = n < gN;
            const size_t v = base + f.P * (in ? n : 0);
            g[c] = in ? f.G4[v] : 0.0f;
            fv[c] = in ? f.F[v] : 0.0f;
          }
        }
#pragma unroll
        for (int c = 0; c < 8; ++c) {
          const int n = n0 + colh + c0 + c;
          if (n >= gN) break;
          const size_t v = base + f.P * n;
          const float r = accRe[c0 + c] * inv;
          f.out[v] = r;
          if (g4) f.G4[v] = g[c] + f.mu * (r - fv[c]);
        }
      }
    } else if (KIND == 0 && gm < g.M) {
      const int sl = slice_of(gm), mr = row_of(gm);
      const int lb = g.lam3_period > 0 ? sl % g.lam3_period : sl;
      float2 *C = g.C + (size_t)sl * g.sC + mr;
#pragma unroll
      for (int c = 0; c < TN / 2; ++c) {
        const int n = n0 + colh + c;
        if (n >= g.N) break;
        float2 v = make_float2(accRe[c], accIm[c]);
        if (EPI == 1) {
          const float den = g.mu * (1.0f + g.lam1[mr] + g.lam2[n] + g.lam3[lb]);
          const float q = g.scale / den;
          v.x *= q;
          v.y *= q;
        }
        C[(size_t)g.ldc * n] = v;
      }
    }
  }
  asm volatile("tcgen05.fence::before_thread_sync;");
  __syncthreads();
  if (warp == 0)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "n"(kCols));
}

// Checks the GEMM's bounded barrier wait and its timeout path: one warp
// allocates tensor memory as the GEMM does, then waits on an mbarrier with
// the wait cut to `tries` tries.  With `arrive`, lane 0 arrives first and the
// phase completes; without, nothing arrives and the wait runs out.  A timeout
// is recorded in out[0]; the tensor memory is freed on both paths, and
// out[1] counts the lanes that got past the free.
__global__ void __launch_bounds__(32) k_wait_probe(long long tries, int arrive, int *out) {
  __shared__ __align__(8) uint64_t bar;
  __shared__ uint32_t slot;
  const uint32_t b = smem_u32(&bar);
  if (threadIdx.x == 0) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(b));
    asm volatile("fence.mbarrier_init.release.cluster;");
  }
  asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], 32;" ::"r"(
                   smem_u32(&slot)));
  asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
  asm volatile("tcgen05.fence::before_thread_sync;");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;");
  const uint32_t tmem = slot;
  if (arrive && threadIdx.x == 0)
    asm volatile("{\n .reg .b64 st;\n mbarrier.arrive.shared::cta.b64 st, [%0];\n}\n" ::"r"(b)
                 : "memory");
  __syncwarp();
  if (!mbar_wait(b, 0u, tries)) atomicOr(out, 1);
  asm volatile("tcgen05.fence::before_thread_sync;");
  __syncthreads();
  asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, 32;" ::"r"(tmem));
  atomicAdd(out + 1, 1);
}

// Tensor-pipe throughput probe: one CTA per SM, one thread issuing n_mma
// MMAs of M = 128, N = 256 (K = 8 TF32 or 16 BF16 per instruction) from
// shared-memory tiles into two alternating TMEM accumulators, then one
// commit and a bounded wait.  The tiles hold a fixed non-zero pattern (the
// tensor core's power, and so its clock under the power cap, depends on the
// data).  A wait that runs out sets *err; tensor memory is freed either way.
constexpr int kProbeN = 256;
constexpr size_t kProbeSmem = 120 * 1024;  // more than half the SM's shared memory: one CTA per SM

template <int PREC>
__global__ void __launch_bounds__(128, 1) k_mma_peak(long long n_mma, int *err) {
  extern __shared__ __align__(1024) char smem[];
  using P = Prec<PREC>;
  __shared__ __align__(8) uint64_t mbar;
  __shared__ uint32_t tslot;
  const int tid = threadIdx.x, warp = tid >> 5;
  const size_t tile_bytes = (size_t)(TM + kProbeN) * P::kKR * P::kBytes;
  for (size_t e = tid; e < tile_bytes / 4; e += blockDim.x) {
    const uint32_t h = (uint32_t)e * 2654435761u;
    const float x = 0.25f + (float)(h >> 9) * (1.0f / 16777216.0f);  // in [0.25, 1.25)
    if (PREC == 0) {
      ((float *)smem)[e] = tf32_hi(x);
    } else {
      __nv_bfloat162 v = __floats2bfloat162_rn(x, 1.5f - x);
      ((__nv_bfloat162 *)smem)[e] = v;
    }
  }
  if (tid == 0) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_u32(&mbar)));
    asm volatile("fence.mbarrier_init.release.cluster;");
  }
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], 512;" ::"r"(
        smem_u32(&tslot)));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
  }
  asm volatile("fence.proxy.async.shared::cta;");
  asm volatile("tcgen05.fence::before_thread_sync;");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;");
  const uint32_t tmem = tslot;
  const uint32_t idesc = (1u << 4) | (P::kFmt << 7) | (P::kFmt << 10) |
                         ((uint32_t)(kProbeN >> 3) << 17) | ((uint32_t)(TM >> 4) << 24);
  const uint32_t bar = smem_u32(&mbar);
  if (tid == 0) {
    const uint64_t a = sdesc(smem_u32(smem));
    const uint64_t b = sdesc(smem_u32(smem + (size_t)TM * P::kKR * P::kBytes));
    for (long long i = 0; i < n_mma; ++i)
      mma<PREC>(tmem + (uint32_t)(i & 1) * kProbeN, a, b, idesc, i > 1 ? 1u : 0u);
    asm volatile(
        "tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar));
  }
  __syncwarp();
  if (!mbar_wait(bar, 0u) && tid == 0) atomicExch(err, 1);
  asm volatile("tcgen05.fence::after_thread_sync;");
  __syncthreads();
  if (warp == 0)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, 512;" ::"r"(tmem));
}

template <int OPB, int EPI, int PREC>
cudaError_t launch_one(CGemm g, int *err, cudaStream_t st) {
  const size_t smem = 2 * stage_bytes(0);
  cudaError_t e = cudaFuncSetAttribute(k_cgemm_tc<OPB, EPI, PREC>,
                                       cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  // Slices that share A or B are one matrix, see the kernel (41 slices of 200 x 200,
  // where 328 tiles left 24 to a second wave: 54 -> 31 us)
  const long long rows = (long long)g.M * g.batch, cols = (long long)g.N * g.batch;
  g.fold = 0;
  if (OPB == 0 && g.batch > 1 && !g.gate && rows < (1 << 30) && cols < (1 << 21)) {
    if (g.sB == 0) {
      g.fold = 1;
      g.slice_m = g.M;
      g.M = (int)rows;
      g.batch = 1;
    } else if (EPI == 0 && g.sA == 0 && g.sB == (long long)g.ldb * g.N &&
               g.sC == (long long)g.ldc * g.N) {
      g.N = (int)cols;
      g.batch = 1;
    }
  }
  const unsigned mt = (g.M + TM - 1) / TM, nt = (g.N + TN - 1) / TN;
  const dim3 grid = g.fold ? dim3(mt * nt) : dim3(mt, nt, g.batch);
  k_cgemm_tc<OPB, EPI, PREC><<<grid, kThreads, smem, st>>>(g, Dft3{}, err);
  return cudaGetLastError();
}

template <int KIND, int PREC>
cudaError_t launch_dft(const Dft3 &f, int nb, int *err, cudaStream_t st) {
  const size_t smem = 2 * stage_bytes(KIND);
  cudaError_t e = cudaFuncSetAttribute(k_cgemm_tc<0, 0, PREC, KIND>,
                                       cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  const size_t mt = (f.P + TM - 1) / TM;
  const size_t nt = ((KIND == 1 ? f.h : f.n3) + TN - 1) / TN;
  dim3 grid((unsigned)(mt * nt), 1, nb);
  k_cgemm_tc<0, 0, PREC, KIND><<<grid, kThreads, smem, st>>>(CGemm{}, f, err);
  return cudaGetLastError();
}

template <int PREC>
cudaError_t launch_prec(const CGemm &g, int *err, cudaStream_t st) {
  if (g.opA == 1) {  // A^H B only
    if constexpr (PREC != 2)
      if (g.opB == 0 && g.epi == 0) return launch_one<2, 0, PREC>(g, err, st);
    return cudaErrorInvalidValue;
  }
  if (g.opB == 0 && g.epi == 0) return launch_one<0, 0, PREC>(g, err, st);
  if (g.opB == 0 && g.epi == 1) return launch_one<0, 1, PREC>(g, err, st);
  if constexpr (PREC != 2)  // the operators' reconstruction is in FP32
    if (g.opB == 1 && g.epi == 0) return launch_one<1, 0, PREC>(g, err, st);
  return cudaErrorInvalidValue;
}

}  // namespace

long long cgemm_tc_wait_limit() { return kWaitLimit; }

cudaError_t launch_wait_probe(long long tries, int arrive, int *out, cudaStream_t st) {
  k_wait_probe<<<1, 32, 0, st>>>(tries, arrive, out);
  return cudaGetLastError();
}

cudaError_t launch_mma_peak(int prec, int nsm, long long n_mma, int *err, cudaStream_t st,
                            double *flops) {
  const double per = 2.0 * TM * kProbeN * (prec ? 16 : 8);
  *flops = per * (double)n_mma * nsm;
  if (prec == 0) {
    cudaError_t e = cudaFuncSetAttribute(k_mma_peak<0>,
                                         cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kProbeSmem);
    if (e != cudaSuccess) return e;
    k_mma_peak<0><<<nsm, 128, kProbeSmem, st>>>(n_mma, err);
  } else {
    cudaError_t e = cudaFuncSetAttribute(k_mma_peak<1>,
                                         cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kProbeSmem);
    if (e != cudaSuccess) return e;
    k_mma_peak<1><<<nsm, 128, kProbeSmem, st>>>(n_mma, err);
  }
  return cudaGetLastError();
}

cudaError_t launch_dft3_tc(int kind, const Dft3 &f, int nb, int *err, cudaStream_t st, int prec) {
  if (f.P == 0 || nb <= 0) return cudaSuccess;
  if (f.P > (size_t)TM * 0x7fffffff / 4) return cudaErrorInvalidValue;
  if (prec == 2 && f.y) return cudaErrorInvalidValue;
  if (kind == 1)
    return prec == 1   ? launch_dft<1, 1>(f, nb, err, st)
           : prec == 2 ? launch_dft<1, 2>(f, nb, err, st)
                       : launch_dft<1, 0>(f, nb, err, st);
  if (kind == 2)
    return prec == 1   ? launch_dft<2, 1>(f, nb, err, st)
           : prec == 2 ? launch_dft<2, 2>(f, nb, err, st)
                       : launch_dft<2, 0>(f, nb, err, st);
  return cudaErrorInvalidValue;
}

cudaError_t launch_cgemm_tc(const CGemm &g, int *err, cudaStream_t st, int prec) {
  if (g.M <= 0 || g.N <= 0 || g.batch <= 0) return cudaSuccess;
  if (g.epi == 2) return cudaErrorInvalidValue;  // SIMT kernel only
  if (prec == 0) return launch_prec<0>(g, err, st);
  if (prec == 1) return launch_prec<1>(g, err, st);
  if (prec == 2) return launch_prec<2>(g, err, st);
  return cudaErrorInvalidValue;
}

}  // namespace lrstv

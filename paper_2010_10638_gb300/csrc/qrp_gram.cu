// K-c, Gram form: the Householder QR with column pivoting of qrp.cu (Section III-D; the same
// pivots, the same Q) of a tall FP32 matrix A (m x n) from its Gram matrix.
//
// The column norms left by j reflectors, and row j of R up to its sign, follow from A^T A: they
// are those of a Cholesky factorisation with the same pivot rule.  So A is read once for
// S = A^T A, on the tensor cores, instead of once per reflector; the chain of k pivot steps
// runs in one block on n numbers; and Q follows from the k pivot columns alone:
//   1  qg_exp_kernel, qg_gram_kernel  S, fixed-point slices as in core.cu (error: see qg_eps;
//                        usually 2^-38 of |a_i| |a_j|), ranges of rows in double-float pairs
//   2  qg_reduce_kernel  the ranges added in order
//   3  qg_pivot_kernel   pivots p_1 .. p_k, the triangle R_1, its inverse (double-float)
//   4  qg_ortho_kernel   E = Q_1^T Q_1 - I for Q_1 = A_p R_1^-1 (double-float): the error of
//                        S, times the squared condition of A_p; its last block forms the
//                        inverse W of the Cholesky factor of I + E to E^2, and the signs
//   5  qg_q_kernel       Q = Q_1 W D: W is within 4e-6 of I, so Q is orthonormal to rounding
//                        whatever the condition (as A_p (R_1^-1 W) it was not: 2e-12)
// Householder's Q is that of the unique QR factorisation with positive diagonal up to the sign
// of each column, -sign(x_j), x_j the top entry of column j as reflector j finds it; the signs
// come from the elimination of the top k x k block of Q (Ballard, Demmel, Grigori, Jacquelin,
// Nguyen, Solomonik: Reconstructing Householder vectors from TSQR, 2014).
//
// Nothing is assumed about A's condition.  Step 3 carries a bound of the error of every norm:
// where the largest remaining norm does not exceed every other by more than their errors (ties,
// near ties), or its own error is not small (rank deficiency), and where E is not small (step
// 4) or A's magnitudes leave FP32's range, a device word is set, the later kernels leave, and
// the cluster form, launched behind them, runs after all; otherwise it leaves at once.  What was done up
// to there is lost, in every sweep anew (what ran before does not tell): 26 to 40 us for magnitudes, 45 to
// 125 us for rank deficiency (50,000 x 256, rank 5, k = 16: 3,080 us, the cluster form alone 2,955;
// 1,000 x 256 2,138 and 2,083; 200 x 64, k = 8 306 and 261).
//
// Why: a reflector of the cluster form takes one pass over A, two reductions and three block-wide
// chains of FP64 operations, 22 us at 50,000 x 256 and 8 us at any size.  50,000 x 256, k = 16:
// 363 -> 180 us (exponents 12, S 76, its sum 6, pivots 22, E 30, Q 13); 1,000 x 256: 186 -> 83;
// 100 x 64, k = 8: 82 -> 61.  Against an FP64 QR the entries of Q differ by 1e-14 to 7e-13, the
// cluster form's by 4e-8 to 2e-6 (its FP32 sums).
#include <algorithm>
#include <climits>

#include "qrp_gram.cuh"
#include "tc.cuh"

namespace tk {
namespace {

constexpr int kGM = 128;             // columns i (MMA M) and j (MMA N) of a tile of S
constexpr int kGBlock = 256;         // rows of A per exact block: level sums stay within 2^24
constexpr int kGRows = 128;          // rows of A: a CTA's range is a multiple
constexpr int kGK = 16;              // rows per stage
constexpr int kGStages = 3;
constexpr int kGSlices = 4, kGLevels = 4;
constexpr int kGT = 512, kGWarps = kGT / 32;  // slicing threads; one more warp issues the products
constexpr uint32_t kGCols = 512;     // tensor-memory columns: kGLevels * kGM
constexpr int kGSlice = kGM * kGK;   // BF16 elements per slice of an operand
constexpr uint32_t kGOperand = kGSlices * kGSlice * 2, kGStage = 2 * kGOperand;  // bytes

// the stages, and the tile's sums (in registers they spill)
__host__ __device__ constexpr size_t qg_smem_bytes() {
  return (size_t)kGStages * kGStage + sizeof(float2) * kGM * kGM + 128;
}

// Exponents: ex[block][c] = e with |A[r, c]| < 2^e for the 256 rows r of the block (-128:
// all zero).  Sets the flag for magnitudes that are not finite or so large or small (outside
// [2^-50, 2^50)) that products of them leave FP32's normal range.  Block = 128 columns, four row lanes.
__global__ void __launch_bounds__(512) qg_exp_kernel(const float *__restrict__ A, int64_t m, int64_t n, int64_t lda,
                                                     int8_t *__restrict__ ex, uint32_t *flag) {
  __shared__ uint32_t mx[4][128];
  const int cl = threadIdx.x & 127, rl = threadIdx.x >> 7;
  const int64_t c = (int64_t)blockIdx.y * 128 + cl, r0 = (int64_t)blockIdx.x * kGBlock;
  const int nr = (int)min((int64_t)kGBlock, m - r0);
  uint32_t v = 0;
  if (c < n) {
    const float *p = A + r0 * lda + c;
#pragma unroll 16
    for (int r = rl; r < kGBlock; r += 4) v = max(v, r < nr ? __float_as_uint(__ldg(p + r * lda)) & 0x7fffffffu : 0u);
  }
  mx[rl][cl] = v;
  __syncthreads();
  if (rl == 0) {
    v = max(max(mx[0][cl], mx[1][cl]), max(mx[2][cl], mx[3][cl]));
    if (c < n) ex[blockIdx.x * n + c] = v ? (int8_t)max(-127, min(127, above_exp_f32(v))) : (int8_t)-128;
    if (v >= 0x58800000u || (v && v < 0x26800000u)) atomicOr(flag, 1u);
  }
}

// Eight values of one column (t: scaled by 2^(8 - e)) into the four slices: t is split, exactly,
// into multiples of 1, 2^-8, 2^-16 and 2^-24 from the top (adding and subtracting 1.5 2^23 units
// rounds to the nearest multiple), each exact in BF16 (at most 2^8 units, after the first 2^7);
// eight consecutive k of a row are 16 bytes of the K-major tile.
__device__ __forceinline__ void qg_slices8(float (&t)[8], float sc, __nv_bfloat16 *out) {
#pragma unroll
  for (int k = 0; k < 8; ++k) t[k] *= sc;
#pragma unroll
  for (int s = 0; s < kGSlices; ++s) {
    const float big = s == 0 ? 12582912.f : s == 1 ? 49152.f : s == 2 ? 192.f : 0.75f;
    uint32_t w[4];
#pragma unroll
    for (int k = 0; k < 8; k += 2) {
      const float m0 = __fadd_rn(__fadd_rn(t[k], big), -big);
      const float m1 = __fadd_rn(__fadd_rn(t[k + 1], big), -big);
      t[k] -= m0;
      t[k + 1] -= m1;
      asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(w[k / 2]) : "f"(m1), "f"(m0));
    }
    *reinterpret_cast<uint4 *>(out + s * kGSlice) = make_uint4(w[0], w[1], w[2], w[3]);
  }
}

// 2^e as FP32 (|e| < 127)
__device__ __forceinline__ float qg_pow2(int e) { return __int_as_float((127 + e) << 23); }

__device__ __forceinline__ void qg_arrive(uint32_t bar) {
  asm volatile("{ .reg .b64 st; mbarrier.arrive.shared::cta.b64 st, [%0]; }" ::"r"(bar) : "memory");
}
__device__ __forceinline__ void qg_commit(uint32_t bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar) : "memory");
}

// Tile (i0 .. i0 + 127) x (j0 .. j0 + 127) of S over a range of rows of A, into part[range] as
// double-float pairs, transposed.  Sixteen warps read A 16 rows at a time, two stages ahead in
// registers (a thread owns a column and eight rows), slice it into one of three shared-memory
// stages, and add the levels of a block, 256 rows, to double-float sums (FP64 additions would
// cost more than the products: one warp instruction per 16 cycles).  A warp of its own issues
// the products (tcgen05.mma): levels 0, 1 and 2 (sums of slices' indices) are exact multiples of
// 2^-8L, 3 and 4 share an accumulator (rounded at 2^-40 of the whole).  The operands of a tile on
// the diagonal are one: its chunks are sliced by the two halves of the warps in turn.
// 50,000 x 256: 76 us; without the products 70, without the sums 66: the slicing (14 instructions
// a value and operand) and the reads of A bound it.  With 128 x 64 tiles, whose operands are sliced
// 4.5 times over instead of twice, blocks of 128 rows and a slicing warp that issues it took 180;
// with the sums in registers, which spill, 132.
__global__ void __launch_bounds__(kGT + 32, 1) qg_gram_kernel(const float *__restrict__ A, int64_t m, int64_t n,
                                                              int64_t lda, int64_t rows_per,
                                                              const int8_t *__restrict__ ex, float2 *__restrict__ part,
                                                              uint32_t *flag, uint32_t *err) {
  extern __shared__ unsigned char qg_raw[];
  unsigned char *base =
      reinterpret_cast<unsigned char *>((reinterpret_cast<uintptr_t>(qg_raw) + 127) & ~static_cast<uintptr_t>(127));
  // full[stage], empty[stage], levels of a block complete, levels read
  __shared__ __align__(8) unsigned long long bars[2 * kGStages + 2];
  __shared__ uint32_t tbase, given_up;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  // (one thread reads it for all: a block that times out may set it meanwhile, and a block has to
  // leave, or come to the allocation and the barriers below, as a whole)
  if (tid == 0) given_up = *flag;
  __syncthreads();
  if (given_up) return;
  int ti = 0, tj = (int)blockIdx.x;  // tiles on and below the diagonal
  while (tj > ti) tj -= ++ti;
  const bool diag = ti == tj;
  const int64_t i0 = (int64_t)ti * kGM, j0 = (int64_t)tj * kGM;
  const int64_t r_begin = (int64_t)blockIdx.y * rows_per, r_end = min(m, r_begin + rows_per);
  const int chunks = (int)((r_end - r_begin + kGK - 1) / kGK);
  const int phase = (int)(r_begin % kGBlock) / kGK;  // of the first chunk in its block
  constexpr int kPer = kGBlock / kGK;
  const uint32_t bar0 = (uint32_t)__cvta_generic_to_shared(bars);
  auto full = [&](int st) { return bar0 + 8u * st; };
  auto empty = [&](int st) { return bar0 + 8u * (kGStages + st); };
  const uint32_t done_bar = bar0 + 8u * 2 * kGStages, read_bar = done_bar + 8u;
  if (tid == 0) {
    for (int st = 0; st < kGStages; ++st) {
      asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(full(st)), "r"(diag ? kGWarps / 2 : kGWarps) : "memory");
      asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(empty(st)) : "memory");
    }
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(done_bar) : "memory");
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(read_bar), "r"(kGWarps) : "memory");
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                     (uint32_t)__cvta_generic_to_shared(&tbase)),
                 "r"(kGCols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem = tbase;
  bool ok = true;  // every wait is bounded: after one that gave up a warp leaves its loop, and so do the others
  const int ci = tid & (kGM - 1), hi = (tid / kGM) & 3;  // of the sums: row, columns 32 hi ..
  float2 *sums = reinterpret_cast<float2 *>(base + kGStages * kGStage) + tid;  // [column - 32 hi][thread]
  if (warp == kGWarps) {
    if (lane == 0) {
      // D f32, A and B bf16, both K-major, N >> 3, M >> 4
      const uint32_t idesc =
          (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(kGM >> 3) << 17) | ((uint32_t)(kGM >> 4) << 24);
      // K-adjacent core matrices are 128 bytes apart, 8-row groups kGK / 8 of them
      const uint64_t d0 = umma_desc((uint32_t)__cvta_generic_to_shared(base), 128, (kGK / 8) * 128);
      int issued = 0;
      for (int g = 0, st = 0; g < chunks && ok; ++g) {
        const int q = (g + phase) % kPer;  // chunk of the block
        const bool first = q == 0 || g == 0;
        const int blk = (g + phase) / kPer;
        if (first && g > 0) ok = tc_wait(read_bar, (uint32_t)((blk - 1) & 1));
        ok = ok && tc_wait(full(st), (uint32_t)((g / kGStages) & 1));
        if (!ok) break;
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        const uint64_t da = d0 + (uint64_t)(st * (kGStage >> 4)), db = diag ? da : da + (kGOperand >> 4);
#pragma unroll
        for (int ks = 0; ks < kGK / 16; ++ks)
#pragma unroll
          for (int L = 0; L <= kGSlices; ++L)
#pragma unroll
            for (int sa = 0; sa < kGSlices; ++sa) {
              const int sb = L - sa;
              if (sb < 0 || sb >= kGSlices) continue;
              const uint32_t add = (!first || ks > 0 || L == kGSlices || sa > 0) ? 1u : 0u;
              asm volatile(
                  "{ .reg .pred p; setp.ne.u32 p, %4, 0; tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p; }" ::"r"(
                      tmem + (uint32_t)(min(L, kGLevels - 1) * kGM)),
                  "l"(da + (uint64_t)((sa * kGSlice * 2 + ks * 256) >> 4)),
                  "l"(db + (uint64_t)((sb * kGSlice * 2 + ks * 256) >> 4)), "r"(idesc), "r"(add)
                  : "memory");
            }
        qg_commit(empty(st));
        if (q == kPer - 1 || g == chunks - 1) qg_commit(done_bar);
        issued = g + 1;
        st = st + 1 == kGStages ? 0 : st + 1;
      }
      // (after a give-up the products in flight get the same time to end)
      if (!ok && issued) tc_wait(empty((issued - 1) % kGStages), (uint32_t)(((issued - 1) / kGStages) & 1));
    }
    __syncwarp();
  } else {
    // slicing: the first eight warps take the columns i, the others the columns j (on the diagonal
    // every second chunk); of a chunk, column ci, rows 8 half .. 8 half + 7
    const int part_j = tid / 256, half = (tid / kGM) & 1;
    const int64_t col = (part_j && !diag ? j0 : i0) + ci;
    const bool in = col < n;
    const float *src = A + (r_begin + 8 * half) * lda + col;
    const int rows = (int)(r_end - r_begin) - 8 * half;  // left from this thread's first row on
    const int step = diag ? 2 : 1;
    auto load = [&](float (&v)[8], int g) {  // chunk g (past the range: zeros, and no read)
#pragma unroll
      for (int k = 0; k < 8; ++k) {
        const int r = g * kGK + k;
        v[k] = (in && r < rows) ? __ldg(src + r * lda) : 0.f;
      }
    };
    // element (row, k) of an operand: ((row / 8) (kGK / 8) + k / 8) 64 + (row % 8) 8 + k % 8
    __nv_bfloat16 *out = reinterpret_cast<__nv_bfloat16 *>(base + (part_j && !diag ? kGOperand : 0)) +
                         ((ci >> 3) * (kGK / 8) + half) * 64 + (ci & 7) * 8;
    const int8_t *exb = ex + (r_begin / kGBlock) * n;  // exponents of block 0 of the range
    // the levels of block blk into the sums
    auto add_levels = [&](int blk) {
      ok = __all_sync(0xffffffffu, tc_wait(done_bar, (uint32_t)(blk & 1)) ? 1 : 0) != 0;
      if (!ok) return;
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      const int64_t jl = j0 + hi * 32 + lane;
      const int ei = i0 + ci < n ? (int)__ldg(exb + blk * n + i0 + ci) : -128;
      const int ej = jl < n ? (int)__ldg(exb + blk * n + jl) : -128;
      const float ps = ei > -128 ? qg_pow2(ei) * (1.f / 65536.f) : 0.f, pl = ej > -128 ? qg_pow2(ej) : 0.f;
#pragma unroll
      for (int q0 = 0; q0 < 32; q0 += 8) {
        uint32_t w[kGLevels][8];
#pragma unroll
        for (int L = 0; L < kGLevels; ++L) {
          const uint32_t taddr = tmem + ((uint32_t)((warp & 3) * 32) << 16) + (uint32_t)(L * kGM + hi * 32 + q0);
          asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
                       : "=r"(w[L][0]), "=r"(w[L][1]), "=r"(w[L][2]), "=r"(w[L][3]), "=r"(w[L][4]), "=r"(w[L][5]),
                         "=r"(w[L][6]), "=r"(w[L][7])
                       : "r"(taddr));
        }
        asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
        for (int q = 0; q < 8; ++q) {
          DF t;
          t.hi = __uint_as_float(w[0][q]);
          df_add1(t, __uint_as_float(w[1][q]));
          t.lo += __uint_as_float(w[2][q]) + __uint_as_float(w[3][q]);
          const float sc = ps * __shfl_sync(0xffffffffu, pl, q0 + q);
          DF x;
          if (blk > 0) {
            const float2 v = sums[(q0 + q) * kGT];
            x.hi = v.x;
            x.lo = v.y;
          }
          x.lo = fmaf(t.lo, sc, x.lo);
          df_add1(x, t.hi * sc);
          sums[(q0 + q) * kGT] = make_float2(x.hi, x.lo);
        }
      }
      asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
      __syncwarp();
      if (lane == 0) qg_arrive(read_bar);
    };
    float sc = 0.f;
    int cur = -1, summed = 0;  // block of sc; blocks in the sums
    auto chunk = [&](float (&v)[8], int g) {
      const int blk = (g + phase) / kPer, st = g % kGStages;
      if (blk != cur) {
        const int e = in ? (int)__ldg(exb + blk * n + col) : -128;
        sc = e > -128 ? qg_pow2(8 - e) : 0.f;
        cur = blk;
      }
      if (g >= kGStages) {  // the products that read this stage
        ok = __all_sync(0xffffffffu, tc_wait(empty(st), (uint32_t)((g / kGStages - 1) & 1)) ? 1 : 0) != 0;
        if (!ok) return;
      }
      qg_slices8(v, sc, out + st * (kGStage / 2));
      load(v, g + 2 * step);
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
      __syncwarp();
      if (lane == 0) qg_arrive(full(st));
      for (; summed < blk && ok; ++summed) add_levels(summed);  // the block before, with a chunk of this one under way
    };
    float v0[8], v1[8];
    int g = diag ? part_j : 0;
    load(v0, g);
    load(v1, g + step);
    for (; g < chunks && ok; g += 2 * step) {
      chunk(v0, g);
      if (g + step < chunks && ok) chunk(v1, g + step);
    }
    for (const int blks = (chunks - 1 + phase) / kPer + 1; summed < blks && ok; ++summed) add_levels(summed);
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  ok = __syncthreads_and(ok ? 1 : 0) != 0;
  if (!ok && tid == 0) {
    atomicOr(err, kErrTimeout);
    atomicOr(flag, 8u);
  }
  if (warp == 0)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(kGCols) : "memory");
  if (warp < kGWarps && ok && i0 + ci < n) {
    const int64_t i = i0 + ci;
    float2 *dst = part + (size_t)blockIdx.y * n * n + i;
#pragma unroll 4
    for (int q = 0; q < 32; ++q) {
      const int64_t j = j0 + hi * 32 + q;
      if (j <= i) dst[j * n] = sums[q * kGT];
    }
  }
}

// S from the ranges' upper triangles, in order, both triangles (normalised pairs)
__global__ void qg_reduce_kernel(const float2 *__restrict__ part, int ranges, int64_t n, float2 *__restrict__ S) {
  const int64_t nn = n * n;
  for (int64_t q = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; q < nn; q += (int64_t)gridDim.x * blockDim.x) {
    const int64_t i = q / n, j = q % n;
    if (j < i) continue;
    DF t;
    int z = 0;
    for (; z + 8 <= ranges; z += 8) {
      float2 v[8];
#pragma unroll
      for (int u = 0; u < 8; ++u) v[u] = __ldcg(part + (int64_t)(z + u) * nn + q);
#pragma unroll
      for (int u = 0; u < 8; ++u) {
        DF x;
        x.hi = v[u].x;
        x.lo = v[u].y;
        df_add(t, x);
      }
    }
    for (; z < ranges; ++z) {
      const float2 v = __ldcg(part + (int64_t)z * nn + q);
      DF x;
      x.hi = v.x;
      x.lo = v.y;
      df_add(t, x);
    }
    S[q] = make_float2(t.hi, t.lo);
    S[j * n + i] = make_float2(t.hi, t.lo);
  }
}

// a b for double-float pairs, normalised
__device__ __forceinline__ DF df_mul(DF a, DF b) {
  const float p = a.hi * b.hi;
  const float e = fmaf(a.hi, b.hi, -p) + fmaf(a.hi, b.lo, a.lo * b.hi);
  DF r;
  r.hi = p + e;
  r.lo = e - (r.hi - p);
  return r;
}
// 1 / sqrt(d): one step of Newton's iteration, y + y (1 - d y^2) / 2, from the FP32 value y,
// with the residual in double-float (square roots and divisions in FP64 take 600 cycles each)
__device__ __forceinline__ DF df_rsqrt(DF d) {
  const float y = rsqrtf(d.hi);
  DF yy;
  yy.hi = y * y;
  yy.lo = fmaf(y, y, -yy.hi);
  const DF p = df_mul(d, yy);
  const float r = (1.f - p.hi) - p.lo;
  const float c = 0.5f * y * fmaf(0.75f * r, r, r);  // (the next term of the series too)
  DF o;
  o.hi = y + c;
  o.lo = c - (o.hi - y);
  return o;
}

// the largest (kh, kl) of a warp and the lowest id with it, in every lane
__device__ __forceinline__ void qg_warp_max(uint32_t &kh, uint32_t &kl, uint32_t &id) {
  const uint32_t h = __reduce_max_sync(0xffffffffu, kh);
  const uint32_t l = __reduce_max_sync(0xffffffffu, kh == h ? kl : 0u);
  id = __reduce_min_sync(0xffffffffu, kh == h && kl == l ? id : 0x7fffffffu);
  kh = h, kl = l;
}

// Pivoted Cholesky of S, k steps, one thread per column (one block), in double-float.
//   r_c = (S[p, c] - sum_l r_lp r_lc) / r_p,  d_c -= r_c^2,  and in FP32 the coefficients w of column c in the
//   pivot columns so far (S_11 w = S_1c): w_j = r_c / r_p, w_l -= w_j w_l(p)
// With an error of at most eps |a_i| |a_j| in every entry of S, that of a remaining norm (a Schur
// complement) is at most eps (|a_c| + sum_l |w_l| |a_l|)^2 to first order.  The pivot has to
// exceed every other norm by more than both errors, and its own error 64 times.
__global__ void __launch_bounds__(kMaxN) qg_pivot_kernel(const float2 *__restrict__ S, int n, int k,
                                                         float eps,
                                                         int *__restrict__ piv, float2 *__restrict__ M,
                                                         uint32_t *flag) {
  extern __shared__ float2 qg_r[];  // [k][n] rows of R
  __shared__ uint32_t s_kh[kMaxN / 32], s_kl[kMaxN / 32], s_idx[kMaxN / 32];
  __shared__ float2 s_inv, s_dp;
  __shared__ float s_pe, s_pn;          // of the pivot: the error of its norm, |a_p|
  __shared__ float s_w[kMaxK];          // its coefficients
  __shared__ float s_na[kMaxK];         // |a_l| of the pivots
  __shared__ float2 s_M[kMaxK];  // a row of R_1^-1
  __shared__ float2 s_iv[kMaxK];  // 1 / R[j][p_j]
  __shared__ int s_piv[kMaxK];
  const int c = threadIdx.x, lane = c & 31, warp = c >> 5, nw = (int)blockDim.x / 32;
  if (*flag) return;
  const bool mine = c < n;
  bool done = !mine, uncertain = false;
  DF d;
  if (mine) {
    const float2 v = __ldcg(S + (size_t)c * n + c);
    d.hi = v.x;
    d.lo = v.y;
  }
  // (a norm whose products leave FP32's normal range, or that is not a number, decides nothing)
  if (!(d.hi < 0x1p100f) || (d.hi > 0.f && d.hi < 0x1p-96f)) uncertain = true;
  const float na = sqrtf(fmaxf(d.hi, 0.f));
  float w[kMaxK], wsum = na;  // wsum = |a_c| + sum |w_l| |a_l|
#pragma unroll
  for (int l = 0; l < kMaxK; ++l) w[l] = 0.f;
#pragma unroll 1
  for (int j = 0; j < k; ++j) {
    // largest remaining norm (lowest column on ties, which are uncertain anyway): pairs ordered as
    // integers, one word after the other; over the warps' results again by every warp
    const bool live = !done && d.hi > 0.f;
    const uint32_t lo = __float_as_uint(d.lo);
    uint32_t kh = live ? __float_as_uint(d.hi) : 0u, kl = lo & 0x80000000u ? ~lo : lo | 0x80000000u, id = live ? c : INT_MAX;
    qg_warp_max(kh, kl, id);
    if (lane == 0) s_kh[warp] = kh, s_kl[warp] = kl, s_idx[warp] = id;
    __syncthreads();
    kh = lane < nw ? s_kh[lane] : 0u, kl = lane < nw ? s_kl[lane] : 0u, id = lane < nw ? s_idx[lane] : INT_MAX;
    qg_warp_max(kh, kl, id);
    const int p = (int)id;
    if (p >= n) {  // nothing left (the same in every thread)
      uncertain = true;
      break;
    }
    DF t, row;  // (the row of S arrives while the products of the earlier rows are taken off)
    if (mine) {
      const float2 v = __ldcg(S + (size_t)p * n + c);
      row.hi = v.x;
      row.lo = v.y;
    }
    const float e = eps * wsum * wsum;
    if (c == p) {
      const DF inv = df_rsqrt(d);
      s_inv = make_float2(inv.hi, inv.lo);
      s_dp = make_float2(d.hi, d.lo);
      s_pe = e;
      s_pn = na;
      s_na[j] = na;
      s_piv[j] = p;
#pragma unroll
      for (int l = 0; l < kMaxK; ++l) s_w[l] = w[l];
      uncertain = uncertain || !(d.hi > 64.f * e);
      done = true;
    }
    if (mine) {
#pragma unroll 4
      for (int l = 0; l < j; ++l) df_sub_prod(t, qg_r[l * n + p], qg_r[l * n + c]);
      df_add(t, row);
    }
    __syncthreads();
    DF inv, dp;
    inv.hi = s_inv.x;
    inv.lo = s_inv.y;
    dp.hi = s_dp.x;
    dp.lo = s_dp.y;
    if (!done) uncertain = uncertain || !((dp.hi - d.hi) + (dp.lo - d.lo) > e + s_pe);
    if (mine) {
      const DF r = df_mul(t, inv);
      qg_r[j * n + c] = make_float2(r.hi, r.lo);
      df_sub_prod(d, make_float2(r.hi, r.lo), make_float2(r.hi, r.lo));
      const float dn = d.hi + d.lo;
      d.lo = d.lo - (dn - d.hi);
      d.hi = dn;
      const float wj = r.hi * inv.hi;
      wsum = fmaf(fabsf(wj), s_pn, na);
#pragma unroll
      for (int l = 0; l < kMaxK; ++l) {
        if (l < j) {
          w[l] = fmaf(-wj, s_w[l], w[l]);
          wsum = fmaf(fabsf(w[l]), s_na[l], wsum);
        } else if (l == j) {
          w[l] = wj;
        }
      }
    }
    if (c == p) s_iv[j] = s_inv;
    __syncthreads();
  }
  if (__syncthreads_or(uncertain ? 1 : 0)) {
    if (c == 0) atomicOr(flag, 2u);
    return;
  }
  // R_1^-1 by rows from the last one up, a thread per entry: row i is done, then leaves the rows above
  const int ri = c / kMaxK, rc = c % kMaxK;
  const bool in = c < kMaxK * kMaxK && ri < k && rc < k && ri <= rc;
  DF x;
  if (in && ri == rc) x.hi = 1.f;
#pragma unroll 1
  for (int i = k - 1; i >= 0; --i) {
    if (in && ri == i) {
      DF iv, xn;
      iv.hi = s_iv[i].x;
      iv.lo = s_iv[i].y;
      xn.hi = x.hi + x.lo;
      xn.lo = x.lo - (xn.hi - x.hi);
      x = df_mul(xn, iv);
      s_M[rc] = make_float2(x.hi, x.lo);
    }
    __syncthreads();
    if (in && ri < i && rc >= i) df_sub_prod(x, qg_r[ri * n + s_piv[i]], s_M[rc]);
    __syncthreads();
  }
  if (c < kMaxK * kMaxK && ri < k && rc < k) M[ri * k + rc] = make_float2(x.hi, x.lo);  // (zero below the diagonal)
  if (c < k) piv[c] = s_piv[c];
}

// Entry (row, c) of A_p M, the row's 16 threads holding one entry of A_p each (a; zero past k), M's
// column c as pairs (zero past the diagonal) in mc.  All lanes of a warp call.
__device__ __forceinline__ DF qg_entry(float a, const float2 (&mc)[kMaxK]) {
  DF t;
#pragma unroll
  for (int l = 0; l < kMaxK; ++l) df_fma(t, __shfl_sync(0xffffffffu, a, l, kMaxK), mc[l].x, mc[l].y);
  return t;
}

// E + I = Q_1^T Q_1 (upper triangle): per block, 128 rows at a time, the entries of Q_1 into
// shared memory (16 threads a row), then one thread per entry of E and half of the rows adds the
// products; the last block adds the blocks' sums in order and finishes (see the top).
constexpr int kOT = 512, kORows = 128;
__global__ void __launch_bounds__(kOT) qg_ortho_kernel(const float *__restrict__ A, int64_t m, int64_t lda, int k,
                                                       const int *__restrict__ piv, const float2 *__restrict__ M1,
                                                       float2 *__restrict__ Q1, float2 *__restrict__ part,
                                                       unsigned *counter,
                                                       float2 *__restrict__ Wout, uint32_t *flag) {
  __shared__ float2 Ms[kMaxK][kMaxK];
  __shared__ int ps[kMaxK];
  __shared__ float2 qs[kMaxK][kORows + 1];
  __shared__ float2 red[kOT];
  __shared__ bool last;
  __shared__ float2 E[kMaxK][kMaxK + 1], W[kMaxK][kMaxK + 1], top[kMaxK][kMaxK + 1];
  __shared__ float T[kMaxK][kMaxK + 1], sgn[kMaxK];
  __shared__ double T64[kMaxK][kMaxK + 1];
  if (*flag) return;  // (written by earlier kernels only, until the last block below)
  const int tid = threadIdx.x;
  const int ne = k * (k + 1) / 2;  // entries (c1 <= c2)
  for (int q = tid; q < k * k; q += kOT) Ms[q / k][q % k] = M1[q];
  if (tid < k) ps[tid] = piv[tid];
  const int H = max(1, min(kOT / ne, 8));  // row lanes per entry
  const int e = tid % ne, h = tid / ne;
  int c1 = 0, c2 = e;
  while (c2 >= k - c1) c2 -= k - c1, ++c1;
  c2 += c1;
  DF s;
  __syncthreads();
  float2 mc[kMaxK];  // column tid % 16 of R_1^-1
#pragma unroll
  for (int l = 0; l < kMaxK; ++l)
    mc[l] = (l < k && tid % kMaxK < k) ? Ms[l][tid % kMaxK] : make_float2(0.f, 0.f);
  constexpr int kOP = kORows * kMaxK / kOT;  // entries of a pass per thread: row tid / 16 + 32 u, column c
  const int64_t stride = (int64_t)gridDim.x * kORows;
  const int c = tid % kMaxK;
  float a[kOP];
  auto load = [&](int64_t r0) {
#pragma unroll
    for (int u = 0; u < kOP; ++u) {
      const int64_t r = r0 + tid / kMaxK + u * (kOT / kMaxK);
      a[u] = (c < k && r < m) ? __ldg(A + r * lda + ps[c]) : 0.f;
    }
  };
  load((int64_t)blockIdx.x * kORows);
  for (int64_t r0 = (int64_t)blockIdx.x * kORows; r0 < m; r0 += stride) {
    const int nr = (int)min((int64_t)kORows, m - r0);
    float b[kOP];
#pragma unroll
    for (int u = 0; u < kOP; ++u) b[u] = a[u];
    load(r0 + stride);
#pragma unroll
    for (int u = 0; u < kOP; ++u) {
      const int r = tid / kMaxK + u * (kOT / kMaxK);
      const DF q = qg_entry(b[u], mc);
      const float hi = q.hi + q.lo;
      const float2 v = make_float2(hi, q.lo - (hi - q.hi));
      qs[c][r] = v;
      if (c < k && r < nr) Q1[(r0 + r) * k + c] = v;
    }
    __syncthreads();
    if (h < H) {
      for (int r = h; r < nr; r += 4 * H) {
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          if (r + u * H >= nr) break;
          const float2 x = qs[c1][r + u * H], y = qs[c2][r + u * H];
          df_fma(s, x.x, y.x, y.y);
          s.lo = fmaf(x.y, y.x, s.lo);
        }
        const float t = s.hi + s.lo;  // (a low part that grows rounds more: Q orthonormal to 5e-14 only)
        s.lo -= t - s.hi;
        s.hi = t;
      }
    }
    __syncthreads();
  }
  auto lanes = [&](DF v) {  // sum of an entry's row lanes, in the first (all threads call)
    red[tid] = make_float2(v.hi, v.lo);
    __syncthreads();
    if (tid < ne)
      for (int g = 1; g < H; ++g) {
        DF x;
        x.hi = red[g * ne + tid].x;
        x.lo = red[g * ne + tid].y;
        df_add(v, x);
      }
    __syncthreads();
    return v;
  };
  s = lanes(s);
  if (tid < ne) part[(size_t)blockIdx.x * ne + tid] = make_float2(s.hi, s.lo);
  __threadfence();
  __syncthreads();
  if (tid == 0) last = atomicAdd(counter, 1u) == gridDim.x - 1u;
  __syncthreads();
  if (!last) return;
  __threadfence();
  if (tid == 0) *counter = 0u;
  // ---- the last block: E, then the factors that make Q_1 orthonormal
  const int i = tid / k, l = tid % k;
  const bool in = tid < k * k;
  if (in) top[i][l] = __ldcg(Q1 + i * k + l);
  DF t;
  if (h < H) {
    const int nb = (int)gridDim.x, b0 = (int)((int64_t)nb * h / H), b1 = (int)((int64_t)nb * (h + 1) / H);
    int b = b0;
    for (; b + 16 <= b1; b += 16) {
      float2 v[16];
#pragma unroll
      for (int u = 0; u < 16; ++u) v[u] = __ldcg(part + (size_t)(b + u) * ne + e);
#pragma unroll
      for (int u = 0; u < 16; ++u) {
        DF x;
        x.hi = v[u].x;
        x.lo = v[u].y;
        df_add(t, x);
      }
    }
    for (; b < b1; ++b) {
      const float2 v = __ldcg(part + (size_t)b * ne + e);
      DF x;
      x.hi = v.x;
      x.lo = v.y;
      df_add(t, x);
    }
  }
  t = lanes(t);
  bool big = false;
  if (tid < ne) {  // less the identity (exact: the high part is near one there, or small)
    if (c1 == c2) t.hi -= 1.f;
    const float hi = t.hi + t.lo;
    const float2 v = make_float2(hi, t.lo - (hi - t.hi));
    big = !(fabsf(hi) < 4e-6f);
    E[c1][c2] = E[c2][c1] = v;
  }
  if (__syncthreads_or(big ? 1 : 0)) {
    if (tid == 0) atomicOr(flag, 4u);
    return;
  }
  // R_2 = I + U_1 + U_2 with U_1 = up(E), U_2 = -up(U_1^T U_1) (up: the strict upper triangle and
  // half of the diagonal); W = R_2^-1 = I - U_1 - U_2 + U_1^2, to E^3.  The squares are below 1e-9
  // and need no more than FP32.
  if (in) T[i][l] = i < l ? E[i][l].x : i == l ? 0.5f * E[i][i].x : 0.f;  // U_1
  __syncthreads();
  if (in) {
    float tt = 0.f, sq = 0.f;
#pragma unroll 4
    for (int a = 0; a < k; ++a) {
      tt = fmaf(T[a][i], T[a][l], tt);  // U_1^T U_1
      sq = fmaf(T[i][a], T[a][l], sq);  // U_1^2
    }
    DF v;  // upper triangle only
    if (i <= l) {
      const float f = i == l ? 0.5f : 1.f;
      v.hi = i == l ? 1.f : 0.f;
      df_add1(v, -f * E[i][l].x);
      v.lo += -f * E[i][l].y + (sq + f * tt);
      const float hi = v.hi + v.lo;
      v.lo -= hi - v.hi;
      v.hi = hi;
    }
    W[i][l] = make_float2(v.hi, v.lo);
  }
  __syncthreads();
  if (in) {  // top block of Q before the signs
    DF v;
    for (int a = 0; a <= l; ++a) {
      df_fma(v, top[i][a].x, W[a][l].x, W[a][l].y);
      v.lo = fmaf(top[i][a].y, W[a][l].x, v.lo);
    }
    T[i][l] = v.hi + v.lo;
    T64[i][l] = (double)v.hi + (double)v.lo;
  }
  __syncthreads();
  // (a sign within FP32's error: again in FP64)
  if (qg_signs(T, k, i, l, in, sgn)) qg_signs(T64, k, i, l, in, sgn);
  if (in) Wout[i * k + l] = i <= l ? make_float2(W[i][l].x * sgn[l], W[i][l].y * sgn[l]) : make_float2(0.f, 0.f);
}

// Q = Q_1 W D, 16 threads a row, FP64 from double-float sums
__global__ void __launch_bounds__(256) qg_q_kernel(const float2 *__restrict__ Q1, int64_t m, int k,
                                                   const float2 *__restrict__ W, const uint32_t *flag,
                                                   double *__restrict__ Q, int64_t ldq) {
  if (*flag) return;
  const int c = threadIdx.x % kMaxK;
  float2 wc[kMaxK];
#pragma unroll
  for (int l = 0; l < kMaxK; ++l) wc[l] = (l < k && c < k) ? W[l * k + c] : make_float2(0.f, 0.f);
  const int64_t step = (int64_t)gridDim.x * (256 / kMaxK);
#pragma unroll 2
  for (int64_t r0 = (int64_t)blockIdx.x * (256 / kMaxK); r0 < m; r0 += step) {
    const int64_t r = r0 + threadIdx.x / kMaxK;
    const bool in = r < m && c < k;
    const float2 v = in ? __ldg(Q1 + r * k + c) : make_float2(0.f, 0.f);
    DF q;
#pragma unroll
    for (int l = 0; l < kMaxK; ++l) {
      df_fma(q, __shfl_sync(0xffffffffu, v.x, l, kMaxK), wc[l].x, wc[l].y);
      q.lo = fmaf(__shfl_sync(0xffffffffu, v.y, l, kMaxK), wc[l].x, q.lo);
    }
    if (in) Q[r * ldq + c] = f2d_exact(q.hi) + f2d_exact(q.lo);
  }
}

// Bound of the error of an entry of S over |a_i| |a_j|, whatever the entries and however their errors
// add up.  In a block of 256 rows let t be a column scaled so that its largest entry lies in
// [2^7, 2^8): its norm is at least 2^7, and its entries' sum at most 16 times its norm.  Over the
// product of two such norms:
//   slicing     an entry is rounded by 2^-25 at most: 2^-25 16 (|t_i| + |t_j|), 2^-27
//   left out    slices 2 x 3 and 3 x 3, 256 (2^-25 + 2^-34): 2^-31
//   levels 3, 4 the shared sum, below 2^-13 (|t_i| + |t_j|) + 0.51, is rounded 112 times by
//               2^-22 of it: 2^-30
//   blocks      the low part, at most 2^-7.8 of the product, is rounded when a level and when
//               the next block of a range is added to it: 2^-31 each
// The sums over blocks are below |a_i| |a_j| (Cauchy-Schwarz).  A column with one large entry
// beside equal small ones comes within a factor of 16 of the first term, and with 2^-33, an estimate
// for errors of either sign, near ties were decided wrongly there.  (156 unfoldings of 18 uniform
// and skewed tensors, three sweeps each: all decided, the nearest tie at 1.1 times what it needs.)
float qg_eps(int64_t rows_per) { return (1.5f + (float)(rows_per / kGBlock + 1) / 16.f) * 0x1p-27f; }

struct Plan {
  int tiles, ranges, oblocks;
  int64_t rows_per;
  size_t part, S, M, W, piv, opart, words, ex, q1, total;
  int64_t blocks;
};

// Six reflectors and more, four and five where the matrix is tall and narrow; up to 64 columns a
// reflector where it is tall and wide.  It takes 50 to 60 us for the smallest matrices and S grows
// with m n^2; the cluster form takes 8 us a reflector for the smallest and 22 us at 50,000 x 256:
//   m x n, k            here   cluster (us)        m x n, k             here   cluster
//   200 x 64, 4           58        52             200 x 64, 6            60        67
//   512 x 128, 4          59        53             512 x 128, 6           59        69
//   2,000 x 128, 4        63        67             6,000 x 256, 4         74        73
//   10,000 x 64, 5        70       151             6,000 x 256, 5         75        84
//   20,000 x 512, 5      174       138             4,000 x 512, 6         89       113
//   100 x 64, 8           61        82             4,000 x 512, 16       112       248
//   1,000 x 256, 16       83       186             50,000 x 256, 16      180       363
bool plan(int64_t m, int64_t n, int k, int num_sms, Plan *p) {
  if (k < 4 || k > kMaxK || n < k || n > kMaxN || m < n || m < 2 * k) return false;
  if (k < 6 && (m < 2000 || n > 128 * (k - 3))) return false;
  if (m > 4000 && n > 64 * k) return false;
  const int t = (int)((n + kGM - 1) / kGM);
  p->tiles = t * (t + 1) / 2;
  const int64_t blocks = (m + kGRows - 1) / kGRows;
  const int64_t want = std::max<int64_t>(1, num_sms / p->tiles);
  const int64_t per = (blocks + std::min(want, blocks) - 1) / std::min(want, blocks);
  p->rows_per = per * kGRows;
  p->ranges = (int)((m + p->rows_per - 1) / p->rows_per);
  p->oblocks = (int)std::min<int64_t>((m + kORows - 1) / kORows, num_sms);
  size_t o = 0;
  auto take = [&](size_t bytes) {
    const size_t r = o;
    o += (bytes + 255) / 256 * 256;
    return r;
  };
  p->words = take(256);  // flag, counter
  p->part = take(sizeof(float2) * (size_t)p->ranges * n * n);
  p->S = take(sizeof(float2) * (size_t)(n * n));
  p->M = take(sizeof(float2) * k * k);
  p->blocks = (m + kGBlock - 1) / kGBlock;
  p->ex = take((size_t)(p->blocks * n));
  p->q1 = take(sizeof(float2) * (size_t)(m * k));
  p->W = take(sizeof(float2) * k * k);
  p->piv = take(sizeof(int) * k);
  p->opart = take(sizeof(float2) * (size_t)p->oblocks * (k * (k + 1) / 2));
  p->total = o;
  return true;
}

}  // namespace

void qg_reduce(const float2 *part, int ranges, int64_t n, float2 *S, cudaStream_t s) {
  qg_reduce_kernel<<<(unsigned)std::min<int64_t>((n * n + 127) / 128, 2048), 128, 0, s>>>(part, ranges, n, S);
  count_launch();
}

cudaError_t qg_pivots(const float2 *S, int64_t n, int k, float eps, int *piv, float2 *M, uint32_t *flag,
                      cudaStream_t s) {
  cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
  cudaStreamIsCapturing(s, &cap);  // the attribute is set by the eager launches before any capture
  if (cap == cudaStreamCaptureStatusNone) {
    const cudaError_t e = cudaFuncSetAttribute(qg_pivot_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                               (int)(sizeof(float2) * kMaxK * kMaxN));
    if (e != cudaSuccess) return e;
  }
  const int threads = std::max(kMaxK * kMaxK, (int)((n + 31) / 32 * 32));
  qg_pivot_kernel<<<1, threads, sizeof(float2) * (size_t)k * n, s>>>(S, (int)n, k, eps, piv, M, flag);
  count_launch();
  return cudaSuccess;
}

size_t qrp_gram_bytes(int64_t m, int64_t n, int k, int num_sms) {
  Plan p;
  return plan(m, n, k, num_sms, &p) ? p.total : 0;
}

bool qrp_gram_takes(const float *, int64_t m, int64_t n, int k, const QrpWork *w, int num_sms) {
  Plan p;
  return w->gram_ws && plan(m, n, k, num_sms, &p) && p.total <= w->gram_bytes;
}

const uint32_t *qrp_gram(const float *A, int64_t m, int64_t n, int64_t lda, int k, double *Q, int64_t ldq, QrpWork *w,
                         int num_sms, cudaStream_t s, cudaError_t *err) {
  *err = cudaSuccess;
  Plan p;
  plan(m, n, k, num_sms, &p);
  char *ws = static_cast<char *>(w->gram_ws);
  uint32_t *words = reinterpret_cast<uint32_t *>(ws + p.words);
  float2 *part = reinterpret_cast<float2 *>(ws + p.part);
  float2 *S = reinterpret_cast<float2 *>(ws + p.S), *M = reinterpret_cast<float2 *>(ws + p.M);
  int8_t *ex = reinterpret_cast<int8_t *>(ws + p.ex);
  float2 *W = reinterpret_cast<float2 *>(ws + p.W), *opart = reinterpret_cast<float2 *>(ws + p.opart);
  int *piv = reinterpret_cast<int *>(ws + p.piv);
  float2 *Q1 = reinterpret_cast<float2 *>(ws + p.q1);
  cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
  cudaStreamIsCapturing(s, &cap);  // the attribute is set by the eager launches before any capture
  if (cap == cudaStreamCaptureStatusNone) {
    *err = cudaFuncSetAttribute(qg_gram_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)qg_smem_bytes());
    if (*err != cudaSuccess) return words;
  }
  if ((*err = cudaMemsetAsync(words, 0, 8, s)) != cudaSuccess) return words;
  qg_exp_kernel<<<dim3((unsigned)p.blocks, (unsigned)((n + 127) / 128)), 512, 0, s>>>(A, m, n, lda, ex, words);
  count_launch();
  qg_gram_kernel<<<dim3((unsigned)p.tiles, (unsigned)p.ranges), kGT + 32, qg_smem_bytes(), s>>>(
      A, m, n, lda, p.rows_per, ex, part, words, w->err_out);
  count_launch();
  qg_reduce(part, p.ranges, n, S, s);
  if ((*err = qg_pivots(S, n, k, qg_eps(p.rows_per), piv, M, words, s)) != cudaSuccess) return words;
  qg_ortho_kernel<<<p.oblocks, kOT, 0, s>>>(A, m, lda, k, piv, M, Q1, opart, words + 1, W, words);
  count_launch();
  qg_q_kernel<<<(unsigned)std::min<int64_t>((m + 15) / 16, 8 * (int64_t)num_sms), 256, 0, s>>>(Q1, m, k, W, words, Q,
                                                                                             ldq);
  count_launch();
  *err = cudaGetLastError();
  return words;
}

}  // namespace tk

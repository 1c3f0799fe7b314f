// K-d: core tensor of one HOOI sweep and the fit (Section III-B, eqs. ttm_ele and
// core_unfolded:  G_(N) = U_N^T Y_(N),  G[c, r] = sum_i U_N(i, r) Y_(N)(i, c)).
// Y_(N) is the FP32 TTMc output of the last mode (I_N x P), U_N the FP64 factor
// (I_N x R).  Two forms: on the tensor cores (core_tc_kernel, exact fixed-point slices,
// below) with a separate reduction of the row ranges (core_reduce_kernel), and an FP64
// SIMT form (core_kernel: split over rows of Y into chunks, each block owns a 16 x 16 tile
// of (column c, rank r) outputs for one row chunk and accumulates in FP64).  Both write G
// (C-order, r fastest), ||G||^2 and fit = 1 - sqrt(max(0, ||X||^2 - ||G||^2)) / ||X||,
// adding the row ranges' partials in a fixed order.
#include <algorithm>
#include <cstdlib>

#include "dfloat.cuh"
#include "internal.cuh"
#include "tc.cuh"

namespace tk {

constexpr int kCoreRows = 64;  // rows of Y per chunk staged at once

__global__ void __launch_bounds__(256) core_kernel(const float *Y, const double *U, int64_t I, int64_t P, int R,
                                                   int rows_per_chunk, double *part, unsigned *counter, double *G,
                                                   const double *norm_x2, double *norm_g2, double *fit) {
  __shared__ float ys[kCoreRows][17];
  __shared__ double us[kCoreRows][17];
  const int tc = threadIdx.x & 15, tr = threadIdx.x >> 4;
  const int64_t c = (int64_t)blockIdx.x * 16 + tc;
  const int r = blockIdx.y * 16 + tr;
  const int64_t i_begin = (int64_t)blockIdx.z * rows_per_chunk;
  const int64_t i_end = std::min<int64_t>(I, i_begin + rows_per_chunk);
  double acc = 0.0;
  for (int64_t i0 = i_begin; i0 < i_end; i0 += kCoreRows) {
    for (int q = threadIdx.x; q < kCoreRows * 16; q += blockDim.x) {
      const int ri = q / 16, cc = q % 16;
      const int64_t i = i0 + ri;
      const int64_t col = (int64_t)blockIdx.x * 16 + cc;
      const int rr = blockIdx.y * 16 + cc;
      ys[ri][cc] = (i < i_end && col < P) ? Y[i * P + col] : 0.f;
      us[ri][cc] = (i < i_end && rr < R) ? U[i * R + rr] : 0.0;
    }
    __syncthreads();
#pragma unroll 8
    for (int ri = 0; ri < kCoreRows; ++ri) acc = fma(us[ri][tr], (double)ys[ri][tc], acc);
    __syncthreads();
  }
  const int64_t PR = P * R;
  if (c < P && r < R) part[(int64_t)blockIdx.z * PR + c * R + r] = acc;

  // last block: reduce chunks, ||G||^2, fit
  __shared__ bool is_last;
  __threadfence();
  __syncthreads();
  if (threadIdx.x == 0) is_last = atomicAdd(counter, 1u) == gridDim.x * gridDim.y * gridDim.z - 1u;
  __syncthreads();
  if (!is_last) return;
  __threadfence();
  __shared__ double red[256];
  double g2 = 0.0;
  for (int64_t q = threadIdx.x; q < PR; q += blockDim.x) {
    double t = 0.0;
    for (int z = 0; z < (int)gridDim.z; ++z) t += __ldcg(part + (int64_t)z * PR + q);
    G[q] = t;
    g2 = fma(t, t, g2);
  }
  red[threadIdx.x] = g2;
  __syncthreads();
  for (int o = 128; o > 0; o >>= 1) {
    if (threadIdx.x < o) red[threadIdx.x] += red[threadIdx.x + o];
    __syncthreads();
  }
  if (threadIdx.x == 0) {
    const double gx = red[0];
    const double nx = *norm_x2;
    *norm_g2 = gx;
    *fit = (nx > 0.0) ? 1.0 - sqrt(fmax(0.0, nx - gx)) / sqrt(nx) : 1.0;
    *counter = 0u;
  }
}

// ---------------------------------------------------------------- tensor-core form
// The same G on the 5th-generation tensor cores: G as a P x R matrix is Y_(N)^T U_N, so one
// CTA computes a tile of 128 columns c of Y (the MMA's M) by all ranks r (N = R rounded up
// to 16) over a range of at most 128 rows i of Y (the K of the product), 16 rows at a time.
//
// Fixed-point slices (an Ozaki-type split): each column of Y over the CTA's rows, and each
// column of U_N (FP64), gets a shared power of two 2^E above its largest magnitude, and
// every value v is written as 2^(E-8) (m_0 + m_1 2^-8 + m_2 2^-16 + m_3 2^-24) with integer
// slices |m_0| <= 256, |m_s| <= 128 (rounded to nearest, remainders exact in FP64; the
// part below the last slice, under 2^(E-33), is dropped).  The slices are exact in BF16.
// For every pair of slices (a, b) one tcgen05.mma kind::f16 adds m_a(Y) m_b(U) over 16 rows
// into the FP32 tensor-memory accumulator of level a + b.  A product is at most 2^16, and a
// level's sum over at most 128 rows stays below 2^24, so every accumulator holds an exact
// integer: the FP32 accumulation never rounds, whatever the tensor core's rounding rule.
// At the end each level is read with tcgen05.ld and added into FP64 with its scale
// 2^(E_c + E_r - 16 - 8 level).  The result differs from the exact G of the FP32 Y and FP64
// U only by the dropped parts (relative ~2^-33 of the columns' largest entries) and the FP64
// additions of the levels and row ranges.  Operands are staged K-major in the no-swizzle
// canonical layout (8-row x 16-byte core matrices) in two buffers: the slices of chunk j + 1
// are written while the products of chunk j run.  The last CTA adds the partials of every row
// range in order, as core_kernel does.
constexpr int kTcM = 128;   // columns of Y per tile (MMA M)
constexpr int kTcK = 16;    // rows of Y per staged chunk (one MMA of K = 16 per slice pair)
constexpr int kTcKC = kTcK * 2 / 16;  // core-matrix columns (16 bytes) along K per chunk
constexpr int kTcRows = 128;  // rows of Y per CTA at most: keeps every level sum below 2^24
constexpr int kTcSlices = 4;  // 8-bit slices per value
constexpr int kTcLevels = 5;  // slice pairs a + b <= 4 (the three pairs above add under 2^-40 of a product)

__host__ __device__ constexpr uint32_t tc_tmem_cols(int np) {
  uint32_t c = 32;
  while (c < (uint32_t)(kTcLevels * np)) c <<= 1;
  return c;
}
__host__ __device__ constexpr size_t tc_rows_bytes(int rows, int np) {  // the CTA's rows of Y and U_N
  return ((size_t)rows * kTcM * 4 + (size_t)rows * np * 8 + 127) / 128 * 128;
}
__host__ __device__ constexpr size_t tc_smem_bytes(int rows, int np) {
  return tc_rows_bytes(rows, np) + (size_t)2 * kTcSlices * (kTcM + np) * kTcK * 2 + 128;  // + two slice buffers
}

// The four integer slices of an FP32 y against 2^e (|y| < 2^e; 2^(8 - e) = sc1 sc2, two
// factors so that neither overflows when the column holds only subnormal values), each
// exact in BF16.  FP32 arithmetic, all exact: t = y 2^(8 - e) has at most 24 significant
// bits below 2^8, and |t - rint(t)| <= 1/2 keeps its bits.
__device__ __forceinline__ void slices_f32(float y, float sc1, float sc2, __nv_bfloat16 *out, int stride) {
  float t = (y * sc1) * sc2;
#pragma unroll
  for (int q = 0; q < kTcSlices; ++q) {
    const float m = rintf(t);
    out[q * stride] = __float2bfloat16_rn(m);
    t = (t - m) * 256.0f;
  }
}
// The four slices of an FP64 u against 2^e (|u| < 2^e): x = u 2^(32 - e) rounded to the
// nearest integer (ties to even), |x| <= 2^32, in balanced base-256 digits
// x = m_0 2^24 + m_1 2^16 + m_2 2^8 + m_3 with |m_s| <= 128 for s >= 1, hence |m_0| <= 256.
// Integer arithmetic on the bits of u (the FP64 pipe is narrow on this part).
__device__ __forceinline__ void slices_f64(double u, int e, __nv_bfloat16 *out, int stride) {
  const unsigned long long bits = (unsigned long long)__double_as_longlong(u);
  const int ex = (int)((bits >> 52) & 0x7ff);
  unsigned long long mant = bits & 0xFFFFFFFFFFFFFull;
  int sh;  // u = mant 2^(ex - 1075) with the hidden bit; x = u 2^(32 - e) = mant 2^-sh
  if (ex == 0) {
    sh = 1042 + e;  // subnormal: u = mant 2^-1074
  } else {
    mant |= 1ull << 52;
    sh = 1043 + e - ex;
  }
  unsigned long long qv = 0;  // sh >= 21 since |u| < 2^e; above 63 the value rounds to 0
  if (sh < 64) {
    const unsigned long long half = 1ull << (sh - 1), rem = mant & ((1ull << sh) - 1ull);
    qv = mant >> sh;
    if (rem > half || (rem == half && (qv & 1ull))) ++qv;
  }
  long long x = (bits >> 63) ? -(long long)qv : (long long)qv;
  int m[kTcSlices];
#pragma unroll
  for (int q = kTcSlices - 1; q > 0; --q) {
    const int d = (int)(((x + 128) & 255) - 128);
    m[q] = d;
    x = (x - d) >> 8;
  }
  m[0] = (int)x;
#pragma unroll
  for (int q = 0; q < kTcSlices; ++q) out[q * stride] = __int2bfloat16_rn(m[q]);
}
// exponent e with |x| < 2^e of a finite FP64 magnitude given by its bits, as above_exp_f32
__device__ __forceinline__ int above_exp_f64(unsigned long long b) {
  const int ef = (int)(b >> 52);
  if (ef) return ef - 1022;
  return b ? -1074 + 64 - __clzll((long long)b) : 0;
}
// 2^k as a double for -1022 <= k <= 1023 (built from its bits)
__device__ __forceinline__ double pow2d(int k) { return __longlong_as_double((long long)(1023 + k) << 52); }
// element (row, k) of a K-major 16-bit operand tile with kTcKC core columns per 8-row group
__device__ __forceinline__ int kmaj16(int row, int k) {
  return ((row >> 3) * kTcKC + (k >> 3)) * 64 + (row & 7) * 8 + (k & 7);
}
template <int NP>  // N of the MMA: R rounded up to 16
__global__ void __launch_bounds__(128) core_tc_kernel(const float *Y, const double *U, int64_t I, int64_t P, int R,
                                                      int rows_per_split, double *part, uint32_t *err) {
  static_assert(NP % 16 == 0 && NP >= 16 && NP <= 64, "N of the MMA");
  constexpr uint32_t kCols = tc_tmem_cols(NP);  // tensor-memory columns: kTcLevels accumulators of NP
  constexpr int kASlice = kTcM * kTcK, kBSlice = NP * kTcK;  // BF16 elements per slice tile
  extern __shared__ unsigned char tc_raw[];
  unsigned char *base = reinterpret_cast<unsigned char *>(
      (reinterpret_cast<uintptr_t>(tc_raw) + 127) & ~static_cast<uintptr_t>(127));
  const int rcap = rows_per_split;  // a multiple of kTcK, at most kTcRows
  float *sY = reinterpret_cast<float *>(base);                              // [rcap][kTcM]
  double *sU = reinterpret_cast<double *>(base + (size_t)rcap * kTcM * 4);  // [rcap][NP]
  __nv_bfloat16 *sA = reinterpret_cast<__nv_bfloat16 *>(base + tc_rows_bytes(rcap, NP));
  __nv_bfloat16 *sB = sA + 2 * kTcSlices * kASlice;  // sA: [2][kTcSlices][kASlice], sB: [2][kTcSlices][kBSlice]
  __shared__ __align__(8) unsigned long long bar[2];
  __shared__ uint32_t tbase;
  __shared__ int s_ok;
  __shared__ int s_eu[NP];
  const int tid = threadIdx.x, warp = tid >> 5;
  const int64_t c0 = (int64_t)blockIdx.x * kTcM;
  const int64_t i_begin = (int64_t)blockIdx.y * rows_per_split;
  const int64_t i_end = min(I, i_begin + rows_per_split);
  uint32_t sb[2];
  sb[0] = (uint32_t)__cvta_generic_to_shared(&bar[0]);
  sb[1] = (uint32_t)__cvta_generic_to_shared(&bar[1]);
  if (tid == 0) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(sb[0]) : "memory");
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(sb[1]) : "memory");
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    s_ok = 1;
  }
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                     (uint32_t)__cvta_generic_to_shared(&tbase)),
                 "r"(kCols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  // the CTA's rows of Y (thread t: column c0 + t) and of U_N into shared memory, loads in flight
  // together; then the shared exponents of the columns
  const int64_t c = c0 + tid;
  const int nrows = (int)(i_end - i_begin);
#pragma unroll 16
  for (int i = 0; i < rcap; ++i)
    sY[i * kTcM + tid] = (i < nrows && c < P) ? __ldg(Y + (i_begin + i) * P + c) : 0.f;
  for (int q = tid; q < rcap * NP; q += 128) {
    const int i = q / NP, n = q % NP;
    sU[q] = (i < nrows && n < R) ? __ldg(U + (i_begin + i) * R + n) : 0.0;
  }
  __syncthreads();
  // (the magnitudes of finite values order like their bit patterns without the sign)
  uint32_t ybits = 0;
  for (int i = 0; i < nrows; ++i) ybits = max(ybits, __float_as_uint(sY[i * kTcM + tid]) & 0x7fffffffu);
  const int ec = above_exp_f32(ybits);
  const int ysh = 8 - ec, ysh1 = min(ysh, 120);
  const float ysc1 = __int_as_float((127 + ysh1) << 23), ysc2 = __int_as_float((127 + ysh - ysh1) << 23);
  for (int n = tid; n < NP; n += 128) {
    unsigned long long ub = 0;
    for (int i = 0; i < nrows; ++i)
      ub = max(ub, (unsigned long long)__double_as_longlong(sU[i * NP + n]) & 0x7FFFFFFFFFFFFFFFull);
    s_eu[n] = above_exp_f64(ub);
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem = tbase;
  // D f32, A and B bf16, both K-major, N >> 3, M >> 4
  const uint32_t idesc = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(NP >> 3) << 17) | ((uint32_t)(kTcM >> 4) << 24);
  const uint32_t lbo = 128, sbo = kTcKC * 128;  // K-adjacent core matrices, 8-row groups
  const uint32_t aS = (uint32_t)__cvta_generic_to_shared(sA), bS = (uint32_t)__cvta_generic_to_shared(sB);
  const int nchunks = (int)((i_end - i_begin + kTcK - 1) / kTcK);
  bool ok = true;
  int issued = 0;  // chunks whose products were issued
  for (int j = 0; j < nchunks && ok; ++j) {
    const int b = j & 1;
    if (j >= 2) ok = tc_wait(sb[b], (uint32_t)(((j >> 1) - 1) & 1));  // the products that read this buffer
    ok = __syncthreads_and(ok ? 1 : 0) != 0;
    if (!ok) break;
    __nv_bfloat16 *a = sA + (size_t)b * kTcSlices * kASlice;
    __nv_bfloat16 *bb = sB + (size_t)b * kTcSlices * kBSlice;
#pragma unroll 4
    for (int k = 0; k < kTcK; ++k)
      slices_f32(sY[(j * kTcK + k) * kTcM + tid], ysc1, ysc2, a + kmaj16(tid, k), kASlice);
    for (int q = tid; q < NP * kTcK; q += 128) {
      const int n = q % NP, k = q / NP;
      slices_f64(sU[(j * kTcK + k) * NP + n], s_eu[n], bb + kmaj16(n, k), kBSlice);
    }
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    if (tid == 0) {
      const uint32_t aB = aS + (uint32_t)(b * kTcSlices * kASlice * 2), bB = bS + (uint32_t)(b * kTcSlices * kBSlice * 2);
#pragma unroll
      for (int L = 0; L < kTcLevels; ++L) {
        const int s0 = L < kTcSlices ? 0 : L - (kTcSlices - 1);
        const int s1 = L < kTcSlices ? L : kTcSlices - 1;  // pairs (a, L - a), both below kTcSlices
        for (int sa = s0; sa <= s1; ++sa) {
          const int sbk = L - sa;
          const uint64_t ad = umma_desc(aB + (uint32_t)(sa * kASlice * 2), lbo, sbo);
          const uint64_t bd = umma_desc(bB + (uint32_t)(sbk * kBSlice * 2), lbo, sbo);
          const uint32_t acc = (j > 0 || sa != s0) ? 1u : 0u;
          asm volatile(
              "{ .reg .pred p; setp.ne.u32 p, %4, 0; tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p; }" ::"r"(
                  tmem + (uint32_t)(L * NP)),
              "l"(ad), "l"(bd), "r"(idesc), "r"(acc)
              : "memory");
        }
      }
      asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(sb[b])
                   : "memory");
    }
    issued = j + 1;
  }
  // the last products of both buffers (bounded; on a give-up the products still in flight get
  // the same bounded time to end before the memory is freed)
  if (tid == 0) {
    bool done = ok;
    for (int b = 0; b < 2; ++b) {
      const int jl = (issued - 1 - b) >= 0 ? ((issued - 1 - b) & ~1) + b : -1;  // last chunk issued in buffer b
      if (jl >= 0) done = tc_wait(sb[b], (uint32_t)((jl >> 1) & 1)) && done;
    }
    if (!done) {
      atomicOr(err, kErrTimeout);
      s_ok = 0;
    }
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  // the levels are exact integers below 2^24: X = sum_L A_L 2^(8 (4 - L)) is exact in 64 bits;
  // then one conversion and one scaling by 2^(E_c + E_r - 16 - 32) (two factors: no overflow)
  long long accx[NP];
#pragma unroll
  for (int q = 0; q < NP; ++q) accx[q] = 0;
  if (s_ok && nchunks > 0) {
#pragma unroll
    for (int L = 0; L < kTcLevels; ++L)
#pragma unroll
      for (int n0 = 0; n0 < NP; n0 += 16) {
        uint32_t v[16];
        const uint32_t taddr = tmem + ((uint32_t)(warp * 32) << 16) + (uint32_t)(L * NP + n0);
        asm volatile(
            "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
            : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]),
              "=r"(v[8]), "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]), "=r"(v[14]), "=r"(v[15])
            : "r"(taddr));
        asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
        for (int q = 0; q < 16; ++q)
          accx[n0 + q] += (long long)__float2int_rn(__uint_as_float(v[q])) << (8 * (kTcLevels - 1 - L));
      }
  }
  double accd[NP];
#pragma unroll
  for (int q = 0; q < NP; ++q) {
    const int sh = ec + s_eu[q] - 16 - 8 * (kTcLevels - 1);
    const int sh1 = min(max(sh, -1000), 1000);  // two exact factors when |sh| is out of range
    accd[q] = ((double)accx[q] * pow2d(sh1)) * pow2d(sh - sh1);
  }
  // warp w holds tensor-memory lanes 32w .. 32w + 31 = columns c0 + 32w + lane (= c: tid)
  const int64_t PR = P * R;
  if (c < P)
#pragma unroll
    for (int q = 0; q < NP; ++q)
      if (q < R) part[(int64_t)blockIdx.y * PR + c * R + q] = s_ok ? accd[q] : __longlong_as_double(0x7ff8000000000000ll);
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  if (warp == 0) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(kCols) : "memory");
}

// G[q] = the partials of every row range added in order (q = c R + r), ||G||^2 from per-block
// sums added by the last block in a fixed tree order, and the fit.
constexpr int kRedT = 64;
__global__ void __launch_bounds__(kRedT) core_reduce_kernel(const double *part, int nz, int64_t PR, double *G,
                                                           double *bsum, unsigned *counter, const double *norm_x2,
                                                           double *norm_g2, double *fit) {
  __shared__ double red[kRedT];
  __shared__ bool is_last;
  const int64_t q = (int64_t)blockIdx.x * kRedT + threadIdx.x;
  double g2 = 0.0;
  if (q < PR) {
    double t = 0.0;
    int z = 0;
    for (; z + 8 <= nz; z += 8) {  // eight loads in flight, added in order
      double v[8];
#pragma unroll
      for (int u = 0; u < 8; ++u) v[u] = __ldcg(part + (int64_t)(z + u) * PR + q);
#pragma unroll
      for (int u = 0; u < 8; ++u) t += v[u];
    }
    for (; z < nz; ++z) t += __ldcg(part + (int64_t)z * PR + q);
    G[q] = t;
    g2 = t * t;
  }
  red[threadIdx.x] = g2;
  __syncthreads();
  for (int o = kRedT / 2; o > 0; o >>= 1) {
    if (threadIdx.x < o) red[threadIdx.x] += red[threadIdx.x + o];
    __syncthreads();
  }
  if (threadIdx.x == 0) {
    bsum[blockIdx.x] = red[0];
    __threadfence();
    is_last = atomicAdd(counter, 1u) == gridDim.x - 1u;
  }
  __syncthreads();
  if (!is_last) return;
  __threadfence();
  double gb = 0.0;  // block sums b = t, t + kRedT, ... then a tree over the threads
  for (unsigned b = threadIdx.x; b < gridDim.x; b += kRedT) gb += __ldcg(bsum + b);
  red[threadIdx.x] = gb;
  __syncthreads();
  for (int o = kRedT / 2; o > 0; o >>= 1) {
    if (threadIdx.x < o) red[threadIdx.x] += red[threadIdx.x + o];
    __syncthreads();
  }
  if (threadIdx.x == 0) {
    const double gx = red[0];
    const double nx = *norm_x2;
    *norm_g2 = gx;
    *fit = (nx > 0.0) ? 1.0 - sqrt(fmax(0.0, nx - gx)) / sqrt(nx) : 1.0;
    *counter = 0u;
  }
}

static bool core_on_tensor_cores();

// ---------------------------------------------------------------- Gram matrix of fat unfoldings
// S = Y Y^T (m x m) of an FP32 m x n matrix (Section III-D, P_n > I_n): a 32 x 32 tile of S on and
// below the diagonal over a range of columns, a 2 x 2 piece a thread.  32 columns at a time, every
// row scaled by the power of two of its largest entry there (any magnitude of FP32 goes), exact
// products are added in double-float (2^-46 of |y_i| |y_j|) and these sums in FP64; both triangles
// are written, and the ranges added in order.
// The FP32 pipe bounds it (11 instructions a product, half of the products by symmetry).  The
// tensor cores on exact 8-bit slices (error 2^-33) took longer at every size, most of it in
// slicing and hand-overs: 200 x 256 32 -> 11 us with the sum of the ranges; with the QRP that
// follows 64 x 3,600 288 -> 191, 200 x 1,280 151 -> 104, 1,000 x 1,056 708 -> 652, 1,000 x 4,096
// 1,682 -> 1,599.
constexpr int kGramMaxRows = 1024;  // above, in FP64 (gram_f32): slower (1,100 x 2,048, with the QRP, 11.7 ms
                                    // for 0.94), but its error is 2^-53 for 2^-46
constexpr int kGramMaxRanges = 8;   // column ranges (partial sets)
constexpr int kGdT = 32, kGdK = 32, kGdLd = kGdK + 4;
__global__ void __launch_bounds__(256) gram_df_kernel(const float *__restrict__ Y, int m, int64_t n,
                                                      int64_t cols_per_range, double *__restrict__ out) {
  __shared__ __align__(16) float sa[kGdT][kGdLd], sb[kGdT][kGdLd];
  __shared__ int ea[kGdT], eb[kGdT];  // the rows' exponents
  int ti = 0, tj = (int)blockIdx.x;
  while (tj > ti) tj -= ++ti;
  const int i0 = ti * kGdT, j0 = tj * kGdT, tid = threadIdx.x;
  const int64_t c_begin = (int64_t)blockIdx.y * cols_per_range, c_end = min(n, c_begin + cols_per_range);
  const int ia = tid / 16, jb = tid % 16;  // rows ia, ia + 16 of the tile, columns jb, jb + 16
  constexpr int kU = kGdT * kGdK / 256;
  float va[kU], vb[kU];
  auto load = [&](int64_t c0) {
#pragma unroll
    for (int u = 0; u < kU; ++u) {
      const int r = tid / kGdK + u * (256 / kGdK);
      const int64_t c = c0 + tid % kGdK;
      va[u] = (c < c_end && i0 + r < m) ? __ldg(Y + (i0 + r) * n + c) : 0.f;
      vb[u] = (c < c_end && j0 + r < m) ? __ldg(Y + (j0 + r) * n + c) : 0.f;
    }
  };
  double sum[4] = {0.0, 0.0, 0.0, 0.0};
  load(c_begin);
  for (int64_t c0 = c_begin; c0 < c_end; c0 += kGdK) {
#pragma unroll
    for (int u = 0; u < kU; ++u) {
      const int r = tid / kGdK + u * (256 / kGdK);  // a warp holds a row
      auto scaled = [](float v, int *e) {
        *e = above_exp_f32(__reduce_max_sync(0xffffffffu, __float_as_uint(v) & 0x7fffffffu));
        const int h = *e / 2;
        return v * __int_as_float((127 - h) << 23) * __int_as_float((127 - (*e - h)) << 23);
      };
      int e0, e1;
      sa[r][tid % kGdK] = scaled(va[u], &e0);
      sb[r][tid % kGdK] = scaled(vb[u], &e1);
      if (tid % kGdK == 0) ea[r] = e0, eb[r] = e1;
    }
    __syncthreads();
    load(c0 + kGdK);
    DF acc[2][2];
#pragma unroll 2
    for (int q = 0; q < kGdK; q += 4) {
      float x[2][4], y[2][4];
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        *reinterpret_cast<float4 *>(x[h]) = *reinterpret_cast<const float4 *>(&sa[ia + 16 * h][q]);
        *reinterpret_cast<float4 *>(y[h]) = *reinterpret_cast<const float4 *>(&sb[jb + 16 * h][q]);
      }
#pragma unroll
      for (int t = 0; t < 4; ++t) {
        DF &s = acc[t >> 1][t & 1];
#pragma unroll
        for (int z = 0; z < 4; ++z) {
          const float a = x[t >> 1][z], b = y[t & 1][z], p = a * b, e = fmaf(a, b, -p);
          const float w = s.hi + p, bp = w - s.hi;
          s.lo += ((s.hi - (w - bp)) + (p - bp)) + e;
          s.hi = w;
        }
        const float w = s.hi + s.lo;
        s.lo -= w - s.hi;
        s.hi = w;
      }
    }
#pragma unroll
    for (int t = 0; t < 4; ++t) {
      const int e = ea[ia + 16 * (t >> 1)] + eb[jb + 16 * (t & 1)];
      auto shifted = [&](float f) {  // f 2^e (of an overflowed row: infinity or NaN as it is)
        if (f == 0.f || !isfinite(f)) return (double)f;
        return __longlong_as_double(__double_as_longlong(f2d_exact(f)) + ((long long)e << 52));
      };
      sum[t] += shifted(acc[t >> 1][t & 1].hi);
      sum[t] += shifted(acc[t >> 1][t & 1].lo);
    }
    __syncthreads();
  }
  double *dst = out + (size_t)blockIdx.y * m * m;
#pragma unroll
  for (int t = 0; t < 4; ++t) {
    const int i = i0 + ia + 16 * (t >> 1), j = j0 + jb + 16 * (t & 1);
    if (j <= i && i < m) dst[(int64_t)i * m + j] = dst[(int64_t)j * m + i] = sum[t];
  }
}

__global__ void gram_reduce_kernel(const double *part, int nr, int64_t mm, double *S) {
  for (int64_t q = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; q < mm; q += (int64_t)gridDim.x * blockDim.x) {
    double t = 0.0;
    for (int r = 0; r < nr; ++r) t += __ldcg(part + (int64_t)r * mm + q);
    S[q] = t;
  }
}

size_t gram_part_elems(int64_t m) {
  return (m > 0 && m <= kGramMaxRows) ? (size_t)kGramMaxRanges * (size_t)(m * m) : 0;
}

void launch_gram(Ctx *c, const float *Y, int64_t m, int64_t n, double *S, cudaStream_t s) {
  if (!core_on_tensor_cores() || !c->gram_part || m > kGramMaxRows || m < 1 || n < 1) {  // TUCKER_CORE_TC=0: FP64
    gram_f32(Y, m, n, S, s);
    return;
  }
  const int64_t t = (m + kGdT - 1) / kGdT, tiles = t * (t + 1) / 2;
  // column ranges: about four blocks an SM
  int64_t nr = std::max<int64_t>(1, std::min<int64_t>(4 * (int64_t)c->num_sms / tiles, kGramMaxRanges));
  const int64_t cpr = ((n + nr - 1) / nr + kGdK - 1) / kGdK * kGdK;
  nr = (n + cpr - 1) / cpr;
  gram_df_kernel<<<dim3((unsigned)tiles, (unsigned)nr), 256, 0, s>>>(Y, (int)m, n, cpr, nr > 1 ? c->gram_part : S);
  ::tk::count_launch();
  if (nr > 1) {
    const int64_t mm = m * m;
    gram_reduce_kernel<<<(unsigned)std::min<int64_t>((mm + 255) / 256, 4096), 256, 0, s>>>(c->gram_part, (int)nr, mm, S);
    ::tk::count_launch();
  }
}

// The core runs on the tensor cores (core_tc_kernel + core_reduce_kernel) where R <= 64 and
// the row ranges fit the partial buffer; TUCKER_CORE_TC=0 selects the FP64 SIMT form
// (core_kernel) instead.  Both agree to FP64 rounding: on the 1M-nonzero Zipf workload
// (fit 0.84) the fits of ten sweeps differ by at most 7e-10.
static bool core_on_tensor_cores() {
  const char *e = std::getenv("TUCKER_CORE_TC");
  return !(e && e[0] == '0');
}

static int core_chunks(int num_sms, int64_t I, int64_t P, int R) {
  const int64_t tiles = ((P + 15) / 16) * ((R + 15) / 16);
  int64_t z = std::max<int64_t>(1, (2 * (int64_t)num_sms) / std::max<int64_t>(tiles, 1));
  z = std::min<int64_t>(z, std::max<int64_t>(1, (I + kCoreRows - 1) / kCoreRows));
  return (int)z;
}

size_t core_part_elems(int num_sms, int64_t P, int R) {
  // enough for the largest chunk count any mode can ask for
  return (size_t)P * R * (size_t)std::max(1, 2 * num_sms);
}

static void launch_core_fp64(Ctx *c, const float *Y, const double *U, double *G, cudaStream_t s);

template <int NP>
static void launch_core_tc(Ctx *c, const float *Y, const double *U, int64_t I, int64_t P, int R, int rows, dim3 grid,
                           double *G, cudaStream_t s) {
  cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
  cudaStreamIsCapturing(s, &cap);  // the attribute is set by the eager launches before any capture
  if (cap == cudaStreamCaptureStatusNone)
    cudaFuncSetAttribute(core_tc_kernel<NP>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                         (int)tc_smem_bytes(kTcRows, NP));
  core_tc_kernel<NP><<<grid, 128, tc_smem_bytes(rows, NP), s>>>(Y, U, I, P, R, rows, c->core_part, c->d_err);
  ::tk::count_launch();
  const int64_t PR = P * R;
  double *bsum = c->core_part + (int64_t)(2 * c->num_sms - 1) * PR;  // after the largest partial set
  core_reduce_kernel<<<(unsigned)((PR + kRedT - 1) / kRedT), kRedT, 0, s>>>(
      c->core_part, (int)grid.y, PR, G, bsum, c->core_counter, c->norm_dev, c->norm_dev + 1, c->fit_dev);
  ::tk::count_launch();
}

void launch_core(Ctx *c, const float *Y, const double *U, double *G, cudaStream_t s) {
  const int N = c->N;
  const int64_t I = c->dims[N - 1];
  const int64_t P = c->mode[N - 1].P;
  const int R = c->ranks[N - 1];
  if (R <= 64 && I > 0 && core_on_tensor_cores()) {
    // tensor-core form: tiles of 128 columns; row ranges of 32 to 128 rows (whole chunks of
    // 16), as many as give about 2 x SMs CTAs; the partial buffer holds 2 x SMs - 1 ranges
    // (its last slot holds the reduction's block sums)
    const int64_t tiles = (P + kTcM - 1) / kTcM;
    const int64_t zmax = 2 * (int64_t)c->num_sms - 1;
    int64_t rows = (I + std::max<int64_t>(1, zmax / tiles) - 1) / std::max<int64_t>(1, zmax / tiles);
    rows = std::min<int64_t>(kTcRows, std::max<int64_t>(32, (rows + kTcK - 1) / kTcK * kTcK));
    const int64_t z = (I + rows - 1) / rows;
    if (z > zmax) return launch_core_fp64(c, Y, U, G, s);  // partials would not fit
    const dim3 grid((unsigned)tiles, (unsigned)z);
    if (R <= 16) launch_core_tc<16>(c, Y, U, I, P, R, (int)rows, grid, G, s);
    else if (R <= 32) launch_core_tc<32>(c, Y, U, I, P, R, (int)rows, grid, G, s);
    else if (R <= 48) launch_core_tc<48>(c, Y, U, I, P, R, (int)rows, grid, G, s);
    else launch_core_tc<64>(c, Y, U, I, P, R, (int)rows, grid, G, s);
    return;
  }
  launch_core_fp64(c, Y, U, G, s);
}

static void launch_core_fp64(Ctx *c, const float *Y, const double *U, double *G, cudaStream_t s) {
  const int N = c->N;
  const int64_t I = c->dims[N - 1];
  const int64_t P = c->mode[N - 1].P;
  const int R = c->ranks[N - 1];
  const int z = core_chunks(c->num_sms, I, P, R);
  const int rows_per_chunk = (int)((I + z - 1) / z);
  const dim3 grid((unsigned)((P + 15) / 16), (unsigned)((R + 15) / 16), (unsigned)z);
  core_kernel<<<grid, 256, 0, s>>>(Y, U, I, P, R, rows_per_chunk, c->core_part, c->core_counter, G, c->norm_dev,
                                   c->norm_dev + 1, c->fit_dev);
  ::tk::count_launch();
}

}  // namespace tk

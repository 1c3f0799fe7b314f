// K-c, Gram form for the square FP64 matrices of the fat branch, A = Y_(n) Y_(n)^T (I_n x I_n,
// I_n <= 512): the scheme of qrp_gram.cu, with S = A^T A in double-float and everything that Q is
// computed from in FP64.  The double-float numbers decide the pivots (within their error bound)
// and precondition: Q_1 = A_p M with M = R_1^-1 taken as exact lies in the span of the pivot
// columns to FP64 rounding, whatever M's own error, and E = Q_1^T Q_1 - I, in FP64, is what W
// corrects: a Cholesky QR of a matrix that is orthonormal already up to M's error (Yamamoto,
// Nakatsukasa, Yanagisawa, Fukaya: Roundoff error analysis of the CholeskyQR2 algorithm, 2015).
//
// Why: the cluster form's chain of FP64 operations, 64 cycles each and 600 for a square root or
// quotient, takes 10 us a reflector however small the matrix is; the FP64 left here is two short
// products.  With the Gram matrix of Y before it (11 us at 200 x 256), k = 16: I_n = 32 140 -> 74
// us, 200 159 -> 76 (S 9, its sum 5, pivots 22, E 17, Q 4), 512 274 -> 165.
#include <algorithm>

#include "qrp_gram.cuh"

namespace tk {
namespace {

constexpr int kHT = 32;      // columns of a tile of S, both ways
constexpr int kHRows = 32;   // rows of A per stage
constexpr int kHThreads = 256;

// Bound of the error of an entry of S over |a_i| |a_j| (u = 2^-24, N = |a_i| |a_j|): a low part stays
// below 5 u N on average, is rounded twice for each of a range's rows, and the terms added to it once
// (11 u^2 N a row); splitting and the product of the low parts come to less than 100 u^2 N, and the
// sum of the ranges and the pivot kernel's own arithmetic to less than 150.  (Equal entries beside one
// large entry reach 0.1 of it; random ones 2^-45 at any number of rows.)
float qh_eps(int rows_per) { return (float)(12 * rows_per + 256) * 0x1p-48f; }

// a as a pair of floats: the leading 24 bits exactly, the other 29 rounded to 24 (integers and one
// conversion from an integer: conversions of doubles take the FP64 pipe).  Zero below 2^-100;
// infinity from 2^127 up and for what is not finite.
__device__ __forceinline__ float2 qh_split(double a) {
  const unsigned long long b = (unsigned long long)__double_as_longlong(a);
  const uint32_t h = (uint32_t)(b >> 32), sign = h & 0x80000000u;
  const int e = (int)((h >> 20) & 0x7ffu) - 1023;
  if (e < -100) return make_float2(0.f, 0.f);
  if (e >= 127) return make_float2(__uint_as_float(sign | 0x7f800000u), 0.f);
  const uint32_t top = (uint32_t)(b >> 29) & 0x7fffffu, rest = (uint32_t)b & 0x1fffffffu;
  const float hi = __uint_as_float(sign | ((uint32_t)(e + 127) << 23) | top);
  // rest 2^(e - 52): in two steps, the first exact
  const float lo = __uint2float_rn(rest) * __uint_as_float((uint32_t)(127 - 26) << 23) *
                   __uint_as_float((uint32_t)(e - 26 + 127) << 23);
  return make_float2(hi, sign ? -lo : lo);
}

// Tile (i0 .. i0 + 31) x (j0 .. j0 + 31), i0 <= j0, of S over a range of rows, a 2 x 2 piece a
// thread: 12 FP32 instructions a product.  200 x 200: 9 us, 512 x 512: 49.
__global__ void __launch_bounds__(kHThreads) qh_gram_kernel(const double *__restrict__ A, int m, int n, int64_t lda,
                                                            int rows_per, float2 *__restrict__ part) {
  __shared__ float2 sa[kHRows][kHT], sb[kHRows][kHT];
  int ti = 0, tj = (int)blockIdx.x;  // ti >= tj
  while (tj > ti) tj -= ++ti;
  const int i0 = tj * kHT, j0 = ti * kHT, tid = threadIdx.x;
  const int r_begin = (int)blockIdx.y * rows_per, r_end = min(m, r_begin + rows_per);
  const int ia = tid / 16, jb = tid % 16;  // rows of the tile ia, ia + 16, columns jb, jb + 16
  DF acc[2][2];
  for (int r0 = r_begin; r0 < r_end; r0 += kHRows) {
    const int nr = min(kHRows, r_end - r0);
#pragma unroll
    for (int u = 0; u < kHRows * kHT / kHThreads; ++u) {
      const int r = tid / kHT + u * (kHThreads / kHT), c = tid % kHT;
      const double *row = A + (int64_t)(r0 + r) * lda;
      const double x = (r < nr && i0 + c < n) ? __ldg(row + i0 + c) : 0.0;
      const double y = (r < nr && j0 + c < n) ? __ldg(row + j0 + c) : 0.0;
      sa[r][c] = qh_split(x);
      sb[r][c] = qh_split(y);
    }
    __syncthreads();
    for (int r = 0; r < nr; r += 4) {  // (rows past nr are zero)
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const float2 x0 = sa[r + q][ia], x1 = sa[r + q][ia + 16], y0 = sb[r + q][jb], y1 = sb[r + q][jb + 16];
        auto add = [](DF &s, float2 x, float2 y) {
          df_fma(s, x.x, y.x, y.y);
          s.lo = fmaf(x.y, y.x, s.lo);
        };
        add(acc[0][0], x0, y0);
        add(acc[0][1], x0, y1);
        add(acc[1][0], x1, y0);
        add(acc[1][1], x1, y1);
      }
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        DF &s = acc[q >> 1][q & 1];
        const float t = s.hi + s.lo;
        s.lo -= t - s.hi;
        s.hi = t;
      }
    }
    __syncthreads();
  }
  float2 *dst = part + (size_t)blockIdx.y * n * n;
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    const int i = i0 + ia + 16 * (q >> 1), j = j0 + jb + 16 * (q & 1);
    if (i <= j && j < n) dst[(int64_t)i * n + j] = make_float2(acc[q >> 1][q & 1].hi, acc[q >> 1][q & 1].lo);
  }
}

// Q_1 = A_p M, a thread per entry of 16 rows a block, and the sums of E; the last block finishes:
// W to E^2, and the signs.
constexpr int kHO = 16;
__global__ void __launch_bounds__(256) qh_ortho_kernel(const double *__restrict__ A, int m, int64_t lda, int k,
                                                       const int *__restrict__ piv, const float2 *__restrict__ M,
                                                       double *__restrict__ Q1, double *__restrict__ part,
                                                       unsigned *counter, double *__restrict__ Wout, uint32_t *flag) {
  __shared__ double qs[kHO][kMaxK + 1], E[kMaxK][kMaxK + 1], W[kMaxK][kMaxK + 1];
  __shared__ float T[kMaxK][kMaxK + 1], U[kMaxK][kMaxK + 1], sgn[kMaxK];
  __shared__ bool last;
  if (*flag) return;
  const int tid = threadIdx.x, r = tid / kMaxK, c = tid % kMaxK;
  const int row = (int)blockIdx.x * kHO + r;
  const bool on = row < m && c < k;
  double q = 0.0;
  if (on) {
    double a[kMaxK];
    float2 mc[kMaxK];
#pragma unroll
    for (int l = 0; l < kMaxK; ++l) {
      a[l] = l <= c ? __ldg(A + (int64_t)row * lda + __ldg(piv + l)) : 0.0;
      mc[l] = l <= c ? __ldg(M + l * k + c) : make_float2(0.f, 0.f);
    }
#pragma unroll
    for (int l = 0; l < kMaxK; ++l) q = fma(a[l], f2d_exact(mc[l].x) + f2d_exact(mc[l].y), q);
    Q1[(int64_t)row * k + c] = q;
  }
  qs[r][c] = q;
  __syncthreads();
  const int i = tid / kMaxK, l = tid % kMaxK;
  const bool in = i < k && l < k;
  double s = 0.0;
  if (in && i <= l) {
    double s1 = 0.0;
#pragma unroll
    for (int x = 0; x < kHO; x += 2) {
      s = fma(qs[x][i], qs[x][l], s);
      s1 = fma(qs[x + 1][i], qs[x + 1][l], s1);
    }
    s += s1;
    part[(size_t)blockIdx.x * kMaxK * kMaxK + tid] = s;
  }
  __threadfence();
  __syncthreads();
  if (tid == 0) last = atomicAdd(counter, 1u) == gridDim.x - 1u;
  __syncthreads();
  if (!last) return;
  __threadfence();
  if (tid == 0) *counter = 0u;
  if (in) qs[i][l] = __ldcg(Q1 + i * k + l);  // the top block of Q_1
  float size = 0.f;
  if (in && i <= l) {
    s = i == l ? -1.0 : 0.0;  // E, the identity first
    for (int b = 0; b < (int)gridDim.x; b += 8) {
      double v[8];
#pragma unroll
      for (int u = 0; u < 8; ++u)
        v[u] = b + u < (int)gridDim.x ? __ldcg(part + (size_t)(b + u) * kMaxK * kMaxK + tid) : 0.0;
      s += ((v[0] + v[1]) + (v[2] + v[3])) + ((v[4] + v[5]) + (v[6] + v[7]));
    }
    E[i][l] = E[l][i] = s;
    size = fabsf((float)s);
    U[i][l] = (float)(i == l ? 0.5 * s : s);
  } else if (in) {
    U[i][l] = 0.f;
  }
  if (__syncthreads_or(!(size < 4e-6f))) {
    if (tid == 0) atomicOr(flag, 4u);
    return;
  }
  double w = 0.0;  // as in qrp_gram.cu: R_2 = I + U + up(-U^T U), W = I - U - up(-U^T U) + U^2
  if (in && i <= l) {
    float tt = 0.f, sq = 0.f;
#pragma unroll 4
    for (int a = 0; a < k; ++a) {
      tt = fmaf(U[a][i], U[a][l], tt);
      sq = fmaf(U[i][a], U[a][l], sq);
    }
    w = i == l ? 1.0 - 0.5 * E[i][i] + (double)(sq + 0.5f * tt) : -E[i][l] + (double)(sq + tt);
  }
  if (in) W[i][l] = w;
  __syncthreads();
  // the top block of Q, and its signs (in FP64 where FP32 leaves one open)
  double t = 0.0;
  if (in)
    for (int a = 0; a <= l; ++a) t = fma(qs[i][a], W[a][l], t);
  if (in) {
    T[i][l] = (float)t;
    E[i][l] = t;
  }
  __syncthreads();
  if (qg_signs(T, k, i, l, in, sgn)) qg_signs(E, k, i, l, in, sgn);
  if (in) Wout[i * k + l] = W[i][l] * (double)sgn[l];
}

// Q = Q_1 W D
__global__ void __launch_bounds__(256) qh_q_kernel(const double *__restrict__ Q1, int m, int k,
                                                   const double *__restrict__ W, const uint32_t *flag,
                                                   double *__restrict__ Q, int64_t ldq) {
  if (*flag) return;
  const int row = (int)blockIdx.x * 16 + threadIdx.x / kMaxK, c = threadIdx.x % kMaxK;
  if (row >= m || c >= k) return;
  double q[kMaxK], w[kMaxK], t = 0.0;
#pragma unroll
  for (int l = 0; l < kMaxK; ++l) {
    q[l] = l <= c ? __ldg(Q1 + (int64_t)row * k + l) : 0.0;
    w[l] = l <= c ? __ldg(W + l * k + c) : 0.0;
  }
#pragma unroll
  for (int l = 0; l < kMaxK; ++l)
    if (l <= c) t = fma(q[l], w[l], t);
  Q[(int64_t)row * ldq + c] = t;
}

struct Plan {
  int tiles, ranges, rows_per, blocks;
  size_t part, S, M, W, piv, opart, words, q1, total;
};

// (m, n: I_n twice)  Six reflectors and more; S grows with the cube of I_n.  With the Gram matrix
// before it, us, here and the cluster form: I_n = 32, k = 6 58, 65; 200, 6 63, 75; 320, 6 83, 102;
// 512, 6 146, 147; 512, 8 146, 171.
bool plan(int64_t m, int64_t n, int k, int num_sms, Plan *p) {
  if (k < 6 || k > kMaxK || m != n || n > kMaxN || m < 2 * k || (n > 400 && k < 8)) return false;
  const int t = (int)((n + kHT - 1) / kHT);
  p->tiles = t * (t + 1) / 2;
  const int stages = (int)((m + kHRows - 1) / kHRows), want = std::max(1, std::min(stages, 4 * num_sms / p->tiles));
  p->rows_per = (stages + want - 1) / want * kHRows;
  p->ranges = (int)((m + p->rows_per - 1) / p->rows_per);
  p->blocks = (int)((m + kHO - 1) / kHO);
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
  p->W = take(sizeof(double) * k * k);
  p->piv = take(sizeof(int) * k);
  p->q1 = take(sizeof(double) * (size_t)(m * k));
  p->opart = take(sizeof(double) * (size_t)p->blocks * kMaxK * kMaxK);
  p->total = o;
  return true;
}

}  // namespace

size_t qrp_gram_bytes64(int64_t m, int64_t n, int k, int num_sms) {
  Plan p;
  return plan(m, n, k, num_sms, &p) ? p.total : 0;
}

bool qrp_gram_takes(const double *, int64_t m, int64_t n, int k, const QrpWork *w, int num_sms) {
  const size_t need = qrp_gram_bytes64(m, n, k, num_sms);
  return w->gram_ws && need && need <= w->gram_bytes;
}

const uint32_t *qrp_gram(const double *A, int64_t m, int64_t n, int64_t lda, int k, double *Q, int64_t ldq, QrpWork *w,
                         int num_sms, cudaStream_t s, cudaError_t *err) {
  Plan p;
  plan(m, n, k, num_sms, &p);
  char *ws = static_cast<char *>(w->gram_ws);
  uint32_t *words = reinterpret_cast<uint32_t *>(ws + p.words);
  float2 *part = reinterpret_cast<float2 *>(ws + p.part);
  float2 *S = reinterpret_cast<float2 *>(ws + p.S), *M = reinterpret_cast<float2 *>(ws + p.M);
  double *W = reinterpret_cast<double *>(ws + p.W), *Q1 = reinterpret_cast<double *>(ws + p.q1);
  double *opart = reinterpret_cast<double *>(ws + p.opart);
  int *piv = reinterpret_cast<int *>(ws + p.piv);
  if ((*err = cudaMemsetAsync(words, 0, 8, s)) != cudaSuccess) return words;
  qh_gram_kernel<<<dim3((unsigned)p.tiles, (unsigned)p.ranges), kHThreads, 0, s>>>(A, (int)m, (int)n, lda, p.rows_per,
                                                                                 part);
  count_launch();
  qg_reduce(part, p.ranges, n, S, s);
  if ((*err = qg_pivots(S, n, k, qh_eps(p.rows_per), piv, M, words, s)) != cudaSuccess) return words;
  qh_ortho_kernel<<<p.blocks, 256, 0, s>>>(A, (int)m, lda, k, piv, M, Q1, opart, words + 1, W, words);
  count_launch();
  qh_q_kernel<<<(unsigned)((m + 15) / 16), 256, 0, s>>>(Q1, (int)m, k, W, words, Q, ldq);
  count_launch();
  *err = cudaGetLastError();
  return words;
}

}  // namespace tk

// What the Gram forms of the QRP share (qrp_gram.cu: tall FP32 matrices, qrp_gram64.cu: small
// square FP64 ones).
#pragma once

#include <algorithm>

#include "dfloat.cuh"
#include "internal.cuh"

namespace tk {

// Reflectors: a row of Q_1 has 16 threads, each with a column of R_1^-1 and of W in registers, and a thread
// of qg_pivot_kernel the 16 coefficients of its column.  More than 16 (32 threads a row, or two columns a
// thread) has not been tried: ranks 17 to 64 run the cluster form.
constexpr int kMaxK = 16;
constexpr int kMaxN = 512;  // columns (one thread each in the pivot kernel)

// s += p, its rounding error into the low part (TwoSum)
__device__ __forceinline__ void df_add1(DF &s, float p) {
  const float t = s.hi + p, bp = t - s.hi;
  s.lo += (s.hi - (t - bp)) + (p - bp);
  s.hi = t;
}

// S = A^T A from its partial sums part[range][n][n] (upper triangles)
void qg_reduce(const float2 *part, int ranges, int64_t n, float2 *S, cudaStream_t s);
// pivots, and R_1^-1 as pairs [k][k]; eps: the error of an entry of S over |a_i| |a_j|
cudaError_t qg_pivots(const float2 *S, int64_t n, int k, float eps, int *piv, float2 *M, uint32_t *flag, cudaStream_t s);

// Signs of the Householder reflectors, from T, the top k x k block of Q before them (a thread per
// entry (i, l), `in` where it has one; overwritten), by elimination: -sign(x_j).  All threads call.
// `close` (the same in every thread) on return: a sign lies within FP32's error.
template <typename T>
__device__ __forceinline__ bool qg_signs(T (*t)[kMaxK + 1], int k, int i, int l, bool in, float *sgn) {
  bool close = false;
  for (int j = 0; j < k; ++j) {
    const T w = t[j][j], sg = w < T(0) ? T(-1) : T(1);
    close = close || (w < T(2e-5) && w > T(-2e-5));
    const T upd = (in && i > j && l > j) ? t[i][j] * (t[j][l] / (w + sg)) : T(0);
    __syncthreads();
    if (in && i > j && l > j) t[i][l] -= upd;
    if (threadIdx.x == 0) sgn[j] = -(float)sg;
    __syncthreads();
  }
  return close;
}

}  // namespace tk

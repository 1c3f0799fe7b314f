// K-e: observed-entry loss of a Tucker model and its adjoint (the differentiation form
// of the sparse TTMc of Algorithm 2):
//     xhat_z = sum_r G[r] prod_m U_m(i_m(z), r_m),   e_z = xhat_z - x_z,   L = 1/2 sum_z e_z^2.
// With E the sparse tensor of residuals e_z at the observed coordinates,
//     dL/dU_n = TTMc_n(E) G_(n)^T          (TTMc_n as in Algorithm 2, values e_z)
//     dL/dG_(1) = U_1^T TTMc_1(E)          (the core-tensor contraction of Section III-B)
// and the forward pass needs only one row of Q = U_1 G_(1) per slice:
//     xhat_z = < Q(i_1(z), :), kron_{m > 1} U_m(i_m(z), :) >.
// So the adjoint is: one small dense product (Q), one pass over mode 1's nonzeros for the
// residuals, the loss and the TTMc of the residuals (ttmc_tile.cuh: the gathers are what it
// costs, so they are made once), then for every other mode a TTMc of the residuals (the
// kernels of ttmc.cu, fed with the caller's FP32 factors; the tiled one reads the residuals
// in place through the source positions, 10M observations 1.34 ms a step against 1.44 ms with
// a gather before it) and small dense contractions.  Kronecker rows are recomputed, never
// stored; every reduction has a fixed order.
#include <algorithm>

#include "internal.cuh"

namespace tk {

constexpr int kAdjRedBlocks = 304;  // fixed grid of the loss reduction (determinism)

// Q[i, c] = sum_r U1[i, r] G[r * P + c]    (U1: I x R1, G as R1 x P)
__global__ void adj_q_kernel(const float *U1, const float *G, int64_t I, int R1, int64_t P, float *Q) {
  for (int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; idx < I * P;
       idx += (int64_t)gridDim.x * blockDim.x) {
    const int64_t i = idx / P, c = idx % P;
    float t = 0.f;
    for (int r = 0; r < R1; ++r) t = fmaf(U1[i * R1 + r], G[(int64_t)r * P + c], t);
    Q[idx] = t;
  }
}

struct AdjFwd {
  int N;
  int64_t Z;
  const uint32_t *coords;  // [N][Z] lexicographic
  const float *vals;
  const float *U[kMaxOrder];
  int R[kMaxOrder];
  const float *Q;
  int64_t P;  // P_1 = prod_{m >= 1} R_m
  float *e;
  double *part;
};

// One thread per nonzero (lexicographic order): xhat = <Q(i_1,:), kron_{m>1} U_m(i_m,:)>
// walked with an odometer over the Kronecker index (last mode fastest).
__global__ void __launch_bounds__(256) adj_forward_kernel(AdjFwd a) {
  __shared__ double red[256];
  double sq = 0.0;
  const int N = a.N;
  for (int64_t z = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; z < a.Z; z += (int64_t)gridDim.x * blockDim.x) {
    const float *q = a.Q + (int64_t)a.coords[z] * a.P;
    const float *row[kMaxOrder];
    for (int m = 1; m < N; ++m) row[m] = a.U[m] + (int64_t)a.coords[(int64_t)m * a.Z + z] * a.R[m];
    float xhat = 0.f;
    if (N == 2) {
      for (int r = 0; r < a.R[1]; ++r) xhat = fmaf(q[r], row[1][r], xhat);
    } else {
      int r[kMaxOrder];
      float pref[kMaxOrder + 1];
      for (int m = 1; m < N; ++m) r[m] = 0;
      pref[1] = 1.f;
      for (int m = 1; m < N - 1; ++m) pref[m + 1] = pref[m] * row[m][0];
      const int Rl = a.R[N - 1];
      const float *rl = row[N - 1];
      for (int64_t c0 = 0; c0 < a.P; c0 += Rl) {
        const float pp = pref[N - 1];
        float t = 0.f;
        for (int x = 0; x < Rl; ++x) t = fmaf(q[c0 + x], rl[x], t);
        xhat = fmaf(pp, t, xhat);
        // advance modes N-2 .. 1
        int m = N - 2;
        while (m >= 1) {
          if (++r[m] < a.R[m]) break;
          r[m] = 0;
          --m;
        }
        if (m < 1) break;
        for (int t2 = m; t2 < N - 1; ++t2) pref[t2 + 1] = pref[t2] * row[t2][r[t2]];
      }
    }
    const float e = xhat - a.vals[z];
    a.e[z] = e;
    sq = fma((double)e, (double)e, sq);
  }
  red[threadIdx.x] = sq;
  __syncthreads();
  for (int o = 128; o > 0; o >>= 1) {
    if (threadIdx.x < o) red[threadIdx.x] += red[threadIdx.x + o];
    __syncthreads();
  }
  if (threadIdx.x == 0) a.part[blockIdx.x] = red[0];
}

__global__ void adj_gather_kernel(int64_t Z, const uint32_t *src, const float *e0, float *en) {
  for (int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; p < Z; p += (int64_t)gridDim.x * blockDim.x)
    en[p] = e0[src[p]];
}

struct Unfold {
  int N, n;
  int R[kMaxOrder];
};

// Gn[r_n, c] = G[r_1, ..., r_N] with c the remaining indices in ascending mode order,
// last fastest (the column order of Y_(n)).
__global__ void adj_unfold_kernel(Unfold u, const float *G, int64_t PR, float *Gn) {
  for (int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; idx < PR; idx += (int64_t)gridDim.x * blockDim.x) {
    // decode the C-order index of G
    int64_t t = idx;
    int r[kMaxOrder];
    for (int m = u.N - 1; m >= 0; --m) {
      r[m] = (int)(t % u.R[m]);
      t /= u.R[m];
    }
    int64_t c = 0;
    for (int m = 0; m < u.N; ++m)
      if (m != u.n) c = c * u.R[m] + r[m];
    const int64_t P = PR / u.R[u.n];
    Gn[(int64_t)r[u.n] * P + c] = G[idx];
  }
}

// dU[i, r] = sum_c Y[i, c] Gn[r, c], one thread per entry; for P and R too large for adj_du_kernel
__global__ void adj_du_wide_kernel(const float *Y, const float *Gn, int64_t I, int64_t P, int R, float *dU) {
  for (int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; idx < I * R;
       idx += (int64_t)gridDim.x * blockDim.x) {
    const int64_t i = idx / R;
    const int r = (int)(idx % R);
    const float *y = Y + i * P;
    const float *g = Gn + (int64_t)r * P;
    float t = 0.f;
    for (int64_t c = 0; c < P; ++c) t = fmaf(y[c], g[c], t);
    dU[idx] = t;
  }
}

// The same with G_(n) (transposed, read from G in place) and a tile of rows of Y in shared
// memory: threads (row, r) with r fastest, so a warp reads one or a few rows of Y (four
// columns at a time, the same address for all r) and adjacent entries of G.  Y is read once,
// coalesced, and G_(n) needs no kernel and no copy of its own.
constexpr int kDuThreads = 256;
__host__ __device__ inline int du_stride(int P) { return (P + 3) / 4 * 4 + 4; }  // rows in different banks
__global__ void __launch_bounds__(kDuThreads) adj_du_kernel(const float *__restrict__ Y, const float *__restrict__ G,
                                                            Unfold u, int64_t I, int P, int nr,
                                                            float *__restrict__ dU) {
  extern __shared__ float4 du_smem[];
  const int R = u.R[u.n], ld = du_stride(P);
  float *ys = reinterpret_cast<float *>(du_smem);  // [nr][ld]
  float *gs = ys + nr * ld;                        // [P][R]
  for (int q = threadIdx.x; q < P * R; q += kDuThreads) {
    int c = q / R, off = 0, stride = 1;
    for (int m = u.N - 1; m >= 0; --m) {  // C-order place of (c, r) in G
      const int i = m == u.n ? q % R : c % u.R[m];
      if (m != u.n) c /= u.R[m];
      off += i * stride;
      stride *= u.R[m];
    }
    gs[q] = __ldg(G + off);
  }
  const int row = (int)threadIdx.x / R, r = (int)threadIdx.x % R;
  for (int64_t i0 = (int64_t)blockIdx.x * nr; i0 < I; i0 += (int64_t)gridDim.x * nr) {
    const int rows = (int)min((int64_t)nr, I - i0);
    if (i0 != (int64_t)blockIdx.x * nr) __syncthreads();  // the previous tile is read
#pragma unroll 4
    for (int q = threadIdx.x; q < rows * P; q += kDuThreads) ys[q / P * ld + q % P] = __ldg(Y + i0 * P + q);
    __syncthreads();  // (the first time, G is there too)
    if (row < rows) {
      const float *y = ys + row * ld, *g = gs + r;
      float t = 0.f;
      int c = 0;
      for (; c + 3 < P; c += 4) {
        const float4 q = *reinterpret_cast<const float4 *>(y + c);
        t = fmaf(q.x, g[c * R], t);
        t = fmaf(q.y, g[(c + 1) * R], t);
        t = fmaf(q.z, g[(c + 2) * R], t);
        t = fmaf(q.w, g[(c + 3) * R], t);
      }
      for (; c < P; ++c) t = fmaf(y[c], g[c * R], t);
      dU[(i0 + row) * R + r] = t;
    }
  }
}

// Row-range partials of dG[r, c] = sum_i U1[i, r] Y[i, c]: a thread owns column c and eight
// ranks for every fourth row of its range, so Y is read once per eight ranks and U's entries
// are the same for a whole warp; the four row lanes are added in order.  At most 256 ranges of
// at least 16 rows: bound by the latency of a thread's chain of loads, so the chains are kept
// short (ncu, cold caches: 20,000 rows, 100 columns, 10 ranks, 20 rows a thread, 19 us, as 313 a
// thread 75 us; 200 rows, 64 columns, 8 ranks 5 us, as one chain of 200 48 us).
constexpr int kDgRanks = 8, kDgCols = 64, kDgLanes = 4, kDgChunks = 256;
__global__ void __launch_bounds__(kDgCols *kDgLanes) adj_dg_partial_kernel(const float *__restrict__ U1,
                                                                           const float *__restrict__ Y, int64_t I,
                                                                           int R, int64_t P, int rows_per,
                                                                           float *__restrict__ gpart) {
  __shared__ float part[kDgLanes - 1][kDgRanks][kDgCols];
  const int cl = (int)threadIdx.x % kDgCols, rl = (int)threadIdx.x / kDgCols;
  const int64_t c = (int64_t)blockIdx.x * kDgCols + cl;
  const int r0 = (int)blockIdx.z * kDgRanks, nr = min(kDgRanks, R - r0);
  const int64_t i0 = (int64_t)blockIdx.y * rows_per, i1 = min(I, i0 + rows_per);
  float t[kDgRanks];
#pragma unroll
  for (int k = 0; k < kDgRanks; ++k) t[k] = 0.f;
  if (c < P) {
#pragma unroll 4
    for (int64_t i = i0 + rl; i < i1; i += kDgLanes) {
      const float y = __ldg(Y + i * P + c);
#pragma unroll
      for (int k = 0; k < kDgRanks; ++k) t[k] = fmaf(k < nr ? __ldg(U1 + i * R + r0 + k) : 0.f, y, t[k]);
    }
  }
  if (rl > 0) {
#pragma unroll
    for (int k = 0; k < kDgRanks; ++k) part[rl - 1][k][cl] = t[k];
  }
  __syncthreads();
  if (rl > 0 || c >= P) return;
#pragma unroll
  for (int k = 0; k < kDgRanks; ++k) {
    if (k >= nr) break;
    for (int l = 0; l < kDgLanes - 1; ++l) t[k] += part[l][k][cl];
    gpart[((int64_t)blockIdx.y * R + r0 + k) * P + c] = t[k];
  }
}

// dG from its partials, a warp per entry (lanes take every 32nd range, then a tree); the last
// block adds the loss from its partials.
__global__ void __launch_bounds__(256) adj_finish_kernel(const float *__restrict__ gpart, int chunks, int64_t RP,
                                                         float *__restrict__ dG, const double *__restrict__ part,
                                                         int64_t np, double *__restrict__ loss) {
  if (blockIdx.x == gridDim.x - 1) {
    __shared__ double red[256];
    double t = 0.0;
    for (int64_t i = threadIdx.x; i < np; i += 256) t += part[i];
    red[threadIdx.x] = t;
    __syncthreads();
    for (int o = 128; o > 0; o >>= 1) {
      if (threadIdx.x < o) red[threadIdx.x] += red[threadIdx.x + o];
      __syncthreads();
    }
    if (threadIdx.x == 0) *loss = 0.5 * red[0];
    return;
  }
  const int lane = threadIdx.x & 31;
  for (int64_t o = (int64_t)blockIdx.x * 8 + (threadIdx.x >> 5); o < RP; o += (int64_t)(gridDim.x - 1) * 8) {
    float t = 0.f;
    for (int q = lane; q < chunks; q += 32) t += __ldg(gpart + (int64_t)q * RP + o);
#pragma unroll
    for (int h = 16; h > 0; h >>= 1) t += __shfl_xor_sync(0xffffffffu, t, h);
    if (lane == 0) dG[o] = t;
  }
}

static unsigned blocks_for(int64_t n, int64_t cap = 65535LL * 8) {
  return (unsigned)std::max<int64_t>(1, std::min<int64_t>((n + 255) / 256, cap));
}

// dU_n from Y_(n) of the residuals
static cudaError_t launch_du(Ctx *c, int n, const float *G, int64_t PR, float *dU, cudaStream_t s) {
  const ModeCopy &mc = c->mode[n];
  const int R = c->ranks[n];
  Unfold uf{};
  uf.N = c->N;
  uf.n = n;
  for (int m = 0; m < c->N; ++m) uf.R[m] = c->ranks[m];
  const int nr = kDuThreads / R;
  const int64_t smem = ((int64_t)nr * (mc.P + 8) + mc.P * R) * (int64_t)sizeof(float);
  constexpr int kDuSmem = 200 * 1024;
  if (smem <= kDuSmem) {
    const size_t bytes = (size_t)(nr * du_stride((int)mc.P) + (int)mc.P * R) * sizeof(float);
    // (the most of any call: the attribute is the function's, shared by all contexts)
    const cudaError_t e = cudaFuncSetAttribute(adj_du_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kDuSmem);
    if (e != cudaSuccess) return e;
    const int64_t tiles = (mc.I + nr - 1) / nr;
    const int64_t per_sm = std::max<int64_t>(1, std::min<int64_t>(4, (int64_t)(220 * 1024) / (int64_t)bytes));
    const unsigned blocks = (unsigned)std::max<int64_t>(1, std::min<int64_t>(tiles, c->num_sms * per_sm));
    adj_du_kernel<<<blocks, kDuThreads, bytes, s>>>(c->adj_Y, G, uf, mc.I, (int)mc.P, nr, dU);
    ::tk::count_launch();
  } else {
    adj_unfold_kernel<<<blocks_for(PR), 256, 0, s>>>(uf, G, PR, c->adj_Gn);
    ::tk::count_launch();
    adj_du_wide_kernel<<<blocks_for(mc.I * R), 256, 0, s>>>(c->adj_Y, c->adj_Gn, mc.I, mc.P, R, dU);
    ::tk::count_launch();
  }
  return cudaGetLastError();
}

tucker_status launch_loss_grad(Ctx *c, const float *const *U, const float *G, double *loss, float *const *dU,
                               float *dG, cudaStream_t s) {
  const int N = c->N;
  const int64_t Z = c->nnz;
  int64_t PR = 1, ymax = 1;
  for (int m = 0; m < N; ++m) PR *= c->ranks[m];
  for (int m = 0; m < N; ++m) ymax = std::max(ymax, c->mode[m].I * c->mode[m].P);
  const ModeCopy &m0 = c->mode[0];
  const int64_t I1 = c->dims[0], P1 = m0.P;
  const int R1 = c->ranks[0];
  const int64_t room = std::max<int64_t>(1, (64ll << 20) / PR);  // partials of dG: 256 MB at most
  const int chunks = (int)std::max<int64_t>(1, std::min<int64_t>({kDgChunks, (I1 + 15) / 16, room}));
  int64_t qrow = 0;  // floats of a row of Q for the fused form
  const bool fused = tile_adj_plan(tile_call(c, 0, nullptr, nullptr), &qrow) && m0.n_units > 0;
  if (!c->adj_e0) {  // first call: buffers allocated in the order of s, ready for any stream after the sync
    c->astream = s;
    TK_CUDA(dev_alloc(c, &c->adj_en, (size_t)std::max<int64_t>(Z, 1)));
    TK_CUDA(dev_alloc(c, &c->adj_Y, (size_t)ymax));
    TK_CUDA(dev_alloc(c, &c->adj_Q, (size_t)(I1 * (fused ? qrow : P1))));
    TK_CUDA(dev_alloc(c, &c->adj_Gn, (size_t)PR));
    int64_t packed = 0;
    for (int m = 0; m < N; ++m) packed += c->dims[m] * tile_layout(c->ranks[m]).row();
    TK_CUDA(dev_alloc(c, &c->adj_U, (size_t)packed));
    TK_CUDA(dev_alloc(c, &c->adj_part, (size_t)std::max<int64_t>(kAdjRedBlocks, m0.n_units)));
    TK_CUDA(dev_alloc(c, &c->adj_gpart, (size_t)(chunks * PR)));
    TK_CUDA(dev_alloc(c, &c->adj_e0, (size_t)std::max<int64_t>(Z, 1)));
    TK_CUDA(cudaStreamSynchronize(s));
    c->astream = 0;
  }
  // (0) the factors as the TTMc reads them: copies in tile_layout, unless the caller's are that already
  const float *Up[kMaxOrder];
  {
    TilePack pk{};
    int copies = 0;
    float *at = c->adj_U;
    for (int m = 0; m < N; ++m) {
      Up[m] = U[m];
      const int64_t n = c->dims[m] * tile_layout(c->ranks[m]).row();
      if (!tile_plain(c->ranks[m]) || reinterpret_cast<uintptr_t>(U[m]) % 16 != 0) {
        pk.in[copies] = U[m];
        pk.out[copies] = at;
        pk.I[copies] = c->dims[m];
        pk.R[copies++] = c->ranks[m];
        Up[m] = at;
      }
      at += n;
    }
    if (copies) launch_tile_pack(pk, copies, s);
  }
  // (1) residuals, their squares, and for mode 1 the TTMc of the residuals: in one kernel, or
  //     where a row has more tiles than that holds, Q = U_1 G_(1), then one thread per nonzero
  int64_t parts = kAdjRedBlocks;
  if (fused) {
    TileAdj a{};
    a.U = U[0];
    a.G = G;
    a.I = I1;
    a.R = R1;
    a.Q = c->adj_Q;
    a.esrc = m0.src;
    a.e_out = c->adj_e0;
    a.sq_part = c->adj_part;
    TK_CUDA(launch_tile_adj(tile_call(c, 0, Up, c->adj_Y), a, s));
    ttmc_finish(c, 0, c->adj_Y, nullptr, s);
    TK_CUDA(cudaGetLastError());
    parts = m0.n_units;
  } else {
    adj_q_kernel<<<blocks_for(I1 * P1), 256, 0, s>>>(U[0], G, I1, R1, P1, c->adj_Q);
    ::tk::count_launch();
    AdjFwd f{};
    f.N = N;
    f.Z = Z;
    f.coords = c->coords;
    f.vals = c->vals;
    for (int m = 0; m < N; ++m) {
      f.U[m] = U[m];
      f.R[m] = c->ranks[m];
    }
    f.Q = c->adj_Q;
    f.P = P1;
    f.e = c->adj_e0;
    f.part = c->adj_part;
    adj_forward_kernel<<<kAdjRedBlocks, 256, 0, s>>>(f);
    ::tk::count_launch();
  }
  // (2) per mode: TTMc of the residuals, then dU_n and (mode 1) dG and the loss
  for (int n = 0; n < N; ++n) {
    const ModeCopy &mc = c->mode[n];
    if (!(n == 0 && fused)) {
      const float *en = c->adj_e0;
      const uint32_t *src = mc.src;  // where this mode's order is not the lexicographic one
      if (src && Z > 0 && !ttmc_tiled(c, n)) {
        adj_gather_kernel<<<blocks_for(Z, 4096), 256, 0, s>>>(Z, src, c->adj_e0, c->adj_en);
        ::tk::count_launch();
        en = c->adj_en;
        src = nullptr;
      }
      tucker_status st = launch_ttmc_ex(c, n, c->adj_Y, en, src, Up, s);
      if (st != TUCKER_OK) return st;
    }
    TK_CUDA(launch_du(c, n, G, PR, dU[n], s));
    if (n == 0) {
      const int rows_per = (int)((I1 + chunks - 1) / chunks);
      const dim3 grid((unsigned)((P1 + kDgCols - 1) / kDgCols), (unsigned)chunks,
                      (unsigned)((R1 + kDgRanks - 1) / kDgRanks));
      adj_dg_partial_kernel<<<grid, kDgCols * kDgLanes, 0, s>>>(U[0], c->adj_Y, I1, R1, P1, rows_per, c->adj_gpart);
      ::tk::count_launch();
      adj_finish_kernel<<<(unsigned)std::min<int64_t>((PR + 7) / 8, 2048) + 1, 256, 0, s>>>(
          c->adj_gpart, chunks, PR, dG, c->adj_part, parts, loss);
      ::tk::count_launch();
    }
  }
  TK_CUDA(cudaGetLastError());
  return TUCKER_OK;
}

}  // namespace tk

// Tiled form of the TTMc (ttmc_tile.cuh): choice of the tile, and the launches for up to two
// remaining modes (orders 2 and 3).
#include <algorithm>

#include "ttmc_tile.cuh"

namespace tk {

// The tile of a mode's TTMc: the ranks of slots 1 and 0 cut into chunks of cA and cB (those of
// the copies, or the halves of chunks of eight), computed by a kernel of TA x TB >= cA x cB.
// The cheapest by this count of issue slots for a step of 32 nonzeros, for slices of `len`
// nonzeros on average:
//   a pass over NG nonzeros   TA TB multiply-adds (packed ones take two cycles), 2 TA products,
//                             the reads and addresses; at least 4 (TA + TB + 1), what its reads
//                             hold of the path to the registers that the schedulers share
//   passes                    32 / NG, and at least one for each slice the step meets
//   a finished slice          for each tile row its stores, reads and sums over the groups
//   few warps                 an SM holds 3 (8 x 8) to 8 (4 x 4) blocks of 128 threads
// Large tiles have the fewest slots per multiply-add, small ones the warps to fill them and
// the cheaper ends of slices.  Measured on 5M nonzeros, ranks 8^4 (four modes): 8 x 8 1.20 ms,
// 8 x 4 1.14 ms, 4 x 4 1.17 ms; on 10,000 nonzeros, ranks 8^3, a mode: 8 x 8 13 us, 4 x 4 11 us.
struct TileChoice {
  int cA, cB, TA, TB;
  double cost;
};

static int tile_width(int c, int no) {  // kernel widths: 4, 5, 6, 7, 8; 7 only with up to two modes
  if (c <= 4) return 4;
  if (no >= 4) return c <= 5 ? 5 : 8;
  if (c == 7 && no == 3) return 8;
  return c;
}

static TileChoice tile_choose(int nother, const int *R /* slot order */, double len, bool adj) {
  TileChoice best{0, 0, 0, 0, 1e300};
  int64_t lead = 1;
  for (int t = 2; t < nother; ++t) lead *= R[t];
  const TileLayout lB = tile_layout(R[0]);
  const TileLayout lA = nother > 1 ? tile_layout(R[1]) : TileLayout{1, 1, 1};
  for (int ha = 0; ha < 2; ++ha)
    for (int hb = 0; hb < 2; ++hb) {  // a chunk of eight may be taken as two of four
      if ((ha && !(nother > 1 && lA.T == 8)) || (hb && lB.T != 8)) continue;
      TileChoice c;
      c.cA = ha ? 4 : lA.T;
      c.cB = hb ? 4 : lB.T;
      c.TA = nother > 1 ? tile_width(c.cA, nother) : 1;
      c.TB = tile_width(c.cB, nother);
      if (adj && !tile_adj_covers(c.TA, c.TB, nother)) continue;
      const int nA = lA.n * (ha ? 2 : 1), nB = lB.n * (hb ? 2 : 1);
      const int64_t G = lead * nA * nB;
      const int Gw = (int)std::min<int64_t>(G, 32), NG = 32 / Gw;
      const double blocks = (double)((G + 31) / 32);
      const int tile = c.TA * c.TB;
      const double slots = tile + 2 * c.TA + (c.TA + 3) / 4 + (c.TB + 3) / 4 + 7 + 2 * (nother - 2);
      const double lds = 4.0 * (c.TA + c.TB + 1 + std::max(nother - 2, 0));
      const double slices = 32.0 / len;
      const double passes = std::max(1.0 + slices, 32.0 / NG + 0.5 * (1.0 + slices));
      const double flush = slices * (20.0 + c.TA * (8.0 + (Gw * c.TB + 31) / 32 * (10.0 + 2.0 * NG)));
      c.cost = blocks * (passes * std::max(slots, lds) + flush + 40.0) * (1.0 + 3.0 / tile_min_blocks(tile));
      if (adj && G > 32) continue;
      if (c.cost < best.cost) best = c;
    }
  return best;
}

#define TK_TILE_B(NO, TA)                                            \
  switch (TB) {                                                      \
    case 4: return run_tile<NO, TA, 4>(p, num_sms, s);               \
    case 5: return run_tile<NO, TA, 5>(p, num_sms, s);               \
    case 6: return run_tile<NO, TA, 6>(p, num_sms, s);               \
    case 7: return run_tile<NO, TA, 7>(p, num_sms, s);               \
    default: return run_tile<NO, TA, 8>(p, num_sms, s);              \
  }

static cudaError_t tile_dispatch_12(int TA, int TB, TileParams &p, int num_sms, cudaStream_t s) {
  switch (TA) {
    case 1: TK_TILE_B(1, 1)
    case 4: TK_TILE_B(2, 4)
    case 5: TK_TILE_B(2, 5)
    case 6: TK_TILE_B(2, 6)
    case 7: TK_TILE_B(2, 7)
    default: TK_TILE_B(2, 8)
  }
}

static TileChoice tile_plan(const TileCall &c, bool adj, TileParams &p) {
  const int no = c.nother;
  p.nother = no;
  int used = 0;
  for (int t = 0; t < no; ++t) {  // slots: the remaining modes backwards
    const int m = no - 1 - t;
    const int row = tile_layout(c.R[m]).row();
    p.idx[t] = c.idx[m];
    p.U[t] = c.U[m];
    p.R[t] = c.R[m];
    p.off[t] = used;
    for (p.lq[t] = 0; (4 << p.lq[t]) < row; ++p.lq[t]) {
    }
    used += row;
  }
  const TileChoice k = tile_choose(no, p.R, c.slice_len, adj);
  const TileLayout lB = tile_layout(p.R[0]);
  p.cB = k.cB;
  p.nB = k.cB == lB.T ? lB.n : 2 * lB.n;
  p.jB = k.cB == lB.T ? lB.jump : 0;
  p.cA = p.nA = 1;
  if (no > 1) {
    const TileLayout lA = tile_layout(p.R[1]);
    p.cA = k.cA;
    p.nA = k.cA == lA.T ? lA.n : 2 * lA.n;
    p.jA = k.cA == lA.T ? lA.jump : 0;
  }
  int64_t G = (int64_t)p.nA * p.nB;
  for (int t = 2; t < no; ++t) G *= p.R[t];
  p.G = (int)G;
  p.Gw = std::min(p.G, 32);
  if (adj)  // a power of two
    for (p.Gw = 1; p.Gw < p.G && p.Gw < 32;) p.Gw *= 2;
  p.NG = 32 / p.Gw;
  p.RS = 4 * tile_record(used / 4, p.Gw, p.nB, p.nA, 1 << p.lq[0], no > 1 ? 1 << p.lq[1] : 1);
  p.val = c.val;
  p.vsrc = c.vsrc;
  p.sptr = c.sptr;
  p.sid = c.sid;
  p.S = c.S;
  p.unit_e0 = c.unit_e0;
  p.unit_k0 = c.unit_k0;
  p.unit_slot = c.unit_slot;
  p.n_units = c.n_units;
  p.Z = c.Z;
  p.Y = c.Y;
  p.carry = c.carry;
  p.P = c.P;
  return k;
}

cudaError_t launch_ttmc_tile(const TileCall &c, cudaStream_t s) {
  TileParams p{};
  const TileChoice k = tile_plan(c, false, p);
  return c.nother <= 2 ? tile_dispatch_12(k.TA, k.TB, p, c.num_sms, s) : tile_dispatch_n(k.TA, k.TB, p, c.num_sms, s);
}

// ---- adjoint form
// Q = U G_(n) in the order of the lanes' tiles: block = 128 places of a row (entry i of lane
// j's tile at i * Gw + j, zero where there is none), some rows; the columns of G of those places
// are held in shared memory.  Rows of U are read by all threads alike.
constexpr int kQCols = 128, kQRows = 16;
__global__ void __launch_bounds__(kQCols) tile_q_kernel(const TileParams p, const float *__restrict__ U,
                                                        const float *__restrict__ G, int64_t I, int R, int TB, int QP,
                                                        float *__restrict__ Q) {
  extern __shared__ float gs[];  // [R][kQCols]
  const int f = (int)blockIdx.y * kQCols + (int)threadIdx.x;
  int64_t col = -1;
  if (f < QP) {
    const int i = f / p.Gw, j = f % p.Gw, a = i / TB, b = i % TB;
    if (j < p.G && a < p.cA && b < p.cB) {
      const int R1 = p.nother == 1 ? 1 : p.R[1], R0 = p.R[0];
      int ja, jb, lead;
      tile_split(j, p.nA, p.nB, ja, jb, lead);
      const int r = ja * (p.cA == 8 ? 4 : p.cA) + a + (a >= 4 ? p.jA : 0);
      const int q = jb * (p.cB == 8 ? 4 : p.cB) + b + (b >= 4 ? p.jB : 0);
      if (r < R1 && q < R0) col = ((int64_t)lead * R1 + r) * R0 + q;
    }
  }
  for (int r = 0; r < R; ++r) gs[r * kQCols + threadIdx.x] = col >= 0 ? __ldg(G + r * p.P + col) : 0.f;
  if (f >= QP) return;
  const int64_t i0 = (int64_t)blockIdx.x * kQRows, i1 = min(I, i0 + kQRows);
  int64_t i = i0;
  for (; i + 3 < i1; i += 4) {  // four rows at a time: their loads are in flight together
    float t[4] = {0.f, 0.f, 0.f, 0.f};
    for (int r = 0; r < R; ++r) {
      const float g = gs[r * kQCols + threadIdx.x];
#pragma unroll
      for (int k = 0; k < 4; ++k) t[k] = fmaf(__ldg(U + (i + k) * R + r), g, t[k]);
    }
#pragma unroll
    for (int k = 0; k < 4; ++k) Q[(i + k) * QP + f] = t[k];
  }
  for (; i < i1; ++i) {
    float t = 0.f;
    for (int r = 0; r < R; ++r) t = fmaf(__ldg(U + i * R + r), gs[r * kQCols + threadIdx.x], t);
    Q[i * QP + f] = t;
  }
}

// The tile the adjoint form runs with, or false where a row has more tiles than a warp lanes.
bool tile_adj_plan(const TileCall &c, int64_t *row_floats) {
  TileParams p{};
  const TileChoice k = tile_plan(c, true, p);
  *row_floats = (int64_t)k.TA * k.TB * p.Gw;
  return p.G <= 32 && k.cost < 1e300;
}

cudaError_t launch_tile_adj(const TileCall &c, const TileAdj &a, cudaStream_t s) {
  TileParams p{};
  const TileChoice k = tile_plan(c, true, p);
  const int QP = k.TA * k.TB * p.Gw;
  const dim3 grid((unsigned)((a.I + kQRows - 1) / kQRows), (unsigned)((QP + kQCols - 1) / kQCols));
  tile_q_kernel<<<grid, kQCols, (size_t)a.R * kQCols * sizeof(float), s>>>(p, a.U, a.G, a.I, a.R, k.TB, QP, a.Q);
  ::tk::count_launch();
  p.Q = a.Q;
  p.esrc = a.esrc;
  p.e_out = a.e_out;
  p.sq_part = a.sq_part;
  return tile_dispatch_adj(k.TA, k.TB, p, c.num_sms, s);
}

// ---- factor copies in the tiled layout
__global__ void tile_pack_kernel(const TilePack p) {
  const int m = (int)blockIdx.y;
  const TileLayout l = tile_layout(p.R[m]);
  const int row = l.row();  // a power of two
  const int sh = 31 - __clz(row);
  const int64_t n = p.I[m] << sh;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
    const int r = l.rank((int)(i & (row - 1)), p.R[m]);
    p.out[m][i] = r >= 0 ? __ldg(p.in[m] + (i >> sh) * p.R[m] + r) : 0.f;
  }
}

void launch_tile_pack(const TilePack &p, int modes, cudaStream_t s) {
  int64_t n = 1;
  for (int m = 0; m < modes; ++m) n = std::max<int64_t>(n, p.I[m] * tile_layout(p.R[m]).row());
  const unsigned blocks = (unsigned)std::min<int64_t>((n + 255) / 256, 1024);
  tile_pack_kernel<<<dim3(blocks, (unsigned)modes), 256, 0, s>>>(p);
  ::tk::count_launch();
}

}  // namespace tk

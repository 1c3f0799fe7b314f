// K-b, tiled form: the sparse TTMc of one mode (Algorithm 2 inner loop, Section III-C) in
// FP32 for any order and any ranks, on register tiles.
//
// One nonzero adds x_z (a_z (x) ... (x) b_z) to a row of Y_(n).  The row is cut into tiles of
// TA x TB entries: TA consecutive ranks of the last remaining mode but one, TB of the last
// one, and one rank of each mode before them.  A lane owns one tile; the G lanes that hold a
// whole row form a group, and the NG = 32 / G groups of a warp take alternate nonzeros of a
// slice.  Per nonzero a lane reads TA + TB floats for TA TB multiply-adds, so large tiles are
// what keeps the path from shared memory to the registers from being the limit.
//
// What bounds it (ncu, 10M uniform nonzeros, ranks 10^3, one mode 0.30 ms): the gathers.  A
// 16-byte cp.async of a warp takes about ten cycles of the load/store path (rows lie in eight
// different lines), 2.7 cycles a nonzero; rows come from L2 at 4.8 TB/s; issue slots 39% busy.
// With 512 columns (5M nonzeros, ranks 8^4, one mode 0.24 - 0.29 ms) the multiply-adds: FMA
// pipe 47%, issue slots 62% busy.
//
// One warp owns one work unit (reorder.cu), in steps of 32 or 16 nonzeros.  The factor rows and
// the values of step t + 1 are copied to shared memory by cp.async while step t is
// computed: no registers hold them, and a warp waits on no gather it has just issued.  A
// nonzero's rows lie side by side in one record, at a record stride chosen for the bank groups
// that the reads of a half-warp fall in (tile_record).
//
// Factors are read from copies with the ranks cut into 1, 2, 4 or 8 equal chunks of at most
// eight (tile_layout), zero-padded so that every piece of a row is a 16-byte copy, whatever
// the rank.  Ranks 4, 8, 16, 32 and 64 need no padding: their copies are the plain matrices.
//
// When a slice ends, its row is finished one tile row at a time through a small buffer in
// shared memory: every lane stores that row of its tile, then lanes take consecutive entries
// of Y, add the groups' parts in group order and store them.  Fixed orders: Y is reproducible
// bit for bit.
#pragma once

#include <algorithm>
#include <climits>

#include "dfloat.cuh"
#include "internal.cuh"

namespace tk {

constexpr int kTileOthers = kMaxOrder - 1;
constexpr int kTileWarps = 4;  // warps per block at most

struct TileParams {
  // slot 0: the last remaining mode, slot 1: the one before it, slots 2 ..: the others, backwards
  const uint32_t *idx[kTileOthers];  // sorted coordinates
  const float *U[kTileOthers];       // factor copies (tile_layout)
  int lq[kTileOthers];               // log2 of the 16-byte pieces of a row
  int off[kTileOthers];              // first float of the row in a record
  int R[kTileOthers];
  int nother;
  const float *val;                  // value of sorted position e: val[vsrc[e]], or val[e] with vsrc null
  const uint32_t *vsrc;
  const uint32_t *sptr, *sid;
  uint32_t S;
  const uint32_t *unit_e0, *unit_k0;
  const int32_t *unit_slot;
  int64_t n_units;
  uint32_t Z;
  float *Y, *carry;
  int64_t P;
  int RS;      // floats in a record
  int G;       // tiles of a row of Y
  int Gw, NG;  // lanes of a group, groups of a warp
  int nA, nB;  // chunks of slots 1 and 0 (nA = 1 with one remaining mode)
  int cA, cB;  // ranks in a chunk
  int jA, jB;  // ranks skipped after the first four of a chunk
  // adjoint form: the model's value is subtracted first, see tile_kernel
  const float *Q;        // [I][TA * TB][Gw] rows of U_n G_(n) in the order of the lanes' tiles
  const uint32_t *esrc;  // where the residual of sorted position e goes: e_out[esrc[e]], or e_out[e]
  float *e_out;
  double *sq_part;       // [n_units] sums of squared residuals
};

__device__ __forceinline__ void tile_cp16(uint32_t dst, const void *src) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 16;\n" ::"r"(dst), "l"(src) : "memory");
}
__device__ __forceinline__ void tile_cp4(uint32_t dst, const void *src) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4;\n" ::"r"(dst), "l"(src) : "memory");
}
__device__ __forceinline__ void tile_commit() { asm volatile("cp.async.commit_group;\n" ::: "memory"); }
template <int N>
__device__ __forceinline__ void tile_wait() {
  asm volatile("cp.async.wait_group %0;\n" ::"n"(N) : "memory");
}

// reads at 32-bit shared-memory addresses (ordered by the barriers around a step's records,
// so not by the compiler's view of memory)
__device__ __forceinline__ float tile_lds1(uint32_t a) {
  float v;
  asm volatile("ld.shared.f32 %0, [%1];" : "=f"(v) : "r"(a));
  return v;
}
// the T ranks of a chunk: its first four at a, the others at a + hop
template <int T>
__device__ __forceinline__ void tile_lds(uint32_t a, uint32_t hop, float (&v)[T]) {
  asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(v[0]), "=f"(v[1]), "=f"(v[2]), "=f"(v[3]) : "r"(a));
  if constexpr (T == 5) {
    v[4] = tile_lds1(a + hop);
  } else if constexpr (T == 6) {
    asm volatile("ld.shared.v2.f32 {%0, %1}, [%2];" : "=f"(v[4]), "=f"(v[5]) : "r"(a + hop));
  } else if constexpr (T >= 7) {
    float w;
    asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(v[4]), "=f"(v[5]), "=f"(v[6]), "=f"(w) : "r"(a + hop));
    if constexpr (T == 8) v[7] = w;
  }
}

// Pairs of FP32 values and the packed multiply-add on them (one issue slot for two products,
// each rounded as fmaf does).
struct TileF2 {
  unsigned long long v;
};
__device__ __forceinline__ TileF2 tile_pack(float lo, float hi) {
  TileF2 r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r.v) : "f"(lo), "f"(hi));
  return r;
}
__device__ __forceinline__ float2 tile_unpack(TileF2 a) {
  float2 r;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(a.v));
  return r;
}
__device__ __forceinline__ TileF2 tile_fma2(TileF2 a, TileF2 b, TileF2 c) {
  TileF2 r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r.v) : "l"(a.v), "l"(b.v), "l"(c.v));
  return r;
}

// A lane's tile, columns in pairs (the reads of b give them; s a[i] is formed twice to fill a
// pair, which costs less than copying), an odd last column by itself.
template <int TA, int TB>
struct TileAcc {
  static constexpr int PB = TB / 2, OB = TB % 2;
  TileF2 p[TA * PB];
  float o[OB ? TA : 1];
  __device__ __forceinline__ void clear() {
    const TileF2 z = tile_pack(0.f, 0.f);
#pragma unroll
    for (int i = 0; i < TA * PB; ++i) p[i] = z;
#pragma unroll
    for (int i = 0; i < OB * TA; ++i) o[i] = 0.f;
  }
  // += s a (x) b
  __device__ __forceinline__ void add(float s, const float (&a)[TA], const float (&b)[TB]) {
    TileF2 b2[PB];
#pragma unroll
    for (int k = 0; k < PB; ++k) b2[k] = tile_pack(b[2 * k], b[2 * k + 1]);
#pragma unroll
    for (int i = 0; i < TA; ++i) {
      const float x0 = __fmul_rn(s, a[i]);
      float x1;  // (volatile: a second product, not a copy of the first)
      asm volatile("mul.rn.f32 %0, %1, %2;" : "=f"(x1) : "f"(s), "f"(a[i]));
      const TileF2 sa = tile_pack(x0, x1);
#pragma unroll
      for (int k = 0; k < PB; ++k) p[i * PB + k] = tile_fma2(sa, b2[k], p[i * PB + k]);
      if constexpr (OB != 0) o[i] = fmaf(tile_unpack(sa).x, b[TB - 1], o[i]);
    }
  }
  template <typename F>
  __device__ __forceinline__ void load(F f) {  // entry i of the flat tile is f(i)
#pragma unroll
    for (int a = 0; a < TA; ++a) {
#pragma unroll
      for (int k = 0; k < PB; ++k) p[a * PB + k] = tile_pack(f(a * TB + 2 * k), f(a * TB + 2 * k + 1));
      if constexpr (OB != 0) o[a] = f(a * TB + TB - 1);
    }
  }
  __device__ __forceinline__ float dot(const float (&a)[TA], const float (&b)[TB]) const {  // a^T tile b
    TileF2 b2[PB];
#pragma unroll
    for (int k = 0; k < PB; ++k) b2[k] = tile_pack(b[2 * k], b[2 * k + 1]);
    float s = 0.f;
#pragma unroll
    for (int i = 0; i < TA; ++i) {
      TileF2 t = tile_pack(0.f, 0.f);
#pragma unroll
      for (int k = 0; k < PB; ++k) t = tile_fma2(p[i * PB + k], b2[k], t);
      const float2 q = tile_unpack(t);
      float r = q.x + q.y;
      if constexpr (OB != 0) r = fmaf(o[i], b[TB - 1], r);
      s = fmaf(a[i], r, s);
    }
    return s;
  }
  __device__ __forceinline__ void row(int a, float (&v)[TB]) const {  // a known at compile time
#pragma unroll
    for (int k = 0; k < PB; ++k) {
      const float2 q = tile_unpack(p[a * PB + k]);
      v[2 * k] = q.x;
      v[2 * k + 1] = q.y;
    }
    if constexpr (OB != 0) v[TB - 1] = o[a];
  }
};

// Cycles the shared-memory path takes for 16-byte accesses of 16 lanes, lane l at 16-byte
// place (l / per) * k + l % per (k: the record stride in 16-byte pieces): the most distinct
// places that share a bank group.
__host__ __device__ constexpr int tile_bank_cycles(int per, int k) {
  if (per > 16) per = 16;
  int most = 0;
  for (int b = 0; b < 8; ++b) {
    int cnt = 0;
    for (int l = 0; l < 16; ++l) cnt += ((l / per) * k + l % per) % 8 == b;
    if (cnt > most) most = cnt;
  }
  return most;
}
// Record stride in 16-byte pieces: the smallest of the `used` pieces and up to seven more with
// the fewest cycles for the reads of both tiles' halves (rows of n chunks, read by G lanes a
// record) and for the copies (rows of q pieces).
__host__ __device__ constexpr int tile_record(int used, int G, int n0, int n1, int q0, int q1) {
  int best = used, cost = 1 << 30;
  for (int k = used; k < used + 8; ++k) {
    const int per = G < 16 ? G : 16;
    int c = 0;
    for (int h = 0; h < 2; ++h) {
      const int n = h ? n1 : n0, q = h ? q1 : q0;
      // the G lanes of a record read n distinct places; 16 / G records side by side
      int most = 0;
      for (int b = 0; b < 8; ++b) {
        int cnt = 0;
        for (int r = 0; r < 16 / per; ++r)
          for (int i = 0; i < (n < per ? n : per); ++i) cnt += (r * k + i) % 8 == b;
        if (cnt > most) most = cnt;
      }
      c += 8 * most + 2 * tile_bank_cycles(q, k);
    }
    if (c < cost) {
      cost = c;
      best = k;
    }
  }
  return best;
}

// Tile j of a row: chunk jb of slot 0, ja of slot 1, and the number of its leading ranks.  Of j's
// low bits the first is jb's, the next ja's, then come jb's others and ja's: a 16-byte read of
// shared memory takes two cycles where no four consecutive lanes read more than two places, and
// four otherwise (measured: with jb's bits lowest and four chunks or more, four).
__host__ __device__ __forceinline__ void tile_split(int j, int nA, int nB, int &ja, int &jb, int &lead) {
  if (nB >= 4 && nA >= 2) {
    jb = (j & 1) | (j / 4 % (nB / 2)) << 1;
    ja = (j / 2 & 1) | (j / (2 * nB) % (nA / 2)) << 1;
  } else {
    jb = j % nB;
    ja = j / nB % nA;
  }
  lead = j / nB / nA;
}

// floats between the lanes' tile rows (an odd number of 16-byte pieces), and of a warp's memory
__host__ __device__ constexpr int tile_row_stride(int TB) { return TB <= 4 ? 4 : 12; }
__host__ __device__ constexpr int tile_warp_floats(int RS, int TB, int KS) {
  return 2 * KS * (RS + 1) + 32 * tile_row_stride(TB) + 2 * 32 * TB;
}

constexpr int tile_min_blocks(int tile) {  // blocks of 128 threads an SM is to hold (registers)
  return tile > 56 ? 3 : tile > 40 ? 4 : tile > 30 ? 5 : tile > 20 ? 6 : 8;
}

// KS: nonzeros of a step.
// NO: remaining modes whose indices are held in registers (1, 2, 3, or 7 for 4 to 7).
//
// ADJ (adjoint.cu): the TTMc of the residuals e_z = <Q(i_n, :), kron rows of z> - x_z, which it
// forms on the way and writes out: a lane holds its tile of the slice's row of Q beside its
// sums, so the gathers, which bound this kernel, are made once for both (10M observations,
// ranks 10^3: 0.40 ms; one thread per nonzero forming e_z alone took 1.71 ms, and the TTMc
// 0.30 ms after it).  A group's lanes add their parts of the inner product by shuffles (Gw a
// power of two; all groups step together).
template <int NO, int TA, int TB, bool ADJ, int KS = 32>
__global__ void __launch_bounds__(kTileWarps * 32, tile_min_blocks(TA * TB * (ADJ ? 2 : 1)))
    ttmc_tile_kernel(const __grid_constant__ TileParams p) {
  static_assert(NO > 1 || TA == 1, "one remaining mode: tiles of one row");
  constexpr unsigned kAll = 0xffffffffu;
  extern __shared__ float4 tile_smem[];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int64_t u = (int64_t)blockIdx.x * (blockDim.x >> 5) + w;
  if (u >= p.n_units) return;
  const int RS = p.RS, nother = NO <= 3 ? NO : p.nother;
  const int Gw = p.Gw, NG = p.NG, nA = p.nA, nB = p.nB;
  float *ring = reinterpret_cast<float *>(tile_smem) + (size_t)w * tile_warp_floats(RS, TB, KS);  // two steps
  float *rows = ring + 2 * KS * (RS + 1);                                                          // one tile row per lane
  int2 *place = reinterpret_cast<int2 *>(rows + 32 * tile_row_stride(TB));  // entries of Gw * TB columns
  const uint32_t ring_s = (uint32_t)__cvta_generic_to_shared(ring);

  // this lane's tile: chunk ja of slot 1, chunk jb of slot 0, one rank of each further slot
  const int g = lane / Gw;
  int j = (int)blockIdx.y * 32 + lane % Gw;
  if (j >= p.G) j = 0;  // no tile of its own: computes one, and `place` holds no place for it
  int jb, ja, lead;
  tile_split(j, nA, nB, ja, jb, lead);
  const int R1 = NO == 1 ? 1 : p.R[1], R0 = p.R[0];
  // where entry (row 0, column b) of tile j of this block's tiles goes in a row of Y, and the
  // tile's first rank of slot 1 (chunks of eight, or fours of them, start at rank 4 j; others at cA j)
  for (int o = lane; o < Gw * TB; o += 32) {
    const int oj = (int)blockIdx.y * 32 + o / TB, b = o % TB;
    int ob, oa, ol;
    tile_split(oj, nA, nB, oa, ob, ol);
    const int c = ob * (p.cB == 8 ? 4 : p.cB) + b + (b >= 4 ? p.jB : 0);
    place[o] = make_int2(ol * R1 * R0 + c,
                         oj < p.G && b < p.cB && c < R0 ? oa * (p.cA == 8 ? 4 : p.cA) : INT_MIN / 2);
  }
  const uint32_t aoff = NO == 1 ? 0u : (uint32_t)(p.off[1] + 4 * ja) * 4u, boff = (uint32_t)(p.off[0] + 4 * jb) * 4u;
  const uint32_t hopA = 16u * (uint32_t)nA, hopB = 16u * (uint32_t)nB;
  uint32_t loff[NO > 2 ? NO - 2 : 1];
  if constexpr (NO > 2) {
#pragma unroll
    for (int t = 2; t < NO; ++t) {
      loff[t - 2] = 0u;
      if (t < nother) {
        loff[t - 2] = (uint32_t)(p.off[t] + tile_layout(p.R[t]).pos(lead % p.R[t])) * 4u;
        lead /= p.R[t];
      }
    }
  }

  const uint32_t e0 = __ldg(p.unit_e0 + u);
  const uint32_t e_end = (u + 1 < p.n_units) ? __ldg(p.unit_e0 + u + 1) : p.Z;
  const int ntiles = (int)((e_end - e0 + (uint32_t)KS - 1u) / (uint32_t)KS);

  uint32_t id[NO], vs = 0u;  // indices of the step whose copies are issued next (lane = position)
  auto load_ids = [&](int t) {
    const uint32_t e = e0 + (uint32_t)KS * (uint32_t)t + (uint32_t)lane;
    const bool in = (KS == 32 || lane < KS) && e < e_end;
#pragma unroll
    for (int m = 0; m < NO; ++m) id[m] = (m < nother && in) ? __ldg(p.idx[m] + e) : 0u;
    vs = !in ? 0xffffffffu : p.vsrc ? __ldg(p.vsrc + e) : e;
  };
  auto issue = [&](int t) {  // copies of step t: values and rows (positions past the unit: row 0, not read)
    const uint32_t st = ring_s + (uint32_t)(t & 1) * (uint32_t)KS * (uint32_t)RS * 4u;
    if (vs != 0xffffffffu) tile_cp4(ring_s + (uint32_t)(2 * KS * RS + KS * (t & 1) + lane) * 4u, p.val + vs);
#pragma unroll
    for (int m = 0; m < NO; ++m) {
      if (m >= nother) break;
      const int lq = p.lq[m], z0 = lane >> lq, c = lane & ((1 << lq) - 1), dz = 32 >> lq;
      const float *U = p.U[m] + 4 * c;
      uint32_t dst = st + (uint32_t)(z0 * RS + p.off[m] + 4 * c) * 4u;
      const uint32_t step = (uint32_t)(dz * RS) * 4u;
      const int rounds = KS == 32 ? 1 << lq : 1 << (lq - 1);  // (KS = 16: rows of two pieces and more)
#pragma unroll 4
      for (int i = 0; i < rounds; ++i, dst += step) {
        const uint32_t r = __shfl_sync(kAll, id[m], z0 + i * dz);
        tile_cp16(dst, U + ((size_t)r << (lq + 2)));
      }
    }
    tile_commit();
  };

  TileAcc<TA, TB> acc;
  acc.clear();
  TileAcc<TA, TB> qt;  // ADJ: this lane's tile of the slice's row of Q
  bool fresh = true;   //      not loaded yet
  double sq = 0.0;  // in FP64: the squares of FP32 residuals leave FP32's range
  uint32_t kb = __ldg(p.unit_k0 + u);
  uint32_t bound = (kb + 1u + lane <= p.S) ? __ldg(p.sptr + kb + 1u + lane) : 0xffffffffu;
  load_ids(0);
  issue(0);
  if (ntiles > 1) load_ids(1);

  for (int t = 0; t < ntiles; ++t) {
    const uint32_t e = e0 + (uint32_t)KS * (uint32_t)t;
    const int nt = (int)min((uint32_t)KS, e_end - e);
    // slices of this step: bit q of `starts` is set where position q >= 1 starts one
    const uint32_t q = bound - e;
    uint32_t starts = __reduce_or_sync(kAll, q < 32u ? (1u << q) : 0u);
    starts &= (nt >= 32) ? kAll : ((1u << nt) - 1u);
    const bool end_is_start = __any_sync(kAll, q == (uint32_t)nt);
    const uint32_t kb_next = kb + __popc(__ballot_sync(kAll, q <= (uint32_t)nt));
    bound = (kb_next + 1u + lane <= p.S) ? __ldg(p.sptr + kb_next + 1u + lane) : 0xffffffffu;
    if (t + 1 < ntiles) {
      issue(t + 1);
      if (t + 2 < ntiles) load_ids(t + 2);
      tile_wait<1>();
    } else {
      tile_wait<0>();
    }
    __syncwarp();
    uint32_t eo = e + (uint32_t)lane;
    if (ADJ && p.esrc && lane < nt) eo = __ldg(p.esrc + eo);
    const uint32_t st = ring_s + (uint32_t)((t & 1) * KS * RS) * 4u;
    const uint32_t xs = ring_s + (uint32_t)(2 * KS * RS + KS * (t & 1)) * 4u;
    uint32_t segs = starts | 1u;
    uint32_t kseg = kb;
    while (segs) {
      const int p0 = __ffs(segs) - 1;
      segs &= segs - 1u;
      const int p1 = segs ? (__ffs(segs) - 1) : nt;
      if constexpr (ADJ) {
        if (fresh) {
          const float *Q = p.Q + (size_t)__ldg(p.sid + kseg) * (size_t)(TA * TB * Gw) + lane % Gw;
          qt.load([&](int i) { return __ldg(Q + i * Gw); });
          fresh = false;
        }
        for (int z0 = p0; z0 < p1; z0 += NG) {
          const int z = min(z0 + g, p1 - 1);  // past the slice: its last position, with no residual
          const uint32_t rec = st + (uint32_t)(z * RS) * 4u;
          float lead_s = 1.f;
          if constexpr (NO > 2) {
#pragma unroll
            for (int m = 2; m < NO; ++m)
              if (m < nother) lead_s *= tile_lds1(rec + loff[m - 2]);
          }
          float av[TA], bv[TB];
          if constexpr (NO == 1)
            av[0] = 1.f;
          else
            tile_lds<TA>(rec + aoff, hopA, av);
          tile_lds<TB>(rec + boff, hopB, bv);
          const float x = tile_lds1(xs + (uint32_t)z * 4u);
          float xhat = lead_s * qt.dot(av, bv);
          for (int o = 1; o < Gw; o <<= 1) xhat += __shfl_xor_sync(kAll, xhat, o);
          const bool in = z0 + g < p1;
          const float r = in ? xhat - x : 0.f;
          acc.add(lead_s * r, av, bv);
          // (its value is no longer read: groups past the slice ignore what they read there)
          if (in && lane % Gw == 0) asm volatile("st.shared.f32 [%0], %1;" ::"r"(xs + (uint32_t)z * 4u), "f"(r) : "memory");
        }
      } else if (g < NG) {
        const uint32_t rec = st + (uint32_t)((p0 + g) * RS) * 4u, adv = (uint32_t)(NG * RS) * 4u;
        uint32_t at_x = xs + (uint32_t)(p0 + g) * 4u, at_a = rec + aoff, at_b = rec + boff;
        uint32_t at_l[NO > 2 ? NO - 2 : 1];
        if constexpr (NO > 2) {
#pragma unroll
          for (int m = 2; m < NO; ++m) at_l[m - 2] = rec + loff[m - 2];
        }
#pragma unroll 1
        for (int left = p1 - p0 - g; left > 0; left -= NG) {
          float s = tile_lds1(at_x);
          if constexpr (NO > 2) {
#pragma unroll
            for (int m = 2; m < NO; ++m)
              if (m < nother) {
                s *= tile_lds1(at_l[m - 2]);
                at_l[m - 2] += adv;
              }
          }
          float av[TA], bv[TB];
          if constexpr (NO == 1)
            av[0] = 1.f;
          else
            tile_lds<TA>(at_a, hopA, av);
          tile_lds<TB>(at_b, hopB, bv);
          acc.add(s, av, bv);
          at_x += (uint32_t)NG * 4u;
          at_a += adv;
          at_b += adv;
        }
      }
      __syncwarp();
      const bool flush = (p1 < nt) || end_is_start || (e + (uint32_t)nt == e_end);
      if (flush) {
        const int slot = __ldg(p.unit_slot + u);
        float *dst = (slot >= 0) ? p.carry + (size_t)slot * p.P : p.Y + (size_t)__ldg(p.sid + kseg) * p.P;
        constexpr int LD = tile_row_stride(TB);
#pragma unroll
        for (int a = 0; a < TA; ++a) {
          if (a >= p.cA) break;
          float v[TB];
          acc.row(a, v);
          float *mine = rows + lane * LD;
          *reinterpret_cast<float4 *>(mine) = make_float4(v[0], v[1], v[2], v[3]);
          if constexpr (TB == 5) mine[4] = v[4];
          if constexpr (TB == 6) *reinterpret_cast<float2 *>(mine + 4) = make_float2(v[4], v[5]);
          if constexpr (TB >= 7)
            *reinterpret_cast<float4 *>(mine + 4) = make_float4(v[4], v[5], v[6], TB == 8 ? v[TB - 1] : 0.f);
          __syncwarp();
          const int skip = a + (a >= 4 ? p.jA : 0);
#pragma unroll 1
          for (int o = lane; o < Gw * TB; o += 32) {
            const float *at = rows + o / TB * LD + o % TB;
            float sum = at[0];
            for (int h = 1; h < NG; ++h) sum += at[h * Gw * LD];
            const int2 pl = place[o];
            const int r = pl.y + skip;
            if (r >= 0 && r < R1) dst[pl.x + r * R0] = sum;
          }
          __syncwarp();
        }
        acc.clear();
        fresh = true;
      }
      ++kseg;
    }
    __syncwarp();
    if constexpr (ADJ) {
      if (lane < nt) {
        const float r = tile_lds1(xs + (uint32_t)lane * 4u);
        p.e_out[eo] = r;
        const double rd = f2d_exact(r);
        sq = fma(rd, rd, sq);
      }
      __syncwarp();  // read before the next step's values are copied there
    }
    kb = kb_next;
  }
  if constexpr (ADJ) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) sq += __shfl_xor_sync(kAll, sq, o);
    if (lane == 0) p.sq_part[u] = sq;
  }
}

constexpr size_t kTileSmem = 227 * 1024;  // shared memory a block may have

template <int NO, int TA, int TB, bool ADJ = false>
static cudaError_t run_tile(TileParams &p, int num_sms, cudaStream_t s) {
  auto kern = ttmc_tile_kernel<NO, TA, TB, ADJ>;
  int KS = 32;
  // Order 3: 16 where the records are so wide (21 KB a warp for two steps of 32 records of 64
  // floats) that an SM holds two blocks at most.  1M nonzeros, three modes: ranks 29^3 491 -> 391 us,
  // 7 x 30 x 30 337 -> 272; where three blocks fit it loses (600,011, 12 x 7 x 20: 111 -> 127).
  if constexpr (NO == 2)
    if (p.lq[0] > 0 && p.lq[1] > 0 &&
        kTileSmem / (kTileWarps * sizeof(float) * (size_t)tile_warp_floats(p.RS, TB, 32) + 1024) < 3) {
      KS = 16;
      kern = ttmc_tile_kernel<NO, TA, TB, ADJ, 16>;
    }
  const size_t per = (size_t)tile_warp_floats(p.RS, TB, KS) * sizeof(float);
  const int most = (int)std::min<size_t>(kTileWarps, kTileSmem / per);
  if (most < 1) return cudaErrorInvalidConfiguration;
  // small tensors: one warp per block reaches every SM
  const int W = (int)std::max<int64_t>(1, std::min<int64_t>(most, p.n_units / num_sms));
  // the most a block may have, not this launch's: the attribute is the function's, and a call on
  // another context may set it between here and the launch
  const cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kTileSmem);
  if (e != cudaSuccess) return e;
  const dim3 grid((unsigned)((p.n_units + W - 1) / W), (unsigned)((p.G + 31) / 32));
  kern<<<grid, 32 * W, per * W, s>>>(p);
  ::tk::count_launch();
  return cudaGetLastError();
}

cudaError_t tile_dispatch_n(int TA, int TB, TileParams &p, int num_sms, cudaStream_t s);    // ttmc_tile_n.cu
cudaError_t tile_dispatch_adj(int TA, int TB, TileParams &p, int num_sms, cudaStream_t s);  // ttmc_tile_adj.cu
bool tile_adj_covers(int TA, int TB, int nother);

}  // namespace tk

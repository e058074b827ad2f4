// Backward pass through the segment aggregation for batches with at most one candidate per user (bf16 inputs): what the
// tensor-core forward path does with such batches (laser_stream.cu) carried over to the gradients.  With one target per
// user neither the keys and values of the items nor their gradients have to exist.  With
//
//   u_h     = W_k[:, h] (t W_q)_h / gamma                 the score of item n is x_n . u_h
//   r_{i,h} = sum_{n in segment i} g_{n,h} x_n            s_i[h] = r_{i,h} W_v[:, h]
//   y_{i,h} = W_v[:, h] ds_i[h]                           dg_{n,h} = x_n . y_{i,h}
//   de      = dg g (1 - g),   p_h = sum_n de_{n,h} x_n
//
// the chain rule through Eq. 8-12 becomes
//
//   dx_n = sum_h de_{n,h} u_h + g_{n,h} y_{i,h},   dW_v[:, h] = sum_{u,i} r_{i,h}^T ds_i[h],
//   d(q_h / gamma) = p_h W_k[:, h],                dW_k[:, h] = sum_u p_h^T q_h / gamma
//
// so a batch costs two passes over the item rows and one over the rows of d_items; every other array has one row per
// (user, segment).  Kernels:
//   bs_fwd_kernel     items -> r [N, Lp, H, d]            (warp per segment, 16 rows per step)
//   bs_rows_kernel    s = r W_v, or y = ds W_v^T          (warp per 16 segments of a user)
//   bs_bwd_kernel     items, u, y -> d_items, p [N, H, d]
//   bs_wv_kernel      dW_v
// fp32 values enter the bf16 MMAs as high and low parts (about 16 bits, more than the TF32 operands of the products around
// them); item rows and weights are bf16 already.
// Bound by HBM: at 2048 users of 200 .. 1000 items, d = 128, 2 heads, segments of 10, the two passes, d_items and the
// per-segment arrays are about 2.5 GB.
#include <algorithm>

#include "laser_common.cuh"
#include "laser_mma.cuh"

namespace laser {
namespace {

using bf16 = __nv_bfloat16;
using namespace mma;

constexpr int kBW = 4;             // warps per block
constexpr int kBThreads = kBW * 32;
constexpr int kBRows = 16;         // item rows per step (one MMA tile)
constexpr int kBStages = 3;        // ring depth per warp
constexpr int kSlotPitch = 48;     // bytes per row of the [slot][item] gate tile (conflict-free ldmatrix)

struct BsParams {
  int U, L, d, H, S, Lp, N;
  const bf16 *items, *Wv;
  const int *lengths, *cand_offsets, *order;
  const float* u;                  // [U, H, d]
  float *r, *s, *y, *p;            // [N, Lp, H, d], [N, Lp, d] (null: s_hi, s_lo), [N, Lp, H, d], [N, H, d]
  bf16 *s_hi, *s_lo;               // H' as bf16 high and low parts, [N, Lp, d] each, instead of s
  const float* ds;                 // [N, Lp, d]
  float *d_items, *dWv;
  int* status;
};

// Candidate of user u (-1: none, or invalid inputs, which are reported) and the user's valid items.
__device__ __forceinline__ int one_candidate(const BsParams& P, int c0, int c1, int len, int* len_out) {
  if (c0 < 0 || c1 < c0 || c1 > P.N || c1 - c0 > 1 || len < 0 || len > P.L) {
    report_status(P.status, LASER_ERR_BAD_INPUT);
    return -1;
  }
  *len_out = len;
  return c1 > c0 ? c0 : -1;
}
__device__ __forceinline__ int one_candidate(const BsParams& P, int u, int* len_out) {
  return one_candidate(P, P.cand_offsets[u], P.cand_offsets[u + 1], P.lengths[u], len_out);
}

__device__ __forceinline__ float gate_of(float x) {
  // 1 / (1 + 2^(-x log2 e)); relative error about 1e-7 per step, an overflowing exponential gives exactly 0
  float e, r;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(e) : "f"(x * -1.4426950408889634f));
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(1.f + e));
  return r;
}

// A fragments (rows h: high parts, rows h + 8: low parts) of the H vectors of d floats at v.
template <int D16>
__device__ __forceinline__ void split_rows(uint32_t (&a)[D16][4], const float* v, int H, int g, int t) {
#pragma unroll
  for (int kt = 0; kt < D16; ++kt) {
    a[kt][0] = a[kt][1] = a[kt][2] = a[kt][3] = 0u;
    if (g < H) {
      const float2 x0 = *reinterpret_cast<const float2*>(v + (size_t)g * 16 * D16 + kt * 16 + 2 * t);
      const float2 x1 = *reinterpret_cast<const float2*>(v + (size_t)g * 16 * D16 + kt * 16 + 2 * t + 8);
      a[kt][0] = pack2(x0.x, x0.y);
      a[kt][1] = pack2(x0.x - bf16_lo(a[kt][0]), x0.y - bf16_hi(a[kt][0]));
      a[kt][2] = pack2(x1.x, x1.y);
      a[kt][3] = pack2(x1.x - bf16_lo(a[kt][2]), x1.y - bf16_hi(a[kt][2]));
    }
  }
}

// A warp's private ring over the rows of its segments (every `stride`-th one of a user), kBRows rows per stage
// (rows past the segment are zeros); a stage that opens a segment also brings `y_bytes` of that segment's y vectors.
template <int D16>
struct RowRing {
  static constexpr int d = 16 * D16, RS = 2 * d + 16;      // bytes per staged row (padded: conflict-free ldmatrix)
  uint32_t base, stage_bytes;
  const bf16* x;                   // the user's rows
  const char* y;                   // the user's y vectors, y_bytes per segment (null: none)
  int y_bytes, len, S, nv, seg, stride, grp, lane;
  bool live;
  __device__ __forceinline__ int groups(int sg) const { return (min(S, len - sg * S) + kBRows - 1) / kBRows; }
  __device__ __forceinline__ void issue(int stage, const bf16* any) {
    if (live) {
      const uint32_t dst = base + stage * stage_bytes;
      const int n0 = seg * S + grp * kBRows, rows = min((seg + 1) * S, len) - n0;
      const bf16* src = x + (size_t)n0 * d;
#pragma unroll
      for (int i = 0; i < D16; ++i) {
        const int piece = i * 32 + lane, row = piece / (2 * D16), q = piece - row * (2 * D16);
        const bool ok = row < rows;
        cp16(dst + row * RS + q * 16, ok ? (const void*)(src + row * d + q * 8) : (const void*)any, ok ? 16u : 0u);
      }
      if (y && grp == 0)
        for (int b = lane * 16; b < y_bytes; b += 512) cp16(dst + kBRows * RS + b, y + (size_t)seg * y_bytes + b, 16u);
      if (++grp >= groups(seg)) {
        grp = 0;
        seg += stride;
        live = seg < nv;
      }
    }
    cp_commit();
  }
};

// r_{i,h} = sum of g_{n,h} x_n over the items of segment i (Eq. 10-12 before the value projection), fp32.
template <int D16>
__global__ void __launch_bounds__(kBThreads) bs_fwd_kernel(BsParams P) {
  constexpr int d = 16 * D16, RS = RowRing<D16>::RS;
  extern __shared__ __align__(128) uint8_t smem[];
  chain_wait();
  chain_release();
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3, H = P.H;
  const int u = P.order ? min(max(P.order[blockIdx.x], 0), P.U - 1) : (int)blockIdx.x;
  int len = 0;
  const int cand = one_candidate(P, u, &len);
  const int nv = (len + P.S - 1) / P.S;
  // gridDim.y blocks share a user, warp by warp (batches of few, long users)
  const int seg0 = blockIdx.y * kBW + warp, stride = kBW * gridDim.y;
  if (cand < 0 || seg0 >= nv) return;                       // (no block-wide barrier below)
  uint32_t ua[D16][4];
  split_rows<D16>(ua, P.u + (size_t)u * H * d, H, g, t);
  RowRing<D16> ring;
  ring.stage_bytes = kBRows * RS;
  ring.base = smem_addr(smem) + warp * kBStages * ring.stage_bytes;
  ring.x = P.items + (size_t)u * P.L * d;
  ring.y = nullptr; ring.y_bytes = 0;
  ring.len = len; ring.S = P.S; ring.nv = nv; ring.seg = seg0; ring.stride = stride;
  ring.grp = 0; ring.lane = lane; ring.live = true;
#pragma unroll
  for (int s = 0; s < kBStages - 1; ++s) ring.issue(s, P.items);
  int stage = 0;
  const uint32_t off1 = ((lane & 7) + ((lane >> 4) & 1) * 8) * RS + ((lane >> 3) & 1) * 16;   // [item][k] operand
  const uint32_t off2 = ((lane & 7) + ((lane >> 3) & 1) * 8) * RS + (lane >> 4) * 16;         // [item][col], transposed
  for (int seg = seg0; seg < nv; seg += stride) {
    float racc[2 * D16][4];
#pragma unroll
    for (int j = 0; j < 2 * D16; ++j) racc[j][0] = racc[j][1] = racc[j][2] = racc[j][3] = 0.f;
    const int ngrp = ring.groups(seg);
    for (int grp = 0; grp < ngrp; ++grp) {
      cp_wait<kBStages - 2>();
      __syncwarp();
      ring.issue(stage ? stage - 1 : kBStages - 1, P.items);
      const uint32_t sb = ring.base + stage * ring.stage_bytes;
      float sc[2][4] = {};
#pragma unroll
      for (int kt = 0; kt < D16; ++kt) {
        uint32_t b[4];
        ldsm_x4(b, sb + off1 + kt * 32);
        mma16816(sc[0], ua[kt][0], ua[kt][1], ua[kt][2], ua[kt][3], b[0], b[1]);
        mma16816(sc[1], ua[kt][0], ua[kt][1], ua[kt][2], ua[kt][3], b[2], b[3]);
      }
      uint32_t ga[4] = {0u, 0u, 0u, 0u};                    // (a zero row has gate 1/2 and adds 1/2 * 0)
      if (g < H) {
#pragma unroll
        for (int nt = 0; nt < 2; ++nt) {
          const float g0 = gate_of(sc[nt][0] + sc[nt][2]), g1 = gate_of(sc[nt][1] + sc[nt][3]);
          ga[2 * nt] = pack2(g0, g1);
          ga[2 * nt + 1] = pack2(g0 - bf16_lo(ga[2 * nt]), g1 - bf16_hi(ga[2 * nt]));
        }
      }
#pragma unroll
      for (int jp = 0; jp < D16; ++jp) {
        uint32_t b[4];
        ldsm_x4_t(b, sb + off2 + jp * 32);
        mma16816(racc[2 * jp], ga[0], ga[1], ga[2], ga[3], b[0], b[1]);
        mma16816(racc[2 * jp + 1], ga[0], ga[1], ga[2], ga[3], b[2], b[3]);
      }
      if (++stage == kBStages) stage = 0;
    }
    if (g < H) {
      float* out = P.r + (((size_t)cand * P.Lp + seg) * H + g) * d + 2 * t;
#pragma unroll
      for (int j = 0; j < 2 * D16; ++j)
        *reinterpret_cast<float2*>(out + j * 8) = make_float2(racc[j][0] + racc[j][2], racc[j][1] + racc[j][3]);
    }
  }
  cp_wait<0>();
}

// One product per (segment row, head) with a slice of W_v (staged once per block): to_y = 0: s[h] = r_h W_v[:, h]
// (K = d, d / H columns); to_y = 1: y_h = ds[h] W_v[:, h]^T (K = d / H, d columns).  A warp takes one head of 16
// segments of a user.
//
// A job is (16-segment tile, user, head), tiles slowest and users in the launch order (longest first): the tiles that exist
// are the first ones of each tile index, so the warps' shares are equal to within a job.  Candidate and segment count of a
// user are two dependent round trips to memory in front of the rows' own, unless the block fills a table of them first
// (tabled; see launch_rows).

// (NPC: the most column pairs a head has; KA: k-tiles requested together.  Half a matrix of columns at most leaves the
// registers for all of a row tile's k-tiles: r -> s 68 -> 58 us, with the high and low products interleaved.)
template <int D16, int NPC, int KA, bool to_y>
__global__ void __launch_bounds__(256, 2) bs_rows_kernel(BsParams P, int tabled) {
  constexpr int d = 16 * D16, WS = 2 * d + 16;
  extern __shared__ __align__(128) uint8_t smem[];
  int2* table = reinterpret_cast<int2*>(smem + d * WS);     // (candidate, segments) by launch position
  chain_wait();
  chain_release();
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, g = lane >> 2, t = lane & 3, H = P.H, dvh = d / H;
  for (int i = tid; i < d * 2 * D16; i += 256) {
    const int row = i / (2 * D16), q = i - row * (2 * D16);
    cp16(smem_addr(smem) + row * WS + q * 16, P.Wv + (size_t)row * d + q * 8, 16u);
  }
  cp_commit();
  auto look_up = [&](int pos) {
    int len = 0;
    const int cand = one_candidate(P, P.order ? min(max(P.order[pos], 0), P.U - 1) : pos, &len);
    return make_int2(cand, cand >= 0 ? (len + P.S - 1) / P.S : 0);
  };
  if (tabled)
    for (int i = tid; i < P.U; i += 256) table[i] = look_up(i);
  cp_wait<0>();
  __syncthreads();
  const int tiles = (P.Lp + 15) >> 4, stride = gridDim.x * 8;
  const uint32_t w = smem_addr(smem);
  const int mi = lane >> 3, lr = lane & 7;
  // cursor (tile, position, head) instead of a job number: no divisions
  const int step_h = stride % H, step_pos = stride / H;
  int tile = 0, pos = (blockIdx.x * 8 + warp) / H, h = (blockIdx.x * 8 + warp) % H;
  for (;; h += step_h, pos += step_pos + (h >= H), h -= h >= H ? H : 0) {
    while (pos >= P.U) pos -= P.U, ++tile;
    if (tile >= tiles) break;
    const int i0 = tile * 16;
    const int2 user = tabled ? table[pos] : look_up(pos);
    const int cand = user.x, rows = user.y - i0;
    if (rows <= 0) continue;
    const size_t row0 = (size_t)cand * P.Lp + i0;
    {
      const float* A = to_y ? P.ds + row0 * d + h * dvh : P.r + (row0 * H + h) * d;
      float* C = to_y ? P.y + (row0 * H + h) * d : P.s + row0 * d + h * dvh;
      const size_t lda = to_y ? d : (size_t)H * d, ldc = to_y ? (size_t)H * d : d;
      const int KT = to_y ? dvh >> 4 : D16, NP = to_y ? D16 : dvh >> 4;      // 16-wide steps of K, pairs of column tiles
      float acc[2 * NPC][4];
#pragma unroll
      for (int j = 0; j < 2 * NPC; ++j) acc[j][0] = acc[j][1] = acc[j][2] = acc[j][3] = 0.f;
      // A several k-tiles at a time, all of their loads in flight together (one tile at a time, each with its own round trip to
      // memory, took 107 us for r -> s and 80 us for ds -> y at 2048 users of 61 segments, d = 128)
      constexpr int kAhead = D16 < KA ? D16 : KA;
#pragma unroll 1
      for (int k0 = 0; k0 < KT; k0 += kAhead) {
        float2 x[kAhead][4];
#pragma unroll
        for (int k = 0; k < kAhead; ++k)
#pragma unroll
          for (int e = 0; e < 4; ++e) {
            const int rr = g + (e & 1) * 8;
            x[k][e] = rr < rows && k0 + k < KT
                          ? *reinterpret_cast<const float2*>(A + rr * lda + (k0 + k) * 16 + (e >> 1) * 8 + 2 * t)
                          : make_float2(0.f, 0.f);
          }
#pragma unroll
        for (int k = 0; k < kAhead; ++k) {
          if (k0 + k >= KT) break;
          const int kt = k0 + k;
          uint32_t hi[4], lo[4];
#pragma unroll
          for (int e = 0; e < 4; ++e) {
            hi[e] = pack2(x[k][e].x, x[k][e].y);
            lo[e] = pack2(x[k][e].x - bf16_lo(hi[e]), x[k][e].y - bf16_hi(hi[e]));
          }
#pragma unroll
          for (int np = 0; np < NPC; ++np) {
            if (np >= NP) break;
            uint32_t b[4];
            if (to_y) ldsm_x4(b, w + (np * 16 + (mi >> 1) * 8 + lr) * WS + (h * dvh + kt * 16 + (mi & 1) * 8) * 2);
            else ldsm_x4_t(b, w + (kt * 16 + (mi & 1) * 8 + lr) * WS + (h * dvh + np * 16 + (mi >> 1) * 8) * 2);
            mma16816(acc[2 * np], hi[0], hi[1], hi[2], hi[3], b[0], b[1]);
            mma16816(acc[2 * np + 1], hi[0], hi[1], hi[2], hi[3], b[2], b[3]);
            mma16816(acc[2 * np], lo[0], lo[1], lo[2], lo[3], b[0], b[1]);
            mma16816(acc[2 * np + 1], lo[0], lo[1], lo[2], lo[3], b[2], b[3]);
          }
        }
      }
#pragma unroll
      for (int j = 0; j < 2 * NPC; ++j) {
        if (j >= 2 * NP) break;
        if (!to_y && !P.s) {
#pragma unroll
          for (int hf = 0; hf < 2; ++hf)
            if (g + 8 * hf < rows) {
              const size_t at = (row0 + g + 8 * hf) * d + h * dvh + j * 8 + 2 * t;
              const uint32_t hi = pack2(acc[j][2 * hf], acc[j][2 * hf + 1]);
              *reinterpret_cast<uint32_t*>(P.s_hi + at) = hi;
              *reinterpret_cast<uint32_t*>(P.s_lo + at) = pack2(acc[j][2 * hf] - bf16_lo(hi), acc[j][2 * hf + 1] - bf16_hi(hi));
            }
          continue;
        }
        if (g < rows) *reinterpret_cast<float2*>(C + g * ldc + j * 8 + 2 * t) = make_float2(acc[j][0], acc[j][1]);
        if (g + 8 < rows) *reinterpret_cast<float2*>(C + (g + 8) * ldc + j * 8 + 2 * t) = make_float2(acc[j][2], acc[j][3]);
      }
    }
  }
}

// Second pass over the items.  Per 16 rows: scores and x_n . y_{i,h} (A operands: u and y, high / low rows), then
// p_h += de x (as r in the forward pass) and dx = de u + g y as one product over slots: with two bf16 parts per factor the
// terms are (de, g)_high (u, y)_high + (de, g)_low (u, y)_high + (de, g)_high (u, y)_low, i.e. 6 H slots of the MMA's
// contraction index, padded to KS 16-slot steps.  The gates of the step go through a small [slot][item] tile in shared
// memory (their accumulators have the heads on the rows, the product wants the items there).
template <int D16>
__global__ void __launch_bounds__(kBThreads, 3) bs_bwd_kernel(BsParams P, int KS, int warp_bytes) {
  constexpr int d = 16 * D16, RS = RowRing<D16>::RS;
  extern __shared__ __align__(128) uint8_t smem[];
  chain_wait();
  chain_release();
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, g = lane >> 2, t = lane & 3, H = P.H;
  const int u = P.order ? min(max(P.order[blockIdx.x], 0), P.U - 1) : (int)blockIdx.x;
  int len = 0;
  const int cand = one_candidate(P, u, &len);
  {                                                         // rows that receive no gradient (all of them without a candidate)
    const int live = cand >= 0 ? len : 0, parts = gridDim.y;
    float4* out = reinterpret_cast<float4*>(P.d_items + ((size_t)u * P.L + live) * d);
    const long long n = (long long)(P.L - live) * (d / 4);
    for (long long i = blockIdx.y * kBThreads + tid; i < n; i += parts * kBThreads) out[i] = make_float4(0.f, 0.f, 0.f, 0.f);
  }
  if (cand < 0) return;
  const int nv = (len + P.S - 1) / P.S;
  uint8_t* mine = smem + (size_t)warp * warp_bytes;
  RowRing<D16> ring;
  ring.stage_bytes = kBRows * RS + H * d * 4;
  ring.base = smem_addr(mine);
  ring.x = P.items + (size_t)u * P.L * d;
  ring.y = reinterpret_cast<const char*>(P.y + (size_t)cand * P.Lp * H * d);
  ring.y_bytes = H * d * 4;
  ring.len = len; ring.S = P.S; ring.nv = nv; ring.seg = blockIdx.y * kBW + warp; ring.stride = kBW * gridDim.y;
  ring.grp = 0; ring.lane = lane; ring.live = ring.seg < nv;
  uint8_t* rows = mine + kBStages * ring.stage_bytes;       // u high [H], y high [H], u low [H], y low [H]
  uint8_t* tile = rows + 4 * H * RS;                        // [16 KS] slots of 16 items
  uint8_t* zero = smem + (size_t)kBW * warp_bytes;          // a zero row, one per block (two heads at d = 128: a third block fits)
  const int seg0 = ring.seg, stride = ring.stride;
#pragma unroll
  for (int s = 0; s < kBStages - 1; ++s) ring.issue(s, P.items);

  // set-up: u as A fragments and as slot rows, zero row, unused slots of the gate tile
  uint32_t ua[D16][4];
  split_rows<D16>(ua, P.u + (size_t)u * H * d, H, g, t);
  if (g < H) {
#pragma unroll
    for (int kt = 0; kt < D16; ++kt) {
      uint8_t* dst = rows + g * RS + kt * 32 + 4 * t;
      *reinterpret_cast<uint32_t*>(dst) = ua[kt][0];
      *reinterpret_cast<uint32_t*>(dst + 16) = ua[kt][2];
      *reinterpret_cast<uint32_t*>(dst + 2 * H * RS) = ua[kt][1];
      *reinterpret_cast<uint32_t*>(dst + 2 * H * RS + 16) = ua[kt][3];
    }
  }
  for (int i = lane; i < RS / 4; i += 32) reinterpret_cast<uint32_t*>(zero)[i] = 0u;      // (every warp: the same zeros)
  for (int i = lane; i < 16 * KS * kSlotPitch / 4; i += 32) reinterpret_cast<uint32_t*>(tile)[i] = 0u;
  __syncwarp();

  const int mi = lane >> 3, lr = lane & 7;
  const uint32_t rows_a = smem_addr(rows), tile_a = smem_addr(tile);
  const uint32_t off1 = ((lane & 7) + ((lane >> 4) & 1) * 8) * RS + ((lane >> 3) & 1) * 16;   // [item][k] operand
  const uint32_t off2 = ((lane & 7) + ((lane >> 3) & 1) * 8) * RS + (lane >> 4) * 16;         // [item][col], transposed
  // y as an A operand: rows 0-7 high parts, rows 8-15 low parts, heads past H read the zero row
  const uint32_t zero_a = smem_addr(zero);
  const uint32_t y_row = (lr < H ? rows_a + (((mi & 1) ? 3 * H : H) + lr) * RS : zero_a) + (mi >> 1) * 16;
  uint32_t slot_row[3];                                     // this lane's row of the slot operand, per 16-slot step
#pragma unroll
  for (int ks = 0; ks < 3; ++ks) {
    const int s = ks * 16 + (mi & 1) * 8 + lr;
    slot_row[ks] = (s >= 6 * H ? zero_a : rows_a + (s < 2 * H ? s : s - 2 * H) * RS) + (mi >> 1) * 16;
  }
  const uint32_t tile_ld = tile_a + ((mi >> 1) * 8 + lr) * kSlotPitch + (mi & 1) * 16;
  uint8_t* tile_st = tile + g * kSlotPitch + 4 * t;

  float pacc[2 * D16][4];
#pragma unroll
  for (int j = 0; j < 2 * D16; ++j) pacc[j][0] = pacc[j][1] = pacc[j][2] = pacc[j][3] = 0.f;
  int stage = 0;
  for (int seg = seg0; seg < nv; seg += stride) {
    const int ngrp = ring.groups(seg), n_end = min((seg + 1) * P.S, len);
    for (int grp = 0; grp < ngrp; ++grp) {
      cp_wait<kBStages - 2>();
      __syncwarp();
      const uint32_t sb = ring.base + stage * ring.stage_bytes;
      if (grp == 0) {                                       // the segment's y vectors as bf16 parts (4 floats per lane and step)
        const uint8_t* ys = mine + stage * ring.stage_bytes + kBRows * RS;
        for (int i = lane; i < H * (d / 4); i += 32) {
          const int h = i / (d / 4), c = i - h * (d / 4);
          const float4 v = *reinterpret_cast<const float4*>(ys + i * 16);
          const uint32_t h0 = pack2(v.x, v.y), h1 = pack2(v.z, v.w);
          *reinterpret_cast<uint2*>(rows + (H + h) * RS + c * 8) = make_uint2(h0, h1);
          *reinterpret_cast<uint2*>(rows + (3 * H + h) * RS + c * 8) =
              make_uint2(pack2(v.x - bf16_lo(h0), v.y - bf16_hi(h0)), pack2(v.z - bf16_lo(h1), v.w - bf16_hi(h1)));
        }
        __syncwarp();
      }
      ring.issue(stage ? stage - 1 : kBStages - 1, P.items);
      float sc[2][4] = {}, dg[2][4] = {};
#pragma unroll
      for (int kt = 0; kt < D16; ++kt) {
        uint32_t b[4], a[4];
        ldsm_x4(b, sb + off1 + kt * 32);
        ldsm_x4(a, y_row + kt * 32);
        mma16816(sc[0], ua[kt][0], ua[kt][1], ua[kt][2], ua[kt][3], b[0], b[1]);
        mma16816(sc[1], ua[kt][0], ua[kt][1], ua[kt][2], ua[kt][3], b[2], b[3]);
        mma16816(dg[0], a[0], a[1], a[2], a[3], b[0], b[1]);
        mma16816(dg[1], a[0], a[1], a[2], a[3], b[2], b[3]);
      }
      uint32_t ea[4] = {0u, 0u, 0u, 0u};
      if (g < H) {
#pragma unroll
        for (int nt = 0; nt < 2; ++nt) {
          const float g0 = gate_of(sc[nt][0] + sc[nt][2]), g1 = gate_of(sc[nt][1] + sc[nt][3]);
          const float e0 = (dg[nt][0] + dg[nt][2]) * (g0 * (1.f - g0)), e1 = (dg[nt][1] + dg[nt][3]) * (g1 * (1.f - g1));
          const uint32_t gh = pack2(g0, g1), gl = pack2(g0 - bf16_lo(gh), g1 - bf16_hi(gh));
          const uint32_t eh = pack2(e0, e1), el = pack2(e0 - bf16_lo(eh), e1 - bf16_hi(eh));
          ea[2 * nt] = eh;
          ea[2 * nt + 1] = el;
          uint8_t* q = tile_st + nt * 16;
          *reinterpret_cast<uint32_t*>(q) = eh;
          *reinterpret_cast<uint32_t*>(q + H * kSlotPitch) = gh;
          *reinterpret_cast<uint32_t*>(q + 2 * H * kSlotPitch) = el;
          *reinterpret_cast<uint32_t*>(q + 3 * H * kSlotPitch) = gl;
          *reinterpret_cast<uint32_t*>(q + 4 * H * kSlotPitch) = eh;
          *reinterpret_cast<uint32_t*>(q + 5 * H * kSlotPitch) = gh;
        }
      }
      __syncwarp();
#pragma unroll
      for (int jp = 0; jp < D16; ++jp) {                    // p += de x
        uint32_t b[4];
        ldsm_x4_t(b, sb + off2 + jp * 32);
        mma16816(pacc[2 * jp], ea[0], ea[1], ea[2], ea[3], b[0], b[1]);
        mma16816(pacc[2 * jp + 1], ea[0], ea[1], ea[2], ea[3], b[2], b[3]);
      }
      // dx of the 16 rows
      uint32_t A[3][4];
#pragma unroll
      for (int ks = 0; ks < 3; ++ks)
        if (ks < KS) ldsm_x4_t(A[ks], tile_ld + ks * 16 * kSlotPitch);
      const int n0 = seg * P.S + grp * kBRows;
      float* out0 = P.d_items + ((size_t)u * P.L + n0 + g) * d + 2 * t;
      float* out1 = out0 + 8 * d;
      const bool in0 = n0 + g < n_end, in1 = n0 + g + 8 < n_end;
#pragma unroll
      for (int jp = 0; jp < D16; ++jp) {
        float c0[4] = {0.f, 0.f, 0.f, 0.f}, c1[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
        for (int ks = 0; ks < 3; ++ks)
          if (ks < KS) {
            uint32_t b[4];
            ldsm_x4_t(b, slot_row[ks] + jp * 32);
            mma16816(c0, A[ks][0], A[ks][1], A[ks][2], A[ks][3], b[0], b[1]);
            mma16816(c1, A[ks][0], A[ks][1], A[ks][2], A[ks][3], b[2], b[3]);
          }
        if (in0) {
          *reinterpret_cast<float2*>(out0 + jp * 16) = make_float2(c0[0], c0[1]);
          *reinterpret_cast<float2*>(out0 + jp * 16 + 8) = make_float2(c1[0], c1[1]);
        }
        if (in1) {
          *reinterpret_cast<float2*>(out1 + jp * 16) = make_float2(c0[2], c0[3]);
          *reinterpret_cast<float2*>(out1 + jp * 16 + 8) = make_float2(c1[2], c1[3]);
        }
      }
      __syncwarp();                        // the gate tile and the y rows are free again
      if (++stage == kBStages) stage = 0;
    }
  }
  cp_wait<0>();
  __syncthreads();                         // every ring is idle: the warps' sums meet in their places
  float* red = reinterpret_cast<float*>(smem);              // [kBW][H][d]
  if (g < H) {
#pragma unroll
    for (int j = 0; j < 2 * D16; ++j)
      *reinterpret_cast<float2*>(red + ((size_t)warp * H + g) * d + j * 8 + 2 * t) =
          make_float2(pacc[j][0] + pacc[j][2], pacc[j][1] + pacc[j][3]);
  }
  __syncthreads();
  for (int i = tid; i < H * d; i += kBThreads) {
    float v = 0.f;
#pragma unroll
    for (int w = 0; w < kBW; ++w) v += red[(size_t)w * H * d + i];
    float* out = P.p + (size_t)cand * H * d + i;
    if (gridDim.y > 1) atomicAdd(out, v);                   // (p is zero before)
    else *out = v;
  }
}

// dW_v[:, h] += sum over the non-empty segments of r_h^T ds[h]: TF32 MMAs (operands rounded to nearest), fp32 partial sums
// of the whole d x d matrix in a block's registers, one reduction per four elements and block.  The rows of a user's segments
// arrive KR at a time by cp.async in two buffers (r: all heads; ds), zero rows past the user's last segment up to a whole step.
// Bound by shared-memory reads: a warp takes two row tiles x half of the column tiles where their number is even (24 words per
// lane and step for 16 MMAs, rounded as they are read; one row tile x all columns took 40 words and, with a pass that rounded
// the buffers in place, 97 us instead of 68 at 2048 users of 61 segments, d = 128).
__device__ __forceinline__ uint32_t tf32_bits(float v) {
  uint32_t r;
  asm("cvt.rna.tf32.f32 %0, %1;" : "=r"(r) : "f"(v));
  return r;
}
template <int D16>
__global__ void __launch_bounds__(256) bs_wv_kernel(BsParams P, int KR) {
  constexpr int d = 16 * D16, kParts = 8 / D16 > 0 ? 8 / D16 : 1;    // warps that share a row tile split the rows
  extern __shared__ __align__(128) uint8_t smem[];
  chain_wait();
  chain_release();
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, g = lane >> 2, t = lane & 3, H = P.H, dvh = d / H;
  const int pa = H * d + 8, pb = d + 8;                     // row pitches in words (conflict-free fragment reads)
  float* buf0 = reinterpret_cast<float*>(smem);
  const int buf_words = KR * (pa + pb);
  constexpr int kM = D16 % 2 == 0 ? 2 : 1, kN = 2 * D16 / kM;        // row tiles and column tiles of a warp
  const int mtile = warp % (D16 / kM) * kM, n0 = warp % D16 / (D16 / kM) * kN, part = warp / D16;
  const bool active = part < kParts;
  uint32_t starts = 0;                                      // column tiles that open a head (no divisions in the loop)
  for (int h = 0; h < H; ++h) starts |= 1u << (h * (dvh >> 3));
  const int h0 = n0 * 8 / dvh;
  float acc[kM][kN][4];
#pragma unroll
  for (int m = 0; m < kM; ++m)
#pragma unroll
    for (int j = 0; j < kN; ++j) acc[m][j][0] = acc[m][j][1] = acc[m][j][2] = acc[m][j][3] = 0.f;
  // cursor over (user, chunk of KR segments).  Users in the launch order (longest first), dealt to the blocks there and back:
  // every block gets about the same number of segments (in index order the busiest of 296 blocks had 1.4 times the mean).
  // What the next user needs is requested while this one's segments are summed.
  int round = 0, i0 = 0, nv = 0, cand = -1;
  auto user_at = [&](int k) {                               // the k-th user of this block, -1 past the last
    const long long pos = (long long)k * gridDim.x + (k & 1 ? gridDim.x - 1 - blockIdx.x : blockIdx.x);
    return pos >= P.U ? -1 : P.order ? min(max(P.order[pos], 0), P.U - 1) : (int)pos;
  };
  int u1 = user_at(0), u2 = user_at(1), c0 = 0, c1 = 0, len1 = 0;     // the next user with its words, and the one after it
  auto request = [&]() {
    if (u1 >= 0) c0 = P.cand_offsets[u1], c1 = P.cand_offsets[u1 + 1], len1 = P.lengths[u1];
  };
  request();
  auto next = [&]() -> bool {                               // to the next chunk with rows; false past the last
    i0 += KR;
    while (i0 >= nv) {
      if (u1 < 0) return false;
      int len = 0;
      cand = one_candidate(P, c0, c1, len1, &len);
      nv = cand >= 0 ? (len + P.S - 1) / P.S : 0;
      i0 = 0;
      u1 = u2;
      request();
      u2 = user_at(++round + 1);
    }
    return true;
  };
  auto stage = [&](int b) {
    float* A = buf0 + b * buf_words;
    float* B = A + KR * pa;
    const size_t row0 = (size_t)cand * P.Lp + i0;
    const int rows = nv - i0, ca = H * d / 4, cb = d / 4, used = min(KR, (rows + 7) & ~7);
    for (int rr = warp; rr < used; rr += 8) {               // a warp per row: no divisions by the run-time row width
      const uint32_t n = rr < rows ? 16u : 0u;
      const size_t at = row0 + min(rr, rows - 1);
      for (int c = lane; c < ca; c += 32) cp16(smem_addr(A + rr * pa + c * 4), P.r + at * H * d + c * 4, n);
      for (int c = lane; c < cb; c += 32) cp16(smem_addr(B + rr * pb + c * 4), P.ds + at * d + c * 4, n);
    }
  };
  bool have = next();
  if (have) stage(0);
  cp_commit();
  int b = 0;
  while (have) {
    const int used = min(KR, (nv - i0 + 7) & ~7);           // rows of this chunk in whole MMA steps
    have = next();
    if (have) stage(b ^ 1);
    cp_commit();
    cp_wait<1>();
    __syncthreads();
    const float* A = buf0 + b * buf_words;
    const float* B = A + KR * pa;
    if (active)
      for (int k = part * 8; k < used; k += kParts * 8) {
        const float* ap = A + (k + t) * pa + h0 * d + mtile * 16 + g;
        const float* bp = B + (k + t) * pb + n0 * 8 + g;
        uint32_t a[kM][4];
#pragma unroll
        for (int j = 0; j < kN; ++j) {
          const bool opens = j > 0 && (starts >> (n0 + j) & 1u);      // first column tile of the next head
          if (opens) ap += d;
          if (j == 0 || opens)
#pragma unroll
            for (int m = 0; m < kM; ++m)
#pragma unroll
              for (int e = 0; e < 4; ++e) a[m][e] = tf32_bits(ap[(e >> 1) * 4 * pa + m * 16 + (e & 1) * 8]);
          const uint32_t b0 = tf32_bits(bp[j * 8]), b1 = tf32_bits(bp[j * 8 + 4 * pb]);
#pragma unroll
          for (int m = 0; m < kM; ++m)
            asm volatile(
                "mma.sync.aligned.m16n8k8.row.col.f32.tf32.tf32.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
                : "+f"(acc[m][j][0]), "+f"(acc[m][j][1]), "+f"(acc[m][j][2]), "+f"(acc[m][j][3])
                : "r"(a[m][0]), "r"(a[m][1]), "r"(a[m][2]), "r"(a[m][3]), "r"(b0), "r"(b1));
        }
      }
    __syncthreads();
    b ^= 1;
  }
  if (!active) return;
#pragma unroll
  for (int m = 0; m < kM; ++m)
#pragma unroll
    for (int j = 0; j < kN; ++j) red_tile(P.dWv + (size_t)(mtile + m) * 16 * d + (n0 + j) * 8, d, acc[m][j], 1.f, lane);
}

size_t ring_bytes(int d, int H, bool with_y) { return (size_t)kBRows * (2 * d + 16) + (with_y ? (size_t)H * d * 4 : 0); }
int slot_steps(int H) { return (6 * H + 15) / 16; }
size_t bwd_warp_bytes(int d, int H) {
  return (kBStages * ring_bytes(d, H, true) + (size_t)4 * H * (2 * d + 16) + (size_t)16 * slot_steps(H) * kSlotPitch + 127) / 128 * 128;
}
int wv_rows(int d, int H) {                                 // rows per step that keep two buffers within about 100 KB
  const size_t row = 2 * ((size_t)H * d + d + 16) * sizeof(float);
  return row * 32 <= 110 * 1024 ? 32 : row * 16 <= 110 * 1024 ? 16 : 8;
}
// Blocks per user: enough that a batch of few users still fills the GPU, at most one per kBW segments.
int user_parts(const Plan& p) {
  const int want = (4 * device_sms() + p.U - 1) / p.U, most = (p.Lp + kBW - 1) / kBW;
  return std::max(1, std::min(std::min(want, most), 65535));
}

struct BsScratch {
  float *u, *r, *y, *p;
  char* fold;
  size_t total;
};
BsScratch carve_bs(const Plan& p, char* base) {
  BsScratch s;
  size_t off = 0;
  auto take = [&](size_t bytes) {
    char* q = base ? base + off : nullptr;
    off = align_up(off + bytes) + kGuardBytes;
    return q;
  };
  const size_t Hd = (size_t)p.H * p.d;
  s.u = (float*)take((size_t)p.U * Hd * 4);
  s.r = (float*)take((size_t)p.N * p.Lp * Hd * 4);
  s.y = (float*)take((size_t)p.N * p.Lp * Hd * 4);
  s.p = (float*)take((size_t)p.N * Hd * 4);
  s.fold = take(stream_fold_bytes(p));
  s.total = off;
  return s;
}

BsParams bs_params(const Plan& p, const BsScratch& s, const void* items, const int32_t* lengths, const int32_t* cand_offsets,
                   const void* Wv, char* ws) {
  BsParams P = {};
  P.U = p.U; P.L = p.L; P.d = p.d; P.H = p.H; P.S = p.S; P.Lp = p.Lp; P.N = p.N;
  P.items = (const bf16*)items; P.Wv = (const bf16*)Wv;
  P.lengths = lengths; P.cand_offsets = cand_offsets;
  P.order = stream_fold_order(p, s.fold);
  P.u = s.u; P.r = s.r; P.y = s.y; P.p = s.p;
  P.status = reinterpret_cast<int*>(ws + p.off_status);
  return P;
}

template <int D16, int NPC, int KA, bool to_y>
int launch_rows(const Plan& p, const BsParams& P, cudaStream_t st) {
  // A table of the users costs a block U look-ups and saves it one per job, of which it has U tiles H / (2 SMs): whatever the
  // number of users, it pays where a user has many jobs.  Both launches together, without | with it, us: 2 jobs per user (9000
  // users, d = 64) 50 | 87, 8 (4096 users) 72 | 77, 14 (2048 users, d = 128) 117 | 116, 16 (2048 users, d = 64) 70 | 68, 24 (4096
  // users, d = 128) 254 | 226, 28 (1024 users) 95 | 87, 32 (2048 users) 166 | 142.
  constexpr size_t kHalfSm = (228 / 2 - 1) * 1024;          // (two blocks per SM beside each other)
  const int tiles = (p.Lp + 15) / 16;
  const size_t w_bytes = (size_t)p.d * (2 * p.d + 16), table = (size_t)p.U * sizeof(int2);
  const bool tabled = tiles * p.H > 16 && w_bytes + table <= kHalfSm;
  const size_t smem = w_bytes + (tabled ? table : 0);
  const long long jobs = (long long)p.U * tiles * p.H;
  auto kernel = bs_rows_kernel<D16, NPC, KA, to_y>;
  LASER_CUDA_OK(allow_smem(kernel, smem));
  LASER_CUDA_OK(launch_chained(kernel, dim3((unsigned)std::min<long long>((jobs + 7) / 8, 2 * device_sms())), dim3(256), smem, st, P, tabled ? 1 : 0));
  return LASER_OK;
}

template <int D16>
int bs_forward_t(const Plan& p, BsParams P, cudaStream_t st) {
  {
    const size_t smem = kBW * kBStages * ring_bytes(p.d, p.H, false);
    LASER_CUDA_OK(allow_smem(bs_fwd_kernel<D16>, smem));
    LaunchScope ls("bs_fwd", st);
    LASER_CUDA_OK(launch_chained(bs_fwd_kernel<D16>, dim3(p.U, user_parts(p)), dim3(kBThreads), smem, st, P));
  }
  LaunchScope ls("bs_rows_s", st);
  return p.H > 1 ? launch_rows<D16, (D16 + 1) / 2, 8, false>(p, P, st) : launch_rows<D16, D16, 4, false>(p, P, st);
}

template <int D16>
int bs_backward_t(const Plan& p, BsParams P, cudaStream_t st) {
  const int sms = device_sms(), parts = user_parts(p);
  {
    LaunchScope ls("bs_rows_y", st);
    const int rc = launch_rows<D16, D16, 4, true>(p, P, st);
    if (rc != LASER_OK) return rc;
  }
  {
    const int warp_bytes = (int)bwd_warp_bytes(p.d, p.H);
    const size_t smem = (size_t)kBW * warp_bytes + 2 * p.d + 16;
    LASER_CUDA_OK(allow_smem(bs_bwd_kernel<D16>, smem));
    LaunchScope ls("bs_bwd", st);
    LASER_CUDA_OK(launch_chained(bs_bwd_kernel<D16>, dim3(p.U, parts), dim3(kBThreads), smem, st, P, slot_steps(p.H), warp_bytes));
  }
  {
    const int KR = wv_rows(p.d, p.H);
    const size_t smem = 2 * (size_t)KR * ((size_t)p.H * p.d + p.d + 16) * sizeof(float);
    LASER_CUDA_OK(allow_smem(bs_wv_kernel<D16>, smem));
    LaunchScope ls("bs_wv", st);
    LASER_CUDA_OK(launch_chained(bs_wv_kernel<D16>, dim3(std::min(p.U, 2 * sms)), dim3(256), smem, st, P, KR));
  }
  LASER_CUDA_OK(cudaGetLastError());
  return LASER_OK;
}

}  // namespace

bool backward_stream_supported(const Plan& p) {
  return p.dtype == LASER_BF16 && p.maxC <= 1 && p.d % 16 == 0 && p.d >= 16 && p.d <= 128 && p.H <= 8 && p.dvh % 16 == 0 &&
         p.dqh % 16 == 0 && kBW * bwd_warp_bytes(p.d, p.H) + 2 * p.d + 16 <= 220 * 1024;
}
float* backward_stream_sums(const Plan& p, char* scratch) { return carve_bs(p, scratch).p; }
size_t backward_stream_scratch_bytes(const Plan& p) { return backward_stream_supported(p) ? carve_bs(p, nullptr).total : 0; }

#define LASER_BS_DISPATCH(fn, ...)                     \
  switch (p.d / 16) {                                  \
    case 1: return fn<1>(__VA_ARGS__);                 \
    case 2: return fn<2>(__VA_ARGS__);                 \
    case 3: return fn<3>(__VA_ARGS__);                 \
    case 4: return fn<4>(__VA_ARGS__);                 \
    case 5: return fn<5>(__VA_ARGS__);                 \
    case 6: return fn<6>(__VA_ARGS__);                 \
    case 7: return fn<7>(__VA_ARGS__);                 \
    case 8: return fn<8>(__VA_ARGS__);                 \
    default: return LASER_ERR_UNSUPPORTED;             \
  }

int backward_stream_forward(const Plan& p, const void* items, const int32_t* lengths, const void* cands,
                            const int32_t* cand_offsets, const void* Wq, const void* Wk, const void* Wv, float* Hp,
                            __nv_bfloat16* Hp_hi, __nv_bfloat16* Hp_lo, char* ws, char* scratch, cudaStream_t st,
                            const ZeroList* zero, const TrainPrep* prep) {
  const BsScratch s = carve_bs(p, scratch);
  const int rc = stream_fold(p, lengths, cands, cand_offsets, Wq, Wk, Wv, s.u, s.fold, reinterpret_cast<int*>(ws + p.off_status), st,
                             zero, prep);
  if (rc != LASER_OK) return rc;
  BsParams P = bs_params(p, s, items, lengths, cand_offsets, Wv, ws);
  P.s = Hp; P.s_hi = Hp_hi; P.s_lo = Hp_lo;
  LASER_BS_DISPATCH(bs_forward_t, p, P, st)
}

int backward_stream(const Plan& p, const void* items, const int32_t* lengths, const int32_t* cand_offsets, const void* Wv,
                    const float* dHp, float* d_items, float* dWv, const float** p_sums, char* ws, char* scratch, cudaStream_t st) {
  const BsScratch s = carve_bs(p, scratch);
  BsParams P = bs_params(p, s, items, lengths, cand_offsets, Wv, ws);
  P.ds = dHp; P.d_items = d_items; P.dWv = dWv;
  *p_sums = s.p;
  LASER_BS_DISPATCH(bs_backward_t, p, P, st)
}

}  // namespace laser

// The dense products of the backward pass over the item rows (bf16 inputs, warp-level MMAs), in two kernels that touch only
// the users' valid rows:
//
//   rows_project_kernel   Y = scale X [W_a | W_b] as bf16: K and V of the recomputed forward (X read once for both), and Q
//   rows_grad_kernel      d_items = dK W_k^T + dV W_v^T (zero rows for padding), dW_k += X^T dK, dW_v += X^T dV, all from one
//                         read of X, dK and dV; and d_cands = dt_0 + dQ W_q^T, dW_q += T^T dQ (16384 candidates: 37 us as two
//                         products on the FP32 ALUs)
//
// dK and dV arrive as bf16 high and low parts (16 bits; TF32 operands, 11 bits, before), so every operand tile is copied to
// shared memory as it is and read with ldmatrix; dQ, summed in fp32, is split on its way into shared memory; the weights stay in shared memory for the block's lifetime, the weight
// gradients in its registers until one atomic add per element at the end.
// Bound by HBM: 0.64 and 1.5 KB per valid row at d = 128, d_qk = 64.  Six kernels over all rows, padding included, and two
// memsets before: 470 us at 64 users of 512 .. 4096 of 4096 rows.
#include <algorithm>

#include "laser_backward.cuh"
#include "laser_common.cuh"
#include "laser_gsta_img.cuh"
#include "laser_mma.cuh"

namespace laser {
namespace {

using bf16 = __nv_bfloat16;
using namespace mma;

constexpr int kRT = 64;                 // rows per tile
constexpr int kRThreads = 512;          // 16 warps: 4 row tiles x 4 column parts

struct RowsParams {
  int groups, rows_per_group, tiles_per_group;       // users x L, or one group of N rows
  int na, nb;                                        // columns of W_a and W_b (nb may be 0)
  const bf16 *X, *Wa, *Wb;                           // X [groups, rows_per_group, d], W_a [d, na], W_b [d, nb]
  const int *lengths, *cand_offsets;                 // null: every row is valid
  int N;
  // projection
  bf16 *Ya, *Yb;
  float scale;
  // gradients
  const bf16 *Ahi, *Alo, *Bhi, *Blo;                 // dK [.., na], dV [.., nb]: high and low parts
  const float* A32;                                  // not null: the gradient [.., na] in fp32 instead, times scale (nb = 0)
  const float* add;                                  // not null: dX = add + the products
  float *dX, *dWa, *dWb;
};

// The items and the candidates in one launch: blocks first[r] .. first[r] + blocks[r] - 1 work on r.  A grid that fills the GPU takes
// one after the other (both ranges are all blocks); where each has few tiles they run beside one another.
struct RowsPair {
  RowsParams r[2];
  int first[2], blocks[2];
};
RowsPair pair_up(const RowsParams& items, const RowsParams& cands, long long most, unsigned* grid) {
  RowsPair P;
  P.r[0] = items;
  P.r[1] = cands;
  long long jobs[2];
  for (int r = 0; r < 2; ++r) jobs[r] = (long long)P.r[r].groups * P.r[r].tiles_per_group;
  const bool apart = jobs[0] + jobs[1] <= most;
  for (int r = 0; r < 2; ++r) {
    P.blocks[r] = (int)std::min(jobs[r], most);
    P.first[r] = apart && r == 1 ? P.blocks[0] : 0;
  }
  *grid = apart ? P.blocks[0] + P.blocks[1] : std::max(P.blocks[0], P.blocks[1]);
  if (!apart) P.first[1] = (int)*grid - P.blocks[1];      // few candidate tiles: to the last blocks, the first have the most item tiles
  return P;
}

// Rows of a group that take part (a user without candidates, or with invalid inputs, has none).
__device__ __forceinline__ int valid_rows(const RowsParams& P, int u) {
  if (!P.lengths) return P.rows_per_group;
  const int len = P.lengths[u], o0 = P.cand_offsets[u], o1 = P.cand_offsets[u + 1];
  return len <= 0 || len > P.rows_per_group || o0 < 0 || o1 <= o0 || o1 > P.N ? 0 : len;
}

// The same from a table in shared memory, when the groups fit (the walks below ask for every tile they pass).
constexpr int kTableGroups = 256;
__device__ __forceinline__ void fill_table(const RowsParams& P, int* table, int tid) {
  if (P.groups <= kTableGroups)
    for (int u = tid; u < P.groups; u += kRThreads) table[u] = valid_rows(P, u);
  __syncthreads();
}

// Tile `tile` of group `u`.  Block `block` of `blocks` takes every blocks-th one, groups fastest: the tiles that only long users have come
// last, spread over the blocks.  (A cursor instead of a tile number: divisions were a third of the gradient kernel's instructions.)
struct RowTile { int tile, u; };
struct RowWalk {
  const RowsParams& P;
  const int* table;
  int dt, du, block;
  __device__ __forceinline__ RowWalk(const RowsParams& params, const int* t, int b, int blocks) : P(params), table(t), block(b) {
    dt = blocks / P.groups;
    du = blocks - dt * P.groups;
  }
  __device__ __forceinline__ RowTile first() const {
    const int tile = block / P.groups;
    return {tile, block - tile * P.groups};
  }
  __device__ __forceinline__ bool in(RowTile c) const { return c.tile < P.tiles_per_group; }
  __device__ __forceinline__ RowTile step(RowTile c) const {
    c.tile += dt;
    c.u += du;
    if (c.u >= P.groups) c.u -= P.groups, ++c.tile;
    return c;
  }
  // valid rows of the tile and beyond it
  __device__ __forceinline__ int rows(RowTile c) const {
    return (P.groups <= kTableGroups ? table[c.u] : valid_rows(P, c.u)) - c.tile * kRT;
  }
  __device__ __forceinline__ size_t row0(RowTile c) const { return (size_t)c.u * P.rows_per_group + c.tile * kRT; }
  // c, or the first tile after it with valid rows
  __device__ __forceinline__ RowTile valid(RowTile c) const {
    while (in(c) && rows(c) <= 0) c = step(c);
    return c;
  }
};

template <int D16>
__device__ __forceinline__ void project_rows(const RowsParams& P, int block, int blocks, uint8_t* smem, int* table) {
  constexpr int d = 16 * D16, XS = 2 * d + 16;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, g = lane >> 2, t = lane & 3;
  const int n = P.na + P.nb, WS = 2 * n + 16;                        // bytes per row of [W_a | W_b] and of the output tile
  uint8_t* Ws = smem;                                                // [d][WS]
  uint8_t* Xs = Ws + (size_t)d * WS;                                 // [2][64][XS]
  uint8_t* Ys = Xs + 2 * kRT * XS;                                   // [64][WS]
  for (int i = tid; i < d * (n / 8); i += kRThreads) {
    const int k = i / (n / 8), c = (i - k * (n / 8)) * 8;
    cp16(smem_addr(Ws) + k * WS + c * 2, c < P.na ? P.Wa + (size_t)k * P.na + c : P.Wb + (size_t)k * P.nb + c - P.na, 16u);
  }
  fill_table(P, table, tid);
  const RowWalk walk(P, table, block, blocks);
  auto stage = [&](RowTile j, int b) {
    const int rows = walk.rows(j);
    const bf16* src = P.X + walk.row0(j) * d;
    for (int i = tid; i < kRT * 2 * D16; i += kRThreads) {
      const int r = i / (2 * D16), q = i - r * (2 * D16);
      cp16(smem_addr(Xs) + b * kRT * XS + r * XS + q * 16, r < rows ? src + (size_t)r * d + q * 8 : P.X, r < rows ? 16u : 0u);
    }
  };
  RowTile job = walk.valid(walk.first());
  if (walk.in(job)) stage(job, 0);
  cp_commit();
  const int m0 = (warp >> 2) * 16, part = warp & 3, pairs = n >> 4;  // column tiles in pairs: part, part + 4, ...
  const uint32_t a_row = ((lane & 7) + ((lane >> 3) & 1) * 8 + m0) * XS + (lane >> 4) * 16;
  const uint32_t b_row = ((lane & 7) + ((lane >> 3) & 1) * 8) * WS + (lane >> 4) * 16;
  int b = 0;
  const int out_c = lane * 8, out_ld = out_c < P.na ? P.na : P.nb;          // this lane's 8 columns of an output row
  bf16* out = out_c < P.na ? P.Ya + out_c : P.Yb + out_c - P.na;
  while (walk.in(job)) {
    const RowTile nxt = walk.valid(walk.step(job));
    if (walk.in(nxt)) stage(nxt, b ^ 1);
    cp_commit();
    cp_wait<1>();
    __syncthreads();
    float acc[4][2][4];
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
      for (int e = 0; e < 4; ++e) acc[i][0][e] = acc[i][1][e] = 0.f;
    const uint32_t xa = smem_addr(Xs) + b * kRT * XS + a_row, wa = smem_addr(Ws) + b_row;
#pragma unroll
    for (int kt = 0; kt < D16; ++kt) {
      uint32_t a[4];
      ldsm_x4(a, xa + kt * 32);
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const int p = part + 4 * i;
        if (p < pairs) {
          uint32_t w[4];
          ldsm_x4_t(w, wa + kt * 16 * WS + p * 32);
          mma16816(acc[i][0], a[0], a[1], a[2], a[3], w[0], w[1]);
          mma16816(acc[i][1], a[0], a[1], a[2], a[3], w[2], w[3]);
        }
      }
    }
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int p = part + 4 * i;
      if (p < pairs) {
        uint8_t* y = Ys + (m0 + g) * WS + p * 32 + 4 * t;
#pragma unroll
        for (int nt = 0; nt < 2; ++nt) {
          *reinterpret_cast<uint32_t*>(y + nt * 16) = pack2(acc[i][nt][0] * P.scale, acc[i][nt][1] * P.scale);
          *reinterpret_cast<uint32_t*>(y + 8 * WS + nt * 16) = pack2(acc[i][nt][2] * P.scale, acc[i][nt][3] * P.scale);
        }
      }
    }
    __syncthreads();
    {
      const int rows = min(walk.rows(job), kRT);
      bf16* y = out + walk.row0(job) * out_ld;
      if (out_c < n)
        for (int r = warp; r < rows; r += kRThreads / 32)
          *reinterpret_cast<uint4*>(y + r * out_ld) = *reinterpret_cast<const uint4*>(Ys + r * WS + out_c * 2);
    }
    job = nxt;
    b ^= 1;
  }
  cp_wait<0>();
}

// The set-up of the backward pass of candidate lists in one launch: both projections, the arrays that are summed into set to zero
// (the status word among them), and in `prep_blocks` blocks of their own what the stacked attention wants (one more sorts its blocks).
// Four launches and a memset before: the small batches are bound by their number.
struct ProjectParams {
  RowsPair rows;
  ZeroList zero;
  TrainPrep prep;
  int row_blocks, prep_blocks;
};
template <int D16>
__global__ void __launch_bounds__(kRThreads, 2) rows_project_kernel(const __grid_constant__ ProjectParams P) {
  extern __shared__ __align__(128) uint8_t smem[];
  __shared__ int table[kTableGroups];
  chain_wait();
  chain_release();
  const int block = blockIdx.x, tid = threadIdx.x;
  zero_share(P.zero, (unsigned long long)block * kRThreads + tid, (unsigned long long)gridDim.x * kRThreads);
  if (block >= P.row_blocks) {
    const int b = block - P.row_blocks;
    if (b < P.prep_blocks) train_prep_share(P.prep, b * kRThreads + tid, P.prep_blocks * kRThreads);
    else gsta_build_order(P.prep.lengths, P.prep.cand_offsets, P.prep.U, P.prep.N, P.prep.L, P.prep.S, P.prep.Lp, P.prep.cpb,
                          P.prep.order, P.prep.keys, reinterpret_cast<int*>(smem));
    return;
  }
#pragma unroll 1
  for (int r = 0; r < 2; ++r) {
    const int b = block - P.rows.first[r];
    if (b < 0 || b >= P.rows.blocks[r]) continue;
    project_rows<D16>(P.rows.r[r], b, P.rows.blocks[r], smem, table);
    __syncthreads();                       // (the next rows' weights and tiles replace these)
  }
}

template <int D16>
__device__ __forceinline__ void row_gradients(const RowsParams& P, int block, int blocks, int nbuf, uint8_t* smem, int* table) {
  constexpr int d = 16 * D16, XS = 2 * d + 16;
  // a warp's share of the weight gradients: kM tiles of 16 features, column pairs wpart, wpart + kParts, ...
  constexpr int kM = D16 % 2 == 0 ? 2 : 1, kParts = 16 * kM / D16, kMaxPairs = (16 + kParts - 1) / kParts;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, g = lane >> 2, t = lane & 3;
  const int n = P.na + P.nb, WS = 2 * n + 16, pairs = n >> 4;
  uint8_t* Ws = smem;                                                // [d][WS]  [W_k | W_v]
  uint8_t* Xs = Ws + (size_t)d * WS;                                 // [nbuf][64][XS]
  uint8_t* Gs = Xs + (size_t)nbuf * kRT * XS;                        // [nbuf][2][64][WS]  [dK | dV], high and low parts
  for (int i = tid; i < d * (n / 8); i += kRThreads) {
    const int k = i / (n / 8), c = (i - k * (n / 8)) * 8;
    cp16(smem_addr(Ws) + k * WS + c * 2, c < P.na ? P.Wa + (size_t)k * P.na + c : P.Wb + (size_t)k * P.nb + c - P.na, 16u);
  }
  fill_table(P, table, tid);
  const RowWalk walk(P, table, block, blocks);
  const int g_c = lane * 8, g_ld = g_c < P.na ? P.na : P.nb;                 // this lane's 8 columns of [dK | dV]
  const bf16 *g_hi = g_c < P.na ? P.Ahi + g_c : P.Bhi + g_c - P.na, *g_lo = g_c < P.na ? P.Alo + g_c : P.Blo + g_c - P.na;
  auto stage = [&](RowTile j, int b) {
    const int rows = walk.rows(j);
    const size_t row0 = walk.row0(j);
    const bf16* x = P.X + row0 * d;
    for (int i = tid; i < kRT * 2 * D16; i += kRThreads) {
      const int r = i / (2 * D16), q = i - r * (2 * D16);
      cp16(smem_addr(Xs) + b * kRT * XS + r * XS + q * 16, r < rows ? x + r * d + q * 8 : P.X, r < rows ? 16u : 0u);
    }
    if (P.A32) {                                                     // fp32: split into its parts on the way
      for (int i = tid; i < kRT * (n / 4); i += kRThreads) {
        const int r = i / (n / 4), q = i - r * (n / 4);
        float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
        if (r < rows) v = *reinterpret_cast<const float4*>(P.A32 + (row0 + r) * n + q * 4);
        v.x *= P.scale; v.y *= P.scale; v.z *= P.scale; v.w *= P.scale;
        const uint32_t h0 = pack2(v.x, v.y), h1 = pack2(v.z, v.w);
        uint8_t* at = Gs + (size_t)b * 2 * kRT * WS + r * WS + q * 8;
        *reinterpret_cast<uint2*>(at) = make_uint2(h0, h1);
        *reinterpret_cast<uint2*>(at + kRT * WS) =
            make_uint2(pack2(v.x - bf16_lo(h0), v.y - bf16_hi(h0)), pack2(v.z - bf16_lo(h1), v.w - bf16_hi(h1)));
      }
    } else if (g_c < n) {                                            // a warp per row, 8 columns per lane
      const bf16 *hi = g_hi + row0 * g_ld, *lo = g_lo + row0 * g_ld;
      uint32_t dst = smem_addr(Gs) + b * 2 * kRT * WS + warp * WS + g_c * 2;
#pragma unroll
      for (int r = warp; r < kRT; r += kRThreads / 32, dst += kRThreads / 32 * WS) {
        const bool ok = r < rows;
        cp16(dst, ok ? hi + r * g_ld : P.X, ok ? 16u : 0u);
        cp16(dst + kRT * WS, ok ? lo + r * g_ld : P.X, ok ? 16u : 0u);
      }
    }
  };
  RowTile job = walk.valid(walk.first());
  if (walk.in(job)) stage(job, 0);
  cp_commit();
  // rows that receive no gradient
  for (RowTile j = walk.first(); walk.in(j); j = walk.step(j)) {
    const int first = max(0, min(kRT, walk.rows(j))), last = min(kRT, P.rows_per_group - j.tile * kRT);
    float4* out = reinterpret_cast<float4*>(P.dX + walk.row0(j) * d);
    for (int i = first * (d / 4) + tid; i < last * (d / 4); i += kRThreads) out[i] = make_float4(0.f, 0.f, 0.f, 0.f);
  }
  const int m0 = (warp >> 2) * 16, part = warp & 3;                  // d_items: 16 rows, feature pairs part, part + 4
  const int mw = warp % (D16 / kM) * kM, wpart = warp / (D16 / kM);
  const int mi = lane >> 3, lr = lane & 7;
  const uint32_t a_row = ((mi & 1) * 8 + lr + m0) * WS + (mi >> 1) * 16;            // [dK | dV] as A (rows, columns)
  const uint32_t w_row = ((mi >> 1) * 8 + lr) * WS + (mi & 1) * 16;                 // W^T as B: W rows are its columns
  const uint32_t xt_row = ((mi >> 1) * 8 + lr) * XS + mw * 32 + (mi & 1) * 16;      // X^T as A
  const uint32_t g_row = ((mi & 1) * 8 + lr) * WS + (mi >> 1) * 16;                 // [dK | dV] as B
  float wacc[kM][kMaxPairs][2][4];
#pragma unroll
  for (int m = 0; m < kM; ++m)
#pragma unroll
    for (int i = 0; i < kMaxPairs; ++i)
#pragma unroll
      for (int e = 0; e < 4; ++e) wacc[m][i][0][e] = wacc[m][i][1][e] = 0.f;
  auto put = [&](float* at, float x0, float x1) {
    if (P.add) {
      const float2 v = *reinterpret_cast<const float2*>(P.add + (at - P.dX));
      x0 += v.x;
      x1 += v.y;
    }
    *reinterpret_cast<float2*>(at) = make_float2(x0, x1);
  };
  int b = 0;
  while (walk.in(job)) {
    const RowTile nxt = walk.valid(walk.step(job));
    if (nbuf == 2) {
      if (walk.in(nxt)) stage(nxt, b ^ 1);
      cp_commit();
      cp_wait<1>();
    } else {
      cp_wait<0>();
    }
    __syncthreads();
    const uint32_t xs = smem_addr(Xs) + b * kRT * XS, hi = smem_addr(Gs) + b * 2 * kRT * WS, lo = hi + kRT * WS;
    // the two products of the tile are independent: half of the warps of every scheduler take them in the other order, so that
    // one's MMAs run beside the other's stores
#pragma unroll 1
    for (int phase = 0; phase < 2; ++phase)
      if (phase == (warp >> 2 & 1)) {
        float acc[2][2][4];
#pragma unroll
        for (int i = 0; i < 2; ++i)
#pragma unroll
          for (int e = 0; e < 4; ++e) acc[i][0][e] = acc[i][1][e] = 0.f;
#pragma unroll 2
        for (int kt = 0; kt < pairs; ++kt) {
          uint32_t ah[4], al[4];
          ldsm_x4(ah, hi + a_row + kt * 32);
          ldsm_x4(al, lo + a_row + kt * 32);
#pragma unroll
          for (int i = 0; i < 2; ++i) {
            const int p = part + 4 * i;
            if (p < D16) {
              uint32_t w[4];
              ldsm_x4(w, smem_addr(Ws) + w_row + p * 16 * WS + kt * 32);
              mma16816(acc[i][0], ah[0], ah[1], ah[2], ah[3], w[0], w[1]);
              mma16816(acc[i][1], ah[0], ah[1], ah[2], ah[3], w[2], w[3]);
              mma16816(acc[i][0], al[0], al[1], al[2], al[3], w[0], w[1]);
              mma16816(acc[i][1], al[0], al[1], al[2], al[3], w[2], w[3]);
            }
          }
        }
        {
          const int rows = walk.rows(job);
          float* out = P.dX + (walk.row0(job) + m0 + g) * d + 2 * t;
#pragma unroll
          for (int i = 0; i < 2; ++i) {
            const int p = part + 4 * i;
            if (p < D16) {
#pragma unroll
              for (int nt = 0; nt < 2; ++nt) {
                const int at = p * 16 + nt * 8;
                if (m0 + g < rows) put(out + at, acc[i][nt][0], acc[i][nt][1]);
                if (m0 + g + 8 < rows) put(out + 8 * d + at, acc[i][nt][2], acc[i][nt][3]);
              }
            }
          }
        }
      } else if (wpart < kParts) {
#pragma unroll
        for (int kt = 0; kt < kRT / 16; ++kt) {
          uint32_t a[kM][4];
#pragma unroll
          for (int m = 0; m < kM; ++m) ldsm_x4_t(a[m], xs + xt_row + kt * 16 * XS + m * 32);
#pragma unroll
          for (int i = 0; i < kMaxPairs; ++i) {
            const int p = wpart + kParts * i;
            if (p < pairs) {
              uint32_t bh[4], bl[4];
              ldsm_x4_t(bh, hi + g_row + kt * 16 * WS + p * 32);
              ldsm_x4_t(bl, lo + g_row + kt * 16 * WS + p * 32);
#pragma unroll
              for (int m = 0; m < kM; ++m) {
                mma16816(wacc[m][i][0], a[m][0], a[m][1], a[m][2], a[m][3], bh[0], bh[1]);
                mma16816(wacc[m][i][1], a[m][0], a[m][1], a[m][2], a[m][3], bh[2], bh[3]);
              }
#pragma unroll
              for (int m = 0; m < kM; ++m) {
                mma16816(wacc[m][i][0], a[m][0], a[m][1], a[m][2], a[m][3], bl[0], bl[1]);
                mma16816(wacc[m][i][1], a[m][0], a[m][1], a[m][2], a[m][3], bl[2], bl[3]);
              }
            }
          }
        }
      }
    __syncthreads();                       // the tile just read may be overwritten
    if (nbuf == 2) {
      b ^= 1;
    } else if (walk.in(nxt)) {
      stage(nxt, 0);
      cp_commit();
    }
    job = nxt;
  }
  cp_wait<0>();
  if (wpart >= kParts) return;
#pragma unroll
  for (int m = 0; m < kM; ++m)
#pragma unroll
    for (int i = 0; i < kMaxPairs; ++i) {
      const int p = wpart + kParts * i;
      if (p < pairs) {
#pragma unroll
        for (int nt = 0; nt < 2; ++nt) {
          const int c = p * 16 + nt * 8;
          if (c < P.na) red_tile(P.dWa + (size_t)(mw + m) * 16 * P.na + c, P.na, wacc[m][i][nt], 1.f, lane);
          else red_tile(P.dWb + (size_t)(mw + m) * 16 * P.nb + c - P.na, P.nb, wacc[m][i][nt], 1.f, lane);
        }
      }
    }
}

template <int D16>
__global__ void __launch_bounds__(kRThreads) rows_grad_kernel(const __grid_constant__ RowsPair P, int nbuf0, int nbuf1) {
  extern __shared__ __align__(128) uint8_t smem[];
  __shared__ int table[kTableGroups];
  chain_wait();
  chain_release();
#pragma unroll 1
  for (int r = 0; r < 2; ++r) {
    const int b = (int)blockIdx.x - P.first[r];
    if (b < 0 || b >= P.blocks[r]) continue;
    row_gradients<D16>(P.r[r], b, P.blocks[r], r ? nbuf1 : nbuf0, smem, table);
    __syncthreads();                       // (the next rows' weights and tiles replace these)
  }
}

size_t project_smem(int d, int n) { return (size_t)d * (2 * n + 16) + 2 * kRT * (2 * (size_t)d + 16) + (size_t)kRT * (2 * n + 16); }
size_t grad_smem(int d, int n, int nbuf) {
  return (size_t)d * (2 * n + 16) + nbuf * (kRT * (2 * (size_t)d + 16) + 2 * kRT * (2 * (size_t)n + 16));
}
constexpr size_t kRowsSmemMax = 226 * 1024;

struct ProjectJob {
  RowsParams items, cands;
  ZeroList zero;
  TrainPrep prep;
};
template <int D16>
int launch_project(const ProjectJob& J, cudaStream_t st) {
  const size_t smem = project_smem(16 * D16, std::max(J.items.na + J.items.nb, J.cands.na));
  LASER_CUDA_OK(allow_smem(rows_project_kernel<D16>, smem));
  const int per_sm = smem <= 112 * 1024 ? 2 : 1, sms = device_sms();
  ProjectParams P;
  unsigned grid;
  P.rows = pair_up(J.items, J.cands, (long long)per_sm * sms, &grid);
  P.zero = J.zero;
  P.prep = J.prep;
  P.row_blocks = (int)grid;
  P.prep_blocks = !J.prep.img ? 0 : std::min((J.prep.M * 6 * D16 * D16 * 32 + kRThreads - 1) / kRThreads, sms);
  LaunchScope ls("bwd_rows_project", st);
  LASER_CUDA_OK(launch_chained(rows_project_kernel<D16>, dim3(grid + P.prep_blocks + (J.prep.order ? 1 : 0)), dim3(kRThreads), smem, st, P));
  return LASER_OK;
}
struct GradJob {
  RowsParams items, cands;
};
template <int D16>
int launch_grad(const GradJob& J, cudaStream_t st) {
  const int n0 = J.items.na + J.items.nb, n1 = J.cands.na;
  auto buffers = [](int n) { return grad_smem(16 * D16, n, 2) <= kRowsSmemMax ? 2 : 1; };
  const size_t smem = std::max(grad_smem(16 * D16, n0, buffers(n0)), grad_smem(16 * D16, n1, buffers(n1)));
  LASER_CUDA_OK(allow_smem(rows_grad_kernel<D16>, smem));
  unsigned grid;
  const RowsPair P = pair_up(J.items, J.cands, device_sms(), &grid);
  LaunchScope ls("bwd_rows_grad", st);
  LASER_CUDA_OK(launch_chained(rows_grad_kernel<D16>, dim3(grid), dim3(kRThreads), smem, st, P, buffers(n0), buffers(n1)));
  return LASER_OK;
}

#define LASER_ROWS_DISPATCH(fn)               \
  switch (p.d / 16) {                         \
    case 1: return fn<1>(J, st);              \
    case 2: return fn<2>(J, st);              \
    case 3: return fn<3>(J, st);              \
    case 4: return fn<4>(J, st);              \
    case 5: return fn<5>(J, st);              \
    case 6: return fn<6>(J, st);              \
    case 7: return fn<7>(J, st);              \
    case 8: return fn<8>(J, st);              \
    default: return LASER_ERR_UNSUPPORTED;    \
  }

}  // namespace

bool rows_mma_supported(const Plan& p) {
  return p.dtype == LASER_BF16 && p.d % 16 == 0 && p.d <= 128 && p.dqk % 16 == 0 && p.dqk <= 128 &&
         grad_smem(p.d, p.dqk + p.d, 1) <= kRowsSmemMax && (long long)p.U * ((p.L + kRT - 1) / kRT) < (1ll << 30);
}

static RowsParams item_rows(const Plan& p, const void* items, const int32_t* lengths, const int32_t* cand_offsets, const void* Wk,
                            const void* Wv) {
  RowsParams P = {};
  P.groups = p.U; P.rows_per_group = p.L; P.tiles_per_group = (p.L + kRT - 1) / kRT; P.na = p.dqk; P.nb = p.d;
  P.X = (const bf16*)items; P.Wa = (const bf16*)Wk; P.Wb = (const bf16*)Wv; P.lengths = lengths; P.cand_offsets = cand_offsets;
  P.N = p.N; P.scale = 1.f;
  return P;
}
static RowsParams cand_rows(const Plan& p, const void* cands, const void* Wq, float scale) {
  RowsParams P = {};
  P.groups = 1; P.rows_per_group = p.N; P.tiles_per_group = (p.N + kRT - 1) / kRT; P.na = p.dqk;
  P.X = (const bf16*)cands; P.Wa = P.Wb = (const bf16*)Wq; P.N = p.N; P.scale = scale;
  return P;
}

int rows_project(const Plan& p, const void* items, const int32_t* lengths, const void* cands, const int32_t* cand_offsets, const void* Wq,
                 const void* Wk, const void* Wv, float q_scale, __nv_bfloat16* Qb, __nv_bfloat16* Kb, __nv_bfloat16* Vb,
                 const ZeroList& zero, const TrainPrep& prep, cudaStream_t st) {
  ProjectJob J;
  J.items = item_rows(p, items, lengths, cand_offsets, Wk, Wv);
  J.items.Ya = Kb; J.items.Yb = Vb;
  J.cands = cand_rows(p, cands, Wq, q_scale);
  J.cands.Ya = Qb;
  J.zero = zero;
  J.prep = prep;
  LASER_ROWS_DISPATCH(launch_project)
}

int rows_gradients(const Plan& p, const void* items, const int32_t* lengths, const void* cands, const int32_t* cand_offsets, const void* Wq,
                   const void* Wk, const void* Wv, const float* dQf, const __nv_bfloat16* dK_hi, const __nv_bfloat16* dK_lo,
                   const __nv_bfloat16* dV_hi, const __nv_bfloat16* dV_lo, const float* dT0, float* d_items, float* d_cands, float* dWq,
                   float* dWk, float* dWv, cudaStream_t st) {
  GradJob J;
  J.items = item_rows(p, items, lengths, cand_offsets, Wk, Wv);
  J.items.Ahi = dK_hi; J.items.Alo = dK_lo; J.items.Bhi = dV_hi; J.items.Blo = dV_lo;
  J.items.dX = d_items; J.items.dWa = dWk; J.items.dWb = dWv;
  J.cands = cand_rows(p, cands, Wq, p.inv_gamma);
  J.cands.A32 = dQf; J.cands.add = dT0; J.cands.dX = d_cands; J.cands.dWa = J.cands.dWb = dWq;
  LASER_ROWS_DISPATCH(launch_grad)
}

}  // namespace laser

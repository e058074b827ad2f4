// Tensor-core kernel of the backward pass through the stacked attention (bf16 inputs): the layers are recomputed and run
// backward for 16 (or 8) candidates inside one block, as the forward kernel (laser_gsta.cu) runs them forward.
//
//   forward, per layer    q = t W_q,   qt_h = q_h W_k[:, h]^T / tau,   a = softmax_j(s_j . qt_h),   m_h = sum_j a s_j,
//                         t += m_h W_v[:, h]
//   backward, per layer   dm_h = dt_h W_v[:, h]^T,   da_j = s_j . dm_h,   de = a (da - m . dm),   dqt_h = sum_j de_j s_j,
//                         dq_h = dqt_h W_k[:, h] / tau,   dt += dq W_q^T
//   at the end            ds_j = sum over layers and heads of de_j qt_h + a_j dm_h   (one product per candidate, its factors
//                         kept per (layer, head) "slot": 2 M H of them)
//
// What used to be seven batched products, two attention kernels and a read-modify-write of dH' per layer, every
// intermediate of 2 MB .. 34 MB crossing L2 between them, leaves only what the weight gradients sum over the candidates
// (t, q, m, dt, dq, dqt) and dH' itself, once.  The targets and every product's left operand are fp32 values split into
// bf16 high and low parts (16 bits; the products had TF32 operands, 11 bits, at the same MMA cost), the weights are bf16.
// Segment vectors and the attention's small factors are bf16 (NP = 1), or bf16 pairs where the caller's recomputed H' is
// fp32 (NP = 2: every product in three terms).
// Bound by instruction issue and latency like the forward kernel: 16 warps per SM where shared memory allows two blocks.
#include <algorithm>

#include "laser_backward.cuh"
#include "laser_common.cuh"
#include "laser_gsta_img.cuh"
#include "laser_mma.cuh"

namespace laser {
namespace {

using bf16 = __nv_bfloat16;
using namespace mma;

constexpr int kTW = 8, kTThreads = kTW * 32;      // warps per block: one or two candidates each
constexpr int kTRows = 16;                        // candidates per tile = rows of the dense MMAs; segments per chunk

struct TrainParams {
  int N, U, L, S, Lp, H, M, cpb, slots, nb, kb;   // slots = 2 M H; nb staging buffers per warp, kb of them hold slot rows
  float inv_tau;
  const bf16 *S0, *S1;                            // [N, Lp, d] segment vectors: high (or only) and low parts
  const bf16* cands;
  const float* dz;
  const uint4* img;                               // [M][3][2][d/16][d/16][32]: W_q, W_k, W_v as stored and transposed
  const int *nseg, *order;
  GstaPlanes G;
  float* stat;                                    // [M, N, H, 2] softmax maximum and 1 / sum
  bf16 *rows0, *rows1;                            // [N, slots, d] qt and dm per slot (high, low)
  float* ad32;                                    // [N, Lp, slots] de and a per slot (NP = 2)
  bf16* ad16;                                     // the same as the bf16 operand it becomes (NP = 1)
  bf16* dS16;                                     // [N, Lp, d] out, rounded to bf16, or
  float* dS32;                                    // [N, Lp, d] out, fp32 (NP = 2, dS16 null)
};

__global__ void __launch_bounds__(256) train_prep_kernel(const __grid_constant__ TrainPrep P) {
  __shared__ int bins[kGstaSortWords];
  chain_wait();
  chain_release();
  const int n_blocks = gridDim.x - (P.order ? 1 : 0);
  if ((int)blockIdx.x == n_blocks) gsta_build_order(P.lengths, P.cand_offsets, P.U, P.N, P.L, P.S, P.Lp, P.cpb, P.order, P.keys, bins);
  else train_prep_share(P, blockIdx.x * 256 + threadIdx.x, n_blocks * 256);
}

// x -> (high, low) bf16 pairs of two floats
__device__ __forceinline__ void split2(float x0, float x1, uint32_t& hi, uint32_t& lo) {
  hi = pack2(x0, x1);
  lo = pack2(x0 - bf16_lo(hi), x1 - bf16_hi(hi));
}

template <int D16, int NP>
struct TrainSmem {
  static constexpr int d = 16 * D16, RS = 2 * d + 16;
  // Bytes from one candidate's head rows to the next's: with an even number of heads 16 bytes more than the rows take, so that
  // the same head of eight candidates (an operand of the dense products) lies in eight different 16-byte bank groups.
  static __host__ __device__ constexpr uint32_t cand_pitch(int H) { return (uint32_t)(H * RS + (H % 2 ? 0 : 16)); }
  static __host__ __device__ constexpr size_t plane(int H) { return (size_t)kTRows * cand_pitch(H); }
  static size_t bytes(int H, int nb) {
    return 2 * (size_t)kTRows * RS + 2 * NP * plane(H) + RS + kTRows * sizeof(int) + 48 + (size_t)kTW * nb * kTRows * RS * NP;
  }
};

template <int D16, int NP>
__global__ void __launch_bounds__(kTThreads, 2) gsta_train_kernel(const __grid_constant__ TrainParams P) {
  using SM = TrainSmem<D16, NP>;
  constexpr int d = SM::d, RS = SM::RS;
  extern __shared__ __align__(128) uint8_t smem[];
  chain_wait();
  chain_release();
  const int H = P.H, Lp = P.Lp, dvh = d / H, KH = dvh >> 4;
  const uint32_t plane = (uint32_t)SM::plane(H), CP = SM::cand_pitch(H);
  uint8_t* Thi = smem;                                               // [16] rows: t, later dt, high and low parts (the fp32
  uint8_t* Tlo = Thi + kTRows * RS;                                  // values live in the registers of the columns' warp)
  uint8_t* Qt = smem + 2 * kTRows * RS;                              // [NP][16] candidates' H rows: qt; m or dqt (high) later
  uint8_t* Dm = Qt + NP * plane;                                     // [NP][16] candidates' H rows: dm; NP = 1: also m or dqt (low)
  uint8_t* Xlo = NP == 1 ? Dm : Qt + plane;                          // low parts of m / dqt (their high parts: Qt)
  uint8_t* zrow = Dm + NP * plane;
  int* nv_s = reinterpret_cast<int*>(zrow + RS);
  uint8_t* stage = reinterpret_cast<uint8_t*>(((uintptr_t)(nv_s + kTRows) + 15) & ~(uintptr_t)15);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, g = lane >> 2, t = lane & 3;
  const uint32_t chunk_bytes = kTRows * RS * NP;                     // one staging buffer: NP planes of 16 rows
  uint8_t* mine = stage + (size_t)warp * P.nb * chunk_bytes;
  const uint32_t mine_a = smem_addr(mine);
  uint8_t* Qhi = stage;                                              // dense phases only: q or dq rows, high and low
  uint8_t* Qlo = stage + kTRows * RS;

  const int blk = P.order ? min(max(P.order[blockIdx.x], 0), (int)gridDim.x - 1) : (int)blockIdx.x;
  const int c_base = blk * P.cpb, c_end = min(c_base + P.cpb, P.N);
  const int n_slots = P.cpb == kTRows ? 2 : 1;                       // candidates per warp
  const size_t Nd = (size_t)P.N * d, NHd = Nd * H;
  const bool dense = warp < D16;
  const int wcol = warp * 16;                                        // this warp's 16 columns of the dense phases
  constexpr int kImg = D16 * D16 * 32;
  if (tid < kTRows) nv_s[tid] = c_base + tid < c_end ? min(max(P.nseg[c_base + tid], 0), Lp) : 0;
  for (int i = tid; i < RS / 4; i += kTThreads) reinterpret_cast<uint32_t*>(zrow)[i] = 0u;
  for (uint32_t i = tid * 4; i < 2 * NP * plane; i += kTThreads * 4) *reinterpret_cast<uint32_t*>(Qt + i) = 0u;   // (rows of absent candidates)
  __syncthreads();

  // ---- dense building blocks.  Weight fragments of k-tile kt for this warp's columns: image entry (kt, warp).
  auto weights = [&](int l, int m, int trans) { return P.img + (size_t)((l * 3 + m) * 2 + trans) * kImg + (size_t)warp * 32 + lane; };
  auto mma_pair = [&](float (&acc)[2][4], const uint32_t (&a)[4], const uint4& b) {
    mma16816(acc[0], a[0], a[1], a[2], a[3], b.x, b.y);
    mma16816(acc[1], a[0], a[1], a[2], a[3], b.z, b.w);
  };
  const uint32_t ldsm_row = (lane & 7) + ((lane >> 3) & 1) * 8, ldsm_kc = lane >> 4;
  // acc = x_h W with x rows (head rows of the planes), h = the head of this warp's columns
  auto from_heads = [&](float (&acc)[2][4], const uint4* w) {
    const uint32_t o = ldsm_row * CP + wcol / dvh * RS + ldsm_kc * 16;
    const uint32_t ah = smem_addr(Qt) + o, al = smem_addr(Xlo) + o;
#pragma unroll
    for (int kt = 0; kt < D16; ++kt) {
      const uint4 b = __ldg(w + kt * D16 * 32);
      uint32_t hi[4], lo[4];
      ldsm_x4(hi, ah + kt * 32);
      ldsm_x4(lo, al + kt * 32);
      mma_pair(acc, hi, b);
      mma_pair(acc, lo, b);
    }
  };
  // this warp's columns of a [16][d] result as high / low rows: to shared memory (hi, lo; the next product's operand) and
  // to global memory (dst: N rows of d, the low parts `lo_at` elements behind)
  auto put_rows = [&](const float (&v)[2][4], float scale, uint8_t* hi, uint8_t* lo, bf16* dst, size_t lo_at) {
#pragma unroll
    for (int nt = 0; nt < 2; ++nt)
#pragma unroll
      for (int hf = 0; hf < 2; ++hf) {
        const int r = g + hf * 8, col = wcol + nt * 8 + 2 * t;
        uint32_t h, l;
        split2(v[nt][2 * hf] * scale, v[nt][2 * hf + 1] * scale, h, l);
        *reinterpret_cast<uint32_t*>(hi + r * RS + col * 2) = h;
        *reinterpret_cast<uint32_t*>(lo + r * RS + col * 2) = l;
        if (dst && c_base + r < c_end) {
          const size_t at = (size_t)(c_base + r) * d + col;
          *reinterpret_cast<uint32_t*>(dst + at) = h;
          *reinterpret_cast<uint32_t*>(dst + lo_at + at) = l;
        }
      }
  };
  // acc += x W with x the 16 high / low rows at hi, lo
  auto from_rows = [&](float (&acc)[2][4], const uint8_t* hi, const uint8_t* lo, const uint4* w) {
    const uint32_t ah = smem_addr(hi + ldsm_row * RS) + ldsm_kc * 16, al = smem_addr(lo + ldsm_row * RS) + ldsm_kc * 16;
#pragma unroll
    for (int kt = 0; kt < D16; ++kt) {
      const uint4 b = __ldg(w + kt * D16 * 32);
      uint32_t x[4];
      ldsm_x4(x, ah + kt * 32);
      mma_pair(acc, x, b);
      ldsm_x4(x, al + kt * 32);
      mma_pair(acc, x, b);
    }
  };
  // the same head by head (k-tiles of head h only), each result as head rows of the planes at dst (low parts: NP = 2)
  auto fold_heads = [&](const uint8_t* hi, const uint8_t* lo, const uint4* w, float scale, uint8_t* dst) {
    const uint32_t ah = smem_addr(hi + ldsm_row * RS) + ldsm_kc * 16, al = smem_addr(lo + ldsm_row * RS) + ldsm_kc * 16;
    float acc[2][4] = {};
#pragma unroll
    for (int kt = 0; kt < D16; ++kt) {
      const uint4 b = __ldg(w + kt * D16 * 32);
      uint32_t x[4];
      ldsm_x4(x, ah + kt * 32);
      mma_pair(acc, x, b);
      ldsm_x4(x, al + kt * 32);
      mma_pair(acc, x, b);
      if ((kt + 1) % KH == 0) {                                      // last k-tile of head kt / KH
        const int h = kt / KH;
#pragma unroll
        for (int nt = 0; nt < 2; ++nt)
#pragma unroll
          for (int hf = 0; hf < 2; ++hf) {
            uint32_t vh, vl;
            split2(acc[nt][2 * hf] * scale, acc[nt][2 * hf + 1] * scale, vh, vl);
            const uint32_t o = (g + hf * 8) * CP + h * RS + (wcol + nt * 8 + 2 * t) * 2;
            *reinterpret_cast<uint32_t*>(dst + o) = vh;
            if (NP == 2) *reinterpret_cast<uint32_t*>(dst + plane + o) = vl;
            acc[nt][2 * hf] = acc[nt][2 * hf + 1] = 0.f;
          }
      }
    }
  };
  float tr[2][4] = {};                                               // t, later dt: this warp's columns, rows g and g + 8
  auto load_rows = [&](auto at) {
#pragma unroll
    for (int nt = 0; nt < 2; ++nt)
#pragma unroll
      for (int hf = 0; hf < 2; ++hf) {
        float2 v = make_float2(0.f, 0.f);
        if (c_base + g + hf * 8 < c_end) v = at((size_t)(c_base + g + hf * 8) * d + wcol + nt * 8 + 2 * t);
        tr[nt][2 * hf] = v.x;
        tr[nt][2 * hf + 1] = v.y;
      }
  };

  // ---- staging of a candidate's segment vectors, 16 rows per buffer (rows past its segments: zeros)
  auto stage_chunk = [&](int cand, int ch, int nv, int b) {
    const uint32_t dst = mine_a + b * chunk_bytes;
#pragma unroll
    for (int pl = 0; pl < NP; ++pl) {
      const bf16* src = (pl ? P.S1 : P.S0) + ((size_t)cand * Lp + ch * kTRows) * d;
#pragma unroll
      for (int i = 0; i < D16; ++i) {
        const int piece = i * 32 + lane, row = piece / (2 * D16), q = piece - row * (2 * D16);
        const bool ok = ch * kTRows + row < nv;
        cp16(dst + pl * (kTRows * RS) + row * RS + q * 16, ok ? (const void*)(src + row * d + q * 8) : (const void*)P.S0, ok ? 16u : 0u);
      }
    }
    cp_commit();
  };
  const uint32_t a_off = ((lane & 7) + ((lane >> 3) & 1) * 8) * RS + (lane >> 4) * 16;       // S as [segment][feature]
  const uint32_t t_off = ((lane & 7) + (lane >> 4) * 8) * RS + ((lane >> 3) & 1) * 16;       // S^T as [feature][segment]
  // B fragments of 8 head rows (row c H + h of a plane; heads past H read zeros)
  auto head_rows = [&](const uint8_t* base, int c) {
    return smem_addr(((lane & 7) < H ? base + c * CP + (lane & 7) * RS : zrow) + ((lane >> 3) & 1) * 16);
  };
  // e += S x^T for one staged chunk, x = head rows at b0 (and b1: low parts)
  auto dot_tile = [&](int kt, const uint32_t (&a0)[4], const uint32_t (&a1)[4], uint32_t b0, uint32_t b1, float (&e)[4]) {
    uint32_t b[2];
    ldsm_x2(b, b0 + kt * 32);
    mma16816(e, a0[0], a0[1], a0[2], a0[3], b[0], b[1]);
    if (NP == 2) {
      mma16816(e, a1[0], a1[1], a1[2], a1[3], b[0], b[1]);
      ldsm_x2(b, b1 + kt * 32);
      mma16816(e, a0[0], a0[1], a0[2], a0[3], b[0], b[1]);
    }
  };
  // x^T (features x heads) += S^T w, w = two rows of weights (segments g, g + 8; heads 2t, 2t + 1)
  auto weigh_chunk = [&](uint32_t sb, float (&x)[D16][4], float w0, float w1, float w2, float w3) {
    uint32_t h0, l0, h1, l1;
    split2(w0, w1, h0, l0);
    split2(w2, w3, h1, l1);
    const uint32_t bh0 = movmatrix_t(h0), bh1 = movmatrix_t(h1);
    const uint32_t bl0 = NP == 2 ? movmatrix_t(l0) : 0u, bl1 = NP == 2 ? movmatrix_t(l1) : 0u;
#pragma unroll
    for (int jt = 0; jt < D16; ++jt) {
      uint32_t a[4];
      ldsm_x4_t(a, sb + t_off + jt * 32);
      mma16816(x[jt], a[0], a[1], a[2], a[3], bh0, bh1);
      if (NP == 2) {
        mma16816(x[jt], a[0], a[1], a[2], a[3], bl0, bl1);
        ldsm_x4_t(a, sb + kTRows * RS + t_off + jt * 32);
        mma16816(x[jt], a[0], a[1], a[2], a[3], bh0, bh1);
      }
    }
  };
  // rows [head][feature] of candidate c from x^T (scaled per head): high parts to Qt, low parts to Xlo
  auto put_heads = [&](int c, const float (&x)[D16][4], float f0, float f1) {
#pragma unroll
    for (int jt = 0; jt < D16; ++jt) {
      uint32_t ha, la, hb, lb;
      split2(x[jt][0] * f0, x[jt][1] * f1, ha, la);
      split2(x[jt][2] * f0, x[jt][3] * f1, hb, lb);
      ha = movmatrix_t(ha); hb = movmatrix_t(hb); la = movmatrix_t(la); lb = movmatrix_t(lb);   // (head g, features 2t, 2t + 1)
      if (g < H) {
        const uint32_t o = c * CP + g * RS + jt * 32 + 4 * t;
        *reinterpret_cast<uint32_t*>(Qt + o) = ha;
        *reinterpret_cast<uint32_t*>(Qt + o + 16) = hb;
        *reinterpret_cast<uint32_t*>(Xlo + o) = la;
        *reinterpret_cast<uint32_t*>(Xlo + o + 16) = lb;
      }
    }
  };
  // 16-byte pieces of a candidate's head rows, lanes over (head, piece): f(head, piece, offset in a plane)
  auto pieces = [&](int c, auto f) {
    for (int i = lane; i < H * 2 * D16; i += 32) {
      const int h = i / (2 * D16), q = i - h * (2 * D16);
      f(h, q, (uint32_t)(c * CP + h * RS + q * 16));
    }
  };
  auto ld16 = [](const void* p) { return *reinterpret_cast<const uint4*>(p); };
  auto unpack = [](float (&v)[8], const uint4& x) {
    v[0] = bf16_lo(x.x); v[1] = bf16_hi(x.x); v[2] = bf16_lo(x.y); v[3] = bf16_hi(x.y);
    v[4] = bf16_lo(x.z); v[5] = bf16_hi(x.z); v[6] = bf16_lo(x.w); v[7] = bf16_hi(x.w);
  };
  auto add_lo = [](float (&v)[8], const uint4& x) {
    v[0] += bf16_lo(x.x); v[1] += bf16_hi(x.x); v[2] += bf16_lo(x.y); v[3] += bf16_hi(x.y);
    v[4] += bf16_lo(x.z); v[5] += bf16_hi(x.z); v[6] += bf16_lo(x.w); v[7] += bf16_hi(x.w);
  };
  auto split8 = [](const float (&v)[8], uint4& hi, uint4& lo) {
    split2(v[0], v[1], hi.x, lo.x); split2(v[2], v[3], hi.y, lo.y); split2(v[4], v[5], hi.z, lo.z); split2(v[6], v[7], hi.w, lo.w);
  };
  const size_t lo_d = (size_t)P.M * Nd, lo_h = (size_t)P.M * NHd;    // distance of the low-part planes in global memory

  // =============================================================================================== forward
  if (dense) {
    load_rows([&](size_t at) {
      const uint32_t v = *reinterpret_cast<const uint32_t*>(P.cands + at);
      return make_float2(bf16_lo(v), bf16_hi(v));
    });
    put_rows(tr, 1.f, Thi, Tlo, P.G.T, lo_d);
  }
  __syncthreads();
  for (int l = 0; l < P.M; ++l) {
    if (dense) {                                                     // q = t W_q
      float acc[2][4] = {};
      from_rows(acc, Thi, Tlo, weights(l, 0, 0));
      put_rows(acc, 1.f, Qhi, Qlo, P.G.Q + l * Nd, lo_d);
    }
    __syncthreads();
    if (dense) fold_heads(Qhi, Qlo, weights(l, 1, 1), P.inv_tau, Qt);   // qt_h = q_h W_k[:, h]^T / tau
    __syncthreads();
#pragma unroll 1
    for (int sl = 0; sl < n_slots; ++sl) {                           // attention, one candidate of this warp after the other
      const int c = warp + kTW * sl, cand = c_base + c, nv = nv_s[c];
      if (cand >= c_end) continue;
      const int nch = (nv + kTRows - 1) / kTRows;
      if (nch > 0) stage_chunk(cand, 0, nv, 0);
      {                                                              // the slot rows of qt, for the backward part
        bf16 *r0 = P.rows0 + ((size_t)cand * P.slots + l * 2 * H) * d, *r1 = P.rows1 + ((size_t)cand * P.slots + l * 2 * H) * d;
        pieces(c, [&](int h, int q, uint32_t o) {
          *reinterpret_cast<uint4*>(r0 + h * d + q * 8) = ld16(Qt + o);
          if (NP == 2) *reinterpret_cast<uint4*>(r1 + h * d + q * 8) = ld16(Qt + plane + o);
        });
      }
      float x[D16][4];
#pragma unroll
      for (int jt = 0; jt < D16; ++jt) x[jt][0] = x[jt][1] = x[jt][2] = x[jt][3] = 0.f;
      float rm0 = -INFINITY, rm1 = -INFINITY, rs0 = 0.f, rs1 = 0.f;
      const uint32_t q0 = head_rows(Qt, c), q1 = head_rows(Qt + plane, c);
      int b = 0;
      for (int ch = 0; ch < nch; ++ch) {
        if (P.nb > 1 && ch + 1 < nch) {
          stage_chunk(cand, ch + 1, nv, b ^ 1);
          cp_wait<1>();
        } else {
          cp_wait<0>();
        }
        __syncwarp();
        const uint32_t sb = mine_a + b * chunk_bytes;
        float e[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
        for (int kt = 0; kt < D16; ++kt) {
          uint32_t a0[4], a1[4];
          ldsm_x4(a0, sb + a_off + kt * 32);
          if (NP == 2) ldsm_x4(a1, sb + kTRows * RS + a_off + kt * 32);
          dot_tile(kt, a0, a1, q0, q1, e);
        }
        const int rows = nv - ch * kTRows;
        if (g >= rows) e[0] = e[1] = -INFINITY;
        if (g + 8 >= rows) e[2] = e[3] = -INFINITY;
        const float nm0 = fmaxf(rm0, group_max(fmaxf(e[0], e[2]))), nm1 = fmaxf(rm1, group_max(fmaxf(e[1], e[3])));
        const float sc0 = __expf(rm0 - nm0), sc1 = __expf(rm1 - nm1);
        rm0 = nm0;
        rm1 = nm1;
        const float w0 = __expf(e[0] - nm0), w1 = __expf(e[1] - nm1), w2 = __expf(e[2] - nm0), w3 = __expf(e[3] - nm1);
        rs0 = rs0 * sc0 + w0 + w2;
        rs1 = rs1 * sc1 + w1 + w3;
        if (ch > 0) {
#pragma unroll
          for (int jt = 0; jt < D16; ++jt) { x[jt][0] *= sc0; x[jt][1] *= sc1; x[jt][2] *= sc0; x[jt][3] *= sc1; }
        }
        weigh_chunk(sb, x, w0, w1, w2, w3);
        __syncwarp();                                                // every lane is done with this buffer
        if (P.nb > 1) b ^= 1;
        else if (ch + 1 < nch) stage_chunk(cand, ch + 1, nv, 0);
      }
      const float s0 = group_sum(rs0), s1 = group_sum(rs1);
      const float i0 = s0 > 0.f ? 1.f / s0 : 0.f, i1 = s1 > 0.f ? 1.f / s1 : 0.f;
      __syncwarp();
      put_heads(c, x, i0, i1);
      if (g == 0) {
        float* st = P.stat + ((size_t)(l * P.N + cand) * H) * 2;
        if (2 * t < H) *reinterpret_cast<float2*>(st + 4 * t) = make_float2(rm0, i0);
        if (2 * t + 1 < H) *reinterpret_cast<float2*>(st + 4 * t + 2) = make_float2(rm1, i1);
      }
      __syncwarp();
      bf16* mg = P.G.Mh + l * NHd + (size_t)cand * H * d;
      pieces(c, [&](int h, int q, uint32_t o) {
        *reinterpret_cast<uint4*>(mg + h * d + q * 8) = ld16(Qt + o);
        *reinterpret_cast<uint4*>(mg + lo_h + h * d + q * 8) = ld16(Xlo + o);
      });
    }
    __syncthreads();
    if (dense && l + 1 < P.M) {                                      // t += m_h W_v[:, h]  (the last layer's t is not needed)
      from_heads(tr, weights(l, 2, 0));
      put_rows(tr, 1.f, Thi, Tlo, P.G.T + (l + 1) * Nd, lo_d);
    }
    __syncthreads();
  }

  // =============================================================================================== backward
  if (dense) {                                                       // dt of the last target
    load_rows([&](size_t at) { return *reinterpret_cast<const float2*>(P.dz + at); });
    put_rows(tr, 1.f, Thi, Tlo, P.G.dT + (P.M - 1) * Nd, lo_d);
  }
  __syncthreads();
  for (int l = P.M - 1; l >= 0; --l) {
    if (dense) fold_heads(Thi, Tlo, weights(l, 2, 1), 1.f, Dm);      // dm_h = dt_h W_v[:, h]^T
    __syncthreads();
#pragma unroll 1
    for (int sl = 0; sl < n_slots; ++sl) {
      const int c = warp + kTW * sl, cand = c_base + c, nv = nv_s[c];
      if (cand >= c_end) continue;
      const int nch = (nv + kTRows - 1) / kTRows;
      if (nch > 0) stage_chunk(cand, 0, nv, 0);
      const bf16* mg = P.G.Mh + l * NHd + (size_t)cand * H * d;
      bf16 *r0 = P.rows0 + ((size_t)cand * P.slots + l * 2 * H) * d, *r1 = P.rows1 + ((size_t)cand * P.slots + l * 2 * H) * d;
      // this layer's qt rows back from the slot rows, and m . dm per head
      float dot0 = 0.f, dot1 = 0.f;                                  // heads 2t, 2t + 1
      auto piece_dot = [&](int h, int q, uint32_t o) {
        *reinterpret_cast<uint4*>(Qt + o) = ld16(r0 + h * d + q * 8);
        if (NP == 2) *reinterpret_cast<uint4*>(Qt + plane + o) = ld16(r1 + h * d + q * 8);
        float m[8], y[8], v = 0.f;
        unpack(m, ld16(mg + h * d + q * 8));
        add_lo(m, ld16(mg + lo_h + h * d + q * 8));
        unpack(y, ld16(Dm + o));
        if (NP == 2) add_lo(y, ld16(Dm + plane + o));
#pragma unroll
        for (int e = 0; e < 8; ++e) v = fmaf(m[e], y[e], v);
        return v;
      };
      if constexpr ((D16 & (D16 - 1)) == 0) {                        // whole heads per step: sums over 2 D16 lanes
        for (int i0 = 0; i0 < H * 2 * D16; i0 += 32) {
          const int i = i0 + lane, h = i / (2 * D16), q = i % (2 * D16);
          float v = h < H ? piece_dot(h, q, (uint32_t)(c * CP + h * RS + q * 16)) : 0.f;
#pragma unroll
          for (int o = 1; o < 2 * D16; o <<= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
          const int h0 = i0 / (2 * D16), per = 32 / (2 * D16);       // heads h0 .. h0 + per - 1 sit in lanes 0, 2 D16, ...
          const float v0 = __shfl_sync(0xffffffffu, v, ((2 * t - h0) * 2 * D16) & 31), v1 = __shfl_sync(0xffffffffu, v, ((2 * t + 1 - h0) * 2 * D16) & 31);
          if (2 * t >= h0 && 2 * t < h0 + per) dot0 = v0;
          if (2 * t + 1 >= h0 && 2 * t + 1 < h0 + per) dot1 = v1;
        }
      } else {
        for (int h = 0; h < H; ++h) {
          float v = lane < 2 * D16 ? piece_dot(h, lane, (uint32_t)(c * CP + h * RS + lane * 16)) : 0.f;
          v = group_sum(quad_sum(v));
          if (h == 2 * t) dot0 = v;
          if (h == 2 * t + 1) dot1 = v;
        }
      }
      __syncwarp();
      float mx0 = 0.f, iv0 = 0.f, mx1 = 0.f, iv1 = 0.f;
      {
        const float* st = P.stat + ((size_t)(l * P.N + cand) * H) * 2;
        if (2 * t < H) { mx0 = st[4 * t]; iv0 = st[4 * t + 1]; }
        if (2 * t + 1 < H) { mx1 = st[4 * t + 2]; iv1 = st[4 * t + 3]; }
      }
      float x[D16][4];
#pragma unroll
      for (int jt = 0; jt < D16; ++jt) x[jt][0] = x[jt][1] = x[jt][2] = x[jt][3] = 0.f;
      float rho0 = 0.f, rho1 = 0.f;
      const uint32_t q0 = head_rows(Qt, c), q1 = head_rows(Qt + plane, c), d0 = head_rows(Dm, c), d1 = head_rows(Dm + (NP - 1) * plane, c);
      int b = 0;
      for (int ch = 0; ch < nch; ++ch) {
        if (P.nb > 1 && ch + 1 < nch) {
          stage_chunk(cand, ch + 1, nv, b ^ 1);
          cp_wait<1>();
        } else {
          cp_wait<0>();
        }
        __syncwarp();
        const uint32_t sb = mine_a + b * chunk_bytes;
        float e[4] = {0.f, 0.f, 0.f, 0.f}, da[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
        for (int kt = 0; kt < D16; ++kt) {
          uint32_t a0[4], a1[4];
          ldsm_x4(a0, sb + a_off + kt * 32);
          if (NP == 2) ldsm_x4(a1, sb + kTRows * RS + a_off + kt * 32);
          dot_tile(kt, a0, a1, q0, q1, e);
          dot_tile(kt, a0, a1, d0, d1, da);
        }
        float a[4], de[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          const bool in = ch * kTRows + g + (k >> 1) * 8 < nv;
          a[k] = in ? __expf(e[k] - ((k & 1) ? mx1 : mx0)) * ((k & 1) ? iv1 : iv0) : 0.f;
          de[k] = a[k] * (da[k] - ((k & 1) ? dot1 : dot0));
        }
        rho0 += de[0] + de[2];
        rho1 += de[1] + de[3];
#pragma unroll
        for (int hf = 0; hf < 2; ++hf) {
          const int j = ch * kTRows + g + hf * 8;
          if (j < nv) {
            const size_t at = ((size_t)cand * Lp + j) * P.slots + l * 2 * H + 2 * t;
            if constexpr (NP == 1) {
              if (H % 2 == 0) {                                      // (slot pairs of two heads: aligned)
                if (2 * t < H) {
                  *reinterpret_cast<uint32_t*>(P.ad16 + at) = pack2(de[2 * hf], de[2 * hf + 1]);
                  *reinterpret_cast<uint32_t*>(P.ad16 + at + H) = pack2(a[2 * hf], a[2 * hf + 1]);
                }
              } else {
                if (2 * t < H) { P.ad16[at] = __float2bfloat16_rn(de[2 * hf]); P.ad16[at + H] = __float2bfloat16_rn(a[2 * hf]); }
                if (2 * t + 1 < H) { P.ad16[at + 1] = __float2bfloat16_rn(de[2 * hf + 1]); P.ad16[at + H + 1] = __float2bfloat16_rn(a[2 * hf + 1]); }
              }
            } else {
              if (2 * t < H) { P.ad32[at] = de[2 * hf]; P.ad32[at + H] = a[2 * hf]; }
              if (2 * t + 1 < H) { P.ad32[at + 1] = de[2 * hf + 1]; P.ad32[at + H + 1] = a[2 * hf + 1]; }
            }
          }
        }
        weigh_chunk(sb, x, de[0], de[1], de[2], de[3]);
        __syncwarp();
        if (P.nb > 1) b ^= 1;
        else if (ch + 1 < nch) stage_chunk(cand, ch + 1, nv, 0);
      }
      // what the rounding of m leaves of sum_j de: taken out of every de_j (rho a_j), i.e. of dqt (rho m) and of the dm rows
      rho0 = group_sum(rho0);
      rho1 = group_sum(rho1);
      auto rho_of = [&](int h) {                                     // (called by all lanes)
        const float a0 = __shfl_sync(0xffffffffu, rho0, (h >> 1) & 3), a1 = __shfl_sync(0xffffffffu, rho1, (h >> 1) & 3);
        return (h & 1) ? a1 : a0;
      };
      const int n_pieces = H * 2 * D16;
      for (int i0 = 0; i0 < n_pieces; i0 += 32) {                    // dm rows
        const int i = min(i0 + lane, n_pieces - 1), h = i / (2 * D16), q = i - h * (2 * D16);
        const uint32_t o = c * CP + h * RS + q * 16;
        const float rho = rho_of(h);
        float m[8], y[8];
        unpack(m, ld16(Qt + o));
        unpack(y, ld16(Dm + o));
        if (NP == 2) { add_lo(m, ld16(Qt + plane + o)); add_lo(y, ld16(Dm + plane + o)); }
#pragma unroll
        for (int e = 0; e < 8; ++e) y[e] = fmaf(-rho, m[e], y[e]);
        uint4 hi, lo;
        split8(y, hi, lo);
        *reinterpret_cast<uint4*>(r0 + (H + h) * d + q * 8) = hi;
        if (NP == 2) *reinterpret_cast<uint4*>(r1 + (H + h) * d + q * 8) = lo;
      }
      __syncwarp();
      put_heads(c, x, 1.f, 1.f);
      __syncwarp();
      bf16* dg = P.G.dQt + l * NHd + (size_t)cand * H * d;
      for (int i0 = 0; i0 < n_pieces; i0 += 32) {                    // dqt rows
        const int i = i0 + lane, h = min(i / (2 * D16), H - 1), q = i % (2 * D16);
        const float rho = rho_of(h);
        if (i < n_pieces) {
          const uint32_t o = c * CP + h * RS + q * 16;
          float m[8], y[8];
          unpack(m, ld16(mg + h * d + q * 8));
          add_lo(m, ld16(mg + lo_h + h * d + q * 8));
          unpack(y, ld16(Qt + o));
          add_lo(y, ld16(Xlo + o));
#pragma unroll
          for (int e = 0; e < 8; ++e) y[e] = fmaf(-rho, m[e], y[e]);
          uint4 hi, lo;
          split8(y, hi, lo);
          *reinterpret_cast<uint4*>(Qt + o) = hi;
          *reinterpret_cast<uint4*>(Xlo + o) = lo;
          *reinterpret_cast<uint4*>(dg + h * d + q * 8) = hi;
          *reinterpret_cast<uint4*>(dg + lo_h + h * d + q * 8) = lo;
        }
      }
    }
    __syncthreads();
    if (dense) {                                                     // dq_h = dqt_h W_k[:, h] / tau
      float acc[2][4] = {};
      from_heads(acc, weights(l, 1, 0));
      put_rows(acc, P.inv_tau, Qhi, Qlo, P.G.dQ + l * Nd, lo_d);
    }
    __syncthreads();
    if (dense) {                                                     // dt += dq W_q^T
      from_rows(tr, Qhi, Qlo, weights(l, 0, 1));
      if (l > 0) put_rows(tr, 1.f, Thi, Tlo, P.G.dT + (l - 1) * Nd, lo_d);
    }
    __syncthreads();
  }
  if (dense) {
#pragma unroll
    for (int nt = 0; nt < 2; ++nt)
#pragma unroll
      for (int hf = 0; hf < 2; ++hf)
        if (c_base + g + hf * 8 < c_end)
          *reinterpret_cast<float2*>(P.G.dT0 + (size_t)(c_base + g + hf * 8) * d + wcol + nt * 8 + 2 * t) =
              make_float2(tr[nt][2 * hf], tr[nt][2 * hf + 1]);
  }

  // =============================================================================================== dH'
  // rows = segments, k = slots: A from the de / a array, B = the candidate's slot rows, staged once if all of them fit the
  // buffers and otherwise kb steps of 16 at a time for every 16 segments (any number of layers and heads, with the sums
  // of all features in registers).  One candidate per user, d = 128, 8 heads: 256 users of 1000 items in 100 segments, 2 layers,
  // 369 us a call (616 with the attention on the FP32 ALUs); 2048 users of 500 items 872 (1172).
  const int KS = (P.slots + 15) >> 4;
  const bool resident = P.kb >= KS, out16 = NP == 1 || P.dS16 != nullptr;
  const bool staged = out16 && (!resident || P.nb > KS);             // 16 rows of a buffer are free for the result
  uint8_t* result = resident ? mine + 16 * KS * NP * RS : mine;
  const int mi = lane >> 3, lr = lane & 7;
  const uint32_t s_trans = ((mi & 1) * 8 + lr) * RS + (mi >> 1) * 16;
  const uint32_t s_plane = P.kb * 16 * RS;
  auto stage_slots = [&](int cand, int k0) {                         // steps k0 .. k0 + kb - 1, planes of 16 kb rows
    const int n = 16 * min(P.kb, KS - k0) * 2 * D16;
#pragma unroll
    for (int pl = 0; pl < NP; ++pl) {
      const bf16* src = (pl ? P.rows1 : P.rows0) + ((size_t)cand * P.slots + k0 * 16) * d;
      for (int i = lane; i < n; i += 32) {
        const int r = i / (2 * D16), q = i % (2 * D16);
        const bool ok = k0 * 16 + r < P.slots;
        cp16(mine_a + pl * s_plane + r * RS + q * 16, ok ? (const void*)(src + r * d + q * 8) : (const void*)P.S0, ok ? 16u : 0u);
      }
    }
    cp_commit();
    cp_wait<0>();
    __syncwarp();
  };
#pragma unroll 1
  for (int sl = 0; sl < n_slots; ++sl) {
    const int c = warp + kTW * sl, cand = c_base + c, nv = nv_s[c];
    if (cand >= c_end) continue;
    __syncwarp();
    if (resident && nv > 0) stage_slots(cand, 0);
    for (int j0 = 0; j0 < nv; j0 += kTRows) {
      float x[D16][2][4];
#pragma unroll
      for (int jp = 0; jp < D16; ++jp)
#pragma unroll
        for (int e = 0; e < 4; ++e) x[jp][0][e] = x[jp][1][e] = 0.f;
#pragma unroll 1
      for (int ks = 0; ks < KS; ++ks) {
        uint32_t ah[4], al[4];
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          const int j = j0 + g + (e & 1) * 8, s = ks * 16 + 2 * t + (e >> 1) * 8;
          const bool in = j < nv && s < P.slots;
          const size_t at = ((size_t)cand * Lp + j) * P.slots + s;
          if constexpr (NP == 1) {
            ah[e] = in ? *reinterpret_cast<const uint32_t*>(P.ad16 + at) : 0u;
          } else {
            const float2 v = in ? *reinterpret_cast<const float2*>(P.ad32 + at) : make_float2(0.f, 0.f);
            split2(v.x, v.y, ah[e], al[e]);
          }
        }
        const int k = ks % P.kb;
        if (!resident && k == 0) {
          __syncwarp();                                              // every lane is done with the rows before
          stage_slots(cand, ks);
        }
        const uint32_t row = mine_a + k * 16 * RS + s_trans;
#pragma unroll
        for (int jp = 0; jp < D16; ++jp) {
          uint32_t b[4];
          ldsm_x4_t(b, row + jp * 32);
          mma16816(x[jp][0], ah[0], ah[1], ah[2], ah[3], b[0], b[1]);
          mma16816(x[jp][1], ah[0], ah[1], ah[2], ah[3], b[2], b[3]);
          if constexpr (NP == 2) {
            mma16816(x[jp][0], al[0], al[1], al[2], al[3], b[0], b[1]);
            mma16816(x[jp][1], al[0], al[1], al[2], al[3], b[2], b[3]);
            ldsm_x4_t(b, row + s_plane + jp * 32);
            mma16816(x[jp][0], ah[0], ah[1], ah[2], ah[3], b[0], b[1]);
            mma16816(x[jp][1], ah[0], ah[1], ah[2], ah[3], b[2], b[3]);
          }
        }
      }
      if (staged) {                                                  // through shared memory: whole rows leave in 16-byte pieces
        if (!resident) __syncwarp();
#pragma unroll
        for (int jp = 0; jp < D16; ++jp) {
          uint8_t* o = result + g * RS + jp * 32 + 4 * t;
          *reinterpret_cast<uint32_t*>(o) = pack2(x[jp][0][0], x[jp][0][1]);
          *reinterpret_cast<uint32_t*>(o + 16) = pack2(x[jp][1][0], x[jp][1][1]);
          *reinterpret_cast<uint32_t*>(o + 8 * RS) = pack2(x[jp][0][2], x[jp][0][3]);
          *reinterpret_cast<uint32_t*>(o + 8 * RS + 16) = pack2(x[jp][1][2], x[jp][1][3]);
        }
        __syncwarp();
        bf16* out = P.dS16 + ((size_t)cand * Lp + j0) * d;
#pragma unroll
        for (int i = 0; i < D16; ++i) {
          const int piece = i * 32 + lane, r = piece / (2 * D16), q = piece - r * (2 * D16);
          if (j0 + r < nv) *reinterpret_cast<uint4*>(out + r * d + q * 8) = ld16(result + r * RS + q * 16);
        }
        __syncwarp();
        continue;
      }
#pragma unroll
      for (int hf = 0; hf < 2; ++hf) {
        const int j = j0 + g + hf * 8;
        if (j >= nv) continue;
#pragma unroll
        for (int jp = 0; jp < D16; ++jp) {
          const size_t at = ((size_t)cand * Lp + j) * d + jp * 16 + 2 * t;
          if (out16) {
            *reinterpret_cast<uint32_t*>(P.dS16 + at) = pack2(x[jp][0][2 * hf], x[jp][0][2 * hf + 1]);
            *reinterpret_cast<uint32_t*>(P.dS16 + at + 8) = pack2(x[jp][1][2 * hf], x[jp][1][2 * hf + 1]);
          } else {
            *reinterpret_cast<float2*>(P.dS32 + at) = make_float2(x[jp][0][2 * hf], x[jp][0][2 * hf + 1]);
            *reinterpret_cast<float2*>(P.dS32 + at + 8) = make_float2(x[jp][1][2 * hf], x[jp][1][2 * hf + 1]);
          }
        }
      }
    }
  }
}

// Weight gradients: C[m][n] += alpha sum_r A_h[r][m] B[r][n], h = the head of column n (A: [rows, heads, d], B: [rows, d],
// both as bf16 high and low parts: three products per term), for up to kMaxSums arrays in one launch.  A block takes a slice
// of the rows, KR at a time through two shared-memory buffers, and keeps the whole d x d sum in its registers: one atomic
// add per element and block at the end.
constexpr int kMaxSums = 24;
struct SumList {
  const bf16 *A[kMaxSums], *B[kMaxSums];
  size_t a_lo[kMaxSums], b_lo[kMaxSums];            // distance of the low parts, in elements
  float* C[kMaxSums];
  float alpha[kMaxSums];
  int heads[kMaxSums];
};
template <int D16>
__global__ void __launch_bounds__(256, 2) weight_sums_kernel(const __grid_constant__ SumList L, int R, int rows_per_block, int KR,
                                                             int dvh) {
  constexpr int d = 16 * D16, kParts = 8 / D16 > 0 ? 8 / D16 : 1, kPairs = (D16 + kParts - 1) / kParts;
  extern __shared__ __align__(128) uint8_t smem[];
  chain_wait();
  chain_release();
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, g = lane >> 2, t = lane & 3;
  const bf16 *A = L.A[blockIdx.y], *B = L.B[blockIdx.y];
  const size_t a_lo = L.a_lo[blockIdx.y], b_lo = L.b_lo[blockIdx.y];
  const int heads = L.heads[blockIdx.y], lda = heads * d, AS = 2 * lda + 16, BS = 2 * d + 16;
  const int hw = heads == 1 ? d : dvh;                               // columns of a head
  const uint32_t a_plane = KR * AS, b_plane = KR * BS, buf_bytes = 2 * (a_plane + b_plane);
  const uint32_t base = smem_addr(smem);
  const int mtile = warp % D16, part = warp / D16;                   // 16 rows of C; column pairs part, part + kParts, ...
  const bool active = part < kParts;
  float acc[kPairs][2][4];
#pragma unroll
  for (int j = 0; j < kPairs; ++j)
#pragma unroll
    for (int e = 0; e < 4; ++e) acc[j][0][e] = acc[j][1][e] = 0.f;
  const int r_lo = blockIdx.x * rows_per_block, r_hi = min(R, r_lo + rows_per_block);
  if (r_lo >= r_hi) return;
  auto stage = [&](int r0, int b) {
    const uint32_t dst = base + b * buf_bytes;
    const int ca = lda / 8, cb = d / 8;
    for (int rr = warp; rr < KR; rr += 8) {                          // a warp per row: no divisions by the run-time row width
      const uint32_t n = r0 + rr < r_hi ? 16u : 0u;
      const bf16 *sa = A + (size_t)min(r0 + rr, r_hi - 1) * lda, *sb = B + (size_t)min(r0 + rr, r_hi - 1) * d;
      for (int c = lane; c < ca; c += 32) {
        cp16(dst + rr * AS + c * 16, sa + c * 8, n);
        cp16(dst + a_plane + rr * AS + c * 16, sa + a_lo + c * 8, n);
      }
      for (int c = lane; c < cb; c += 32) {
        cp16(dst + 2 * a_plane + rr * BS + c * 16, sb + c * 8, n);
        cp16(dst + 2 * a_plane + b_plane + rr * BS + c * 16, sb + b_lo + c * 8, n);
      }
    }
    cp_commit();
  };
  const int mi = lane >> 3, lr = lane & 7;
  const uint32_t a_off = ((mi >> 1) * 8 + lr) * AS + mtile * 32 + (mi & 1) * 16;      // A^T: rows = columns of A
  const uint32_t b_off = ((mi & 1) * 8 + lr) * BS + (mi >> 1) * 16;
  uint32_t head_at[kPairs];                                          // byte offset of each column pair's head in a row of A
#pragma unroll
  for (int j = 0; j < kPairs; ++j) head_at[j] = (uint32_t)min((part + kParts * j) * 16 / hw, heads - 1) * (2 * d);
  stage(r_lo, 0);
  int b = 0;
  for (int r0 = r_lo; r0 < r_hi; r0 += KR, b ^= 1) {
    if (r0 + KR < r_hi) {
      stage(r0 + KR, b ^ 1);
      cp_wait<1>();
    } else {
      cp_wait<0>();
    }
    __syncthreads();
    const uint32_t as = base + b * buf_bytes + a_off, bs = base + b * buf_bytes + 2 * a_plane + b_off;
    if (active)
      for (int k = 0; k < KR; k += 16) {
        uint32_t ah[4], al[4];
#pragma unroll
        for (int j = 0; j < kPairs; ++j) {
          const int p = part + kParts * j;
          if (p < D16) {
            if (j == 0 || head_at[j] != head_at[j > 0 ? j - 1 : 0]) {
              ldsm_x4_t(ah, as + k * AS + head_at[j]);
              ldsm_x4_t(al, as + a_plane + k * AS + head_at[j]);
            }
            uint32_t bh[4], bl[4];
            ldsm_x4_t(bh, bs + k * BS + p * 32);
            ldsm_x4_t(bl, bs + b_plane + k * BS + p * 32);
            mma16816(acc[j][0], ah[0], ah[1], ah[2], ah[3], bh[0], bh[1]);
            mma16816(acc[j][1], ah[0], ah[1], ah[2], ah[3], bh[2], bh[3]);
            mma16816(acc[j][0], al[0], al[1], al[2], al[3], bh[0], bh[1]);
            mma16816(acc[j][1], al[0], al[1], al[2], al[3], bh[2], bh[3]);
            mma16816(acc[j][0], ah[0], ah[1], ah[2], ah[3], bl[0], bl[1]);
            mma16816(acc[j][1], ah[0], ah[1], ah[2], ah[3], bl[2], bl[3]);
          }
        }
      }
    __syncthreads();
  }
  if (!active) return;
  float* C = L.C[blockIdx.y];
  const float alpha = L.alpha[blockIdx.y];
#pragma unroll
  for (int j = 0; j < kPairs; ++j) {
    const int p = part + kParts * j;
    if (p < D16) {
#pragma unroll
      for (int nt = 0; nt < 2; ++nt) red_tile(C + (size_t)mtile * 16 * d + p * 16 + nt * 8, d, acc[j][nt], alpha, lane);
    }
  }
}

struct TrainScratch {
  uint4* img;
  int *nseg, *order, *keys;
  float *stat, *ad32;
  bf16* ad16;
  bf16 *rows0, *rows1;
  size_t total;
};
TrainScratch carve_train(const Plan& p, int np, char* base) {
  TrainScratch s;
  size_t off = 0;
  auto take = [&](size_t bytes) {
    char* q = base ? base + off : nullptr;
    off = align_up(off + bytes) + kGuardBytes;
    return q;
  };
  const size_t N = p.N, slots = 2 * (size_t)p.M * p.H, blocks = (N + 7) / 8;
  s.img = (uint4*)take((size_t)p.M * 6 * p.d * p.d * 2);
  s.nseg = (int*)take(N * sizeof(int));
  s.order = (int*)take(blocks * sizeof(int));
  s.keys = (int*)take(blocks * sizeof(int));
  s.stat = (float*)take((size_t)p.M * N * p.H * 2 * sizeof(float));
  s.ad16 = np == 1 ? (bf16*)take(N * p.Lp * slots * sizeof(bf16)) : nullptr;
  s.ad32 = np == 2 ? (float*)take(N * p.Lp * slots * sizeof(float)) : nullptr;
  s.rows0 = (bf16*)take(N * slots * p.d * sizeof(bf16));
  s.rows1 = np == 2 ? (bf16*)take(N * slots * p.d * sizeof(bf16)) : nullptr;
  s.total = off;
  return s;
}

// 8 candidates per block (one per warp) while all blocks still run at once, two per SM
int train_cpb(const Plan& p) { return (p.N + 7) / 8 <= 2 * device_sms() ? 8 : kTRows; }

template <int D16, int NP>
int launch_train(TrainParams P, const TrainPrep& prep, const Plan& p, bool prepared, cudaStream_t st) {
  P.cpb = prep.cpb;
  P.order = prep.order;
  const int blocks = (p.N + P.cpb - 1) / P.cpb;
  if (!prepared) {
    const int total = p.M * 6 * D16 * D16 * 32;
    LaunchScope ls("gsta_train_prep", st);
    LASER_CUDA_OK(launch_chained(train_prep_kernel, dim3(std::min((total + 255) / 256, 4 * device_sms()) + (prep.order ? 1 : 0)), dim3(256),
                                 0, st, prep));
  }
  const size_t smem = TrainSmem<D16, NP>::bytes(p.H, P.nb);
  LASER_CUDA_OK(allow_smem(gsta_train_kernel<D16, NP>, smem));
  LaunchScope ls("gsta_train", st);
  LASER_CUDA_OK(launch_chained(gsta_train_kernel<D16, NP>, dim3(blocks), dim3(kTThreads), smem, st, P));
  return LASER_OK;
}

template <int D16>
int launch_sums(const Plan& p, const GstaPlanes& G, float* dWg, cudaStream_t st) {
  const size_t Nd = (size_t)p.N * p.d, dd = (size_t)p.d * p.d, lo_d = (size_t)p.M * Nd, lo_h = lo_d * p.H;
  const size_t row = 2 * 2 * (2 * ((size_t)p.H * p.d + p.d) + 32);    // bytes per row in two buffers of two parts
  const int KR = row * 32 <= 110 * 1024 ? 32 : 16;
  const size_t smem = row * KR;
  LASER_CUDA_OK(allow_smem(weight_sums_kernel<D16>, smem));
  for (int l0 = 0; l0 < p.M; l0 += kMaxSums / 3) {
    SumList L;
    int n = 0;
    for (int l = l0; l < p.M && n + 3 <= kMaxSums; ++l) {
      float *gWq = dWg + (size_t)(l * 3) * dd, *gWk = gWq + dd, *gWv = gWk + dd;
      auto add = [&](const bf16* A, size_t a_lo, int heads, const bf16* B, float* C, float alpha) {
        L.A[n] = A; L.a_lo[n] = a_lo; L.B[n] = B; L.b_lo[n] = lo_d; L.C[n] = C; L.alpha[n] = alpha; L.heads[n] = heads;
        ++n;
      };
      add(G.Mh + l * Nd * p.H, lo_h, p.H, G.dT + l * Nd, gWv, 1.f);
      add(G.dQt + l * Nd * p.H, lo_h, p.H, G.Q + l * Nd, gWk, p.inv_tau);
      add(G.T + l * Nd, lo_d, 1, G.dQ + l * Nd, gWq, 1.f);
    }
    // about one wave of two blocks per SM over all sums
    const int want = std::max(1, 2 * device_sms() / n);
    const int per = std::max(KR, ((p.N + want - 1) / want + KR - 1) / KR * KR);
    LaunchScope ls("gsta_weight_sums", st);
    LASER_CUDA_OK(launch_chained(weight_sums_kernel<D16>, dim3((p.N + per - 1) / per, n), dim3(256), smem, st, L, p.N, per, KR, p.dvh));
  }
  return LASER_OK;
}

int train_slot_steps(const Plan& p) { return (2 * p.M * p.H + 15) / 16; }

size_t train_smem(const Plan& p, int np, int nb) {
  const size_t RS = 2 * p.d + 16;
  return 2 * (size_t)kTRows * RS + 2 * np * (size_t)kTRows * (p.H * RS + (p.H % 2 ? 0 : 16)) + RS + kTRows * sizeof(int) + 48 +
         (size_t)kTW * nb * kTRows * RS * np;
}

constexpr size_t kTrainSmemMax = 226 * 1024, kSmemPerSm = 228 * 1024, kSmemPerBlock = 1024;    // (the last: reserved by the system)
int train_blocks_per_sm(const Plan& p, int np, int nb) { return (int)std::min<size_t>(2, kSmemPerSm / (train_smem(p, np, nb) + kSmemPerBlock)); }

// Staging buffers of a warp: two of one part (the next 16 segments arrive while these are worked on), one of two parts (a second
// one, where it costs no block, changed nothing: 116 us at 256 users, 8 heads; 420 at lists of d = 96, 6 heads), and as many as the
// slot rows need where that costs no block per SM.
int train_buffers(const Plan& p, int np) {
  const int base = np == 1 ? 2 : 1, all = train_slot_steps(p);
  return all > base && train_smem(p, np, all) <= kTrainSmemMax && train_blocks_per_sm(p, np, all) == train_blocks_per_sm(p, np, base) ? all : base;
}

}  // namespace

bool gsta_train_supported(const Plan& p, int np) {
  return p.dtype == LASER_BF16 && p.M > 0 && p.d % 16 == 0 && p.d >= 16 && p.d <= 128 && p.H <= 8 && p.dvh % 16 == 0 &&
         train_smem(p, np, np == 1 ? 2 : 1) <= kTrainSmemMax;
}
size_t gsta_train_scratch_bytes(const Plan& p, int np) { return gsta_train_supported(p, np) ? carve_train(p, np, nullptr).total : 0; }

#define LASER_TRAIN_DISPATCH(call)        \
  switch (p.d / 16) {                     \
    case 1: return call(1);               \
    case 2: return call(2);               \
    case 3: return call(3);               \
    case 4: return call(4);               \
    case 5: return call(5);               \
    case 6: return call(6);               \
    case 7: return call(7);               \
    case 8: return call(8);               \
    default: return LASER_ERR_UNSUPPORTED; \
  }

TrainPrep gsta_train_prep(const Plan& p, int np, const void* Wg, const int32_t* lengths, const int32_t* cand_offsets, char* scratch) {
  const TrainScratch s = carve_train(p, np, scratch);
  TrainPrep P;
  P.Wg = (const bf16*)Wg; P.img = s.img; P.lengths = lengths; P.cand_offsets = cand_offsets;
  P.d = p.d; P.M = p.M; P.U = p.U; P.N = p.N; P.L = p.L; P.S = p.S; P.Lp = p.Lp; P.cpb = train_cpb(p);
  P.nseg = s.nseg;
  P.order = (p.N + P.cpb - 1) / P.cpb > 2 * device_sms() ? s.order : nullptr;
  P.keys = s.keys;
  return P;
}

int gsta_train(const Plan& p, int np, const void* S0, const void* S1, const int32_t* lengths, const int32_t* cand_offsets,
               const void* cands, const void* Wg, const float* dz, const GstaPlanes& G, float* dS32, __nv_bfloat16* dS16, char* scratch,
               cudaStream_t st, bool prepared) {
  const TrainScratch s = carve_train(p, np, scratch);
  const TrainPrep prep = gsta_train_prep(p, np, Wg, lengths, cand_offsets, scratch);
  TrainParams P = {};
  P.N = p.N; P.U = p.U; P.L = p.L; P.S = p.S; P.Lp = p.Lp; P.H = p.H; P.M = p.M; P.slots = 2 * p.M * p.H; P.nb = train_buffers(p, np);
  P.kb = std::min(P.nb, train_slot_steps(p));
  P.inv_tau = p.inv_tau;
  P.S0 = (const bf16*)S0; P.S1 = (const bf16*)S1; P.cands = (const bf16*)cands; P.dz = dz;
  P.img = s.img; P.nseg = s.nseg; P.G = G; P.stat = s.stat; P.rows0 = s.rows0; P.rows1 = s.rows1; P.ad16 = s.ad16; P.ad32 = s.ad32;
  P.dS16 = dS16; P.dS32 = dS32;
#define LASER_TRAIN_CALL(D) (np == 1 ? launch_train<D, 1>(P, prep, p, prepared, st) : launch_train<D, 2>(P, prep, p, prepared, st))
  LASER_TRAIN_DISPATCH(LASER_TRAIN_CALL)
#undef LASER_TRAIN_CALL
}

int gsta_weight_sums(const Plan& p, const GstaPlanes& G, float* dWg, cudaStream_t st) {
#define LASER_TRAIN_CALL(D) launch_sums<D>(p, G, dWg, st)
  LASER_TRAIN_DISPATCH(LASER_TRAIN_CALL)
#undef LASER_TRAIN_CALL
}

}  // namespace laser

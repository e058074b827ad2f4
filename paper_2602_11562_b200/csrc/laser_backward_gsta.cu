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
  int N, U, L, S, Lp, H, M, cpb, slots, nb;       // slots = 2 M H; nb staging buffers per warp
  float inv_tau;
  const bf16 *S0, *S1;                            // [N, Lp, d] segment vectors: high (or only) and low parts
  const bf16* cands;
  const float* dz;
  const uint4* img;                               // [M][3][2][d/16][d/16][32]: W_q, W_k, W_v as stored and transposed
  const int *nseg, *order;
  GstaTrain G;
  float* stat;                                    // [M, N, H, 2] softmax maximum and 1 / sum
  bf16 *rows0, *rows1;                            // [N, slots, d] qt and dm per slot (high, low)
  float* ad;                                      // [N, Lp, slots] de and a per slot
  bf16* dS16;                                     // [N, Lp, d] out (NP = 1)
  float* dS32;                                    // [N, Lp, d] out (NP = 2)
};

// Weight images in MMA fragment order (see laser_gsta_img.cuh), each matrix as stored (B[k][n] = W[k][n]) and transposed.
__global__ void __launch_bounds__(256) train_prep_kernel(const bf16* Wg, uint4* img, int d, int M, const int* lengths,
                                                         const int* cand_offsets, int U, int N, int L, int S, int Lp, int cpb,
                                                         int* nseg, int* order, int* keys) {
  const int n_blocks = gridDim.x - (order ? 1 : 0);
  if ((int)blockIdx.x == n_blocks) {
    gsta_build_order(lengths, cand_offsets, U, N, L, S, Lp, cpb, order, keys);
    return;
  }
  const int D16 = d >> 4, total = M * 6 * D16 * D16 * 32, workers = n_blocks * 256;
  const int worker = blockIdx.x * 256 + threadIdx.x;
  for (int i = worker; i < total; i += workers) {
    const int lane = i & 31;
    int r = i >> 5;
    const int p = r % D16; r /= D16;
    const int kt = r % D16; r /= D16;
    const bool trans = r & 1;
    const uint16_t* W = reinterpret_cast<const uint16_t*>(Wg) + (size_t)(r >> 1) * d * d;
    const int g = lane >> 2, t = lane & 3;
    uint32_t v[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const int n = (2 * p + (q >> 1)) * 8 + g, k = kt * 16 + 2 * t + (q & 1) * 8;
      const uint32_t lo = trans ? W[(size_t)n * d + k] : W[(size_t)k * d + n];
      const uint32_t hi = trans ? W[(size_t)n * d + k + 1] : W[(size_t)(k + 1) * d + n];
      v[q] = lo | (hi << 16);
    }
    img[i] = make_uint4(v[0], v[1], v[2], v[3]);
  }
  gsta_build_nseg(lengths, cand_offsets, U, N, L, S, Lp, nullptr, nseg, worker >> 5, workers >> 5, threadIdx.x & 31);
}

// x -> (high, low) bf16 pairs of two floats
__device__ __forceinline__ void split2(float x0, float x1, uint32_t& hi, uint32_t& lo) {
  hi = pack2(x0, x1);
  lo = pack2(x0 - bf16_lo(hi), x1 - bf16_hi(hi));
}

template <int D16, int NP>
struct TrainSmem {
  static constexpr int d = 16 * D16, RS = 2 * d + 16, TS = d + 8;
  static __host__ __device__ constexpr size_t plane(int H) { return (size_t)kTRows * H * RS; }
  static size_t bytes(int H, int nb) {
    return (size_t)kTRows * TS * 4 + 2 * NP * plane(H) + RS + kTRows * sizeof(int) + 48 + (size_t)kTW * nb * kTRows * RS * NP;
  }
};

template <int D16, int NP>
__global__ void __launch_bounds__(kTThreads, 2) gsta_train_kernel(const __grid_constant__ TrainParams P) {
  using SM = TrainSmem<D16, NP>;
  constexpr int d = SM::d, RS = SM::RS, TS = SM::TS;
  extern __shared__ __align__(128) uint8_t smem[];
  const int H = P.H, Lp = P.Lp, dvh = d / H, KH = dvh >> 4;
  const uint32_t plane = (uint32_t)SM::plane(H);
  float* Ts = reinterpret_cast<float*>(smem);                        // [16][TS]  t, later dt
  uint8_t* Qt = smem + kTRows * TS * 4;                              // [NP][16][H] rows: qt; m or dqt (high) later
  uint8_t* Dm = Qt + NP * plane;                                     // [NP][16][H] rows: dm; NP = 1: also m or dqt (low)
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
  for (int i = tid; i < kTRows * (d / 8); i += kTThreads) {
    const int r = i / (d / 8), c8 = (i - r * (d / 8)) * 8;
    uint4 v = make_uint4(0, 0, 0, 0);
    if (c_base + r < c_end) v = *reinterpret_cast<const uint4*>(P.cands + (size_t)(c_base + r) * d + c8);
    float* dst = Ts + r * TS + c8;
    dst[0] = bf16_lo(v.x); dst[1] = bf16_hi(v.x); dst[2] = bf16_lo(v.y); dst[3] = bf16_hi(v.y);
    dst[4] = bf16_lo(v.z); dst[5] = bf16_hi(v.z); dst[6] = bf16_lo(v.w); dst[7] = bf16_hi(v.w);
  }
  for (int i = tid; i < RS / 4; i += kTThreads) reinterpret_cast<uint32_t*>(zrow)[i] = 0u;
  for (uint32_t i = tid * 4; i < 2 * NP * plane; i += kTThreads * 4) *reinterpret_cast<uint32_t*>(Qt + i) = 0u;   // (rows of absent candidates)
  __syncthreads();

  // ---- dense building blocks.  Weight fragments of k-tile kt for this warp's columns: image entry (kt, warp).
  auto weights = [&](int l, int m, int trans) { return P.img + (size_t)((l * 3 + m) * 2 + trans) * kImg + (size_t)warp * 32 + lane; };
  // high / low A fragments of k-tile kt of the fp32 rows in Ts
  auto ts_frag = [&](int kt, uint32_t (&hi)[4], uint32_t (&lo)[4]) {
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      const float2 x = *reinterpret_cast<const float2*>(Ts + (g + (e & 1) * 8) * TS + kt * 16 + 2 * t + (e >> 1) * 8);
      split2(x.x, x.y, hi[e], lo[e]);
    }
  };
  auto mma_pair = [&](float (&acc)[2][4], const uint32_t (&a)[4], const uint4& b) {
    mma16816(acc[0], a[0], a[1], a[2], a[3], b.x, b.y);
    mma16816(acc[1], a[0], a[1], a[2], a[3], b.z, b.w);
  };
  const uint32_t ldsm_row = (lane & 7) + ((lane >> 3) & 1) * 8, ldsm_kc = lane >> 4;
  // acc = x_h W with x rows (row r H + h of the planes hi, lo), h = the head of this warp's columns
  auto from_heads = [&](float (&acc)[2][4], const uint4* w) {
    const uint32_t o = (ldsm_row * H + wcol / dvh) * RS + ldsm_kc * 16;
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
  // rows of a [16][d] result: fp32 to global memory (dst, N rows of d) and as high / low rows for the next product
  auto put_rows = [&](const float (&acc)[2][4], float scale, float* dst, bool split) {
#pragma unroll
    for (int nt = 0; nt < 2; ++nt)
#pragma unroll
      for (int hf = 0; hf < 2; ++hf) {
        const int r = g + hf * 8, col = wcol + nt * 8 + 2 * t;
        const float x0 = acc[nt][2 * hf] * scale, x1 = acc[nt][2 * hf + 1] * scale;
        if (c_base + r < c_end) *reinterpret_cast<float2*>(dst + (size_t)(c_base + r) * d + col) = make_float2(x0, x1);
        if (split) {
          uint32_t hi, lo;
          split2(x0, x1, hi, lo);
          *reinterpret_cast<uint32_t*>(Qhi + r * RS + col * 2) = hi;
          *reinterpret_cast<uint32_t*>(Qlo + r * RS + col * 2) = lo;
        }
      }
  };
  auto save_rows = [&](float* dst) {                                 // the block's rows of Ts to global memory
    for (int i = tid; i < kTRows * (d / 4); i += kTThreads) {
      const int r = i / (d / 4), c4 = (i - r * (d / 4)) * 4;
      if (c_base + r < c_end)
        *reinterpret_cast<float4*>(dst + (size_t)(c_base + r) * d + c4) = *reinterpret_cast<const float4*>(Ts + r * TS + c4);
    }
  };
  auto add_rows = [&](const float (&acc)[2][4]) {                    // Ts += this warp's columns
#pragma unroll
    for (int nt = 0; nt < 2; ++nt) {
      const int col = wcol + nt * 8 + 2 * t;
      float2* r0 = reinterpret_cast<float2*>(Ts + g * TS + col);
      float2* r1 = reinterpret_cast<float2*>(Ts + (g + 8) * TS + col);
      float2 v0 = *r0, v1 = *r1;
      v0.x += acc[nt][0]; v0.y += acc[nt][1];
      v1.x += acc[nt][2]; v1.y += acc[nt][3];
      *r0 = v0;
      *r1 = v1;
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
    return smem_addr(((lane & 7) < H ? base + (c * H + (lane & 7)) * RS : zrow) + ((lane >> 3) & 1) * 16);
  };
  // e += S x^T for one staged chunk, x = head rows at b0 (and b1: low parts)
  auto dot_tile = [&](uint32_t sb, int kt, const uint32_t (&a0)[4], const uint32_t (&a1)[4], uint32_t b0, uint32_t b1, float (&e)[4]) {
    (void)sb;
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
  // rows [head][feature] of candidate c from x^T (scaled per head): high parts to Qt, low parts to Xlo, fp32 to dst [H, d]
  auto put_heads = [&](int c, const float (&x)[D16][4], float f0, float f1, float* dst) {
    const int h0 = 2 * t, h1 = 2 * t + 1;
#pragma unroll
    for (int jt = 0; jt < D16; ++jt) {
      const float v0 = x[jt][0] * f0, v1 = x[jt][1] * f1, v2 = x[jt][2] * f0, v3 = x[jt][3] * f1;
      if (dst) {
        if (h0 < H) { dst[h0 * d + jt * 16 + g] = v0; dst[h0 * d + jt * 16 + g + 8] = v2; }
        if (h1 < H) { dst[h1 * d + jt * 16 + g] = v1; dst[h1 * d + jt * 16 + g + 8] = v3; }
      }
      uint32_t ha, la, hb, lb;
      split2(v0, v1, ha, la);
      split2(v2, v3, hb, lb);
      ha = movmatrix_t(ha); hb = movmatrix_t(hb); la = movmatrix_t(la); lb = movmatrix_t(lb);   // (head g, features 2t, 2t + 1)
      if (g < H) {
        const uint32_t o = (c * H + g) * RS + jt * 32 + 4 * t;
        *reinterpret_cast<uint32_t*>(Qt + o) = ha;
        *reinterpret_cast<uint32_t*>(Qt + o + 16) = hb;
        *reinterpret_cast<uint32_t*>(Xlo + o) = la;
        *reinterpret_cast<uint32_t*>(Xlo + o + 16) = lb;
      }
    }
  };

  // =============================================================================================== forward
  for (int l = 0; l < P.M; ++l) {
    save_rows(P.G.T + l * Nd);
    if (dense) {                                                     // q = t W_q
      float acc[2][4] = {};
      const uint4* w = weights(l, 0, 0);
#pragma unroll
      for (int kt = 0; kt < D16; ++kt) {
        const uint4 b = __ldg(w + kt * D16 * 32);
        uint32_t hi[4], lo[4];
        ts_frag(kt, hi, lo);
        mma_pair(acc, hi, b);
        mma_pair(acc, lo, b);
      }
      put_rows(acc, 1.f, P.G.Q + l * Nd, true);
    }
    __syncthreads();
    if (dense) {                                                     // qt_h = q_h W_k[:, h]^T / tau
      float acc[2][4] = {};
      const uint4* w = weights(l, 1, 1);
#pragma unroll
      for (int kt = 0; kt < D16; ++kt) {
        const uint4 b = __ldg(w + kt * D16 * 32);
        uint32_t hi[4], lo[4];
        ldsm_x4(hi, smem_addr(Qhi + ldsm_row * RS + (kt * 2 + ldsm_kc) * 16));
        ldsm_x4(lo, smem_addr(Qlo + ldsm_row * RS + (kt * 2 + ldsm_kc) * 16));
        mma_pair(acc, hi, b);
        mma_pair(acc, lo, b);
        if ((kt + 1) % KH == 0) {                                    // last k-tile of head kt / KH
          const int h = kt / KH;
#pragma unroll
          for (int nt = 0; nt < 2; ++nt)
#pragma unroll
            for (int hf = 0; hf < 2; ++hf) {
              uint32_t hi2, lo2;
              split2(acc[nt][2 * hf] * P.inv_tau, acc[nt][2 * hf + 1] * P.inv_tau, hi2, lo2);
              const uint32_t o = ((g + hf * 8) * H + h) * RS + (wcol + nt * 8 + 2 * t) * 2;
              *reinterpret_cast<uint32_t*>(Qt + o) = hi2;
              if (NP == 2) *reinterpret_cast<uint32_t*>(Qt + plane + o) = lo2;
              acc[nt][2 * hf] = acc[nt][2 * hf + 1] = 0.f;
            }
        }
      }
    }
    __syncthreads();
#pragma unroll 1
    for (int sl = 0; sl < n_slots; ++sl) {                           // attention, one candidate of this warp after the other
      const int c = warp + kTW * sl, cand = c_base + c, nv = nv_s[c];
      if (cand >= c_end) continue;
      // the slot rows (qt of this layer): kept for the backward part
      for (int i = lane; i < H * 2 * D16; i += 32) {
        const int h = i / (2 * D16), q = i - h * (2 * D16);
        const size_t at = ((size_t)cand * P.slots + l * 2 * H + h) * d + q * 8;
        *reinterpret_cast<uint4*>(P.rows0 + at) = *reinterpret_cast<const uint4*>(Qt + (c * H + h) * RS + q * 16);
        if (NP == 2) *reinterpret_cast<uint4*>(P.rows1 + at) = *reinterpret_cast<const uint4*>(Qt + plane + (c * H + h) * RS + q * 16);
      }
      float x[D16][4];
#pragma unroll
      for (int jt = 0; jt < D16; ++jt) x[jt][0] = x[jt][1] = x[jt][2] = x[jt][3] = 0.f;
      float rm0 = -INFINITY, rm1 = -INFINITY, rs0 = 0.f, rs1 = 0.f;
      const uint32_t q0 = head_rows(Qt, c), q1 = head_rows(Qt + plane, c);
      const int nch = (nv + kTRows - 1) / kTRows;
      if (nch > 0) stage_chunk(cand, 0, nv, 0);
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
          dot_tile(sb, kt, a0, a1, q0, q1, e);
        }
        const int rows = nv - ch * kTRows;
        if (g >= rows) e[0] = e[1] = -INFINITY;
        if (g + 8 >= rows) e[2] = e[3] = -INFINITY;
        const float nm0 = fmaxf(rm0, group_max(fmaxf(e[0], e[2]))), nm1 = fmaxf(rm1, group_max(fmaxf(e[1], e[3])));
        const float sc0 = __expf(rm0 - nm0), sc1 = __expf(rm1 - nm1);
        rm0 = nm0;
        rm1 = nm1;
        float w0 = __expf(e[0] - nm0), w1 = __expf(e[1] - nm1), w2 = __expf(e[2] - nm0), w3 = __expf(e[3] - nm1);
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
      put_heads(c, x, i0, i1, P.G.Mh + l * NHd + (size_t)cand * H * d);
      if (g == 0) {
        float* st = P.stat + ((size_t)(l * P.N + cand) * H) * 2;
        if (2 * t < H) *reinterpret_cast<float2*>(st + 4 * t) = make_float2(rm0, i0);
        if (2 * t + 1 < H) *reinterpret_cast<float2*>(st + 4 * t + 2) = make_float2(rm1, i1);
      }
    }
    __syncthreads();
    if (dense && l + 1 < P.M) {                                      // t += m_h W_v[:, h]  (the last layer's t is not needed)
      float acc[2][4] = {};
      from_heads(acc, weights(l, 2, 0));
      add_rows(acc);
    }
    __syncthreads();
  }

  // =============================================================================================== backward
  for (int i = tid; i < kTRows * (d / 4); i += kTThreads) {          // dt of the last target
    const int r = i / (d / 4), c4 = (i - r * (d / 4)) * 4;
    *reinterpret_cast<float4*>(Ts + r * TS + c4) =
        c_base + r < c_end ? *reinterpret_cast<const float4*>(P.dz + (size_t)(c_base + r) * d + c4) : make_float4(0.f, 0.f, 0.f, 0.f);
  }
  __syncthreads();
  for (int l = P.M - 1; l >= 0; --l) {
    save_rows(P.G.dT + l * Nd);
    if (dense) {                                                     // dm_h = dt_h W_v[:, h]^T
      float acc[2][4] = {};
      const uint4* w = weights(l, 2, 1);
#pragma unroll
      for (int kt = 0; kt < D16; ++kt) {
        const uint4 b = __ldg(w + kt * D16 * 32);
        uint32_t hi[4], lo[4];
        ts_frag(kt, hi, lo);
        mma_pair(acc, hi, b);
        mma_pair(acc, lo, b);
        if ((kt + 1) % KH == 0) {
          const int h = kt / KH;
#pragma unroll
          for (int nt = 0; nt < 2; ++nt)
#pragma unroll
            for (int hf = 0; hf < 2; ++hf) {
              uint32_t hi2, lo2;
              split2(acc[nt][2 * hf], acc[nt][2 * hf + 1], hi2, lo2);
              const uint32_t o = ((g + hf * 8) * H + h) * RS + (wcol + nt * 8 + 2 * t) * 2;
              *reinterpret_cast<uint32_t*>(Dm + o) = hi2;
              if (NP == 2) *reinterpret_cast<uint32_t*>(Dm + plane + o) = lo2;
              acc[nt][2 * hf] = acc[nt][2 * hf + 1] = 0.f;
            }
        }
      }
    }
    __syncthreads();
#pragma unroll 1
    for (int sl = 0; sl < n_slots; ++sl) {
      const int c = warp + kTW * sl, cand = c_base + c, nv = nv_s[c];
      if (cand >= c_end) continue;
      const int nch = (nv + kTRows - 1) / kTRows;
      if (nch > 0) stage_chunk(cand, 0, nv, 0);
      // this layer's qt rows back from the slot rows; m . dm per head (lanes split the features)
      const float* mg = P.G.Mh + l * NHd + (size_t)cand * H * d;
      float dot0 = 0.f, dot1 = 0.f;                                  // heads 2t, 2t + 1
      for (int h = 0; h < H; ++h) {
        float v = 0.f;
        for (int q = lane; q < 2 * D16; q += 32) {
          const size_t at = ((size_t)cand * P.slots + l * 2 * H + h) * d + q * 8;
          const uint32_t o = (c * H + h) * RS + q * 16;
          *reinterpret_cast<uint4*>(Qt + o) = *reinterpret_cast<const uint4*>(P.rows0 + at);
          if (NP == 2) *reinterpret_cast<uint4*>(Qt + plane + o) = *reinterpret_cast<const uint4*>(P.rows1 + at);
          const float4 m0 = *reinterpret_cast<const float4*>(mg + h * d + q * 8), m1 = *reinterpret_cast<const float4*>(mg + h * d + q * 8 + 4);
#pragma unroll
          for (int pl = 0; pl < NP; ++pl) {
            const uint4 x = *reinterpret_cast<const uint4*>(Dm + pl * plane + o);
            v += m0.x * bf16_lo(x.x) + m0.y * bf16_hi(x.x) + m0.z * bf16_lo(x.y) + m0.w * bf16_hi(x.y) + m1.x * bf16_lo(x.z) +
                 m1.y * bf16_hi(x.z) + m1.z * bf16_lo(x.w) + m1.w * bf16_hi(x.w);
          }
        }
        v = group_sum(quad_sum(v));
        if (h == 2 * t) dot0 = v;
        if (h == 2 * t + 1) dot1 = v;
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
          dot_tile(sb, kt, a0, a1, q0, q1, e);
          dot_tile(sb, kt, a0, a1, d0, d1, da);
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
            float* o = P.ad + ((size_t)cand * Lp + j) * P.slots + l * 2 * H;
            if (2 * t < H) { o[2 * t] = de[2 * hf]; o[H + 2 * t] = a[2 * hf]; }
            if (2 * t + 1 < H) { o[2 * t + 1] = de[2 * hf + 1]; o[H + 2 * t + 1] = a[2 * hf + 1]; }
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
#pragma unroll
      for (int jt = 0; jt < D16; ++jt) {
        const float* mp = mg + jt * 16 + g;
        if (2 * t < H) { x[jt][0] -= rho0 * mp[2 * t * d]; x[jt][2] -= rho0 * mp[2 * t * d + 8]; }
        if (2 * t + 1 < H) { x[jt][1] -= rho1 * mp[(2 * t + 1) * d]; x[jt][3] -= rho1 * mp[(2 * t + 1) * d + 8]; }
      }
      for (int h = 0; h < H; ++h) {
        const float r0 = __shfl_sync(0xffffffffu, rho0, (h >> 1) & 3), r1 = __shfl_sync(0xffffffffu, rho1, (h >> 1) & 3);
        const float rho = (h & 1) ? r1 : r0;
        for (int q = lane; q < d / 2; q += 32) {
          const uint32_t o = (c * H + h) * RS + q * 4;
          const size_t at = ((size_t)cand * P.slots + l * 2 * H + H + h) * d + q * 2;
          float2 q2 = make_float2(0.f, 0.f), m2 = make_float2(0.f, 0.f);
#pragma unroll
          for (int pl = 0; pl < NP; ++pl) {
            const uint32_t qv = *reinterpret_cast<const uint32_t*>(Qt + pl * plane + o), mv = *reinterpret_cast<const uint32_t*>(Dm + pl * plane + o);
            q2.x += bf16_lo(qv); q2.y += bf16_hi(qv);
            m2.x += bf16_lo(mv); m2.y += bf16_hi(mv);
          }
          uint32_t hi, lo;
          split2(m2.x - rho * q2.x, m2.y - rho * q2.y, hi, lo);
          *reinterpret_cast<uint32_t*>(P.rows0 + at) = hi;
          if (NP == 2) *reinterpret_cast<uint32_t*>(P.rows1 + at) = lo;
        }
      }
      __syncwarp();
      put_heads(c, x, 1.f, 1.f, P.G.dQt + l * NHd + (size_t)cand * H * d);
    }
    __syncthreads();
    if (dense) {                                                     // dq_h = dqt_h W_k[:, h] / tau
      float acc[2][4] = {};
      from_heads(acc, weights(l, 1, 0));
      put_rows(acc, P.inv_tau, P.G.dQ + l * Nd, true);
    }
    __syncthreads();
    if (dense) {                                                     // dt += dq W_q^T
      float acc[2][4] = {};
      const uint4* w = weights(l, 0, 1);
#pragma unroll
      for (int kt = 0; kt < D16; ++kt) {
        const uint4 b = __ldg(w + kt * D16 * 32);
        uint32_t hi[4], lo[4];
        ldsm_x4(hi, smem_addr(Qhi + ldsm_row * RS + (kt * 2 + ldsm_kc) * 16));
        ldsm_x4(lo, smem_addr(Qlo + ldsm_row * RS + (kt * 2 + ldsm_kc) * 16));
        mma_pair(acc, hi, b);
        mma_pair(acc, lo, b);
      }
      add_rows(acc);
    }
    __syncthreads();
  }
  save_rows(P.G.dT0);

  // =============================================================================================== dH'
  // rows = segments, k = slots: A from the de / a array, B = the candidate's slot rows (staged once: slots <= 64)
  const int KS = (P.slots + 15) >> 4;
  const int mi = lane >> 3, lr = lane & 7;
  const uint32_t s_trans = ((mi & 1) * 8 + lr) * RS + (mi >> 1) * 16;
#pragma unroll 1
  for (int sl = 0; sl < n_slots; ++sl) {
    const int c = warp + kTW * sl, cand = c_base + c, nv = nv_s[c];
    if (cand >= c_end) continue;
    __syncwarp();
    for (int i = lane; i < 16 * KS * 2 * D16 * NP; i += 32) {        // planes of 16 KS rows
      const int pl = i / (16 * KS * 2 * D16), r = (i - pl * (16 * KS * 2 * D16)) / (2 * D16), q = i % (2 * D16);
      const bf16* src = (pl ? P.rows1 : P.rows0) + ((size_t)cand * P.slots + r) * d + q * 8;
      cp16(mine_a + (pl * 16 * KS + r) * RS + q * 16, r < P.slots ? (const void*)src : (const void*)P.S0, r < P.slots ? 16u : 0u);
    }
    cp_commit();
    cp_wait<0>();
    __syncwarp();
    for (int j0 = 0; j0 < nv; j0 += kTRows) {
      uint32_t ah[4][4], al[4][4];
#pragma unroll
      for (int ks = 0; ks < 4; ++ks)
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          const int j = j0 + g + (e & 1) * 8, s = ks * 16 + 2 * t + (e >> 1) * 8;
          float2 v = make_float2(0.f, 0.f);
          if (ks < KS && j < nv && s < P.slots) v = *reinterpret_cast<const float2*>(P.ad + ((size_t)cand * Lp + j) * P.slots + s);
          split2(v.x, v.y, ah[ks][e], al[ks][e]);
        }
#pragma unroll
      for (int jp = 0; jp < D16; ++jp) {
        float c0[4] = {0.f, 0.f, 0.f, 0.f}, c1[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
        for (int ks = 0; ks < 4; ++ks) {
          if (ks >= KS) break;
          uint32_t b[4];
          ldsm_x4_t(b, mine_a + ks * 16 * RS + s_trans + jp * 32);
          mma16816(c0, ah[ks][0], ah[ks][1], ah[ks][2], ah[ks][3], b[0], b[1]);
          mma16816(c1, ah[ks][0], ah[ks][1], ah[ks][2], ah[ks][3], b[2], b[3]);
          if (NP == 2) {
            mma16816(c0, al[ks][0], al[ks][1], al[ks][2], al[ks][3], b[0], b[1]);
            mma16816(c1, al[ks][0], al[ks][1], al[ks][2], al[ks][3], b[2], b[3]);
            ldsm_x4_t(b, mine_a + (16 * KS + ks * 16) * RS + s_trans + jp * 32);
            mma16816(c0, ah[ks][0], ah[ks][1], ah[ks][2], ah[ks][3], b[0], b[1]);
            mma16816(c1, ah[ks][0], ah[ks][1], ah[ks][2], ah[ks][3], b[2], b[3]);
          }
        }
#pragma unroll
        for (int hf = 0; hf < 2; ++hf) {
          const int j = j0 + g + hf * 8;
          if (j >= nv) continue;
          const size_t at = ((size_t)cand * Lp + j) * d + jp * 16 + 2 * t;
          if (NP == 1) {
            *reinterpret_cast<uint32_t*>(P.dS16 + at) = pack2(c0[2 * hf], c0[2 * hf + 1]);
            *reinterpret_cast<uint32_t*>(P.dS16 + at + 8) = pack2(c1[2 * hf], c1[2 * hf + 1]);
          } else {
            *reinterpret_cast<float2*>(P.dS32 + at) = make_float2(c0[2 * hf], c0[2 * hf + 1]);
            *reinterpret_cast<float2*>(P.dS32 + at + 8) = make_float2(c1[2 * hf], c1[2 * hf + 1]);
          }
        }
      }
    }
  }
}

// Weight gradients: C[m][n] += alpha sum_r A_h[r][m] B[r][n], h = the head of column n (A: [rows, heads, d], B: [rows, d]),
// for up to 3 M arrays in one launch.  TF32 MMAs (operands rounded to nearest), fp32 sums of the whole d x d matrix in a
// block's registers over its slice of the rows, one atomic add per element and block.
constexpr int kMaxSums = 24;
struct SumList {
  const float *A[kMaxSums], *B[kMaxSums];
  float* C[kMaxSums];
  float alpha[kMaxSums];
  int heads[kMaxSums];
};
__device__ __forceinline__ uint32_t to_tf32(float v) {
  uint32_t r;
  asm("cvt.rna.tf32.f32 %0, %1;" : "=r"(r) : "f"(v));
  return r;
}
template <int D16>
__global__ void __launch_bounds__(256, 2) weight_sums_kernel(const __grid_constant__ SumList L, int R, int rows_per_block, int KR,
                                                             int dvh) {
  constexpr int d = 16 * D16, kParts = 8 / D16 > 0 ? 8 / D16 : 1;    // warps that share a row tile split the rows
  extern __shared__ __align__(128) uint8_t smem[];
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, g = lane >> 2, t = lane & 3;
  const float *A = L.A[blockIdx.y], *B = L.B[blockIdx.y];
  const int heads = L.heads[blockIdx.y], lda = heads * d, pa = lda + 8, pb = d + 8;
  const int hw = heads == 1 ? d : dvh;                               // columns of a head
  float* buf0 = reinterpret_cast<float*>(smem);
  const int buf_words = KR * (pa + pb);
  const int mtile = warp % D16, part = warp / D16;
  const bool active = part < kParts;
  float acc[2 * D16][4];
#pragma unroll
  for (int j = 0; j < 2 * D16; ++j) acc[j][0] = acc[j][1] = acc[j][2] = acc[j][3] = 0.f;
  const int r_lo = blockIdx.x * rows_per_block, r_hi = min(R, r_lo + rows_per_block);
  auto stage = [&](int r0, int b) {
    float* As = buf0 + b * buf_words;
    float* Bs = As + KR * pa;
    const int ca = lda / 4, cb = d / 4;
    for (int i = tid; i < KR * ca; i += 256) {
      const int rr = i / ca, c = i - rr * ca;
      cp16(smem_addr(As + rr * pa + c * 4), A + (size_t)min(r0 + rr, r_hi - 1) * lda + c * 4, r0 + rr < r_hi ? 16u : 0u);
    }
    for (int i = tid; i < KR * cb; i += 256) {
      const int rr = i / cb, c = i - rr * cb;
      cp16(smem_addr(Bs + rr * pb + c * 4), B + (size_t)min(r0 + rr, r_hi - 1) * d + c * 4, r0 + rr < r_hi ? 16u : 0u);
    }
    cp_commit();
  };
  if (r_lo >= r_hi) return;
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
    const float* As = buf0 + b * buf_words;
    const float* Bs = As + KR * pa;
    if (active)
      for (int k = part * 8; k < KR; k += kParts * 8) {
        const float* ap = As + (k + t) * pa + mtile * 16 + g;
        const float* bp = Bs + (k + t) * pb + g;
        uint32_t a[4];
#pragma unroll
        for (int j = 0; j < 2 * D16; ++j) {
          if ((j * 8) % hw == 0) {                                   // first column tile of a head
            const float* q = ap + (j * 8) / hw * d;
            a[0] = to_tf32(q[0]); a[1] = to_tf32(q[8]);
            a[2] = to_tf32(q[4 * pa]); a[3] = to_tf32(q[4 * pa + 8]);
          }
          const uint32_t b0 = to_tf32(bp[j * 8]), b1 = to_tf32(bp[j * 8 + 4 * pb]);
          asm volatile(
              "mma.sync.aligned.m16n8k8.row.col.f32.tf32.tf32.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
              : "+f"(acc[j][0]), "+f"(acc[j][1]), "+f"(acc[j][2]), "+f"(acc[j][3])
              : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
        }
      }
    __syncthreads();
  }
  if (!active) return;
  float* C = L.C[blockIdx.y];
  const float alpha = L.alpha[blockIdx.y];
#pragma unroll
  for (int j = 0; j < 2 * D16; ++j)
#pragma unroll
    for (int e = 0; e < 4; ++e)
      atomicAdd(C + (size_t)(mtile * 16 + g + (e >> 1) * 8) * d + j * 8 + 2 * t + (e & 1), alpha * acc[j][e]);
}

struct TrainScratch {
  uint4* img;
  int *nseg, *order, *keys;
  float *stat, *ad;
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
  s.ad = (float*)take(N * p.Lp * slots * sizeof(float));
  s.rows0 = (bf16*)take(N * slots * p.d * sizeof(bf16));
  s.rows1 = np == 2 ? (bf16*)take(N * slots * p.d * sizeof(bf16)) : nullptr;
  s.total = off;
  return s;
}

int train_slot_steps(const Plan& p) { return (2 * p.M * p.H + 15) / 16; }
int train_buffers(const Plan& p, int np) { return std::max(np == 1 ? 2 : 1, train_slot_steps(p)); }

template <int D16, int NP>
int launch_train(TrainParams P, const Plan& p, const TrainScratch& s, const void* Wg, const int32_t* lengths,
                 const int32_t* cand_offsets, cudaStream_t st) {
  const int sms = device_sms();
  // 8 candidates per block (one per warp) while all blocks still run at once, two per SM
  P.cpb = (p.N + 7) / 8 <= 2 * sms ? 8 : kTRows;
  const int blocks = (p.N + P.cpb - 1) / P.cpb;
  P.order = blocks > 2 * sms ? s.order : nullptr;
  {
    const int total = p.M * 6 * D16 * D16 * 32;
    LaunchScope ls("gsta_train_prep", st);
    train_prep_kernel<<<std::min((total + 255) / 256, 4 * sms) + (P.order ? 1 : 0), 256, 0, st>>>(
        (const bf16*)Wg, s.img, p.d, p.M, lengths, cand_offsets, p.U, p.N, p.L, p.S, p.Lp, P.cpb, s.nseg,
        P.order ? s.order : nullptr, s.keys);
  }
  const size_t smem = TrainSmem<D16, NP>::bytes(p.H, P.nb);
  LASER_CUDA_OK(allow_smem(gsta_train_kernel<D16, NP>, smem));
  LaunchScope ls("gsta_train", st);
  gsta_train_kernel<D16, NP><<<blocks, kTThreads, smem, st>>>(P);
  LASER_CUDA_OK(cudaGetLastError());
  return LASER_OK;
}

template <int D16>
int launch_sums(const Plan& p, const GstaTrain& G, float* dWg, cudaStream_t st) {
  const size_t Nd = (size_t)p.N * p.d, dd = (size_t)p.d * p.d;
  const size_t row = 2 * ((size_t)p.H * p.d + p.d + 16) * sizeof(float);
  const int KR = row * 32 <= 110 * 1024 ? 32 : row * 16 <= 110 * 1024 ? 16 : 8;
  const size_t smem = row * KR;
  LASER_CUDA_OK(allow_smem(weight_sums_kernel<D16>, smem));
  for (int l0 = 0; l0 < p.M; l0 += kMaxSums / 3) {
    SumList L;
    int n = 0;
    for (int l = l0; l < p.M && n + 3 <= kMaxSums; ++l) {
      float *gWq = dWg + (size_t)(l * 3) * dd, *gWk = gWq + dd, *gWv = gWk + dd;
      auto add = [&](const float* A, int heads, const float* B, float* C, float alpha) {
        L.A[n] = A; L.B[n] = B; L.C[n] = C; L.alpha[n] = alpha; L.heads[n] = heads;
        ++n;
      };
      add(G.Mh + l * Nd * p.H, p.H, G.dT + l * Nd, gWv, 1.f);
      add(G.dQt + l * Nd * p.H, p.H, G.Q + l * Nd, gWk, p.inv_tau);
      add(G.T + l * Nd, 1, G.dQ + l * Nd, gWq, 1.f);
    }
    // about one wave of two blocks per SM over all sums
    const int want = std::max(1, 2 * device_sms() / n);
    const int per = std::max(KR, ((p.N + want - 1) / want + KR - 1) / KR * KR);
    LaunchScope ls("gsta_weight_sums", st);
    weight_sums_kernel<D16><<<dim3((p.N + per - 1) / per, n), 256, smem, st>>>(L, p.N, per, KR, p.dvh);
    LASER_CUDA_OK(cudaGetLastError());
  }
  return LASER_OK;
}

size_t train_smem(const Plan& p, int np) {
  const size_t RS = 2 * p.d + 16;
  return (size_t)kTRows * (p.d + 8) * 4 + 2 * np * (size_t)kTRows * p.H * RS + RS + kTRows * sizeof(int) + 48 +
         (size_t)kTW * train_buffers(p, np) * kTRows * RS * np;
}

}  // namespace

bool gsta_train_supported(const Plan& p, int np) {
  return p.dtype == LASER_BF16 && p.M > 0 && p.d % 16 == 0 && p.d >= 16 && p.d <= 128 && p.H <= 8 && p.dvh % 16 == 0 &&
         train_slot_steps(p) <= 4 && train_smem(p, np) <= 226 * 1024;
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

int gsta_train(const Plan& p, int np, const void* S0, const void* S1, const int32_t* lengths, const int32_t* cand_offsets,
               const void* cands, const void* Wg, const float* dz, const GstaTrain& G, void* dS, char* scratch, cudaStream_t st) {
  const TrainScratch s = carve_train(p, np, scratch);
  TrainParams P = {};
  P.N = p.N; P.U = p.U; P.L = p.L; P.S = p.S; P.Lp = p.Lp; P.H = p.H; P.M = p.M; P.slots = 2 * p.M * p.H; P.nb = train_buffers(p, np);
  P.inv_tau = p.inv_tau;
  P.S0 = (const bf16*)S0; P.S1 = (const bf16*)S1; P.cands = (const bf16*)cands; P.dz = dz;
  P.img = s.img; P.nseg = s.nseg; P.G = G; P.stat = s.stat; P.rows0 = s.rows0; P.rows1 = s.rows1; P.ad = s.ad;
  P.dS16 = (bf16*)dS; P.dS32 = (float*)dS;
#define LASER_TRAIN_CALL(D) (np == 1 ? launch_train<D, 1>(P, p, s, Wg, lengths, cand_offsets, st) : launch_train<D, 2>(P, p, s, Wg, lengths, cand_offsets, st))
  LASER_TRAIN_DISPATCH(LASER_TRAIN_CALL)
#undef LASER_TRAIN_CALL
}

int gsta_weight_sums(const Plan& p, const GstaTrain& G, float* dWg, cudaStream_t st) {
#define LASER_TRAIN_CALL(D) launch_sums<D>(p, G, dWg, st)
  LASER_TRAIN_DISPATCH(LASER_TRAIN_CALL)
#undef LASER_TRAIN_CALL
}

}  // namespace laser

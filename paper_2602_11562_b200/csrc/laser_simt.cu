// FP32-ALU kernels for STA and GSTA: fp32 arithmetic for either I/O dtype.  This is the path of the fp32
// configuration (tf32 tensor cores carry a 10-bit mantissa and cannot hold a 1e-4 bound) and a second,
// independent GPU implementation for any shape the tensor-core path does not take.
#include "laser_common.cuh"

namespace laser {
namespace {

constexpr int kProjRows = 32;     // rows per projection block
constexpr int kProjThreads = 128;
constexpr int kStaCands = 32;     // candidates per STA block
constexpr int kStaItems = 32;     // items per chunk
constexpr int kStaThreads = 128;
constexpr int kStaMaxJ = 64;      // columns per thread = d/4 <= 64  (d <= 256)
constexpr int kGstaThreads = 256;

// Eq. 4 / Eq. 8-9 in one launch, for widths that the tiled kernels (laser_simt_proj.cu) do not take: Q = t W_q / gamma for the
// candidates (the first q_tiles blocks of grid.x), K = H W_k and V = H W_v for every user's valid items (padded [U, L, .]
// outputs).  A block owns 32 rows x 32 columns, a thread eight rows of one column: the weights come straight from L2, a warp
// reading one 128-byte row piece per step, sixteen steps in flight; the rows sit in shared memory and are read as 128-bit
// broadcasts.  Block 0 clears the status word for the kernels behind this one.
struct ProjParams {
  const void *items, *cands, *Wq, *Wk, *Wv;
  float *Q, *K, *V;
  const int *lengths, *row_off;          // row_off: packed item layout (null: padded)
  int* status;
  int U, L, N, d, dqk, q_tiles, tiles_per_user;
  float inv_gamma;
};
template <typename T>
__global__ void __launch_bounds__(kProjThreads) proj_simt_kernel(ProjParams P) {
  extern __shared__ __align__(16) float xs[];   // [kProjRows][dp], dp = d rounded up to a multiple of 4
  chain_wait();                                 // (the kernels of this path are chained: launch latencies overlap)
  chain_release();
  if (blockIdx.x == 0 && blockIdx.y == 0 && threadIdx.x == 0) set_status(P.status, 0);
  const int d = P.d, dqk = P.dqk, tid = threadIdx.x, lane = tid & 31, part = tid >> 5;
  const bool is_q = (int)blockIdx.x < P.q_tiles;
  const int n_cols = is_q ? dqk : dqk + d, col = blockIdx.y * 32 + lane;
  if ((int)blockIdx.y * 32 >= n_cols) return;
  int rows;
  size_t in_row, out_row;
  if (is_q) {
    const int r0 = blockIdx.x * kProjRows;
    rows = min(kProjRows, P.N - r0);
    in_row = out_row = r0;
  } else {
    const int x = blockIdx.x - P.q_tiles, u = x / P.tiles_per_user, r0 = (x - u * P.tiles_per_user) * kProjRows;
    int len = P.lengths[u];                     // (invalid lengths and row offsets are reported by the STA kernel)
    if (len < 0 || len > P.L) len = 0;
    if (P.row_off && len > 0 && (P.row_off[u] < 0 || P.row_off[u] > P.row_off[P.U] - len)) len = 0;
    rows = min(kProjRows, len - r0);
    in_row = (P.row_off ? (size_t)P.row_off[u] : (size_t)u * P.L) + r0;
    out_row = (size_t)u * P.L + r0;
  }
  if (rows <= 0) return;
  const int dp = (d + 3) & ~3;
  const T* X = static_cast<const T*>(is_q ? P.cands : P.items) + in_row * d;
  for (int i = tid; i < kProjRows * dp; i += kProjThreads) {
    const int r = i / dp, c = i - r * dp;
    xs[i] = r < rows && c < d ? to_f32<T>(X[(size_t)r * d + c]) : 0.f;
  }
  const bool first = col < dqk;                 // W_q or W_k, else W_v
  const T* W = static_cast<const T*>(is_q ? P.Wq : first ? P.Wk : P.Wv) + (first ? col : col - dqk);
  const int ldw = first ? dqk : d;
  const bool live = col < n_cols;
  float acc[8] = {};
  __syncthreads();
  const float* xr = xs + part * 8 * dp;
  for (int k0 = 0; k0 < d; k0 += 16) {
    float w[16];
#pragma unroll
    for (int k = 0; k < 16; ++k) w[k] = live && k0 + k < d ? to_f32<T>(W[(size_t)(k0 + k) * ldw]) : 0.f;
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      if (k0 + 4 * q >= d) break;
#pragma unroll
      for (int r = 0; r < 8; ++r) {
        const float4 x = *reinterpret_cast<const float4*>(xr + r * dp + k0 + 4 * q);
        acc[r] = fmaf(x.x, w[4 * q], acc[r]);
        acc[r] = fmaf(x.y, w[4 * q + 1], acc[r]);
        acc[r] = fmaf(x.z, w[4 * q + 2], acc[r]);
        acc[r] = fmaf(x.w, w[4 * q + 3], acc[r]);
      }
    }
  }
  if (!live) return;
  float* Y = (is_q ? P.Q : first ? P.K : P.V) + (out_row + part * 8) * ldw + (first ? col : col - dqk);
  const float scale = is_q ? P.inv_gamma : 1.f;
#pragma unroll
  for (int r = 0; r < 8; ++r)
    if (part * 8 + r < rows) Y[(size_t)r * ldw] = acc[r] * scale;
}

__device__ __forceinline__ float sigmoid_accurate(float x) {
  // 1 / (1 + e^-x) with the accurate expf; e^-x overflowing to +inf gives exactly 0.
  return 1.f / (1.f + expf(-x));
}

__device__ __forceinline__ float warp_sum(float v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}
__device__ __forceinline__ float warp_max(float v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, o));
  return v;
}

// One block = (segment, 32-candidate tile, user).  Gates (Eq. 5 / Eq. 10) for a 32x32 (candidate, item) chunk go to
// shared memory, then every thread accumulates gate * value for its candidate and its interleaved columns (Eq. 12).
// kSoftmax selects the ablation variant: the weights of a segment's valid items are exp(score) normalised to sum to one
// per (candidate, head), computed online over the 32-item chunks (running maximum, running sum, rescaled accumulators).
template <typename T, bool kSoftmax>
__global__ void __launch_bounds__(kStaThreads)
sta_simt_kernel(const float* __restrict__ Q, const float* __restrict__ K, const float* __restrict__ V,
                const int* __restrict__ lengths, const int* __restrict__ cand_offsets, T* __restrict__ Hp,
                int L, int d, int dqk, int H, int S, int Lp, int N, const int* __restrict__ row_off,
                int* __restrict__ status) {
  extern __shared__ float sm[];
  chain_wait();
  chain_release();
  const int u = blockIdx.z, seg = blockIdx.x;
  const int off0 = cand_offsets[u], off1 = cand_offsets[u + 1];
  const int len = lengths[u];
  if (row_off && len > 0 && len <= L && (row_off[u] < 0 || row_off[u] > row_off[gridDim.z] - len)) {   // packed rows out of range
    if (threadIdx.x == 0) report_status(status, LASER_ERR_BAD_INPUT);
    return;
  }
  // (a user with more candidates than the grid was sized for, i.e. than max_cands_per_user, would leave rows unwritten)
  if (off0 < 0 || off1 < off0 || off1 > N || len < 0 || len > L || off1 - off0 > (int)gridDim.y * kStaCands) {
    if (threadIdx.x == 0) report_status(status, LASER_ERR_BAD_INPUT);
    return;
  }
  const int c0 = off0 + blockIdx.y * kStaCands;
  if (c0 >= off1) return;
  const int nc = min(kStaCands, off1 - c0);
  const int dqh = dqk / H, dvh = d / H;
  const int qld = dqk + 1;
  float* Qs = sm;                              // [32][dqk+1]
  float* Ks = Qs + kStaCands * qld;            // [32][dqk+1]
  float* Vs = Ks + kStaItems * qld;            // [32][d]
  float* G = Vs + kStaItems * d;               // [H][32][33]
  float* st_m = G + H * kStaCands * 33;        // softmax variant: running maximum   [H][32]
  float* st_z = st_m + H * kStaCands;          //                  running sum       [H][32]
  float* st_s = st_z + H * kStaCands;          //                  this chunk's rescale factor [H][32]

  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int c = tid >> 2, cg = tid & 3;        // accumulate phase: candidate, column group
  const int nj = (d + 3 - cg) / 4;             // columns cg, cg+4, ...
  float acc[kStaMaxJ];
  int goff[kStaMaxJ];
#pragma unroll
  for (int j = 0; j < kStaMaxJ; ++j) {
    acc[j] = 0.f;
    int col = cg + 4 * j;
    goff[j] = col < d ? ((col / dvh) * kStaCands + c) * 33 : 0;
  }

  for (int idx = tid; idx < kStaCands * dqk; idx += kStaThreads) {
    int r = idx / dqk, a = idx - r * dqk;
    Qs[r * qld + a] = r < nc ? Q[(size_t)(c0 + r) * dqk + a] : 0.f;
  }
  if (kSoftmax) {
    for (int idx = tid; idx < H * kStaCands; idx += kStaThreads) {
      st_m[idx] = -INFINITY;
      st_z[idx] = 0.f;
    }
  }

  const int n_begin = seg * S;
  const int n_end = min(min(n_begin + S, L), len);
  const float* Ku = K + (size_t)u * L * dqk;
  const float* Vu = V + (size_t)u * L * d;
  for (int nb = n_begin; nb < n_end; nb += kStaItems) {
    const int cnt = min(kStaItems, n_end - nb);
    __syncthreads();   // previous chunk fully consumed (and Qs visible on the first trip)
    for (int idx = tid; idx < kStaItems * dqk; idx += kStaThreads) {
      int r = idx / dqk, a = idx - r * dqk;
      Ks[r * qld + a] = r < cnt ? Ku[(size_t)(nb + r) * dqk + a] : 0.f;
    }
    for (int idx = tid; idx < kStaItems * d; idx += kStaThreads) {
      int r = idx / d, a = idx - r * d;
      Vs[idx] = r < cnt ? Vu[(size_t)(nb + r) * d + a] : 0.f;
    }
    __syncthreads();
    // gates: item = lane, candidate = warp + 4k
    for (int cc = warp; cc < kStaCands; cc += kStaThreads / 32) {
      for (int h = 0; h < H; ++h) {
        float dot = 0.f;
        for (int a = 0; a < dqh; ++a) dot = fmaf(Qs[cc * qld + h * dqh + a], Ks[lane * qld + h * dqh + a], dot);
        if (!kSoftmax) {
          G[(h * kStaCands + cc) * 33 + lane] = lane < cnt ? sigmoid_accurate(dot) : 0.f;
        } else {
          const float m_old = st_m[h * kStaCands + cc], z_old = st_z[h * kStaCands + cc];
          const float m_new = fmaxf(m_old, warp_max(lane < cnt ? dot : -INFINITY));   // finite: the chunk has an item
          const float pw = lane < cnt ? expf(dot - m_new) : 0.f;
          const float psum = warp_sum(pw);
          G[(h * kStaCands + cc) * 33 + lane] = pw;
          __syncwarp();
          if (lane == 0) {
            const float sc = expf(m_old - m_new);           // 0 on the first chunk (m_old = -inf)
            st_s[h * kStaCands + cc] = sc;
            st_z[h * kStaCands + cc] = z_old * sc + psum;
            st_m[h * kStaCands + cc] = m_new;
          }
        }
      }
    }
    __syncthreads();
    if (kSoftmax) {
#pragma unroll
      for (int j = 0; j < kStaMaxJ; ++j)
        if (j < nj) acc[j] *= st_s[goff[j] / 33];
    }
    // (the column loop is unrolled over the accumulator registers; its bound follows the width in use, so that a narrow
    // d does not pay for 64 predicated steps per item)
    if (nj <= 8) {
      for (int n = 0; n < cnt; ++n) {
#pragma unroll
        for (int j = 0; j < 8; ++j)
          if (j < nj) acc[j] = fmaf(G[goff[j] + n], Vs[n * d + cg + 4 * j], acc[j]);
      }
    } else if (nj <= 16) {
      for (int n = 0; n < cnt; ++n) {
#pragma unroll
        for (int j = 0; j < 16; ++j)
          if (j < nj) acc[j] = fmaf(G[goff[j] + n], Vs[n * d + cg + 4 * j], acc[j]);
      }
    } else if (nj <= 32) {
      for (int n = 0; n < cnt; ++n) {
#pragma unroll
        for (int j = 0; j < 32; ++j)
          if (j < nj) acc[j] = fmaf(G[goff[j] + n], Vs[n * d + cg + 4 * j], acc[j]);
      }
    } else {
      for (int n = 0; n < cnt; ++n) {
#pragma unroll
        for (int j = 0; j < kStaMaxJ; ++j)
          if (j < nj) acc[j] = fmaf(G[goff[j] + n], Vs[n * d + cg + 4 * j], acc[j]);
      }
    }
  }
  if (c < nc) {
    T* out = Hp + ((size_t)(c0 + c) * Lp + seg) * d;
#pragma unroll
    for (int j = 0; j < kStaMaxJ; ++j) {
      if (j < nj) {
        float v = acc[j];
        if (kSoftmax) {
          const float z = st_z[goff[j] / 33];
          v = z > 0.f ? v / z : 0.f;                        // a segment without valid items stays a zero row
        }
        out[cg + 4 * j] = from_f32<T>(v);
      }
    }
  }
}


// The same aggregation (sigmoid gates) for 16-wide query / key heads and 16-, 32- or 64-wide value heads: thread = (candidate,
// head, item part) with its query slice and its accumulators in registers; the segment's items pass through shared memory
// 32 at a time and every lane reads them as 128-bit broadcasts, so an item costs a thread 4 + DVH / 4 shared-memory reads
// for 16 + DVH multiply-adds (the kernel above reads two words per multiply-add).  `parts` warps share a (candidate tile,
// head): part k takes items k, k + parts, ... of a chunk and the parts' sums meet in shared memory; without them a small
// batch would run one warp per head through the whole segment (latency: 32 serial items at d_qh = 16).
template <typename TO, int DVH, int kMaxThreads>
__global__ void __launch_bounds__(kMaxThreads) sta_regs_kernel(const float* __restrict__ Qf, const float* __restrict__ Kf,
                                                       const float* __restrict__ Vf, const int* __restrict__ lengths,
                                                       const int* __restrict__ cand_offsets, TO* __restrict__ Hp, int L, int d,
                                                       int dqk, int H, int S, int Lp, int N, int parts,
                                                       const int* __restrict__ row_off, int* __restrict__ status) {
  constexpr int DQH = 16;
  extern __shared__ __align__(16) float sm[];
  float* Ks = sm;                        // [32][dqk]
  float* Vs = Ks + kStaItems * dqk;      // [32][d]
  float* red = Vs + kStaItems * d;       // [parts - 1][H][DVH][33]
  chain_wait();
  chain_release();
  const int u = blockIdx.z, seg = blockIdx.x;
  const int len = lengths[u], off0 = cand_offsets[u], off1 = cand_offsets[u + 1];
  if (len < 0 || len > L || off0 < 0 || off1 < off0 || off1 > N || off1 - off0 > (int)gridDim.y * kStaCands ||
      (row_off && len > 0 && (row_off[u] < 0 || row_off[u] > row_off[gridDim.z] - len))) {
    if (threadIdx.x == 0) report_status(status, LASER_ERR_BAD_INPUT);
    return;
  }
  const int c0 = off0 + blockIdx.y * kStaCands;
  if (c0 >= off1) return;
  const int tid = threadIdx.x, nt = blockDim.x, ci = tid & 31, warp = tid >> 5, h = warp % H, part = warp / H, c = c0 + ci;
  const bool live = c < off1;
  float q[DQH], acc[DVH];
#pragma unroll
  for (int a = 0; a < DQH / 4; ++a) {
    const float4 x = live ? reinterpret_cast<const float4*>(Qf + (size_t)c * dqk + h * DQH)[a] : make_float4(0.f, 0.f, 0.f, 0.f);
    q[4 * a] = x.x; q[4 * a + 1] = x.y; q[4 * a + 2] = x.z; q[4 * a + 3] = x.w;
  }
#pragma unroll
  for (int v = 0; v < DVH; ++v) acc[v] = 0.f;
  const int n_begin = seg * S, n_end = min(min(n_begin + S, L), len);
  for (int nb = n_begin; nb < n_end; nb += kStaItems) {
    const int cnt = min(kStaItems, n_end - nb);
    __syncthreads();
    const float4* Kg = reinterpret_cast<const float4*>(Kf + ((size_t)u * L + nb) * dqk);
    const float4* Vg = reinterpret_cast<const float4*>(Vf + ((size_t)u * L + nb) * d);
    for (int i = tid; i < cnt * dqk / 4; i += nt) reinterpret_cast<float4*>(Ks)[i] = Kg[i];
    for (int i = tid; i < cnt * d / 4; i += nt) reinterpret_cast<float4*>(Vs)[i] = Vg[i];
    __syncthreads();
    if (live) {
      for (int n = part; n < cnt; n += parts) {
        const float4* kp = reinterpret_cast<const float4*>(Ks + n * dqk + h * DQH);
        const float4* vp = reinterpret_cast<const float4*>(Vs + n * d + h * DVH);
        float e0 = 0.f, e1 = 0.f;
#pragma unroll
        for (int a = 0; a < DQH / 4; ++a) {
          const float4 x = kp[a];
          e0 = fmaf(q[4 * a], x.x, e0); e1 = fmaf(q[4 * a + 1], x.y, e1);
          e0 = fmaf(q[4 * a + 2], x.z, e0); e1 = fmaf(q[4 * a + 3], x.w, e1);
        }
        const float g = sigmoid_accurate(e0 + e1);
#pragma unroll
        for (int v = 0; v < DVH / 4; ++v) {
          const float4 x = vp[v];
          acc[4 * v] = fmaf(g, x.x, acc[4 * v]); acc[4 * v + 1] = fmaf(g, x.y, acc[4 * v + 1]);
          acc[4 * v + 2] = fmaf(g, x.z, acc[4 * v + 2]); acc[4 * v + 3] = fmaf(g, x.w, acc[4 * v + 3]);
        }
      }
    }
  }
  if (parts > 1) {
    if (part > 0) {
      float* mine = red + (size_t)((part - 1) * H + h) * DVH * 33 + ci;
#pragma unroll
      for (int v = 0; v < DVH; ++v) mine[v * 33] = acc[v];
    }
    __syncthreads();
    if (part > 0) return;
    for (int k = 0; k < parts - 1; ++k) {
      const float* other = red + (size_t)(k * H + h) * DVH * 33 + ci;
#pragma unroll
      for (int v = 0; v < DVH; ++v) acc[v] += other[v * 33];
    }
  }
  if (!live) return;
  TO* out = Hp + ((size_t)c * Lp + seg) * d + h * DVH;
#pragma unroll
  for (int v = 0; v < DVH; v += 4) {
    if constexpr (sizeof(TO) == 4) {
      *reinterpret_cast<float4*>(out + v) = make_float4(acc[v], acc[v + 1], acc[v + 2], acc[v + 3]);
    } else {
#pragma unroll
      for (int e = 0; e < 4; ++e) out[v + e] = from_f32<TO>(acc[v + e]);
    }
  }
}

template <typename TO, int DVH>
int launch_sta_regs(const Plan& p, const int32_t* lengths, const int32_t* cand_offsets, TO* Hp, char* ws, cudaStream_t st) {
  // Up to four warps per (tile, head), each with at least four items of a chunk, while there are few of them: with 8 warps per SM and
  // more two, with 32 one.  One | two | four, us: 5 users x 61 candidates (640 warps) 21 | 17 | 15; 20 x 60, segments of 60 (1120) 29
  // | 23 | 25; 32 x 3, d = 128 (2560) 18 | 15 | 22; 4 x 300 (2720) 23 | 21 | 25; 40 x 60 (5120) 31 | 33 | 39; 256 x 6, segments of
  // 20 (25600) 60 | 76 | 150.
  const int per_chunk = p.S < kStaItems ? p.S : kStaItems, ctiles = (p.maxC + kStaCands - 1) / kStaCands;
  const long long warps = (long long)p.Lp * ctiles * p.U * p.H, sms = device_sms();
  const int most = warps > 32 * sms ? 1 : warps > 8 * sms ? 2 : 4;
  int parts = 1;
  while (parts < most && 2 * parts * p.H <= 16 && per_chunk / (2 * parts) >= 4) parts *= 2;
  const size_t smem = ((size_t)kStaItems * (p.dqk + p.d) + (size_t)(parts - 1) * p.H * DVH * 33) * sizeof(float);
  if (smem > 200 * 1024) return LASER_ERR_UNSUPPORTED;
  auto kernel = p.H <= 16 ? sta_regs_kernel<TO, DVH, 512> : sta_regs_kernel<TO, DVH, 1024>;
  LASER_CUDA_OK(allow_smem(kernel, smem));
  LaunchScope ls("sta_simt", st);
  LASER_CUDA_OK(launch_chained(kernel, dim3(p.Lp, ctiles, p.U), dim3(32 * p.H * parts), smem, st,
                               (const float*)(ws + p.off_q), (const float*)(ws + p.off_k), (const float*)(ws + p.off_v),
                               (const int*)lengths, (const int*)cand_offsets, Hp, p.L, p.d, p.dqk, p.H, p.S, p.Lp, p.N, parts, (const int*)p.item_offsets,
                               reinterpret_cast<int*>(ws + p.off_status)));
  return LASER_OK;
}

// One block per CB candidates, for widths that gsta_f32_kernel (laser_simt_gsta.cu) does not take.  Eq. 7 in the reassociated form
// (exact in real arithmetic):
//   q = t W_q;  qt_h = W_k[:, head h] q_h  (so that (s_j W_k)_h . q_h = s_j . qt_h);  e_{j,h} = s_j . qt_h / tau;
//   a = softmax_j(e);  m_h = sum_j a_{j,h} s_j;  o[head h] = m_h W_v[:, head h];  t += o.
// Small batches are bound by the latency of these phases, so each of them spreads its outputs AND its sums over all 256
// threads: the two d x d products split the contraction index into `parts` partial sums, a score belongs to four lanes,
// each with a quarter of the features (segment vectors sit in rows padded by four words, so the eight rows a warp reads at a
// time do not share banks).  With more candidates than two blocks per SM, a block takes CB of them and reads every weight
// once for all.
template <typename T, int CB>
__global__ void __launch_bounds__(kGstaThreads)
gsta_simt_kernel(const T* __restrict__ Hp, const int* __restrict__ lengths, const int* __restrict__ cand_offsets,
                 const T* __restrict__ cands, const T* __restrict__ Wg, T* __restrict__ z, int U, int L, int d, int H,
                 int S, int Lp, int M, int N, int ds, float inv_tau, int* __restrict__ status) {
  extern __shared__ __align__(16) float sm[];
  __shared__ int s_nv[CB];
  chain_wait();
  chain_release();
  const int c_base = blockIdx.x * CB, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  constexpr int nwarps = kGstaThreads / 32;
  const int dh = d / H;                      // ds: row pitch of the segment vectors
  float* Hs = sm;                            // [CB][Lp][ds]
  float* t = Hs + (size_t)CB * Lp * ds;      // [CB][d]
  float* q = t + CB * d;                     // [CB][d]
  float* qt = q + CB * d;                    // [CB][H][ds]   qt, later m
  float* e = qt + CB * H * ds;               // [CB][H][Lp]
  float* red = e + CB * H * Lp;              // [parts][CB][d]
  if (tid < CB) {
    // user of this candidate: the largest u with cand_offsets[u] <= cand (skipping users without candidates)
    const int cand = c_base + tid;
    int nv = -1;                             // no candidate here, or one that nothing is written for
    if (cand < N) {
      int lo = 0, hi = U;                    // invariant: cand_offsets[lo] <= cand < cand_offsets[hi]
      if (cand_offsets[0] > cand || cand_offsets[U] <= cand) {
        report_status(status, LASER_ERR_BAD_INPUT);
      } else {
        while (hi - lo > 1) {
          const int mid = (lo + hi) >> 1;
          if (cand_offsets[mid] <= cand) lo = mid; else hi = mid;
        }
        const int len = lengths[lo];
        if (len < 0 || len > L) report_status(status, LASER_ERR_BAD_INPUT);
        else nv = min((len + S - 1) / S, Lp);
      }
    }
    s_nv[tid] = nv;
  }
  for (int i = tid; i < CB * d; i += kGstaThreads) t[i] = c_base + i / d < N ? to_f32<T>(cands[(size_t)c_base * d + i]) : 0.f;
  __syncthreads();
  int most = 0;
#pragma unroll
  for (int c = 0; c < CB; ++c) {
    const int n = s_nv[c] * d;
    most = max(most, s_nv[c]);
    const T* Hc = Hp + (size_t)(c_base + c) * Lp * d;
    for (int i = tid; i < n; i += kGstaThreads) Hs[(c * Lp + i / d) * ds + i % d] = to_f32<T>(Hc[i]);
  }
  const int parts = d >= kGstaThreads ? 1 : kGstaThreads / d;           // threads (j, part) of the d x d products
  const int kj = tid % d, kpart = tid / d, klen = (d + parts - 1) / parts;
  __syncthreads();

  for (int l = 0; l < M && most > 0; ++l) {
    const T* Wq = Wg + (size_t)(l * 3 + 0) * d * d;
    const T* Wk = Wg + (size_t)(l * 3 + 1) * d * d;
    const T* Wv = Wg + (size_t)(l * 3 + 2) * d * d;
    // y[c][j] (+)= sum_i x(c, j)[i] W[i][j]
    auto product = [&](const T* W, auto x_of, float* y, bool add) {
      for (int j0 = 0; j0 < d; j0 += kGstaThreads) {                    // (one pass unless d > 256)
        const int j = parts > 1 ? kj : j0 + tid;
        float a[CB];
#pragma unroll
        for (int c = 0; c < CB; ++c) a[c] = 0.f;
        if (j < d && kpart < parts) {
          const int i1 = min(d, (kpart + 1) * klen);
#pragma unroll 16
          for (int i = kpart * klen; i < i1; ++i) {
            const float w = to_f32<T>(W[(size_t)i * d + j]);
#pragma unroll
            for (int c = 0; c < CB; ++c) a[c] = fmaf(x_of(c, j)[i], w, a[c]);
          }
#pragma unroll
          for (int c = 0; c < CB; ++c) red[((parts > 1 ? kpart : 0) * CB + c) * d + j] = a[c];
        }
      }
      __syncthreads();
      for (int i = tid; i < CB * d; i += kGstaThreads) {
        float v = 0.f;
        for (int k = 0; k < parts; ++k) v += red[k * CB * d + i];
        if (add) y[i] += v; else y[i] = v;
      }
      __syncthreads();
    };
    product(Wq, [&](int c, int) { return (const float*)(t + c * d); }, q, false);
    // qt[c][h][i] = sum_{j in head h} Wk[i][j] q[c][j]
    for (int o = tid; o < H * d; o += kGstaThreads) {
      const int h = o % H, i = o / H;                                   // (a row's heads side by side: whole sectors)
      const T* w = Wk + (size_t)i * d + h * dh;
      float a[CB];
#pragma unroll
      for (int c = 0; c < CB; ++c) a[c] = 0.f;
#pragma unroll 16
      for (int j = 0; j < dh; ++j) {
        const float wv = to_f32<T>(w[j]);
#pragma unroll
        for (int c = 0; c < CB; ++c) a[c] = fmaf(wv, q[c * d + h * dh + j], a[c]);
      }
#pragma unroll
      for (int c = 0; c < CB; ++c) qt[(c * H + h) * ds + i] = a[c];
    }
    __syncthreads();
    // scores: four lanes per (candidate, head, segment)
    for (int c = 0; c < CB; ++c) {
      const int nv = s_nv[c], n = nv * H * 4;
      for (int o0 = warp * 32; o0 < n; o0 += kGstaThreads) {
        const int o = o0 + lane, p = o & 3, x = o >> 2, h = x / max(nv, 1), j = x - h * nv;
        float a = 0.f;
        if (o < n) {
          const float *s = Hs + (c * Lp + j) * ds, *w = qt + (c * H + h) * ds;
          if (d % 16 == 0) {
#pragma unroll 4
            for (int i = p * 4; i < d; i += 16) {
              const float4 sv = *reinterpret_cast<const float4*>(s + i), wv = *reinterpret_cast<const float4*>(w + i);
              a = fmaf(sv.x, wv.x, a); a = fmaf(sv.y, wv.y, a); a = fmaf(sv.z, wv.z, a); a = fmaf(sv.w, wv.w, a);
            }
          } else {
            for (int i = p; i < d; i += 4) a = fmaf(s[i], w[i], a);
          }
        }
        a += __shfl_xor_sync(0xffffffffu, a, 1);
        a += __shfl_xor_sync(0xffffffffu, a, 2);
        if (o < n && p == 0) e[(c * H + h) * Lp + j] = a * inv_tau;
      }
    }
    __syncthreads();
    // softmax over the non-empty segments: one warp per (candidate, head)
    for (int ch = warp; ch < CB * H; ch += nwarps) {
      const int nv = s_nv[ch / H];
      float* ec = e + ch * Lp;
      float mx = -INFINITY;
      for (int j = lane; j < nv; j += 32) mx = fmaxf(mx, ec[j]);
      mx = warp_max(mx);
      float s = 0.f;
      for (int j = lane; j < nv; j += 32) {
        const float w = expf(ec[j] - mx);
        ec[j] = w;
        s += w;
      }
      s = warp_sum(s);
      const float inv = 1.f / s;
      for (int j = lane; j < nv; j += 32) ec[j] *= inv;
    }
    __syncthreads();
    // m[c][h] = sum_j a_{j,h} s_j   (a candidate without segments: m = 0)
    for (int o = tid; o < CB * H * d; o += kGstaThreads) {
      const int ch = o / d, i = o - ch * d, c = ch / H, nv = s_nv[c];
      const float *ec = e + ch * Lp, *s = Hs + c * Lp * ds + i;
      float a = 0.f;
#pragma unroll 8
      for (int j = 0; j < nv; ++j) a = fmaf(ec[j], s[j * ds], a);
      qt[ch * ds + i] = a;
    }
    __syncthreads();
    product(Wv, [&](int c, int j) { return (const float*)(qt + (c * H + j / dh) * ds); }, t, true);
  }
  for (int i = tid; i < CB * d; i += kGstaThreads)
    if (s_nv[i / d] >= 0) z[(size_t)c_base * d + i] = from_f32<T>(t[i]);
}

// Eq. 8-9 in fp32: Q / gamma, K, V into the workspace (off_q, off_k, off_v).
template <typename T>
int simt_project_t(const Plan& p, const T* items, const int32_t* lengths, const T* cands, const T* Wq, const T* Wk,
                   const T* Wv, char* ws, cudaStream_t st, const ZeroList* zero = nullptr) {
  if (p.N == 0 || p.U == 0) return LASER_OK;
  int rc = simt_project_tiles(p, items, lengths, cands, Wq, Wk, Wv, ws, st, zero);
  if (rc != LASER_ERR_UNSUPPORTED) return rc;
  if (zero && (rc = zero_arrays(*zero, st)) != LASER_OK) return rc;
  ProjParams P;
  P.items = items; P.cands = cands; P.Wq = Wq; P.Wk = Wk; P.Wv = Wv;
  P.Q = reinterpret_cast<float*>(ws + p.off_q);
  P.K = reinterpret_cast<float*>(ws + p.off_k);
  P.V = reinterpret_cast<float*>(ws + p.off_v);
  P.lengths = lengths; P.row_off = p.item_offsets;
  P.status = reinterpret_cast<int*>(ws + p.off_status);
  P.U = p.U; P.L = p.L; P.N = p.N; P.d = p.d; P.dqk = p.dqk; P.inv_gamma = p.inv_gamma;
  P.q_tiles = (p.N + kProjRows - 1) / kProjRows;
  P.tiles_per_user = (p.L + kProjRows - 1) / kProjRows;
  const long long tiles = P.q_tiles + (long long)p.U * P.tiles_per_user;
  const int col_tiles = (p.dqk + p.d + 31) / 32;
  const size_t smem = (size_t)kProjRows * ((p.d + 3) & ~3) * sizeof(float);
  if (p.U > 65535 || tiles > 0x7fffffffLL || col_tiles > 65535 || smem > 200 * 1024) return LASER_ERR_UNSUPPORTED;
  LASER_CUDA_OK(allow_smem(proj_simt_kernel<T>, smem));
  LaunchScope ls("proj_simt", st);
  LASER_CUDA_OK(launch_chained(proj_simt_kernel<T>, dim3((unsigned)tiles, col_tiles), dim3(kProjThreads), smem, st, P));
  return LASER_OK;
}

// T: dtype of the inputs; TO: dtype of H' (T itself, or float when the caller keeps fp32 intermediates)
template <typename T, typename TO>
int simt_sta_t(const Plan& p, const T* items, const int32_t* lengths, const T* cands, const int32_t* cand_offsets,
               const T* Wq, const T* Wk, const T* Wv, TO* Hp, char* ws, cudaStream_t st, bool softmax) {
  int* status = reinterpret_cast<int*>(ws + p.off_status);
  float* Qf = reinterpret_cast<float*>(ws + p.off_q);
  float* Kf = reinterpret_cast<float*>(ws + p.off_k);
  float* Vf = reinterpret_cast<float*>(ws + p.off_v);
  if (p.N == 0 || p.U == 0) return LASER_OK;
  // users and candidate tiles index grid.y / grid.z of the launches below
  if (p.U > 65535 || (p.maxC + kStaCands - 1) / kStaCands > 65535) return LASER_ERR_UNSUPPORTED;
  const int rc = simt_project_t<T>(p, items, lengths, cands, Wq, Wk, Wv, ws, st);
  if (rc != LASER_OK) return rc;
  if (!softmax && p.dqh == 16 && p.H <= 32) {
    if (p.dvh == 16) return launch_sta_regs<TO, 16>(p, lengths, cand_offsets, Hp, ws, st);
    if (p.dvh == 32) return launch_sta_regs<TO, 32>(p, lengths, cand_offsets, Hp, ws, st);
    if (p.dvh == 64) return launch_sta_regs<TO, 64>(p, lengths, cand_offsets, Hp, ws, st);
  }
  {
    const size_t smem = ((size_t)(kStaCands + kStaItems) * (p.dqk + 1) + (size_t)kStaItems * p.d +
                         (size_t)p.H * kStaCands * (33 + 3)) * sizeof(float);
    if (smem > 200 * 1024) return LASER_ERR_UNSUPPORTED;
    dim3 grid(p.Lp, (p.maxC + kStaCands - 1) / kStaCands, p.U);
    if (softmax) {
      LASER_CUDA_OK(allow_smem(sta_simt_kernel<TO, true>, smem));
      LaunchScope ls("sta_simt_softmax", st);
      LASER_CUDA_OK(launch_chained(sta_simt_kernel<TO, true>, grid, dim3(kStaThreads), smem, st, (const float*)Qf,
                                   (const float*)Kf, (const float*)Vf, (const int*)lengths, (const int*)cand_offsets, Hp,
                                   p.L, p.d, p.dqk, p.H, p.S, p.Lp, p.N, p.item_offsets, status));
    } else {
      LASER_CUDA_OK(allow_smem(sta_simt_kernel<TO, false>, smem));
      LaunchScope ls("sta_simt", st);
      LASER_CUDA_OK(launch_chained(sta_simt_kernel<TO, false>, grid, dim3(kStaThreads), smem, st, (const float*)Qf,
                                   (const float*)Kf, (const float*)Vf, (const int*)lengths, (const int*)cand_offsets, Hp,
                                   p.L, p.d, p.dqk, p.H, p.S, p.Lp, p.N, p.item_offsets, status));
    }
  }
  LASER_CUDA_OK(cudaGetLastError());
  return LASER_OK;
}

// pad: words between the rows of the segment vectors (four, or none where only that fits).
size_t gsta_simt_smem(const Plan& p, int cb, int pad) {
  const int parts = p.d >= kGstaThreads ? 1 : kGstaThreads / p.d;
  return (size_t)cb * ((size_t)p.Lp * (p.d + pad) + 2 * p.d + (size_t)p.H * (p.d + pad) + (size_t)p.H * p.Lp + (size_t)parts * p.d) *
         sizeof(float);
}

template <typename T, int CB>
int launch_gsta_simt(const Plan& p, const T* Hp, const int32_t* lengths, const int32_t* cand_offsets, const T* cands,
                     const T* Wg, T* z, int pad, char* ws, cudaStream_t st) {
  const size_t smem = gsta_simt_smem(p, CB, pad);
  LASER_CUDA_OK(allow_smem(gsta_simt_kernel<T, CB>, smem));
  LaunchScope ls("gsta_simt", st);
  LASER_CUDA_OK(launch_chained(gsta_simt_kernel<T, CB>, dim3((p.N + CB - 1) / CB), dim3(kGstaThreads), smem, st, Hp,
                               (const int*)lengths, (const int*)cand_offsets, cands, Wg, z, p.U, p.L, p.d, p.H, p.S, p.Lp, p.M,
                               p.N, p.d + pad, p.inv_tau, reinterpret_cast<int*>(ws + p.off_status)));
  return LASER_OK;
}

// Candidates per block: four when that leaves at least two blocks per SM and two blocks' shared memory fit one.
template <typename T>
int simt_gsta_t(const Plan& p, const T* Hp, const int32_t* lengths, const int32_t* cand_offsets, const T* cands,
                const T* Wg, T* z, char* ws, cudaStream_t st) {
  if (p.N == 0) return LASER_OK;
  constexpr size_t most = 226 * 1024;
  if (gsta_simt_smem(p, 1, 0) > most) return LASER_ERR_UNSUPPORTED;
  const int pad = gsta_simt_smem(p, 1, 4) <= most ? 4 : 0;
  if ((p.N + 3) / 4 >= 2 * device_sms() && gsta_simt_smem(p, 4, 4) <= 110 * 1024)
    return launch_gsta_simt<T, 4>(p, Hp, lengths, cand_offsets, cands, Wg, z, pad, ws, st);
  return launch_gsta_simt<T, 1>(p, Hp, lengths, cand_offsets, cands, Wg, z, pad, ws, st);
}

}  // namespace

static int simt_sta_any(const Plan& p, const void* items, const int32_t* lengths, const void* cands,
                        const int32_t* cand_offsets, const void* Wq, const void* Wk, const void* Wv, void* Hprime,
                        char* ws, cudaStream_t st, bool softmax) {
  if (p.d > 4 * kStaMaxJ) return LASER_ERR_UNSUPPORTED;
  if (p.dtype == LASER_F32)
    return simt_sta_t<float, float>(p, (const float*)items, lengths, (const float*)cands, cand_offsets, (const float*)Wq,
                                    (const float*)Wk, (const float*)Wv, (float*)Hprime, ws, st, softmax);
  using B = __nv_bfloat16;
  return simt_sta_t<B, B>(p, (const B*)items, lengths, (const B*)cands, cand_offsets, (const B*)Wq, (const B*)Wk,
                          (const B*)Wv, (B*)Hprime, ws, st, softmax);
}

// STA with H' kept in fp32 whatever the I/O dtype (the backward pass recomputes the forward this way); the projections
// stay in the workspace as fp32 Q / gamma, K, V.
int simt_sta_f32(const Plan& p, const void* items, const int32_t* lengths, const void* cands, const int32_t* cand_offsets,
                 const void* Wq, const void* Wk, const void* Wv, float* Hprime32, char* ws, cudaStream_t st) {
  if (p.d > 4 * kStaMaxJ) return LASER_ERR_UNSUPPORTED;
  if (p.dtype == LASER_F32)
    return simt_sta_t<float, float>(p, (const float*)items, lengths, (const float*)cands, cand_offsets, (const float*)Wq,
                                    (const float*)Wk, (const float*)Wv, Hprime32, ws, st, false);
  using B = __nv_bfloat16;
  return simt_sta_t<B, float>(p, (const B*)items, lengths, (const B*)cands, cand_offsets, (const B*)Wq, (const B*)Wk,
                              (const B*)Wv, Hprime32, ws, st, false);
}

int simt_project(const Plan& p, const void* items, const int32_t* lengths, const void* cands, const void* Wq,
                 const void* Wk, const void* Wv, char* ws, cudaStream_t st, const ZeroList* zero) {
  if (p.dtype == LASER_F32)
    return simt_project_t<float>(p, (const float*)items, lengths, (const float*)cands, (const float*)Wq, (const float*)Wk,
                                 (const float*)Wv, ws, st, zero);
  using B = __nv_bfloat16;
  return simt_project_t<B>(p, (const B*)items, lengths, (const B*)cands, (const B*)Wq, (const B*)Wk, (const B*)Wv, ws, st, zero);
}

int simt_attend_f32(const Plan& p, const int32_t* lengths, const int32_t* cand_offsets, float* Hprime32, char* ws,
                    cudaStream_t st) {
  if (p.dqh != 16 || p.H > 32 || p.U > 65535 || (p.maxC + kStaCands - 1) / kStaCands > 65535) return LASER_ERR_UNSUPPORTED;
  if (p.dvh == 16) return launch_sta_regs<float, 16>(p, lengths, cand_offsets, Hprime32, ws, st);
  if (p.dvh == 32) return launch_sta_regs<float, 32>(p, lengths, cand_offsets, Hprime32, ws, st);
  if (p.dvh == 64) return launch_sta_regs<float, 64>(p, lengths, cand_offsets, Hprime32, ws, st);
  return LASER_ERR_UNSUPPORTED;
}

int simt_sta(const Plan& p, const void* items, const int32_t* lengths, const void* cands, const int32_t* cand_offsets,
             const void* Wq, const void* Wk, const void* Wv, void* Hprime, char* ws, cudaStream_t st) {
  return simt_sta_any(p, items, lengths, cands, cand_offsets, Wq, Wk, Wv, Hprime, ws, st, false);
}

int simt_sta_softmax(const Plan& p, const void* items, const int32_t* lengths, const void* cands,
                     const int32_t* cand_offsets, const void* Wq, const void* Wk, const void* Wv, void* Hprime, char* ws,
                     cudaStream_t st) {
  return simt_sta_any(p, items, lengths, cands, cand_offsets, Wq, Wk, Wv, Hprime, ws, st, true);
}

int simt_gsta(const Plan& p, const void* Hprime, const int32_t* lengths, const int32_t* cand_offsets, const void* cands,
              const void* Wg, void* z, char* ws, cudaStream_t st, bool follows_call) {
  const int rc = gsta_f32(p, Hprime, lengths, cand_offsets, cands, Wg, z, ws, st, follows_call);
  if (rc != LASER_ERR_UNSUPPORTED) return rc;
  if (p.dtype == LASER_F32)
    return simt_gsta_t<float>(p, (const float*)Hprime, lengths, cand_offsets, (const float*)cands, (const float*)Wg,
                              (float*)z, ws, st);
  using B = __nv_bfloat16;
  return simt_gsta_t<B>(p, (const B*)Hprime, lengths, cand_offsets, (const B*)cands, (const B*)Wg, (B*)z, ws, st);
}

}  // namespace laser

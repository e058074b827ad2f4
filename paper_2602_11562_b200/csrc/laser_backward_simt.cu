// FP32-ALU kernels of the backward pass that replace many small launches by few: the stacked attention of a candidate
// forward and backward in one kernel, and all dense products that do not depend on one another in one launch.
#include <algorithm>

#include "laser_backward.cuh"
#include "laser_common.cuh"
#include "laser_mma.cuh"

namespace laser {
namespace {

using bf16 = __nv_bfloat16;

constexpr int kTrainThreads = 256;

// Four consecutive weights (16- or 8-byte aligned).
__device__ __forceinline__ void load4(float (&v)[4], const float* p) {
  const float4 q = *reinterpret_cast<const float4*>(p);
  v[0] = q.x; v[1] = q.y; v[2] = q.z; v[3] = q.w;
}
__device__ __forceinline__ void load4(float (&v)[4], const bf16* p) {
  const uint2 q = *reinterpret_cast<const uint2*>(p);
  v[0] = __uint_as_float(q.x << 16); v[1] = __uint_as_float(q.x & 0xFFFF0000u);
  v[2] = __uint_as_float(q.y << 16); v[3] = __uint_as_float(q.y & 0xFFFF0000u);
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

// Stacked attention, recomputed forward and backward, one block per CB candidates with everything of a candidate in shared
// memory: segment vectors, and per layer t, q, qt_h = W_k[:, h] q_h / tau, a, m.  Layers last to first:
//   dm_h = dt_h W_v[:, h]^T,   de_{j,h} = a_{j,h} (s_j . dm_h - m_h . dm_h)       (sum_j a_j (s_j . dm) = m . dm)
//   dqt_h = sum_j de_{j,h} s_j,   ds_j += sum_h de_{j,h} qt_h + a_{j,h} dm_h
//   dq_h = dqt_h W_k[:, h] / tau,   dt += dq W_q^T
// What the weight gradients sum over the candidates (t, q, m, dt, dq, dqt per layer) goes to global memory.  The phases are
// latency-bound like those of the forward kernel and spread over all threads the same way.  Six launches and two copies per
// layer and direction before: 6 users x 23 candidates, d = 64, two layers, 0.40 ms; now one launch of 30 us.
template <typename T, int CB>
__global__ void __launch_bounds__(kTrainThreads)
gsta_train_simt_kernel(const float* __restrict__ Hp, const int* __restrict__ lengths, const int* __restrict__ cand_offsets,
                       const T* __restrict__ cands, const T* __restrict__ Wg, const float* __restrict__ dz, GstaTrain G,
                       float* __restrict__ dHp, int U, int L, int d, int H, int S, int Lp, int M, int N, int ds, float inv_tau) {
  extern __shared__ __align__(16) float sm[];
  __shared__ int s_nv[CB];
  const int c_base = blockIdx.x * CB, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  constexpr int nwarps = kTrainThreads / 32;
  const int dh = d / H, HL = H * Lp, Hd = H * ds;
  // (everything that is read in groups of four floats comes first: with d a multiple of 16 those offsets stay aligned)
  float* Hs = sm;                               // [CB][Lp][ds]
  float* t = Hs + (size_t)CB * Lp * ds;         // [M + 1][CB][d]
  float* q = t + (M + 1) * CB * d;              // [M][CB][d]
  float* qt = q + M * CB * d;                   // [M][CB][H][ds]
  float* m = qt + M * CB * Hd;                  // [M][CB][H][ds]
  float* dm = m + M * CB * Hd;                  // [CB][H][ds]
  float* dqt = dm + CB * Hd;                    // [CB][H][ds]
  float* dt = dqt + CB * Hd;                    // [CB][d]
  float* dq = dt + CB * d;                      // [CB][d]
  float* red = dq + CB * d;                     // [parts][CB][d]
  float* a = red + CB * d * (d >= kTrainThreads ? 1 : kTrainThreads / d);   // [M][CB][H][Lp]
  float* de = a + M * CB * HL;                  // [CB][H][Lp]
  float* mdm = de + CB * HL;                    // [CB][H]
  if (tid < CB) {
    const int cand = c_base + tid;
    int nv = 0;
    if (cand < N) {
      int lo = 0, hi = U - 1;                   // the last user whose first candidate is <= cand
      while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (cand_offsets[mid] <= cand) lo = mid; else hi = mid - 1;
      }
      const int len = lengths[lo];
      nv = len <= 0 || len > L ? 0 : min((len + S - 1) / S, Lp);
    }
    s_nv[tid] = nv;
  }
  const int live = min(CB, N - c_base) * d;     // elements of the candidates' rows
  for (int i = tid; i < CB * d; i += kTrainThreads) {
    t[i] = i < live ? to_f32<T>(cands[(size_t)c_base * d + i]) : 0.f;
    dt[i] = i < live ? dz[(size_t)c_base * d + i] : 0.f;
  }
  __syncthreads();
#pragma unroll
  for (int c = 0; c < CB; ++c) {
    const int n = s_nv[c] * d;
    const float* Hc = Hp + (size_t)(c_base + c) * Lp * d;
    for (int i = tid; i < n; i += kTrainThreads) Hs[(c * Lp + i / d) * ds + i % d] = Hc[i];
  }
  const int parts = d >= kTrainThreads ? 1 : kTrainThreads / d;        // threads (j, part) of the d x d products
  const int kj = tid % d, kpart = tid / d, klen = (d + parts - 1) / parts;
  const bool rows4 = dh % 4 == 0;               // whole groups of four in a row and in a head's slice of it
  __syncthreads();

  // y[c][j] = scale sum_i x(c, j)[i] W[i][j], or with the transposed matrix sum_i x(c, j)[i] W[j][i], plus add[c][j]
  auto product = [&](const T* W, bool trans, auto x_of, float scale, const float* add, float* y) {
    for (int j0 = 0; j0 < d; j0 += kTrainThreads) {
      const int j = parts > 1 ? kj : j0 + tid;
      if (j < d && kpart < parts) {
        float acc[CB];
#pragma unroll
        for (int c = 0; c < CB; ++c) acc[c] = 0.f;
        const int i0 = kpart * klen, i1 = min(d, i0 + klen);
        const T* w = trans ? W + (size_t)j * d : W + j;
        const int step = trans ? 1 : d;
        int i = i0;
        if (trans && rows4 && klen % 4 == 0) {
#pragma unroll 4
          for (; i < i1; i += 4) {
            float wv[4];
            load4(wv, w + i);
#pragma unroll
            for (int c = 0; c < CB; ++c)
#pragma unroll
              for (int e = 0; e < 4; ++e) acc[c] = fmaf(x_of(c, j)[i + e], wv[e], acc[c]);
          }
        }
#pragma unroll 16
        for (; i < i1; ++i) {
          const float wv = to_f32<T>(w[(size_t)i * step]);
#pragma unroll
          for (int c = 0; c < CB; ++c) acc[c] = fmaf(x_of(c, j)[i], wv, acc[c]);
        }
#pragma unroll
        for (int c = 0; c < CB; ++c) red[((parts > 1 ? kpart : 0) * CB + c) * d + j] = acc[c];
      }
    }
    __syncthreads();
    for (int i = tid; i < CB * d; i += kTrainThreads) {
      float v = 0.f;
      for (int k = 0; k < parts; ++k) v += red[k * CB * d + i];
      y[i] = fmaf(v, scale, add ? add[i] : 0.f);
    }
    __syncthreads();
  };
  // y[c][h][i] = scale sum_{j in head h} W[i][j] x[c][j]
  auto fold = [&](const T* W, const float* x, float scale, float* y) {
    for (int o = tid; o < H * d; o += kTrainThreads) {
      const int h = o % H, i = o / H;
      const T* w = W + (size_t)i * d + h * dh;
      float acc[CB];
#pragma unroll
      for (int c = 0; c < CB; ++c) acc[c] = 0.f;
      int j = 0;
      if (rows4) {
#pragma unroll 4
        for (; j < dh; j += 4) {
          float wv[4];
          load4(wv, w + j);
#pragma unroll
          for (int c = 0; c < CB; ++c)
#pragma unroll
            for (int e = 0; e < 4; ++e) acc[c] = fmaf(wv[e], x[c * d + h * dh + j + e], acc[c]);
        }
      }
      for (; j < dh; ++j) {
        const float wv = to_f32<T>(w[j]);
#pragma unroll
        for (int c = 0; c < CB; ++c) acc[c] = fmaf(wv, x[c * d + h * dh + j], acc[c]);
      }
#pragma unroll
      for (int c = 0; c < CB; ++c) y[(c * H + h) * ds + i] = acc[c] * scale;
    }
    __syncthreads();
  };
  // y[c][h][j] = s_j . x[c][h], four lanes per value
  auto scores = [&](const float* x, float* y) {
    for (int c = 0; c < CB; ++c) {
      const int nv = s_nv[c], n = nv * H * 4;
      for (int o0 = warp * 32; o0 < n; o0 += kTrainThreads) {
        const int o = o0 + lane, p = o & 3, r = o >> 2, h = r / nv, j = r - h * nv;
        float acc = 0.f;
        if (o < n) {
          const float *s = Hs + (c * Lp + j) * ds, *w = x + (c * H + h) * ds;
          if (d % 16 == 0) {
#pragma unroll 4
            for (int i = p * 4; i < d; i += 16) {
              const float4 sv = *reinterpret_cast<const float4*>(s + i), wv = *reinterpret_cast<const float4*>(w + i);
              acc = fmaf(sv.x, wv.x, acc); acc = fmaf(sv.y, wv.y, acc); acc = fmaf(sv.z, wv.z, acc); acc = fmaf(sv.w, wv.w, acc);
            }
          } else {
            for (int i = p; i < d; i += 4) acc = fmaf(s[i], w[i], acc);
          }
        }
        acc += __shfl_xor_sync(0xffffffffu, acc, 1);
        acc += __shfl_xor_sync(0xffffffffu, acc, 2);
        if (o < n && p == 0) y[(c * H + h) * Lp + j] = acc;
      }
    }
    __syncthreads();
  };
  // y[c][h] = sum_j w[c][h][j] s_j
  auto weighted = [&](const float* w, float* y) {
    for (int o = tid; o < CB * H * d; o += kTrainThreads) {
      const int ch = o / d, i = o - ch * d, c = ch / H, nv = s_nv[c];
      const float *wc = w + ch * Lp, *s = Hs + c * Lp * ds + i;
      float acc = 0.f;
#pragma unroll 8
      for (int j = 0; j < nv; ++j) acc = fmaf(wc[j], s[j * ds], acc);
      y[ch * ds + i] = acc;
    }
    __syncthreads();
  };
  auto keep = [&](float* dst, const float* src) {          // [CB][d] to the candidates' rows
    for (int i = tid; i < live; i += kTrainThreads) dst[(size_t)c_base * d + i] = src[i];
  };
  auto keep_heads = [&](float* dst, const float* src) {    // [CB][H][ds] to [N, H, d]
    for (int i = tid; i < live * H; i += kTrainThreads) dst[(size_t)c_base * H * d + i] = src[i / d * ds + i % d];
  };
  const size_t Nd = (size_t)N * d;

  for (int l = 0; l < M; ++l) {
    const T *Wq = Wg + (size_t)(l * 3) * d * d, *Wk = Wq + (size_t)d * d, *Wv = Wk + (size_t)d * d;
    float *tl = t + l * CB * d, *ql = q + l * CB * d, *qtl = qt + l * CB * Hd, *ml = m + l * CB * Hd, *al = a + l * CB * HL;
    product(Wq, false, [&](int c, int) { return (const float*)(tl + c * d); }, 1.f, nullptr, ql);
    fold(Wk, ql, inv_tau, qtl);
    scores(qtl, al);
    for (int ch = warp; ch < CB * H; ch += nwarps) {       // softmax over the non-empty segments
      const int nv = s_nv[ch / H];
      float* e = al + ch * Lp;
      float mx = -INFINITY, sum = 0.f;
      for (int j = lane; j < nv; j += 32) mx = fmaxf(mx, e[j]);
      mx = warp_max(mx);
      for (int j = lane; j < nv; j += 32) {
        e[j] = expf(e[j] - mx);
        sum += e[j];
      }
      sum = warp_sum(sum);
      const float inv = 1.f / sum;
      for (int j = lane; j < nv; j += 32) e[j] *= inv;
    }
    __syncthreads();
    weighted(al, ml);
    product(Wv, false, [&](int c, int j) { return (const float*)(ml + (c * H + j / dh) * ds); }, 1.f, tl, tl + CB * d);
    keep(G.T + l * Nd, tl);
    keep(G.Q + l * Nd, ql);
    keep_heads(G.Mh + l * Nd * H, ml);
  }
  for (int l = M - 1; l >= 0; --l) {
    const T *Wq = Wg + (size_t)(l * 3) * d * d, *Wk = Wq + (size_t)d * d, *Wv = Wk + (size_t)d * d;
    float *qtl = qt + l * CB * Hd, *ml = m + l * CB * Hd, *al = a + l * CB * HL;
    keep(G.dT + l * Nd, dt);
    fold(Wv, dt, 1.f, dm);
    for (int ch = warp; ch < CB * H; ch += nwarps) {
      float v = 0.f;
      for (int i = lane; i < d; i += 32) v = fmaf(ml[ch * ds + i], dm[ch * ds + i], v);
      v = warp_sum(v);
      if (lane == 0) mdm[ch] = v;
    }
    scores(dm, de);
    for (int i = tid; i < CB * HL; i += kTrainThreads) {
      const int ch = i / Lp, j = i - ch * Lp;
      de[i] = j < s_nv[ch / H] ? al[i] * (de[i] - mdm[ch]) : 0.f;
    }
    __syncthreads();
    weighted(de, dqt);
    // ds: every entry belongs to one thread in every layer; the layer processed first writes all rows
    for (int c = 0; c < CB && c_base + c < N; ++c) {
      const int nv = s_nv[c];
      float* out = dHp + (size_t)(c_base + c) * Lp * d;
      for (int o = tid; o < Lp * d; o += kTrainThreads) {
        const int j = o / d, i = o - j * d;
        if (j >= nv) {
          if (l == M - 1) out[o] = 0.f;
          continue;
        }
        float v = l == M - 1 ? 0.f : out[o];
        for (int h = 0; h < H; ++h) {
          const int ch = c * H + h;
          v = fmaf(de[ch * Lp + j], qtl[ch * ds + i], fmaf(al[ch * Lp + j], dm[ch * ds + i], v));
        }
        out[o] = v;
      }
    }
    product(Wk, false, [&](int c, int j) { return (const float*)(dqt + (c * H + j / dh) * ds); }, inv_tau, nullptr, dq);
    product(Wq, true, [&](int c, int) { return (const float*)(dq + c * d); }, 1.f, dt, dt);
    keep(G.dQ + l * Nd, dq);
    keep_heads(G.dQt + l * Nd * H, dqt);
    __syncthreads();                                       // (the next layer writes dqt and dm)
  }
  keep(G.dT0, dt);
}

size_t train_simt_smem(const Plan& p, int cb, int pad) {
  const int parts = p.d >= kTrainThreads ? 1 : kTrainThreads / p.d;
  const size_t ds = p.d + pad, Hd = p.H * ds, HL = (size_t)p.H * p.Lp, M = p.M;
  return ((size_t)cb * (p.Lp * ds + (M + 1) * p.d + M * (p.d + 2 * Hd + HL) + 2 * Hd + HL + 2 * p.d + (size_t)parts * p.d) +
          (size_t)cb * p.H) * sizeof(float);
}
constexpr size_t kTrainSmemMax = 226 * 1024;

template <typename T, int CB>
int launch_train(const Plan& p, const float* Hp, const int32_t* lengths, const int32_t* cand_offsets, const T* cands,
                 const T* Wg, const float* dz, const GstaTrain& G, float* dHp, int pad, cudaStream_t st) {
  const size_t smem = train_simt_smem(p, CB, pad);
  LASER_CUDA_OK(allow_smem(gsta_train_simt_kernel<T, CB>, smem));
  LaunchScope ls("gsta_train_simt", st);
  gsta_train_simt_kernel<T, CB><<<(p.N + CB - 1) / CB, kTrainThreads, smem, st>>>(
      Hp, lengths, cand_offsets, cands, Wg, dz, G, dHp, p.U, p.L, p.d, p.H, p.S, p.Lp, p.M, p.N, p.d + pad, p.inv_tau);
  LASER_CUDA_OK(cudaGetLastError());
  return LASER_OK;
}

template <typename T>
int train_t(const Plan& p, const float* Hp, const int32_t* lengths, const int32_t* cand_offsets, const T* cands, const T* Wg,
            const float* dz, const GstaTrain& G, float* dHp, cudaStream_t st) {
  // four candidates per block (weights read once for all four) when that leaves two blocks per SM
  if ((p.N + 3) / 4 >= 2 * device_sms() && train_simt_smem(p, 4, 4) <= 110 * 1024)
    return launch_train<T, 4>(p, Hp, lengths, cand_offsets, cands, Wg, dz, G, dHp, 4, st);
  const int pad = train_simt_smem(p, 1, 4) <= kTrainSmemMax ? 4 : 0;
  return launch_train<T, 1>(p, Hp, lengths, cand_offsets, cands, Wg, dz, G, dHp, pad, st);
}

// ------------------------------------------------------------------------------------------------ dense products
// Every product of a list in one launch: C = D + alpha (A B + A2 B2), or C += by atomic adds of slices of the contraction.  A block
// finds its product, tile, batch entry and slice from its index.  Tiles of 64 rows x 64, 32 or 16 columns, as many as the product has:
// a thread has 4 x 4 of them, and in the narrow ones (a head's 16 or 32 columns) two or four groups of threads take every second or
// fourth step of the contraction (in 64-wide tiles three quarters of the weight sums of 16-wide heads were multiplications by zero).
// Contraction steps come 32 at a time, fetched a round ahead into registers, four consecutive elements at a time where the layout
// allows.  27 users x 49 candidates of 315 items, d = 96, six heads, two layers 62 -> 56 us, 75 x 23 of 169, d = 32
// 19 -> 15, the two lists of 63 users with one candidate each, d = 96, six heads 11 + 9 -> 7 + 7.  Bound by issue (64 %) and shared-memory
// reads (67 %).
constexpr int kTile = 64, kStep = 32, kPitch = kTile + 4;
struct ProductList {
  Product p[kMaxProducts];
  int first[kMaxProducts + 1];             // first block of each product
  int n;
};
__host__ __device__ inline int tile_cols(int N) { return N <= 16 ? 16 : (N + 31) % kTile < 32 ? kTile : 32; }

template <typename TX>
__device__ __forceinline__ void fetch4(float (&v)[4], const TX* X, int ld, bool k_major, int r, int R, int k, int K, bool vec) {
  // k_major: X[k ld + r], four rows; else X[r ld + k], four k
  const TX* src = k_major ? X + (size_t)k * ld + r : X + (size_t)r * ld + k;
  if (vec && r + (k_major ? 4 : 1) <= R && k + (k_major ? 1 : 4) <= K) {
    if constexpr (sizeof(TX) == 4) {
      const float4 q = *reinterpret_cast<const float4*>(src);
      v[0] = q.x; v[1] = q.y; v[2] = q.z; v[3] = q.w;
    } else {
      const uint2 q = *reinterpret_cast<const uint2*>(src);
      v[0] = __uint_as_float(q.x << 16); v[1] = __uint_as_float(q.x & 0xFFFF0000u);
      v[2] = __uint_as_float(q.y << 16); v[3] = __uint_as_float(q.y & 0xFFFF0000u);
    }
    return;
  }
#pragma unroll
  for (int e = 0; e < 4; ++e) {
    const bool in = k_major ? r + e < R && k < K : r < R && k + e < K;
    v[e] = in ? to_f32<TX>(src[e]) : 0.f;
  }
}
// A thread's share of a round: four elements of each half.  k_major: thread = (k, four rows), else (row, four k).
struct Fetch {
  const void* X;
  int ld, r0, R;
  bool is16, k_major, vec;
  __device__ __forceinline__ Fetch(const void* x, bool b16, int l, bool km, int r, int rows)
      : X(x), ld(l), r0(r), R(rows), is16(b16), k_major(km), vec(l % 4 == 0 && (reinterpret_cast<uintptr_t>(x) & (b16 ? 7 : 15)) == 0) {}
  __device__ __forceinline__ void load(float (&v)[2][4], int k0, int K, int tid) const {
#pragma unroll
    for (int half = 0; half < 2; ++half) {
      const int r = r0 + (k_major ? (tid & 15) * 4 : tid >> 2), k = k0 + (k_major ? (tid >> 4) + 16 * half : ((tid & 3) + 4 * half) * 4);
      if (is16) fetch4<bf16>(v[half], static_cast<const bf16*>(X), ld, k_major, r, R, k, K, vec);
      else fetch4<float>(v[half], static_cast<const float*>(X), ld, k_major, r, R, k, K, vec);
    }
  }
  // shared layout [k][64 + 4]
  __device__ __forceinline__ void put(float* sm, const float (&v)[2][4], int tid) const {
#pragma unroll
    for (int half = 0; half < 2; ++half) {
      if (k_major) {
        *reinterpret_cast<float4*>(sm + ((tid >> 4) + 16 * half) * kPitch + (tid & 15) * 4) = make_float4(v[half][0], v[half][1], v[half][2], v[half][3]);
      } else {
#pragma unroll
        for (int e = 0; e < 4; ++e) sm[(((tid & 3) + 4 * half) * 4 + e) * kPitch + (tid >> 2)] = v[half][e];
      }
    }
  }
};

template <int COLS>
__device__ __forceinline__ void multiply(float (&acc)[4][4], const float* As, const float* Bs, int tid) {
  constexpr int kGroups = kTile / COLS, kTx = COLS / 4;
  const int grp = tid / (16 * kTx), tx = tid % kTx, ty = tid / kTx % 16;
#pragma unroll
  for (int kk = 0; kk < kStep; kk += kGroups) {
    const float4 a4 = *reinterpret_cast<const float4*>(As + (kk + grp) * kPitch + ty * 4);
    const float4 b4 = *reinterpret_cast<const float4*>(Bs + (kk + grp) * kPitch + tx * 4);
    const float a[4] = {a4.x, a4.y, a4.z, a4.w}, b[4] = {b4.x, b4.y, b4.z, b4.w};
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
      for (int j = 0; j < 4; ++j) acc[i][j] = fmaf(a[i], b[j], acc[i][j]);
  }
}

__global__ void __launch_bounds__(256) products_kernel(const __grid_constant__ ProductList L) {
  __shared__ __align__(16) float sm[4 * kStep * kPitch];   // A and B, two buffers each; the groups' sums at the end
  chain_wait();
  const int tid = threadIdx.x;
  int which = 0;
  while (which + 1 < L.n && (int)blockIdx.x >= L.first[which + 1]) ++which;
  const Product& P = L.p[which];
  int b = blockIdx.x - L.first[which];
  const int cols = tile_cols(P.N), tiles_n = (P.N + cols - 1) / cols, tiles = (P.M + kTile - 1) / kTile * tiles_n;
  const int slice = b / (tiles * P.batch);
  b -= slice * tiles * P.batch;
  const int bat = b / tiles, tile = b - bat * tiles;
  const int m0 = tile / tiles_n * kTile, n0 = tile % tiles_n * cols;
  float acc[4][4] = {};
  for (int seg = 0; seg < (P.A2 ? 2 : 1); ++seg) {
    const Fetch A(seg ? P.A2 : (const char*)P.A + (size_t)bat * P.sa * (P.a16 ? 2 : 4), P.a16, seg ? P.lda2 : P.lda, P.ta, m0, P.M);
    const Fetch B(seg ? P.B2 : (const char*)P.B + (size_t)bat * P.sb * (P.b16 ? 2 : 4), P.b16, seg ? P.ldb2 : P.ldb, !P.tb, n0, P.N);
    const int K = seg ? P.K2 : P.K, k_lo = slice * P.k_per, k_hi = seg ? K : min(K, k_lo + P.k_per);
    float va[2][4], vb[2][4];
    int buf = 0;
    A.load(va, k_lo, k_hi, tid);
    B.load(vb, k_lo, k_hi, tid);
    for (int k0 = k_lo; k0 < k_hi; k0 += kStep, buf ^= 1) {
      float *As = sm + buf * kStep * kPitch, *Bs = As + 2 * kStep * kPitch;
      A.put(As, va, tid);
      B.put(Bs, vb, tid);
      __syncthreads();
      if (k0 + kStep < k_hi) {
        A.load(va, k0 + kStep, k_hi, tid);
        B.load(vb, k0 + kStep, k_hi, tid);
      }
      if (cols == kTile) multiply<64>(acc, As, Bs, tid);
      else if (cols == 32) multiply<32>(acc, As, Bs, tid);
      else multiply<16>(acc, As, Bs, tid);
    }
    __syncthreads();                       // (two buffers: one barrier per round, and one before the other pair of operands)
  }
  const int tx = tid % (cols / 4), ty = tid / (cols / 4) % 16;
  if (cols < kTile) {                      // the groups' sums, to the first group
    const int groups = kTile / cols, per = 256 / groups, grp = tid / per;
    float4* mine = reinterpret_cast<float4*>(sm) + (size_t)grp * per * 4 + tid % per;
#pragma unroll
    for (int i = 0; i < 4; ++i) mine[i * per] = make_float4(acc[i][0], acc[i][1], acc[i][2], acc[i][3]);
    __syncthreads();
    if (grp > 0) return;
    for (int k = 1; k < groups; ++k)
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const float4 v = mine[(k * 4 + i) * per];
        acc[i][0] += v.x; acc[i][1] += v.y; acc[i][2] += v.z; acc[i][3] += v.w;
      }
  }
  float* C = P.C + (size_t)bat * P.sc;
  const bool whole = n0 + tx * 4 + 4 <= P.N && P.ldc % 4 == 0 && (reinterpret_cast<uintptr_t>(C) & 15) == 0 &&
                     (reinterpret_cast<uintptr_t>(P.D) & 15) == 0;      // four columns with one access
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const int m = m0 + ty * 4 + i;
    if (m >= P.M) continue;
    if (whole) {
      const size_t at = (size_t)m * P.ldc + n0 + tx * 4;
      float4 v = make_float4(P.alpha * acc[i][0], P.alpha * acc[i][1], P.alpha * acc[i][2], P.alpha * acc[i][3]);
      if (P.atomic) {
        mma::red_add4(C + at, v.x, v.y, v.z, v.w);
      } else {
        if (P.D) {
          const float4 w = *reinterpret_cast<const float4*>(P.D + at);
          v.x += w.x; v.y += w.y; v.z += w.z; v.w += w.w;
        }
        *reinterpret_cast<float4*>(C + at) = v;
      }
      continue;
    }
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const int n = n0 + tx * 4 + j;
      if (n >= P.N) continue;
      const float v = P.alpha * acc[i][j];
      float* c = C + (size_t)m * P.ldc + n;
      if (P.atomic) atomicAdd(c, v);
      else *c = P.D ? P.D[(size_t)m * P.ldc + n] + v : v;
    }
  }
}

}  // namespace

bool gsta_train_simt_supported(const Plan& p) { return p.M > 0 && train_simt_smem(p, 1, 0) <= kTrainSmemMax; }

int gsta_train_simt(const Plan& p, const float* Hp, const int32_t* lengths, const int32_t* cand_offsets, const void* cands,
                    const void* Wg, const float* dz, const GstaTrain& G, float* dHp, cudaStream_t st) {
  const int rc = gsta_train_f32(p, Hp, lengths, cand_offsets, cands, Wg, dz, &G, nullptr, dHp, nullptr, st);
  if (rc != LASER_ERR_UNSUPPORTED) return rc;
  if (p.dtype == LASER_F32)
    return train_t<float>(p, Hp, lengths, cand_offsets, (const float*)cands, (const float*)Wg, dz, G, dHp, st);
  return train_t<bf16>(p, Hp, lengths, cand_offsets, (const bf16*)cands, (const bf16*)Wg, dz, G, dHp, st);
}

int run_products(Product* list, int n, cudaStream_t st) {
  for (int i0 = 0; i0 < n; i0 += kMaxProducts) {
    ProductList L;
    L.n = std::min(kMaxProducts, n - i0);
    long long blocks = 0;
    for (int i = 0; i < L.n; ++i) {
      Product& P = list[i0 + i];
      const int cols = tile_cols(P.N);
      const long long tiles = (long long)((P.M + kTile - 1) / kTile) * ((P.N + cols - 1) / cols) * P.batch;
      int slices = 1;
      P.k_per = std::max(P.K, 1);
      if (P.atomic) {                      // slices of at least 64 rows, longer when a product still gets about two blocks per SM
        P.k_per = (int)std::min<long long>(std::max<long long>(64, ((long long)P.K * tiles / (2 * device_sms()) + kStep - 1) / kStep * kStep), 1 << 24);
        slices = (P.K + P.k_per - 1) / P.k_per;
      }
      L.p[i] = P;
      L.first[i] = (int)blocks;
      blocks += tiles * slices;
      if (blocks > 0x7fffffffLL) return LASER_ERR_UNSUPPORTED;
    }
    L.first[L.n] = (int)blocks;
    if (blocks == 0) continue;
    LaunchScope ls("bwd_products", st);
    LASER_CUDA_OK(launch_chained(products_kernel, dim3((unsigned)blocks), dim3(256), 0, st, L));
  }
  return LASER_OK;
}

}  // namespace laser

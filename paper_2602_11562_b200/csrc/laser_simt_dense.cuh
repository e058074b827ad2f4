// Building blocks of the FP32-ALU kernels of the stacked attention (forward and backward): a block of 256 threads holds CB
// candidates in shared memory and multiplies them by d x d weights that it reads once for all of them.  D (width) and H
// (heads) are compile-time constants; head widths are powers of two, so that a head's slice of a weight row belongs to an
// aligned group of lanes.
//
// What bounds these products at the sizes they run at is the latency of the weight reads: every thread has all its reads of a
// product in flight at once (up to sixteen of four weights), and load() can be called a phase ahead of run().
#pragma once

#include "laser_common.cuh"

namespace laser {
namespace dense {

constexpr int kThreads = 256, kWarps = kThreads / 32;

// Four consecutive values as they lie in memory.
template <typename T> struct Raw4;
template <> struct Raw4<float> { using type = float4; };
template <> struct Raw4<__nv_bfloat16> { using type = uint2; };
__device__ __forceinline__ void unpack4(float (&v)[4], float4 q) { v[0] = q.x; v[1] = q.y; v[2] = q.z; v[3] = q.w; }
__device__ __forceinline__ void unpack4(float (&v)[4], uint2 q) {
  v[0] = __uint_as_float(q.x << 16); v[1] = __uint_as_float(q.x & 0xFFFF0000u);
  v[2] = __uint_as_float(q.y << 16); v[3] = __uint_as_float(q.y & 0xFFFF0000u);
}
template <typename T>
__device__ __forceinline__ typename Raw4<T>::type load4(const T* p) {
  return __ldg(reinterpret_cast<const typename Raw4<T>::type*>(p));
}
__device__ __forceinline__ void lds4(float (&v)[4], const float* p) { unpack4(v, *reinterpret_cast<const float4*>(p)); }

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

// y[c][j] = sum_i x(c, j)[i] W[i][j].  Thread = (eighth of the rows, four columns); the eight partial sums meet in shared
// memory (`red`: 8 CB D floats).
template <typename T, int D, int CB>
struct ProductNN {
  static constexpr int kCols = D / 4, kRows = D / 8;
  typename Raw4<T>::type w[kRows];
  __device__ __forceinline__ void load(const T* W, int tid) {
    if (D == 128 || tid < 8 * kCols) {
      const T* p = W + (size_t)(tid / kCols * kRows) * D + tid % kCols * 4;
#pragma unroll
      for (int r = 0; r < kRows; ++r) w[r] = load4(p + (size_t)r * D);
    }
  }
  // x(c, j): the row that candidate c's column j is multiplied with (16-byte aligned).  Ends before the barrier that
  // finish() needs in front of it.
  template <typename X>
  __device__ __forceinline__ void run(X x, float* red, int tid) {
    if (D == 128 || tid < 8 * kCols) {
      const int part = tid / kCols, j = tid % kCols * 4;
      float acc[CB][4];
#pragma unroll
      for (int c = 0; c < CB; ++c) acc[c][0] = acc[c][1] = acc[c][2] = acc[c][3] = 0.f;
      const float* xp[CB];
#pragma unroll
      for (int c = 0; c < CB; ++c) xp[c] = x(c, j) + part * kRows;
#pragma unroll
      for (int r = 0; r < kRows; r += 4) {
        float wv[4][4];
#pragma unroll
        for (int e = 0; e < 4; ++e) unpack4(wv[e], w[r + e]);
#pragma unroll
        for (int c = 0; c < CB; ++c) {
          float xv[4];
          lds4(xv, xp[c] + r);
#pragma unroll
          for (int e = 0; e < 4; ++e)
#pragma unroll
            for (int k = 0; k < 4; ++k) acc[c][k] = fmaf(xv[e], wv[e][k], acc[c][k]);
        }
      }
#pragma unroll
      for (int c = 0; c < CB; ++c)
        *reinterpret_cast<float4*>(red + (part * CB + c) * D + j) = make_float4(acc[c][0], acc[c][1], acc[c][2], acc[c][3]);
    }
  }
  // after a barrier: put(index of four consecutive values in [CB][D], the sums)
  template <typename Put>
  __device__ __forceinline__ static void finish(const float* red, int tid, Put put) {
    for (int i = tid; i < CB * kCols; i += kThreads) {
      float v[4], s[4];
      lds4(s, red + 4 * i);
#pragma unroll
      for (int k = 1; k < 8; ++k) {
        lds4(v, red + k * CB * D + 4 * i);
#pragma unroll
        for (int e = 0; e < 4; ++e) s[e] += v[e];
      }
      put(4 * i, s);
    }
  }
};

// y(c, h, i) = sum_{j in head h} W[i][j] x[c][j], HN heads of D / HN columns (HN = 1: a product with the transposed matrix).
// Every lane takes four consecutive columns of a row per step; the lanes of a head add up with the steps dealt out among
// them (a reduction that also scatters), so that a sum costs about one shuffle.
template <typename T, int D, int HN, int CB>
struct ProductNT {
  static constexpr int G = D / HN / 4 < 32 ? D / HN / 4 : 32;         // lanes of a head's slice of a row
  static constexpr int NS = D * D / (4 * kThreads) > 0 ? D * D / (4 * kThreads) : 1;
  static_assert((G & (G - 1)) == 0, "head widths are powers of two");
  static_assert(D / HN <= 128 && D * D % (4 * kThreads) == 0, "a step takes whole rows or a row takes whole steps");
  typename Raw4<T>::type w[NS];
  __device__ __forceinline__ void load(const T* W, int tid) {
#pragma unroll
    for (int s = 0; s < NS; ++s) w[s] = load4(W + (size_t)(s * kThreads + tid) * 4);
  }
  // x: [CB][D]
  template <typename Put>
  __device__ __forceinline__ void run(const float* x, int tid, Put put) {
    const int lane = tid & 31;
#pragma unroll
    for (int c = 0; c < CB; ++c) {
      float v[NS];
#pragma unroll
      for (int s = 0; s < NS; ++s) {
        const int col = (s * kThreads + tid) * 4 % D;
        float xv[4], wv[4];
        lds4(xv, x + c * D + col);
        unpack4(wv, w[s]);
        v[s] = fmaf(xv[3], wv[3], fmaf(xv[2], wv[2], fmaf(xv[1], wv[1], xv[0] * wv[0])));
      }
      reduce(v, lane, tid, c, put);
    }
  }
  template <typename Put>
  __device__ __forceinline__ static void reduce(float (&v)[NS], int lane, int tid, int c, Put put) {
    // stages that halve the number of values a lane holds (NS a power of two), then plain ones
    constexpr int kHalve = (NS & (NS - 1)) ? 0 : ilog2(NS < G ? NS : G);
    int base = 0;                                                     // first step whose sum this lane ends up with
#pragma unroll
    for (int k = 0; k < kHalve; ++k) {
      const int o = G >> (k + 1), n = NS >> (k + 1);
      const bool upper = lane & o;
#pragma unroll
      for (int i = 0; i < n; ++i) {
        const float keep = upper ? v[i + n] : v[i], send = upper ? v[i] : v[i + n];
        v[i] = keep + __shfl_xor_sync(0xffffffffu, send, o);
      }
      base += upper ? n : 0;
    }
    constexpr int kLeft = NS >> kHalve, kGroup = G >> kHalve;          // values left, lanes that still share each
#pragma unroll
    for (int o = kGroup >> 1; o > 0; o >>= 1)
#pragma unroll
      for (int i = 0; i < kLeft; ++i) v[i] += __shfl_xor_sync(0xffffffffu, v[i], o);
    if ((lane & (kGroup - 1)) == 0) {
#pragma unroll
      for (int i = 0; i < kLeft; ++i) {
        const int f = ((base + i) * kThreads + tid) * 4, row = f / D, h = f % D / (D / HN);
        put(c, h, row, v[i]);
      }
    }
  }
  __host__ __device__ static constexpr int ilog2(int n) { return n <= 1 ? 0 : 1 + ilog2(n / 2); }
};

// The warps of a block are dealt to its candidates: kWarps / CB each.

// y[c][h][j] = scale s_j . x[c][h] for the nv[c] segment vectors of candidate c (Hs: Lp rows of pitch DS per candidate; y: rows of
// pitch yp), four lanes per segment, all heads at once.
template <int D, int H, int CB, int DS>
__device__ __forceinline__ void scores(const float* Hs, const float* x, const int* nv, int Lp, int yp, float scale, float* y, int tid) {
  constexpr int kPer = kWarps / CB;
  const int warp = tid >> 5, lane = tid & 31, c = warp / kPer, p = lane & 3, n = nv[c];
  const float* xc = x + (size_t)c * H * DS + p * 4;
  for (int j0 = warp % kPer * 8; j0 < n; j0 += kPer * 8) {
    const int j = j0 + (lane >> 2);
    const float* s = Hs + ((size_t)c * Lp + min(j, n - 1)) * DS + p * 4;
    float acc[H];
#pragma unroll
    for (int h = 0; h < H; ++h) acc[h] = 0.f;
#pragma unroll
    for (int i = 0; i < D; i += 16) {
      float sv[4];
      lds4(sv, s + i);
#pragma unroll
      for (int h = 0; h < H; ++h) {
        float wv[4];
        lds4(wv, xc + h * DS + i);
#pragma unroll
        for (int e = 0; e < 4; ++e) acc[h] = fmaf(sv[e], wv[e], acc[h]);
      }
    }
#pragma unroll
    for (int h = 0; h < H; ++h) {
      acc[h] += __shfl_xor_sync(0xffffffffu, acc[h], 1);
      acc[h] += __shfl_xor_sync(0xffffffffu, acc[h], 2);
    }
    if (j < n) {
#pragma unroll
      for (int h = 0; h < H; ++h)
        if ((h & 3) == p) y[((size_t)c * H + h) * yp + j] = acc[h] * scale;
    }
  }
}

// softmax over a candidate's segments (rows of pitch ep), one warp per (candidate, head); a candidate without segments has no weights
template <int H, int CB>
__device__ __forceinline__ void softmax(float* e, const int* nv, int ep, int tid) {
  const int warp = tid >> 5, lane = tid & 31;
  for (int ch = warp; ch < CB * H; ch += kWarps) {
    const int n = nv[ch / H];
    float* ec = e + (size_t)ch * ep;
    float mx = -INFINITY, s = 0.f;
    for (int j = lane; j < n; j += 32) mx = fmaxf(mx, ec[j]);
    mx = warp_max(mx);
    for (int j = lane; j < n; j += 32) {
      const float w = expf(ec[j] - mx);
      ec[j] = w;
      s += w;
    }
    const float inv = 1.f / warp_sum(s);
    for (int j = lane; j < n; j += 32) ec[j] *= inv;
  }
}

// y[c][h] = sum_j w[c][h][j] s_j (w: rows of pitch wp): a group of D / 4 lanes (four features each) takes every kGroups-th segment of its
// candidate, all heads at once; the groups' sums meet in `red` (kFloats).
template <int D, int H, int CB>
struct Weighted {
  static constexpr int kPer = kWarps / CB, kCols = D / 4, kInWarp = 32 / kCols, kGroups = kPer * kInWarp;
  static constexpr int kFloats = CB * kGroups * H * D;                 // of `red`
  template <int DS>
  __device__ __forceinline__ static void run(const float* Hs, const float* w, const int* nv, int Lp, int wp, float* red, int tid) {
    const int warp = tid >> 5, lane = tid & 31, c = warp / kPer, sub = lane / kCols, n = nv[c];
    if (kInWarp * kCols < 32 && sub >= kInWarp) return;
    const int grp = warp % kPer * kInWarp + sub, i = lane % kCols * 4;
    float acc[H][4];
#pragma unroll
    for (int h = 0; h < H; ++h) acc[h][0] = acc[h][1] = acc[h][2] = acc[h][3] = 0.f;
    const float* s = Hs + (size_t)c * Lp * DS + i;
    const float* wc = w + (size_t)c * H * wp;
#pragma unroll 4
    for (int j = grp; j < n; j += kGroups) {
      float sv[4];
      lds4(sv, s + (size_t)j * DS);
#pragma unroll
      for (int h = 0; h < H; ++h) {
        const float a = wc[h * wp + j];
#pragma unroll
        for (int e = 0; e < 4; ++e) acc[h][e] = fmaf(a, sv[e], acc[h][e]);
      }
    }
#pragma unroll
    for (int h = 0; h < H; ++h)
      *reinterpret_cast<float4*>(red + (((size_t)c * kGroups + grp) * H + h) * D + i) =
          make_float4(acc[h][0], acc[h][1], acc[h][2], acc[h][3]);
  }
  // after a barrier: y rows of pitch DS
  template <int DS>
  __device__ __forceinline__ static void finish(const float* red, float* y, int tid) {
    for (int o = tid; o < CB * H * kCols; o += kThreads) {
      const int ch = o / kCols, i = o % kCols * 4, c = ch / H, h = ch % H;
      float s[4], v[4];
      lds4(s, red + (((size_t)c * kGroups) * H + h) * D + i);
#pragma unroll
      for (int g = 1; g < kGroups; ++g) {
        lds4(v, red + (((size_t)c * kGroups + g) * H + h) * D + i);
#pragma unroll
        for (int e = 0; e < 4; ++e) s[e] += v[e];
      }
      *reinterpret_cast<float4*>(y + (size_t)ch * DS + i) = make_float4(s[0], s[1], s[2], s[3]);
    }
  }
};

// Segment vectors of the block's candidates (rows of D values in global memory) to shared memory, fp32, rows of pitch DS.
template <typename T, int D, int CB, int DS>
__device__ __forceinline__ void stage_segments(float* Hs, const T* Hp, const int* nv, int c_base, int Lp, int tid) {
  constexpr int kPer = kWarps / CB * 32, kCols = D / 4;
  const int c = tid / kPer, n = nv[c] * kCols;
  const T* src = Hp + (size_t)(c_base + c) * Lp * D;
  float* dst = Hs + (size_t)c * Lp * DS;
#pragma unroll 8
  for (int i = tid % kPer; i < n; i += kPer) {
    float v[4];
    unpack4(v, *reinterpret_cast<const typename Raw4<T>::type*>(src + 4 * i));
    *reinterpret_cast<float4*>(dst + i / kCols * DS + i % kCols * 4) = make_float4(v[0], v[1], v[2], v[3]);
  }
}

}  // namespace dense
}  // namespace laser

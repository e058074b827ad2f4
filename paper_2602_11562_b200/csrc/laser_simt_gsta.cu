// Stacked attention in fp32 arithmetic for the widths in use (d = 32, 64, 96, 128; head widths 16, 32, 64, 128), for either
// I/O dtype: Eq. 7 re-associated as in gsta_simt_kernel (laser_simt.cu), which takes all other shapes.
//
// One block per CB candidates, everything of a candidate in shared memory, all layers in one launch.  Bound by latency: per
// layer three reads of weights from L2, a dozen barriers and the serial walk over the segments.  The weights of the next
// product are requested before the barrier in front of it, a product has all its reads in flight at once, and the
// contractions over the segment vectors read 16 bytes per shared-memory access for all heads.  Against the general kernel (CUDA
// events, about 6 us too long): 185 candidates, d = 64, four heads, 16 segments, two layers 23 -> 13 us, 9600 of them 384 -> 105;
// d = 128, eight heads, 48 segments, three layers, 370 candidates 156 -> 37, 4800 of them 1340 -> 271.
#include "laser_common.cuh"
#include "laser_simt_dense.cuh"

namespace laser {
namespace {

using namespace dense;

struct GstaF32Params {
  const void *Hp, *cands, *Wg;
  void* z;
  const int *lengths, *cand_offsets;
  int* status;
  int U, L, S, Lp, M, N;
  float inv_tau;
  int early;                     // the inputs are complete before this kernel starts (it follows another kernel of the call)
};

template <int D, int H, int CB>
__host__ __device__ constexpr int red_floats() {
  return Weighted<D, H, CB>::kFloats > 8 * CB * D ? Weighted<D, H, CB>::kFloats : 8 * CB * D;
}

template <typename T, int D, int H, int CB>
__global__ void __launch_bounds__(kThreads, 2) gsta_f32_kernel(const GstaF32Params P) {
  constexpr int DS = D + 4;                  // row pitch: eight consecutive rows start in different banks
  extern __shared__ __align__(16) float sm[];
  __shared__ int s_nv[CB], s_put[CB];
  const int Lp = P.Lp, c_base = blockIdx.x * CB, tid = threadIdx.x;
  float* t = sm;                             // [CB][D]
  float* q = t + CB * D;                     // [CB][D]
  float* qt = q + CB * D;                    // [CB][H][DS]   qt, later m
  float* red = qt + CB * H * DS;             // partial sums
  float* Hs = red + red_floats<D, H, CB>();  // [CB][Lp][DS]
  float* e = Hs + (size_t)CB * Lp * DS;      // [CB][H][Lp]
  const T* Wg = static_cast<const T*>(P.Wg);
  if (!P.early) chain_wait();
  ProductNN<T, D, CB> nn;
  ProductNT<T, D, H, CB> nt;
  if (P.M > 0) nn.load(Wg, tid);
  if (tid < CB) {
    // user of this candidate: the largest u with cand_offsets[u] <= cand (skipping users without candidates)
    const int cand = c_base + tid;
    int nv = -1;                             // no candidate here, or one that nothing is written for
    bool bad = false;
    if (cand < P.N) {
      int lo = 0, hi = P.U;                  // invariant: cand_offsets[lo] <= cand < cand_offsets[hi]
      if (P.cand_offsets[0] > cand || P.cand_offsets[P.U] <= cand) {
        bad = true;
      } else {
        while (hi - lo > 1) {
          const int mid = (lo + hi) >> 1;
          if (P.cand_offsets[mid] <= cand) lo = mid; else hi = mid;
        }
        const int len = P.lengths[lo];
        if (len < 0 || len > P.L) bad = true;
        else nv = min((len + P.S - 1) / P.S, Lp);
      }
    }
    s_put[tid] = nv >= 0;
    s_nv[tid] = bad ? -2 : max(nv, 0);       // (-2: reported below, once the status word has been cleared)
  }
  for (int i = tid; i < CB * D; i += kThreads)
    t[i] = c_base + i / D < P.N ? to_f32<T>(static_cast<const T*>(P.cands)[(size_t)c_base * D + i]) : 0.f;
  if (P.early) chain_wait();
  __syncthreads();
  if (tid < CB && s_nv[tid] == -2) {
    report_status(P.status, LASER_ERR_BAD_INPUT);
    s_nv[tid] = 0;
  }
  __syncthreads();
  int most = 0;
#pragma unroll
  for (int c = 0; c < CB; ++c) most = max(most, s_nv[c]);
  stage_segments<T, D, CB, DS>(Hs, static_cast<const T*>(P.Hp), s_nv, c_base, Lp, tid);

  for (int l = 0; l < P.M && most > 0; ++l) {
    const T *Wk = Wg + (size_t)(l * 3 + 1) * D * D, *Wv = Wk + D * D;
    nn.run([&](int c, int) { return (const float*)(t + c * D); }, red, tid);
    nt.load(Wk, tid);
    __syncthreads();
    nn.finish(red, tid, [&](int i, const float (&s)[4]) { *reinterpret_cast<float4*>(q + i) = make_float4(s[0], s[1], s[2], s[3]); });
    __syncthreads();
    nt.run(q, tid, [&](int c, int h, int i, float v) { qt[(c * H + h) * DS + i] = v; });
    __syncthreads();
    scores<D, H, CB, DS>(Hs, qt, s_nv, Lp, Lp, P.inv_tau, e, tid);
    __syncthreads();
    softmax<H, CB>(e, s_nv, Lp, tid);
    __syncthreads();
    Weighted<D, H, CB>::template run<DS>(Hs, e, s_nv, Lp, Lp, red, tid);
    nn.load(Wv, tid);
    __syncthreads();
    Weighted<D, H, CB>::template finish<DS>(red, qt, tid);
    __syncthreads();
    nn.run([&](int c, int j) { return (const float*)(qt + (c * H + j / (D / H)) * DS); }, red, tid);
    if (l + 1 < P.M) nn.load(Wv + D * D, tid);
    __syncthreads();
    nn.finish(red, tid, [&](int i, const float (&s)[4]) {
      float4* y = reinterpret_cast<float4*>(t + i);
      float4 v = *y;
      v.x += s[0]; v.y += s[1]; v.z += s[2]; v.w += s[3];
      *y = v;
    });
    __syncthreads();
  }
  for (int i = tid; i < CB * D; i += kThreads)
    if (s_put[i / D]) static_cast<T*>(P.z)[(size_t)c_base * D + i] = from_f32<T>(t[i]);
}

template <int D, int H, int CB>
size_t smem_bytes(int Lp) {
  return ((size_t)CB * (2 * D + H * (D + 4) + (size_t)Lp * (D + 4) + (size_t)H * Lp) + red_floats<D, H, CB>()) * sizeof(float);
}

template <typename T, int D, int H, int CB>
int launch_cb(const Plan& p, const GstaF32Params& P, cudaStream_t st) {
  const size_t smem = smem_bytes<D, H, CB>(p.Lp);
  LASER_CUDA_OK(allow_smem(gsta_f32_kernel<T, D, H, CB>, smem));
  LaunchScope ls("gsta_simt", st);
  LASER_CUDA_OK(launch_chained(gsta_f32_kernel<T, D, H, CB>, dim3((p.N + CB - 1) / CB), dim3(kThreads), smem, st, P));
  return LASER_OK;
}

constexpr size_t kMost = 226 * 1024;

template <typename T, int D, int H>
int launch(const Plan& p, const GstaF32Params& P, cudaStream_t st) {
  // Candidates per block, us (CUDA events, about 6 too long; fp32, one | two | four): while one per block makes a single wave of two
  // blocks per SM nothing is gained by sharing the weights (d = 64, four heads, 16 segments, two layers: 185 candidates 13 | 13
  // | 15; d = 128, two heads: 15 | 15 | 19); then two (370: 17 | 13 | 15; 25 | 19 | 19), from six per SM on four (600: 23 | 17 | 17; 33
  // | 25 | 23; 1200: 35 | 25 | 23; 52 | 37 | 33; 9600: 216 | 136 | 105; 353 | 228 | 166) unless four candidates' segments leave room for
  // one block per SM only (d = 128, eight heads, 48 segments, three layers, 1200: 95 | 78 | 89; 4800: 341 | 271 | 293).
  const int sms = device_sms();
  if (p.N > 6 * sms && smem_bytes<D, H, 4>(p.Lp) <= kMost / 2) return launch_cb<T, D, H, 4>(p, P, st);
  if (p.N > 2 * sms && smem_bytes<D, H, 2>(p.Lp) <= kMost) return launch_cb<T, D, H, 2>(p, P, st);
  if (smem_bytes<D, H, 1>(p.Lp) > kMost) return LASER_ERR_UNSUPPORTED;
  return launch_cb<T, D, H, 1>(p, P, st);
}

template <typename T>
int dispatch(const Plan& p, const GstaF32Params& P, cudaStream_t st) {
  switch (p.d * 16 + p.H) {
    case 32 * 16 + 1: return launch<T, 32, 1>(p, P, st);
    case 32 * 16 + 2: return launch<T, 32, 2>(p, P, st);
    case 64 * 16 + 1: return launch<T, 64, 1>(p, P, st);
    case 64 * 16 + 2: return launch<T, 64, 2>(p, P, st);
    case 64 * 16 + 4: return launch<T, 64, 4>(p, P, st);
    case 96 * 16 + 3: return launch<T, 96, 3>(p, P, st);
    case 96 * 16 + 6: return launch<T, 96, 6>(p, P, st);
    case 128 * 16 + 1: return launch<T, 128, 1>(p, P, st);
    case 128 * 16 + 2: return launch<T, 128, 2>(p, P, st);
    case 128 * 16 + 4: return launch<T, 128, 4>(p, P, st);
    case 128 * 16 + 8: return launch<T, 128, 8>(p, P, st);
    default: return LASER_ERR_UNSUPPORTED;
  }
}

}  // namespace

int gsta_f32(const Plan& p, const void* Hprime, const int32_t* lengths, const int32_t* cand_offsets, const void* cands,
             const void* Wg, void* z, char* ws, cudaStream_t st, bool follows_call) {
  if (p.N == 0) return LASER_OK;
  GstaF32Params P;
  P.Hp = Hprime; P.cands = cands; P.Wg = Wg; P.z = z; P.lengths = lengths; P.cand_offsets = cand_offsets;
  P.status = reinterpret_cast<int*>(ws + p.off_status);
  P.U = p.U; P.L = p.L; P.S = p.S; P.Lp = p.Lp; P.M = p.M; P.N = p.N; P.inv_tau = p.inv_tau; P.early = follows_call ? 1 : 0;
  return p.dtype == LASER_F32 ? dispatch<float>(p, P, st) : dispatch<__nv_bfloat16>(p, P, st);
}

}  // namespace laser

// Interfaces between the source files of the backward pass.  The kernels of the two tensor-core routes are chained (the next
// one's blocks are placed while the last blocks of this one run: 1.2 % of a call of 0.75-0.85 ms).  Those of the FP32 route and of the
// FP32 forward are chained too, but (the segment sums apart) they let their successor start only as they end: their grids are
// smaller than the GPU, and blocks placed early crowd the SMs that happen to be idle.  6 users x 45 candidates, backward: early
// release everywhere 60.8 us, no chaining 55.3, this 49.4; 2 x 63 of 2507 items, forward: 38.1 and 34.7.
#pragma once

#include "laser_common.cuh"
#include "laser_gsta_img.cuh"

namespace laser {

// What the stacked-attention kernels leave for the weight gradients, per layer (l = 0 .. M - 1): the targets t_l, q, m_h,
// and the gradients of t_{l+1}, q, qt_h; and, in dT0, the gradient of t_0.
struct GstaTrain {
  float *T, *Q, *dT, *dQ;         // [M, N, d]
  float *Mh, *dQt;                // [M, N, H, d]
  float* dT0;                     // [N, d]
};

// FP32 ALUs (laser_backward_simt.cu): recomputes the layers from the fp32 H' and runs them backward; writes every row of dHp.
bool gsta_train_simt_supported(const Plan& p);
int gsta_train_simt(const Plan& p, const float* Hp, const int32_t* lengths, const int32_t* cand_offsets, const void* cands,
                    const void* Wg, const float* dz, const GstaTrain& G, float* dHp, cudaStream_t st);

// The same for the tensor-core kernel, as bf16 high and low parts: arrays of [2][M, N, d] and [2][M, N, H, d].
struct GstaPlanes {
  __nv_bfloat16 *T, *Q, *dT, *dQ, *Mh, *dQt;
  float* dT0;
};

// FP32 ALUs, the widths in use (laser_backward_f32.cu).  The stacked attention as gsta_train_simt, leaving G or the same as bf16 parts, dH'
// in fp32 or rounded to bf16 (one of each pair is null); and the gates: every row of dK and dV, adds to dQf (zeroed before).
// LASER_ERR_UNSUPPORTED for all other shapes.
bool gsta_train_f32_pays(const Plan& p);      // in place of the tensor-core kernel
int gsta_train_f32(const Plan& p, const float* Hp, const int32_t* lengths, const int32_t* cand_offsets, const void* cands,
                   const void* Wg, const float* dz, const GstaTrain* G, const GstaPlanes* planes, float* dHp, __nv_bfloat16* dHp16,
                   cudaStream_t st);
bool sta_bwd_f32_supported(const Plan& p);
int sta_bwd_f32(const Plan& p, const float* Qf, const float* Kf, const float* Vf, const float* dHp, const int32_t* lengths,
                const int32_t* cand_offsets, float* dQf, float* dK, float* dV, cudaStream_t st);

// Tensor cores (laser_backward_gsta.cu), bf16 inputs: np = 1: segment vectors S0 in bf16; np = 2: segment vectors S0 + S1 (bf16
// high and low parts of fp32 values).  dS [N, Lp, d] leaves as fp32 in dS32 (np = 2) or rounded to bf16 in dS16, whichever is not
// null.  Rows of empty segments are neither read nor written.  gsta_weight_sums adds the layers' weight gradients from what
// gsta_train left in G.
// prepared: an earlier launch of the call did the work of gsta_train_prep(..) (train_prep_share, and gsta_build_order where it asks
// for an order).
bool gsta_train_supported(const Plan& p, int np);
size_t gsta_train_scratch_bytes(const Plan& p, int np);
TrainPrep gsta_train_prep(const Plan& p, int np, const void* Wg, const int32_t* lengths, const int32_t* cand_offsets, char* scratch);
int gsta_train(const Plan& p, int np, const void* S0, const void* S1, const int32_t* lengths, const int32_t* cand_offsets,
               const void* cands, const void* Wg, const float* dz, const GstaPlanes& G, float* dS32, __nv_bfloat16* dS16, char* scratch,
               cudaStream_t st, bool prepared);
int gsta_weight_sums(const Plan& p, const GstaPlanes& G, float* dWg, cudaStream_t st);

// Products over the item rows on the tensor cores (laser_backward_rows.cu), users' valid rows only, bf16 inputs.  rows_project: K, V
// and q_scale Q as bf16; the same launch sets arrays to zero and runs gsta_train's preparation.  rows_gradients: every row of d_items
// (zeros for padding) and the sums into dWk, dWv from dK and dV as bf16 high and low parts; d_cands = dT0 + dQf W_q^T / gamma and
// dWq += T^T dQf / gamma.
bool rows_mma_supported(const Plan& p);
int rows_project(const Plan& p, const void* items, const int32_t* lengths, const void* cands, const int32_t* cand_offsets, const void* Wq,
                 const void* Wk, const void* Wv, float q_scale, __nv_bfloat16* Qb, __nv_bfloat16* Kb, __nv_bfloat16* Vb,
                 const ZeroList& zero, const TrainPrep& prep, cudaStream_t st);
int rows_gradients(const Plan& p, const void* items, const int32_t* lengths, const void* cands, const int32_t* cand_offsets, const void* Wq,
                   const void* Wk, const void* Wv, const float* dQf, const __nv_bfloat16* dK_hi, const __nv_bfloat16* dK_lo,
                   const __nv_bfloat16* dV_hi, const __nv_bfloat16* dV_lo, const float* dT0, float* d_items, float* d_cands, float* dWq,
                   float* dWk, float* dWv, cudaStream_t st);

// A dense product on the FP32 ALUs: C[m][n] = D[m][n] + alpha (sum_k A(m, k) B(k, n) + sum_k A2(m, k) B2(k, n)), or, with
// atomic, C += alpha A B in slices of the contraction.  A(m, k) = ta ? A[k lda + m] : A[m lda + k], B(k, n) = tb ?
// B[n ldb + k] : B[k ldb + n] (A2, B2 alike); a16 / b16: bf16 operands.  `batch` products sa, sb, sc elements apart.
struct Product {
  const void *A, *B, *A2, *B2;
  const float* D;
  float* C;
  int lda, ldb, lda2, ldb2, ldc, M, N, K, K2, batch, sa, sb, sc, k_per;
  float alpha;
  bool ta, tb, a16, b16, atomic;
};
constexpr int kMaxProducts = 24;
// Independent products in as few launches as possible (k_per is filled in).
int run_products(Product* list, int n, cudaStream_t st);

}  // namespace laser

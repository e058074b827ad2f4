// laser_sta_forward_static: STA for callers that cannot provide (or obtain) a device workspace.
//
// Some callers of this library have no way to allocate device memory: a plug-in running inside a serving
// process whose GPU memory is owned, down to the last byte, by the host framework's pool; a request thread
// with a hard latency bound, where cudaMalloc's implicit device-wide synchronisation is not acceptable; a
// client that was handed a fixed set of input and output buffers and nothing else.  For them the scratch
// that the FP32-ALU STA kernels need (fp32 Q, K, V and the status word) lives in a fixed array that is part
// of the library image itself: every GPU that loads the library holds kStaticScratchBytes of it until the
// process exits.
#include <mutex>

#include "laser_common.cuh"

namespace laser {
namespace {

constexpr size_t kStaticScratchBytes = LASER_STATIC_SCRATCH_BYTES;
constexpr unsigned kMaxContexts = 64;

// The scratch itself.  In host code this name is only a host-side stand-in for the symbol, NOT a device
// address: host code must go through cudaGetSymbolAddress (below) and hand the result to the kernels.
static __device__ __align__(256) unsigned char g_static_scratch[kStaticScratchBytes];

std::mutex g_mu;
struct { unsigned ctx; char* ptr; } g_scratch[kMaxContexts];   // device address of g_static_scratch by context, once resolved
unsigned g_next;                                               // entry that is overwritten next

// Where g_static_scratch lives in the current context.  (Every context has its own copy: one that came after a reset, or beside
// another on the same device, must not be given the address that the library had in the other.)
int static_scratch_for_current_context(char** out) {
  const unsigned ctx = current_context();
  std::lock_guard<std::mutex> lock(g_mu);
  for (const auto& e : g_scratch)
    if (ctx && e.ctx == ctx) {
      *out = e.ptr;
      return LASER_OK;
    }
  void* ptr = nullptr;
  if (cudaGetSymbolAddress(&ptr, g_static_scratch) != cudaSuccess || !ptr) return LASER_ERR_CUDA;
  *out = static_cast<char*>(ptr);
  const unsigned now = current_context();                      // (the first call of a thread may have made one current)
  if (now) g_scratch[g_next++ % kMaxContexts] = {now, *out};
  return LASER_OK;
}

}  // namespace
}  // namespace laser

using namespace laser;

extern "C" int laser_sta_forward_static(const laser_config* cfg, const void* items, const int32_t* lengths,
                                        const void* cands, const int32_t* cand_offsets, const void* Wq,
                                        const void* Wk, const void* Wv, void* Hprime, int32_t* status_out,
                                        void* cuda_stream) {
  reset_launch_count();
  if (!cfg) return LASER_ERR_INVALID_ARG;
  laser_config c = *cfg;
  c.path = LASER_PATH_SIMT;     // the kernels whose scratch the static array replaces
  Plan p;
  int rc = make_plan(&c, &p);
  if (rc != LASER_OK) return rc;
  // Re-carve the scratch without the internal H' region (the caller supplies H'): status, Q, K, V.
  size_t off = 0;
  p.off_status = off; off = align_up(off + kStatusWords * sizeof(int));
  p.off_hp = 0;
  p.off_q = off; off = align_up(off + (size_t)p.N * p.dqk * sizeof(float));
  p.off_k = off; off = align_up(off + (size_t)p.U * p.L * p.dqk * sizeof(float));
  p.off_v = off; off = align_up(off + (size_t)p.U * p.L * p.d * sizeof(float));
  p.total = off;
  if (p.total > kStaticScratchBytes) return LASER_ERR_WORKSPACE;   // problem too large for the built-in scratch
  if (!lengths || !cand_offsets) return LASER_ERR_INVALID_ARG;
  if (p.N > 0) {
    const void* ptrs[] = {items, cands, Wq, Wk, Wv, Hprime};
    for (const void* q : ptrs)
      if (!q || (reinterpret_cast<uintptr_t>(q) & 15u)) return LASER_ERR_INVALID_ARG;
  }
  char* scratch = nullptr;
  if ((rc = static_scratch_for_current_context(&scratch)) != LASER_OK) return rc;
  cudaStream_t st = static_cast<cudaStream_t>(cuda_stream);
  // The array keeps whatever the previous call left in it.  Only the status word must start at zero (the first
  // kernel clears it): Q, K and V are fully rewritten for every row that is read afterwards.
  if (p.N == 0) {
    LASER_CUDA_OK(cudaMemsetAsync(scratch + p.off_status, 0, sizeof(int), st));
  } else {
    rc = simt_sta(p, items, lengths, cands, cand_offsets, Wq, Wk, Wv, Hprime, scratch, st);
    if (rc != LASER_OK) return rc;
  }
  if (status_out)
    LASER_CUDA_OK(cudaMemcpyAsync(status_out, scratch + p.off_status, sizeof(int32_t), cudaMemcpyDeviceToDevice, st));
  return LASER_OK;
}

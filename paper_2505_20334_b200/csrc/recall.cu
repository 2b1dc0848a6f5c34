// Recall of one selection against another (Section 3, Eq. 1-3): per unit
// |M_pred n M_gold| / |M_gold| for two index tensors as laq_select / laq_evict write them
// (ascending positions). One block per unit: M_gold is staged in shared memory (up to 48 KB of it),
// every thread takes elements of M_pred in turn and looks them up by binary search. Bound: the latency
// of the search's dependent reads (256 units of 1024 against 1024: 56 us with one warp per unit and the
// search in global memory).
#include "laq_internal.cuh"

namespace laq {
namespace {

constexpr int kRecallWarps = 8;
// What a launch may have in shared memory without an opt-in, less the kernel's own static array.
constexpr int kMaxStaged = (48 * 1024 - kRecallWarps * (int)sizeof(int)) / (int)sizeof(int32_t);

__global__ void __launch_bounds__(256) recall_kernel(const int32_t* pred, int n_pred, const int32_t* gold,
                                                     int n_gold, int32_t* n_common, float* recall,
                                                     int staged) {
  extern __shared__ int32_t s_gold[];
  __shared__ int s_hits[kRecallWarps];
  wait_for_predecessor();
  const int64_t u = blockIdx.x;
  const int32_t* a = pred + u * n_pred;
  const int32_t* g = gold + u * n_gold;
  if (staged) {
    for (int i = threadIdx.x; i < n_gold; i += 256) s_gold[i] = g[i];
    __syncthreads();
    g = s_gold;
  }
  int hits = 0;
  for (int i = threadIdx.x; i < n_pred; i += 256) {
    const int32_t x = a[i];
    int lo = 0, hi = n_gold;  // first position of g with g[pos] >= x
    while (lo < hi) {
      const int mid = (lo + hi) >> 1;
      if (g[mid] < x) lo = mid + 1;
      else hi = mid;
    }
    hits += (lo < n_gold && g[lo] == x) ? 1 : 0;
  }
  hits = __reduce_add_sync(0xffffffffu, hits);
  if ((threadIdx.x & 31) == 0) s_hits[threadIdx.x >> 5] = hits;
  __syncthreads();
  if (threadIdx.x == 0) {
    hits = 0;
    for (int w = 0; w < kRecallWarps; ++w) hits += s_hits[w];
    if (n_common) n_common[u] = hits;
    if (recall) recall[u] = n_gold > 0 ? (float)hits / (float)n_gold : 0.f;
  }
}

}  // namespace
}  // namespace laq

using namespace laq;

extern "C" laq_status laq_recall(int64_t n_units, const int32_t* idx_pred, int32_t n_pred,
                                 const int32_t* idx_gold, int32_t n_gold, int32_t* n_common,
                                 float* recall, void* cuda_stream) {
  if (n_units < 1 || n_pred < 1 || n_gold < 1 || !idx_pred || !idx_gold || (!n_common && !recall))
    return LAQ_ERR_INVALID_ARG;
  if ((reinterpret_cast<uintptr_t>(idx_pred) | reinterpret_cast<uintptr_t>(idx_gold) |
       reinterpret_cast<uintptr_t>(n_common) | reinterpret_cast<uintptr_t>(recall)) & 3u)
    return LAQ_ERR_INVALID_ARG;
  if (n_units > (1ll << 34)) return LAQ_ERR_UNSUPPORTED;
  const bool staged = n_gold <= kMaxStaged;
  cudaLaunchAttribute attr;
  programmatic_launch(&attr);
  cudaLaunchConfig_t cfg = {};
  cfg.blockDim = dim3(256);
  cfg.dynamicSmemBytes = staged ? (size_t)n_gold * sizeof(int32_t) : 0;
  cfg.stream = (cudaStream_t)cuda_stream;
  cfg.attrs = &attr;
  cfg.numAttrs = 1;
  constexpr int64_t kSlab = 1ll << 30;  // units per launch (one block each)
  for (int64_t u0 = 0; u0 < n_units; u0 += kSlab) {
    cfg.gridDim = dim3((unsigned)(n_units - u0 < kSlab ? n_units - u0 : kSlab));
    if (!cuda_ok(cudaLaunchKernelEx(&cfg, recall_kernel, idx_pred + u0 * n_pred, (int)n_pred,
                                    idx_gold + u0 * n_gold, (int)n_gold, n_common ? n_common + u0 : nullptr,
                                    recall ? recall + u0 : nullptr, staged ? 1 : 0)))
      return LAQ_ERR_CUDA;
  }
  return LAQ_OK;
}

// Recall of one selection against another (Section 3, Eq. 1-3): per unit
// |M_pred n M_gold| / |M_gold| for two index tensors as laq_select / laq_evict write them
// (ascending positions). Every thread takes elements of M_pred in turn and looks them up in M_gold by
// binary search. Bound: the latency of the search's dependent reads where there are few units, the cost of
// a block where there are many. So a unit has a block of its own, with M_gold staged in shared memory (up
// to 48 KB of it), or one warp that searches in global memory (see recall_by_warps).
#include "laq_internal.cuh"

namespace laq {
namespace {

constexpr int kRecallWarps = 8;
// What a launch may have in shared memory without an opt-in, less the kernel's own static array.
constexpr int kMaxStaged = (48 * 1024 - kRecallWarps * (int)sizeof(int)) / (int)sizeof(int32_t);

// kBlock: a block per unit, else a warp.
template <bool kBlock>
__global__ void __launch_bounds__(32 * kRecallWarps)
recall_kernel(const int32_t* pred, int n_pred, const int32_t* gold, int n_gold, int64_t n_units,
              int32_t* n_common, float* recall, int staged) {
  extern __shared__ int32_t s_gold[];
  __shared__ int s_hits[kRecallWarps];
  wait_for_predecessor();
  const int64_t u = kBlock ? (int64_t)blockIdx.x : (int64_t)blockIdx.x * kRecallWarps + (threadIdx.x >> 5);
  if (u >= n_units) return;  // (a warp of its own)
  const int n_threads = kBlock ? 32 * kRecallWarps : 32, tid = (int)threadIdx.x & (n_threads - 1);
  const int32_t* a = pred + u * n_pred;
  const int32_t* g = gold + u * n_gold;
  if (kBlock && staged) {
    for (int i = tid; i < n_gold; i += n_threads) s_gold[i] = g[i];
    __syncthreads();
    g = s_gold;
  }
  int hits = 0;
  for (int i = tid; i < n_pred; i += n_threads) {
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
  if (kBlock) {
    if ((threadIdx.x & 31) == 0) s_hits[threadIdx.x >> 5] = hits;
    __syncthreads();
    if (tid == 0) {
      hits = 0;
      for (int w = 0; w < kRecallWarps; ++w) hits += s_hits[w];
    }
  }
  if (tid == 0) {
    if (n_common) n_common[u] = hits;
    if (recall) recall[u] = n_gold > 0 ? (float)hits / (float)n_gold : 0.f;
  }
}

// Whether a warp per unit is the faster one. Measured on B200: a block adds 1.05 ns to the launch, 0.8 ns
// more for every 1000 staged positions (1.6 where M_gold is too long to be staged) and 2.9 for every 1000
// lookups; a warp 0.15 and 6.5 for every 1000 lookups, but its chain of lookups takes 3 us + 33 ns a lookup
// however few the units are. us with a warp / with a block, n_pred = n_gold unless given: 64: 10000 units
// 8.3 / 12.9, 5000 6.2 / 7.2, 2500 5.3 / 4.6; 256: 40000 57.7 / 69.4, 5000 12.4 / 9.9; 1024: 40000 289 / 221,
// 256 37.0 / 4.6; 128 against 12000: 2500 10.5 / 33.4, 256 8.9 / 4.2; 64 against 20000: 2500 7.3 / 9.2, 1184
// 7.3 / 4.1; 512 against 20000: 10000 57.5 / 45.2.
bool recall_by_warps(int64_t n_units, int n_pred, int n_gold, bool staged) {
  const double stage = staged ? n_gold / 1200.0 : 1.6;
  return n_pred < 250 + (staged ? n_gold / 5 : 0) && n_units * (1.05 + stage) > 3000.0 + 33.0 * n_pred;
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
  const bool by_warps = recall_by_warps(n_units, n_pred, n_gold, staged);
  const int64_t per_block = by_warps ? kRecallWarps : 1;
  cudaLaunchConfig_t cfg = {};
  cfg.blockDim = dim3(32 * kRecallWarps);
  cfg.dynamicSmemBytes = staged && !by_warps ? (size_t)n_gold * sizeof(int32_t) : 0;
  cfg.stream = (cudaStream_t)cuda_stream;
  cfg.attrs = &attr;
  cfg.numAttrs = 1;
  constexpr int64_t kSlab = 1ll << 30;  // units per launch (at most one block each)
  for (int64_t u0 = 0; u0 < n_units; u0 += kSlab) {
    const int64_t nu = n_units - u0 < kSlab ? n_units - u0 : kSlab;
    cfg.gridDim = dim3((unsigned)((nu + per_block - 1) / per_block));
    if (!cuda_ok(cudaLaunchKernelEx(&cfg, by_warps ? recall_kernel<false> : recall_kernel<true>,
                                    idx_pred + u0 * n_pred, (int)n_pred, idx_gold + u0 * n_gold, (int)n_gold, nu,
                                    n_common ? n_common + u0 : nullptr, recall ? recall + u0 : nullptr,
                                    staged ? 1 : 0)))
      return LAQ_ERR_CUDA;
  }
  return LAQ_OK;
}

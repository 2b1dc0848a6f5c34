// Step 4 (average or maximum pooling of the column sums) and step 5 (Eq. 4's ArgSort(...)[:B]: per-unit
// top-k by radix select on the fp32 bit patterns, ties to the lower position, ascending output
// followed by the retained tail).
#include <atomic>

#include "laq_internal.cuh"

namespace laq {
namespace {

constexpr int kSelThreads = 1024;
constexpr int kSelWarps = kSelThreads / 32;

// Geometry shared by the kernels below. Ls_full = L - R is the row length of the score tensor;
// a unit whose prompt is shorter (per-prompt lengths) scores only its first Lb - R positions.
// The tables are 5 KB of kernel parameters, which every launch has to carry: calls with neither
// per-prompt lengths nor per-layer budgets take the kernels without them.
struct SelGeom {
  int Ls_full, R, B, Bt, Hkv;
};
struct SelGeomTables : SelGeom {
  SeqLens sl;
  LayerBudgets lb;
};
__device__ __forceinline__ int unit_scored(const SelGeom& g, int64_t u) { return g.Ls_full; }
__device__ __forceinline__ int unit_scored(const SelGeomTables& g, int64_t u) {
  return unit_len(g.sl, (int)((u / g.Hkv) % g.Bt), g.Ls_full + g.R) - g.R;
}
// Slots unit u selects (its budget without the tail) and where its row of kept positions starts.
__device__ __forceinline__ int unit_kb(const SelGeom& g, int64_t u) { return g.B - g.R; }
__device__ __forceinline__ int unit_kb(const SelGeomTables& g, int64_t u) {
  return unit_budget(g.lb, u, g.Bt * g.Hkv, g.B) - g.R;
}
__device__ __forceinline__ int32_t* unit_out(const SelGeom& g, int32_t* idx, int64_t u) {
  return idx + u * (int64_t)g.B;
}
__device__ __forceinline__ int32_t* unit_out(const SelGeomTables& g, int32_t* idx, int64_t u) {
  return idx + unit_out_row(g.lb, u, g.Bt * g.Hkv, g.B);
}

// Average pooling: p_j = (1/k) * sum_{|t| <= k/2, 0 <= j+t < Ls} c_{j+t} (zero padding, divisor
// always k). Maximum pooling: the largest c_{j+t} over the same window positions that exist.
// One position near an edge of [0, Ls), or any position when the window is not unrolled.
__device__ __forceinline__ float pool_at(const float* c, int j, int h, int Ls, float inv_k,
                                         int pool_max) {
  if (pool_max) {
    float best = c[j];
    for (int t = -h; t <= h; ++t) {
      const int jj = j + t;
      if (jj >= 0 && jj < Ls) best = fmaxf(best, c[jj]);
    }
    return best;
  }
  float acc = 0.f;
  for (int t = -h; t <= h; ++t) {
    const int jj = j + t;
    if (jj >= 0 && jj < Ls) acc += c[jj];
  }
  return acc * inv_k;
}

// Four consecutive positions per thread: three 16-byte loads (rows of column sums are 512-byte aligned)
// hold every tap of a pooling kernel of up to nine. kPool: pooling kernel at compile time, 0 = kpool: one
// position per thread and a load per tap. kVec: the score rows allow 16-byte stores.
// Bound: HBM. 256 units of 32736 scores: 68 us with one position and a load per tap and thread.
template <int kPool, bool kVec, class Geom>
__global__ void __launch_bounds__(256)
pool_kernel(const float* __restrict__ colsum, int L_pad, float* __restrict__ pooled, int kpool, float inv_k,
            int pool_max, int64_t u0, const __grid_constant__ Geom g) {
  const int64_t u = u0 + blockIdx.y;
  const int Ls = unit_scored(g, u);
  const float* c = colsum + u * L_pad;
  if constexpr (kPool == 0) {
    const int j = 256 * blockIdx.x + threadIdx.x;
    if (j < g.Ls_full)
      pooled[u * (int64_t)g.Ls_full + j] = j < Ls ? pool_at(c, j, kpool / 2, Ls, inv_k, pool_max) : 0.f;
  } else {
    const int j = 4 * (blockIdx.x * 256 + threadIdx.x);
    if (j >= g.Ls_full) return;
    float r[4];
    constexpr int h = kPool / 2;
    static_assert(h <= 4, "one vector of halo");
    const float fill = pool_max ? __int_as_float(0xff800000) : 0.f;
    float x[12];
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      const int p = j - 4 + 4 * k;
      float4 v = make_float4(fill, fill, fill, fill);
      if (p >= 0 && p < Ls) v = *reinterpret_cast<const float4*>(c + p);  // (rows are padded to 128)
      x[4 * k] = v.x;
      x[4 * k + 1] = p + 1 < Ls ? v.y : fill;
      x[4 * k + 2] = p + 2 < Ls ? v.z : fill;
      x[4 * k + 3] = p + 3 < Ls ? v.w : fill;
    }
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      float acc = pool_max ? x[4 + i] : 0.f;
#pragma unroll
      for (int t = -h; t <= h; ++t) acc = pool_max ? fmaxf(acc, x[4 + i + t]) : acc + x[4 + i + t];
      r[i] = j + i < Ls ? (pool_max ? acc : acc * inv_k) : 0.f;
    }
    float* dst = pooled + u * (int64_t)g.Ls_full + j;
    if (kVec) {
      *reinterpret_cast<float4*>(dst) = make_float4(r[0], r[1], r[2], r[3]);
    } else {
#pragma unroll
      for (int i = 0; i < 4; ++i)
        if (j + i < g.Ls_full) dst[i] = r[i];
    }
  }
}

// Order-preserving map from fp32 bits to uint32 (larger float <=> larger key).
__device__ __forceinline__ uint32_t order_key(float f) {
  const uint32_t b = __float_as_uint(f);
  return (b & 0x80000000u) ? ~b : (b | 0x80000000u);
}

// One block per unit. Four 8-bit radix passes find the key of the Kb-th largest score and how
// many positions holding exactly that key are still needed; an ordered two-step compaction then
// writes the kept positions in ascending order.
__device__ __forceinline__ void select_unit(const float* p, int32_t* out, int Ls, int Kb, int R) {
  __shared__ uint32_t hist[256];
  __shared__ uint32_t s_prefix, s_need;
  __shared__ uint32_t s_gt[kSelWarps], s_eq[kSelWarps];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;

  if (tid == 0) {
    s_prefix = 0;
    s_need = (uint32_t)Kb;
  }
  uint32_t mask = 0;
  for (int pass = 0; pass < 4; ++pass) {
    const int shift = 24 - 8 * pass;
    if (tid < 256) hist[tid] = 0;
    __syncthreads();
    const uint32_t prefix = s_prefix;
    for (int i0 = 0; i0 < Ls; i0 += kSelThreads) {
      const int i = i0 + tid;
      uint32_t digit = 0xffffffffu;
      if (i < Ls) {
        const uint32_t key = order_key(p[i]);
        if ((key & mask) == prefix) digit = (key >> shift) & 255u;
      }
      // one shared-memory atomic per distinct digit in the warp
      const uint32_t peers = __match_any_sync(0xffffffffu, digit);
      if (digit != 0xffffffffu && lane == __ffs(peers) - 1) atomicAdd(&hist[digit], __popc(peers));
    }
    __syncthreads();
    if (warp == 0) {
      // lane owns bins [8*lane, 8*lane+8); find the bin where the count from the top reaches need
      uint32_t own = 0;
#pragma unroll
      for (int b = 0; b < 8; ++b) own += hist[lane * 8 + b];
      uint32_t suffix = own;  // inclusive suffix sum over lanes >= lane
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const uint32_t v = __shfl_down_sync(0xffffffffu, suffix, o);
        if (lane + o < 32) suffix += v;
      }
      const uint32_t above = suffix - own;
      const uint32_t need = s_need;
      if (above < need && need <= above + own) {
        uint32_t acc = above;
        for (int b = 7; b >= 0; --b) {
          const uint32_t hcount = hist[lane * 8 + b];
          if (acc + hcount >= need) {
            s_prefix = prefix | ((uint32_t)(lane * 8 + b) << shift);
            s_need = need - acc;
            break;
          }
          acc += hcount;
        }
      }
    }
    mask |= 255u << shift;
    __syncthreads();
  }
  const uint32_t theta = s_prefix;  // key of the Kb-th largest score
  const uint32_t need = s_need;     // positions holding exactly theta that are kept (lowest first)

  // warp w owns the contiguous positions [w*chunk, (w+1)*chunk)
  const int chunk = ((Ls + kSelWarps - 1) / kSelWarps + 31) / 32 * 32;
  const int beg = warp * chunk, end = min(Ls, beg + chunk);
  uint32_t n_gt = 0, n_eq = 0;
  for (int i0 = beg; i0 < end; i0 += 32) {
    const int i = i0 + lane;
    const uint32_t key = i < end ? order_key(p[i]) : 0u;
    n_gt += __popc(__ballot_sync(0xffffffffu, i < end && key > theta));
    n_eq += __popc(__ballot_sync(0xffffffffu, i < end && key == theta));
  }
  if (lane == 0) {
    s_gt[warp] = n_gt;
    s_eq[warp] = n_eq;
  }
  __syncthreads();
  uint32_t gt_run = 0, eq_run = 0;
  for (int w = 0; w < warp; ++w) {
    gt_run += s_gt[w];
    eq_run += s_eq[w];
  }
  const uint32_t lt_mask = (1u << lane) - 1u;
  for (int i0 = beg; i0 < end; i0 += 32) {
    const int i = i0 + lane;
    const uint32_t key = i < end ? order_key(p[i]) : 0u;
    const bool gt = i < end && key > theta;
    const bool eq = i < end && key == theta;
    const uint32_t bg = __ballot_sync(0xffffffffu, gt);
    const uint32_t be = __ballot_sync(0xffffffffu, eq);
    const uint32_t gt_before = gt_run + __popc(bg & lt_mask);
    const uint32_t eq_before = eq_run + __popc(be & lt_mask);
    if (gt || (eq && eq_before < need)) out[gt_before + min(eq_before, need)] = i;
    gt_run += __popc(bg);
    eq_run += __popc(be);
  }
  for (int t = tid; t < R; t += kSelThreads) out[Kb + t] = Ls + t;
}

// Step 5 alone, for units too long for the registers of two CTAs: scores of unit blockIdx.x in global
// memory.
__global__ void __launch_bounds__(kSelThreads) select_kernel(const float* __restrict__ pooled,
                                                             int32_t* __restrict__ idx,
                                                             const __grid_constant__ SelGeomTables g) {
  const int64_t u = blockIdx.x;
  select_unit(pooled + u * (int64_t)g.Ls_full, unit_out(g, idx, u), unit_scored(g, u), unit_kb(g, u), g.R);
}

// Steps 4 and 5 with the unit's scores held in registers. Thread t owns the consecutive positions
// [kItems t, kItems t + kItems), so kept positions leave in ascending order after one block-wide scan.
// The key of the Kb-th largest score is found from the top, two bits per step: `alive` marks a
// thread's keys that agree with the threshold's bits so far, and three block-wide counts (alive keys
// whose next bits are 11, 10, 01) tell which of the four go on and which lie above. The search ends
// as soon as the alive keys are exactly as many as are still wanted (for scores without ties, after
// about two thirds of the bits).
// kItems = 32: the keys are transposed into bit planes (word b holds bit b of all 32), so that a step
// is a handful of ANDs and population counts. kItems = 8, for a few short units, where nothing but the
// length of the dependent chain counts: four times the threads, bits taken from the keys one by one.
// Bound: issue slots (B200, 1024 units of 32736 scores: about 40 instructions per score; the layout
// with lane-strided positions, 7 shared-memory reads per pooled score, 32 one-bit steps and a ballot
// per position took 70).
// The pooling arithmetic is that of pool_kernel, so the scores are bit-identical to laq_score's.
constexpr int kRegItems = 32;
constexpr int kMaxSelWarps = 32;
constexpr int kCopy = -1;  // kPool: the scores are given, no pooling

// In-register transpose of a 32 x 32 bit matrix: on return bit i of a[b] is bit b of the old a[i].
__device__ __forceinline__ void transpose32(uint32_t (&a)[32]) {
  uint32_t m = 0x0000ffffu;
#pragma unroll
  for (int j = 16; j != 0; j >>= 1, m ^= m << j) {
#pragma unroll
    for (int k = 0; k < 32; ++k) {
      if ((k & j) == 0) {
        // swap the high-j block of row k with the low-j block of row k + j
        const uint32_t t = ((a[k] >> j) ^ a[k + j]) & m;
        a[k + j] ^= t;
        a[k] ^= t << j;
      }
    }
  }
}

// kPair: a unit of up to 65536 scored positions is taken by a cluster of two 1024-thread CTAs,
// CTA r holding positions [32768 r, 32768 r + 32768) in registers as before. What the threshold
// search needs from the other half is its counts of each step, read from the peer's shared memory
// after a cluster barrier; the kept positions of the second half are written behind those of the
// first. Both CTAs execute the same barriers whatever their data, so neither can be left waiting.
constexpr int kPairHalf = kRegItems * 1024;  // positions per CTA of a pair
constexpr int kHalo = 32;                    // staged positions on either side of a CTA's own

__device__ __forceinline__ void cluster_sync_all() {
  asm volatile("barrier.cluster.arrive.release.aligned;\nbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
// Reads the 32-bit word at the same shared-memory address in CTA `rank` of the cluster.
__device__ __forceinline__ uint32_t ld_peer_u32(const uint32_t* p, uint32_t rank) {
  const uint32_t local = (uint32_t)__cvta_generic_to_shared(p);
  uint32_t remote, v;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(remote) : "r"(local), "r"(rank));
  asm volatile("ld.shared::cluster.u32 %0, [%1];" : "=r"(v) : "r"(remote) : "memory");
  return v;
}

struct SelArgs {
  const float* src;   // column sums, or the scores themselves (kCopy)
  int64_t src_row;    // floats per unit in src
  float* pooled_out;  // may be NULL
  int32_t* idx;
  int kpool, pool_max;
  float inv_k;
  int halo;  // kPool == 0: staged positions on either side, as many as a window reaches (a multiple of 4)
};

// Shared memory holds the source from kHalo positions before the CTA's first to kHalo behind its last,
// every 32 floats followed by 4 unused ones: a thread's 16-byte reads of its own 32 floats then hit
// the banks of its neighbours' once. (kPool == 0 reads it by neighbouring threads, stages args.halo
// positions on either side and leaves no gaps until the pooled scores change hands.)
__device__ __forceinline__ int staged_at(int i) { return i + ((i >> 5) << 2); }
inline size_t staged_floats(int n) { return (size_t)(n + 2 * kHalo + 31) / 32 * 36; }

// kPool: pooling kernel at compile time (1, 3, 5, 7, 9: the window fits the vectors of halo), kCopy, or 0 =
// args.kpool.
template <int kPool, int kItems, bool kPair, class Geom>
__global__ void __launch_bounds__(1024, 1)
pool_select_reg_kernel(const __grid_constant__ SelArgs args, const __grid_constant__ Geom g) {
  __shared__ uint32_t s_cnt[2][2][kMaxSelWarps];
  __shared__ uint32_t s_scan[kMaxSelWarps];
  __shared__ uint32_t s_x[2][2], s_tot;  // pair: this CTA's counts of the current step; its totals
  extern __shared__ __align__(16) float s_c[];
  const int n_threads = blockDim.x, n_warps = n_threads >> 5;
  const uint32_t rank = kPair ? (blockIdx.x & 1u) : 0u;  // cluster of (2, 1, 1): rank = blockIdx.x % 2
  const int64_t u = kPair ? (int64_t)(blockIdx.x >> 1) : (int64_t)blockIdx.x;
  const int Ls = unit_scored(g, u), Kb = unit_kb(g, u), R = g.R;
  int32_t* out = unit_out(g, args.idx, u);
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int pos0 = kPair ? (int)rank * kPairHalf : 0;  // first position this CTA holds
  const int n_own = n_threads * kItems;
  allow_successor();
  wait_for_predecessor();

  // ---- stage: positions that do not exist count nothing in a sum and lose every maximum
  const float fill = kPool != kCopy && args.pool_max ? __int_as_float(0xff800000) : 0.f;
  const float* src = args.src + u * args.src_row;
  {
    const int halo = kPool == 0 ? args.halo : kHalo;
    const int n4 = (min(n_own, max(0, Ls - pos0)) + 2 * halo + 3) >> 2;  // what any thread reads
    const float* from = src + pos0 - halo;
    const bool aligned = kPool != kCopy;  // rows of column sums are 512-byte aligned
#pragma unroll 4
    for (int i = tid; i < n4; i += n_threads) {
      const int p = pos0 - halo + 4 * i;
      float4 v = make_float4(fill, fill, fill, fill);
      if (aligned && p >= 0 && p + 4 <= Ls) {
        v = __ldcs(reinterpret_cast<const float4*>(from) + i);
      } else if (p >= 0) {
        if (p < Ls) v.x = __ldcs(from + 4 * i);
        if (p + 1 < Ls) v.y = __ldcs(from + 4 * i + 1);
        if (p + 2 < Ls) v.z = __ldcs(from + 4 * i + 2);
        if (p + 3 < Ls) v.w = __ldcs(from + 4 * i + 3);
      }
      *reinterpret_cast<float4*>(s_c + (kPool == 0 ? 4 * i : staged_at(4 * i))) = v;
    }
  }
  __syncthreads();

  // ---- pool: keys of this thread's positions
  const int own = tid * kItems, base = pos0 + own;
  const int n_real = min(kItems, max(0, Ls - base));
  uint32_t w[kItems];
  if constexpr (kPool == 0) {
    // One load per tap. Item k of a thread is position k * n_threads + tid here: neighbouring threads load
    // neighbouring words, and the pooled scores change hands through shared memory. Positions that do not
    // exist hold `fill`; a window that reaches beyond the halo finds none there either. Four positions at a
    // time share the loop over the taps. (256 units of 4088 scores, kernel 31: the whole call 150 us with a
    // thread's consecutive positions one after the other, 96 so; kernel 65: 221 and 114.)
    const int h = min(args.kpool / 2, args.halo);
#pragma unroll
    for (int k0 = 0; k0 < kItems; k0 += 4) {
      const float* c[4];
      float acc[4];
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        // (beyond the last position: anything)
        c[k] = s_c + args.halo + min((k0 + k) * n_threads + tid, max(0, Ls - 1 - pos0));
        acc[k] = args.pool_max ? *c[k] : 0.f;
      }
      if (args.pool_max) {
#pragma unroll 4
        for (int t = -h; t <= h; ++t)
#pragma unroll
          for (int k = 0; k < 4; ++k) acc[k] = fmaxf(acc[k], c[k][t]);
      } else {
#pragma unroll 4
        for (int t = -h; t <= h; ++t)
#pragma unroll
          for (int k = 0; k < 4; ++k) acc[k] += c[k][t];
      }
#pragma unroll
      for (int k = 0; k < 4; ++k) w[k0 + k] = __float_as_uint(args.pool_max ? acc[k] : acc[k] * args.inv_k);
    }
    __syncthreads();
#pragma unroll
    for (int k = 0; k < kItems; ++k) s_c[staged_at(kHalo + k * n_threads + tid)] = __uint_as_float(w[k]);
    __syncthreads();
#pragma unroll
    for (int k = 0; k < kItems; ++k) w[k] = __float_as_uint(s_c[staged_at(kHalo + own + k)]);
  } else {
    constexpr int h = kPool > 0 ? kPool / 2 : 0;
    static_assert(h <= 4, "one vector of halo");
    const float4* row = reinterpret_cast<const float4*>(s_c);
    // eight positions at a time from a window of sixteen: with all 40 words in registers at once next
    // to the keys the block of 1024 threads spills
#pragma unroll
    for (int k0 = 0; k0 < kItems; k0 += 8) {
      float x[16];  // [own + k0 - 4, own + k0 + 12)
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        const float4 v = row[staged_at(kHalo + own + k0 - 4 + 4 * k) >> 2];
        x[4 * k] = v.x; x[4 * k + 1] = v.y; x[4 * k + 2] = v.z; x[4 * k + 3] = v.w;
      }
      if (kPool == kCopy) {
#pragma unroll
        for (int k = 0; k < 8; ++k) w[k0 + k] = __float_as_uint(x[4 + k]);
      } else if (args.pool_max) {
#pragma unroll
        for (int k = 0; k < 8; ++k) {
          float m = x[4 + k];
#pragma unroll
          for (int t = -h; t <= h; ++t) m = fmaxf(m, x[4 + k + t]);
          w[k0 + k] = __float_as_uint(m);
        }
      } else {
#pragma unroll
        for (int k = 0; k < 8; ++k) {
          float acc = 0.f;
#pragma unroll
          for (int t = -h; t <= h; ++t) acc += x[4 + k + t];
          w[k0 + k] = __float_as_uint(acc * args.inv_k);
        }
      }
    }
  }
  if (args.pooled_out) {  // through shared memory, so that the stores are coalesced
    __syncthreads();
#pragma unroll
    for (int k = 0; k < kItems; ++k) s_c[staged_at(kHalo + own + k)] = k < n_real ? __uint_as_float(w[k]) : 0.f;
    __syncthreads();
    float* dst = args.pooled_out + u * (int64_t)g.Ls_full + pos0;
    for (int i = tid; i < min(n_own, g.Ls_full - pos0); i += n_threads) dst[i] = s_c[staged_at(kHalo + i)];
  }
#pragma unroll
  for (int k = 0; k < kItems; ++k) w[k] = order_key(__uint_as_float(w[k]));
  if constexpr (kItems == 32) transpose32(w);  // w[i] bit b -> w[b] bit i

  // ---- threshold
  uint32_t alive = n_real >= 32 ? 0xffffffffu : (1u << n_real) - 1u;
  uint32_t above_mask = 0u;  // items known to lie above the threshold
  uint32_t above = 0u;       // their number in the whole unit
  uint32_t n_alive = (uint32_t)Ls;
#pragma unroll
  for (int bit = 30; bit >= 0; bit -= 2) {
    if (above + n_alive == (uint32_t)Kb) break;  // uniform: every alive item is wanted
    uint32_t hi, lo;
    if constexpr (kItems == 32) {
      hi = w[bit + 1];
      lo = w[bit];
    } else {
      hi = lo = 0u;
#pragma unroll
      for (int k = 0; k < kItems; ++k) {
        hi |= ((w[k] >> (bit + 1)) & 1u) << k;
        lo |= ((w[k] >> bit) & 1u) << k;
      }
    }
    const uint32_t m3 = alive & hi & lo, m2 = alive & hi & ~lo, m1 = alive & ~hi & lo;
    // per warp at most 1024 of each, per CTA 32768: two counts share a word
    uint32_t n32 = __reduce_add_sync(0xffffffffu, (uint32_t)__popc(m3) | ((uint32_t)__popc(m2) << 16));
    uint32_t n1 = __reduce_add_sync(0xffffffffu, (uint32_t)__popc(m1));
    const int buf = (bit >> 1) & 1;
    if (lane == 0) {
      s_cnt[buf][0][warp] = n32;
      s_cnt[buf][1][warp] = n1;
    }
    __syncthreads();
    n32 = __reduce_add_sync(0xffffffffu, lane < n_warps ? s_cnt[buf][0][lane] : 0u);
    n1 = __reduce_add_sync(0xffffffffu, lane < n_warps ? s_cnt[buf][1][lane] : 0u);
    uint32_t n3 = n32 & 0xffffu, n2 = n32 >> 16;
    if (kPair) {
      // add the other half's counts of this step (the two slots alternate: a slot is rewritten
      // only after the peer has passed the next barrier, i.e. after it has read it)
      if (tid == 0) {
        s_x[buf][0] = n32;
        s_x[buf][1] = n1;
      }
      cluster_sync_all();
      const uint32_t p32 = ld_peer_u32(&s_x[buf][0], rank ^ 1u);
      n3 += p32 & 0xffffu;
      n2 += p32 >> 16;
      n1 += ld_peer_u32(&s_x[buf][1], rank ^ 1u);
    }
    const uint32_t want = (uint32_t)Kb - above;
    if (n3 >= want) {
      alive = m3;
      n_alive = n3;
    } else if (n3 + n2 >= want) {
      above += n3;
      above_mask |= m3;
      alive = m2;
      n_alive = n2;
    } else if (n3 + n2 + n1 >= want) {
      above += n3 + n2;
      above_mask |= m3 | m2;
      alive = m1;
      n_alive = n1;
    } else {
      above += n3 + n2 + n1;
      above_mask |= m3 | m2 | m1;
      alive &= ~(hi | lo);
      n_alive -= n3 + n2 + n1;
    }
  }
  // `alive` now marks the items whose keys agree as far as they were looked at; `need` of them are
  // kept (the lowest positions first), with all `above` items
  const uint32_t need = (uint32_t)Kb - above;

  // ---- write the kept positions in ascending order: one scan of (above, alive) counts, 16 bits each
  const uint32_t mine = (uint32_t)__popc(above_mask) | ((uint32_t)__popc(alive) << 16);
  uint32_t scan = mine;
#pragma unroll
  for (int s = 1; s < 32; s <<= 1) {
    const uint32_t v = __shfl_up_sync(0xffffffffu, scan, s);
    if (lane >= s) scan += v;
  }
  if (lane == 31) s_scan[warp] = scan;
  __syncthreads();
  const uint32_t of_warp = lane < n_warps ? s_scan[lane] : 0u;
  const uint32_t before = __reduce_add_sync(0xffffffffu, lane < warp ? of_warp : 0u) + scan - mine;
  uint32_t gt = before & 0xffffu, eq = before >> 16;
  if (kPair) {
    // the second half writes behind the first: its running counts start from the first half's totals
    const uint32_t total = __reduce_add_sync(0xffffffffu, of_warp);
    if (tid == 0) s_tot = total;
    cluster_sync_all();
    if (rank == 1u) {
      const uint32_t t = ld_peer_u32(&s_tot, 0u);
      gt += t & 0xffffu;
      eq += t >> 16;
    }
  }
  for (uint32_t m = above_mask | alive; m != 0u; m &= m - 1u) {
    const int k = __ffs(m) - 1;
    if ((above_mask >> k) & 1u) {
      out[gt + min(eq, need)] = base + k;
      ++gt;
    } else {
      if (eq < need) out[gt + eq] = base + k;
      ++eq;
    }
  }
  if (rank == 0u)
    for (int t = tid; t < R; t += n_threads) out[Kb + t] = Ls + t;
  if (kPair) cluster_sync_all();  // no CTA leaves while its peer may still read its shared memory
}

// c[u][j] = max over the G heads of c_h[u*G + g][j] (LAQ_GROUP_MAX); rows are L_pad floats,
// a multiple of 128, read and written four at a time.
__global__ void group_max_kernel(const float4* __restrict__ colsum_h, float4* __restrict__ colsum,
                                 int row4, int G, int64_t total4) {
  const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (i >= total4) return;
  const int64_t u = i / row4;
  const int j = (int)(i % row4);
  const float4* src = colsum_h + u * G * (int64_t)row4 + j;
  float4 m = __ldcs(src);
  for (int g = 1; g < G; ++g) {
    const float4 x = __ldcs(src + g * (int64_t)row4);
    m.x = fmaxf(m.x, x.x); m.y = fmaxf(m.y, x.y); m.z = fmaxf(m.z, x.z); m.w = fmaxf(m.w, x.w);
  }
  colsum[i] = m;
}

}  // namespace

laq_status group_max_launch(const Dims& d, const float* colsum_h, int L_pad, float* colsum,
                            cudaStream_t stream, int* launches) {
  const int row4 = L_pad / 4;
  const int64_t total4 = d.U * (int64_t)row4;
  const int64_t blocks = (total4 + 255) / 256;
  if (blocks > 0x7fffffff) return LAQ_ERR_UNSUPPORTED;
  group_max_kernel<<<(unsigned)blocks, 256, 0, stream>>>((const float4*)colsum_h, (float4*)colsum, row4,
                                                         d.G, total4);
  *launches += 1;
  return cudaGetLastError() == cudaSuccess ? LAQ_OK : LAQ_ERR_CUDA;
}

static void fill_geom(const Dims& d, SelGeom* g) {
  g->Ls_full = d.Ls; g->R = d.R; g->B = d.B; g->Bt = d.Bt; g->Hkv = d.Hkv;
}
static SelGeomTables geom_tables(const Dims& d) {
  SelGeomTables g;
  fill_geom(d, &g);
  g.sl = d.sl;
  g.lb = d.lb;
  return g;
}
static SelGeom geom_plain(const Dims& d) {
  SelGeom g;
  fill_geom(d, &g);
  return g;
}
static bool has_tables(const Dims& d) { return d.sl.n > 0 || d.lb.n > 0; }

namespace {

template <bool kVec, class Geom>
void launch_pool(dim3 grid, cudaStream_t stream, const Dims& d, const float* colsum, int L_pad, float* pooled,
                 int64_t u0, const Geom& g) {
  const float inv_k = 1.0f / (float)d.kpool;
#define LAQ_POOL(K) \
  pool_kernel<K, kVec, Geom><<<grid, 256, 0, stream>>>(colsum, L_pad, pooled, d.kpool, inv_k, d.pool_max, u0, g)
  switch (d.kpool) {
    case 1: LAQ_POOL(1); break;
    case 3: LAQ_POOL(3); break;
    case 5: LAQ_POOL(5); break;
    case 7: LAQ_POOL(7); break;
    case 9: LAQ_POOL(9); break;
    default: LAQ_POOL(0); break;
  }
#undef LAQ_POOL
}

// Floats of shared memory that the kernel for any pooling window (kPool == 0) may take.
constexpr size_t kMaxWindowed = 56 * 1024;
// Positions it stages on either side of a CTA's own: what a window reaches of the Ls there are.
int window_halo(const Dims& d) {
  const int h = d.kpool / 2 < d.Ls ? d.kpool / 2 : d.Ls;
  return (h + 3) / 4 * 4;
}

// Shared memory opt-in of a kernel: a per-device attribute, set once per device and kernel.
template <class K>
bool opt_in(K kernel, size_t bytes, std::atomic<uint64_t>& devices) {
  int dev = 0;
  if (!cuda_ok(cudaGetDevice(&dev))) return false;
  if (dev < 64 && ((devices.load(std::memory_order_acquire) >> dev) & 1u)) return true;
  if (!cuda_ok(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes))) return false;
  if (dev < 64) devices.fetch_or(1ull << dev, std::memory_order_release);
  return true;
}

template <int kPool, int kItems, bool kPair, class Geom>
bool launch_select(unsigned units, int threads, cudaStream_t stream, const SelArgs& args, const Geom& g) {
  static std::atomic<uint64_t> devices{0};
  if (!opt_in(pool_select_reg_kernel<kPool, kItems, kPair, Geom>,
              (kPool == 0 ? kMaxWindowed : staged_floats(kPairHalf)) * sizeof(float), devices))
    return false;
  size_t floats = staged_floats(threads * kItems);
  if (kPool == 0 && floats < (size_t)threads * kItems + 2 * args.halo)
    floats = (size_t)threads * kItems + 2 * args.halo;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(kPair ? 2 * units : units);
  cfg.blockDim = dim3((unsigned)threads);
  cfg.dynamicSmemBytes = floats * sizeof(float);
  cfg.stream = stream;
  cudaLaunchAttribute attr[2];
  programmatic_launch(&attr[0]);
  attr[1].id = cudaLaunchAttributeClusterDimension;
  attr[1].val.clusterDim.x = 2;
  attr[1].val.clusterDim.y = attr[1].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = kPair ? 2 : 1;
  return cuda_ok(cudaLaunchKernelEx(&cfg, pool_select_reg_kernel<kPool, kItems, kPair, Geom>, args, g));
}

// Which of the kernels takes units of Ls scores: up to 32768 one CTA with 32 scores per thread, up to
// 65536 a pair of CTAs. Where the units are so few and short that every one has an SM to itself and
// waits for its own chain of steps only, 8 scores per thread (one unit of 1016: 14.4 us with 128
// threads); and where a wide window makes the taps most of the work, which wants more threads to a unit
// (256 units of 4088, kernel 1001: the whole call 618 us with 32 scores per thread, 208 with 8; kernel
// 129: 94; kernel 101, still with 32: 134).
template <int kPool, class Geom>
bool launch_select_sized(const Dims& d, cudaStream_t stream, const SelArgs& args, const Geom& g) {
  const unsigned units = (unsigned)d.U;
  if (d.Ls > kPairHalf) return launch_select<kPool, 32, true, Geom>(units, 1024, stream, args, g);
  if (d.Ls <= 8 * 1024 && (d.U <= 148 || (kPool == 0 && d.kpool > 128)))
    return launch_select<kPool, 8, false, Geom>(units, ((d.Ls + 7) / 8 + 31) / 32 * 32, stream, args, g);
  return launch_select<kPool, 32, false, Geom>(units, ((d.Ls + 31) / 32 + 31) / 32 * 32, stream, args, g);
}

// pool: 0 the scores are given, 1 pool them first.
template <class Geom>
bool launch_select_pooled(const Dims& d, bool pool, cudaStream_t stream, const SelArgs& args, const Geom& g) {
  if (!pool) return launch_select_sized<kCopy, Geom>(d, stream, args, g);
  switch (d.kpool) {
    case 1: return launch_select_sized<1, Geom>(d, stream, args, g);
    case 3: return launch_select_sized<3, Geom>(d, stream, args, g);
    case 5: return launch_select_sized<5, Geom>(d, stream, args, g);
    case 7: return launch_select_sized<7, Geom>(d, stream, args, g);
    case 9: return launch_select_sized<9, Geom>(d, stream, args, g);
    default: return launch_select_sized<0, Geom>(d, stream, args, g);
  }
}

}  // namespace

laq_status pool_launch(const Dims& d, const float* colsum, int L_pad, float* pooled,
                       cudaStream_t stream, int* launches) {
  const bool vec = d.Ls % 4 == 0 && (reinterpret_cast<uintptr_t>(pooled) & 15u) == 0;
  // grid.y limit: launch in slabs of units
  for (int64_t u0 = 0; u0 < d.U; u0 += 65535) {
    const unsigned nu = (unsigned)((d.U - u0 < 65535) ? d.U - u0 : 65535);
    const int per_block = d.kpool > 9 ? 256 : 1024;  // a position per thread, or four
    const dim3 grid((d.Ls + per_block - 1) / per_block, nu);
    if (has_tables(d)) {
      const SelGeomTables g = geom_tables(d);
      if (vec) launch_pool<true>(grid, stream, d, colsum, L_pad, pooled, u0, g);
      else launch_pool<false>(grid, stream, d, colsum, L_pad, pooled, u0, g);
    } else {
      const SelGeom g = geom_plain(d);
      if (vec) launch_pool<true>(grid, stream, d, colsum, L_pad, pooled, u0, g);
      else launch_pool<false>(grid, stream, d, colsum, L_pad, pooled, u0, g);
    }
    *launches += 1;
  }
  return cudaGetLastError() == cudaSuccess ? LAQ_OK : LAQ_ERR_CUDA;
}

// Units that the register kernels take.
static bool fits_registers(const Dims& d) { return d.Ls <= 2 * kPairHalf && d.U <= 0x3fffffff; }

static laq_status select_reg_launch(const Dims& d, bool pool, const float* src, int64_t src_row, float* pooled_out,
                                    int32_t* idx, cudaStream_t stream, int* launches) {
  SelArgs args;
  args.src = src;
  args.src_row = src_row;
  args.pooled_out = pooled_out;
  args.idx = idx;
  args.kpool = pool ? d.kpool : 1;
  args.pool_max = pool ? d.pool_max : 0;
  args.inv_k = 1.0f / (float)args.kpool;
  args.halo = pool ? window_halo(d) : 0;
  const bool ok = has_tables(d) ? launch_select_pooled(d, pool, stream, args, geom_tables(d))
                                : launch_select_pooled(d, pool, stream, args, geom_plain(d));
  if (!ok) return LAQ_ERR_CUDA;
  *launches += 1;
  return LAQ_OK;
}

laq_status select_launch(const Dims& d, const float* pooled, int32_t* idx, cudaStream_t stream,
                         int* launches) {
  if (d.U > 0x7fffffff) return LAQ_ERR_UNSUPPORTED;
  if (fits_registers(d)) return select_reg_launch(d, false, pooled, d.Ls, nullptr, idx, stream, launches);
  select_kernel<<<(unsigned)d.U, kSelThreads, 0, stream>>>(pooled, idx, geom_tables(d));
  *launches += 1;
  return cudaGetLastError() == cudaSuccess ? LAQ_OK : LAQ_ERR_CUDA;
}

laq_status pool_select_launch(const Dims& d, const float* colsum, int L_pad, float* pooled_out,
                              int32_t* idx, cudaStream_t stream, int* launches, bool* done) {
  *done = false;
  // else the caller uses the two-kernel path: units too long, or windows that do not fit next to them
  if (!fits_registers(d)) return LAQ_OK;
  const int own = d.Ls < kPairHalf ? (d.Ls + 1023) / 1024 * 1024 : kPairHalf;
  if (d.kpool > 9 && own + 2 * (size_t)window_halo(d) > kMaxWindowed) return LAQ_OK;
  const laq_status st = select_reg_launch(d, true, colsum, L_pad, pooled_out, idx, stream, launches);
  *done = st == LAQ_OK;
  return st;
}

}  // namespace laq

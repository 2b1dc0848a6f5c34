// Tensor-core scoring kernel for units whose logits fit the tensor memory of one thread-block
// cluster: steps 1-3 of the unit computation (Eq. 4 of Section 4.3 read as attention weights) with
// ONE pass over K and ONE matrix product per (row, key) pair.
//
// Softmax needs every row's sum before any column can be normalised. score_tc.cu therefore forms the
// logits twice (two sweeps over K). Here a cluster of C CTAs (one per SM) owns a whole unit: CTA r
// takes the 128-key tiles r, r + C, r + 2C, ... and keeps their logits S^T = K Q^T (keys on the TMEM
// lanes, fp32) in tensor memory while the row sums are formed and exchanged:
//   pass 1   adds 2^(t[r][j] - ref_r) over the keys. The logits are read in the fragment layout: a
//            thread holds a quarter of the rows, one accumulator each, for a quarter of its warp's
//            keys, and the cross-lane sum is taken once per unit, not once per tile;
//   exchange each CTA sends its (ref, sum) pairs to every CTA of the cluster through distributed
//            shared memory (st.async), and each merges them into b_r = m_r + log2(l_r);
//   pass 2   reads the same logits from tensor memory again and sums 2^(t[r][j] - b_r) over the rows.
// K crosses HBM and L2 once, the tensor cores do a third of the work of score_tc.cu (which for up to
// 64 rows holds them twice), and nothing goes through global memory but K, Q and the column sums: no
// counters, no partials, nothing to clear.
//
// The two passes run on warps of their own, so that pass 2 of a unit overlaps pass 1 of the next: a
// tile's TMEM slot goes back to the MMA issuer when pass 2 has read it, whatever unit comes next.
// 512 TMEM columns hold 512 / stride tiles, stride = rows rounded up to a power of two >= 16.
//
// The reference ref_r of a warp is the logit of its first key. Sums are scale
// free in fp32, so any reference within 2^100 of the largest logit will do; a warp whose sums
// overflow that (a key 69 nats above the reference) takes the maximum from tensor memory and redoes
// its sums.
//
// Warp roles (640 threads):
//   warp 0       TMA producer (one lane)
//   warp 1       tcgen05.mma issuer (an elected lane of the converged warp); owns the tensor memory
//   warps 2-3    exchange: merge the warps' pairs, send them, wait for the cluster's, publish -b_r
//   warps 4-11   pass 1, two warpgroups on alternate tiles
//   warps 12-19  pass 2, likewise, all rows of a key in one thread
// Every wait is bounded, as in score_tc.cu; clusters meet at a cluster barrier before they leave, so
// that no CTA exits while another may still write into its shared memory.
#include <cuda.h>
#include <cuda_runtime.h>
#include <math.h>

#include <atomic>
#include <mutex>

#include "laq_internal.cuh"
#include "softmax_math.cuh"
#include "tc_ptx.cuh"

namespace laq {
namespace {

using namespace laq::math;
using namespace laq::ptx;

constexpr int kThreads = 640;
constexpr int kPass1Warp = 4, kPass1Warps = 8;
constexpr int kPass2Warp = 12, kPass2Warps = 8;
constexpr int kExchangeWarps = 2;
constexpr int kMaxStages = 12;   // K stages in shared memory
constexpr int kMaxSlots = 32;    // TMEM tiles
constexpr int kMaxRows = 64;
constexpr uint32_t kTmemCols = 512;
constexpr uint32_t kBoxBytes = TILE_KEYS * 128;  // one 64-dim box of a K tile
#ifndef LAQ_TIMEOUT_CYCLES
#define LAQ_TIMEOUT_CYCLES 4000000000LL  // ~2 s: every device-side wait gives up after this
#endif
constexpr long long kTimeoutCycles = LAQ_TIMEOUT_CYCLES;
constexpr long long kDrainCycles = 2000000LL;
constexpr float kLog2e = 1.4426950408889634f;
constexpr float kNoKeys = -1e30f;  // reference of a row without keys
constexpr float kSumLimit = 1.2676506e30f;  // 2^100: above it a warp redoes its sums
constexpr int kMaxDevices = 64;

// Pass 2: how many of every four row pairs take the FMA-pipe exponential. Measured on B200 (64 rows,
// 32 layers x 8 heads): L 16384, batch 8: 2.26 ms at 0, 2.17 at 1, 2.18 at 2; L 4096: 67 / 66 / 68 us.
// In pass 1 any share is neutral.
constexpr int kPolyPass2 = 1;

struct ClArgs {
  int U;
  int Bt, Hkv, G, W, W_local, L, M, L_pad;
  int groups;        // ceil(M / 8): groups of eight rows
  int n16;           // rows of the kernel variant rounded up to 16: the N of the MMAs
  int boxes;         // 64-dim boxes per row (ceil(head_dim / 64))
  int ksteps;        // 16-dim MMA steps (ceil(head_dim / 16))
  int n_stages;      // K stages
  int slots_log2;    // TMEM tiles
  int stride_log2;   // TMEM columns per tile
  int c_log2;        // log2 of the cluster size where that is a whole number
  float scale_log2;
  int keep_status;    // the status words keep what an earlier piece of the call recorded
  int withhold_unit;  // test hook: this unit's statistics are never sent (-1: none)
  int32_t* hdr;
  float* colsum;
  SeqLens sl;
  // For cluster sizes between the powers of two, and behind the rest: between the fields above they changed
  // which of those one load fetches, and with it the registers of the kernels that never read them (64 rows
  // 96 for 94, with spills; us, 32 units of 2943 keys 15.4, so 14.6; 16 units of 7353 keys, 64 dims 19.8 / 18.9).
  int C;                       // CTAs per cluster
  int full_tiles, more_tiles;  // prompts of L positions: tiles of every CTA; CTAs that have one more
};

// Control block in dynamic shared memory, behind the K and Q stages.
struct Ctl {
  uint64_t q_full[2], q_empty[2];
  uint64_t k_full[kMaxStages], k_empty[kMaxStages];
  uint64_t slot_full[kMaxSlots], slot_empty[kMaxSlots];
  uint64_t stat_full[2], stat_empty[2];  // the pass-1 warps' pairs of a unit: delivered / read
  uint64_t lse_full[2];  // every CTA of the cluster has sent its pairs of a unit; both exchange warps
                         // arrive, so that neither can be two phases behind (a parity wait would miss one)
  uint64_t boff_full[2], boff_empty[2];  // -b_r of a unit: written / no longer needed
  uint64_t drain;
  uint32_t tmem_base;
  volatile int abort;
  alignas(16) float2 part[2][kPass1Warps][kMaxRows];  // (ref, sum) of the rows over a warp's keys
  alignas(16) float nboff[2][kMaxRows];          // -b_r (rows beyond M: -1e30)
  // followed by float2 lse_in[2][C][8 * groups]: the pairs each CTA of the cluster has sent
};
constexpr uint32_t kCtlBytes = (sizeof(Ctl) + 127u) / 128u * 128u;

// ------------------------------------------------------------------ cluster primitives
__device__ __forceinline__ uint32_t cluster_rank() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}
__device__ __forceinline__ uint32_t cluster_index() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%clusterid.x;" : "=r"(r));
  return r;
}
__device__ __forceinline__ uint32_t cluster_count() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%nclusterid.x;" : "=r"(r));
  return r;
}
__device__ __forceinline__ void cluster_sync() {
  asm volatile("barrier.cluster.arrive.release.aligned;\nbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
__device__ __forceinline__ uint32_t map_to_rank(uint32_t addr, uint32_t rank) {
  uint32_t r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(rank));
  return r;
}
// Writes a pair into a CTA of the cluster and counts its 8 bytes on a barrier of that CTA.
__device__ __forceinline__ void st_async_pair(uint32_t addr, float2 v, uint32_t bar) {
  asm volatile(
      "st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.v2.f32 [%0], {%1, %2}, [%3];" ::"r"(addr),
      "f"(v.x), "f"(v.y), "r"(bar)
      : "memory");
}
__device__ __forceinline__ bool mbar_try_wait_cluster(uint32_t bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n.reg .pred p;\n"
      "mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2, 2000;\n"
      "selp.u32 %0, 1, 0, p;\n}"
      : "=r"(ok)
      : "r"(bar), "r"(parity)
      : "memory");
  return ok != 0;
}

// ------------------------------------------------------------------ bounded waits
__device__ __noinline__ void give_up(int32_t* hdr, Ctl* ctl, int site) {
  ctl->abort = 1;
  if (atomicCAS(&hdr[HDR_STATUS], 0, (int)LAQ_ERR_TIMEOUT) == 0)
    hdr[HDR_WHERE] = (site << 16) | (int)(blockIdx.x & 0xffff);
}
template <bool kCluster = false>
__device__ __forceinline__ bool bounded_wait(const ClArgs& a, Ctl* ctl, uint64_t* barrier, uint32_t parity, int site) {
  const uint32_t bar = smem_u32(barrier);
  if (kCluster ? mbar_try_wait_cluster(bar, parity) : mbar_try_wait(bar, parity)) return true;
  const long long t0 = clock64();
  uint32_t spins = 0;
  while (!(kCluster ? mbar_try_wait_cluster(bar, parity) : mbar_try_wait_for(bar, parity, 2000))) {
    if ((++spins & 63u) == 0) {
      if (ctl->abort) return false;
      if (clock64() - t0 > kTimeoutCycles) {
        give_up(a.hdr, ctl, site);
        return false;
      }
    }
  }
  return true;
}
__device__ __forceinline__ void drain_wait(uint64_t* barrier, uint32_t parity) {
  const long long t0 = clock64();
  while (!mbar_try_wait_for(smem_u32(barrier), parity, 1000) && clock64() - t0 < kDrainCycles) {
  }
}

// ------------------------------------------------------------------ units
struct Unit {
  int u;
  int Lu;     // length of the unit's prompt
  int tiles;  // tiles of the unit that this CTA holds
};
// kShift: the cluster size is a power of two, c_log2 its logarithm. (Kernels of their own: with a product in
// place of the shift and a division of the tiles the others took up to 4 % longer, 256 units of 12000 keys and
// 64 rows 190 -> 197 us.)
// Place in the unit of the i-th tile of the CTA of that rank.
template <bool kShift>
__device__ __forceinline__ int tile_at(const ClArgs& a, int rank, int i) {
  return rank + (kShift ? i << a.c_log2 : i * a.C);
}
template <bool kShift>
__device__ __forceinline__ Unit unit_at(const ClArgs& a, int u, int rank) {
  Unit x;
  x.u = u;
  x.Lu = a.L;
  if (!kShift) {  // (all prompts have L positions)
    x.tiles = a.full_tiles + (rank < a.more_tiles ? 1 : 0);
    return x;
  }
  if (a.sl.n > 0) x.Lu = a.sl.len[((uint32_t)u / (uint32_t)a.Hkv) % (uint32_t)a.Bt];
  const int n_tiles = (x.Lu + TILE_KEYS - 1) / TILE_KEYS;
  x.tiles = rank < n_tiles ? (int)((uint32_t)(n_tiles - rank - 1) >> a.c_log2) + 1 : 0;
  return x;
}

// ------------------------------------------------------------------ pass 1
// Pass 1 needs sums over the keys, which are the TMEM lanes. It reads the logits in the fragment
// layout: a thread gets 2 rows of every 8 and, per 16 lanes, two keys, so that it holds a quarter of
// the rows for a quarter of the warp's keys. That leaves one accumulator and one reference per row
// it holds (16 of 64) in registers, and three shuffle steps per unit instead of five.
// 16 keys x 8 * kGroups rows, requested; v[4 g .. 4 g + 3] as in tmem_ld_frag*.
template <int kGroups>
__device__ __forceinline__ void request_frag(uint32_t taddr, float* v) {
  if constexpr (kGroups == 8) {
    tmem_ld_frag8(taddr, v);
  } else {
    if constexpr (kGroups & 4) tmem_ld_frag4(taddr, v);
    if constexpr (kGroups & 2) tmem_ld_frag2(taddr + 8u * (kGroups & 4), v + 4 * (kGroups & 4));
    if constexpr (kGroups & 1) tmem_ld_frag1(taddr + 8u * (kGroups & 6), v + 4 * (kGroups & 6));
  }
}
// Hides from this thread what its rows may not see: keys beyond the prompt, and, for the causal
// local queries of a LAQ++ window (Eq. 5), keys behind their own position.
template <int kGroups>
__device__ __forceinline__ void mask_frag(const ClArgs& a, int key, int lane, int Lu, float* v) {
  const int step = 8 % a.W;
  int i0 = (2 * (lane & 3)) % a.W, i1 = (2 * (lane & 3) + 1) % a.W;  // query indices inside their heads
#pragma unroll
  for (int g = 0; g < kGroups; ++g) {
    const int vis0 = i0 < a.W_local ? Lu - a.W_local + i0 + 1 : Lu;
    const int vis1 = i1 < a.W_local ? Lu - a.W_local + i1 + 1 : Lu;
    if (key >= vis0) v[4 * g] = __int_as_float(0xff800000);  // -inf
    if (key >= vis1) v[4 * g + 1] = __int_as_float(0xff800000);
    if (key + 8 >= vis0) v[4 * g + 2] = __int_as_float(0xff800000);
    if (key + 8 >= vis1) v[4 * g + 3] = __int_as_float(0xff800000);
    if ((i0 += step) >= a.W) i0 -= a.W;
    if ((i1 += step) >= a.W) i1 -= a.W;
  }
}
// Two values summed over the lanes that hold the same rows (lane bits 2-4).
__device__ __forceinline__ void sum_lanes(float* x) {
#pragma unroll
  for (int s = 4; s <= 16; s <<= 1) {
    x[0] += __shfl_xor_sync(0xffffffffu, x[0], s);
    x[1] += __shfl_xor_sync(0xffffffffu, x[1], s);
  }
}
// One step of the same for kN groups (a power of two): where there is more than one left, the lanes
// with bit kBit set go on with the upper half and the others with the lower half.
template <int kN, int kBit>
__device__ __forceinline__ void sum_step(float2* acc, float2* nref, int& group, int lane) {
  if constexpr (kN > 1) {
    const bool up = (lane & kBit) != 0;
#pragma unroll
    for (int i = 0; i < kN / 2; ++i) {
      const float2 send = up ? acc[i] : acc[i + kN / 2], keep = up ? acc[i + kN / 2] : acc[i];
      acc[i] = make_float2(keep.x + __shfl_xor_sync(0xffffffffu, send.x, kBit),
                           keep.y + __shfl_xor_sync(0xffffffffu, send.y, kBit));
      if (up) nref[i] = nref[i + kN / 2];
    }
    if (up) group += kN / 2;
  } else {
    acc[0].x += __shfl_xor_sync(0xffffffffu, acc[0].x, kBit);
    acc[0].y += __shfl_xor_sync(0xffffffffu, acc[0].y, kBit);
  }
}

// What a pass-1 warp knows about itself.
struct Warp1 {
  int lane, quad, index;  // index: 0 .. 7
  uint32_t lane_addr;     // tensor memory at this warp's 32 lanes
};
__device__ __forceinline__ Warp1 make_warp1(uint32_t tmem_base) {
  Warp1 w;
  w.lane = threadIdx.x & 31;
  w.index = (int)(threadIdx.x >> 5) - kPass1Warp;
  w.quad = w.index & 3;
  w.lane_addr = tmem_base + ((uint32_t)(w.quad * 32) << 16);
  return w;
}

// Pass 1 again for a warp whose sums overflowed: the largest logit of every row becomes its
// reference. Rare (a key more than 69 nats above the first one), so eight rows at a time; writes the
// warp's pairs. A row whose logits hold NaN or +inf ends here too, with a sum that is NaN, as its scores are to be.
// With one sum over the rows, pass 2 takes rows 2 and 3 of every four on the FMA pipe, whose exponential
// makes 2^-126 of a NaN, so rows 0 and 1 of those four, which the MUFU takes, pass it on.
template <bool kPerHead, bool kShift>
__device__ __noinline__ void redo_sums(const ClArgs& a, Ctl* ctl, int u, int rank, uint32_t tile0, int buf) {
  const Warp1 w = make_warp1(ctl->tmem_base);
  const Unit x = unit_at<kShift>(a, u, rank);
  const float c = a.scale_log2;
  const uint32_t slot_mask = (1u << a.slots_log2) - 1u;
  for (int g = 0; g < a.groups; ++g) {
    float m[2] = {-3.0e38f, -3.0e38f}, s[2] = {0.f, 0.f};
    for (int sweep = 0; sweep < 2; ++sweep) {
      for (int i = w.index >> 2; i < x.tiles; i += 2) {
        const int key0 = tile_at<kShift>(a, rank, i) * TILE_KEYS + w.quad * 32;
        if (key0 >= x.Lu) continue;
        const uint32_t slot = (tile0 + (uint32_t)i) & slot_mask;
        for (int half = 0; half < 2; ++half) {
          float v[4];
          tmem_ld_frag1(w.lane_addr + ((uint32_t)(16 * half) << 16) + (slot << a.stride_log2) + (uint32_t)(8 * g), v);
          tmem_ld_wait_n<4>(v);
          const int key = key0 + 16 * half + (w.lane >> 2);
          for (int k = 0; k < 4; ++k) {
            const int q = (8 * g + 2 * (w.lane & 3) + (k & 1)) % a.W;
            const int vis = q < a.W_local ? x.Lu - a.W_local + q + 1 : x.Lu;
            if (key + 8 * (k >> 1) >= vis) continue;
            if (sweep == 0) m[k & 1] = fmaxf(m[k & 1], v[k] * c);
            else s[k & 1] += ex2(fmaf(v[k], c, -m[k & 1]));
          }
        }
      }
      if (sweep == 0)
        for (int o = 4; o <= 16; o <<= 1) {
          m[0] = fmaxf(m[0], __shfl_xor_sync(0xffffffffu, m[0], o));
          m[1] = fmaxf(m[1], __shfl_xor_sync(0xffffffffu, m[1], o));
        }
    }
    sum_lanes(s);
    if (!kPerHead) {
      const float s2 = __shfl_xor_sync(0xffffffffu, s[0], 1), s3 = __shfl_xor_sync(0xffffffffu, s[1], 1);
      if ((w.lane & 1) == 0) {
        s[0] += 0.f * s2;
        s[1] += 0.f * s3;
      }
    }
    if (w.lane < 4) {
      ctl->part[buf][w.index][8 * g + 2 * w.lane] = make_float2(m[0], s[0]);
      ctl->part[buf][w.index][8 * g + 2 * w.lane + 1] = make_float2(m[1], s[1]);
    }
  }
}

// Pass 1 over this warp's tiles of a unit; tile0 is the CTA's running number of the unit's first
// tile, n the running number of the unit.
template <int kGroups, bool kPerHead, bool kShift>
__device__ __forceinline__ bool pass1(const ClArgs& a, Ctl* ctl, const Warp1& w, const Unit& x, int rank,
                                      uint32_t tile0, int n) {
  const float c = a.scale_log2;
  const float2 c2 = make_float2(c, c);
  const uint32_t slot_mask = (1u << a.slots_log2) - 1u;
  constexpr int kPow2 = kGroups > 4 ? 8 : (kGroups > 2 ? 4 : kGroups);
  float2 acc[kPow2], nref[kPow2];  // this thread's rows 8 g + 2 (lane % 4) and the next
#pragma unroll
  for (int g = 0; g < kPow2; ++g) acc[g] = nref[g] = make_float2(0.f, 0.f);
  bool have_ref = false;
  for (int i = w.index >> 2; i < x.tiles; i += 2) {
    const uint32_t t = tile0 + (uint32_t)i, slot = t & slot_mask;
    if (!bounded_wait(a, ctl, &ctl->slot_full[slot], (t >> a.slots_log2) & 1u, 21)) return false;
    __syncwarp();
    tc_fence_after();
    const int key0 = tile_at<kShift>(a, rank, i) * TILE_KEYS + w.quad * 32;
    if (key0 >= x.Lu) continue;  // warp-uniform: the prompt ends before this warp's keys
    const uint32_t taddr = w.lane_addr + (slot << a.stride_log2);
    const bool masked = key0 + 32 > x.Lu - a.W_local;
#pragma unroll
    for (int half = 0; half < 2; ++half) {
      float v[4 * kGroups];
      request_frag<kGroups>(taddr + ((uint32_t)(16 * half) << 16), v);
      tmem_ld_wait_n<4 * kGroups>(v);
      if (!have_ref) {  // the logits of the warp's first key
        have_ref = true;
#pragma unroll
        for (int g = 0; g < kGroups; ++g)
          nref[g] = make_float2(-c * __shfl_sync(0xffffffffu, v[4 * g], w.lane & 3),
                                -c * __shfl_sync(0xffffffffu, v[4 * g + 1], w.lane & 3));
      }
      if (masked) mask_frag<kGroups>(a, key0 + 16 * half + (w.lane >> 2), w.lane, x.Lu, v);
#pragma unroll
      for (int g = 0; g < kGroups; ++g) {
        const float2 e0 = exp2_mufu_pair(__ffma2_rn(make_float2(v[4 * g], v[4 * g + 1]), c2, nref[g]));
        const float2 e1 = exp2_mufu_pair(__ffma2_rn(make_float2(v[4 * g + 2], v[4 * g + 3]), c2, nref[g]));
        acc[g] = __fadd2_rn(acc[g], __fadd2_rn(e0, e1));
      }
    }
  }
  const int buf = n & 1;
  if (!bounded_wait(a, ctl, &ctl->stat_empty[buf], ((uint32_t)(n >> 1) & 1u) ^ 1u, 24)) return false;
  // sums over the warp's keys; a lane ends with one group's pair of rows
  int group = 0;
  sum_step<kPow2, 16>(acc, nref, group, w.lane);
  sum_step<(kPow2 > 1 ? kPow2 / 2 : 1), 8>(acc, nref, group, w.lane);
  sum_step<(kPow2 > 2 ? kPow2 / 4 : 1), 4>(acc, nref, group, w.lane);
  const int row = 8 * group + 2 * (w.lane & 3);
  const bool high = (row < a.M && !(acc[0].x < kSumLimit)) || (row + 1 < a.M && !(acc[0].y < kSumLimit));
  if (group < kGroups)  // (rows beyond M hold anything; lanes with the same rows write the same pairs)
    *reinterpret_cast<float4*>(&ctl->part[buf][w.index][row]) =
        make_float4(-nref[0].x, acc[0].x, -nref[0].y, acc[0].y);
  __syncwarp();
  if (__any_sync(0xffffffffu, high)) redo_sums<kPerHead, kShift>(a, ctl, x.u, rank, tile0, buf);
  tc_fence_before();
  __syncwarp();
  if (w.lane == 0) mbar_arrive(smem_u32(&ctl->stat_full[buf]));
  return true;
}

// ------------------------------------------------------------------ pass 2
// 8 * kGroups (up to 32) consecutive fp32 columns of this thread's TMEM lane, requested and waited for.
template <int kGroups>
__device__ __forceinline__ void load_groups(uint32_t taddr, float* v) {
  if constexpr (kGroups == 4) {
    tmem_ld32(taddr, v);
  } else {
    if constexpr (kGroups >= 2) tmem_ld16(taddr, v);
    if constexpr (kGroups != 2) tmem_ld8(taddr + 8u * (kGroups - 1), v + 8 * (kGroups - 1));
  }
  tmem_ld_wait_n<8 * kGroups>(v);
}

// Eight rows of this thread's key: 2^(c * v - b_r), added in packed pairs.
__device__ __forceinline__ void colsum_group(const float* v, float c, const float* nb, float2* acc) {
  const float2 c2 = make_float2(c, c);
  const float4* nb4 = reinterpret_cast<const float4*>(nb);
#pragma unroll
  for (int k = 0; k < 2; ++k) {
    const float4 b = nb4[k];
    const float* x = v + 4 * k;
    const float2 t0 = __ffma2_rn(make_float2(x[0], x[1]), c2, make_float2(b.x, b.y));
    const float2 t1 = __ffma2_rn(make_float2(x[2], x[3]), c2, make_float2(b.z, b.w));
    acc[2 * k] = __fadd2_rn(acc[2 * k], exp2_mufu_pair(t0));
    acc[2 * k + 1] = __fadd2_rn(acc[2 * k + 1], k < kPolyPass2 ? exp2_fma_pair(t1) : exp2_mufu_pair(t1));
  }
}

// One sum per query head: rows arrive in order, a head ends after every W of them.
struct HeadSums {
  float* out;      // column sum of the current head at this thread's key
  int64_t stride;  // to the next head
  int W, left;     // rows per head, rows left of the current one
  int heads_left;
  bool store;      // this thread's key exists
  float run;
  __device__ __forceinline__ void close() {
    if (heads_left > 0) {
      if (store) *out = run;
      out += stride;
      --heads_left;
    }
    run = 0.f;
    left = W;
  }
};
__device__ __forceinline__ void head_group(const float* v, float c, const float* nb, HeadSums& hs) {
  if ((hs.W & 3) == 0) {  // a head's rows fill whole groups of four
    const float4* nb4 = reinterpret_cast<const float4*>(nb);
    const float2 c2 = make_float2(c, c);
#pragma unroll
    for (int k = 0; k < 2; ++k) {
      const float4 b = nb4[k];
      const float* x = v + 4 * k;
      const float2 e0 = exp2_mufu_pair(__ffma2_rn(make_float2(x[0], x[1]), c2, make_float2(b.x, b.y)));
      const float2 e1 = exp2_mufu_pair(__ffma2_rn(make_float2(x[2], x[3]), c2, make_float2(b.z, b.w)));
      hs.run += (e0.x + e0.y) + (e1.x + e1.y);
      if ((hs.left -= 4) == 0) hs.close();
    }
  } else {
#pragma unroll
    for (int r = 0; r < 8; ++r) {
      hs.run += ex2(fmaf(v[r], c, nb[r]));
      if (--hs.left == 0) hs.close();
    }
  }
}

// Everything of the tile is in registers: the slot goes back to the MMA issuer.
__device__ __forceinline__ void release_slot(Ctl* ctl, uint32_t slot, int lane) {
  tc_fence_before();
  __syncwarp();
  if (lane == 0) mbar_arrive(smem_u32(&ctl->slot_empty[slot]));
}

template <int kGroups, bool kPerHead, bool kShift>
__device__ __forceinline__ bool pass2(const ClArgs& a, Ctl* ctl, uint32_t tmem_base, const Unit& x, int rank,
                                      uint32_t tile0, int n) {
  constexpr int kFirst = kGroups < 4 ? kGroups : 4, kRest = kGroups - kFirst;  // one or two loads
  const float c = a.scale_log2;
  const uint32_t slot_mask = (1u << a.slots_log2) - 1u;
  const int lane = threadIdx.x & 31, quad = (threadIdx.x >> 5) & 3;
  const int wg = (int)((threadIdx.x >> 5) - kPass2Warp) >> 2;
  const int buf = n & 1;
  if (!bounded_wait(a, ctl, &ctl->boff_full[buf], (uint32_t)(n >> 1) & 1u, 22)) return false;
  __syncwarp();
  tc_fence_after();
  const float* nb = ctl->nboff[buf];
  const uint32_t lane_addr = tmem_base + ((uint32_t)(quad * 32) << 16);
  // the unit's tiles are all complete: pass 1 has been through them
  for (int i = wg; i < x.tiles; i += 2) {
    const uint32_t slot = (tile0 + (uint32_t)i) & slot_mask;
    const int key = tile_at<kShift>(a, rank, i) * TILE_KEYS + quad * 32 + lane;
    const bool any = key - lane < x.Lu;  // warp-uniform: the prompt reaches this warp's keys
    float2 acc[4];
    HeadSums hs;
    if (any) {
      const uint32_t taddr = lane_addr + (slot << a.stride_log2);
#pragma unroll
      for (int k = 0; k < 4; ++k) acc[k] = make_float2(0.f, 0.f);
      if (kPerHead) {
        hs.out = a.colsum + (int64_t)x.u * a.G * a.L_pad + key;
        hs.stride = a.L_pad;
        hs.W = hs.left = a.W;
        hs.heads_left = a.G;
        hs.store = key < x.Lu;
        hs.run = 0.f;
      }
      float v[8 * kFirst];
      load_groups<kFirst>(taddr, v);
      if (kRest == 0) release_slot(ctl, slot, lane);
#pragma unroll
      for (int g = 0; g < kFirst; ++g) {
        if (kPerHead) head_group(v + 8 * g, c, nb + 8 * g, hs);
        else colsum_group(v + 8 * g, c, nb + 8 * g, acc);
      }
      if constexpr (kRest > 0) {
        load_groups<kRest>(taddr + 32u, v);
        release_slot(ctl, slot, lane);
#pragma unroll
        for (int g = 0; g < kRest; ++g) {
          if (kPerHead) head_group(v + 8 * g, c, nb + 32 + 8 * g, hs);
          else colsum_group(v + 8 * g, c, nb + 32 + 8 * g, acc);
        }
      }
      if (!kPerHead && key < x.Lu) {
        const float2 s2 = __fadd2_rn(__fadd2_rn(acc[0], acc[1]), __fadd2_rn(acc[2], acc[3]));
        a.colsum[(int64_t)x.u * a.L_pad + key] = s2.x + s2.y;
      }
    } else if (lane == 0) {
      mbar_arrive(smem_u32(&ctl->slot_empty[slot]));
    }
  }
  __syncwarp();
  if (lane == 0) mbar_arrive(smem_u32(&ctl->boff_empty[buf]));
  return true;
}

// ------------------------------------------------------------------ the kernel
template <int kGroups, bool kPerHead, bool kShift>
__global__ void __launch_bounds__(kThreads, 1)
score_cluster_kernel(const __grid_constant__ CUtensorMap tmap_q, const __grid_constant__ CUtensorMap tmap_k,
                     const __grid_constant__ ClArgs a) {
  long long clk0 = 0;
  unsigned long long ns0 = 0;
  if (threadIdx.x == 0) {
    prefetch_tensor_map(&tmap_q);
    prefetch_tensor_map(&tmap_k);
  }
  extern __shared__ __align__(1024) uint8_t smem_raw[];
  // stages first: the swizzled layout needs 1024-byte aligned addresses
  const uint32_t smem_base = smem_u32(smem_raw);
  const uint32_t k_stage_bytes = (uint32_t)a.boxes * kBoxBytes;
  const uint32_t q_box_bytes = (uint32_t)a.n16 * 128u;
  const uint32_t q_stage_bytes = (uint32_t)a.boxes * q_box_bytes;
  const uint32_t q_off = (uint32_t)a.n_stages * k_stage_bytes;
  const uint32_t ctl_off = q_off + 2u * q_stage_bytes;
  Ctl* ctl = reinterpret_cast<Ctl*>(smem_raw + ctl_off);
  float2* lse_in = reinterpret_cast<float2*>(smem_raw + ctl_off + kCtlBytes);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int rank = (int)cluster_rank();
  const int C = kShift ? 1 << a.c_log2 : a.C;
  const int n_clusters = (int)(kShift ? gridDim.x >> a.c_log2 : cluster_count());
  const int u_first = (int)(kShift ? blockIdx.x >> a.c_log2 : cluster_index());
  const int rows8 = a.groups * 8;

  if ((smem_base & 1023u) != 0) {  // the same in every CTA
    if (threadIdx.x == 0) atomicCAS(&a.hdr[HDR_STATUS], 0, (int)LAQ_ERR_INTERNAL);
    return;
  }

  // ---- set-up: barriers, zeroed Q stages (rows the loads never write stay zero), TMEM
  if (threadIdx.x == 0) {
    for (int i = 0; i < 2; ++i) {
      mbar_init(smem_u32(&ctl->q_full[i]), 1);
      mbar_init(smem_u32(&ctl->q_empty[i]), 1);
      mbar_init(smem_u32(&ctl->stat_full[i]), kPass1Warps);
      mbar_init(smem_u32(&ctl->stat_empty[i]), kExchangeWarps);
      mbar_init(smem_u32(&ctl->lse_full[i]), kExchangeWarps);
      mbar_init(smem_u32(&ctl->boff_full[i]), kExchangeWarps);
      mbar_init(smem_u32(&ctl->boff_empty[i]), kPass2Warps);
    }
    for (int i = 0; i < a.n_stages; ++i) {
      mbar_init(smem_u32(&ctl->k_full[i]), 1);
      mbar_init(smem_u32(&ctl->k_empty[i]), 1);
    }
    for (int i = 0; i < (1 << a.slots_log2); ++i) {
      mbar_init(smem_u32(&ctl->slot_full[i]), 1);
      mbar_init(smem_u32(&ctl->slot_empty[i]), 4);  // the four pass-2 warps that read the tile
    }
    mbar_init(smem_u32(&ctl->drain), 1);
    ctl->abort = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  {
    uint4* qz = reinterpret_cast<uint4*>(smem_raw + q_off);
    const int n16 = (int)(2u * q_stage_bytes / 16u);
    for (int i = threadIdx.x; i < n16; i += kThreads) qz[i] = make_uint4(0, 0, 0, 0);
    for (int i = threadIdx.x; i < 2 * kMaxRows; i += kThreads) (&ctl->nboff[0][0])[i] = -1e30f;
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                     smem_u32(&ctl->tmem_base)),
                 "r"(kTmemCols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  // Up to here nothing outside the SM was touched: the set-up overlaps the predecessor's end.
  wait_for_predecessor();
  allow_successor();
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    clk0 = clock64();
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(ns0));
    // The status words start at OK. CTAs start in order and a wait runs out long after that, so
    // no record of this launch is lost.
    if (!a.keep_status) a.hdr[HDR_STATUS] = a.hdr[HDR_WHERE] = 0;
  }
  cluster_sync();  // the cluster's barriers are initialised before anything is sent to them
  const uint32_t tmem_base = ctl->tmem_base;
  const uint32_t slot_mask = (1u << a.slots_log2) - 1u;

  if (warp == 0) {
    // ================= producer =================
    if (lane == 0) {
      uint32_t qc = 0, kc = 0, stage = 0, phase = 0;
      const uint64_t pol = l2_policy_evict_first();
      bool ok = true;
      for (int u = u_first; ok && u < a.U; u += n_clusters) {
        const Unit x = unit_at<kShift>(a, u, rank);
        const int h = u % a.Hkv, b = (u / a.Hkv) % a.Bt, layer = u / (a.Hkv * a.Bt);
        {
          const uint32_t qs = qc & 1u;
          if (!bounded_wait(a, ctl, &ctl->q_empty[qs], ((qc >> 1) & 1u) ^ 1u, 3)) break;
          const uint32_t bar = smem_u32(&ctl->q_full[qs]);
          mbar_expect_tx(bar, (uint32_t)(a.boxes * a.M) * 128u);
          const uint32_t dst = smem_base + q_off + qs * q_stage_bytes;
          for (int i = 0; i < a.boxes; ++i)
            tma_load_5d(dst + (uint32_t)i * q_box_bytes, &tmap_q, bar, 64 * i, 0, h * a.G, b, layer);
          ++qc;
        }
        for (int i = 0; i < x.tiles; ++i) {
          if (!bounded_wait(a, ctl, &ctl->k_empty[stage], phase ^ 1u, 4)) {
            ok = false;
            break;
          }
          const uint32_t bar = smem_u32(&ctl->k_full[stage]);
          mbar_expect_tx(bar, k_stage_bytes);
          const uint32_t dst = smem_base + stage * k_stage_bytes;
          const int key0 = tile_at<kShift>(a, rank, i) * TILE_KEYS;
          for (int j = 0; j < a.boxes; ++j)
            tma_load_5d_hint(dst + (uint32_t)j * kBoxBytes, &tmap_k, bar, 64 * j, key0, h, b, layer, pol);
          ++kc;
          if (++stage == (uint32_t)a.n_stages) {
            stage = 0;
            phase ^= 1u;
          }
        }
      }
      if (ctl->abort) {
        // loads that this lane has requested must not land after the CTA has exited
        const uint32_t n = (uint32_t)a.n_stages;
        for (uint32_t t = kc > n ? kc - n : 0u; t < kc; ++t) drain_wait(&ctl->k_full[t % n], (t / n) & 1u);
        for (uint32_t t = qc > 2u ? qc - 2u : 0u; t < qc; ++t) drain_wait(&ctl->q_full[t & 1u], (t >> 1) & 1u);
      }
    }
  } else if (warp == 1) {
    // ================= MMA issuer =================
    const uint32_t idesc = instr_desc(TILE_KEYS, a.n16);
    const uint32_t k_lo0 = smem_desc_lo(smem_base), q_lo0 = smem_desc_lo(smem_base + q_off);
    const uint32_t q_box = q_box_bytes >> 4;
    uint32_t qc = 0, stage = 0, phase = 0, t = 0;
    bool ok = true;
    for (int u = u_first; ok && u < a.U; u += n_clusters) {
      const Unit x = unit_at<kShift>(a, u, rank);
      const uint32_t qs = qc & 1u;
      if (!bounded_wait(a, ctl, &ctl->q_full[qs], (qc >> 1) & 1u, 11)) break;
      const uint32_t q_lo = q_lo0 + qs * (q_stage_bytes >> 4);
      for (int i = 0; i < x.tiles; ++i, ++t) {
        const uint32_t slot = t & slot_mask;
        if (!bounded_wait(a, ctl, &ctl->slot_empty[slot], ((t >> a.slots_log2) & 1u) ^ 1u, 13) ||
            !bounded_wait(a, ctl, &ctl->k_full[stage], phase, 12)) {
          ok = false;
          break;
        }
        __syncwarp();
        tc_fence_after();
        const uint32_t k_lo = k_lo0 + stage * (k_stage_bytes >> 4);
        const uint32_t d = tmem_base + (slot << a.stride_log2);
        const uint32_t full = smem_u32(&ctl->slot_full[slot]), empty = smem_u32(&ctl->k_empty[stage]);
        if (elect_one()) {
          // step kk covers dims [16 kk, 16 kk + 16): 32 bytes inside the 64-dim box kk >> 2
          if (a.ksteps == 8) {
#pragma unroll
            for (int kk = 0; kk < 8; ++kk)
              umma_bf16(d, k_lo + (uint32_t)(kk >> 2) * (kBoxBytes >> 4) + (uint32_t)(kk & 3) * 2u,
                        q_lo + (uint32_t)(kk >> 2) * q_box + (uint32_t)(kk & 3) * 2u, kSmemDescHi, idesc, kk > 0);
          } else {
#pragma unroll 1
            for (int kk = 0; kk < a.ksteps; ++kk)
              umma_bf16(d, k_lo + (uint32_t)(kk >> 2) * (kBoxBytes >> 4) + (uint32_t)(kk & 3) * 2u,
                        q_lo + (uint32_t)(kk >> 2) * q_box + (uint32_t)(kk & 3) * 2u, kSmemDescHi, idesc, kk > 0);
          }
          umma_commit(full);
          umma_commit(empty);
        }
        __syncwarp();
        if (++stage == (uint32_t)a.n_stages) {
          stage = 0;
          phase ^= 1u;
        }
      }
      if (!ok) break;
      if (elect_one()) umma_commit(smem_u32(&ctl->q_empty[qs]));
      __syncwarp();
      ++qc;
    }
    __syncwarp();
    if (ctl->abort && elect_one()) {  // MMAs still running must end before tensor memory is given back
      umma_commit(smem_u32(&ctl->drain));
      drain_wait(&ctl->drain, 0u);
    }
  } else if (warp < kPass1Warp) {
    // ================= exchange =================
    const int tid = threadIdx.x - 64;
    int n = 0;
    for (int u = u_first; u < a.U; u += n_clusters, ++n) {
      const int buf = n & 1;
      const uint32_t parity = (uint32_t)(n >> 1) & 1u;
      if (!bounded_wait(a, ctl, &ctl->stat_full[buf], parity, 31)) break;
      const uint32_t bar = smem_u32(&ctl->lse_full[buf]);
      if (tid == 0) mbar_expect_tx(bar, (uint32_t)(C * a.M) * 8u);
      else if (lane == 0) mbar_arrive(bar);
      float2* in = lse_in + (size_t)buf * C * rows8;
      if (u != a.withhold_unit) {
        for (int r = tid; r < a.M; r += 32 * kExchangeWarps) {
          // all pairs at once: a chain of pairwise merges took 600 cycles here and 1250 below (16 CTAs)
          float2 p[kPass1Warps];
          float m = kNoKeys, l = 0.f;
#pragma unroll
          for (int i = 0; i < kPass1Warps; ++i) {
            p[i] = ctl->part[buf][i][r];
            if (p[i].y == 0.f) p[i].x = kNoKeys;  // a warp without keys has no say
            m = fmaxf(m, p[i].x);
          }
#pragma unroll
          for (int i = 0; i < kPass1Warps; ++i) l = fmaf(p[i].y, ex2(p[i].x - m), l);
          const uint32_t addr = smem_u32(in + (size_t)rank * rows8 + r);
          for (int cc = 0; cc < C; ++cc)
            st_async_pair(map_to_rank(addr, (uint32_t)cc), make_float2(m, l), map_to_rank(bar, (uint32_t)cc));
        }
      }
      __syncwarp();
      if (lane == 0) mbar_arrive(smem_u32(&ctl->stat_empty[buf]));
      if (!bounded_wait(a, ctl, &ctl->boff_empty[buf], parity ^ 1u, 33)) break;
      if (!bounded_wait<true>(a, ctl, &ctl->lse_full[buf], parity, 32)) break;
      for (int r = tid; r < a.M; r += 32 * kExchangeWarps) {
        float m = kNoKeys, l = 0.f;
#pragma unroll 8
        for (int cc = 0; cc < C; ++cc) m = fmaxf(m, in[(size_t)cc * rows8 + r].x);
#pragma unroll 8
        for (int cc = 0; cc < C; ++cc) {
          const float2 p = in[(size_t)cc * rows8 + r];
          l = fmaf(p.y, ex2(p.x - m), l);
        }
        ctl->nboff[buf][r] = -(m + log2f(l));
      }
      __syncwarp();
      if (lane == 0) mbar_arrive(smem_u32(&ctl->boff_full[buf]));
    }
  } else if (warp < kPass2Warp) {
    // ================= pass 1 =================
    const Warp1 w = make_warp1(tmem_base);
    uint32_t tile0 = 0;
    int n = 0;
    for (int u = u_first; u < a.U; u += n_clusters, ++n) {
      const Unit x = unit_at<kShift>(a, u, rank);
      if (!pass1<kGroups, kPerHead, kShift>(a, ctl, w, x, rank, tile0, n)) break;
      tile0 += (uint32_t)x.tiles;
    }
  } else {
    // ================= pass 2 =================
    uint32_t tile0 = 0;
    int n = 0;
    for (int u = u_first; u < a.U; u += n_clusters, ++n) {
      const Unit x = unit_at<kShift>(a, u, rank);
      if (!pass2<kGroups, kPerHead, kShift>(a, ctl, tmem_base, x, rank, tile0, n)) break;
      tile0 += (uint32_t)x.tiles;
    }
  }

  // ---- teardown
  __syncwarp();
  if (ctl->abort) __nanosleep(20000);  // pairs this CTA has sent arrive within microseconds
  tc_fence_before();
  __syncthreads();
  cluster_sync();
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    unsigned long long ns1;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(ns1));
    *reinterpret_cast<long long*>(&a.hdr[HDR_CYCLES]) = clock64() - clk0;
    *reinterpret_cast<long long*>(&a.hdr[HDR_NANOS]) = (long long)(ns1 - ns0);
  }
  if (warp == 1) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(kTmemCols)
                 : "memory");
  }
}

#ifdef LAQ_SIZES_BETWEEN
constexpr bool kPow2 = false;
#else
constexpr bool kPow2 = true;
#endif
// [per head][groups of eight rows - 1] (seven groups run as eight)
constexpr int kVariants = 8;
#define LAQ_VARIANTS(H)                                                                                      \
  {(const void*)score_cluster_kernel<1, H, kPow2>, (const void*)score_cluster_kernel<2, H, kPow2>,           \
   (const void*)score_cluster_kernel<3, H, kPow2>, (const void*)score_cluster_kernel<4, H, kPow2>,           \
   (const void*)score_cluster_kernel<5, H, kPow2>, (const void*)score_cluster_kernel<6, H, kPow2>,           \
   (const void*)score_cluster_kernel<8, H, kPow2>, (const void*)score_cluster_kernel<8, H, kPow2>}
const void* const kKernels[2][kVariants] = {LAQ_VARIANTS(false), LAQ_VARIANTS(true)};
#undef LAQ_VARIANTS

#ifdef LAQ_SIZES_BETWEEN
}  // namespace

const void* cluster_kernel_between(bool per_head, int variant) { return kKernels[per_head ? 1 : 0][variant]; }
#else

// Clusters of each size that the device keeps resident with these kernels' resources, one CTA per SM;
// looked up once per device. 0: that cluster size cannot be launched.
constexpr int kMaxCluster = 16;
struct ClusterCounts {
  int resident[kMaxCluster + 1];
};
constexpr size_t kSmemBytes = 227 * 1024;

// What a kernel needs to be launched with all shared memory and in clusters of any size, per device.
bool allow_launch(const void* kernel) {
  return cuda_ok(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmemBytes)) &&
         cuda_ok(cudaFuncSetAttribute(kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1));
}

bool cluster_counts(int dev, ClusterCounts* out) {
  static std::mutex mutex;
  static ClusterCounts cached[kMaxDevices];
  static std::atomic<bool> known[kMaxDevices];
  if (dev < 0 || dev >= kMaxDevices) return false;
  if (!known[dev].load(std::memory_order_acquire)) {
    std::lock_guard<std::mutex> lock(mutex);
    if (!known[dev].load(std::memory_order_relaxed)) {
      for (int i = 0; i < 2 * kVariants; ++i)
        if (!allow_launch(kKernels[i / kVariants][i % kVariants])) return false;
      for (int i = 1; i <= kMaxCluster; ++i) {
        cudaLaunchAttribute attr;
        attr.id = cudaLaunchAttributeClusterDimension;
        attr.val.clusterDim.x = (unsigned)i;
        attr.val.clusterDim.y = attr.val.clusterDim.z = 1;
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3((unsigned)i);
        cfg.blockDim = dim3(kThreads);
        cfg.dynamicSmemBytes = kSmemBytes;
        cfg.attrs = &attr;
        cfg.numAttrs = 1;
        int n = 0;
        if (!cuda_ok(cudaOccupancyMaxActiveClusters(&n, kKernels[0][kVariants - 1], &cfg))) n = 0;
        cached[dev].resident[i] = n;
      }
      known[dev].store(true, std::memory_order_release);
    }
  }
  *out = cached[dev];
  return true;
}

// CTAs per cluster for a call whose units have up to n_tiles tiles; 0: no cluster holds a unit.
int cluster_size(const Dims& d, int n_tiles, int slots, const ClusterCounts& counts) {
  // Among the powers of two: ceil(U / clusters) rounds of T tiles per CTA. Cycles as measured on B200: a
  // tile takes the arithmetic of both passes or the CTA's share of the HBM stream (3600 bytes per cycle, at
  // most 30 per SM). The exchange of a unit is hidden where its tiles leave room for as many of the next
  // unit's, costs about 1000 where they leave some, and 3000 where they leave none. Large clusters leave
  // SMs idle (15 of 8 CTAs and 7 of 16 fit the 148), small ones fit fewer keys.
  const int boxes = (d.D + 63) / 64;
  int best = 0;
  double best_cost = 0.0;
  for (int C = 1; C <= kMaxCluster; C *= 2) {
    const int n = counts.resident[C], T = (n_tiles + C - 1) / C;
    if (n < 1 || T > slots || C > n_tiles) continue;
    const double rounds = (double)((d.U + n - 1) / n);
    const double tile = fmax(200.0 + 20.0 * d.M, (double)(boxes * kBoxBytes) * fmax(n * C, 120.0) / 3600.0);
    const double exchange = 2 * T <= slots ? 60.0 * C : (T < slots ? 1000.0 : 3000.0);
    const double cost = rounds * (T * tile + exchange);
    if (best == 0 || cost < best_cost) {
      best = C;
      best_cost = cost;
    }
  }
  if (best == 0 || d.sl.n > 0) return best;
  // A size between the powers of two (the 148 SMs hold 45 clusters of 3 CTAs, 26 of 5, 22 of 6, 15 of 7 to
  // 9, 11 of 10, 7 of 11 to 16) where 3 % or more are expected of it. A round takes the longest of: the HBM
  // stream, shared by the clusters of an average round, with its end exposed where the tiles leave no room
  // for the next unit's; the arithmetic, likewise; the chain from the first MMA of a unit through the exchange
  // to the end of pass 2, of which two can be under way (what short units are bound by: without it 512
  // units of 582 keys and 16 rows took 31.7 us in clusters of 5, 20.1 alone); and, with one sum per head,
  // pass 2 of the busier of the two warpgroups. The last unit's pass 2 ends the call. Fitted to the times of
  // all sizes on 9500 shapes of up to 65536 keys, K from HBM in 4500 of them and from L2 in the others: 2 %
  // faster than the powers of two alone on average, 48 shapes more than 1.5 % slower, the worst 7 %. With K from
  // HBM the size taken is 2.1 % above the best one on average, powers of two 4.4 %. To rank those by the same
  // costs gains another 0.3 %, but makes some 3 % of the shapes slower than they were.
  // Not for prompts of different lengths, which leave CTAs of a cluster without tiles in ways that this does
  // not foresee (3 prompts of 1319 to 6597 keys: 4 % slower).
  const auto cycles = [&](int C) {
    const int n = counts.resident[C], T = (n_tiles + C - 1) / C;
    const double rounds = (double)((d.U + n - 1) / n), full = (double)T / slots;
    const double sms = (double)d.U / rounds * C;  // of an average round
    const double stream = T * (d.D / 64.0) * fmax(477.0, kBoxBytes * sms / 3853.0) + fmax(0.0, 3400.0 * (full - 0.602));
    const double math = T * (751.0 + 6.4 * d.M) + fmax(0.0, 2185.0 * (full - 0.505));
    const double chain = 2467.0 + 30.0 * d.M + 7.2 * C;
    const double heads = d.group_mode == LAQ_GROUP_SUM ? 0.0 : (T + 1) / 2 * (682.0 + 18.8 * d.M);
    return rounds * fmax(fmax(stream, math), fmax(chain, heads)) + T * (122.0 + 0.7 * d.M);
  };
  best_cost = 0.967 * cycles(best);
  for (int C = 3; C < kMaxCluster; ++C) {
    if ((C & (C - 1)) == 0 || counts.resident[C] < 1 || (n_tiles + C - 1) / C > slots || C > n_tiles) continue;
    const double cost = cycles(C);
    if (cost < best_cost) {
      best = C;
      best_cost = cost;
    }
  }
  return best;
}

// The kernel of these rows for a size, ready to be launched on this device (0 <= dev < kMaxDevices). Those for
// sizes between the powers of two are a module of their own (score_cluster_between.cu), loaded when one of
// them is first wanted: a process's first scoring call took 12.6 ms with all of them in one, and takes 10.3;
// the first call of such a size 1.7.
const void* use_size(int dev, bool pow2, bool per_head, int variant) {
  if (pow2) return kKernels[per_head ? 1 : 0][variant];
  static std::atomic<uint32_t> allowed[kMaxDevices];
  const void* kernel = cluster_kernel_between(per_head, variant);
  const uint32_t bit = 1u << (variant + (per_head ? kVariants : 0));
  if (!(allowed[dev].load(std::memory_order_acquire) & bit)) {
    if (!allow_launch(kernel)) return nullptr;
    allowed[dev].fetch_or(bit, std::memory_order_release);
  }
  return kernel;
}

int log2_ceil(int x) {
  int l = 0;
  while ((1 << l) < x) ++l;
  return l;
}

#ifdef LAQ_TEST_HOOKS
std::atomic<int> g_last_cluster{0};
#endif

}  // namespace
}  // namespace laq

#ifdef LAQ_TEST_HOOKS
// Test builds only: CTAs per cluster of the last scoring call that took this kernel, 0 if the last one did not.
extern "C" __attribute__((visibility("default"))) int laq_test_last_cluster() { return laq::g_last_cluster.load(); }
#endif

namespace laq {
laq_status score_cluster_launch(const laq_params& p, const Dims& d, const Workspace& w, const void* q,
                                const void* k, char* ws, cudaStream_t stream, int* launches, bool* done) {
  *done = false;
#ifdef LAQ_TEST_HOOKS
  g_last_cluster = 0;
#endif
  // the caller's scheduling knobs belong to the two-sweep kernel
  if (d.M > kMaxRows || d.U > 0x3fffffff || d.D > 256 || d.tiles_per_task > 0 || d.sched_lag_tasks > 0)
    return LAQ_OK;
  int dev = 0;
  ClusterCounts counts;
  if (!cuda_ok(cudaGetDevice(&dev))) return LAQ_ERR_CUDA;
  if (!cluster_counts(dev, &counts)) return LAQ_OK;
  ClArgs a;
  a.groups = (d.M + 7) / 8;
  a.boxes = (d.D + 63) / 64;
  a.ksteps = (d.D + 15) / 16;
  a.stride_log2 = d.M <= 16 ? 4 : log2_ceil(d.M);
  a.slots_log2 = 9 - a.stride_log2;
  const int n_tiles = w.L_pad / TILE_KEYS, slots = 1 << a.slots_log2;
  const int best = cluster_size(d, n_tiles, slots, counts);
  if (best == 0) return LAQ_OK;
  const int C = best;
  const bool pow2 = (C & (C - 1)) == 0;
  a.C = C;
  a.c_log2 = log2_ceil(C);
  a.full_tiles = n_tiles / C;
  a.more_tiles = n_tiles % C;
  const int64_t clusters = d.U < counts.resident[C] ? d.U : counts.resident[C];
  const int variant = a.groups - 1;
  a.n16 = ((a.groups == 7 ? 64 : 8 * a.groups) + 15) / 16 * 16;
  const size_t stage = (size_t)a.boxes * kBoxBytes, qs = 2 * (size_t)a.boxes * a.n16 * 128;
  const size_t tail = kCtlBytes + 2 * (size_t)C * a.groups * 8 * sizeof(float2);
  if (qs + tail + 2 * stage > kSmemBytes) return LAQ_OK;
  a.n_stages = (int)((kSmemBytes - qs - tail) / stage);
  if (a.n_stages > kMaxStages) a.n_stages = kMaxStages;
  a.U = (int)d.U;
  a.Bt = d.Bt; a.Hkv = d.Hkv; a.G = d.G; a.W = d.W; a.W_local = d.W_local; a.L = d.L; a.M = d.M;
  a.L_pad = w.L_pad;
  a.scale_log2 = d.scale * kLog2e;
  a.keep_status = d.keep_status;
  a.withhold_unit = (int)test_withhold_unit();
  a.hdr = (int32_t*)(ws + w.off_hdr);
  const bool per_head = d.group_mode != LAQ_GROUP_SUM;
  a.colsum = (float*)(ws + (per_head ? w.off_colsum_h : w.off_colsum));
  a.sl = d.sl;

  CUtensorMap tmap_q, tmap_k;
  const uint64_t qdims[5] = {(uint64_t)d.D, (uint64_t)d.W, (uint64_t)d.Hq, (uint64_t)d.Bt, (uint64_t)d.NL};
  const int64_t qstr[4] = {p.q_stride_pos, p.q_stride_head, p.q_stride_batch, p.q_stride_layer};
  const uint32_t qbox[5] = {64, (uint32_t)d.W, (uint32_t)d.G, 1, 1};
  const uint64_t kdims[5] = {(uint64_t)d.D, (uint64_t)d.L, (uint64_t)d.Hkv, (uint64_t)d.Bt, (uint64_t)d.NL};
  const int64_t kstr[4] = {p.k_stride_pos, p.k_stride_head, p.k_stride_batch, p.k_stride_layer};
  const uint32_t kbox[5] = {64, TILE_KEYS, 1, 1, 1};
  if (!make_tensor_map(&tmap_q, q, qdims, qstr, qbox) || !make_tensor_map(&tmap_k, k, kdims, kstr, kbox))
    return LAQ_OK;  // layout TMA cannot describe

  cudaLaunchAttribute attr[2];
  programmatic_launch(&attr[0]);
  attr[1].id = cudaLaunchAttributeClusterDimension;
  attr[1].val.clusterDim.x = (unsigned)C;
  attr[1].val.clusterDim.y = attr[1].val.clusterDim.z = 1;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)(clusters * C));
  cfg.blockDim = dim3(kThreads);
  cfg.dynamicSmemBytes = kSmemBytes;
  cfg.stream = stream;
  cfg.attrs = attr;
  cfg.numAttrs = 2;
  const void* kernel = use_size(dev, pow2, per_head, variant);
  void* args[] = {&tmap_q, &tmap_k, &a};
  if (!kernel || !cuda_ok(cudaLaunchKernelExC(&cfg, kernel, args))) return LAQ_ERR_CUDA;
  *launches += 1;
  *done = true;
#ifdef LAQ_TEST_HOOKS
  g_last_cluster = C;
#endif
  return LAQ_OK;
}
#endif  // !LAQ_SIZES_BETWEEN

}  // namespace laq

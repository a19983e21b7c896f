// Shared device helpers and the workspace layout of libasd (sm_103a).
#pragma once

#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include "asd.h"

namespace asd {

constexpr int kMaxNodes = ASD_MAX_TREE_NODES;
constexpr int kMaxLmRanges = 256;   // upper bound on LM-head vocabulary ranges (CTAs)
constexpr int kMaxAttnParts = 8;    // attention context splits = cluster size (portable max)
constexpr float kLog2e = 1.4426950408889634f;
constexpr float kLn2 = 0.6931471805599453f;
// Bounded waits give up after this many SM clock cycles (about 2 s at 2 GHz).
constexpr long long kWaitCycles = 4000000000LL;

// Per-sequence flags written by the tree preparation kernel.
enum SeqFlag : int { kSeqBadTree = 1, kSeqBadToken = 2, kSeqBadCtx = 4 };

// One vocabulary range's running softmax statistics of one LM-head row.
struct LmPartial {
  float m;   // max logit in the range
  float s;   // sum of exp(logit - m) over the range
  int a;     // lowest vocab id attaining m
  int pad;
};

// Offsets (bytes) of the workspace regions; every region is 256-byte aligned.
struct WsLayout {
  size_t status;       // int32[2]: [0] first device error code; [1] a bounded wait gave up
  size_t seq_flags;    // int32[B]
  size_t child_start;  // int32[T]: global slot of the node's first child
  size_t child_cnt;    // int32[T]
  size_t child_tok;    // int32[T]: children tokens, grouped by parent, sorted by (token, id)
  size_t child_id;     // int32[T]: global node id of each slot
  size_t lm_part;      // LmPartial[T][g_lm]
  size_t total;        // everything above: what every call needs
  size_t at_part;      // attention partials: plan int2[B], then (max, sum) and output rows
  size_t full;         // total and the attention partials (asd_workspace_bytes)
  int g_lm;            // CTAs of the LM-head kernel (vocabulary ranges)
  int n_parts;         // context splits of the mma.sync and fp32 attention kernels (the
                       // tree keys ride with the last one)
  // lazy LM-head schedule only (0 otherwise)
  size_t lz_count;     // int32[2][max_path + 1]: rows, then active sequences per pass
  size_t lz_seq;       // int2[B]: a sequence's first row and rows in the pass
  size_t lz_rows;      // int32[2][T]: node ids of a pass's rows (two passes in flight)
  size_t lz_h;         // bf16[2][lz_cap][hidden]: their hidden rows
  int lz_cap;          // T rounded up to 128
  int attn_tc;         // tensor-core attention (attention has the SMs to itself): 1 one
                       // query tile per CTA, 2 two query tiles in ping-pong, 3 either, by
                       // the context lengths; 0: the bf16 mma.sync or the fp32 kernel
};

// ---------------------------------------------------------------- device utils

// Programmatic dependent launch: a kernel launched with programmatic stream
// serialisation may start while its predecessor in the stream still runs;
// pdl_wait() blocks until every predecessor grid has completed and its memory
// is visible, pdl_launch_dependents() lets the next kernel start launching.
// Both are no-ops for kernels launched without the attribute.
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void pdl_launch_dependents() {
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}

// The first error of a call, in its status word.  The call's first kernel
// clears the word, so a later kernel that started early waits for it here.
__device__ __forceinline__ void set_status(int* status, int code) {
  pdl_wait();
  atomicCAS(status, 0, code);
}

// A bounded wait gave up: ASD_ERR_TIMEOUT as the call's status (unless an
// earlier error came first) and word 1 of the status block set, which tells
// the later kernels of the call that results of this one are incomplete.
__device__ __forceinline__ void note_timeout(int* status) {
  set_status(status, ASD_ERR_TIMEOUT);
  atomicExch(status + 1, 1);
}

// Merges the g_lm per-range LM-head statistics of one row (max m, sum of
// exp(logit - m) s, lowest argmax a) into the row's, one warp per row with up
// to 8 ranges per lane; every lane returns them.  The tail kernel and the lazy
// pass kernel use this, so their rows agree bit for bit.  The maximum comes
// first, so that the sums' exponentials do not wait for one another (folding
// range into range, two of them per step and lane, the merge of 60 rows stood
// 4.9 us in the headline step's tail; now 3.5).
__device__ __forceinline__ void merge_row(const LmPartial* part, int g_lm, float& m, float& s,
                                          int& a) {
  constexpr int kPerLane = kMaxLmRanges / 32;
  const int lane = threadIdx.x & 31;
  const float4* src = reinterpret_cast<const float4*>(part);
  float4 q[kPerLane];
#pragma unroll
  for (int k = 0; k < kPerLane; ++k)
    q[k] = lane + 32 * k < g_lm ? __ldcg(src + lane + 32 * k) : make_float4(-INFINITY, 0.f, 0.f, 0.f);
  m = q[0].x;
#pragma unroll
  for (int k = 1; k < kPerLane; ++k) m = fmaxf(m, q[k].x);
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
  s = 0.f;
  a = 0x7fffffff;
#pragma unroll
  for (int k = 0; k < kPerLane; ++k) {
    if (q[k].x == -INFINITY) continue;
    s = fmaf(q[k].y, exp2f((q[k].x - m) * kLog2e), s);
    if (q[k].x == m) a = min(a, __float_as_int(q[k].z));
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  a = __reduce_min_sync(0xffffffffu, a);
}

__device__ __forceinline__ uint32_t smem_u32(const void* p) {
  return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}

__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
}

__device__ __forceinline__ void fence_mbar_init() {
  asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}

__device__ __forceinline__ void fence_proxy_async() {
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
}

__device__ __forceinline__ void mbar_expect_tx(uint32_t bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes)
               : "memory");
}

__device__ __forceinline__ void mbar_arrive(uint32_t bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}

__device__ __forceinline__ bool mbar_try_wait(uint32_t bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok)
      : "r"(bar), "r"(parity)
      : "memory");
  return ok != 0;
}

// Non-blocking test of the phase with the given parity.
__device__ __forceinline__ bool mbar_test_wait(uint32_t bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok)
      : "r"(bar), "r"(parity)
      : "memory");
  return ok != 0;
}

// Waits until the phase with the given parity has completed.  Gives up after
// `budget` SM clock cycles (kWaitCycles unless the call set another) and
// returns false (the caller records ASD_ERR_TIMEOUT).  try_wait may suspend
// the thread for a while by itself, so a shortened budget (a test making a
// wait give up) polls with the non-blocking test_wait instead.
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity,
                                          long long budget = kWaitCycles) {
  if (budget < kWaitCycles) {
    const long long t0 = clock64();
    while (!mbar_test_wait(bar, parity))
      if (clock64() - t0 > budget) return false;
    return true;
  }
  if (mbar_try_wait(bar, parity)) return true;
  const long long t0 = clock64();
  while (true) {
#pragma unroll 1
    for (int i = 0; i < 32; ++i)
      if (mbar_try_wait(bar, parity)) return true;
    if (clock64() - t0 > budget) return false;
  }
}

// The wait budget of a call: the host's, where a test set a shorter one
// (asd_debug_set_wait_cycles).  Waits for copies and MMAs already in flight
// always use the full kWaitCycles.
__device__ __forceinline__ long long wait_budget(long long set) {
  return set > 0 ? set : kWaitCycles;
}

__device__ __forceinline__ uint64_t l2_policy_evict_first() {
  uint64_t p;
  asm volatile("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(p));
  return p;
}

__device__ __forceinline__ uint64_t l2_policy_evict_last() {
  uint64_t p;
  asm volatile("createpolicy.fractional.L2::evict_last.b64 %0, 1.0;" : "=l"(p));
  return p;
}

// 2D tiled TMA load into this CTA's shared memory, completing on `bar`.
// x (innermost coordinate) must be a multiple of 16 bytes / element size.
__device__ __forceinline__ void tma_load_2d(uint32_t dst, const CUtensorMap* tmap, uint32_t bar,
                                            int x, int y, uint64_t policy) {
  asm volatile(
      "cp.async.bulk.tensor.2d.shared::cluster.global.tile.mbarrier::complete_tx::bytes"
      ".L2::cache_hint [%0], [%1, {%3, %4}], [%2], %5;" ::"r"(dst),
      "l"(reinterpret_cast<uint64_t>(tmap)), "r"(bar), "r"(x), "r"(y), "l"(policy)
      : "memory");
}

// 3D tiled TMA load (coordinates x innermost) into shared memory.
__device__ __forceinline__ void tma_load_3d(uint32_t dst, const CUtensorMap* tmap, uint32_t bar,
                                            int x, int y, int z, uint64_t policy) {
  asm volatile(
      "cp.async.bulk.tensor.3d.shared::cluster.global.tile.mbarrier::complete_tx::bytes"
      ".L2::cache_hint [%0], [%1, {%3, %4, %5}], [%2], %6;" ::"r"(dst),
      "l"(reinterpret_cast<uint64_t>(tmap)), "r"(bar), "r"(x), "r"(y), "r"(z), "l"(policy)
      : "memory");
}

// Plain bulk copy global -> shared (both 16-byte aligned, bytes % 16 == 0).
__device__ __forceinline__ void bulk_load(uint32_t dst, const void* src, uint32_t bytes,
                                          uint32_t bar, uint64_t policy) {
  asm volatile(
      "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes.L2::cache_hint"
      " [%0], [%1], %2, [%3], %4;" ::"r"(dst),
      "l"(reinterpret_cast<uint64_t>(src)), "r"(bytes), "r"(bar), "l"(policy)
      : "memory");
}

// `bytes` (4 or 16) of global memory -> shared memory by cp.async, zeros unless `in`.
template <int bytes>
__device__ __forceinline__ void copy_async(float* dst, const float* src, bool in) {
  const int n = in ? bytes : 0;
  if (bytes == 16)
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(smem_u32(dst)), "l"(src),
                 "r"(n)
                 : "memory");
  else
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(smem_u32(dst)), "l"(src),
                 "r"(n)
                 : "memory");
}

// Barrier of all threads of the thread-block cluster.
__device__ __forceinline__ void cluster_barrier() {
  asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;"
               ::: "memory");
}

__device__ __forceinline__ uint32_t cta_rank_in_cluster() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}

__device__ __forceinline__ void prefetch_tmap(const CUtensorMap* tmap) {
  asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(tmap)) : "memory");
}

template <typename T>
__device__ __forceinline__ T from_f32(float v);
template <>
__device__ __forceinline__ float from_f32<float>(float v) { return v; }
template <>
__device__ __forceinline__ __nv_bfloat16 from_f32<__nv_bfloat16>(float v) {
  return __float2bfloat16_rn(v);
}

}  // namespace asd

// LM head fused with the margin-rule statistics (Eq. 1) for fp32 inputs:
// exact fp32 FMA on the CUDA cores (the tensor cores have no fp32-exact mode).
//
// One CTA per (vocabulary range, tile of NT nodes); the ranges are those of the
// tensor-core kernel.  A CTA walks its range in chunks of 64 vocabulary rows and
// 64 hidden elements at a time, W and hidden rows through a ring of cp.async
// stages, each thread accumulating a VP x NP block of logits from 16-byte
// shared-memory reads along the hidden dimension.  The logits of a chunk meet in
// shared memory, where a warp per node row folds them into the row's running
// (max, lowest argmax, sum-exp) and picks the drafted tokens' logits of the
// node's children.  One partial per node and range.
//
// Bound: W traffic up to some 25 nodes, FMA issue beyond; on small shapes the
// latency of the loads, hence all stages in flight at once.  Whole fp32 step of
// 8 nodes, hidden 256, vocabulary 4096, this kernel 34.4 -> 8.8 us (profiled): one
// node per thread and 32 columns, loads between two barriers before.
#include <type_traits>

#include "kernels.h"

namespace asd {
namespace {

constexpr int kThreads = 256;
constexpr int kVt = 64;          // vocabulary rows of a chunk
constexpr int kKc = 64;          // hidden elements of a stage
constexpr int kLd = kKc + 4;     // padded row: 8 rows' 16-byte reads touch all 32 banks

template <int NT>
struct Geom {
  static constexpr int kTn = NT < 16 ? NT : 16;      // thread groups along the nodes
  static constexpr int kTv = kThreads / kTn;         // and along the vocabulary
  static constexpr int kVp = kVt / kTv;              // a thread's vocabulary rows
  static constexpr int kNp = NT / kTn;               // and nodes
  static constexpr int kStages = NT <= 16 ? 4 : 3;
  static constexpr int kCtas = NT <= 32 ? 2 : 1;     // per SM: 82 to 91 KB each, 119 for 64 nodes
  static constexpr int kStageFloats = (kVt + NT) * kLd;
  static constexpr size_t kBytes = sizeof(float) * kStages * kStageFloats;
};

template <int NT>
__global__ void __launch_bounds__(kThreads, Geom<NT>::kCtas) lmhead_f32_kernel(const LmParams p) {
  using G = Geom<NT>;
  extern __shared__ __align__(16) float smem[];
  __shared__ float s_x[NT][kVt + 1];                 // logits of a chunk
  __shared__ float s_m[NT], s_s[NT];                 // running statistics of a row
  __shared__ int s_a[NT];
  pdl_launch_dependents();
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int tn = tid / G::kTv, tv = tid % G::kTv;
  const float* hid = static_cast<const float*>(p.hidden);
  const float* w = static_cast<const float*>(p.w);

  const int ngroups = (p.V + kLmBoxRows - 1) / kLmBoxRows;
  const int tile = blockIdx.x / p.g_lm, range = blockIdx.x - tile * p.g_lm;
  const int vs = lm_range_begin(range, p.g_lm, ngroups) * kLmBoxRows;
  const int ve = min(p.V, lm_range_begin(range + 1, p.g_lm, ngroups) * kLmBoxRows);
  const int node0 = tile * NT;
  const int nk = (p.K + kKc - 1) / kKc;
  const int total = (ve - vs + kVt - 1) / kVt * nk;

  if (tid < NT) {
    s_m[tid] = -INFINITY;
    s_s[tid] = 0.f;
    s_a[tid] = -1;
  }

  // stage `it`: 64 hidden elements of the chunk's W rows, then of the nodes' rows
  auto load = [&](int it) {
    float* st = smem + (it % G::kStages) * G::kStageFloats;
    const int v0 = vs + it / nk * kVt, k0 = it % nk * kKc;
    auto rows = [&](auto step) {   // 4 or 1 elements per copy
      constexpr int kE = decltype(step)::value;
#pragma unroll 4
      for (int i = tid; i < (kVt + NT) * (kKc / kE); i += kThreads) {
        const int r = i / (kKc / kE), k = k0 + i % (kKc / kE) * kE;
        const bool is_w = r < kVt;
        const int row = is_w ? v0 + r : node0 + r - kVt;
        const bool in = k < p.K && row < (is_w ? ve : p.T);
        const float* src = (is_w ? w : hid) + (in ? static_cast<size_t>(row) * p.K + k : 0);
        copy_async<4 * kE>(st + r * kLd + (k - k0), src, in);
      }
    };
    if (p.K % 4 == 0)   // rows start 16-byte aligned
      rows(std::integral_constant<int, 4>());
    else
      rows(std::integral_constant<int, 1>());
  };

#pragma unroll
  for (int s = 0; s < G::kStages - 1; ++s) {
    if (s < total) load(s);
    asm volatile("cp.async.commit_group;" ::: "memory");
  }
  float acc[G::kVp][G::kNp];
  bool waited = false;
  for (int it = 0; it < total; ++it) {
    asm volatile("cp.async.wait_group %0;" ::"n"(G::kStages - 2) : "memory");
    __syncthreads();   // stage `it` has landed, everyone is done with the one before
    if (it + G::kStages - 1 < total) load(it + G::kStages - 1);
    asm volatile("cp.async.commit_group;" ::: "memory");
    if (it % nk == 0) {
#pragma unroll
      for (int a = 0; a < G::kVp; ++a)
#pragma unroll
        for (int b = 0; b < G::kNp; ++b) acc[a][b] = 0.f;
    }
    const float* st = smem + (it % G::kStages) * G::kStageFloats;
    const float* sw = st + tv * kLd;
    const float* sh = st + (kVt + tn) * kLd;
#pragma unroll 4
    for (int k = 0; k < kKc; k += 4) {
      float4 x[G::kVp], y[G::kNp];
#pragma unroll
      for (int a = 0; a < G::kVp; ++a)
        x[a] = *reinterpret_cast<const float4*>(sw + a * G::kTv * kLd + k);
#pragma unroll
      for (int b = 0; b < G::kNp; ++b)
        y[b] = *reinterpret_cast<const float4*>(sh + b * G::kTn * kLd + k);
#pragma unroll
      for (int a = 0; a < G::kVp; ++a)
#pragma unroll
        for (int b = 0; b < G::kNp; ++b) {
          acc[a][b] = fmaf(x[a].x, y[b].x, acc[a][b]);
          acc[a][b] = fmaf(x[a].y, y[b].y, acc[a][b]);
          acc[a][b] = fmaf(x[a].z, y[b].z, acc[a][b]);
          acc[a][b] = fmaf(x[a].w, y[b].w, acc[a][b]);
        }
    }
    if (it % nk != nk - 1) continue;

    // the chunk's logits are complete
    const int v0 = vs + it / nk * kVt, nv = min(kVt, ve - v0);
#pragma unroll
    for (int a = 0; a < G::kVp; ++a)
#pragma unroll
      for (int b = 0; b < G::kNp; ++b) s_x[tn + b * G::kTn][tv + a * G::kTv] = acc[a][b];
    if (!waited) {   // the children lists come from the tree preparation
      pdl_wait();
      waited = true;
    }
    __syncthreads();
    for (int r = warp; r < NT; r += kThreads / 32) {
      const int node = node0 + r;
      if (node >= p.T) break;
      const float x0 = lane < nv ? s_x[r][lane] : -INFINITY;
      const float x1 = lane + 32 < nv ? s_x[r][lane + 32] : -INFINITY;
      float cm = fmaxf(x0, x1);
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) cm = fmaxf(cm, __shfl_xor_sync(0xffffffffu, cm, o));
      float m = s_m[r], sum = s_s[r];
      __syncwarp();
      if (cm > m) {   // uniform over the warp
        const unsigned lo = __ballot_sync(0xffffffffu, x0 == cm);
        const unsigned hi = __ballot_sync(0xffffffffu, x1 == cm);
        if (lane == 0) s_a[r] = v0 + (lo ? __ffs(lo) - 1 : 31 + __ffs(hi));
        sum *= exp2f((m - cm) * kLog2e);
        m = cm;
      }
      const float nm = -m * kLog2e;
      float e0, e1;
      asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(e0) : "f"(fmaf(x0, kLog2e, nm)));
      asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(e1) : "f"(fmaf(x1, kLog2e, nm)));
      e0 += e1;
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) e0 += __shfl_xor_sync(0xffffffffu, e0, o);
      if (lane == 0) {
        s_m[r] = m;
        s_s[r] = sum + e0;
      }
      int cs = p.child_start[node], cnt = p.child_cnt[node];
      if (cs < 0 || cnt < 0 || cnt > p.T || cs > p.T - cnt) cnt = 0;  // malformed tree: no children
      for (int c = lane; c < cnt; c += 32) {
        const int j = p.child_tok[cs + c] - v0;
        const int cid = p.child_id[cs + c];
        if (j >= 0 && j < nv && static_cast<unsigned>(cid) < static_cast<unsigned>(p.T))
          p.l_draft[cid] = s_x[r][j];
      }
    }
  }
  pdl_wait();
  __syncthreads();
  if (tid < NT && node0 + tid < p.T) {
    LmPartial part;
    part.m = s_m[tid];
    part.s = s_s[tid];
    part.a = s_a[tid];
    part.pad = 0;
    p.part[static_cast<size_t>(node0 + tid) * p.g_lm + range] = part;
  }
}

template <int NT>
cudaError_t launch(const LmParams& p, cudaStream_t s) {
  const cudaError_t err = set_smem_attrs(lmhead_f32_kernel<NT>, Geom<NT>::kBytes);
  if (err != cudaSuccess) return err;
  return launch_pdl(lmhead_f32_kernel<NT>, dim3(p.g_lm * ((p.T + NT - 1) / NT)), dim3(kThreads),
                    Geom<NT>::kBytes, s, p);
}

}  // namespace

cudaError_t launch_lmhead_f32(const LmParams& p, cudaStream_t s) {
  // the smallest tile that holds the nodes, up to 64: wider tiles read W less
  // often and feed more FMAs per shared-memory read
  if (p.T <= 8) return launch<8>(p, s);
  if (p.T <= 16) return launch<16>(p, s);
  if (p.T <= 32) return launch<32>(p, s);
  return launch<64>(p, s);
}

}  // namespace asd

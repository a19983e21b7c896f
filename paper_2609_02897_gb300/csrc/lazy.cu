// Lazy LM head (asd_lm_schedule ASD_LM_LAZY_LEVELS).
//
// The verify walk only ever reads the accept verdicts of nodes whose every
// ancestor was accepted, and a verdict needs the parent's LM-head row (Eq. 1
// and the kappa rule), so only the rows of the roots and of nodes reached
// through accepted nodes are needed.  They are computed in passes over W.  A
// pass holds, of every sequence, its frontier (the root, then the accepted
// nodes whose rows are still missing) and, as far as kLazyRows rows of the
// whole pass allow, nodes below the frontier in breadth-first order, ahead of
// their ancestors' verdicts: a pass costs one stream of W whether it computes
// 32 rows or 256, and with the rows below at hand it settles two or three tree
// levels instead of one.  lazy_pass_kernel then merges the rows' partials,
// judges their children, follows the accepted nodes down through the rows of
// the pass, writes what was reached, and lists the next pass.  Rows that were
// computed ahead and not reached leave no trace.
//
// 32 sequences of 128 nodes at tau 1 (contexts of 2048 to 4096): two or three W
// passes by the inputs instead of nine to eleven, the whole step 1784 -> 837 us (the
// same inputs, with three).
//
// The merge of the partials and the kappa rule are the tail kernel's, in the
// same order, so every computed row and verdict is bit-identical to the
// every-row schedule's.  Which sequence's rows come first within a pass depends
// on atomic appends; no result depends on it.
#include "kernels.h"

namespace asd {
namespace {

constexpr int kLazyThreads = 256;
constexpr int kWarps = kLazyThreads / 32;
// Rows of a pass that are computed ahead at most: two 128-row node tiles, which
// the wide LM head takes over one stream of W.
constexpr int kLazyRows = 256;

struct LazySmem {
  int par[kMaxNodes], tok[kMaxNodes];
  int slot[kMaxNodes];     // row of the pass that holds the node, or -1
  float m[kMaxNodes], s[kMaxNodes];
  int a[kMaxNodes];        // the row's merged statistics
  int acc[kMaxNodes];      // judged in this pass: the node's verdict
  int lvl[kMaxNodes];      // next pass: steps below the frontier (0: frontier), or -1
  int list[kMaxNodes];     // next pass: its nodes
  int warp_cnt[kMaxNodes / 32];
  int base;
};

// Copies hidden row `src` (K bf16) to row `dst` of the next pass's buffer,
// one warp, 16 bytes per lane and step (K % 8 == 0).
__device__ __forceinline__ void copy_row(const LazyParams& p, int src, int dst, int lane) {
  const uint4* from = reinterpret_cast<const uint4*>(static_cast<const __nv_bfloat16*>(p.hidden) +
                                                     static_cast<size_t>(src) * p.K);
  uint4* to = reinterpret_cast<uint4*>(static_cast<__nv_bfloat16*>(p.h_next) +
                                       static_cast<size_t>(dst) * p.K);
#pragma unroll 4
  for (int k = lane; k < p.K / 8; k += 32) to[k] = __ldg(from + k);
}

// Rank of this thread among the CTA's first kMaxNodes threads with `flag`, in
// thread order, and their number.  Synchronises the CTA.
__device__ __forceinline__ int rank_of(bool flag, LazySmem& s, int& total) {
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const unsigned bits = __ballot_sync(0xffffffffu, flag);
  if (lane == 0 && warp < kMaxNodes / 32) s.warp_cnt[warp] = __popc(bits);
  __syncthreads();
  int before = __popc(bits & ((1u << lane) - 1u));
  total = 0;
#pragma unroll
  for (int w = 0; w < kMaxNodes / 32; ++w) {
    before += w < warp ? s.warp_cnt[w] : 0;
    total += s.warp_cnt[w];
  }
  __syncthreads();
  return before;
}

// Lists the next pass of the sequence starting at node s0 (n nodes): the
// frontier nodes and, up to `quota` rows in all, nodes below them, level by
// level in index order; nodes at depth max_path or deeper are never reached
// (the caller reports reached ones).  Copies their hidden rows.
__device__ __forceinline__ void list_next(const LazyParams& p, int b, int s0, int n, bool frontier,
                                          int quota, LazySmem& s) {
  const int i = threadIdx.x, warp = i >> 5, lane = i & 31;
  int depth = 0;
  if (i < n)
    for (int u = i; s.par[u] >= 0; u = s.par[u]) ++depth;
  int total = 0;
  int r = rank_of(frontier, s, total);
  if (i < n) s.lvl[i] = frontier ? 0 : -1;
  if (frontier) s.list[r] = i;
  int used = total;
  __syncthreads();
  for (int step = 0; used > 0 && used < quota && step < n; ++step) {
    const bool cand = i > 0 && i < n && s.lvl[i] < 0 && s.slot[i] < 0 && depth < p.levels &&
                      s.lvl[s.par[i]] == step;
    r = rank_of(cand, s, total);
    if (total == 0) break;
    if (cand && used + r < quota) {
      s.lvl[i] = step + 1;
      s.list[used + r] = i;
    }
    used = min(quota, used + total);
    __syncthreads();
  }
  if (i == 0) {
    int base = 0;
    if (used > 0) {
      base = atomicAdd(p.count + p.pass + 1, used);
      atomicAdd(p.active + p.pass + 1, 1);
    }
    p.seq_rows[b] = make_int2(base, used);
    s.base = base;
  }
  __syncthreads();
  const int base = s.base;
  if (i < used) p.rows_next[base + i] = s0 + s.list[i];
  for (int k = warp; k < used; k += kWarps) copy_row(p, s0 + s.list[k], base + k, lane);
}

// The sequence's tree in shared memory; false for a malformed sequence
// (uniform over the CTA).
__device__ __forceinline__ bool load_tree(const LazyParams& p, int b, int& s0, int& n,
                                          LazySmem& s) {
  const int i = threadIdx.x;
  s0 = p.cu_nodes[b];
  n = p.cu_nodes[b + 1] - s0;
  if (p.seq_flags[b] != 0 || n <= 0 || n > kMaxNodes || s0 < 0 || s0 + n > p.T) return false;
  if (i < n) {
    const int par = p.parent[s0 + i];
    s.par[i] = par < i ? max(par, -1) : -1;   // topological (checked by the tree preparation)
    s.tok[i] = p.tokens[s0 + i];
    s.slot[i] = -1;
  }
  __syncthreads();
  return true;
}

// Pass 0: every unflagged sequence's root and nodes below it; the outputs' fills.
// count and active were zeroed on the stream before this kernel.
__global__ void __launch_bounds__(kLazyThreads) lazy_init_kernel(const LazyParams p) {
  __shared__ LazySmem s;
  pdl_launch_dependents();
  pdl_wait();
  const float nan = __int_as_float(0x7fc00000);
  for (int i = blockIdx.x * kLazyThreads + threadIdx.x; i < p.T; i += gridDim.x * kLazyThreads) {
    p.row_max[i] = nan;
    p.row_argmax[i] = -1;
    p.row_lse[i] = nan;
    p.ratio[i] = nan;
    p.accept[i] = 0;
  }
  const int b = blockIdx.x;
  int s0, n;
  if (!load_tree(p, b, s0, n, s)) {   // malformed: no row, the walk skips it
    if (threadIdx.x == 0) p.seq_rows[b] = make_int2(0, 0);
    return;
  }
  list_next(p, b, s0, n, threadIdx.x == 0, kLazyRows / p.B, s);
}

// After the LM head of pass `pass`, one CTA per sequence.
__global__ void __launch_bounds__(kLazyThreads) lazy_pass_kernel(const LazyParams p) {
  __shared__ LazySmem s;
  pdl_launch_dependents();
  pdl_wait();
  const int b = blockIdx.x, i = threadIdx.x, warp = i >> 5, lane = i & 31;
  const int2 mine = p.seq_rows[b];
  if (mine.y <= 0) return;
  int s0, n;
  if (!load_tree(p, b, s0, n, s)) return;
  if (i < n) s.acc[i] = 0;

  // one warp per row
  for (int k = warp; k < mine.y; k += kWarps) {
    const int r = mine.x + k;
    if (r < 0 || r >= p.T) break;
    const int node = p.rows_cur[r] - s0;
    if (node < 0 || node >= n) continue;
    float m, sm;
    int a;
    merge_row(p.part + static_cast<size_t>(r) * p.g_lm, p.g_lm, m, sm, a);
    if (lane == 0) {
      s.slot[node] = r;
      s.m[node] = m;
      s.s[node] = sm;
      s.a[node] = a;
    }
  }
  __syncthreads();

  // the verdicts of the rows' children (Eq. 1 and the kappa rule)
  const int pp = i > 0 && i < n ? s.par[i] : -1;
  const bool judged = pp >= 0 && s.slot[pp] >= 0;
  float d = 0.f;
  if (judged) {
    d = __ldcg(p.l_draft + s0 + i) - s.m[pp];
    s.acc[i] = (s.tok[i] == s.a[pp] || d >= p.ln_tau) ? 1 : 0;
  }
  __syncthreads();
  // a row is reached when every node from it up to a frontier node (one whose
  // parent's row is not of this pass) was accepted
  auto reached = [&](int u) -> bool {
    while (u > 0 && s.slot[s.par[u]] >= 0) {
      if (!s.acc[u]) return false;
      u = s.par[u];
    }
    return true;
  };
  const bool below = judged && reached(pp);   // judged by a reached row
  if (i < n && s.slot[i] >= 0 && reached(i)) {
    p.row_max[s0 + i] = s.m[i];
    p.row_argmax[s0 + i] = s.a[i];
    p.row_lse[s0 + i] = s.m[i] + logf(s.s[i]);
    if (i == 0) p.accept[s0] = 1;
  }
  bool frontier = false;
  if (below) {
    p.ratio[s0 + i] = expf(d);
    p.accept[s0 + i] = static_cast<uint8_t>(s.acc[i]);
    if (s.acc[i] && s.slot[i] < 0) {
      int depth = 0;
      for (int u = i; s.par[u] >= 0; u = s.par[u]) ++depth;
      frontier = depth < p.levels;
      // a reached node one level deeper than max_path allows
      if (!frontier) set_status(p.status, ASD_ERR_SHAPE);
    }
  } else if (judged) {
    p.l_draft[s0 + i] = __int_as_float(0x7fc00000);   // judged ahead, not reached
  }
  list_next(p, b, s0, n, frontier, kLazyRows / max(p.active[p.pass], 1), s);
}

}  // namespace

cudaError_t launch_lazy_init(const LazyParams& p, cudaStream_t s) {
  // rows per pass, then active sequences per pass
  cudaError_t err =
      cudaMemsetAsync(p.count, 0, sizeof(int) * 2 * (static_cast<size_t>(p.levels) + 1), s);
  if (err != cudaSuccess) return err;
  return launch_pdl(lazy_init_kernel, dim3(p.B), dim3(kLazyThreads), 0, s, p);
}

cudaError_t launch_lazy_pass(const LazyParams& p, cudaStream_t s) {
  return launch_pdl(lazy_pass_kernel, dim3(p.B), dim3(kLazyThreads), 0, s, p);
}

}  // namespace asd

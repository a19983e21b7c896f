// Tree preparation: clears the call's status word, validates each draft tree
// (parent array, drafted token range, context length) into it and the
// per-sequence flags, and derives what the LM-head epilogue consumes:
//  - children of every node grouped by parent and sorted by (token, node id),
//    so the LM-head epilogue can pick l_draft = logits[parent, token] while it
//    sweeps the vocabulary in increasing order (Eq. 1 needs the parent row's
//    logit of each drafted token).
// 128 threads per sequence (thread i owns local node i), eight sequences side
// by side in a CTA.  Batches of up to kOneCta sequences take one CTA, which can
// then clear the status word itself, and the call's kernels follow one another
// by programmatic launches from the previous call's on: a memset in front of
// the call cost it about 4 us (headline step 175.5 -> 171.4 us).  Nothing waits
// for the later rounds of such a batch but the LM head's first epilogue, some 10
// us into the call.
#include <algorithm>

#include "kernels.h"

namespace asd {
namespace {

constexpr int kSeqs = 8;       // sequences of one round of a CTA
constexpr int kOneCta = 32;    // sequences that one CTA takes in rounds

struct PrepSmem {
  int par[kMaxNodes], tok[kMaxNodes];
  int cnt[kMaxNodes], start[kMaxNodes], filled[kMaxNodes];
  int list_tok[kMaxNodes], list_id[kMaxNodes];   // children grouped by parent, any order
  int warp_sum[kMaxNodes / 32];
  int bad;
};

__global__ void __launch_bounds__(kSeqs* kMaxNodes) tree_prep_kernel(const PrepParams p) {
  __shared__ PrepSmem smem[kSeqs];

  // every kernel of the call may start from here on: the stream's earlier work
  // is complete
  pdl_wait();
  pdl_launch_dependents();
  const int group = threadIdx.x / kMaxNodes, groups = blockDim.x / kMaxNodes;
  const int i = threadIdx.x % kMaxNodes, lane = threadIdx.x & 31, warp = i >> 5;
  PrepSmem& sm = smem[group];
  if (p.clear_status && threadIdx.x == 0) p.status[0] = p.status[1] = 0;

  for (int b0 = blockIdx.x * groups; b0 < p.B; b0 += gridDim.x * groups) {
    const int b = b0 + group;
    const bool here = b < p.B;
    const int s = here ? p.cu_nodes[b] : 0;
    const int e = here ? p.cu_nodes[b + 1] : 0;
    __syncthreads();   // the status word is clear, the last round is over
    if (i == 0) sm.bad = 0;
    sm.cnt[i] = 0;
    sm.filled[i] = 0;
    bool seq_ok = (s >= 0) && (e > s) && (e <= p.T) && (e - s <= p.max_nodes);
    if (b == 0) seq_ok = seq_ok && (s == 0);
    if (b == p.B - 1) seq_ok = seq_ok && (e == p.T);
    if (here && !seq_ok && i == 0) {
      p.seq_flags[b] = kSeqBadTree;
      set_status(p.status, ASD_ERR_TREE);
    }
    const int n = here && seq_ok ? e - s : 0;
    __syncthreads();

    if (i < n) {
      const int par = p.parent[s + i];
      const int tok = p.tokens ? p.tokens[s + i] : 0;
      const bool ok = (i == 0) ? (par == -1) : (par >= 0 && par < i);
      if (!ok) atomicOr(&sm.bad, kSeqBadTree);
      if (p.tokens && i > 0 && (tok < 0 || tok >= p.vocab)) atomicOr(&sm.bad, kSeqBadToken);
      sm.par[i] = ok ? par : (i == 0 ? -1 : 0);
      sm.tok[i] = tok;
      if (i == 0 && p.ctx_len) {
        const int c = p.ctx_len[b];
        if (c < 0 || c > p.ctx_max) atomicOr(&sm.bad, kSeqBadCtx);
      }
      if (i > 0) atomicAdd(&sm.cnt[sm.par[i]], 1);
    }
    __syncthreads();
    const int bad = sm.bad;
    if (i == 0 && n > 0) {
      p.seq_flags[b] = bad;
      if (bad & kSeqBadTree) set_status(p.status, ASD_ERR_TREE);
      else if (bad & kSeqBadToken) set_status(p.status, ASD_ERR_TOKEN_RANGE);
      else if (bad & kSeqBadCtx) set_status(p.status, ASD_ERR_CTX_RANGE);
    }
    if (!p.tokens) continue;   // an attention call has no use for the children
    const bool tree_ok = !(bad & kSeqBadTree);

    // children of node i at [start, start + cnt) of the sequence's slots
    const int cnt = i < n && tree_ok ? sm.cnt[i] : 0;
    int incl = cnt;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int v = __shfl_up_sync(0xffffffffu, incl, o);
      incl += lane >= o ? v : 0;
    }
    if (lane == 31) sm.warp_sum[warp] = incl;
    __syncthreads();
    int start = incl - cnt;
#pragma unroll
    for (int w = 0; w < kMaxNodes / 32; ++w) start += w < warp ? sm.warp_sum[w] : 0;
    sm.start[i] = start;
    if (i < n) {
      p.child_start[s + i] = s + start;
      p.child_cnt[s + i] = cnt;
      if (p.l_draft) p.l_draft[s + i] = __int_as_float(0x7fc00000);  // NaN
    }
    __syncthreads();
    const int pp = i > 0 && i < n && tree_ok ? sm.par[i] : -1;
    if (pp >= 0) {
      const int at = sm.start[pp] + atomicAdd(&sm.filled[pp], 1);
      sm.list_tok[at] = sm.tok[i];
      sm.list_id[at] = i;
    }
    __syncthreads();
    if (pp >= 0) {   // its place among its siblings by (token, id)
      const int first = sm.start[pp], last = first + sm.cnt[pp], tok = sm.tok[i];
      int rank = 0;
      for (int k = first; k < last; ++k) {
        const int t = sm.list_tok[k];
        rank += (t < tok || (t == tok && sm.list_id[k] < i)) ? 1 : 0;
      }
      p.child_tok[s + first + rank] = tok;
      p.child_id[s + first + rank] = s + i;
    }
  }
}

// The status word of a call whose first large kernel has several CTAs that may
// set it.  A kernel and not a memset: both neighbours overlap it (accepted path
// and commit of 16 sequences, two calls: 16.3 us with memsets, 8.8 with this).
__global__ void clear_status_kernel(int* status) {
  pdl_wait();
  pdl_launch_dependents();
  if (threadIdx.x < 2) status[threadIdx.x] = 0;
}

}  // namespace

cudaError_t launch_clear_status(int* status, cudaStream_t s) {
  return launch_pdl(clear_status_kernel, dim3(1), dim3(32), 0, s, status);
}

cudaError_t launch_tree_prep(PrepParams p, cudaStream_t s) {
  p.clear_status = p.B <= kOneCta ? 1 : 0;
  if (!p.clear_status) {
    const cudaError_t err = launch_clear_status(p.status, s);
    if (err != cudaSuccess) return err;
  }
  const int ctas = p.clear_status ? 1 : (p.B + kSeqs - 1) / kSeqs;
  return launch_pdl(tree_prep_kernel, dim3(ctas), dim3(kMaxNodes * std::min(p.B, kSeqs)), 0, s, p);
}

}  // namespace asd

// Internal interface between the C-ABI layer (asd_api.cu) and the kernels.
#pragma once

#include <cuda.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include <utility>

#include "common.cuh"

namespace asd {

// Launches `kernel` with programmatic stream serialisation, so it may begin
// while the previous kernel in the stream finishes (see pdl_wait()).
template <typename... KArgs, typename... Args>
cudaError_t launch_pdl(void (*kernel)(KArgs...), dim3 grid, dim3 block, size_t smem,
                       cudaStream_t s, Args&&... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kernel, std::forward<Args>(args)...);
}

// Dynamic shared memory limit of `kernel`, and the whole unified L1 as shared
// memory, so that an LM-head CTA and an attention CTA fit on one SM together
// (the default carveout is sized for one kernel's CTAs alone).
template <typename K>
cudaError_t set_smem_attrs(K* kernel, size_t smem) {
  cudaError_t err = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         static_cast<int>(smem));
  if (err != cudaSuccess) return err;
  return cudaFuncSetAttribute(kernel, cudaFuncAttributePreferredSharedMemoryCarveout,
                              cudaSharedmemCarveoutMaxShared);
}

// ------------------------------------------------------------ tree preparation
struct PrepParams {
  const int32_t* parent;
  const int32_t* tokens;    // may be null (attention-only call)
  const int32_t* cu_nodes;
  const int32_t* ctx_len;   // may be null
  int* status;
  int* seq_flags;
  int32_t* child_start;
  int32_t* child_cnt;
  int32_t* child_tok;
  int32_t* child_id;
  float* l_draft;           // may be null; set to NaN
  int B, T, vocab, max_nodes, ctx_max;
  int clear_status;         // set by launch_tree_prep: the kernel clears the status word
};
// Also clears the status word (the call's first launch).
cudaError_t launch_tree_prep(PrepParams p, cudaStream_t s);
cudaError_t launch_clear_status(int* status, cudaStream_t s);

// ------------------------------------------------------------------ attention
struct AttnParams {
  const void* q;            // [T, Hq, D]
  const void* k_cache;      // contiguous [B,Hkv,ctx_max,D] / paged [P,Hkv,ps,D]
  const void* v_cache;
  const void* tree_k;       // [T, Hkv, D]
  const void* tree_v;
  const int32_t* cu_nodes;
  const int32_t* ctx_len;
  const int32_t* page_table;  // [B, ctx_max / ps] or null
  const int32_t* parent;      // local parent ids (ancestor masks are derived in-kernel)
  int* status;
  long long wait_cycles;    // bound of the kernel's waits (0: the default)
  void* out;                // [T, Hq, D]
  int B, T, Hq, Hkv, G, D;
  int ctx_max, page_size, pages_per_seq, num_pages;
  int n_parts, max_nodes;
  float scale_log2;         // log2(e) / sqrt(D)
  int q_tma;                // tensor-core kernels: the query tiles by TMA (tm_q)
  int nsm;                  // SMs of the device
  // bf16 calls of up to 128 nodes that the context lengths decide about: the
  // 32-key tiles up to which the mma.sync kernel takes the call, beyond which the
  // tensor-core kernel does (both are launched and decide alike,
  // attention_takes_mma); -1: no choice.  A step whose cache could hold more keys
  // than the LM head hides (attention_co_tiles_limit), or, with `alone`, a call
  // without an LM head and with several items per SM (attention_alone_rule)
  int co_tiles;
  int alone;
  // calls that the context lengths decide between the two tensor-core forms about:
  // attention_pair_ratio (0: no choice)
  float pair_ratio;
  // one-tile tensor-core kernel: half of P goes to the P.V MMA in two bf16 terms
  // (calls of up to 128 nodes, which another kernel took before)
  int p_two;
  // one-tile tensor-core kernel: partial results of sequences cut into chunks
  long long part_cap;       // rows that part_o / part_ml hold (0: no splitting)
  float* part_o;            // [part_cap][D]: a chunk's unnormalised output row
  float2* part_ml;          // [part_cap]: its reference max (log2 domain) and sum
  int2* plan;               // [B]: first partial row and chunks of a sequence
};
// Whether the mma.sync kernel takes this call (p.co_tiles): in a step the key
// tiles of its longest split, or an even share of all of them per SM, against
// the limit; in a call by itself the mean of the key tiles over the query row
// blocks, and half of the longest.  Every lane of a warp calls it; the answer is
// uniform over the grid.  B <= 128 here; unrolled, so that the loads of all
// sequences are in flight at once.
constexpr int kCoKeys = 32, kCoRows = 64;   // keys per tile, query rows per CTA
struct AloneTiles {   // sums of a call by itself
  int longest, total, blocks;
};
// Sequence of n nodes and context ctx: query row blocks and key tiles.
__device__ __forceinline__ AloneTiles alone_tiles(const AttnParams& p, int n, int ctx) {
  const int rows = (n * p.G + kCoRows - 1) / kCoRows;
  // key tiles cut off far beyond any limit and far from overflow
  const int t = min((ctx + kCoKeys - 1) / kCoKeys + (n + kCoKeys - 1) / kCoKeys, 1 << 12);
  return {t, rows * t, rows};
}
__device__ __forceinline__ bool alone_takes_mma(const AttnParams& p, const AloneTiles& a) {
  return a.longest <= 2 * p.co_tiles && a.total <= p.co_tiles * a.blocks;
}
__device__ __forceinline__ bool attention_takes_mma(const AttnParams& p) {
  int longest = 0, total = 0, blocks = 0;
#pragma unroll
  for (int k = 0; k < kMaxNodes / 32; ++k) {
    const int q = (threadIdx.x & 31) + 32 * k;
    if (q >= p.B) continue;
    const int n = min(max(p.cu_nodes[q + 1] - p.cu_nodes[q], 0), kMaxNodes);
    const int ctx = min(max(p.ctx_len[q], 0), p.ctx_max);
    if (p.alone) {
      const AloneTiles a = alone_tiles(p, n, ctx);
      longest = max(longest, a.longest);
      total += a.total;
      blocks += a.blocks;
      continue;
    }
    const int tree = (n + kCoKeys - 1) / kCoKeys;
    const int tiles = (ctx + kCoKeys - 1) / kCoKeys;
    longest = max(longest, (tiles + p.n_parts - 1) / p.n_parts + tree);
    // a share per SM (rounded up per sequence): far from overflow
    const long long work = static_cast<long long>((n * p.G + kCoRows - 1) / kCoRows) * p.Hkv *
                           (tiles + tree);
    total += static_cast<int>(min((work + p.nsm - 1) / p.nsm, 1LL << 20));
  }
  longest = __reduce_max_sync(0xffffffffu, longest);
  total = __reduce_add_sync(0xffffffffu, total);
  if (!p.alone) return max(longest, total) <= p.co_tiles;
  blocks = __reduce_add_sync(0xffffffffu, blocks);
  return alone_takes_mma(p, {longest, total, blocks});
}
// bf16 path: tensor-core (mma.sync) split-KV kernel fed by TMA; tm_k / tm_v are
// 2D tensor maps over the context cache rows (box 64 columns x
// min(attention_keys_per_tile(), rows per page) rows).
// Both paths merge the splits of a group inside its thread-block cluster.
cudaError_t launch_attention_bf16(const AttnParams& p, const CUtensorMap& tm_k,
                                  const CUtensorMap& tm_v, cudaStream_t s);
cudaError_t launch_attention_f32(const AttnParams& p, cudaStream_t s);
int attention_row_blocks(int max_nodes, int G);
// Key tiles of the busiest SM of the kernel beside the LM head, for contexts of
// the cache's capacity, and up to how many of them it is the faster choice.
long long attention_co_tiles_max(const asd_dims& d, int n_parts, int nsm);
int attention_co_tiles_limit(const asd_dims& d);
// The same limit for a call by itself (-1: the tensor-core kernel takes it), and
// whether the contexts may exceed it, so that both kernels are launched.
struct AloneRule {
  int tiles;
  bool both;
};
AloneRule attention_alone_rule(const asd_dims& d, int total_nodes, int nsm);
int attention_keys_per_tile();   // context keys per K/V tile = TMA box rows
// bf16 path on the 5th-generation tensor cores, where attention has the SMs to
// itself (a step of more than 128 tree nodes, or of fewer with long contexts, or a
// call by itself): one CTA per (128 query rows, sequence x KV head, chunk of the
// keys), and a merge kernel behind it where chunks are possible (p.part_cap > 0).
// tm_k / tm_v: 2D maps over the cache rows with boxes of 64 columns x
// min(kAttnTcKeys, rows per page) rows; tm_tk / tm_tv: 3D maps over the tree
// K/V [T, Hkv, D] with boxes of 64 columns x 1 head x kAttnTcKeys nodes;
// tm_q (with p.q_tma, where attention_q_tma_ok(G)): a 3D map over
// q [T, Hq, D] with boxes of 64 columns x G heads x kAttnTcRows / G nodes.
// pingpong: the two-query-tile form (256 rows per CTA: one tile's MMAs run
// during the other's softmax), chosen by attention_pair_rule() by how many waves of
// CTAs its items make, and about one wave by the context lengths: both forms are
// then launched and decide alike.
constexpr int kAttnTcRows = 128;   // query rows per CTA (per tile of the ping-pong form)
constexpr int kAttnTcKeys = 128;   // keys per tile
size_t attention_tc_smem_bytes(int head_dim, bool pingpong);
enum class PairRule { kOneTile, kPairs, kByContext };
PairRule attention_pair_rule(int batch, int num_kv_heads, int G, int total_nodes, int page_size,
                             int nsm);
float attention_pair_ratio(int page_size);
// Partial rows that the one-tile kernel can use to cut sequences into chunks
// (0: the items of these dims and nodes fill the GPU anyway).
long long attention_split_rows(const asd_dims& d, int total_nodes, int nsm);
bool attention_q_tma_ok(int G);   // G divides kAttnTcRows: a query box of whole nodes
cudaError_t launch_attention_tc(const AttnParams& p, const CUtensorMap& tm_k,
                                const CUtensorMap& tm_v, const CUtensorMap& tm_tk,
                                const CUtensorMap& tm_tv, const CUtensorMap& tm_q, bool pingpong,
                                cudaStream_t s);

// -------------------------------------------------------------------- LM head
struct LmParams {
  const void* hidden;       // [T, K]
  const void* w;            // [V, K]
  const int32_t* child_start;
  const int32_t* child_cnt;
  const int32_t* child_tok;
  const int32_t* child_id;
  LmPartial* part;          // [T][g_lm]
  float* l_draft;           // [T]
  int* status;
  long long wait_cycles;    // bound of the kernel's waits (0: the default)
  int T, K, V, g_lm;
  int a_rows;               // node rows per hidden-state TMA box: min(128, T rounded to 8);
                            // accumulator rows past it belong to no node
  const uint8_t* w_packed;  // W in the packed streaming layout, or null ([V, K] rows via TMA)
  // Lazy LM head (one pass per launch): the number of hidden rows is
  // read from *t_dev (at most T), written by the previous kernel; row r
  // belongs to node row_node[r].  Both null: T rows, row r = node r.
  const int* t_dev;
  const int32_t* row_node;
  // 1: W is memory of the launching device, the only one this process sees, so the
  // wide kernel may run in clusters of two that multicast W between their SMs (set
  // by the host)
  int w_local;
};
constexpr int kLmStages = 3;       // 3 x 48 KB (a_rows <= 64): room for an attention CTA
constexpr int kLmTileN = 128;      // vocabulary rows per MMA tile
constexpr int kLmBoxRows = 32;     // vocabulary rows per range group (and per small TMA box)
size_t lmhead_tc_smem_bytes(int a_rows);
// Tensor maps of the bf16 LM head (128-byte swizzle, 64-element inner boxes):
// h: hidden [T, K], box a_rows rows; w64 / w32: W [V, K], boxes of 64 and 32
// rows (unused with a packed weight).
struct LmMaps {
  CUtensorMap h, w64, w32;
};
// bf16 path: tcgen05/TMEM GEMM with the fused max/argmax/sum-exp/l_draft epilogue.
cudaError_t launch_lmhead_bf16(const LmParams& p, const LmMaps& maps, cudaStream_t s);
// Which bf16 LM-head kernel launch_lmhead_bf16 runs for these parameters
// (asd_lm_head_variant values: 1 weight-streaming, 2 wide, 3 wide in clusters).
int lmhead_bf16_variant(const LmParams& p);

// Vocabulary ranges of the LM head: range c of g covers the 32-row groups
// [c * ngroups / g, (c + 1) * ngroups / g); each range is cut into tiles of
// up to kLmTileN rows starting at its first group.
__host__ __device__ inline int lm_range_begin(int c, int g, int ngroups) {
  return static_cast<int>(static_cast<long long>(c) * ngroups / g);
}
int lm_ranges(int vocab, int nsm);

// Packed streaming layout of the LM-head weight (asd_pack_lm_head): a header
// of kLmPackHeader bytes, then for every tile in range order and every
// k-block kb, the tile's rows (ng whole 32-row groups, zeros past V and past
// K) x 128 bytes with the 128-byte swizzle applied (16-byte chunk c of row r
// at chunk c ^ (r & 7)).  The block of a tile starting at group g0 for
// k-block kb begins at byte kLmPackHeader + 4096 * (nkb * g0 + kb * ng), so a
// stage's two k-blocks are one contiguous run.
constexpr uint32_t kLmPackMagic = 0x57445341u;  // "ASDW"
constexpr uint32_t kLmPackVersion = 1;
constexpr int kLmPackHeader = 256;
struct LmPackHeader {
  uint32_t magic, version;
  int32_t vocab, hidden, ranges;
};
size_t lm_packed_bytes(int vocab, int hidden);
cudaError_t launch_lm_pack(const void* w, void* w_packed, int vocab, int hidden, int ranges,
                           cudaStream_t s);
cudaError_t launch_lmhead_f32(const LmParams& p, cudaStream_t s);

// --------------------------------------- finalize / accepted path / K/V commit
enum TailMode : int { kTailFinalize = 1, kTailWalk = 2, kTailCompact = 4 };
struct TailParams {
  int mode;
  const int32_t* parent;
  const int32_t* tokens;
  const int32_t* cu_nodes;
  const int* seq_flags;       // from tree preparation, or null
  // finalize
  const LmPartial* part;
  int g_lm;
  float ln_tau;
  float* row_max;
  int32_t* row_argmax;        // written by finalize, read by walk
  float* row_lse;
  const float* l_draft;
  float* ratio;               // written by finalize; read by the greedy walks otherwise
  uint8_t* accept;            // written by finalize, read by walk
  // walk
  int32_t* path;              // [B, max_path]
  int32_t* path_len;
  int32_t* bonus;
  int32_t* n_promoted;
  // compact
  const void* tree_k;
  const void* tree_v;
  void* k_cache;
  void* v_cache;
  const int32_t* ctx_len;
  const int32_t* page_table;
  int32_t* ctx_len_out;
  int* status;
  int rule;                   // accepted-path reading (asd_accept_rule)
  int clear_status;           // set by launch_tail_alone: the grid is one cluster, whose
                              // first CTA clears the status word
  int B, T, Hkv, D, elem_bytes, max_nodes, max_path;
  int ctx_max, page_size, pages_per_seq, num_pages;
};
cudaError_t launch_tail(const TailParams& p, cudaStream_t s);
// The same as a call's only work (walk or commit): it also clears the status word.
cudaError_t launch_tail_alone(TailParams p, cudaStream_t s);

// Lazy LM head: rows are computed for the roots and for nodes reached through
// accepted nodes only, in passes over W (lazy.cu).
struct LazyParams {
  const int32_t* parent;
  const int32_t* tokens;
  const int32_t* cu_nodes;
  const int* seq_flags;
  const void* hidden;         // [T, K] bf16
  const LmPartial* part;      // [rows of the pass][g_lm]
  float* row_max;
  int32_t* row_argmax;
  float* row_lse;
  float* l_draft;
  float* ratio;
  uint8_t* accept;
  int* count;                 // [levels + 1] rows per pass
  int* active;                // [levels + 1] sequences with rows per pass (behind count)
  int2* seq_rows;             // [B] first row of the pass and rows of a sequence
  const int32_t* rows_cur;    // node ids of this pass's rows
  int32_t* rows_next;
  void* h_next;               // [cap, K] bf16: hidden rows of the next pass
  int* status;
  int B, T, K, g_lm, pass;
  int levels;                 // max_path: passes at most, and levels of a tree
  float ln_tau;
};
cudaError_t launch_lazy_init(const LazyParams& p, cudaStream_t s);
cudaError_t launch_lazy_pass(const LazyParams& p, cudaStream_t s);

}  // namespace asd

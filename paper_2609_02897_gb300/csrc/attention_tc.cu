// Tree attention (Sec. 2 "Verify": the target scores every drafted node in
// one forward pass) on the 5th-generation tensor cores, where the attention
// kernel has the SMs to itself: a step of more than 128 tree nodes (the LM head
// then takes most of an SM's shared memory and runs first); a smaller one whose
// contexts are longer than its LM head hides, behind the LM head (decided on the
// device, AttnParams::co_tiles); and an attention call by itself, unless many
// short sequences are better off with the mma.sync kernel.  bf16 in, fp32
// accumulate.
//
// Measured, a whole asd_tree_attention call: one sequence, 8 nodes, context
// 32768 in a cache of 40960 slots 186.5 -> 32.3 us (134 MB of K/V; the
// mma.sync kernel in 8 splits of the cache's capacity before), 4 sequences of
// 60 nodes, contexts 901 to 3625 41.0 -> 24.8 us (unsplit before).
//
// Work item (one CTA): 128 query rows of one (sequence, KV head) pair and a
// chunk of its keys: the whole context, or, when the items would leave SMs
// idle, one of up to kMaxChunks equal runs of key tiles.  The chunk length is
// one for the whole step and is chosen in-kernel from the context lengths
// (chunk_length: the host knows the cache's capacity only, which says little
// about them), so a cache sized for many times the context splits like a tight
// one.  A chunk leaves its unnormalised O, reference max and row sum in the
// workspace, and attn_merge_kernel, one warp or four per query row, combines
// them.  The CTAs take the chunks in decreasing order of work, so the longest
// start first.  The rows of a pair are its N nodes times the G query heads that
// share the KV head, node-major (row r -> node r / G, head g*G + r % G); row r
// lives in TMEM lane r.  Keys come in tiles of 128, K and V through TMA rings of
// their own (128-byte swizzle; paged caches one box per page; the tree K/V
// through a 3D map over [T, Hkv, D]), so a K slot is refilled as soon as its S
// MMA is done rather than after the tile's P.V; the last tile of a pair holds
// its tree keys, where a node sees only its ancestors (bitmasks derived here
// from the parent array).
//
//   Q             loaded once into shared memory by one TMA (G dividing 128:
//                 boxes of G heads x 128/G nodes), else by the softmax warps
//   S = Q . K^T   tcgen05.mma, Q and K K-major in shared memory
//   P = exp2(S*c - m), per row by the thread that owns the row, written back
//                 over the tile's S columns as bf16 pairs
//   O += P . V    tcgen05.mma, A (= P) from TMEM, V MN-major straight from its
//                 TMA tile, O in TMEM for the whole item
//
// The softmax keeps a per-row reference max m and rescales O only when the
// running max exceeds m by more than 2^8 in the exp2 domain (P then stays
// below 2^8 and the result equals that with the exact running max, but for the
// rounding of P: exp2_tile_two).  S/P is triple-buffered: S of tile t+1 is ready
// when the softmax finishes tile t, and S of tile t+2 does not wait for O += P V of
// tile t (with two buffers it did, which put the P.V, its commit and the next S on
// the softmax's path every second tile).
//
// TMEM (512 columns): O [0, D), S/P [128, 256), [256, 384), [384, 512).
// Shared memory: Q, a 3-stage K ring and a V ring (160 KB of rings for D =
// 128).
// Warp roles (384 threads): warp 0 K producer, warp 1 issuer of the S MMAs,
// warps 2-9 softmax and epilogue, two per TMEM lane quarter, each on one half
// of every tile's keys, warp 10 TMEM allocator and issuer of the P.V MMAs,
// warp 11 V producer.
#include <algorithm>

#include "kernels.h"
#include "tc.cuh"

namespace asd {
namespace {

constexpr int kRows = kAttnTcRows;   // query rows per CTA = TMEM lanes
constexpr int kKeys = kAttnTcKeys;   // keys per tile
constexpr int kThreads = 384;   // twelve warps (the roles above; the ping-pong form's below)
constexpr int kSoftmaxThreads = 256;   // eight warps: two per TMEM lane quarter
constexpr float kRescaleLog2 = 8.f;
constexpr uint32_t kTmemCols = 512;
constexpr int kSBufs = 3;              // S/P buffers in TMEM
constexpr uint32_t kSCol0 = 128;       // S/P buffer b at columns [128 (b + 1), 128 (b + 2))

// Dynamic shared memory, 1024-byte aligned: Q [D/64][128 rows][128 B], the K
// ring [stage][D/64][128 keys][128 B], then the V ring likewise (two stages
// for D = 128, where a third does not fit beside Q).
template <int D>
struct TcGeom {
  static constexpr int kNH = D / 64;
  static constexpr int kTileBytes = kNH * kKeys * 128;   // one K or one V tile
  static constexpr int kKStages = 3;
  static constexpr int kVStages = D == 64 ? 3 : 2;
  static constexpr int kQOff = 0;
  static constexpr int kKOff = kNH * kRows * 128;
  static constexpr int kVOff = kKOff + kKStages * kTileBytes;
  static constexpr int kBytes = kVOff + kVStages * kTileBytes;
};

// Named barrier 1 of the eight softmax warps.
__device__ __forceinline__ void softmax_sync() {
  asm volatile("bar.sync 1, %0;" ::"n"(kSoftmaxThreads) : "memory");
}

// AND of `v` over the eight softmax warps (named barrier 1); uniform result.
__device__ __forceinline__ bool softmax_all(bool v) {
  uint32_t r;
  asm volatile(
      "{\n\t.reg .pred p, q;\n\t"
      "setp.ne.u32 q, %1, 0;\n\t"
      "barrier.cta.red.and.pred p, 1, %2, q;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(r)
      : "r"(v ? 1u : 0u), "n"(kSoftmaxThreads)
      : "memory");
  return r != 0;
}

// OR of `v` over the eight softmax warps (named barrier 1); uniform result.
__device__ __forceinline__ bool softmax_any(bool v) {
  uint32_t r;
  asm volatile(
      "{\n\t.reg .pred p, q;\n\t"
      "setp.ne.u32 q, %1, 0;\n\t"
      "barrier.cta.red.or.pred p, 1, %2, q;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(r)
      : "r"(v ? 1u : 0u), "n"(kSoftmaxThreads)
      : "memory");
  return r != 0;
}

// Every lane polls (bounded by `budget` cycles); the result is lane 0's,
// uniform over the warp.
__device__ __forceinline__ bool wait_all(uint64_t* bar, uint32_t parity, long long budget) {
  return __shfl_sync(0xffffffffu, mbar_wait(smem_u32(bar), parity, budget) ? 1 : 0, 0) != 0;
}

__device__ __forceinline__ bool aborted_warp(volatile int* s_abort) {
  return __shfl_sync(0xffffffffu, *s_abort, 0) != 0;
}

// Whether a call of about one wave of pairs of query tiles is the ping-pong form's
// (p.pair_ratio > 0: both forms are launched and decide alike).  Its pairs take 1.8
// us a key tile together at D = 128 (1.5 at D = 64), and the call the longest pair's
// time.  Of the one-tile form's items, one to two waves in decreasing order, an SM's
// second starts as its first ends: the call takes the longest item, or 1.15 times
// an even share of all, at 1.0 us a key tile (1.2 with pages of 32 tokens or more,
// 1.4 with smaller ones; D = 64 0.85 and 1.1), and 4 us more than the pairs for the
// second start.  The idle form's grid costs the call some 3 us.  One tile / pairs by
// themselves, 8 KV heads, G = 4:
//   16 x 64 nodes, context 2048 47.7 / 41.1 us, pages of 16 60.7 / 42.3, of 32 53.7 /
//     42.1, D = 64 41.9 / 33.3; contexts 300-1000 30.4 / 26.0
//   16 x 64, contexts 1000-6000 59.1 / 78.0, pages of 16 100.2 / 94.6, of 32 81.2 /
//     95.8, D = 64 53.1 / 78.3; 9 x 128 67.7 / 89.3, D = 64 76.3 / 74.7
// Every lane of a warp calls it; the answer is uniform over the grid.
constexpr int kPairSeqs = 192;   // sequences at most (one pair each and KV head, one wave)
__device__ __forceinline__ bool attention_takes_pairs(const AttnParams& p) {
  int longest = 0, pairs = 0, work = 0;
#pragma unroll
  for (int k = 0; k < kPairSeqs / 32; ++k) {   // unrolled: all loads in flight at once
    const int q = (threadIdx.x & 31) + 32 * k;
    if (q >= p.B) continue;
    const int n = min(max(p.cu_nodes[q + 1] - p.cu_nodes[q], 0), kMaxNodes);
    const int ctx = min(max(p.ctx_len[q], 0), p.ctx_max);
    const int t = n > 0 ? (ctx + kKeys - 1) / kKeys + 1 : 0, r = n * p.G;
    longest = max(longest, t);
    pairs += (r + 2 * kRows - 1) / (2 * kRows) * p.Hkv;
    work += (r + kRows - 1) / kRows * p.Hkv * min(t, 1 << 20);
  }
  longest = __reduce_max_sync(0xffffffffu, longest);
  pairs = __reduce_add_sync(0xffffffffu, pairs);
  work = __reduce_add_sync(0xffffffffu, work);
  const float one = fmaxf(static_cast<float>(longest), 1.15f * static_cast<float>(work) / p.nsm);
  return pairs <= p.nsm && static_cast<float>(longest) <= p.pair_ratio * one + 3.f;
}

struct Item {
  int b, g, s0, n, r0, nrows, R;
  int key_base;              // first context key of the chunk (a multiple of kKeys)
  int ctx;                   // context length past key_base
  int nctx, ntree, ntiles;   // context, tree and all key tiles of the chunk
  int chunks, chunk, part0;  // chunks of the sequence, this one, the sequence's partial rows
};

constexpr int kOrderMax = 256;   // batches ordered by work in-kernel (larger ones: index order)

// Forms of the kernels compiled apart, since code that a call skips still costs it
// up to 1 %: calls of up to 128 nodes hand half of P over in two bf16 terms and may
// be the mma.sync kernel's (AttnParams::p_two, co_tiles); calls of about one wave of
// pairs go to either form by their context lengths (pair_ratio).
enum Mode { kPlain, kTwoTerms, kByContext };

constexpr int kMaxChunks = 32;   // chunks per sequence: one lane of the merging warp each
constexpr int kMergeOverhead = 3;   // cost of the merge in key tiles of ~1 us

// Shared-memory scratch of make_item, one entry per sequence.
struct PlanSmem {
  int s0[kOrderMax], n[kOrderMax], ctx[kOrderMax];   // first node, nodes, context length
  int tiles[kOrderMax];    // key tiles (0: no query rows)
  int items[kOrderMax];    // query row blocks x KV heads
  int key[kOrderMax];      // key tiles of the longest chunk
  int2 order[kOrderMax];   // larger first: by key, then by index; the sequence's CTAs
  int part[kOrderMax];     // partial rows (0: one chunk)
  int chunks[kOrderMax];
  int cut_ctas[kMaxChunks];   // CTAs and partial rows when the longest sequence is
  int cut_part[kMaxChunks];   // cut into 1, 2, ... chunks
  AloneTiles alone[kMaxNodes / 32];   // a call by itself: sums over 32 sequences each
  int past;                // items in all where they are more than the grid's CTAs, else 0
  int seq, first, part0;   // the sequence of this CTA, its first CTA and partial row
};

// ceil(t / len) and a / b for quotients up to about 2^12, from an approximate
// reciprocal (the estimate is then off by one at most).
__device__ __forceinline__ int ceil_div_est(int t, int len, float inv) {
  int c = static_cast<int>(static_cast<float>(t) * inv);
  c -= (c - 1) * len >= t ? 1 : 0;
  c += c * len < t ? 1 : 0;
  c += c * len < t ? 1 : 0;
  return c;
}
__device__ __forceinline__ int div_est(int a, int b) {
  int q = static_cast<int>(static_cast<float>(a) * __frcp_rn(static_cast<float>(b)));
  q -= q * b > a ? 1 : 0;
  q += (q + 1) * b <= a ? 1 : 0;
  return q;
}

// Sort key of a sequence: the length of its chunks, then its index, ascending.
__device__ __forceinline__ int order_key(int tiles, int q) {
  static_assert(kOrderMax <= 512, "9 bits of index");
  return (min(tiles, 1 << 21) << 9) | (511 - q);
}

// Key tiles per chunk.  Lane k weighs cutting the longest sequence into k + 1
// chunks (and the others into chunks no longer than its), each warp adding up
// some of the sequences.  The chunks run at once, one CTA per SM (a second wave
// would pay a CTA's overhead again), so a step takes its longest chunk: the
// shortest length that fits, unless the merge costs more than the cut saves.
// Every thread of the CTA calls it (it synchronises the CTA) and returns the
// same length; s.cut_* are zero on entry.  It stands between the start of every
// CTA and its first copy: 1.0 us (1.9 with three candidates per warp, a lane per
// sequence).
__device__ __forceinline__ int chunk_length(const AttnParams& p, PlanSmem& s) {
  static_assert(kMaxChunks == 32, "a lane per candidate");
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  int longest = 1, items = 0;
  for (int q = lane; q < p.B; q += 32) {
    longest = max(longest, s.tiles[q]);
    items += s.items[q];
  }
  longest = __reduce_max_sync(0xffffffffu, longest);
  items = __reduce_add_sync(0xffffffffu, items);
  if (items == 0 || items > p.nsm) return longest;   // uniform over the CTA
  const int len = (longest + lane) / (lane + 1);
  const float inv = __frcp_rn(static_cast<float>(len));
  int ctas = 0, part = 0;
  for (int q = warp; q < p.B; q += kThreads / 32) {
    const int c = ceil_div_est(s.tiles[q], len, inv);
    ctas += s.items[q] * c;
    part += c > 1 ? s.n[q] * p.Hq * c : 0;
  }
  if (warp < p.B) {
    atomicAdd(&s.cut_ctas[lane], ctas);
    atomicAdd(&s.cut_part[lane], part);
  }
  __syncthreads();
  ctas = s.cut_ctas[lane];
  part = s.cut_part[lane];
  // one chunk each (lane 0) is always possible
  const unsigned cost = lane > 0 && (part > p.part_cap || ctas > p.nsm)
                            ? 0xffffffffu
                            : static_cast<unsigned>(len + (part > 0 ? kMergeOverhead : 0));
  const unsigned best = __reduce_min_sync(0xffffffffu, cost);
  return __shfl_sync(0xffffffffu, len, __ffs(__ballot_sync(0xffffffffu, cost == best)) - 1);
}

// The chunk of CTA blockIdx.x: sequences in decreasing order of their chunks'
// length (ties by index), within one its KV heads, its chunks, its blocks of
// query rows (which read the same keys) innermost.  The hardware dispatches
// CTAs in blockIdx order, so the longest run first and the short ones fill the
// last wave.  False when the CTA has none.  Every thread of the CTA calls it (it
// synchronises the CTA).
template <int ROWS, int MODE>
__device__ __forceinline__ bool make_item(const AttnParams& p, Item& it, PlanSmem& s) {
  const int idx = blockIdx.x;
  int local, ctx, longest;   // longest: key tiles of the sequence's longest chunk
  if (ROWS == kRows && threadIdx.x == 0) s.past = 0;
  if (p.B > kOrderMax) {   // index order, unsplit
    const int rbmax = (p.max_nodes * p.G + ROWS - 1) / ROWS;
    it.b = idx / (rbmax * p.Hkv);
    if (it.b >= p.B) {
      __syncthreads();
      return false;
    }
    local = idx - it.b * rbmax * p.Hkv;
    it.g = local / rbmax;
    it.r0 = (local - it.g * rbmax) * ROWS;
    it.chunks = 1;
    it.chunk = 0;
    it.part0 = 0;
    it.s0 = p.cu_nodes[it.b];
    it.n = p.cu_nodes[it.b + 1] - it.s0;
    ctx = min(max(p.ctx_len[it.b], 0), p.ctx_max);
    longest = 0x3fffffff;
    __syncthreads();
  } else {
    // sequence extents and context lengths are caller inputs (the tree
    // preparation reports bad ones): a malformed sequence gets no CTA
    if (threadIdx.x == 0) s.seq = -1;
    if (threadIdx.x < kMaxChunks) s.cut_ctas[threadIdx.x] = s.cut_part[threadIdx.x] = 0;
    for (int q = threadIdx.x; q < p.B; q += blockDim.x) {
      const int s0 = p.cu_nodes[q], n = p.cu_nodes[q + 1] - s0;
      const int c = min(max(p.ctx_len[q], 0), p.ctx_max);
      const bool okq = n > 0 && n <= kMaxNodes && s0 >= 0 && s0 + n <= p.T;
      s.s0[q] = s0;
      s.n[q] = n;
      s.ctx[q] = c;
      s.tiles[q] = okq ? (c + kKeys - 1) / kKeys + (n + kKeys - 1) / kKeys : 0;
      s.items[q] = okq ? (n * p.G + ROWS - 1) / ROWS * p.Hkv : 0;
      s.key[q] = s.tiles[q];
      s.part[q] = 0;
      s.chunks[q] = 1;
      s.order[q] = make_int2(order_key(s.tiles[q], q), s.items[q]);
    }
    // B <= 128 here: a sequence per thread
    const bool choice = MODE == kTwoTerms && p.alone && p.co_tiles >= 0;
    if (choice && threadIdx.x < kMaxNodes) {
      const int q = threadIdx.x;
      AloneTiles a{0, 0, 0};
      if (q < p.B) a = alone_tiles(p, min(max(s.n[q], 0), kMaxNodes), s.ctx[q]);
      a = {__reduce_max_sync(0xffffffffu, a.longest), __reduce_add_sync(0xffffffffu, a.total),
           __reduce_add_sync(0xffffffffu, a.blocks)};
      if ((q & 31) == 0) s.alone[q >> 5] = a;
    }
    __syncthreads();
    // The mma.sync kernel's call: decided here, where the extents are at hand,
    // since in front of every CTA's set-up (attention_takes_mma) it cost the several
    // waves of such a call 1.3 us each.
    if (choice) {
      AloneTiles a = s.alone[0];
#pragma unroll
      for (int w = 1; w < kMaxNodes / 32; ++w)
        a = {max(a.longest, s.alone[w].longest), a.total + s.alone[w].total,
             a.blocks + s.alone[w].blocks};
      if (alone_takes_mma(p, a)) return false;
    }
    if (p.part_cap > 0) {
      const int len = chunk_length(p, s);
      const float inv = __frcp_rn(static_cast<float>(len));
      for (int q = threadIdx.x; q < p.B; q += blockDim.x) {
        const int t = s.tiles[q], c = ceil_div_est(t, len, inv);
        s.chunks[q] = c;
        if (c > 1) {
          s.key[q] = (t + c - 1) / c;
          s.part[q] = s.n[q] * p.Hq * c;
          s.order[q] = make_int2(order_key(s.key[q], q), s.items[q] * c);
        }
      }
      __syncthreads();
    }
    // the CTAs (and partial rows) of the sequences before each one, a thread per
    // sequence: on the way of every CTA's first copy (a warp per sequence, its
    // lanes over the others, was slower: 64 sequences of 8 nodes at contexts 300
    // to 1000, 3.4 waves of CTAs, 68.5 us against 61.2)
    for (int q = threadIdx.x; q < p.B; q += blockDim.x) {
      const int2 mine = s.order[q];
      int first = 0, part = 0;
#pragma unroll 8
      for (int j = 0; j < p.B; ++j) {
        const int2 o = s.order[j];
        first += o.x > mine.x ? o.y : 0;
      }
      if (ROWS == kRows && first + mine.y > static_cast<int>(gridDim.x))
        atomicMax(&s.past, first + mine.y);
      if (idx < first || idx >= first + mine.y) continue;
      if (p.part_cap > 0) {
        for (int j = 0; j < p.B; ++j) part += s.order[j].x > mine.x ? s.part[j] : 0;
        if (idx == first) p.plan[q] = make_int2(part, s.chunks[q]);
      }
      s.seq = q;
      s.first = first;
      s.part0 = part;
    }
    __syncthreads();
    it.b = s.seq;
    if (it.b < 0) return false;
    it.s0 = s.s0[it.b];
    it.n = s.n[it.b];
    ctx = s.ctx[it.b];
    it.chunks = s.chunks[it.b];
    it.part0 = s.part0;
    const int rb = (it.n * p.G + ROWS - 1) / ROWS;
    local = idx - s.first;
    const int gz = div_est(local, rb);
    it.r0 = (local - gz * rb) * ROWS;
    it.g = div_est(gz, it.chunks);
    it.chunk = gz - it.g * it.chunks;
    longest = s.key[it.b];
  }
  it.R = it.n * p.G;
  if (it.n <= 0 || it.n > kMaxNodes || it.s0 < 0 || it.s0 + it.n > p.T || it.r0 >= it.R)
    return false;
  it.nrows = min(ROWS, it.R - it.r0);
  const int nctx = (ctx + kKeys - 1) / kKeys, all = nctx + (it.n + kKeys - 1) / kKeys;
  // of the context's tiles, then the tree's, the first chunks take one more
  // than the others where they do not divide
  const int few = it.chunks == 1 ? all : (longest * it.chunks == all ? longest : longest - 1);
  const int more = all - few * it.chunks;
  const int t0 = it.chunk * few + min(it.chunk, more);
  const int t1 = t0 + few + (it.chunk < more ? 1 : 0);
  it.ntiles = t1 - t0;
  it.nctx = min(t1, nctx) - t0;
  it.ntree = it.ntiles - it.nctx;
  it.key_base = t0 * kKeys;
  it.ctx = ctx - it.key_base;
  return true;
}

// One-tile form: the items past the grid, which has a CTA for every item of
// sequences that do not overlap.  A batch whose cu_nodes run backwards (reported as
// ASD_ERR_TREE) can make more, and its well-formed sequences keep their outputs.
// Plain loops over the keys, a warp per query row, by the eight softmax warps (tid:
// thread among them) of every CTA when it is done.  (In the ping-pong form the
// branch cost the tile loop 2 %; its grid covers every item instead.)
template <int D>
__device__ __forceinline__ void items_past_grid(const AttnParams& p, PlanSmem& s, int tid) {
  constexpr int kV = D / 32;   // a lane's columns
  const int lane = tid & 31;
  const __nv_bfloat16* kc = static_cast<const __nv_bfloat16*>(p.k_cache);
  const __nv_bfloat16* vc = static_cast<const __nv_bfloat16*>(p.v_cache);
  for (int idx = gridDim.x + blockIdx.x; idx < s.past; idx += gridDim.x) {
    softmax_sync();   // everyone is done with the last item's sequence
    for (int q = tid; q < p.B; q += kSoftmaxThreads) {
      int first = 0;
      for (int j = 0; j < p.B; ++j) first += s.order[j].x > s.order[q].x ? s.order[j].y : 0;
      if (idx < first || idx >= first + s.order[q].y) continue;
      s.seq = q;
      s.first = first;
      if (idx == first && p.part_cap > 0) p.plan[q] = make_int2(0, 1);   // nothing to merge
    }
    softmax_sync();
    const int b = s.seq, s0 = s.s0[b], R = s.n[b] * p.G, rb = (R + kRows - 1) / kRows;
    const int g = (idx - s.first) / rb, r0 = (idx - s.first - g * rb) * kRows;
    for (int r = r0 + (tid >> 5); r < min(r0 + kRows, R); r += kSoftmaxThreads / 32) {
      const int node = r / p.G;
      const size_t row = static_cast<size_t>(s0 + node) * p.Hq + g * p.G + (r - node * p.G);
      const __nv_bfloat16* qr = static_cast<const __nv_bfloat16*>(p.q) + row * D;
      __nv_bfloat16* out = static_cast<__nv_bfloat16*>(p.out) + row * D;
      float q[kV], o[kV], m = -INFINITY, l = 0.f;
#pragma unroll
      for (int k = 0; k < kV; ++k) {
        q[k] = __bfloat162float(qr[lane * kV + k]) * p.scale_log2;
        o[k] = 0.f;
      }
      auto key = [&](const __nv_bfloat16* kr, const __nv_bfloat16* vr) {
        float x = 0.f;
#pragma unroll
        for (int k = 0; k < kV; ++k) x = fmaf(q[k], __bfloat162float(kr[lane * kV + k]), x);
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) x += __shfl_xor_sync(0xffffffffu, x, off);
        const float mn = fmaxf(m, x);
        const float al = m == -INFINITY ? 0.f : exp2f(m - mn);
        const float pe = x == -INFINITY ? 0.f : exp2f(x - mn);
        l = l * al + pe;
#pragma unroll
        for (int k = 0; k < kV; ++k) o[k] = fmaf(pe, __bfloat162float(vr[lane * kV + k]), o[k] * al);
        m = mn;
      };
      for (int j = 0; j < s.ctx[b]; ++j) {
        size_t at = (static_cast<size_t>(b) * p.Hkv + g) * p.ctx_max + j;
        if (p.page_size) {
          const int page = p.page_table[static_cast<size_t>(b) * p.pages_per_seq + j / p.page_size];
          if (page < 0 || page >= p.num_pages) {
            set_status(p.status, ASD_ERR_CTX_RANGE);
            continue;
          }
          at = (static_cast<size_t>(page) * p.Hkv + g) * p.page_size + j % p.page_size;
        }
        key(kc + at * D, vc + at * D);
      }
      for (int u = node; u >= 0;) {   // the node and its ancestors
        const size_t at = (static_cast<size_t>(s0 + u) * p.Hkv + g) * D;
        key(static_cast<const __nv_bfloat16*>(p.tree_k) + at,
            static_cast<const __nv_bfloat16*>(p.tree_v) + at);
        const int pu = p.parent[s0 + u];
        u = pu < u ? pu : -1;
      }
      const float inv = l > 0.f ? 1.f / l : 0.f;
#pragma unroll
      for (int k = 0; k < kV; ++k)
        out[lane * kV + k] = __float2bfloat16_rn(o[k] * inv);
    }
  }
}

__device__ __forceinline__ size_t grow_of(const AttnParams& p, const Item& it, int r) {
  const int rr = it.r0 + r;
  const int i = rr / p.G;
  return static_cast<size_t>(it.s0 + i) * p.Hq + it.g * p.G + (rr - i * p.G);
}

constexpr int kPageChunk = 512;   // page-table entries staged in shared memory

// Issues one K (which = 0) or V (which = 1) tile t into `dst` (producer lane 0;
// contiguous cache or tree keys).
template <int D>
__device__ __forceinline__ void issue_half_tile(const AttnParams& p, const Item& it, int t,
                                                uint32_t dst, uint32_t bar,
                                                const CUtensorMap* tm, const CUtensorMap* tm_tree,
                                                uint64_t pol) {
  using G = TcGeom<D>;
  mbar_expect_tx(bar, G::kTileBytes);
  if (t >= it.nctx) {
    const int key0 = (t - it.nctx) * kKeys;
#pragma unroll
    for (int h = 0; h < G::kNH; ++h)
      tma_load_3d(dst + h * (kKeys * 128), tm_tree, bar, h * 64, it.g, it.s0 + key0, pol);
    return;
  }
  const int row = (it.b * p.Hkv + it.g) * p.ctx_max + it.key_base + t * kKeys;
#pragma unroll
  for (int h = 0; h < G::kNH; ++h) tma_load_2d(dst + h * (kKeys * 128), tm, bar, h * 64, row, pol);
}

// Paged context tile t, K or V (the whole producer warp): one box of
// min(page, 128) rows per page the tile touches, lane j taking page j of the
// tile, its page id read from a chunk of the sequence's page-table row that
// the warp stages in shared memory (`chunk0`: first staged entry, -1 before
// the first chunk).  Pages past the context are not loaded; an out-of-range
// page id is reported and not loaded.
template <int D>
__device__ __forceinline__ void issue_paged_half(const AttnParams& p, const Item& it, int t,
                                                 uint32_t dst, uint32_t bar, const CUtensorMap* tm,
                                                 uint64_t pol, int* s_pages, int& chunk0,
                                                 int lane) {
  using G = TcGeom<D>;
  const int ps = p.page_size;
  const int br = ps < kKeys ? ps : kKeys;
  const int nbox = kKeys / br;
  const int key0 = it.key_base + t * kKeys;
  const int e_first = key0 / ps, e_last = (key0 + (nbox - 1) * br) / ps;
  if (chunk0 < 0 || e_first < chunk0 || e_last >= chunk0 + kPageChunk) {
    chunk0 = e_first;
    const int32_t* row_pt = p.page_table + static_cast<size_t>(it.b) * p.pages_per_seq;
    for (int i = lane; i < kPageChunk; i += 32) {
      const int e = chunk0 + i;
      s_pages[i] = e < p.pages_per_seq ? row_pt[e] : -1;
    }
    __syncwarp();
  }
  int row = -1;
  if (lane < nbox) {
    const int key = key0 + lane * br;
    if (key < it.key_base + it.ctx) {
      const int page = s_pages[key / ps - chunk0];
      if (page < 0 || page >= p.num_pages)
        set_status(p.status, ASD_ERR_CTX_RANGE);
      else
        row = (page * p.Hkv + it.g) * ps + (key % ps);
    }
  }
  const uint32_t valid = __ballot_sync(0xffffffffu, row >= 0);
  if (lane == 0) mbar_expect_tx(bar, static_cast<uint32_t>(__popc(valid) * G::kNH * br * 128));
  __syncwarp();
  if (row >= 0) {
#pragma unroll
    for (int h = 0; h < G::kNH; ++h)
      tma_load_2d(dst + h * (kKeys * 128) + lane * br * 128, tm, bar, h * 64, row, pol);
  }
  __syncwarp();
}

// The query tile of an item by TMA (p.q_tma): a 3D map over q [T, Hq, D]
// with boxes of 64 columns x G heads x 128/G nodes lands as the item's 128
// rows (node-major, head-minor, as grow_of numbers them), 128-byte swizzled;
// rows past the item's hold the next nodes' queries (or zeros past T), which
// no output row reads.
template <int D>
__device__ __forceinline__ void issue_q_tile(const AttnParams& p, const Item& it, uint32_t q_s,
                                             uint32_t bar, const CUtensorMap* tm_q,
                                             uint64_t pol) {
  using G = TcGeom<D>;
  mbar_expect_tx(bar, static_cast<uint32_t>(G::kNH * kRows * 128));
#pragma unroll
  for (int h = 0; h < G::kNH; ++h)
    tma_load_3d(q_s + h * (kRows * 128), tm_q, bar, h * 64, it.g * p.G, it.s0 + it.r0 / p.G,
                pol);
}

// Ancestor bitmasks (self included) of the sequence's nodes for the tree tile,
// by the eight softmax warps (tid: thread among them); a malformed parent ends
// the walk, so it is bounded.
__device__ __forceinline__ void tree_masks(const AttnParams& p, const Item& it, int tid, int* s_par,
                                           uint64_t (*s_anc)[2]) {
  for (int i = tid; i < it.n; i += kSoftmaxThreads) s_par[i] = p.parent[it.s0 + i];
  softmax_sync();
  for (int i = tid; i < it.n; i += kSoftmaxThreads) {
    uint64_t lo = 0, hi = 0;
    int u = i;
    while (true) {
      if (u < 64) lo |= 1ull << u; else hi |= 1ull << (u - 64);
      const int pu = s_par[u];
      if (pu < 0 || pu >= u) break;
      u = pu;
    }
    s_anc[i][0] = lo;
    s_anc[i][1] = hi;
  }
  softmax_sync();
}

// One thread's share of a softmax tile: P = exp2(x c - mu) of N scores as bf16
// pairs, and their sum.  Two scores per multiply-add and per addition: the
// softmax sets the pace at D = 64 and in the ping-pong form (8 x 64 nodes at
// context 16384, one-tile form: D = 64 123.2 -> 116.3 us, D = 128 129.6 -> 124.4).
template <int N>
__device__ __forceinline__ float exp2_tile(const float* x, float c, float mu,
                                           uint32_t (&pk)[N / 2]) {
  const uint64_t c2 = pack_f32x2(c, c), nmu2 = pack_f32x2(-mu, -mu);
  uint64_t sum = 0ull;
#pragma unroll
  for (int k = 0; k < N; k += 2) {
    float y0, y1;
    unpack_f32x2(fma_f32x2(pack_f32x2(x[k], x[k + 1]), c2, nmu2), y0, y1);
    const float p0 = ex2_approx(y0), p1 = ex2_approx(y1);
    sum = add_f32x2(sum, pack_f32x2(p0, p1));
    __nv_bfloat162 h = __floats2bfloat162_rn(p0, p1);
    pk[k / 2] = *reinterpret_cast<uint32_t*>(&h);
  }
  float lo, hi;
  unpack_f32x2(sum, lo, hi);
  return lo + hi;
}

// The same, P as the sum of two bf16 numbers.  Calls of up to 128 nodes hand half
// of P to the tensor cores so (kTwoTerms): the mma.sync kernel, which took them
// before this one did, rescales to the running maximum of every 32 keys, which
// makes the largest weights exact, and with P in one term this kernel's error
// against 64 bits was up to 7 % above its.  Half of P in two terms leaves it 6 to
// 14 % below; all of P 19 to 25 %, for twice the time.  8 nodes at context 32768:
// one term 31.2 us, half 32.3, all 33.4; 128 nodes 90, 102, 117.
// `hi` is cut off behind its 8 bits, `lo` the rest rounded to bf16, so that hi + lo is
// within 2^-16 of P.  `lo` is taken from P (1 + 2^-20), which keeps it above zero
// wherever P is: an infinite V then stays infinite (0 * inf would be NaN); the sum
// is scaled likewise.
constexpr float kTwoTermScale = 1.f + 0x1p-20f;
template <int N>
__device__ __forceinline__ float exp2_tile_two(const float* x, float c, float mu,
                                               uint32_t (&hi)[N / 2], uint32_t (&lo)[N / 2]) {
  const uint64_t c2 = pack_f32x2(c, c), nmu2 = pack_f32x2(-mu, -mu);
  const uint64_t k2 = pack_f32x2(kTwoTermScale, kTwoTermScale);
  uint64_t sum = 0ull;
#pragma unroll
  for (int k = 0; k < N; k += 2) {
    float y0, y1;
    unpack_f32x2(fma_f32x2(pack_f32x2(x[k], x[k + 1]), c2, nmu2), y0, y1);
    const float p0 = ex2_approx(y0), p1 = ex2_approx(y1);
    const uint64_t p2 = pack_f32x2(p0, p1);
    sum = add_f32x2(sum, p2);
    const uint32_t u0 = __float_as_uint(p0), u1 = __float_as_uint(p1);
    hi[k / 2] = __byte_perm(u0, u1, 0x7632);
    const uint64_t nhi2 = pack_f32x2(__uint_as_float((u0 & 0xffff0000u) ^ 0x80000000u),
                                     __uint_as_float((u1 & 0xffff0000u) ^ 0x80000000u));
    unpack_f32x2(fma_f32x2(p2, k2, nhi2), y0, y1);
    __nv_bfloat162 h = __floats2bfloat162_rn(y0, y1);
    lo[k / 2] = *reinterpret_cast<uint32_t*>(&h);
  }
  float a, b;
  unpack_f32x2(sum, a, b);
  return (a + b) * kTwoTermScale;
}

// Softmax warps (eight): warp w handles TMEM lane quarter w % 4 (its 32 query
// rows, one thread per row) and half h = (w - 2) / 4 of every tile's 128 keys.
// Per tile: read its 64 S columns, mask, exchange the row's partial max with
// the warp that holds the other half, keep the reference max, and write P
// (bf16 pairs) over the tile's S columns: half h's keys go to P columns
// [32h, 32h + 32), which overlap S columns that both halves have read before
// the exchange.  The row sum stays split between the two threads of a row
// until the end.  Returns false (uniformly over the eight warps) when a
// bounded wait gave up; otherwise m_out and l_out are the row's reference max
// and sum, with O complete in TMEM.
template <int D, int MODE>
__device__ __forceinline__ bool softmax_role(const AttnParams& p, const Item& it, uint32_t tmem,
                                             uint8_t* gbase, int* s_par, uint64_t (*s_anc)[2],
                                             float (*s_mx)[2][kRows], float (*s_l)[kRows],
                                             uint64_t* q_ready, uint64_t* s_full,
                                             uint64_t* p_full, uint64_t* pv_done,
                                             uint64_t* v_full, volatile int* s_abort,
                                             long long budget, float& m_out, float& l_out) {
  using G = TcGeom<D>;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int hf = (warp - 2) >> 2;              // key half of every tile
  const int row = (warp & 3) * 32 + lane;      // = TMEM lane
  const int tid = threadIdx.x - 64;            // 0..255
  const uint32_t lane_base = tmem + (static_cast<uint32_t>((warp & 3) * 32) << 16);

  // this half of the row's query (16-byte chunks [hf D/16, (hf+1) D/16)) ->
  // shared memory, 128-byte swizzled like a TMA tile; zeros past nrows
  // (unless the query tile comes by TMA)
  if (!p.q_tma) {
    const bool mine = row < it.nrows;
    const uint4* qg = reinterpret_cast<const uint4*>(static_cast<const __nv_bfloat16*>(p.q) +
                                                     (mine ? grow_of(p, it, row) : 0) * D);
    uint8_t* qs = gbase + G::kQOff;
#pragma unroll
    for (int k = 0; k < D / 16; ++k) {
      const int c = hf * (D / 16) + k;
      const uint4 v = mine ? qg[c] : make_uint4(0u, 0u, 0u, 0u);
      *reinterpret_cast<uint4*>(qs + (c >> 3) * (kRows * 128) + row * 128 +
                                (((c & 7) ^ (row & 7)) << 4)) = v;
    }
  }
  if (!p.q_tma) {
    fence_proxy_async();   // the tensor cores read these rows
    __syncwarp();
    if (lane == 0) mbar_arrive(smem_u32(q_ready));
  }

  tree_masks(p, it, tid, s_par, s_anc);
  // ancestors among the keys of this half of the tree tile
  const uint64_t anc = row < it.nrows ? s_anc[(it.r0 + row) / p.G][hf] : 0ull;
  const float c = p.scale_log2;
  float m_ref = -INFINITY, l = 0.f;
  bool ok = true, bad = false;
  bool s_seen = false;   // S of tile t already seen complete (probed during tile t-1)
  for (int t = 0; t < it.ntiles; ++t) {
    const int b = t % kSBufs, e = t & 1;
    const uint32_t sb = lane_base + kSCol0 + b * kKeys;
    const bool tree = t >= it.nctx;
    const int key0 = tree ? (t - it.nctx) * kKeys : t * kKeys;
    const int valid = min(kKeys, (tree ? it.n : it.ctx) - key0);
    float x[64];
    float mt = -INFINITY;
    const bool here = !bad && (s_seen || wait_all(&s_full[b], (t / kSBufs) & 1, budget)) &&
                      !aborted_warp(s_abort);
    if (here) {
      tc_fence_after();
      tmem_ld64(sb + 64 * hf, x);
      if (tree || valid < kKeys) {
        // a bit per key (a 64-bit shift and a comparison per key, and one chain
        // of 32 maxima below: 16 ragged sequences of 20-100 nodes 71.0 us, now
        // 68.9; 4 x 60 nodes at contexts to 3600 25.2 -> 24.6); the tree tile
        // holds every node of the sequence, at most 128, from key 0
        const int own = min(max(valid - 64 * hf, 0), 64);
        uint64_t am = own == 64 ? ~0ull : (1ull << own) - 1ull;
        if (tree) am &= anc;
        const uint32_t w[2] = {static_cast<uint32_t>(am), static_cast<uint32_t>(am >> 32)};
#pragma unroll
        for (int k = 0; k < 64; ++k) x[k] = (w[k >> 5] >> (k & 31)) & 1u ? x[k] : -INFINITY;
      }
      float m2[2] = {fmaxf(x[0], x[1]), fmaxf(x[2], x[3])};   // two chains of maxima
#pragma unroll
      for (int k = 4; k < 64; k += 4)
#pragma unroll
        for (int q = 0; q < 2; ++q) m2[q] = fmaxf(fmaxf(m2[q], x[k + 2 * q]), x[k + 2 * q + 1]);
      mt = fmaxf(m2[0], m2[1]);
      s_mx[e][hf][row] = mt;
    }
    // probe S of the next tile now (non-blocking), so that the barrier's
    // latency passes under this tile's exponentials; once complete, that
    // phase stays complete until this warp has consumed the tile
    s_seen = __all_sync(0xffffffffu,
                        t + 1 < it.ntiles &&
                            mbar_test_wait(smem_u32(&s_full[(t + 1) % kSBufs]),
                                           static_cast<uint32_t>(((t + 1) / kSBufs) & 1)));
    // every softmax warp decides together whether to go on (no warp may be
    // left waiting at a barrier), and the partial maxima become visible
    ok = softmax_all(here);
    if (!ok) break;
    // the row's max over both halves (raw scores; the scale is positive)
    mt = fmaxf(mt, s_mx[e][hf ^ 1][row]) * c;
    const float mn = fmaxf(m_ref, mt);
    const bool had = m_ref != -INFINITY;
    const bool need = had ? (mn > m_ref + kRescaleLog2) : (mn != -INFINITY);
    if (__any_sync(0xffffffffu, need && had)) {
      // O holds earlier tiles of this row: rescale this half of it once
      // O += P V of tile t-1 is done
      // (a wait that gives up marks the thread; all leave at the next tile)
      if (!wait_all(&pv_done[(t - 1) % kSBufs], ((t - 1) / kSBufs) & 1, budget)) {
        bad = true;
      } else {
        tc_fence_after();
        const float alpha = (need && had) ? exp2f(m_ref - mn) : 1.f;
#pragma unroll 1
        for (int cc = 0; cc < D / 64; ++cc) {
          float o[32];
          const uint32_t oc = lane_base + hf * (D / 2) + 32 * cc;
          tmem_ld32(oc, o);
#pragma unroll
          for (int i = 0; i < 32; ++i) o[i] *= alpha;
          tmem_st32(oc, o);
        }
      }
    }
    if (need) {
      l = had ? l * exp2f(m_ref - mn) : 0.f;
      m_ref = mn;
    }
    const float mu = (m_ref == -INFINITY) ? 0.f : m_ref;
    if (MODE == kTwoTerms) {   // the first 32 of this half's keys
      uint32_t hi[16], lo[16], pk[16];
      l += exp2_tile_two<32>(x, c, mu, hi, lo);
      tmem_st16u(sb + 32 * hf, hi);
      tmem_st16u(sb + kKeys / 2 + 16 * hf, lo);
      l += exp2_tile<32>(x + 32, c, mu, pk);
      tmem_st16u(sb + 32 * hf + 16, pk);
    } else {
      uint32_t pk[32];
      l += exp2_tile<64>(x, c, mu, pk);
      tmem_st32u(sb + 32 * hf, pk);
    }
    if (valid < kKeys) {
      // ragged tile: V rows past the last valid key may hold anything; zero
      // them so that 0 * V stays 0, once the V tile has landed (it comes
      // through its own ring and may still be in flight).  The slot's previous
      // tile must have been consumed first: S runs up to three tiles ahead of
      // P.V, so with a late V ring that tile may not even have landed, and the
      // parity of its phase would then pass for this tile's.
      const int pt = t - G::kVStages;
      if (!bad && pt >= 0 && !wait_all(&pv_done[pt % kSBufs], (pt / kSBufs) & 1, budget))
        bad = true;
      if (!bad && wait_all(&v_full[t % G::kVStages], (t / G::kVStages) & 1, budget)) {
        uint8_t* vt = gbase + G::kVOff + (t % G::kVStages) * G::kTileBytes;
        constexpr int kChunksPerRow = G::kNH * 8;
        for (int i = tid; i < (kKeys - valid) * kChunksPerRow; i += kSoftmaxThreads) {
          const int r = valid + i / kChunksPerRow, rem = i % kChunksPerRow;
          *reinterpret_cast<uint4*>(vt + (rem >> 3) * (kKeys * 128) + r * 128 + (rem & 7) * 16) =
              make_uint4(0u, 0u, 0u, 0u);
        }
        fence_proxy_async();  // the zeroed rows are read by the tensor cores
      } else {
        bad = true;
      }
    }
    tmem_wait_st();   // P is in place
    tc_fence_before();
    __syncwarp();
    if (lane == 0) mbar_arrive(smem_u32(&p_full[b]));
  }
  if (ok) {
    // O is complete once the last P.V is done (S of the last tile waited for
    // the P.V three tiles back, so that buffer's pending phase is the last's)
    const int last = it.ntiles - 1;
    ok = !bad && wait_all(&pv_done[last % kSBufs], (last / kSBufs) & 1, budget) &&
         !aborted_warp(s_abort);
    if (ok) tc_fence_after();
  }
  if (softmax_any(!ok)) {
    if (tid == 0) {
      note_timeout(p.status);
      *s_abort = 1;
    }
    return false;
  }
  // the row sum over both halves
  s_l[hf][row] = l;
  softmax_sync();
  l_out = l + s_l[hf ^ 1][row];
  m_out = m_ref;
  return true;
}

template <int D, int MODE>
__global__ void __launch_bounds__(kThreads, 1)
    attn_tc_kernel(const __grid_constant__ CUtensorMap tm_k, const __grid_constant__ CUtensorMap tm_v,
                   const __grid_constant__ CUtensorMap tm_tk,
                   const __grid_constant__ CUtensorMap tm_tv,
                   const __grid_constant__ CUtensorMap tm_q, const AttnParams p) {
  using G = TcGeom<D>;
  extern __shared__ uint8_t smem_raw[];
  constexpr int KS = G::kKStages, VS = G::kVStages;
  __shared__ __align__(8) uint64_t s_k_full[KS], s_k_empty[KS];
  __shared__ __align__(8) uint64_t s_v_full[VS], s_v_empty[VS];
  __shared__ __align__(8) uint64_t s_s_full[kSBufs];    // S of a tile in TMEM (MMA -> softmax)
  __shared__ __align__(8) uint64_t s_p_full[kSBufs];    // P of a tile in TMEM (softmax -> MMA)
  __shared__ __align__(8) uint64_t s_pv_done[kSBufs];   // O += P V of a tile done (MMA -> softmax)
  __shared__ __align__(8) uint64_t s_q_ready;
  __shared__ __align__(8) uint64_t s_mma_done[2];   // each MMA issuer's own drain
  __shared__ uint32_t s_tmem;
  __shared__ volatile int s_abort;
  __shared__ int s_par[kMaxNodes];
  __shared__ uint64_t s_anc[kMaxNodes][2];
  __shared__ float s_mx[2][2][kRows];   // [tile parity][key half][row]: partial row max
  __shared__ float s_l[2][kRows];       // [key half][row]: partial row sum
  __shared__ int s_pages[2][kPageChunk];   // K / V producer: staged page-table entries
  __shared__ int s_issued[2][KS > VS ? KS : VS];  // producer: K (0) / V (1) fills per stage

  __shared__ PlanSmem s_plan;

  pdl_launch_dependents();
  if (MODE == kByContext && attention_takes_pairs(p)) {   // the ping-pong form's call
    pdl_wait();
    return;
  }
  // the mma.sync kernel's step (a call by itself: make_item)
  if (MODE == kTwoTerms && p.co_tiles >= 0 && !p.alone && attention_takes_mma(p)) {
    pdl_wait();
    return;
  }
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const long long budget = wait_budget(p.wait_cycles);

  uint32_t base = smem_u32(smem_raw);
  const uint32_t pad = (1024u - (base & 1023u)) & 1023u;
  uint8_t* gbase = smem_raw + pad;
  base += pad;
  const uint32_t q_s = base + G::kQOff, k_s0 = base + G::kKOff, v_s0 = base + G::kVOff;

  // The set-up that needs no item runs while the first loads of make_item are
  // on their way; make_item synchronises the CTA, and from then on every role
  // runs by itself (32 ragged sequences of 4 to 8 nodes, paged: 123.5 -> 120.9 us
  // with the masks built by the softmax warps, beside the first copies).
  if (threadIdx.x == 32 * 11) {
    for (int s = 0; s < KS; ++s) {
      mbar_init(smem_u32(&s_k_full[s]), 1);
      mbar_init(smem_u32(&s_k_empty[s]), 1);
      s_issued[0][s] = 0;
    }
    for (int s = 0; s < VS; ++s) {
      mbar_init(smem_u32(&s_v_full[s]), 1);
      mbar_init(smem_u32(&s_v_empty[s]), 1);
      s_issued[1][s] = 0;
    }
    for (int b = 0; b < kSBufs; ++b) {
      mbar_init(smem_u32(&s_s_full[b]), 1);
      mbar_init(smem_u32(&s_p_full[b]), kSoftmaxThreads / 32);
      mbar_init(smem_u32(&s_pv_done[b]), 1);
    }
    // the query: one TMA (p.q_tma) or the eight softmax warps' stores
    mbar_init(smem_u32(&s_q_ready), p.q_tma ? 1 : kSoftmaxThreads / 32);
    mbar_init(smem_u32(&s_mma_done[0]), 1);
    mbar_init(smem_u32(&s_mma_done[1]), 1);
    s_abort = 0;
    fence_mbar_init();
  }
  if (warp == 10) {
    tmem_alloc(smem_u32(&s_tmem), kTmemCols);
    tmem_relinquish();
    tc_fence_before();
  }
  Item it;
  const bool some = make_item<kRows, MODE>(p, it, s_plan);   // uniform over the CTA
  tc_fence_after();
  if (!some) {   // no query rows here
    if (warp == 10) tmem_dealloc(s_tmem, kTmemCols);
    pdl_wait();
    return;
  }
  const uint32_t tmem = s_tmem;

  bool ok = false;           // softmax warps: O complete in TMEM
  float m_row = 0.f, l_row = 0.f;
  if (warp == 0 || warp == 11) {
    // ----------------------------------------------------------- TMA producers
    // K and V come through rings of their own, each filled by its own warp
    // (warp 0 K, warp 11 V), so that neither ring waits behind the other: a K
    // slot is free again once the S MMA of its tile is done, a V slot once the
    // P.V MMA is.
    const int which = warp == 0 ? 0 : 1;
    const int ns = which ? VS : KS;
    if (lane == 0) {
      prefetch_tmap(which ? &tm_v : &tm_k);
      prefetch_tmap(which ? &tm_tv : &tm_tk);
    }
    const uint64_t pol = l2_policy_evict_first();
    if (which == 0 && lane == 0 && p.q_tma)
      issue_q_tile<D>(p, it, q_s, smem_u32(&s_q_ready), &tm_q, pol);
    int chunk0 = -1;
    bool pok = true;
    for (int t = 0; pok && t < it.ntiles; ++t) {
      const int stage = t % ns;
      uint64_t* empty = which ? &s_v_empty[stage] : &s_k_empty[stage];
      uint64_t* full = which ? &s_v_full[stage] : &s_k_full[stage];
      if (!wait_all(empty, ((t / ns) & 1) ^ 1u, budget) || aborted_warp(&s_abort)) {
        pok = false;
        break;
      }
      const uint32_t dst = base + (which ? G::kVOff : G::kKOff) + stage * G::kTileBytes;
      if (p.page_size != 0 && t < it.nctx)
        issue_paged_half<D>(p, it, t, dst, smem_u32(full), which ? &tm_v : &tm_k, pol,
                            s_pages[which], chunk0, lane);
      else if (lane == 0)
        issue_half_tile<D>(p, it, t, dst, smem_u32(full), which ? &tm_v : &tm_k,
                           which ? &tm_tv : &tm_tk, pol);
      if (lane == 0) ++s_issued[which][stage];
      __syncwarp();
    }
    if (!pok && lane == 0) {
      note_timeout(p.status);
      s_abort = 1;
    }
    // every copy issued has landed before the buffers are reused or left
    // (the query tile's too, which a wait that gave up may have left in flight)
    if (lane == 0) {
      for (int st = 0; st < ns; ++st)
        if (s_issued[which][st] > 0)
          mbar_wait(smem_u32(which ? &s_v_full[st] : &s_k_full[st]),
                    static_cast<uint32_t>((s_issued[which][st] - 1) & 1));
      if (which == 0 && p.q_tma) mbar_wait(smem_u32(&s_q_ready), 0);
    }
    __syncwarp();
  } else if (warp == 1 || warp == 10) {
    // ------------------------------------------------------------ MMA issuers
    // Two issuing threads, so that the one's barrier waits (each a few hundred
    // cycles even on a completed phase) overlap the other's MMAs: warp 1
    // issues S = Q K^T of every tile, warp 10 O += P V.  Each commit tracks the
    // issuing thread's own MMAs.
    if (lane == 0) {
      bool mok = true;
      if (warp == 1) {
        const uint32_t idesc_s = idesc_bf16(kRows, kKeys);   // S = Q K^T
        mok = mbar_wait(smem_u32(&s_q_ready), 0, budget);
        if (mok) tc_fence_after();
        for (int t = 0; mok && t < it.ntiles; ++t) {
          const int stage = t % KS, b = t % kSBufs;
          mok = mbar_wait(smem_u32(&s_k_full[stage]), (t / KS) & 1, budget);
          // the S/P buffer is free once O += P V of tile t-3 is done
          if (mok && t >= kSBufs)
            mok = mbar_wait(smem_u32(&s_pv_done[b]), ((t / kSBufs) - 1) & 1, budget);
          if (!mok || s_abort) break;
          tc_fence_after();
          const uint32_t kst = k_s0 + stage * G::kTileBytes;
#pragma unroll
          for (int ks = 0; ks < D / 16; ++ks) {
            const int h = ks >> 2, kk = ks & 3;
            tc_mma(tmem + kSCol0 + b * kKeys, sw128_desc(q_s + h * (kRows * 128) + 32 * kk),
                   sw128_desc(kst + h * (kKeys * 128) + 32 * kk), idesc_s, ks > 0 ? 1u : 0u);
          }
          tc_commit(smem_u32(&s_s_full[b]));
          tc_commit(smem_u32(&s_k_empty[stage]));
        }
      } else {
        const uint32_t idesc_o = idesc_bf16(kRows, D, true);   // O += P V, V MN-major
        for (int j = 0; mok && j < it.ntiles; ++j) {
          // O += P_j V_j once tile j's softmax has written P_j
          const int stage = j % VS, b = j % kSBufs;
          mok = mbar_wait(smem_u32(&s_p_full[b]), (j / kSBufs) & 1, budget) &&
                mbar_wait(smem_u32(&s_v_full[stage]), (j / VS) & 1, budget);
          if (!mok || s_abort) break;
          tc_fence_after();
          const uint32_t vst = v_s0 + stage * G::kTileBytes;
#pragma unroll
          for (int kk = 0; kk < kKeys / 16; ++kk)
            tc_mma_ts(tmem, tmem + kSCol0 + b * kKeys + kk * 8,
                      sw128_desc_mn(vst + kk * 2048, kKeys * 128, 1024), idesc_o,
                      (j > 0 || kk > 0) ? 1u : 0u);
          if (MODE == kTwoTerms)   // second terms of keys 0-31 and 64-95
#pragma unroll
            for (int i = 0; i < 4; ++i)
              tc_mma_ts(tmem, tmem + kSCol0 + b * kKeys + kKeys / 2 + i * 8,
                        sw128_desc_mn(vst + ((i & 1) + 4 * (i >> 1)) * 2048, kKeys * 128, 1024),
                        idesc_o, 1u);
          tc_commit(smem_u32(&s_pv_done[b]));
          tc_commit(smem_u32(&s_v_empty[stage]));
        }
      }
      if (!mok) {
        note_timeout(p.status);
        s_abort = 1;
      }
      // every MMA this thread issued has finished before TMEM or the buffers
      // are reused
      uint64_t* done = &s_mma_done[warp == 1 ? 0 : 1];
      tc_commit(smem_u32(done));
      mbar_wait(smem_u32(done), 0);
    }
    __syncwarp();
  } else {
    ok = softmax_role<D, MODE>(p, it, tmem, gbase, s_par, s_anc, s_mx, s_l, &s_q_ready, s_s_full, s_p_full,
                         s_pv_done, s_v_full, &s_abort, budget, m_row, l_row);
  }

  // ------------------------------------------------------------------ finish
  tc_fence_before();
  __syncthreads();   // the tile buffers and the tensor cores are idle from here on
  tc_fence_after();
  if (warp >= 2 && warp < 10 && ok) {
    // Each thread holds its key half's share of a row, D/2 columns: the output,
    // or (one of several chunks) the fp32 partial that attn_merge_kernel
    // combines.
    const int hf = (warp - 2) >> 2;
    const int row0 = (warp & 3) * 32, row = row0 + lane;   // TMEM lane = query row
    const uint32_t lane_base = tmem + (static_cast<uint32_t>(row0) << 16) +
                               static_cast<uint32_t>(hf * (D / 2));
    const bool mine = row < it.nrows;
    if (it.chunks == 1) {
      const float inv = l_row > 0.f ? 1.f / l_row : 0.f;
      __nv_bfloat16* out = static_cast<__nv_bfloat16*>(p.out) +
                           (mine ? grow_of(p, it, row) : 0) * D + hf * (D / 2);
#pragma unroll 1
      for (int c = 0; c < D / 64; ++c) {
        float o[32];
        tmem_ld32(lane_base + 32 * c, o);   // every lane takes part in the warp-wide load
        if (mine) {
#pragma unroll
          for (int k = 0; k < 32; k += 8) {
            uint4 pk;
            __nv_bfloat162 h0 = __floats2bfloat162_rn(o[k] * inv, o[k + 1] * inv);
            __nv_bfloat162 h1 = __floats2bfloat162_rn(o[k + 2] * inv, o[k + 3] * inv);
            __nv_bfloat162 h2 = __floats2bfloat162_rn(o[k + 4] * inv, o[k + 5] * inv);
            __nv_bfloat162 h3 = __floats2bfloat162_rn(o[k + 6] * inv, o[k + 7] * inv);
            pk.x = *reinterpret_cast<uint32_t*>(&h0);
            pk.y = *reinterpret_cast<uint32_t*>(&h1);
            pk.z = *reinterpret_cast<uint32_t*>(&h2);
            pk.w = *reinterpret_cast<uint32_t*>(&h3);
            *reinterpret_cast<uint4*>(out + 32 * c + k) = pk;
          }
        }
      }
    } else if (row0 < it.nrows) {
      // Written by the lanes that hold them, the partials' 16-byte stores would
      // touch 32 rows each; turned through shared memory (the tile buffers are
      // free), eight lanes write 128 consecutive bytes: 2.6 -> 1.6 us for a
      // CTA's 128 rows of 128 columns.  (The bf16 output, half the bytes, is
      // faster as it is: 0.6 us against 1.4 for 32 rows.)
      const size_t prow = static_cast<size_t>(it.part0) +
                          static_cast<size_t>(it.g * it.chunks + it.chunk) * it.R + it.r0 + row0;
      if (mine && hf == 0) p.part_ml[prow + lane] = make_float2(m_row, l_row);
      constexpr int kStLd = 36;   // padded row of 32 columns
      float* stg = reinterpret_cast<float*>(gbase) + (warp - 2) * 32 * kStLd;
#pragma unroll 1
      for (int c = 0; c < D / 64; ++c) {
        float o[32];
        tmem_ld32(lane_base + 32 * c, o);
#pragma unroll
        for (int k = 0; k < 8; ++k)
          *reinterpret_cast<float4*>(stg + lane * kStLd + 4 * k) =
              make_float4(o[4 * k], o[4 * k + 1], o[4 * k + 2], o[4 * k + 3]);
        __syncwarp();
        const int col = 4 * (lane & 7);
        float* po = p.part_o + prow * D + hf * (D / 2) + 32 * c + col;
#pragma unroll
        for (int i = 0; i < 8; ++i) {
          const int r = 4 * i + (lane >> 3);
          if (row0 + r < it.nrows)
            *reinterpret_cast<float4*>(po + static_cast<size_t>(r) * D) =
                *reinterpret_cast<const float4*>(stg + r * kStLd + col);
        }
        __syncwarp();
      }
    }
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  if (warp == 10) tmem_dealloc(tmem, kTmemCols);
  if (s_plan.past > 0 && warp >= 2 && warp < 10)
    items_past_grid<D>(p, s_plan, threadIdx.x - 64);
  pdl_wait();   // the next kernel's wait covers every earlier kernel
}

// Combines the chunks of every query row that attn_tc_kernel split:
//   out = sum_z 2^(m_z - M) O_z / sum_z 2^(m_z - M) l_z,  M = max_z m_z.
// W warps per row: lane z of each reads chunk z's (reference max, row sum),
// warp w adds up chunks w, w + W, ..., each lane D/32 columns, four or eight
// loads in flight, and the W sums meet in shared memory.  Few rows come in many chunks
// and take W = 4 (256 rows in 19 chunks: 3.9 us, 9.7 with a warp per row),
// many rows in few chunks and take W = 1 (7680 rows in up to 3 chunks: 3.4 us,
// 11 with four warps, all of it CTA launches).  Sequences in one chunk
// (plan[b].y == 1) were written by attn_tc_kernel.
constexpr int kMergeThreads = 256;
constexpr int kMergeFewRows = 2048;   // query rows of a step up to which W = 4

template <int D, int W>
__global__ void __launch_bounds__(kMergeThreads) attn_merge_kernel(const AttnParams p) {
  constexpr int kV = D / 32, kMergeWarps = W, kMergeRows = kMergeThreads / 32 / W;
  constexpr int kMergeLoads = W == 1 ? 4 : 8;   // of 3 and 19 chunks in the cases above
  __shared__ float s_acc[kMergeRows][kMergeWarps][D];
  pdl_launch_dependents();
  const int b = blockIdx.y / p.Hkv, g = blockIdx.y - b * p.Hkv;
  const int lane = threadIdx.x & 31;
  const int w = (threadIdx.x >> 5) % kMergeWarps, rl = (threadIdx.x >> 5) / kMergeWarps;
  const int s0 = p.cu_nodes[b], n = p.cu_nodes[b + 1] - s0, R = n * p.G;
  pdl_wait();
  if (p.co_tiles >= 0 && attention_takes_mma(p)) return;   // nothing was cut
  if (n <= 0 || n > kMaxNodes || s0 < 0 || s0 + n > p.T || static_cast<int>(blockIdx.x) * kMergeRows >= R)
    return;
  const int2 plan = __ldcg(p.plan + b);
  const int c = plan.y;
  if (c < 2 || c > kMaxChunks || plan.x < 0 ||
      plan.x + static_cast<long long>(R) * p.Hkv * c > p.part_cap)
    return;
  const int row = blockIdx.x * kMergeRows + rl;
  const bool mine = row < R;
  const size_t base = static_cast<size_t>(plan.x) + static_cast<size_t>(g) * c * R + (mine ? row : 0);
  float wt = 0.f, sum = 0.f, acc[kV];
#pragma unroll
  for (int j = 0; j < kV; ++j) acc[j] = 0.f;
#pragma unroll 1
  for (int z0 = w; z0 < c; z0 += kMergeLoads * W) {   // uniform over the warp
    float v[kMergeLoads][kV];
#pragma unroll
    for (int k = 0; k < kMergeLoads; ++k) {
      const int z = z0 + k * W;
      const float* po = p.part_o + (base + static_cast<size_t>(z < c ? z : 0) * R) * D + lane * kV;
      if (kV == 4) {
        const float4 x = z < c ? __ldcg(reinterpret_cast<const float4*>(po))
                               : make_float4(0.f, 0.f, 0.f, 0.f);
        v[k][0] = x.x;
        v[k][1] = x.y;
        v[k][kV - 2] = x.z;
        v[k][kV - 1] = x.w;
      } else {
        const float2 x = z < c ? __ldcg(reinterpret_cast<const float2*>(po)) : make_float2(0.f, 0.f);
        v[k][0] = x.x;
        v[k][1] = x.y;
      }
    }
    if (z0 == w) {   // the weights, while the first chunks' rows are on their way
      const float2 ml = lane < c ? __ldcg(p.part_ml + base + static_cast<size_t>(lane) * R)
                                 : make_float2(-INFINITY, 0.f);
      float M = ml.x;
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) M = fmaxf(M, __shfl_xor_sync(0xffffffffu, M, o));
      wt = ml.x == -INFINITY ? 0.f : exp2f(ml.x - M);
      sum = wt * ml.y;
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
    }
#pragma unroll
    for (int k = 0; k < kMergeLoads; ++k) {
      const float wz = __shfl_sync(0xffffffffu, wt, (z0 + k * W) & 31);   // 0 from c on
#pragma unroll
      for (int j = 0; j < kV; ++j) acc[j] = fmaf(z0 + k * W < c ? wz : 0.f, v[k][j], acc[j]);
    }
  }
#pragma unroll
  for (int j = 0; j < kV; ++j) s_acc[rl][w][lane * kV + j] = acc[j];
  __syncthreads();
  // two columns per lane and step, the row's W warps side by side
  const float inv = sum > 0.f ? 1.f / sum : 0.f;
  const int i = row / p.G;
  if (!mine) return;
  __nv_bfloat16* out = static_cast<__nv_bfloat16*>(p.out) +
                       (static_cast<size_t>(s0 + i) * p.Hq + g * p.G + (row - i * p.G)) * D;
  for (int col = w * 64 + 2 * lane; col < D; col += 64 * W) {
    float x = 0.f, y = 0.f;
#pragma unroll
    for (int k = 0; k < W; ++k) {
      x += s_acc[rl][k][col];
      y += s_acc[rl][k][col + 1];
    }
    *reinterpret_cast<__nv_bfloat162*>(out + col) = __floats2bfloat162_rn(x * inv, y * inv);
  }
}

// ----------------------------------------------------------------------------
// Ping-pong variant: one CTA per (256 query rows, sequence x KV head) = two
// 128-row query tiles A and B that see the same keys.  Every K/V tile serves
// both: S_A = Q_A.K^T and S_B = Q_B.K^T, then O_A += P_A.V and O_B += P_B.V, so
// the MMAs of one tile run while the other tile's softmax works, and a K/V
// byte feeds twice the products.  Q stays in shared memory (both tiles, 128-byte
// swizzled, by TMA or written by the softmax threads).  K and V come through
// separate rings with their own barriers, so a K slot is refilled as soon as
// both S MMAs have read it.  Warps: 0 K producer, 1 S-MMA issuer (lane 0),
// 2 P.V-MMA issuer (lane 0), 3 V producer, 4-7 softmax of tile A, 8-11 softmax
// of tile B; a softmax thread owns one row of its tile and all 128 keys of
// every key tile, so no exchange between warps is needed.  It takes the row's
// 128 scores into registers with one TMEM load, which frees the S columns: S of
// the next tile does not wait for the softmax or for P.V.  P has columns of its
// own (bf16 pairs, half as many), so TMEM holds O_A, O_B, one S buffer and P_A,
// P_B at D = 128, an S buffer per query tile at D = 64.  The 128 scores need
// more than 168 registers a thread, so the softmax warpgroups take what the
// issuing one leaves (setmaxnreg).
//
// Measured against S and P sharing their columns, the scores read twice (before
// -> now, 8 KV heads, G = 4): 64 x 128 nodes at context 2048 303.5 -> 274.5 us
// (D = 128), 265.6 -> 225 us (D = 64); contexts 300-1000 180.7 -> 149 us; 62 x
// 60 nodes at 17-137 66.8 -> 53.5 us.  What bounds it: a pair of key tiles takes
// ~3,950 cycles, of which the MMAs alone ~3,200 (shared memory feeds the S ones);
// the rest is S read -> next S.  No faster: two warps per row quarter, 64 keys
// each and a pair barrier (299 us), P handed over by key halves (274.3, D = 64
// 252), P.V held back while S MMAs are issued (282), waits that spin on test_wait
// instead of try_wait (288).
constexpr int kPPRows = 2 * kRows;   // query rows per CTA

template <int D>
struct PPGeom {
  static constexpr int kNH = D / 64;
  static constexpr int kStages = D == 64 ? 3 : 2;
  static constexpr int kQTile = kNH * kRows * 128;    // one query tile
  static constexpr int kKVTile = kNH * kKeys * 128;   // one K or one V tile
  static constexpr int kQOff = 0;
  static constexpr int kKOff = 2 * kQTile;
  static constexpr int kVOff = kKOff + kStages * kKVTile;
  static constexpr int kBytes = kVOff + kStages * kKVTile;
  // TMEM columns: O_A, O_B, then the S buffers (at D = 128 one for both query
  // tiles), then P_A and P_B
  static constexpr int kSBufs = D == 64 ? 2 : 1;
  static __device__ __forceinline__ uint32_t s_col(int x) {
    return 2 * D + (kSBufs == 2 ? kKeys * static_cast<uint32_t>(x) : 0u);
  }
  static __device__ __forceinline__ uint32_t p_col(int x) {
    return 384u + kKeys / 2 * static_cast<uint32_t>(x);
  }
};

// Registers per thread of the issuing warpgroup (warps 0-3) and of the two
// softmax ones, out of the 168 each that the block is launched with (a split
// whose sum is above that would wait forever).  88 / 208: D = 64 229 us, not 225.
constexpr int kPPIssueRegs = 120, kPPSoftmaxRegs = 192;
static_assert(128 * kPPIssueRegs + 256 * kPPSoftmaxRegs <= kThreads * 168,
              "more registers than the block is launched with");

template <int N>
__device__ __forceinline__ void regs_inc() {
  asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(N));
}

template <int N>
__device__ __forceinline__ void regs_dec() {
  asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(N));
}

template <int D, int MODE>
__global__ void __launch_bounds__(kThreads, 1)
    attn_pp_kernel(const __grid_constant__ CUtensorMap tm_k, const __grid_constant__ CUtensorMap tm_v,
                   const __grid_constant__ CUtensorMap tm_tk,
                   const __grid_constant__ CUtensorMap tm_tv,
                   const __grid_constant__ CUtensorMap tm_q, const AttnParams p) {
  using G = PPGeom<D>;
  constexpr int S = G::kStages;
  extern __shared__ uint8_t smem_raw[];
  __shared__ __align__(8) uint64_t s_k_full[S], s_k_empty[S], s_v_full[S], s_v_empty[S];
  __shared__ __align__(8) uint64_t s_s_full[2];    // S of tile X computed (MMA -> softmax X)
  __shared__ __align__(8) uint64_t s_s_read[2];    // S of tile X read (softmax X -> MMA)
  __shared__ __align__(8) uint64_t s_p_full[2];    // P of tile X written (softmax X -> MMA)
  __shared__ __align__(8) uint64_t s_pv_done[2];   // O_X += P_X V done (MMA -> softmax X)
  __shared__ __align__(8) uint64_t s_q_ready;
  __shared__ __align__(8) uint64_t s_mma_done[2];   // each MMA issuer's own drain
  __shared__ uint32_t s_tmem;
  __shared__ volatile int s_abort;
  __shared__ int s_par[kMaxNodes];
  __shared__ uint64_t s_anc[kMaxNodes][2];
  __shared__ int s_pages[2][kPageChunk];   // K / V producer: staged page-table entries
  __shared__ int s_issued[2][S];   // producer: K (0) and V (1) fills issued per stage

  __shared__ PlanSmem s_plan;

  pdl_launch_dependents();
  if (MODE == kByContext && !attention_takes_pairs(p)) {   // the one-tile form's call
    pdl_wait();
    return;
  }
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const long long budget = wait_budget(p.wait_cycles);

  uint32_t base = smem_u32(smem_raw);
  const uint32_t pad = (1024u - (base & 1023u)) & 1023u;
  uint8_t* gbase = smem_raw + pad;
  base += pad;

  // as in the one-tile kernel: the set-up that needs no item under make_item's
  // first loads, then every role by itself
  if (threadIdx.x == 32 * 3) {
    for (int s = 0; s < S; ++s) {
      mbar_init(smem_u32(&s_k_full[s]), 1);
      mbar_init(smem_u32(&s_k_empty[s]), 1);
      mbar_init(smem_u32(&s_v_full[s]), 1);
      mbar_init(smem_u32(&s_v_empty[s]), 1);
      s_issued[0][s] = s_issued[1][s] = 0;
    }
    for (int x = 0; x < 2; ++x) {
      mbar_init(smem_u32(&s_s_full[x]), 1);
      mbar_init(smem_u32(&s_s_read[x]), 4);
      mbar_init(smem_u32(&s_p_full[x]), 4);
      mbar_init(smem_u32(&s_pv_done[x]), 1);
    }
    // the query tiles: TMA (p.q_tma) or the eight softmax warps' stores
    mbar_init(smem_u32(&s_q_ready), p.q_tma ? 1 : 8);
    mbar_init(smem_u32(&s_mma_done[0]), 1);
    mbar_init(smem_u32(&s_mma_done[1]), 1);
    s_abort = 0;
    fence_mbar_init();
  }
  if (warp == 2) {
    tmem_alloc(smem_u32(&s_tmem), kTmemCols);
    tmem_relinquish();
    tc_fence_before();
  }
  Item it;
  const bool some = make_item<kPPRows, MODE>(p, it, s_plan);   // uniform over the CTA
  tc_fence_after();
  if (!some) {   // no query rows here
    if (warp == 2) tmem_dealloc(s_tmem, kTmemCols);
    pdl_wait();
    return;
  }
  const int nx = it.nrows > kRows ? 2 : 1;   // query tiles present
  const uint32_t tmem = s_tmem;

  if (warp < 4) {
    regs_dec<kPPIssueRegs>();
    if (warp == 0 || warp == 3) {
      // ----------------------------------------------------------- TMA producers
      // K (warp 0) and V (warp 3), each into its own ring; K slots free up as
      // soon as both S MMAs of their tile are done, V slots after both P.V MMAs
      const int which = warp == 0 ? 0 : 1;
      if (lane == 0) {
        prefetch_tmap(which ? &tm_v : &tm_k);
        prefetch_tmap(which ? &tm_tv : &tm_tk);
      }
      const uint64_t pol = l2_policy_evict_first();
      if (which == 0 && lane == 0 && p.q_tma) {
        const uint32_t bar = smem_u32(&s_q_ready);
        mbar_expect_tx(bar, static_cast<uint32_t>(nx * G::kQTile));
        for (int x = 0; x < nx; ++x)
#pragma unroll
          for (int h = 0; h < G::kNH; ++h)
            tma_load_3d(base + G::kQOff + x * G::kQTile + h * (kRows * 128), &tm_q, bar, h * 64,
                        it.g * p.G, it.s0 + (it.r0 + x * kRows) / p.G, pol);
      }
      int chunk0 = -1;
      bool pok = true;
      for (int t = 0; t < it.ntiles; ++t) {
        const int stage = t % S;
        uint64_t* empty = which ? &s_v_empty[stage] : &s_k_empty[stage];
        uint64_t* full = which ? &s_v_full[stage] : &s_k_full[stage];
        if (!wait_all(empty, ((t / S) & 1) ^ 1u, budget) || aborted_warp(&s_abort)) {
          pok = false;
          break;
        }
        const uint32_t dst = base + (which ? G::kVOff : G::kKOff) + stage * G::kKVTile;
        if (p.page_size != 0 && t < it.nctx)
          issue_paged_half<D>(p, it, t, dst, smem_u32(full), which ? &tm_v : &tm_k, pol,
                              s_pages[which], chunk0, lane);
        else if (lane == 0)
          issue_half_tile<D>(p, it, t, dst, smem_u32(full), which ? &tm_v : &tm_k,
                             which ? &tm_tv : &tm_tk, pol);
        if (lane == 0) ++s_issued[which][stage];
        __syncwarp();
      }
      if (!pok && lane == 0) {
        note_timeout(p.status);
        s_abort = 1;
      }
      // every copy issued has landed before the buffers are reused or left
      // (the query tiles' too, which a wait that gave up may have left in flight)
      if (lane == 0) {
        for (int st = 0; st < S; ++st)
          if (s_issued[which][st] > 0)
            mbar_wait(smem_u32(which ? &s_v_full[st] : &s_k_full[st]),
                      static_cast<uint32_t>((s_issued[which][st] - 1) & 1));
        if (which == 0 && p.q_tma) mbar_wait(smem_u32(&s_q_ready), 0);
      }
      __syncwarp();
    } else {
      // ------------------------------------------------------------ MMA issuers
      // Two issuing threads, so that the one's barrier waits overlap the other's
      // MMAs: warp 1 issues S_x(t) = Q_x K(t)^T, warp 2 O_x += P_x(t) V(t).
      // While tile A's softmax works on key tile t, the tensor cores run
      // O_B += P_B V(t-1) and S_B(t); while B's works, O_A += P_A V(t) and
      // S_A(t+1).  Each commit tracks the issuing thread's own MMAs.
      if (lane == 0) {
        bool mok = true;
        if (warp == 1) {
          const uint32_t idesc_s = idesc_bf16(kRows, kKeys);   // S = Q K^T
          mok = mbar_wait(smem_u32(&s_q_ready), 0, budget);
          if (mok) tc_fence_after();
          for (int t = 0; mok && t < it.ntiles; ++t) {
            const int stage = t % S;
            mok = mbar_wait(smem_u32(&s_k_full[stage]), (t / S) & 1, budget);
            for (int x = 0; mok && x < nx; ++x) {
              // the S columns are free once their last tile has been read: tile x's
              // own, or (one buffer) that of the query tile before it
              const int px = G::kSBufs == 2 ? x : (x == 0 ? nx - 1 : 0);
              const int pt = px < x ? t : t - 1;
              if (pt >= 0) mok = mbar_wait(smem_u32(&s_s_read[px]), pt & 1, budget);
              if (!mok || s_abort) {
                mok = false;
                break;
              }
              tc_fence_after();
              const uint32_t kst = base + G::kKOff + stage * G::kKVTile;
              const uint32_t qst = base + G::kQOff + x * G::kQTile;
#pragma unroll
              for (int ks = 0; ks < D / 16; ++ks) {
                const int h = ks >> 2, kk = ks & 3;
                tc_mma(tmem + G::s_col(x), sw128_desc(qst + h * (kRows * 128) + 32 * kk),
                       sw128_desc(kst + h * (kKeys * 128) + 32 * kk), idesc_s, ks > 0 ? 1u : 0u);
              }
              tc_commit(smem_u32(&s_s_full[x]));
            }
            // the last S of tile t releases K(t)
            if (mok) tc_commit(smem_u32(&s_k_empty[stage]));
          }
        } else {
          const uint32_t idesc_o = idesc_bf16(kRows, D, true);   // O += P V, V MN-major
          for (int t = 0; mok && t < it.ntiles; ++t) {
            const int stage = t % S;
            mok = mbar_wait(smem_u32(&s_v_full[stage]), (t / S) & 1, budget);
            for (int x = 0; mok && x < nx; ++x) {
              // O_x += P_x(t) V(t) once tile x's softmax of key tile t is done
              mok = mbar_wait(smem_u32(&s_p_full[x]), t & 1, budget);
              if (!mok || s_abort) {
                mok = false;
                break;
              }
              tc_fence_after();
              const uint32_t vst = base + G::kVOff + stage * G::kKVTile;
#pragma unroll
              for (int kk = 0; kk < kKeys / 16; ++kk)
                tc_mma_ts(tmem + static_cast<uint32_t>(x * D), tmem + G::p_col(x) + kk * 8,
                          sw128_desc_mn(vst + kk * 2048, kKeys * 128, 1024), idesc_o,
                          (t > 0 || kk > 0) ? 1u : 0u);
              tc_commit(smem_u32(&s_pv_done[x]));
            }
            // the last P.V of tile t releases V(t)
            if (mok) tc_commit(smem_u32(&s_v_empty[stage]));
          }
        }
        if (!mok) {
          note_timeout(p.status);
          s_abort = 1;
        }
        // every MMA this thread issued has finished before TMEM or the buffers
        // are reused
        uint64_t* done = &s_mma_done[warp == 1 ? 0 : 1];
        tc_commit(smem_u32(done));
        mbar_wait(smem_u32(done), 0);
      }
      __syncwarp();
    }
  } else {
    regs_inc<kPPSoftmaxRegs>();
    // ------------------------------------------------------------ softmax of tile x
    const int x = (warp - 4) >> 2;
    const int row = (warp & 3) * 32 + lane;    // = TMEM lane = row of the tile
    const int rr = x * kRows + row;            // row of the item
    const bool mine = rr < it.nrows;
    const uint32_t lane_base = tmem + (static_cast<uint32_t>((warp & 3) * 32) << 16);
    const uint32_t sb = lane_base + G::s_col(x), pb = lane_base + G::p_col(x);
    // the row's query -> shared memory, 128-byte swizzled like a TMA tile
    // (unless the query tiles come by TMA)
    if (!p.q_tma) {
      const int q_row = it.r0 + rr;
      const int node = q_row / p.G;
      const uint4* qg = reinterpret_cast<const uint4*>(
          static_cast<const __nv_bfloat16*>(p.q) +
          (mine ? (static_cast<size_t>(it.s0 + node) * p.Hq + it.g * p.G + (q_row - node * p.G)) : 0) *
              D);
      uint8_t* qs = gbase + G::kQOff + x * G::kQTile;
#pragma unroll
      for (int c = 0; c < D / 8; ++c) {
        const uint4 v = mine ? qg[c] : make_uint4(0u, 0u, 0u, 0u);
        *reinterpret_cast<uint4*>(qs + (c >> 3) * (kRows * 128) + row * 128 +
                                  (((c & 7) ^ (row & 7)) << 4)) = v;
      }
      fence_proxy_async();   // the tensor cores read these rows
      __syncwarp();
      if (lane == 0) mbar_arrive(smem_u32(&s_q_ready));
    }
    tree_masks(p, it, threadIdx.x - 128, s_par, s_anc);
    uint64_t alo = 0, ahi = 0;
    if (mine) {
      const int node = (it.r0 + rr) / p.G;
      alo = s_anc[node][0];
      ahi = s_anc[node][1];
    }
    // a second query tile with no rows: its warps only staged the zero rows
    if (x < nx) {
    const float c = p.scale_log2;
    float m_ref = -INFINITY, l = 0.f;
    bool ok = true;
    for (int t = 0; t < it.ntiles; ++t) {
      const bool tree = t >= it.nctx;
      const int key0 = tree ? (t - it.nctx) * kKeys : t * kKeys;
      const int valid = min(kKeys, (tree ? it.n : it.ctx) - key0);
      ok = wait_all(&s_s_full[x], t & 1, budget) && !aborted_warp(&s_abort);
      if (!ok) break;
      tc_fence_after();
      // the row's scores -> registers, which frees the S columns for the next
      // S; only a ragged context tile and the tree tile need the key mask
      float xs[128];
      tmem_ld128(sb, xs);
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(smem_u32(&s_s_read[x]));
      if (tree || valid < kKeys) {
#pragma unroll
        for (int q = 0; q < 4; ++q) {   // 32 keys each, a bit per key
          // the tree tile holds every node of the sequence (at most 128) from key 0
          const int own = min(max(valid - 32 * q, 0), 32);
          uint32_t w = own == 32 ? ~0u : (1u << own) - 1u;
          if (tree) w &= static_cast<uint32_t>((q & 2 ? ahi : alo) >> (32 * (q & 1)));
#pragma unroll
          for (int k = 0; k < 32; ++k)
            xs[32 * q + k] = (w >> k) & 1u ? xs[32 * q + k] : -INFINITY;
        }
      }
      float m4[4];   // four chains of maxima
#pragma unroll
      for (int q = 0; q < 4; ++q) m4[q] = fmaxf(xs[2 * q], xs[2 * q + 1]);
#pragma unroll
      for (int k = 8; k < 128; k += 8)
#pragma unroll
        for (int q = 0; q < 4; ++q)
          m4[q] = fmaxf(fmaxf(m4[q], xs[k + 2 * q]), xs[k + 2 * q + 1]);
      float mt = fmaxf(fmaxf(m4[0], m4[1]), fmaxf(m4[2], m4[3]));
      mt *= c;
      const float mn = fmaxf(m_ref, mt);
      const bool had = m_ref != -INFINITY;
      const bool need = had ? (mn > m_ref + kRescaleLog2) : (mn != -INFINITY);
      // O += P V of tile t-1 is done: P may be written again, O rescaled
      if (t > 0) {
        ok = wait_all(&s_pv_done[x], (t - 1) & 1, budget);
        if (!ok) break;
        tc_fence_after();
      }
      if (__any_sync(0xffffffffu, need && had)) {
        const float alpha = (need && had) ? exp2f(m_ref - mn) : 1.f;
#pragma unroll 1
        for (int cc = 0; cc < D / 16; ++cc) {
          uint32_t o[16];
          const uint32_t oc = lane_base + static_cast<uint32_t>(x * D) + 16 * cc;
          tmem_ld16(oc, o);
#pragma unroll
          for (int i = 0; i < 16; ++i) o[i] = __float_as_uint(__uint_as_float(o[i]) * alpha);
          tmem_st16(oc, o);
        }
      }
      if (need) {
        l = had ? l * exp2f(m_ref - mn) : 0.f;
        m_ref = mn;
      }
      const float mu = (m_ref == -INFINITY) ? 0.f : m_ref;
      // P = exp2(s c - m) as bf16 pairs
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        uint32_t pk[16];
        l += exp2_tile<32>(xs + 32 * q, c, mu, pk);
        tmem_st16u(pb + 16 * q, pk);
      }
      if (valid < kKeys && x == 0) {
        // ragged tile: V rows past the last valid key may hold anything; zero
        // them (once the tile has landed) so that 0 * V stays 0 for both tiles
        const int stage = t % S;
        if (!wait_all(&s_v_full[stage], (t / S) & 1, budget)) {
          ok = false;
          break;
        }
        uint8_t* vt = gbase + G::kVOff + stage * G::kKVTile;
        constexpr int kChunksPerRow = G::kNH * 8;
        for (int i = threadIdx.x - 128; i < (kKeys - valid) * kChunksPerRow; i += 128) {
          const int r = valid + i / kChunksPerRow, rem = i % kChunksPerRow;
          *reinterpret_cast<uint4*>(vt + (rem >> 3) * (kKeys * 128) + r * 128 + (rem & 7) * 16) =
              make_uint4(0u, 0u, 0u, 0u);
        }
        fence_proxy_async();
        // the four warps of tile A zero disjoint rows; each arrives for itself
      }
      tmem_wait_st();   // P is in place
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(smem_u32(&s_p_full[x]));
    }
    if (ok) {
      const int last = it.ntiles - 1;
      ok = wait_all(&s_pv_done[x], last & 1, budget) && !aborted_warp(&s_abort);
      if (ok) tc_fence_after();
    }
    if (!ok) {
      if (lane == 0) {
        note_timeout(p.status);
        s_abort = 1;
      }
    } else {
      // O_x / l -> the row's output, D columns
      const float inv = l > 0.f ? 1.f / l : 0.f;
      __nv_bfloat16* out = nullptr;
      if (mine) {
        const int q_row = it.r0 + rr;
        const int node = q_row / p.G;
        out = static_cast<__nv_bfloat16*>(p.out) +
              (static_cast<size_t>(it.s0 + node) * p.Hq + it.g * p.G + (q_row - node * p.G)) * D;
      }
#pragma unroll 1
      for (int cc = 0; cc < D / 32; ++cc) {
        float o[32];
        tmem_ld32(lane_base + static_cast<uint32_t>(x * D) + 32 * cc, o);
        if (mine) {
#pragma unroll
          for (int k = 0; k < 32; k += 8) {
            uint4 pk;
            __nv_bfloat162 h0 = __floats2bfloat162_rn(o[k] * inv, o[k + 1] * inv);
            __nv_bfloat162 h1 = __floats2bfloat162_rn(o[k + 2] * inv, o[k + 3] * inv);
            __nv_bfloat162 h2 = __floats2bfloat162_rn(o[k + 4] * inv, o[k + 5] * inv);
            __nv_bfloat162 h3 = __floats2bfloat162_rn(o[k + 6] * inv, o[k + 7] * inv);
            pk.x = *reinterpret_cast<uint32_t*>(&h0);
            pk.y = *reinterpret_cast<uint32_t*>(&h1);
            pk.z = *reinterpret_cast<uint32_t*>(&h2);
            pk.w = *reinterpret_cast<uint32_t*>(&h3);
            *reinterpret_cast<uint4*>(out + 32 * cc + k) = pk;
          }
        }
      }
    }
    }
  }

  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  if (warp == 2) tmem_dealloc(tmem, kTmemCols);
  pdl_wait();   // the next kernel's wait covers every earlier kernel
}

}  // namespace

size_t attention_tc_smem_bytes(int head_dim, bool pingpong) {
  if (pingpong)
    return 1024 + static_cast<size_t>(head_dim == 64 ? PPGeom<64>::kBytes : PPGeom<128>::kBytes);
  return 1024 + static_cast<size_t>(head_dim == 64 ? TcGeom<64>::kBytes : TcGeom<128>::kBytes);
}

// A pair of query tiles takes 1.7 times as long as one tile on another SM does
// (1.4 with small pages, where the copies of K and V count), so the line lies in
// the waves of CTAs: measured with 8 KV heads, G = 4, 152 SMs, one tile against
// two, contiguous unless said.
//   above 1.5 waves of pairs: 16 x 128 nodes 90.0 / 77.0 us, 24 x 128 133.6 /
//     114.6, 32 x 60 at contexts 1000-6000 136 / 124, 48 x 33 149.5 / 124.5
//   1 to 1.5 (three waves of single tiles against two of pairs): 12 x 128
//     68.0 / 75.7, pages of 64 75.0 / 77.5, of 32 79.9 / 77.7, of 16 90.1 / 78.2;
//     20 x 60 (160 pairs) with pages of 16 89 / 78, at contexts 1000-6000 113 / 89
//   up to 1: by the context lengths (attention_takes_pairs); below 5/6 of a wave the
//     single tiles' second wave is short: 15 ragged sequences of 20-100 nodes (0.78
//     of a wave) 54.0 / 63.7
//   128 rows per sequence or fewer leave the second tile empty: 128 x 20 nodes
//     153.8 / 157.6, 64 x 31 83.6 / 84.5; 257 to 384 rows make 3 tiles but 2 pairs
//     (4 KV heads, G = 7): 32 x 40 71.1 / 86.2, 64 x 40 136.4 / 138.9
// Pairs are counted for sequences of the average size; two waves of all rows are
// enough whatever the sizes.
PairRule attention_pair_rule(int batch, int num_kv_heads, int G, int total_nodes, int page_size,
                             int nsm) {
  const long long rows = static_cast<long long>(total_nodes) * G;
  if (batch <= 0 || rows <= static_cast<long long>(batch) * kRows) return PairRule::kOneTile;
  const long long heads = num_kv_heads;
  const long long least = heads * ((rows + kPPRows - 1) / kPPRows);
  if (least >= 2LL * nsm) return PairRule::kPairs;
  const long long avg = (rows + batch - 1) / batch;
  const long long pairs = heads * batch * ((avg + kPPRows - 1) / kPPRows);
  const long long tiles = heads * batch * ((avg + kRows - 1) / kRows);
  const bool small = page_size > 0 && page_size <= 32;
  if (10 * tiles < (small ? 14 : 17) * pairs || 6 * least < 5LL * nsm) return PairRule::kOneTile;
  if (pairs <= nsm) return batch <= kPairSeqs ? PairRule::kByContext : PairRule::kOneTile;
  return small || 2 * least > 3LL * nsm ? PairRule::kPairs : PairRule::kOneTile;
}

float attention_pair_ratio(int page_size) {
  // a key tile of the one-tile form over a pair's (attention_takes_pairs)
  return page_size == 0 ? 0.56f : page_size >= 32 ? 0.65f : 0.75f;
}

bool attention_q_tma_ok(int G) { return G >= 1 && kRows % G == 0; }

cudaError_t launch_attention_tc(const AttnParams& p, const CUtensorMap& tm_k,
                                const CUtensorMap& tm_v, const CUtensorMap& tm_tk,
                                const CUtensorMap& tm_tv, const CUtensorMap& tm_q, bool pingpong,
                                cudaStream_t s) {
  const size_t smem = attention_tc_smem_bytes(p.D, pingpong);
  if (p.D != 64 && p.D != 128) return cudaErrorInvalidValue;
  cudaError_t err;
  // row blocks: at most max_nodes * G rows of each of B sequences (index order, B >
  // kOrderMax, numbers these; the ping-pong form's sequences are large, so that few
  // of them lie idle), and T * G rows of which every sequence may leave one block
  // ragged (sequences that overlap can make more: items_past_grid)
  const int rows = pingpong ? kPPRows : kRows;
  const long long full = static_cast<long long>((p.max_nodes * p.G + rows - 1) / rows) * p.B;
  const long long blocks =
      p.B > kOrderMax || pingpong
          ? full
          : std::min(full, static_cast<long long>(p.T) * p.G / rows + p.B);
  const long long ctas =
      std::max<long long>(blocks * p.Hkv, p.part_cap > 0 ? p.nsm : 0);
  if (ctas > 0x7fffffffLL) return cudaErrorInvalidValue;
  const bool d64 = p.D == 64, by_context = p.pair_ratio > 0.f;
  auto* k = d64 ? attn_tc_kernel<64, kPlain> : attn_tc_kernel<128, kPlain>;
  if (pingpong)
    k = by_context ? (d64 ? attn_pp_kernel<64, kByContext> : attn_pp_kernel<128, kByContext>)
                   : (d64 ? attn_pp_kernel<64, kPlain> : attn_pp_kernel<128, kPlain>);
  else if (by_context)
    k = d64 ? attn_tc_kernel<64, kByContext> : attn_tc_kernel<128, kByContext>;
  else if (p.p_two)
    k = d64 ? attn_tc_kernel<64, kTwoTerms> : attn_tc_kernel<128, kTwoTerms>;
  err = set_smem_attrs(k, smem);
  if (err != cudaSuccess) return err;
  err = launch_pdl(k, dim3(static_cast<unsigned>(ctas)), dim3(kThreads), smem, s, tm_k, tm_v, tm_tk,
                   tm_tv, tm_q, p);
  if (err != cudaSuccess || p.part_cap == 0) return err;
  const bool few = static_cast<long long>(p.T) * p.Hq <= kMergeFewRows;
  const int mrows = kMergeThreads / 32 / (few ? 4 : 1);
  const dim3 mgrid((p.max_nodes * p.G + mrows - 1) / mrows, p.B * p.Hkv);
  auto* merge = p.D == 64 ? (few ? attn_merge_kernel<64, 4> : attn_merge_kernel<64, 1>)
                          : (few ? attn_merge_kernel<128, 4> : attn_merge_kernel<128, 1>);
  return launch_pdl(merge, mgrid, dim3(kMergeThreads), 0, s, p);
}

long long attention_split_rows(const asd_dims& d, int total_nodes, int nsm) {
  // worth its plan and merge kernel only while the unsplit items leave a
  // quarter of the SMs idle; the device decides from the context lengths.
  // (Allowed for 128 items on 152 SMs, which an even batch cannot split, the
  // step of 8 sequences at context 16384 took 584 us instead of 580; for 256
  // items, 32 ragged sequences took 128.5 us instead of 121.)
  const long long G = d.num_q_heads / d.num_kv_heads;
  const long long blocks = std::max<long long>(d.batch, total_nodes * G / kRows);
  if (d.batch > kOrderMax || 4 * d.num_kv_heads * blocks > 3LL * nsm || d.ctx_max < 2 * kKeys)
    return 0;
  return static_cast<long long>(nsm) * std::min<long long>(kRows, d.max_nodes * G);
}

}  // namespace asd

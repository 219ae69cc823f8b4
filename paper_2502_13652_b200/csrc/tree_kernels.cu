// Per-sequence kernels: classification and pruning of a level, the Top-N rerank, the
// verification inputs and the acceptance walk.  One CTA per sequence; all of this is
// O(F*K) or O(tree) work per sequence, done in double precision where it is floating point.
#include <string.h>

#include "c2t_internal.h"
#include "level_prune.cuh"

namespace c2t {
namespace {

constexpr int kTreeThreads = 512;
constexpr int kTreeWarps = kTreeThreads / 32;
constexpr unsigned kFull = 0xFFFFFFFFu;

__global__ void begin_step_kernel(TreeState t, const int32_t *root_tok, const int32_t *prefix_len) {
  chain_enter();
  const int b = blockIdx.x * blockDim.x + threadIdx.x;
  if (b >= t.B) return;
  const size_t o = (size_t)b * t.cap;
  t.tree_n[b] = 1;
  t.tree_token[o] = root_tok[b];
  t.tree_parent[o] = -1;
  t.tree_level[o] = 0;
  t.tree_logP[o] = 0.0;
  t.tree_C[o] = 1.0;
  t.tree_Chat[o] = INFINITY;
  t.frontier_n[0][b] = 1;
  t.frontier_n[1][b] = 0;
  t.frontier_node[0][(size_t)b * t.F] = 0;
  t.frontier_logP[0][(size_t)b * t.F] = 0.0;
  t.frontier_chat[0][(size_t)b * t.F] = INFINITY;
  t.cand_n[b] = 0;
  t.final_n[b] = 0;
  t.root_tok[b] = root_tok[b];
  t.prefix_len[b] = prefix_len[b];
  t.status[b] = 0u;
}

// The record of every active row of the last (sharded) expand pass, for c2t_export_row_records: a warp per row.
constexpr int kExportWarps = 4;
__global__ void __launch_bounds__(kExportWarps * 32) export_rows_kernel(TreeState t, int level, int tok_base, c2t_row_record *out) {
  chain_enter();
  const int lane = threadIdx.x & 31;
  const long long i = (long long)blockIdx.x * kExportWarps + (threadIdx.x >> 5);
  if (i >= (long long)t.B * t.F) return;
  const int b = (int)(i / t.F), j = (int)(i % t.F);
  const int n = t.frontier_n[level & 1][b];
  const RowResult r = t.rows[i];                     // (loads issued together; rows past n hold anything)
  const unsigned long long key = lane < t.K ? t.row_keys[i * t.K + lane] : 0ull;
  if (j >= n) return;
  c2t_row_record *o = out + i;
  if (lane < t.K) {
    o->x[lane] = key ? key_value(key) : -INFINITY;
    o->tok[lane] = key ? key_token(key) + tok_base : -1;
  }
  if (lane == 0) {
    o->M = r.M; o->S = r.S; o->T = r.T;
    o->n = r.n_valid;
    o->fault = r.fault;
  }
}

// ROUNDS: candidates of a thread at most; GATHERED: the rows come from gathered records of n_shards shards, not from this context's own
// expand pass
template <int ROUNDS, bool GATHERED>
__global__ void __launch_bounds__(kTreeThreads) prune_level_kernel(TreeState t, int level, c2t_frontier out,
                                                                   const c2t_row_record *records, int n_shards) {
  extern __shared__ __align__(16) unsigned char s_prune[];
  __shared__ __align__(16) double s_w[kWCount];
  PruneShared &sh = *reinterpret_cast<PruneShared *>(s_prune);
  GatherShared *gs = reinterpret_cast<GatherShared *>(s_prune + sizeof(PruneShared));
  chain_release();
  stage_classifier(t, s_w, threadIdx.x, kTreeThreads);   // (written at init, not by the chain: while the expand pass is finishing)
  chain_wait();
  prune_level_body<kTreeThreads, ROUNDS, GATHERED>(t, level, out, records, n_shards, blockIdx.x, sh, s_w, gs);
}
constexpr int kPruneRounds = kMaxCand / kTreeThreads;

// ---------------------------------------------------------------- rerank ----

// Top-N rerank (Sec. 2.2): root + the N-1 nodes first under (Chat desc, id asc), renumbered
// in id order.  Chat never exceeds the parent's and parents have lower ids, so the kept set
// is closed under "parent of".  A chain of dependent steps: the tree is fetched into shared memory in one go, the scores as
// orderable integers.  Up to kRankNodes nodes a warp ranks a node against 32 others at a time; beyond that the work of
// all pairs is the longer way (511 nodes: 30.9 us) and the cut is searched by its bits, one count of the whole tree per bit.
constexpr int kRankNodes = 192;
__global__ void __launch_bounds__(kTreeThreads) final_prune_kernel(TreeState t) {
  extern __shared__ unsigned long long s_score[];              // [cap], behind it [cap] parents, [cap] new ids
  __shared__ int s_count[kTreeWarps];
  __shared__ unsigned long long s_and, s_or;
  int *s_parent = reinterpret_cast<int *>(s_score + t.cap), *s_remap = s_parent + t.cap;
  chain_enter();
  const int b = blockIdx.x, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const size_t tb = (size_t)b * t.cap, fb = (size_t)b * t.Nw;
  int n = t.tree_n[b];
  int token = 0, level = 0;                                    // of node tid
  if (tid < t.cap) { token = t.tree_token[tb + tid]; level = t.tree_level[tb + tid]; }
  for (int i = tid; i < t.cap; i += kTreeThreads) {            // (past n: anything, unused)
    const unsigned long long cb = (unsigned long long)__double_as_longlong(t.tree_Chat[tb + i]);
    s_score[i] = cb ^ ((cb >> 63) ? ~0ull : 0x8000000000000000ull);
    s_parent[i] = t.tree_parent[tb + i];
  }
  n = n > t.cap ? t.cap : n;
  __syncthreads();
  const bool all = (t.N <= 0 || n <= t.N);
  if (!all && n > kRankNodes) {
    // the (N-1)-th largest score by its bits, from the highest in which the scores differ down, until a count fits exactly
    // (equal scores at the cut: the lower ids)
    const int quota = t.N - 1;
    if (tid == 0) { s_and = ~0ull; s_or = 0ull; }
    __syncthreads();
    unsigned long long al = ~0ull, ol = 0ull;
    for (int i = 1 + tid; i < n; i += kTreeThreads) { al &= s_score[i]; ol |= s_score[i]; }
    atomicAnd(&s_and, al);
    atomicOr(&s_or, ol);
    __syncthreads();
    const unsigned long long common = s_and, differ = common ^ s_or;
    int bit = differ ? 63 - __clzll((long long)differ) : -1;
    unsigned long long cutoff = bit >= 63 ? 0ull : common & ~((1ull << (bit + 1)) - 1ull);
    if (bit < 0) cutoff = common;
    bool exact = false;
    for (; bit >= 0 && !exact; --bit) {
      const unsigned long long trial = cutoff | (1ull << bit);
      int reach = 0;
      for (int base = 0; base < n; base += kTreeThreads) {
        const int i = base + tid;
        reach += __syncthreads_count(i > 0 && i < n && s_score[i] >= trial);
      }
      if (reach >= quota) cutoff = trial;
      exact = reach == quota;
    }
    int ties = n;                                              // nodes with the cutoff's score that may stay
    if (!exact) {
      ties = quota;
      for (int base = 0; base < n; base += kTreeThreads) {
        const int i = base + tid;
        ties -= __syncthreads_count(i > 0 && i < n && s_score[i] > cutoff);
      }
    }
    int seen = 0;
    for (int base = 0; base < n; base += kTreeThreads) {
      const int i = base + tid;
      const bool tie = i > 0 && i < n && s_score[i] == cutoff;
      const unsigned mask = __ballot_sync(kFull, tie);
      if (lane == 0) s_count[warp] = __popc(mask);
      __syncthreads();
      const int c = lane < kTreeWarps ? s_count[lane] : 0;
      const int before = seen + __reduce_add_sync(kFull, lane < warp ? c : 0) + __popc(mask & ((1u << lane) - 1u));
      if (i < n) s_remap[i] = i == 0 || s_score[i] > cutoff || (tie && before < ties);
      seen += __reduce_add_sync(kFull, c);
      __syncthreads();
    }
  } else if (!all) {
    for (int i = warp; i < n; i += kTreeWarps) {               // 1: kept (for now)
      const unsigned long long mine = s_score[i];
      int before = 0;
#pragma unroll 4
      for (int o = lane; o < n; o += 32) {
        const unsigned long long other = s_score[o];
        before += o > 0 && (other > mine || (other == mine && o < i));
      }
      before = __reduce_add_sync(kFull, before);
      if (lane == 0) s_remap[i] = i == 0 || before < t.N - 1;
    }
    __syncthreads();
  }
  int run = 0;                                                 // nodes kept below the chunk
  for (int base = 0; base < n; base += kTreeThreads) {
    const int i = base + tid;
    const bool keep = i < n && (all || s_remap[i]);
    const unsigned mask = __ballot_sync(kFull, keep);
    if (lane == 0) s_count[warp] = __popc(mask);
    __syncthreads();
    const int c = lane < kTreeWarps ? s_count[lane] : 0;
    const int before = __reduce_add_sync(kFull, lane < warp ? c : 0);
    if (i < n) s_remap[i] = keep ? run + before + __popc(mask & ((1u << lane) - 1u)) : -1;
    run += __reduce_add_sync(kFull, c);
    __syncthreads();
  }
  const int n_final = run > t.Nw ? t.Nw : run;
  for (int i = tid; i < n; i += kTreeThreads) {
    const int m = s_remap[i];
    if (m < 0 || m >= t.Nw) continue;
    const int par = s_parent[i];
    t.final_src[fb + m] = i;
    t.final_token[fb + m] = i == tid ? token : t.tree_token[tb + i];
    t.final_parent[fb + m] = par < 0 ? -1 : s_remap[par];
    t.final_level[fb + m] = i == tid ? level : t.tree_level[tb + i];
  }
  for (int m = n_final + tid; m < t.Nw; m += kTreeThreads) {
    t.final_src[fb + m] = -1;
    t.final_token[fb + m] = 0;
    t.final_parent[fb + m] = -1;
    t.final_level[fb + m] = 0;
  }
  if (tid == 0) t.final_n[b] = n_final;
}

// ---------------------------------------------------------------- verify ----

// The tree is fetched into shared memory in one go; ancestors are found there.
__global__ void __launch_bounds__(kTreeThreads) build_verify_kernel(TreeState t, c2t_verify out) {
  extern __shared__ int s_verify[];                            // [Nw] parents, [Nw] levels, [Nw] has-child
  __shared__ int s_count[kTreeWarps];
  chain_enter();
  const int b = blockIdx.x, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int n = t.final_n[b], Nw = t.Nw, W = t.W, width = t.D + 1;
  const int prefix = t.prefix_len[b];
  const size_t fb = (size_t)b * Nw;
  int *parent = s_verify, *level = s_verify + Nw, *has_child = s_verify + 2 * Nw;
  for (int i = tid; i < Nw; i += kTreeThreads) {               // (past n: parent -1, level and token 0)
    parent[i] = t.final_parent[fb + i];
    level[i] = t.final_level[fb + i];
    has_child[i] = 0;
    if (out.tokens) out.tokens[fb + i] = t.final_token[fb + i];
  }
  if (out.retrieve)
    for (int k = tid; k < Nw * width; k += kTreeThreads) out.retrieve[fb * width + k] = -1;
  __syncthreads();
  for (int i = tid; i < n; i += kTreeThreads)
    if (parent[i] >= 0) has_child[parent[i]] = 1;
  for (int i = tid; i < Nw; i += kTreeThreads) {
    if (out.parents) out.parents[fb + i] = parent[i];
    if (out.position_ids) out.position_ids[fb + i] = i < n ? prefix + level[i] : 0;
  }
  if (out.mask_bits) {
    for (int k = tid; k < Nw * W; k += kTreeThreads) {         // a thread per word
      const int i = k / W, w = k - i * W;
      unsigned long long bits = 0ull;
      if (i < n)
        for (int a = i, g = 0; a >= 0 && g <= t.D + 1; a = parent[a], ++g)
          if ((a >> 6) == w) bits |= 1ull << (a & 63);
      out.mask_bits[fb * W + k] = bits;
    }
  }
  __syncthreads();
  // leaves in ascending id order
  int run = 0;
  for (int base = 0; base < n; base += kTreeThreads) {
    const int i = base + tid;
    const bool leaf = i < n && !has_child[i];
    const unsigned mask = __ballot_sync(kFull, leaf);
    if (lane == 0) s_count[warp] = __popc(mask);
    __syncthreads();
    const int c = lane < kTreeWarps ? s_count[lane] : 0;
    const int at = run + __reduce_add_sync(kFull, lane < warp ? c : 0) + __popc(mask & ((1u << lane) - 1u));
    if (leaf && out.retrieve) {
      int32_t *row = out.retrieve + (fb + at) * width;
      for (int a = i, g = 0; a >= 0 && g <= t.D + 1; a = parent[a], ++g) {
        const int l = level[a];
        if (l >= 0 && l < width) row[l] = a;
      }
    }
    run += __reduce_add_sync(kFull, c);
    __syncthreads();
  }
  if (tid == 0) {
    if (out.n_nodes) out.n_nodes[b] = n;
    if (out.n_leaves) out.n_leaves[b] = run;
  }
}

// ---------------------------------------------------------------- accept ----

// takes a key of the last arg-max pass (0: none) and leaves the zero that the next pass starts from
__device__ __forceinline__ unsigned long long take_best(const TreeState &t, size_t slot) {
  const unsigned long long best = t.best[slot];
  if (best) t.best[slot] = 0ull;
  return best;
}

// The best key of every final node's row over one token range, token ids made global, for c2t_argmax_shard.
__global__ void __launch_bounds__(kTreeThreads) export_best_kernel(TreeState t, int tok_base, unsigned long long *out) {
  chain_enter();
  const size_t i = (size_t)blockIdx.x * kTreeThreads + threadIdx.x;
  if (i >= (size_t)t.B * t.Nw) return;
  const unsigned long long best = take_best(t, i);             // (nodes that do not exist have none)
  out[i] = best ? (best & 0xFFFFFFFF00000000ull) | (0xFFFFFFFFu - (uint32_t)(key_token(best) + tok_base)) : 0ull;
}

// gathered == nullptr: the arg-max of this context's own pass; else the best of n_shards gathered keys per node.
// The tree and the nodes' arg-maxes meet in shared memory, where every node looks for the child that carries its token, so
// that the walk itself is a chain of one load per step.
__global__ void __launch_bounds__(kTreeThreads) accept_walk_kernel(TreeState t, c2t_accept_out out,
                                                                   const unsigned long long *gathered, int n_shards) {
  extern __shared__ int s_walk[];                              // [Nw] arg-maxes, [Nw] the child to go to
  chain_enter();
  const int b = blockIdx.x, tid = threadIdx.x;
  const int n = t.final_n[b], Nw = t.Nw, width = t.D + 1;
  const size_t fb = (size_t)b * Nw;
  int *want = s_walk, *next = s_walk + Nw;
  int parent = -1, token = 0;                                  // of node 1 + tid
  if (1 + tid < Nw) { parent = t.final_parent[fb + 1 + tid]; token = t.final_token[fb + 1 + tid]; }
  if (out.path)
    for (int k = tid; k < width; k += kTreeThreads) out.path[(size_t)b * width + k] = k == 0 ? 0 : -1;
  for (int i = tid; i < Nw; i += kTreeThreads) {
    unsigned long long best = 0ull;
    if (gathered) {                                 // equal logits in two shards: the larger key is the lower token id
#pragma unroll 4
      for (int s = 0; s < n_shards; ++s) {
        const unsigned long long k = gathered[((size_t)s * t.B + b) * Nw + i];
        best = k > best ? k : best;
      }
    } else {
      best = take_best(t, fb + i);
    }
    const int tok = best && i < n ? key_token(best) : -1;
    want[i] = tok;
    next[i] = 0x7FFFFFFF;
    t.node_argmax[fb + i] = tok;
  }
  __syncthreads();
  for (int c = 1 + tid; c < n; c += kTreeThreads) {
    if (c != 1 + tid) { parent = t.final_parent[fb + c]; token = t.final_token[fb + c]; }
    if (parent >= 0 && token == want[parent]) atomicMin(&next[parent], c);
  }
  __syncthreads();
  if (tid != 0) return;
  int cur = 0, len = 0;
  while (n > 0 && len + 1 < width) {
    const int found = next[cur];
    if (found == 0x7FFFFFFF) break;
    cur = found;
    ++len;
    if (out.path) out.path[(size_t)b * width + len] = cur;
  }
  if (out.accept_len) out.accept_len[b] = len;
  if (out.next_token) out.next_token[b] = n > 0 ? want[cur] : -1;
}

// ---------------------------------------------------------------- dense mask -

// Four rows of a sequence's final tree per CTA, two warps per row.  Most of a row does not depend on the tree (its
// prefix, and what lies behind the tree), and is stored first, 16 bytes at a time; then the row's ancestor-or-self set (Sec. 2.2)
// is found by a walk up the parent pointers in shared memory (at most D+1 steps; through global memory it costs
// microseconds), and the few vectors that hold tree nodes follow.  Bound by the stores: 64 x 60 rows of 4160 bf16
// values 26.6 -> 9.8 us per call (32 MB).
constexpr int kMaskRows = 4, kMaskThreads = kMaskRows * 64;
template <typename T>
__global__ void __launch_bounds__(kMaskThreads) dense_mask_kernel(TreeState t, T *out, long long kv_len, T ninf) {
  extern __shared__ int s_parent[];                  // [Nw], behind it the rows' bits
  constexpr int E = 16 / sizeof(T);
  const int b = blockIdx.y, tid = threadIdx.x, r = tid >> 6, k0 = tid & 63, i = (int)blockIdx.x * kMaskRows + r;
  const int Nw = t.Nw, words = (Nw + 31) / 32;
  unsigned *bits = reinterpret_cast<unsigned *>(s_parent + Nw) + r * words;
  chain_enter();
  const long long prefix = t.prefix_len[b];
  const int n = t.final_n[b];
  for (int j = tid; j < Nw; j += kMaskThreads) s_parent[j] = t.final_parent[(size_t)b * Nw + j];
  for (int w = k0; w < words; w += 64) bits[w] = 0u;
  T *row = out + ((size_t)b * Nw + i) * kv_len;
  long long head = (long long)((16 - (reinterpret_cast<uintptr_t>(row) & 15)) & 15) / (int)sizeof(T);     // up to the first 16-byte boundary
  head = head < kv_len ? head : kv_len;
  const long long body = (kv_len - head) / E;
  uint4 *dst = reinterpret_cast<uint4 *>(row + head);
  // vectors [0, k1) lie in the prefix, [k2, body) behind the tree
  long long k1 = prefix > head ? (prefix - head) / E : 0, k2 = prefix + Nw > head ? (prefix + Nw - head + E - 1) / E : 0;
  k1 = k1 < body ? k1 : body;
  k2 = k2 < body ? k2 : body;
  union { uint4 v; T e[E]; } fill, mixed;
  if (i < Nw) {
#pragma unroll 4
    for (long long k = k0; k < k1; k += 64) dst[k] = make_uint4(0u, 0u, 0u, 0u);
#pragma unroll
    for (int q = 0; q < E; ++q) fill.e[q] = ninf;
#pragma unroll 4
    for (long long k = k2 + k0; k < body; k += 64) dst[k] = fill.v;
  }
  __syncthreads();
  if (k0 == 0 && i < n)
    for (int j = i, guard = 0; j >= 0 && j < Nw && guard <= Nw; j = s_parent[j], ++guard) bits[j >> 5] |= 1u << (j & 31);
  __syncthreads();
  if (i >= Nw) return;
  auto value = [&](long long c) -> T {
    const long long j = c - prefix;
    return c < prefix || (j < Nw && ((bits[j >> 5] >> (j & 31)) & 1u)) ? (T)0 : ninf;
  };
  for (long long k = k1 + k0; k < k2; k += 64) {
#pragma unroll
    for (int q = 0; q < E; ++q) mixed.e[q] = value(head + k * E + q);
    dst[k] = mixed.v;
  }
  if (k0 < head) row[k0] = value(k0);
  const long long done = head + body * E;
  if (k0 < kv_len - done) row[done + k0] = value(done + k0);
}

// ---------------------------------------------------------------- lazy walk --

// One round of the acceptance walk over target rows sharded over the vocabulary, reading only the rows it visits (Sec. 5
// Metrics).  Round 0 puts every sequence with a tree on its root.  Round r > 0 takes the best of the n_shards gathered keys
// per sequence ([n_shards, B], one key for the sequence's current node, 0 for a sequence that has stopped): the
// sequence moves to the child that carries that token, or stops.  A thread per sequence.
constexpr int kWalkThreads = 128;
__global__ void __launch_bounds__(kWalkThreads) lazy_walk_round_kernel(TreeState t, int round, c2t_accept_out out,
                                                                       const unsigned long long *gathered, int n_shards) {
  chain_enter();
  const int b = blockIdx.x * kWalkThreads + threadIdx.x;
  const int Nw = t.Nw, width = t.D + 1;
  if (b >= t.B) return;
  const size_t fb = (size_t)b * Nw;
  const int n = t.final_n[b];
  if (round == 0) {
    for (int i = 0; i < Nw; ++i) t.node_argmax[fb + i] = -1;
    if (out.path)
      for (int w = 0; w < width; ++w) out.path[(size_t)b * width + w] = w == 0 ? 0 : -1;
    t.walk_cur[b] = 0;
    t.walk_len[b] = 0;
    t.walk_active[b] = n > 0;
    if (n <= 0) {
      if (out.accept_len) out.accept_len[b] = 0;
      if (out.next_token) out.next_token[b] = -1;
    }
    return;
  }
  if (!t.walk_active[b]) return;
  unsigned long long best = 0ull;                      // equal logits in two shards: the larger key is the lower token id
#pragma unroll 4
  for (int sh = 0; sh < n_shards; ++sh) {
    const unsigned long long k = gathered[(size_t)sh * t.B + b];
    best = k > best ? k : best;
  }
  const int want = best ? key_token(best) : -1;
  int cur = t.walk_cur[b], len = t.walk_len[b];
  t.node_argmax[fb + cur] = want;
  int found = -1;
  if (len + 1 < width)
    for (int c = cur + 1; c < n; ++c)
      if (t.final_parent[fb + c] == cur && t.final_token[fb + c] == want) { found = c; break; }
  if (found >= 0) {
    ++len;
    t.walk_cur[b] = found;
    t.walk_len[b] = len;
    if (out.path) out.path[(size_t)b * width + len] = found;
  } else {
    t.walk_active[b] = 0;
    if (out.accept_len) out.accept_len[b] = len;
    if (out.next_token) out.next_token[b] = want;
  }
}

// After an arg-max pass over one token range of the walking sequences' current rows: per sequence the best key of
// that range with the token id made global (0 for a sequence that has stopped), for c2t_lazy_argmax_shard.
__global__ void __launch_bounds__(kWalkThreads) export_lazy_best_kernel(TreeState t, int tok_base, unsigned long long *out) {
  chain_enter();
  const int b = blockIdx.x * kWalkThreads + threadIdx.x;
  if (b >= t.B) return;
  const unsigned long long best = take_best(t, b);
  out[b] = best ? (best & 0xFFFFFFFF00000000ull) | (0xFFFFFFFFu - (uint32_t)(key_token(best) + tok_base)) : 0ull;
}

}  // namespace

cudaError_t launch_dense_mask(const TreeState &t, void *out, int out_dtype, int64_t kv_len, cudaStream_t s) {
  const dim3 grid((t.Nw + kMaskRows - 1) / kMaskRows, t.B);
  const size_t smem = (size_t)t.Nw * sizeof(int) + (size_t)kMaskRows * ((t.Nw + 31) / 32) * sizeof(unsigned);    // (at most 40 KB)
  if (out_dtype == C2T_F32)                          // the values as raw words: +0 and -inf
    return launch_chained(dense_mask_kernel<unsigned>, grid, dim3(kMaskThreads), smem, s, t, reinterpret_cast<unsigned *>(out),
                          (long long)kv_len, 0xFF800000u);
  return launch_chained(dense_mask_kernel<unsigned short>, grid, dim3(kMaskThreads), smem, s, t, reinterpret_cast<unsigned short *>(out),
                        (long long)kv_len, (unsigned short)0xFF80);
}

cudaError_t launch_lazy_walk_round(const TreeState &t, int round, const c2t_accept_out *out,
                                   const unsigned long long *gathered, int n_shards, cudaStream_t s) {
  c2t_accept_out o;
  memset(&o, 0, sizeof o);
  if (out) o = *out;
  return launch_chained(lazy_walk_round_kernel, dim3((t.B + kWalkThreads - 1) / kWalkThreads), dim3(kWalkThreads), 0, s, t, round, o, gathered, n_shards);
}

cudaError_t launch_export_lazy_best(const TreeState &t, int vocab_begin, unsigned long long *out, cudaStream_t s) {
  return launch_chained(export_lazy_best_kernel, dim3((t.B + kWalkThreads - 1) / kWalkThreads), dim3(kWalkThreads), 0, s, t, vocab_begin, out);
}

cudaError_t launch_begin_step(const TreeState &t, const int32_t *root_tok, const int32_t *prefix_len,
                              cudaStream_t s) {
  return launch_chained(begin_step_kernel, dim3((t.B + 127) / 128), dim3(128), 0, s, t, root_tok, prefix_len);
}

cudaError_t launch_export_rows(const TreeState &t, int level, int vocab_begin, c2t_row_record *out, cudaStream_t s) {
  const long long rows = (long long)t.B * t.F;
  return launch_chained(export_rows_kernel, dim3((unsigned)((rows + kExportWarps - 1) / kExportWarps)), dim3(kExportWarps * 32), 0, s,
                        t, level, vocab_begin, out);
}

cudaError_t launch_prune_level(const TreeState &t, int level, const c2t_frontier *out, const c2t_row_record *records,
                               int n_shards, cudaStream_t s) {
  c2t_frontier o = {nullptr, nullptr, nullptr, nullptr};
  if (out) o = *out;
  const bool small = t.F * t.K <= kTreeThreads;
  const auto kernel = records ? (small ? prune_level_kernel<1, true> : prune_level_kernel<kPruneRounds, true>)
                              : (small ? prune_level_kernel<1, false> : prune_level_kernel<kPruneRounds, false>);
  return launch_chained(kernel, dim3(t.B), dim3(kTreeThreads), sizeof(PruneShared) + (records ? sizeof(GatherShared) : 0),
                        s, t, level, o, records, n_shards);
}

// dynamic shared memory: up to 128 KB for the rerank of the largest tree
static size_t final_smem(int cap) { return (size_t)cap * (sizeof(unsigned long long) + 2 * sizeof(int)); }

cudaError_t prepare_tree_kernels() {
  const int gather = (int)(sizeof(PruneShared) + sizeof(GatherShared));
  cudaError_t e = cudaFuncSetAttribute(prune_level_kernel<1, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, gather);
  if (e == cudaSuccess) e = cudaFuncSetAttribute(prune_level_kernel<kPruneRounds, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, gather);
  if (e == cudaSuccess) e = cudaFuncSetAttribute(final_prune_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)final_smem(C2T_MAX_TREE));
  if (e == cudaSuccess) e = cudaFuncSetAttribute(build_verify_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, 3 * C2T_MAX_TREE * (int)sizeof(int));
  if (e == cudaSuccess) e = cudaFuncSetAttribute(accept_walk_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, 2 * C2T_MAX_TREE * (int)sizeof(int));
  return e;
}

cudaError_t launch_final_prune(const TreeState &t, cudaStream_t s) {
  return launch_chained(final_prune_kernel, dim3(t.B), dim3(kTreeThreads), final_smem(t.cap), s, t);
}

cudaError_t launch_build_verify(const TreeState &t, const c2t_verify *out, cudaStream_t s) {
  c2t_verify o = {nullptr, nullptr, nullptr, nullptr, nullptr, nullptr, nullptr};
  if (out) o = *out;
  return launch_chained(build_verify_kernel, dim3(t.B), dim3(kTreeThreads), 3 * (size_t)t.Nw * sizeof(int), s, t, o);
}

cudaError_t launch_export_best(const TreeState &t, int vocab_begin, unsigned long long *out, cudaStream_t s) {
  return launch_chained(export_best_kernel, dim3((unsigned)(((size_t)t.B * t.Nw + kTreeThreads - 1) / kTreeThreads)), dim3(kTreeThreads), 0, s, t, vocab_begin, out);
}

cudaError_t launch_accept_walk(const TreeState &t, const c2t_accept_out *out, const unsigned long long *gathered,
                               int n_shards, cudaStream_t s) {
  c2t_accept_out o = {nullptr, nullptr, nullptr};
  if (out) o = *out;
  return launch_chained(accept_walk_kernel, dim3(t.B), dim3(kTreeThreads), 2 * (size_t)t.Nw * sizeof(int), s, t, o, gathered, n_shards);
}

}  // namespace c2t

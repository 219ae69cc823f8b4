// Internal declarations shared by the CUDA translation units of libc2t.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "c2t.h"

namespace c2t {

// ---------------------------------------------------------------- keys ------
// Total order used everywhere a "largest logit, then lowest token id" decision is taken:
// key = (orderable(value) << 32) | (0xFFFFFFFF - token).  A larger key wins.  0 = empty.

__host__ __device__ __forceinline__ uint32_t f32_orderable(uint32_t bits) {
  return bits ^ ((bits & 0x80000000u) ? 0xFFFFFFFFu : 0x80000000u);
}
__host__ __device__ __forceinline__ uint32_t f32_from_orderable(uint32_t o) {
  return o ^ ((o & 0x80000000u) ? 0x80000000u : 0xFFFFFFFFu);
}
__device__ __forceinline__ unsigned long long make_key(float x, uint32_t tok) {
  return ((unsigned long long)f32_orderable(__float_as_uint(x)) << 32) | (0xFFFFFFFFu - tok);
}
__device__ __forceinline__ float key_value(unsigned long long k) {
  return __uint_as_float(f32_from_orderable((uint32_t)(k >> 32)));
}
__device__ __forceinline__ int32_t key_token(unsigned long long k) {
  return (int32_t)(0xFFFFFFFFu - (uint32_t)k);
}

// Logits of -inf (and anything below -2^127) are read as -2^127, so that "probability zero"
// never produces inf - inf or 0 * inf in the running sums.
constexpr float kNegInfAsFinite = -1.7e38f;   // anything at or below this was -inf (or as good as)

// ---------------------------------------------------------------- index checks
// A build with -DC2T_DEBUG_BOUNDS checks the indices of the kernels' writes to shared memory queues, pools and
// workspace records: a failed check sets C2T_ST_INTERNAL in the given status word (if there is one) and the guarded
// access is skipped.  It stands in for a memory checker where none can be run.  In a normal build the check is the
// constant `true`.
#ifdef __CUDACC__
#ifdef C2T_DEBUG_BOUNDS
__device__ __forceinline__ bool c2t_in_bounds(unsigned long long i, unsigned long long n, uint32_t *status) {
  if (i < n) return true;
  if (status) atomicOr(status, (uint32_t)C2T_ST_INTERNAL);
  return false;
}
#define C2T_IN_BOUNDS(i, n, status) c2t_in_bounds((unsigned long long)(i), (unsigned long long)(n), (status))
#else
#define C2T_IN_BOUNDS(i, n, status) true
#endif
#endif

// ---------------------------------------------------------------- launch chain
// The kernels of a decode step form a chain in which each one consumes what the one before wrote.
// They are launched with programmatic stream serialisation: the next kernel's CTAs may be placed
// on SMs (and its launch latency paid) while the previous kernel is still finishing.  Every kernel
// of the chain therefore starts with chain_enter(): it lets its own successor be scheduled and then
// waits until the predecessor has completed and its writes are visible.  Nothing touches global
// memory before that, so the chain behaves exactly like plain stream order.  One exception: the pruning
// kernels read the classifier's weights before they wait.  That is sound only because c2t_init writes
// the weights, waits for them, and nothing changes them afterwards.
#ifdef __CUDACC__
__device__ __forceinline__ void chain_release() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void chain_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void chain_enter() {
  chain_release();
  chain_wait();
}

template <typename... KArgs, typename... Args>
cudaError_t launch_chained(void (*kernel)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t s,
                           Args &&...args) {
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
  return cudaLaunchKernelEx(&cfg, kernel, KArgs(args)...);
}
#endif

// ---------------------------------------------------------------- vocab pass -

constexpr int kPassThreads = 512;     // threads per CTA of the vocabulary pass
constexpr int kPassCtasPerSm = 2;
// the expand pass: one CTA per SM, 12 warps that stream and 4 that complete rows.  Measured on eight levels of 640 rows of
// 128256 tokens with the pruning of the time (bf16 / fp32; these 12 warps are at 314 / 467 with today's): 12 streaming warps
// 323 / 472 us, 16 325 / 462, 20 342 / 477, 24 372 / 550 (fewer registers per thread: spills); chunks of 8 KB in 12 warps
// 335 / 468 (the unrolled chunk no longer fits the instruction caches).
constexpr int kExpandWarps = 12;
constexpr int kExpandThreads = (kExpandWarps + 4) * 32;
constexpr int kChunkVecs = 256;       // 16-byte vectors of a chunk: 8 per lane

// How the expand pass cut the rows (with M > 0: for the selection kernels).
struct PassInfo {
  int32_t n_rows;       // active rows
  int32_t row_chunks;   // chunks per row
  int32_t cta_chunks;   // chunks per CTA
  int32_t reserved;
};

// What the expand pass leaves per active row, at (b, j) of [B, F]; its K largest keys are in row_keys.
struct RowResult {
  double M, S, T, L, H;         // row maximum; sums over every other element of e^(x - M) and e^(x - M)(x - M); ln(1 + S);
                                // the entropy of Eq. 2 with natural log
  unsigned long long top;       // the row's best key (0: none)
  int32_t n_valid;              // keys that exist (at most K)
  uint32_t fault;               // C2T_ST_* bits of the row's data
};

// The sums over the chunks of a row that one warp streamed, base 2, relative to an integer offset; the lane and chunk with
// the largest value are kept apart, so that a row can be completed without its largest element by summing one lane's
// vectors of one chunk again.
struct alignas(16) SumRecord {
  float4 rest;                  // S and U of everything else, the offset, the largest value
  float4 held;                  // S and U of that lane and chunk, their numbers (as int bits)
};

struct TopmSegment;

struct PassParams {
  const void *logits;
  int64_t seq_stride, row_stride;   // elements
  int32_t V, K, B;
  int32_t rows_per_seq_max;         // F (draft) or Nw (target)
  int32_t rows_bound;               // expand: no sequence has more active rows at this level
  const int32_t *counts;            // [B] active rows per sequence, device
  const int32_t *row_sel;           // arg-max pass only, may be null: [B] the row of sequence b to read (then counts is 0 or 1)
  uint32_t *status;                 // may be null: a status word for C2T_ST_INTERNAL (the first sequence's)
  PassInfo *info;                   // expand with M > 0: written by CTA 0
  int32_t *row_off;                 // expand with M > 0: [B+1] first active row of every sequence, written by CTA 0
  // expand: results per row, and what the warps that stream a row leave for the pair that completes it
  RowResult *rows;                  // [B, F]
  unsigned long long *row_keys;     // [B, F, K] the row's K largest keys, sorted descending, 0-padded
  int32_t *row_done;                // [B * F] finished chunks of a row shared by several CTAs (rows in registers: [b F] finished rows of sequence b);
                                    // 0 between launches
  uint32_t *cells, *cell_low;       // [row, two chunks, 32] lane maxima, rounded; fp32: their lower halves (expand_pass.cu)
  SumRecord *sums;                  // [chunk] at a warp's last chunk of a row
  int64_t n_chunks, n_segs;
  int32_t cta_tasks;                // barriers in a CTA's shared memory (set at launch)
  int32_t near_cells;               // where the cells of a CTA's own rows begin in its shared memory, 0: in the workspace (set at launch)
  int32_t wait_limit;               // tries of such a barrier (set at launch)
  // expand with M > 0 (else null): the pool of candidate vectors, cut evenly among the warps, and a record per segment
  uint4 *topm_pool;
  long long topm_pool_vecs;
  int32_t topm_place;               // the floor's place among the lane maxima (topm_floor_place)
  TopmSegment *topm_seg;            // [warp + row]
  // argmax: [B, rows_per_seq_max] best key per row, the largest of what is there and of the row's keys (0 before the pass;
  // the kernel that reads a key puts the 0 back)
  unsigned long long *best;
  int64_t n_slots;
};

// ---------------------------------------------------------------- candidates of the truncated entropy (Eq. 3)
// With entropy_top_m = M > 0 the expand pass also sets aside every 16-byte vector that holds an element at or above
// a floor of its segment (the part of a row that one warp streams): one of the 32 lane maxima over the segment's first two
// groups, the place among them chosen so that about 3 M of the row's elements reach it (if the segment's head looks like
// the row).  The vectors go, in stream order, to
// a region of the warp's own in a pool in global memory; the segment's record says where they are and what the floor
// was.  A small kernel per row then takes the elements at or above the row's highest floor F from those vectors: if
// there are at least M of them the M-th largest is among them and so is everything above it, and Eq. 3's sums follow
// without reading the row again.  Rows for which that fails (a region ran full, fewer than M elements at or above F,
// more than fit in shared memory) are left to the pass that reads the row again.
constexpr int kTopmPoolDivisor = 3;      // the pool holds a third of the largest level's vectors (twice what is expected)
constexpr float kTopmLowestFloor = -1.7e38f;   // above -2^127, the value that pads a ragged vector
struct TopmSegment {
  int first;       // the segment's first vector in the pool
  int n;           // vectors, or -1: the region ran full
  float floor;
  int pad;
};
int topm_floor_place(int vocab, int elem_bytes, int M);
size_t topm_pool_vectors(size_t batch, size_t rows_per_seq, int vocab, int elem_bytes);

int row_chunks(int vocab, int elem_bytes);   // chunks of a row of the expand pass

// ---------------------------------------------------------------- rows in registers (row_pass.cu)
constexpr int kRowThreads = 512;                // threads of a block at most (or half as many)
constexpr int kRowPart = kRowThreads * 8;       // 16-byte vectors of a row that a block of so many holds
constexpr int kRowCluster = 8;                  // blocks of a row at most
struct RowPlan {
  int cluster, threads;                         // blocks per row (0: the level is not for that pass), threads of a block
};
struct TreeState;

// tries of a barrier in shared memory before the row is given up
constexpr int kTaskWaitLimit = 1 << 22;
#ifdef C2T_DEBUG_BOUNDS
extern "C" int c2t_debug_task_wait_limit;       // tests let the wait run out: then every level takes a pass that waits
#define C2T_TASK_WAIT_LIMIT c2t_debug_task_wait_limit
#else
#define C2T_TASK_WAIT_LIMIT kTaskWaitLimit
#endif

// How a level is cut, if its rows leave an SM no more than 512 threads of them: the smaller blocks where a row fits eight of them, and while
// half the chip would be idle more of them to a row.  Where the line lies: 64 rows of 128256 bf16 tokens (a step's level 0) in 512 blocks of
// 256 threads take 7 us more than streamed, 32 of fp32 in 256 blocks of 512 6 us more; 80 rows of 32000 in 160 blocks 4 us less per level.
// Blocks of 512 threads in clusters of eight where those of 256 would do: 16 rows of 128256 19 us per level instead of 14 (a GPC
// holds two such clusters only while all its SMs are free).
// And only rows that give data to 1.5 K of the groups whose maxima make the floor, so that few elements reach the K-th of those;
// for the same reason no more blocks to a row than it has vectors for their threads.  With less data the K largest are found in rounds:
// five levels of 3 sequences of 1000 bf16 tokens, K = 10, with eight blocks to a row 123 us, with one 45 (streamed 52); of one sequence of
// 500, K = 16, 139 us, streamed 58.
inline RowPlan row_pass_plan(int vocab, int elem_bytes, long long rows, int K, int sms) {
  RowPlan plan = {0, 0};
  const int vec = 16 / elem_bytes, vpr = (vocab + vec - 1) / vec;
  const int threads = vpr <= kRowCluster * kRowPart / 2 ? kRowThreads / 2 : kRowThreads, part = threads * 8;
  if (vpr < 6 * K) return plan;                         // (a group of a single block is four of its threads)
  int cluster = 1;
  while (cluster < kRowCluster && (vpr + cluster - 1) / cluster > part) cluster *= 2;
  if ((vpr + cluster - 1) / cluster > part || rows * cluster > (long long)sms * (kRowThreads / threads)) return plan;
  while (cluster < kRowCluster && 2 * cluster * rows <= sms && vpr >= 2 * cluster * threads) cluster *= 2;
  if (C2T_TASK_WAIT_LIMIT != kTaskWaitLimit && cluster == 1) return plan;      // (nothing waits there)
  plan.cluster = cluster;
  plan.threads = threads;
  return plan;
}
cudaError_t launch_expand_rows(PassParams p, int dtype, RowPlan plan, cudaStream_t s);
cudaError_t launch_expand_rows_prune(PassParams p, const TreeState &t, int level, const c2t_frontier &out, int dtype, RowPlan plan, cudaStream_t s);

cudaError_t prepare_expand_pass();   // once per device: opt in to the kernel's shared-memory size
cudaError_t launch_expand_pass(PassParams p, int dtype, int grid, cudaStream_t s);
cudaError_t launch_argmax_pass(const PassParams &p, int dtype, int grid, cudaStream_t s);
// arg-max of every row of a matrix; pieces: [grid] device scratch, a CTA's best keys of the rows it shares with the CTA before it
// (first) and behind it (last); ticket: 0 between calls, which all have the same grid of at most kMaxArgmaxCtas
constexpr int kMaxArgmaxCtas = kPassThreads;
struct ArgmaxPieces {
  unsigned long long first, last;
};
cudaError_t launch_row_argmax(const void *logits, int64_t row_stride, int rows, int V, int dtype, ArgmaxPieces *pieces, unsigned *ticket,
                              int32_t *out, int grid, cudaStream_t s);
struct TreeState;
cudaError_t prepare_accept_lazy();   // once per device
// the acceptance walk reading only the rows it visits; grid: CTAs of kPassThreads threads that the chip holds
cudaError_t launch_accept_lazy(const TreeState &t, const void *logits, int64_t seq_stride, int64_t row_stride, const c2t_accept_out *out,
                               int dtype, int grid, cudaStream_t s);
// expand and prune of a level in one launch (which levels: c2t_expand_prune_level)
cudaError_t launch_expand_prune(PassParams p, const TreeState &t, int level, const c2t_frontier *out, int dtype,
                                int grid, cudaStream_t s);
// ---------------------------------------------------------------- tree state -

struct TreeState {
  int32_t B, V, K, F, D, N, Nw, W, cap, hidden, classifier, tree_add;
  float beta;
  // frontier, double buffered by level parity
  int32_t *frontier_n[2];      // [B]
  int32_t *frontier_node[2];   // [B, F]
  double *frontier_logP[2], *frontier_chat[2];      // [B, F] the nodes' tree_logP and tree_Chat
  // tree
  int32_t *tree_n;             // [B]
  int32_t *tree_token, *tree_parent, *tree_level;   // [B, cap]
  double *tree_logP, *tree_C, *tree_Chat;           // [B, cap]
  // candidates of the last level
  int32_t *cand_n;             // [B]
  int32_t *cand_token, *cand_flags;                 // [B, F*K]
  double *cand_lp, *cand_logP, *cand_H, *cand_C;    // [B, F*K]
  // final tree
  int32_t *final_n;            // [B]
  int32_t *final_src, *final_token, *final_parent, *final_level;   // [B, Nw]
  int32_t *node_argmax;        // [B, Nw]
  int32_t *root_tok, *prefix_len;                   // [B]
  int32_t *walk_active, *walk_cur, *walk_len;       // [B] state of the lazy acceptance walk
  int32_t entropy_top_m, topm_place;   // M of Eq. 3 (0: exact entropy); the place of the collection floor
  double2 *topm;               // [B, F] {S_M, T_M} of the last expand call when M > 0
  uint4 *topm_pool;            // M > 0: candidate vectors set aside by the expand pass
  long long topm_pool_vecs;
  TopmSegment *topm_seg;       // M > 0: [n_segs] where each segment's candidates are
  int32_t *topm_done;          // M > 0: [B, F] 1 where the row's sums came from the candidate vectors
  uint32_t *status;            // [B]
  uint32_t *ticket;            // one counter: CTAs of a fused expand + prune launch that have finished (0 between launches)
  PassInfo *info_draft;
  int32_t *row_off_draft;          // [B+1] first row of every sequence in the last expand pass
  RowResult *rows;                 // the expand pass: see PassParams
  unsigned long long *row_keys;
  int32_t *row_done;
  uint32_t *cells, *cell_low;
  SumRecord *sums;
  int64_t n_chunks, n_segs;
  unsigned long long *best;        // [B, Nw] best key per row of the last arg-max pass; zeros between passes
  float *w1, *b1, *w2, *b2;
};

// truncated entropy (Eq. 3): per active row (b, j) the sums over its M largest logits, out[b * F + j] = {S_M, T_M};
// runs after the expand pass of the same level, whose partial records give it the row maxima
cudaError_t prepare_topm_pass();     // once per device: opt in to the kernel's shared-memory size
cudaError_t prepare_tree_kernels();  // the same for the pruning kernel
cudaError_t launch_topm_entropy(const void *logits, int64_t seq_stride, int64_t row_stride, int V, int M, int F,
                                int B, const int32_t *counts, const TreeState &t, double2 *out, const int32_t *done,
                                int n_ctas, int dtype, cudaStream_t s);
// the same sums from the candidate vectors of the expand pass, for the rows where they suffice (t.topm_done says
// which; launch_topm_entropy skips those when given t.topm_done)
cudaError_t launch_topm_finish(int M, int F, int B, const int32_t *counts, const TreeState &t, double2 *out, int dtype,
                               cudaStream_t s);
cudaError_t launch_begin_step(const TreeState &t, const int32_t *root_tok, const int32_t *prefix_len,
                              cudaStream_t s);
// records == nullptr: rows merged from this context's own expand pass; else from n_shards gathered records per row
cudaError_t launch_prune_level(const TreeState &t, int level, const c2t_frontier *out, const c2t_row_record *records,
                               int n_shards, cudaStream_t s);
cudaError_t launch_export_rows(const TreeState &t, int level, int vocab_begin, c2t_row_record *out, cudaStream_t s);
cudaError_t launch_final_prune(const TreeState &t, cudaStream_t s);
cudaError_t launch_build_verify(const TreeState &t, const c2t_verify *out, cudaStream_t s);
cudaError_t launch_dense_mask(const TreeState &t, void *out, int out_dtype, int64_t kv_len, cudaStream_t s);
// gathered == nullptr: node arg-maxes from this context's own pass; else the best of n_shards gathered keys per node
cudaError_t launch_accept_walk(const TreeState &t, const c2t_accept_out *out, const unsigned long long *gathered,
                               int n_shards, cudaStream_t s);
cudaError_t launch_export_best(const TreeState &t, int vocab_begin, unsigned long long *out, cudaStream_t s);
// one round of the lazy walk over sharded rows: round 0 starts it, round r > 0 takes n_shards gathered keys per sequence
cudaError_t launch_lazy_walk_round(const TreeState &t, int round, const c2t_accept_out *out,
                                   const unsigned long long *gathered, int n_shards, cudaStream_t s);
cudaError_t launch_export_lazy_best(const TreeState &t, int vocab_begin, unsigned long long *out, cudaStream_t s);

}  // namespace c2t

// Host side of libc2t: argument validation, workspace carving, call ordering, launches.
#include <new>
#include <string.h>

#include "c2t_internal.h"

using namespace c2t;

struct c2t_ctx {
  c2t_config cfg;
  TreeState t;
  int grid;              // CTAs of the arg-max pass
  int grid_expand;       // CTAs of the expand pass
  int next_level;        // level the next c2t_expand_level must carry
  int expanded;          // 1 after expand_level(next_level), before its prune
  int shard_expanded;    // 1 after expand_level_shard(next_level), before its export
  int shard_vocab;       // tokens of that shard
  int finalized;         // 1 after c2t_prune(C2T_FINAL)
  int started;
  int keys_unread;       // 1 between an arg-max pass and the launch that reads its keys and puts the zeros back
  int64_t launches;
  size_t elem_bytes;
  // c2t_decode_step_host only (made at its first call): its copies run ahead on a stream of their own
  cudaStream_t copy_stream;
  cudaEvent_t entered, copied[2], consumed[2];
};

namespace {

struct Carver {
  char *base;
  size_t off;
  template <typename T>
  T *take(size_t count) {
    off = (off + 255) & ~(size_t)255;
    T *p = base ? reinterpret_cast<T *>(base + off) : nullptr;
    off += count * sizeof(T);
    return p;
  }
};

int validate(const c2t_config *c) {
  if (!c) return C2T_EINVAL;
  if (c->batch < 1 || c->vocab < 1 || c->max_depth < 1 || c->topk < 1 || c->frontier_cap < 1 ||
      c->budget < 0 || c->device < 0)
    return C2T_EINVAL;
  if (c->dtype != C2T_F32 && c->dtype != C2T_BF16) return C2T_EINVAL;
  if (c->classifier != C2T_CLS_MLP && c->classifier != C2T_CLS_IDENTITY_JOINT &&
      c->classifier != C2T_CLS_IDENTITY_COND)
    return C2T_EINVAL;
  if (c->tree_add != C2T_ADD_FRONTIER && c->tree_add != C2T_ADD_ALL_SURVIVORS) return C2T_EINVAL;
  if (c->entropy_top_m < 0) return C2T_EINVAL;
  if (!(c->threshold == c->threshold)) return C2T_EINVAL;
  if (c->classifier == C2T_CLS_MLP) {
    if (c->hidden < 1 || !c->w1 || !c->b1 || !c->w2 || !c->b2) return C2T_EINVAL;
    if (c->hidden > C2T_MAX_HIDDEN) return C2T_ERANGE;
  }
  if (c->batch > C2T_MAX_BATCH || c->topk > C2T_MAX_TOPK || c->frontier_cap > C2T_MAX_FRONTIER ||
      c->max_depth > C2T_MAX_DEPTH || c->budget > C2T_MAX_BUDGET)
    return C2T_ERANGE;
  if (c2t_tree_capacity(c) > C2T_MAX_TREE) return C2T_ERANGE;
  return C2T_OK;
}

int tree_capacity_unchecked(const c2t_config *c) {
  const long long K = c->topk, F = c->frontier_cap, D = c->max_depth;
  long long cap;
  if (c->tree_add == C2T_ADD_ALL_SURVIVORS) cap = 1 + K + (D - 1) * F * K;
  else cap = 1 + (K < F ? K : F) + (D - 1) * F;
  return cap > 0x7FFFFFFF ? 0x7FFFFFFF : (int)cap;
}

// The grid of the vocabulary pass is fixed per device: 2 CTAs per SM.  Workspace sizing must
// not depend on a device query failing, so sizes assume at most this many SMs.
constexpr int kMaxSms = 256;

int pass_grid(int device) {
  int sms = 0;
  if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, device) != cudaSuccess || sms < 1)
    return -1;
  if (sms > kMaxSms) sms = kMaxSms;
  return sms * kPassCtasPerSm;
}

size_t carve(const c2t_config *c, void *base, TreeState *t) {
  Carver w{reinterpret_cast<char *>(base), 0};
  const size_t B = c->batch, F = c->frontier_cap, K = c->topk;
  const size_t cap = tree_capacity_unchecked(c), Nw = c2t_final_width(c);
  const int eb = c->dtype == C2T_BF16 ? 2 : 4;
  TreeState s;
  memset(&s, 0, sizeof s);
  for (int i = 0; i < 2; ++i) {
    s.frontier_n[i] = w.take<int32_t>(B);
    s.frontier_node[i] = w.take<int32_t>(B * F);
    s.frontier_logP[i] = w.take<double>(B * F);
    s.frontier_chat[i] = w.take<double>(B * F);
  }
  s.tree_n = w.take<int32_t>(B);
  s.tree_token = w.take<int32_t>(B * cap);
  s.tree_parent = w.take<int32_t>(B * cap);
  s.tree_level = w.take<int32_t>(B * cap);
  s.tree_logP = w.take<double>(B * cap);
  s.tree_C = w.take<double>(B * cap);
  s.tree_Chat = w.take<double>(B * cap);
  s.cand_n = w.take<int32_t>(B);
  s.cand_token = w.take<int32_t>(B * F * K);
  s.cand_flags = w.take<int32_t>(B * F * K);
  s.cand_lp = w.take<double>(B * F * K);
  s.cand_logP = w.take<double>(B * F * K);
  s.cand_H = w.take<double>(B * F * K);
  s.cand_C = w.take<double>(B * F * K);
  s.final_n = w.take<int32_t>(B);
  s.final_src = w.take<int32_t>(B * Nw);
  s.final_token = w.take<int32_t>(B * Nw);
  s.final_parent = w.take<int32_t>(B * Nw);
  s.final_level = w.take<int32_t>(B * Nw);
  s.node_argmax = w.take<int32_t>(B * Nw);
  s.root_tok = w.take<int32_t>(B);
  s.prefix_len = w.take<int32_t>(B);
  s.walk_active = w.take<int32_t>(B);
  s.walk_cur = w.take<int32_t>(B);
  s.walk_len = w.take<int32_t>(B);
  s.status = w.take<uint32_t>(B);
  s.ticket = w.take<uint32_t>(1);
  s.info_draft = w.take<PassInfo>(1);
  s.row_off_draft = w.take<int32_t>(B + 1);
  s.topm = w.take<double2>(B * F);
  // every segment of the expand pass (with M > 0) ends a warp's span or a row
  const size_t segs = B * F + (size_t)kMaxSms * kExpandWarps;
  s.n_segs = (int64_t)segs;
  s.n_chunks = (int64_t)(B * F * row_chunks(c->vocab, eb));
  const bool truncated = c->entropy_top_m > 0 && c->entropy_top_m < c->vocab;
  if (truncated) s.topm_done = w.take<int32_t>(B * F);
  if (truncated && topm_floor_place(c->vocab, eb, c->entropy_top_m) > 0) {     // the expand pass sets Eq. 3's candidates aside
    s.topm_pool_vecs = (long long)topm_pool_vectors(B, F, c->vocab, eb);
    s.topm_pool = w.take<uint4>((size_t)s.topm_pool_vecs);
    s.topm_seg = w.take<TopmSegment>(segs);
  }
  s.rows = w.take<RowResult>(B * F);
  s.row_keys = w.take<unsigned long long>(B * F * K);
  s.row_done = w.take<int32_t>(B * F);
  const size_t cells = B * F * ((row_chunks(c->vocab, eb) + 1) / 2) * 32;
  s.cells = w.take<uint32_t>(cells);
  if (eb == 4) s.cell_low = w.take<uint32_t>(cells);
  s.sums = w.take<SumRecord>((size_t)s.n_chunks);
  s.best = w.take<unsigned long long>(B * Nw);
  s.w1 = w.take<float>(3 * C2T_MAX_HIDDEN);
  s.b1 = w.take<float>(C2T_MAX_HIDDEN);
  s.w2 = w.take<float>(C2T_MAX_HIDDEN);
  s.b2 = w.take<float>(4);
  if (t) *t = s;
  return (w.off + 255) & ~(size_t)255;
}

// no sequence has more active rows at this level
int rows_bound(const TreeState &t, int level) {
  long long bound = 1;
  for (int l = 0; l < level && bound < t.F; ++l) bound *= t.K;
  return bound < t.F ? (int)bound : t.F;
}

constexpr long long kFusedRowBytes = 32768;            // (c2t_expand_prune_level)

// the expand pass of a level over rows of `vocab` tokens (the whole vocabulary, or one shard of it)
PassParams expand_params(const TreeState &t, int level, const void *logits, int64_t seq_stride, int64_t row_stride, int vocab) {
  PassParams p;
  memset(&p, 0, sizeof p);
  p.logits = logits; p.seq_stride = seq_stride; p.row_stride = row_stride;
  p.V = vocab; p.K = t.K; p.B = t.B; p.rows_per_seq_max = t.F;
  p.rows_bound = rows_bound(t, level);
  p.counts = t.frontier_n[level & 1];
  p.status = t.status;
  p.info = t.info_draft;
  p.row_off = t.row_off_draft;
  p.rows = t.rows; p.row_keys = t.row_keys; p.row_done = t.row_done;
  p.cells = t.cells; p.cell_low = t.cell_low; p.sums = t.sums;
  p.n_chunks = t.n_chunks; p.n_segs = t.n_segs;
  return p;
}

// the arg-max pass over the rows of all final nodes, or (walk) over the current node's row of every walking sequence
PassParams argmax_params(const TreeState &t, const void *logits, int64_t seq_stride, int64_t row_stride, int vocab, bool walk) {
  PassParams p;
  memset(&p, 0, sizeof p);
  p.logits = logits; p.seq_stride = seq_stride; p.row_stride = row_stride;
  p.V = vocab; p.K = 1; p.B = t.B; p.rows_per_seq_max = walk ? 1 : t.Nw;
  p.counts = walk ? t.walk_active : t.final_n;
  p.row_sel = walk ? t.walk_cur : nullptr;
  p.status = t.status;
  p.best = t.best;
  p.n_slots = (int64_t)t.B * t.Nw;
  return p;
}

// The arg-max pass.  It takes the largest of a row's keys and of what is in its place; the launch behind it reads the places and
// leaves zeros.  Where that launch failed after an earlier pass, its keys are cleared first.
cudaError_t argmax_pass(c2t_ctx *ctx, const PassParams &p, cudaStream_t s) {
  if (ctx->keys_unread) {
    const cudaError_t e = cudaMemsetAsync(p.best, 0, sizeof(unsigned long long) * (size_t)p.n_slots, s);
    if (e != cudaSuccess) return e;
  }
  ctx->keys_unread = 1;
  return launch_argmax_pass(p, ctx->cfg.dtype, ctx->grid, s);
}

// The stream of c2t_decode_step_host's copies and its events, on the context's device: all of them or none.
void drop_copy_stream(c2t_ctx *ctx) {
  cudaEvent_t *events[] = {&ctx->entered, &ctx->copied[0], &ctx->copied[1], &ctx->consumed[0], &ctx->consumed[1]};
  for (cudaEvent_t *e : events) {
    if (*e) cudaEventDestroy(*e);
    *e = nullptr;
  }
  if (ctx->copy_stream) cudaStreamDestroy(ctx->copy_stream);
  ctx->copy_stream = nullptr;
}

cudaError_t make_copy_stream(c2t_ctx *ctx) {
  int current = 0;
  cudaError_t e = cudaGetDevice(&current);
  if (e == cudaSuccess && current != ctx->cfg.device) e = cudaSetDevice(ctx->cfg.device);
  if (e != cudaSuccess) return e;
  cudaEvent_t *events[] = {&ctx->entered, &ctx->copied[0], &ctx->copied[1], &ctx->consumed[0], &ctx->consumed[1]};
  for (cudaEvent_t *ev : events) {
    if (e == cudaSuccess) e = cudaEventCreateWithFlags(ev, cudaEventDisableTiming);
    if (e != cudaSuccess) *ev = nullptr;
  }
  if (e == cudaSuccess) {
    e = cudaStreamCreateWithFlags(&ctx->copy_stream, cudaStreamNonBlocking);
    if (e != cudaSuccess) ctx->copy_stream = nullptr;
  }
  if (e != cudaSuccess) drop_copy_stream(ctx);
  if (current != ctx->cfg.device) cudaSetDevice(current);
  return e;
}

// Waits for a stream on the way out, unless told that there is nothing left to wait for.
struct WaitOnExit {
  cudaStream_t stream;
  ~WaitOnExit() { if (stream) cudaStreamSynchronize(stream); }
};

bool aligned16(const void *p) { return (reinterpret_cast<uintptr_t>(p) & 15) == 0; }

}  // namespace

extern "C" {

int32_t c2t_tree_capacity(const c2t_config *cfg) {
  if (!cfg || cfg->topk < 1 || cfg->frontier_cap < 1 || cfg->max_depth < 1) return 0;
  return tree_capacity_unchecked(cfg);
}

int32_t c2t_final_width(const c2t_config *cfg) {
  const int32_t cap = c2t_tree_capacity(cfg);
  if (cap == 0) return 0;
  return (cfg->budget > 0 && cfg->budget < cap) ? cfg->budget : cap;
}

int32_t c2t_mask_words(const c2t_config *cfg) { return (c2t_final_width(cfg) + 63) / 64; }

size_t c2t_workspace_bytes(const c2t_config *cfg) {
  if (validate(cfg) != C2T_OK) return 0;
  return carve(cfg, nullptr, nullptr);
}

size_t c2t_host_step_ints(const c2t_config *cfg) {
  if (validate(cfg) != C2T_OK) return 0;
  const size_t B = cfg->batch, Nw = c2t_final_width(cfg), W = c2t_mask_words(cfg), D = cfg->max_depth;
  // roots, prefix lengths, n_nodes, tokens, parents, positions, mask (2 ints per word),
  // retrieve, n_leaves, accept_len, path, next_token; each padded to an even count
  size_t n = 0;
  const size_t parts[] = {B, B, B, B * Nw, B * Nw, B * Nw, 2 * B * Nw * W, B * Nw * (D + 1), B, B, B * (D + 1), B};
  for (size_t p : parts) n += (p + 1) & ~(size_t)1;
  return n;
}

int c2t_init(const c2t_config *cfg, void *workspace_dev, size_t workspace_bytes, c2t_ctx **out) {
  if (!out) return C2T_EINVAL;
  *out = nullptr;
  int rc = validate(cfg);
  if (rc != C2T_OK) return rc;
  if (!workspace_dev) return C2T_EINVAL;
  if (reinterpret_cast<uintptr_t>(workspace_dev) & 255) return C2T_EALIGN;
  if (workspace_bytes < carve(cfg, nullptr, nullptr)) return C2T_ERANGE;
  if (cudaSetDevice(cfg->device) != cudaSuccess) { cudaGetLastError(); return C2T_ECUDA; }
  const int grid = pass_grid(cfg->device);
  if (grid < 0 || prepare_expand_pass() != cudaSuccess || prepare_topm_pass() != cudaSuccess ||
      prepare_tree_kernels() != cudaSuccess || prepare_accept_lazy() != cudaSuccess) {
    cudaGetLastError();
    return C2T_ECUDA;
  }

  c2t_ctx *ctx = new (std::nothrow) c2t_ctx;
  if (!ctx) return C2T_ENOMEM;
  memset(ctx, 0, sizeof *ctx);
  ctx->cfg = *cfg;
  ctx->cfg.w1 = ctx->cfg.b1 = ctx->cfg.w2 = ctx->cfg.b2 = nullptr;
  ctx->grid = grid;
  ctx->grid_expand = grid / kPassCtasPerSm;
  ctx->elem_bytes = cfg->dtype == C2T_BF16 ? 2 : 4;
  carve(cfg, workspace_dev, &ctx->t);
  TreeState &t = ctx->t;
  t.B = cfg->batch; t.V = cfg->vocab; t.K = cfg->topk; t.F = cfg->frontier_cap; t.D = cfg->max_depth;
  t.N = cfg->budget; t.Nw = c2t_final_width(cfg); t.W = c2t_mask_words(cfg);
  t.cap = tree_capacity_unchecked(cfg);
  t.hidden = cfg->classifier == C2T_CLS_MLP ? cfg->hidden : 0;
  t.classifier = cfg->classifier; t.tree_add = cfg->tree_add; t.beta = cfg->threshold;
  t.entropy_top_m = cfg->entropy_top_m;
  t.topm_place = topm_floor_place(cfg->vocab, (int)ctx->elem_bytes, cfg->entropy_top_m);
  cudaError_t e = cudaSuccess;
  if (cfg->classifier == C2T_CLS_MLP) {
    const size_t h = cfg->hidden;
    e = cudaMemcpy(t.w1, cfg->w1, 3 * h * sizeof(float), cudaMemcpyHostToDevice);
    if (e == cudaSuccess) e = cudaMemcpy(t.b1, cfg->b1, h * sizeof(float), cudaMemcpyHostToDevice);
    if (e == cudaSuccess) e = cudaMemcpy(t.w2, cfg->w2, h * sizeof(float), cudaMemcpyHostToDevice);
    if (e == cudaSuccess) e = cudaMemcpy(t.b2, cfg->b2, sizeof(float), cudaMemcpyHostToDevice);
  }
  if (e == cudaSuccess) e = cudaMemset(t.status, 0, sizeof(uint32_t) * cfg->batch);
  if (e == cudaSuccess) e = cudaMemset(t.ticket, 0, sizeof(uint32_t));
  if (e == cudaSuccess) e = cudaMemset(t.best, 0, sizeof(unsigned long long) * cfg->batch * t.Nw);
  if (e == cudaSuccess && t.topm_done) e = cudaMemset(t.topm_done, 0, sizeof(int32_t) * cfg->batch * cfg->frontier_cap);
  if (e == cudaSuccess) e = cudaMemset(t.row_done, 0, sizeof(int32_t) * cfg->batch * cfg->frontier_cap);
  // all of this is on the default stream, which the stream of the first step need not wait for
  if (e == cudaSuccess) e = cudaStreamSynchronize(cudaStreamLegacy);
  if (e != cudaSuccess) { cudaGetLastError(); delete ctx; return C2T_ECUDA; }
  *out = ctx;
  return C2T_OK;
}

void c2t_destroy(c2t_ctx *ctx) {
  if (ctx) drop_copy_stream(ctx);
  delete ctx;
}

int c2t_begin_step(c2t_ctx *ctx, const int32_t *root_tok_dev, const int32_t *prefix_len_dev, void *stream) {
  if (!ctx || !root_tok_dev || !prefix_len_dev) return C2T_EINVAL;
  if (launch_begin_step(ctx->t, root_tok_dev, prefix_len_dev, (cudaStream_t)stream) != cudaSuccess)
    return C2T_ECUDA;
  ctx->launches += 1;
  ctx->next_level = 0;
  ctx->expanded = 0;
  ctx->shard_expanded = 0;
  ctx->finalized = 0;
  ctx->started = 1;
  return C2T_OK;
}

int c2t_expand_level(c2t_ctx *ctx, int level, const void *logits_dev, int64_t seq_stride,
                     int64_t row_stride, void *stream) {
  if (!ctx || !logits_dev) return C2T_EINVAL;
  if (!ctx->started || ctx->finalized || ctx->expanded || ctx->shard_expanded || level != ctx->next_level ||
      level >= ctx->cfg.max_depth)
    return C2T_EORDER;
  if (seq_stride < 0 || row_stride < ctx->cfg.vocab) return C2T_EINVAL;
  if (!aligned16(logits_dev) || (seq_stride * ctx->elem_bytes) % 16 || (row_stride * ctx->elem_bytes) % 16)
    return C2T_EALIGN;
  const TreeState &t = ctx->t;
  PassParams p = expand_params(t, level, logits_dev, seq_stride, row_stride, t.V);
  const bool truncated = t.entropy_top_m > 0 && t.entropy_top_m < t.V;   // Eq. 3: the sums over the M most probable tokens
  const bool set_aside = truncated && t.topm_place > 0;
  if (set_aside) { p.topm_pool = t.topm_pool; p.topm_pool_vecs = t.topm_pool_vecs; p.topm_seg = t.topm_seg; p.topm_place = t.topm_place; }
  if (launch_expand_pass(p, ctx->cfg.dtype, ctx->grid_expand, (cudaStream_t)stream) != cudaSuccess)
    return C2T_ECUDA;
  ctx->launches += 1;
  if (truncated) {
    // from the vectors the pass set aside; then, for the rows where those did not suffice, from the rows themselves
    if (set_aside && launch_topm_finish(t.entropy_top_m, t.F, t.B, p.counts, t, t.topm, ctx->cfg.dtype, (cudaStream_t)stream) != cudaSuccess)
      return C2T_ECUDA;
    if (launch_topm_entropy(logits_dev, seq_stride, row_stride, t.V, t.entropy_top_m, t.F, t.B, p.counts, t, t.topm,
                            t.topm_done, ctx->grid_expand, ctx->cfg.dtype, (cudaStream_t)stream) != cudaSuccess)
      return C2T_ECUDA;
    ctx->launches += set_aside ? 2 : 1;
  }
  ctx->expanded = 1;
  return C2T_OK;
}

int c2t_prune(c2t_ctx *ctx, int level, const c2t_frontier *out, void *stream) {
  if (!ctx) return C2T_EINVAL;
  if (!ctx->started || ctx->finalized) return C2T_EORDER;
  if (level == C2T_FINAL) {
    if (ctx->expanded) return C2T_EORDER;
    if (launch_final_prune(ctx->t, (cudaStream_t)stream) != cudaSuccess) return C2T_ECUDA;
    ctx->launches += 1;
    ctx->finalized = 1;
    return C2T_OK;
  }
  if (!ctx->expanded || level != ctx->next_level) return C2T_EORDER;
  if (launch_prune_level(ctx->t, level, out, nullptr, 0, (cudaStream_t)stream) != cudaSuccess) return C2T_ECUDA;
  ctx->launches += 1;
  ctx->expanded = 0;
  ctx->next_level = level + 1;
  return C2T_OK;
}

int c2t_expand_prune_level(c2t_ctx *ctx, int level, const void *logits_dev, int64_t seq_stride, int64_t row_stride,
                           const c2t_frontier *out, void *stream) {
  if (!ctx || !logits_dev) return C2T_EINVAL;
  const TreeState &t = ctx->t;
  // One launch where a level is small: few sequences, or long rows in registers.  On the device one or two launches are alike there, to 0.2 us
  // of a level of 9 (in a graph; 3 to 12 sequences of 32000 bf16 tokens 8.8, 9.5, 9.8 us in one, 8.7, 9.4, 9.9 in two), and a launch less is 2.5 us
  // less for the caller.  Below kFusedRowBytes two stay: one is within 0.3 us for 3 and 6 sequences, from 12 on 0.1 to 0.5 us better.  Where
  // a block's threads do not suffice for the candidates two are better: 3 sequences of 32000, K = 16, F = 24, 12.4 us in one, 11.3 in two.
  const RowPlan rows = row_pass_plan(t.V, (int)ctx->elem_bytes, (long long)t.B * rows_bound(t, level), t.K, ctx->grid_expand);
  const bool small = t.B <= C2T_FUSED_MAX_BATCH ||
                     (rows.cluster > 0 && t.V * (long long)ctx->elem_bytes >= kFusedRowBytes && t.F * t.K <= rows.threads);
  if (!small || (t.entropy_top_m > 0 && t.entropy_top_m < t.V)) {
    const int rc = c2t_expand_level(ctx, level, logits_dev, seq_stride, row_stride, stream);
    return rc != C2T_OK ? rc : c2t_prune(ctx, level, out, stream);
  }
  if (!ctx->started || ctx->finalized || ctx->expanded || ctx->shard_expanded || level != ctx->next_level ||
      level >= ctx->cfg.max_depth)
    return C2T_EORDER;
  if (seq_stride < 0 || row_stride < ctx->cfg.vocab) return C2T_EINVAL;
  if (!aligned16(logits_dev) || (seq_stride * ctx->elem_bytes) % 16 || (row_stride * ctx->elem_bytes) % 16)
    return C2T_EALIGN;
  PassParams p = expand_params(t, level, logits_dev, seq_stride, row_stride, t.V);
  if (launch_expand_prune(p, t, level, out, ctx->cfg.dtype, ctx->grid_expand, (cudaStream_t)stream) != cudaSuccess)
    return C2T_ECUDA;
  ctx->launches += 1;
  ctx->next_level = level + 1;
  return C2T_OK;
}

int c2t_expand_level_shard(c2t_ctx *ctx, int level, const void *logits_dev, int64_t seq_stride,
                           int64_t row_stride, int32_t vocab_count, void *stream) {
  if (!ctx || !logits_dev) return C2T_EINVAL;
  if (!ctx->started || ctx->finalized || ctx->expanded || ctx->shard_expanded || level != ctx->next_level ||
      level >= ctx->cfg.max_depth)
    return C2T_EORDER;
  if (vocab_count < 1 || vocab_count > ctx->cfg.vocab || seq_stride < 0 || row_stride < vocab_count) return C2T_EINVAL;
  if (ctx->t.entropy_top_m > 0 && ctx->t.entropy_top_m < ctx->t.V) return C2T_EINVAL;   // Eq. 3 needs whole rows
  if (!aligned16(logits_dev) || (seq_stride * ctx->elem_bytes) % 16 || (row_stride * ctx->elem_bytes) % 16)
    return C2T_EALIGN;
  const TreeState &t = ctx->t;
  PassParams p = expand_params(t, level, logits_dev, seq_stride, row_stride, vocab_count);
  if (launch_expand_pass(p, ctx->cfg.dtype, ctx->grid_expand, (cudaStream_t)stream) != cudaSuccess)
    return C2T_ECUDA;
  ctx->launches += 1;
  ctx->shard_expanded = 1;
  ctx->shard_vocab = vocab_count;
  return C2T_OK;
}

int c2t_export_row_records(c2t_ctx *ctx, int level, int32_t vocab_begin, c2t_row_record *records_dev,
                           void *stream) {
  if (!ctx || !records_dev) return C2T_EINVAL;
  if (!ctx->shard_expanded || level != ctx->next_level) return C2T_EORDER;
  if (vocab_begin < 0 || (int64_t)vocab_begin + ctx->shard_vocab > ctx->cfg.vocab) return C2T_EINVAL;
  if (launch_export_rows(ctx->t, level, vocab_begin, records_dev, (cudaStream_t)stream) !=
      cudaSuccess)
    return C2T_ECUDA;
  ctx->launches += 1;
  ctx->shard_expanded = 0;
  return C2T_OK;
}

int c2t_prune_gathered(c2t_ctx *ctx, int level, const c2t_row_record *records_dev, int32_t n_shards,
                       const c2t_frontier *out, void *stream) {
  if (!ctx || !records_dev) return C2T_EINVAL;
  if (n_shards < 1) return C2T_EINVAL;
  if (n_shards > C2T_MAX_SHARDS) return C2T_ERANGE;
  if (!ctx->started || ctx->finalized || ctx->expanded || ctx->shard_expanded || level != ctx->next_level ||
      level >= ctx->cfg.max_depth)
    return C2T_EORDER;
  if (launch_prune_level(ctx->t, level, out, records_dev, n_shards, (cudaStream_t)stream) != cudaSuccess)
    return C2T_ECUDA;
  ctx->launches += 1;
  ctx->next_level = level + 1;
  return C2T_OK;
}

int c2t_build_verify(c2t_ctx *ctx, const c2t_verify *out, void *stream) {
  if (!ctx) return C2T_EINVAL;
  if (!ctx->finalized) return C2T_EORDER;
  if (launch_build_verify(ctx->t, out, (cudaStream_t)stream) != cudaSuccess) return C2T_ECUDA;
  ctx->launches += 1;
  return C2T_OK;
}

int c2t_dense_mask(c2t_ctx *ctx, void *out_dev, int32_t out_dtype, int64_t kv_len, void *stream) {
  if (!ctx || !out_dev || kv_len < 1) return C2T_EINVAL;
  if (out_dtype != C2T_F32 && out_dtype != C2T_BF16) return C2T_EINVAL;
  if (!ctx->finalized) return C2T_EORDER;
  if (launch_dense_mask(ctx->t, out_dev, out_dtype, kv_len, (cudaStream_t)stream) != cudaSuccess) return C2T_ECUDA;
  ctx->launches += 1;
  return C2T_OK;
}

int c2t_accept(c2t_ctx *ctx, const void *target_logits_dev, int64_t seq_stride, int64_t row_stride,
               const c2t_accept_out *out, void *stream) {
  if (!ctx || !target_logits_dev) return C2T_EINVAL;
  if (!ctx->finalized) return C2T_EORDER;
  if (seq_stride < 0 || row_stride < ctx->cfg.vocab) return C2T_EINVAL;
  if (!aligned16(target_logits_dev) || (seq_stride * ctx->elem_bytes) % 16 ||
      (row_stride * ctx->elem_bytes) % 16)
    return C2T_EALIGN;
  const TreeState &t = ctx->t;
  const PassParams p = argmax_params(t, target_logits_dev, seq_stride, row_stride, t.V, false);
  if (argmax_pass(ctx, p, (cudaStream_t)stream) != cudaSuccess) return C2T_ECUDA;
  if (launch_accept_walk(t, out, nullptr, 0, (cudaStream_t)stream) != cudaSuccess) return C2T_ECUDA;
  ctx->keys_unread = 0;
  ctx->launches += 2;
  return C2T_OK;
}

int c2t_argmax_shard(c2t_ctx *ctx, const void *target_logits_dev, int64_t seq_stride, int64_t row_stride,
                     int32_t vocab_count, int32_t vocab_begin, uint64_t *keys_dev, void *stream) {
  if (!ctx || !target_logits_dev || !keys_dev) return C2T_EINVAL;
  if (!ctx->finalized) return C2T_EORDER;
  if (vocab_count < 1 || vocab_begin < 0 || (int64_t)vocab_begin + vocab_count > ctx->cfg.vocab || seq_stride < 0 ||
      row_stride < vocab_count)
    return C2T_EINVAL;
  if (!aligned16(target_logits_dev) || (seq_stride * ctx->elem_bytes) % 16 ||
      (row_stride * ctx->elem_bytes) % 16)
    return C2T_EALIGN;
  const TreeState &t = ctx->t;
  const PassParams p = argmax_params(t, target_logits_dev, seq_stride, row_stride, vocab_count, false);
  if (argmax_pass(ctx, p, (cudaStream_t)stream) != cudaSuccess) return C2T_ECUDA;
  if (launch_export_best(t, vocab_begin, reinterpret_cast<unsigned long long *>(keys_dev), (cudaStream_t)stream) !=
      cudaSuccess)
    return C2T_ECUDA;
  ctx->keys_unread = 0;
  ctx->launches += 2;
  return C2T_OK;
}

int c2t_accept_gathered(c2t_ctx *ctx, const uint64_t *keys_dev, int32_t n_shards, const c2t_accept_out *out,
                        void *stream) {
  if (!ctx || !keys_dev || n_shards < 1) return C2T_EINVAL;
  if (n_shards > C2T_MAX_SHARDS) return C2T_ERANGE;
  if (!ctx->finalized) return C2T_EORDER;
  if (launch_accept_walk(ctx->t, out, reinterpret_cast<const unsigned long long *>(keys_dev), n_shards,
                         (cudaStream_t)stream) != cudaSuccess)
    return C2T_ECUDA;
  ctx->launches += 1;
  return C2T_OK;
}

int c2t_accept_lazy(c2t_ctx *ctx, const void *target_logits_dev, int64_t seq_stride, int64_t row_stride,
                    const c2t_accept_out *out, void *stream) {
  if (!ctx || !target_logits_dev) return C2T_EINVAL;
  if (!ctx->finalized) return C2T_EORDER;
  if (seq_stride < 0 || row_stride < ctx->cfg.vocab) return C2T_EINVAL;
  if (!aligned16(target_logits_dev) || (seq_stride * ctx->elem_bytes) % 16 ||
      (row_stride * ctx->elem_bytes) % 16)
    return C2T_EALIGN;
  if (launch_accept_lazy(ctx->t, target_logits_dev, seq_stride, row_stride, out, ctx->cfg.dtype, ctx->grid, (cudaStream_t)stream) !=
      cudaSuccess)
    return C2T_ECUDA;
  ctx->launches += 1;
  return C2T_OK;
}

int c2t_lazy_begin(c2t_ctx *ctx, const c2t_accept_out *out, void *stream) {
  if (!ctx) return C2T_EINVAL;
  if (!ctx->finalized) return C2T_EORDER;
  if (launch_lazy_walk_round(ctx->t, 0, out, nullptr, 0, (cudaStream_t)stream) != cudaSuccess) return C2T_ECUDA;
  ctx->launches += 1;
  return C2T_OK;
}

int c2t_lazy_argmax_shard(c2t_ctx *ctx, const void *target_logits_dev, int64_t seq_stride, int64_t row_stride,
                          int32_t vocab_count, int32_t vocab_begin, uint64_t *keys_dev, void *stream) {
  if (!ctx || !target_logits_dev || !keys_dev) return C2T_EINVAL;
  if (!ctx->finalized) return C2T_EORDER;
  if (vocab_count < 1 || vocab_begin < 0 || (int64_t)vocab_begin + vocab_count > ctx->cfg.vocab || seq_stride < 0 ||
      row_stride < vocab_count)
    return C2T_EINVAL;
  if (!aligned16(target_logits_dev) || (seq_stride * ctx->elem_bytes) % 16 || (row_stride * ctx->elem_bytes) % 16)
    return C2T_EALIGN;
  const TreeState &t = ctx->t;
  const PassParams p = argmax_params(t, target_logits_dev, seq_stride, row_stride, vocab_count, true);
  cudaStream_t s = (cudaStream_t)stream;
  if (argmax_pass(ctx, p, s) != cudaSuccess) return C2T_ECUDA;
  if (launch_export_lazy_best(t, vocab_begin, reinterpret_cast<unsigned long long *>(keys_dev), s) != cudaSuccess)
    return C2T_ECUDA;
  ctx->keys_unread = 0;
  ctx->launches += 2;
  return C2T_OK;
}

int c2t_lazy_step_gathered(c2t_ctx *ctx, int round, const uint64_t *keys_dev, int32_t n_shards,
                           const c2t_accept_out *out, void *stream) {
  if (!ctx || !keys_dev || n_shards < 1 || round < 1) return C2T_EINVAL;
  if (n_shards > C2T_MAX_SHARDS) return C2T_ERANGE;
  if (!ctx->finalized) return C2T_EORDER;
  if (launch_lazy_walk_round(ctx->t, round, out, reinterpret_cast<const unsigned long long *>(keys_dev), n_shards,
                             (cudaStream_t)stream) != cudaSuccess)
    return C2T_ECUDA;
  ctx->launches += 1;
  return C2T_OK;
}

int c2t_status(c2t_ctx *ctx, uint32_t *bits_host, uint32_t *per_seq_host, void *stream) {
  if (!ctx || !bits_host) return C2T_EINVAL;
  const int B = ctx->cfg.batch;
  uint32_t *tmp = per_seq_host ? per_seq_host : new (std::nothrow) uint32_t[B];
  if (!tmp) return C2T_ENOMEM;
  cudaError_t e = cudaMemcpyAsync(tmp, ctx->t.status, sizeof(uint32_t) * B, cudaMemcpyDeviceToHost,
                                  (cudaStream_t)stream);
  if (e == cudaSuccess) e = cudaStreamSynchronize((cudaStream_t)stream);
  uint32_t bits = 0;
  if (e == cudaSuccess)
    for (int b = 0; b < B; ++b) bits |= tmp[b];
  if (!per_seq_host) delete[] tmp;
  if (e != cudaSuccess) { cudaGetLastError(); return C2T_ECUDA; }
  *bits_host = bits;
  return C2T_OK;
}

int c2t_get_view(c2t_ctx *ctx, c2t_view *v) {
  if (!ctx || !v) return C2T_EINVAL;
  const TreeState &t = ctx->t;
  v->tree_n = t.tree_n; v->tree_token = t.tree_token; v->tree_parent = t.tree_parent;
  v->tree_level = t.tree_level; v->tree_logP = t.tree_logP; v->tree_C = t.tree_C; v->tree_Chat = t.tree_Chat;
  v->cand_n = t.cand_n; v->cand_token = t.cand_token; v->cand_lp = t.cand_lp; v->cand_logP = t.cand_logP;
  v->cand_H = t.cand_H; v->cand_C = t.cand_C; v->cand_flags = t.cand_flags;
  v->frontier_n = t.frontier_n[ctx->next_level & 1];
  v->frontier_node = t.frontier_node[ctx->next_level & 1];
  v->final_n = t.final_n; v->final_src = t.final_src; v->final_token = t.final_token;
  v->final_parent = t.final_parent; v->final_level = t.final_level; v->node_argmax = t.node_argmax;
  v->topm_from_pass = t.topm_done;
  return C2T_OK;
}

int c2t_decode_step(c2t_ctx *ctx, const c2t_step *step, void *stream) {
  if (!ctx || !step || !step->draft_logits_dev || !step->draft_strides) return C2T_EINVAL;
  int rc = c2t_begin_step(ctx, step->root_tok_dev, step->prefix_len_dev, stream);
  for (int l = 0; l < ctx->cfg.max_depth && rc == C2T_OK; ++l)
    rc = c2t_expand_prune_level(ctx, l, step->draft_logits_dev[l], step->draft_strides[2 * l], step->draft_strides[2 * l + 1], step->frontier, stream);
  if (rc == C2T_OK) rc = c2t_prune(ctx, C2T_FINAL, nullptr, stream);
  if (rc == C2T_OK) rc = c2t_build_verify(ctx, step->verify, stream);
  if (rc == C2T_OK) rc = c2t_accept(ctx, step->target_logits_dev, step->target_seq_stride, step->target_row_stride, step->accept, stream);
  return rc;
}

int c2t_decode_step_host(c2t_ctx *ctx, const c2t_host_step *io, void *stream) {
  if (!ctx || !io || !io->draft_logits_host || !io->target_logits_host || !io->root_tok_host ||
      !io->prefix_len_host || !io->draft_stage_dev || !io->target_stage_dev || !io->int_stage_dev)
    return C2T_EINVAL;
  cudaStream_t s = (cudaStream_t)stream;
  const c2t_config &c = ctx->cfg;
  const size_t B = c.batch, F = c.frontier_cap, V = c.vocab, D = c.max_depth, eb = ctx->elem_bytes;
  const size_t Nw = ctx->t.Nw, W = ctx->t.W;
  for (size_t l = 0; l < D; ++l)
    if (!io->draft_logits_host[l]) return C2T_EINVAL;

  // carve the integer staging buffer (each part padded to an even count: mask words need 8-byte alignment)
  int32_t *ip = io->int_stage_dev;
  if (reinterpret_cast<uintptr_t>(ip) & 7) return C2T_EALIGN;
  auto take = [&](size_t n) { int32_t *p = ip; ip += (n + 1) & ~(size_t)1; return p; };
  int32_t *root = take(B), *prefix = take(B);
  c2t_verify vo;
  vo.n_nodes = take(B); vo.tokens = take(B * Nw); vo.parents = take(B * Nw); vo.position_ids = take(B * Nw);
  vo.mask_bits = reinterpret_cast<uint64_t *>(take(2 * B * Nw * W));
  vo.retrieve = take(B * Nw * (D + 1)); vo.n_leaves = take(B);
  c2t_accept_out ao;
  ao.accept_len = take(B); ao.path = take(B * (D + 1)); ao.next_token = take(B);

#define C2T_CUDA(x) do { if ((x) != cudaSuccess) { cudaGetLastError(); return C2T_ECUDA; } } while (0)
#define C2T_CALL(x) do { int rc_ = (x); if (rc_ != C2T_OK) return rc_; } while (0)
  if (!ctx->copy_stream) C2T_CUDA(make_copy_stream(ctx));
  cudaStream_t cs = ctx->copy_stream;
  WaitOnExit copies{cs};                         // (a call that fails in the middle: its copies use the caller's buffers)
  // The step is bound by the host link, so it is kept busy: the levels' rows are copied ahead of the kernels into the two
  // staging buffers in turn (the target's is free until the target rows come, and holds a level's rows if Nw >= F), the last level's
  // into its own; the target rows follow them.  8 sequences, 32000 tokens, bf16: 1512 -> 1309 us per step, 67 MB over a link of 55 GB/s.
  // (With the walk reading the rows it visits from the pinned buffer in place 821 us, but then neither the arg-max of the other
  // nodes nor the staged target rows are there, which this call has always left behind; c2t_accept_lazy takes such a buffer.)
  void *stage[2] = {io->draft_stage_dev, io->target_stage_dev};
  const uintptr_t d0 = reinterpret_cast<uintptr_t>(stage[0]), t0 = reinterpret_cast<uintptr_t>(stage[1]);
  const bool apart = d0 + B * F * V * eb <= t0 || t0 + B * Nw * V * eb <= d0;     // (one buffer may serve as both)
  const bool two = Nw >= F && apart;
  bool used[2] = {false, false};

  C2T_CUDA(cudaEventRecord(ctx->entered, s));    // (earlier work of the stream may still use the staging buffers)
  C2T_CUDA(cudaStreamWaitEvent(cs, ctx->entered, 0));
  C2T_CUDA(cudaMemcpyAsync(root, io->root_tok_host, B * 4, cudaMemcpyHostToDevice, s));
  C2T_CUDA(cudaMemcpyAsync(prefix, io->prefix_len_host, B * 4, cudaMemcpyHostToDevice, s));
  C2T_CALL(c2t_begin_step(ctx, root, prefix, s));
  for (size_t l = 0; l < D; ++l) {
    const int i = two ? (int)((D - 1 - l) & 1) : 0;
    if (used[i]) C2T_CUDA(cudaStreamWaitEvent(cs, ctx->consumed[i], 0));
    used[i] = true;
    if (l == 0)   // only the root's row of each sequence is ever read at level 0
      C2T_CUDA(cudaMemcpy2DAsync(stage[i], F * V * eb, io->draft_logits_host[0], F * V * eb, V * eb, B, cudaMemcpyHostToDevice, cs));
    else
      C2T_CUDA(cudaMemcpyAsync(stage[i], io->draft_logits_host[l], B * F * V * eb, cudaMemcpyHostToDevice, cs));
    C2T_CUDA(cudaEventRecord(ctx->copied[i], cs));
    C2T_CUDA(cudaStreamWaitEvent(s, ctx->copied[i], 0));
    C2T_CALL(c2t_expand_level(ctx, (int)l, stage[i], (int64_t)(F * V), (int64_t)V, s));
    C2T_CUDA(cudaEventRecord(ctx->consumed[i], s));
    C2T_CALL(c2t_prune(ctx, (int)l, nullptr, s));
  }
  C2T_CALL(c2t_prune(ctx, C2T_FINAL, nullptr, s));
  C2T_CALL(c2t_build_verify(ctx, &vo, s));
  if (used[1] || !apart) C2T_CUDA(cudaStreamWaitEvent(cs, ctx->consumed[used[1]], 0));
  C2T_CUDA(cudaMemcpyAsync(io->target_stage_dev, io->target_logits_host, B * Nw * V * eb, cudaMemcpyHostToDevice, cs));
  C2T_CUDA(cudaEventRecord(ctx->copied[1], cs));
  C2T_CUDA(cudaStreamWaitEvent(s, ctx->copied[1], 0));
  C2T_CALL(c2t_accept(ctx, io->target_stage_dev, (int64_t)(Nw * V), (int64_t)V, &ao, s));
  if (io->n_nodes_host) C2T_CUDA(cudaMemcpyAsync(io->n_nodes_host, vo.n_nodes, B * 4, cudaMemcpyDeviceToHost, s));
  if (io->tokens_host) C2T_CUDA(cudaMemcpyAsync(io->tokens_host, vo.tokens, B * Nw * 4, cudaMemcpyDeviceToHost, s));
  if (io->accept_len_host) C2T_CUDA(cudaMemcpyAsync(io->accept_len_host, ao.accept_len, B * 4, cudaMemcpyDeviceToHost, s));
  if (io->path_host) C2T_CUDA(cudaMemcpyAsync(io->path_host, ao.path, B * (D + 1) * 4, cudaMemcpyDeviceToHost, s));
  if (io->next_token_host) C2T_CUDA(cudaMemcpyAsync(io->next_token_host, ao.next_token, B * 4, cudaMemcpyDeviceToHost, s));
  C2T_CUDA(cudaStreamSynchronize(s));
  copies.stream = nullptr;                       // (every copy has a kernel behind it)
#undef C2T_CUDA
#undef C2T_CALL
  return C2T_OK;
}

int64_t c2t_launch_count(const c2t_ctx *ctx) { return ctx ? ctx->launches : 0; }

const char *c2t_strerror(int code) {
  switch (code) {
    case C2T_OK: return "ok";
    case C2T_EINVAL: return "invalid argument";
    case C2T_EALIGN: return "pointer or stride not aligned";
    case C2T_ERANGE: return "size out of range";
    case C2T_EORDER: return "call out of order";
    case C2T_ECUDA: return "CUDA runtime error";
    case C2T_ENOMEM: return "out of host memory";
    default: return "unknown error";
  }
}

}  // extern "C"

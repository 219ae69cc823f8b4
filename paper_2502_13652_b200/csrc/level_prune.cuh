// The per-sequence work of a level (Eq. 1, Eq. 4, Alg. 1, Sec. 4.2.2): features, classifier, the two prunings,
// compaction, tree append, from the results that the expand pass (or the merge of gathered records) has per row.  A device function, so that the pruning kernel
// (one CTA per sequence) and the expand kernels that prune in the same launch (by their last CTA, or a sequence's last) share it.
#pragma once

#include "c2t_internal.h"

namespace c2t {
namespace {

constexpr int kMaxCand = C2T_MAX_TOPK * C2T_MAX_FRONTIER;   // 1024
constexpr unsigned kFullMask = 0xFFFFFFFFu;

__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(kFullMask, v, o);
  return __shfl_sync(kFullMask, v, 0);
}

// ---------------------------------------------------------------- a level ---

// The classifier's weights in shared memory, as doubles (a conversion per use costs more than the arithmetic): per hidden
// unit its three input weights, its bias, its output weight; w[kW0] is the output bias.
constexpr int kWStride = 6;                       // (16-byte loads)
constexpr int kHiddenBatch = 4;
constexpr int kW0 = kWStride * C2T_MAX_HIDDEN;
static_assert(C2T_MAX_HIDDEN % kHiddenBatch == 0, "");
constexpr int kWCount = kW0 + 2;
__device__ __forceinline__ void stage_classifier(const TreeState &t, double *w, int tid, int n_threads) {
  if (t.classifier != C2T_CLS_MLP) return;
  for (int i = tid; i < 3 * t.hidden; i += n_threads) w[(i / 3) * kWStride + i % 3] = (double)t.w1[i];
  for (int i = tid; i < t.hidden; i += n_threads) {
    w[i * kWStride + 3] = (double)t.b1[i];
    w[i * kWStride + 4] = (double)t.w2[i];
  }
  const int padded = (t.hidden + kHiddenBatch - 1) & ~(kHiddenBatch - 1);
  for (int i = t.hidden * kWStride + tid; i < padded * kWStride; i += n_threads) w[i] = 0.0;
  if (tid == 0) w[kW0] = (double)t.b2[0];
}

// One copy of exp for all its callers in a kernel.  The kernels here are chains that run through their code once, and what code costs
// then is fetching it: about 400 cycles for a jump over something that is not in the instruction caches yet.
__device__ __noinline__ double exp_shared(double x) { return exp(x); }

// Confidence of one child (Eq. 4): two-layer FFN on (P, H, d), ReLU, sigmoid.
//   The hidden units are taken kHiddenBatch at a time, without a branch and with all of a batch's loads first: one after the other they are a
// chain of loads, additions and a comparison each (89 cycles per unit; the classification of a level 1.3 -> 0.6 us).
__device__ __forceinline__ double classify(int hidden, const double *w, double P, double H, double d) {
  double z[kHiddenBatch] = {w[kW0], 0.0, 0.0, 0.0};
#pragma unroll 1
  for (int k0 = 0; k0 < hidden; k0 += kHiddenBatch) {            // (units of weight 0 behind the last one)
    double2 a01[kHiddenBatch], a23[kHiddenBatch];
    double v[kHiddenBatch];
#pragma unroll
    for (int i = 0; i < kHiddenBatch; ++i) {
      const double *u = w + (k0 + i) * kWStride;
      a01[i] = *reinterpret_cast<const double2 *>(u);
      a23[i] = *reinterpret_cast<const double2 *>(u + 2);
      v[i] = u[4];
    }
#pragma unroll
    for (int i = 0; i < kHiddenBatch; ++i) {
      const double a = fma(a01[i].x, P, fma(a01[i].y, H, fma(a23[i].x, d, a23[i].y)));
      z[i] = fma(v[i], a < 0.0 ? 0.0 : a, z[i]);
    }
  }
  return 1.0 / (1.0 + exp_shared(-((z[0] + z[1]) + (z[2] + z[3]))));
}

// A row's merged sums, as one warp holds them.
struct RowMerge {
  double M, S, T;              // row maximum; sums over every other element of e^(x - M) and e^(x - M)(x - M)
  unsigned long long top;      // the row's best key (0: none)
  int n_valid;                 // candidates written (at most K)
};

// status bits of a row from its maximum and its sums
__device__ __forceinline__ uint32_t row_fault_bits(float top_x, double S, double T) {
  if (!(top_x > kNegInfAsFinite)) return C2T_ST_ALL_NEGINF;
  if (top_x == INFINITY) return C2T_ST_POSINF_LOGIT;
  if (S != S || T != T || isinf(S)) return C2T_ST_NAN_LOGIT;
  return 0u;
}

constexpr int kStageKeys = 320;
// One warp merges the gathered records of row (b, j): lane s holds shard s's record.  Writes the K
// best candidates to out_x / out_tok and returns the merged maximum and sums; *fault_out collects the
// shards' status bits ("all -inf" only if every shard says so).  stage: room for kStageKeys keys in shared memory, where
// the shards' lists are copied first if they fit (one after the other from global memory, a head costs a round trip).
__device__ RowMerge merge_row_records(const TreeState &t, const c2t_row_record *records, int n_shards, int b, int j,
                                      int K, float *out_x, int *out_tok, uint32_t *fault_out, unsigned long long *stage) {
  const int lane = threadIdx.x & 31;
  const size_t row = (size_t)b * t.F + j, shard_rows = (size_t)t.B * t.F;
  const c2t_row_record *rec = records + lane * shard_rows + row;
  const bool staged = n_shards * K <= kStageKeys;
  if (staged) {
#pragma unroll 4
    for (int i = lane; i < n_shards * K; i += 32) {
      const c2t_row_record *r = records + (i / K) * shard_rows + row;
      stage[i] = make_key(r->x[i % K], (uint32_t)r->tok[i % K]);
    }
  }
  double Mg = 0.0, Sg = 0.0, Tg = 0.0;
  int ng = 0;
  uint32_t fg = 0u;
  bool live = false;
  if (lane < n_shards) {
    Mg = rec->M; Sg = rec->S; Tg = rec->T; ng = rec->n; fg = rec->fault;
    ng = ng < 0 ? 0 : (ng > K ? K : ng);
    live = !(fg & C2T_ST_ALL_NEGINF);
  }
  const uint32_t fault = __reduce_or_sync(kFullMask, fg & ~(uint32_t)C2T_ST_ALL_NEGINF);
  // the row maximum is the best of the shards' maxima; equal values go to the lower shard, whose token ids are lower
  unsigned long long top = live ? (((unsigned long long)f32_orderable(__float_as_uint((float)Mg)) << 32) |
                                   (0xFFFFFFFFu - (uint32_t)lane)) : 0ull;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    unsigned long long other = __shfl_xor_sync(kFullMask, top, o);
    top = other > top ? other : top;
  }
  const int winner = (int)(0xFFFFFFFFu - (uint32_t)top);
  const double M = (double)key_value(top);
  double S = 0.0, T = 0.0;
  if (live) {
    const double d = Mg - M, f = exp(d);          // this shard's sums are relative to its own maximum
    S = f * Sg;
    T = f * (Tg + d * Sg);
    if (lane != winner) { S += f; T += f * d; }   // its maximum is an ordinary element of the row
  }
  S = warp_sum(S);
  T = warp_sum(T);
  __syncwarp();
  int n_valid = 0, pos = 0;
  for (; n_valid < K; ++n_valid) {                // the shards' lists are sorted: take the largest head K times
    unsigned long long h = 0ull;
    if (live && pos < ng) h = staged ? stage[lane * K + pos] : make_key(rec->x[pos], (uint32_t)rec->tok[pos]);
    const uint32_t hi = (uint32_t)(h >> 32), mx_hi = __reduce_max_sync(kFullMask, hi);
    const uint32_t mx_lo = __reduce_max_sync(kFullMask, hi == mx_hi ? (uint32_t)h : 0u);
    const unsigned long long mx = ((unsigned long long)mx_hi << 32) | mx_lo;
    if (mx == 0ull) break;
    if (lane == 0) { out_x[n_valid] = key_value(mx); out_tok[n_valid] = key_token(mx); }
    if (h == mx) ++pos;
  }
  for (int r = n_valid + lane; r < K; r += 32) { out_x[r] = -INFINITY; out_tok[r] = -1; }
  __syncwarp();
  *fault_out = fault;
  RowMerge m;
  m.M = M; m.S = S; m.T = T; m.top = top; m.n_valid = n_valid;
  return m;
}

constexpr int kCapBlock = 128;                 // keys that the frontier cap compares with at a time
static_assert(kMaxCand % kCapBlock == 0 && 256 % kCapBlock == 0, "the last block ends within the threads' last round");
// The shared memory of prune_level_body.
struct PruneShared {
  double rowM[C2T_MAX_FRONTIER], rowL[C2T_MAX_FRONTIER], rowH[C2T_MAX_FRONTIER];
  double flogP[C2T_MAX_FRONTIER];              // joint log-probability of every frontier node
  double fchat[C2T_MAX_FRONTIER];              // its smallest confidence on the path from the root
  int fnode[C2T_MAX_FRONTIER];                 // tree id of every frontier node
  int rowfault[C2T_MAX_FRONTIER];
  alignas(16) unsigned long long ckey[kMaxCand + 2];   // confidence of every candidate as an orderable integer, 0 for a dropped one and behind the last
  alignas(16) unsigned chi[kMaxCand];           // its upper half, zeros behind the last one up to a whole block of kCapBlock
  int count[32];                               // candidates added and selected, per 32
  int next, n_equal;                           // first_of_equals: the smallest reach above the cap, candidates that have it
  short reach[kMaxCand];                       // survivors whose upper halves are at or above a candidate's
};
// ... and with gathered records, behind it:
struct GatherShared {
  float x[kMaxCand];
  int tok[kMaxCand];
  unsigned long long stage[16][kStageKeys];
};

// One row's maximum, normaliser and entropy into shared memory; its fault into the status word.
__device__ __forceinline__ void row_stats(const TreeState &t, const RowResult &r, const double2 &sm, int b, int j, PruneShared &sh) {
  sh.rowM[j] = r.M;
  sh.rowL[j] = r.L;
  if (t.entropy_top_m > 0 && t.entropy_top_m < t.V) sh.rowH[j] = (r.L * sm.x - sm.y) / (1.0 + r.S);   // Eq. 3: only the M most
                                                                // probable tokens, probabilities of the full softmax
  else sh.rowH[j] = r.H;                                        // Eq. 2
  sh.rowfault[j] = (int)r.fault;
  if (r.fault) atomicOr(&t.status[b], r.fault);
}

// Where the upper halves leave less than F selected: the candidates of the next larger reach, all with the same upper half, share the room that
// is left by lower half and index.  `have` are selected; kept: which of the thread's candidates survive (a bit per round).  Returns
// which of them are among the first.  Called by all threads (sh.n_equal and sh.next are as at the level's start).
template <int NT, int ROUNDS>
__device__ __noinline__ unsigned first_of_equals(PruneShared &sh, unsigned kept, int have, int F) {
  const int tid = threadIdx.x, lane = tid & 31;
  unsigned least = 0x7FFFu;
#pragma unroll
  for (int r = 0; r < ROUNDS; ++r) {
    const unsigned reach = kept >> r & 1u ? (unsigned)sh.reach[tid + r * NT] : 0u;
    if (reach > (unsigned)F && reach < least) least = reach;
  }
  least = __reduce_min_sync(kFullMask, least);
  if (lane == 0) atomicMin(&sh.next, (int)least);
  __syncthreads();
  const int next = sh.next, n = next - have;
  unsigned long long key[ROUNDS];
#pragma unroll
  for (int r = 0; r < ROUNDS; ++r) {
    const int c = tid + r * NT;
    key[r] = (kept >> r & 1u) && sh.reach[c] == next ? sh.ckey[c] << 32 | (0xFFFFFFFFu - (unsigned)c) : 0ull;
  }
  __syncthreads();                                // the keys are free now: the list takes their place
#pragma unroll
  for (int r = 0; r < ROUNDS; ++r)
    if (key[r]) sh.ckey[atomicAdd(&sh.n_equal, 1)] = key[r];
  if (tid == 0) sh.ckey[n] = 0ull;
  __syncthreads();
  unsigned first = 0u;
#pragma unroll
  for (int r = 0; r < ROUNDS; ++r) {
    if (!key[r]) continue;
    int before = 0;
#pragma unroll 4
    for (int o = 0; o < n; o += 2) {
      const ulonglong2 k = *reinterpret_cast<const ulonglong2 *>(&sh.ckey[o]);
      before += (k.x > key[r]) + (k.y > key[r]);
    }
    first |= (unsigned)(before < F - have) << r;
  }
  return first;
}

// NT: threads of the CTA; b: the sequence; w: the classifier's staged weights.  records == nullptr: the rows come from
// this context's own expand pass; else from gathered records of n_shards shards (gs: room for their merge).
//   The work is a chain of dependent steps over at most F K candidates, on the critical path of every level, so it is short
// in steps rather than in operations: every global load whose address does not depend on another is issued at the top
// (frontier nodes carry their log-probabilities and path confidences with them for that), a thread keeps its
// candidates in registers, the cap ranks a candidate with several threads, and the compaction needs one barrier.
// Eight levels of 64 sequences: 323 -> 314 us (expand and prune).  And it is short in code, which is cold whenever a level's last block is
// on another SM than the last level's: a candidate per thread where that is enough (ROUNDS 1), what is rarely needed in functions of its
// own, loops that are not unrolled.
template <int NT, int ROUNDS, bool GATHERED>
__device__ __forceinline__ void prune_level_body(const TreeState &t, int level, const c2t_frontier &out, const c2t_row_record *records,
                                                 int n_shards, int b, PruneShared &sh, const double *w, GatherShared *gs) {
  constexpr int kRounds = ROUNDS, kNW = NT / 32;               // candidates per thread; warps
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int K = t.K, F = t.F;
  const int cur = level & 1, nxt = cur ^ 1;
  const size_t cbase = (size_t)b * F * K, fbase = (size_t)b * F;
  const unsigned per_k = (65536u + (unsigned)K - 1u) / (unsigned)K;       // c / K = c per_k >> 16 for c < 1024, K <= 32

  // ---- loads (slots past the frontier's size hold anything: kept in bounds, unused)
  int n = t.frontier_n[cur][b];
  const int base = t.tree_n[b];
  unsigned long long key[kRounds];
#pragma unroll
  for (int r = 0; r < kRounds; ++r) {
    const int c = tid + r * NT;
    key[r] = !GATHERED && c < F * K ? __ldcg(&t.row_keys[cbase + c]) : 0ull;
  }
  const int jr = tid - (NT - 64), jf = tid - (NT - 32);        // the last two warps fetch the rows' and the frontier's data
  RowResult row;
  double2 sm = make_double2(0.0, 0.0);
  if (!GATHERED && jr >= 0 && jr < F) {
    row = t.rows[fbase + jr];
    if (t.entropy_top_m > 0) sm = t.topm[fbase + jr];
  }
  int fnode = 0;
  double flogP = 0.0, fchat = 0.0;
  if (jf >= 0 && jf < F) {
    fnode = t.frontier_node[cur][fbase + jf];
    flogP = t.frontier_logP[cur][fbase + jf];
    fchat = t.frontier_chat[cur][fbase + jf];
  }
  n = n < 0 ? 0 : (n > F ? F : n);
  if (n == 0) {                                   // the loop of Alg. 1 has ended for this sequence
    if (tid == 0) {
      t.frontier_n[nxt][b] = 0;
      t.cand_n[b] = 0;
      if (out.count) out.count[b] = 0;
    }
    return;
  }
  __syncthreads();                                // (a CTA that serves several sequences: the last one's reads are done)
  if (!GATHERED) {
    if (jr >= 0 && jr < n) row_stats(t, row, sm, b, jr, sh);
  } else {
    for (int j = warp; j < n; j += kNW) {
      uint32_t shard_faults = 0u;
      const RowMerge m = merge_row_records(t, records, n_shards, b, j, K, &gs->x[j * K], &gs->tok[j * K], &shard_faults, gs->stage[warp]);
      if (lane == 0) {
        RowResult r;
        r.M = m.M; r.S = m.S; r.T = m.T;
        r.L = log1p(m.S);
        r.H = r.L - m.T / (1.0 + m.S);
        r.fault = shard_faults ? shard_faults : row_fault_bits(m.top ? key_value(m.top) : -INFINITY, m.S, m.T);
        row_stats(t, r, sm, b, j, sh);
      }
    }
  }
  if (jf >= 0 && jf < n) {
    sh.fnode[jf] = fnode;
    sh.flogP[jf] = flogP;
    sh.fchat[jf] = fchat;
  }
  if (tid == 0) { sh.next = 0x7FFF; sh.n_equal = 0; }
  __syncthreads();

  // ---- features and confidence, a thread per candidate child
  const int nc = n * K, nc_blocks = (nc + kCapBlock - 1) & ~(kCapBlock - 1);
  double C[kRounds], logP[kRounds];
  int tok[kRounds];
  bool keep[kRounds], sel[kRounds];
  int n_keep = 0;
#pragma unroll
  for (int r = 0; r < kRounds; ++r) {
    const int c = tid + r * NT;
    keep[r] = false;
    if (r * NT < nc) {                            // (uniform)
      if (c >= nc && c < nc_blocks) { sh.chi[c] = 0u; sh.ckey[c] = 0ull; }
      if (c < nc) {
        const int j = (int)((unsigned)c * per_k >> 16);
        float x;
        if (GATHERED) { x = gs->x[c]; tok[r] = gs->tok[c]; }
        else { x = key[r] ? key_value(key[r]) : -INFINITY; tok[r] = key[r] ? key_token(key[r]) : -1; }
        const bool ok = tok[r] >= 0 && !sh.rowfault[j];
        const double lp = (x > kNegInfAsFinite) ? ((double)x - sh.rowM[j]) - sh.rowL[j] : -INFINITY;
        logP[r] = sh.flogP[j] + lp;                                             // Eq. 1 in log space
        const double P = exp_shared(logP[r]);
        const double H = sh.rowH[j];
        if (!ok) C[r] = NAN;
        else if (t.classifier == C2T_CLS_IDENTITY_JOINT) C[r] = P;
        else if (t.classifier == C2T_CLS_IDENTITY_COND) C[r] = exp_shared(lp);
        else C[r] = classify(t.hidden, w, P, H, (double)level);
        keep[r] = ok && C[r] >= (double)t.beta;                                 // first pruning
        // (C desc, index asc) as integer compares: an orderable image of C, 0 for a dropped candidate
        const unsigned long long cb = (unsigned long long)__double_as_longlong(C[r]);
        sh.ckey[c] = keep[r] ? (cb ^ ((cb >> 63) ? ~0ull : 0x8000000000000000ull)) : 0ull;
        sh.chi[c] = (unsigned)(sh.ckey[c] >> 32);
        t.cand_token[cbase + c] = tok[r];
        t.cand_lp[cbase + c] = ok ? lp : NAN;
        t.cand_logP[cbase + c] = ok ? logP[r] : NAN;
        t.cand_H[cbase + c] = ok ? H : NAN;
        t.cand_C[cbase + c] = C[r];
      }
      n_keep += __syncthreads_count(keep[r]);
    }
    sel[r] = keep[r];
  }

  // ---- second pruning: the F survivors that come first under (C desc, index asc).  kParts threads count the survivors at or above a
  // candidate by the upper halves of the keys, four to a load.  Where no more than F of them are, it is selected; those that share the
  // next larger count have equal upper halves and share what is left: the usual case where K > F, whose cut falls among one row's children (of
  // ever smaller joint probabilities: their keys share 35 to 60 bits).  Five levels of 9 x 23862 fp32 tokens, K = 10, 12, 14, 16, F = 10: 92, 97,
  // 106, 106 us; ranked a second time by whole keys where the halves do not decide 92, 102, 120, 121; by whole keys alone 99, 102, 117, 121.
  if (n_keep > F) {
    constexpr int kParts = NT >= 512 ? 4 : 2, kLoads = kCapBlock / kParts / 4;
    const int part = tid % kParts;
    for (int c0 = 0; c0 < nc; c0 += NT / kParts) {
      const int c = c0 + tid / kParts;
      const unsigned kc = c < nc ? sh.chi[c] : 0xFFFFFFFFu;
      int n_reach = 0;                              // (itself among them)
#pragma unroll 1
      for (int o = 0; o < nc; o += kCapBlock) {
#pragma unroll 1
        for (int i0 = 0; i0 < kLoads; i0 += 8) {
          uint4 k[8];
#pragma unroll
          for (int i = 0; i < 8; ++i) k[i] = *reinterpret_cast<const uint4 *>(&sh.chi[o + ((i0 + i) * kParts + part) * 4]);
          int more[4] = {0, 0, 0, 0};
#pragma unroll
          for (int i = 0; i < 8; ++i) {
            more[0] += k[i].x >= kc;
            more[1] += k[i].y >= kc;
            more[2] += k[i].z >= kc;
            more[3] += k[i].w >= kc;
          }
          n_reach += (more[0] + more[1]) + (more[2] + more[3]);
        }
      }
#pragma unroll
      for (int m = 1; m < kParts; m <<= 1) n_reach += __shfl_xor_sync(kFullMask, n_reach, m);
      if (part == 0 && c < nc) sh.reach[c] = (short)n_reach;
    }
    __syncthreads();
#pragma unroll
    for (int r = 0; r < kRounds; ++r)
      if (tid + r * NT < nc) sel[r] = keep[r] && sh.reach[tid + r * NT] <= F;
  }

  // ---- stable compaction in candidate order; append to the tree, emit the frontier
  const bool add_all = t.tree_add == C2T_ADD_ALL_SURVIVORS;
  unsigned add_mask[kRounds], sel_mask[kRounds];
  auto count_up = [&] {
#pragma unroll
    for (int r = 0; r < kRounds; ++r) {
      add_mask[r] = __ballot_sync(kFullMask, add_all ? keep[r] : sel[r]);
      sel_mask[r] = __ballot_sync(kFullMask, sel[r]);
      if (lane == 0) sh.count[r * kNW + warp] = __popc(add_mask[r]) | (__popc(sel_mask[r]) << 16);    // (each total at most 1024)
    }
    __syncthreads();
    return lane < kRounds * kNW ? sh.count[lane] : 0;
  };
  int counts = count_up(), total = __reduce_add_sync(kFullMask, counts);
  if (n_keep > F && (total >> 16) != F) {           // (uniform)
    unsigned kept = 0u;
#pragma unroll
    for (int r = 0; r < kRounds; ++r) kept |= (unsigned)keep[r] << r;
    const unsigned first = first_of_equals<NT, kRounds>(sh, kept, total >> 16, F);
#pragma unroll
    for (int r = 0; r < kRounds; ++r) sel[r] = sel[r] || (first >> r & 1u);
    counts = count_up();
    total = __reduce_add_sync(kFullMask, counts);
  }
  static_assert(kRounds * kNW <= 32, "a count per lane");
  const int tot_add = total & 0xFFFF, tot_sel = total >> 16;
  const bool overflow = base + tot_add > t.cap;
  const size_t tb = (size_t)b * t.cap;
#pragma unroll
  for (int r = 0; r < kRounds; ++r) {
    const int c = tid + r * NT;
    if (r * NT >= nc) break;                      // (uniform)
    const int before = __reduce_add_sync(kFullMask, lane < r * kNW + warp ? counts : 0);
    if (c >= nc) continue;
    t.cand_flags[cbase + c] = (keep[r] ? 1 : 0) | (sel[r] ? 2 : 0);
    if (!(add_all ? keep[r] : sel[r])) continue;
    const unsigned lt = (1u << lane) - 1u;
    const int id = base + (before & 0xFFFF) + __popc(add_mask[r] & lt);
    const int j = (int)((unsigned)c * per_k >> 16);
    const double chat = C[r] < sh.fchat[j] ? C[r] : sh.fchat[j];
    if (id < t.cap) {
      t.tree_token[tb + id] = tok[r];
      t.tree_parent[tb + id] = sh.fnode[j];
      t.tree_level[tb + id] = level + 1;
      t.tree_logP[tb + id] = logP[r];             // (a node is only added if its candidate was in order)
      t.tree_C[tb + id] = C[r];
      t.tree_Chat[tb + id] = chat;
    }
    if (sel[r] && !overflow) {
      const int slot = (before >> 16) + __popc(sel_mask[r] & lt);
      if (!C2T_IN_BOUNDS(slot, F, &t.status[b])) continue;
      t.frontier_node[nxt][fbase + slot] = id;
      t.frontier_logP[nxt][fbase + slot] = logP[r];
      t.frontier_chat[nxt][fbase + slot] = chat;
      if (out.token) out.token[fbase + slot] = tok[r];
      if (out.node_id) out.node_id[fbase + slot] = id;
      if (out.parent_slot) out.parent_slot[fbase + slot] = j;
    }
  }
  if (tid == 0) {
    const int next_n = overflow ? 0 : tot_sel;
    t.tree_n[b] = overflow ? t.cap : base + tot_add;
    t.frontier_n[nxt][b] = next_n;
    t.cand_n[b] = nc;
    if (out.count) out.count[b] = next_n;
    if (overflow) atomicOr(&t.status[b], C2T_ST_TREE_OVERFLOW);
  }
}

}  // namespace
}  // namespace c2t

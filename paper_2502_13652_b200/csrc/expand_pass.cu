// The expand pass: one streaming read of every active draft-logits row, giving per row the
// softmax normaliser and entropy sums and the K largest logits (ties to the lower token id)
//                                                        (Sec. 4.2.1, Eq. 2, Sec. 4.2.2).
//
// Work partition.  A row is cut into chunks of 256 consecutive 16-byte vectors (4 KB).  The chunks
// of the active rows (a device-side count per sequence), laid end to end, are dealt out in
// contiguous equal ranges, one per CTA of a persistent grid (one CTA per SM).  Most warps of a CTA
// stream, taking its chunks in turn; the others complete rows, in pairs, as soon as all chunks of
// a row are done: while the stream goes on, but for the last row.
//
// Stream.  A warp keeps one chunk in registers, 8 vectors per lane, in two groups; as soon as a
// group has been consumed the same registers are requested for the same group of the warp's next chunk,
// so one to two groups (2 to 4 KB per warp) are in flight all the time.  Per element the
// stream does nothing but the sums and a running maximum: no comparison with a filter, no vote, no
// branch that depends on the data.  Selection of the K largest is left to the row's end, where the
// maxima say where to look.
//
// Sums.  Per lane, in base-2 units relative to an integer offset c = floor(-m log2(e)), m the largest value of the row that
// the lane has met, the group at hand included:  t = x log2(e) + c,  S = sum 2^t,  U = sum 2^t t,  two elements at a time
// (packed fp32 FMA and add).  The offset follows m before a group is summed, without a branch and without asking other lanes,
// so t is never positive: the elements that make up most of the sums have the smallest t and with it the smallest
// rounding of t, U is a sum of one sign that rescaling does not cancel, and no row overflows.  Offsets are integers, so
// rescaling is by exact powers of two.  (Rows of 128256 values of scale 8: a probability's error is 7e-9 r.m.s. and 4e-8 at most,
// an entropy's 1e-7; relative to the largest value of a row's first group they were 2e-7, 1e-6 and 3e-6, and rows whose head lies 87 nats
// below their maximum lost sums.  A warp-wide reference, raised after a vote per group, costs 3 % of a level, a lane's own nothing.)
//
// Top-K.  Every lane records the maximum of its vectors of a chunk, its "cell".  When all chunks of a
// row are done the row is completed: the K-th largest of the 32 lanes' column maxima
// is a lower bound on the row's K-th largest element, the few cells that reach it are read again (128 bytes each,
// usually from L2), their elements at or above the bound are ranked by key, and the warps' sums are merged in double
// precision.  The row's largest element stays out of the sums, so that they keep fp32 relative accuracy with respect to
// "everything but the maximum" however peaked the row is: the one lane and chunk that holds it is summed again without it.
// Everything is computed in an order that does not depend on timing, so the results are reproducible bit for bit.
#include "row_sums.cuh"

namespace c2t {
namespace {

constexpr int kStreamWarps = kExpandWarps;            // the first warps of a CTA stream ...
constexpr int kEWarps = kExpandThreads / 32;          // ... the others only complete rows
constexpr int kPairs = kEWarps / 2;
constexpr int kGroups = kChunkVecs / 128;             // groups of a chunk; a lane holds 4 vectors of each, 32 apart
constexpr int kListCap = 128;                         // cells of a row that are read again
static_assert(kStreamWarps % 2 == 0 && kPairs <= 15, "pairs of warps, one named barrier each");

// What a pair of warps needs in shared memory to complete a row.
struct PairShared {
  unsigned long long pool[kPoolCap];
  __align__(16) float colmax[64];
  int list[kListCap], vecs[kListCap];
  __align__(16) uint4 data[kListCap];
};

// A CTA's shared memory; behind it a transaction barrier per task (a row, or the CTA's part of one) and the row list.
struct CtaShared {
  PairShared scratch[kPairs];
  int task, flag[kPairs], task_of[kPairs];            // the next task; what the first warp of a pair tells the other
  int pad;
  __device__ unsigned long long *bars() { return reinterpret_cast<unsigned long long *>(this + 1); }
};

// the float just above a value
__device__ __forceinline__ float just_above(float x) {
  return __uint_as_float(f32_from_orderable(f32_orderable(__float_as_uint(x)) + 1u));
}

// ---------------------------------------------------------------- a warp's sums of a row

// A lane's sums of the chunks of a row that its warp streams; the chunk with the lane's largest value is kept apart.
struct LaneSums {
  Acc acc;                   // the current chunk, relative to c
  float S, U;                // finished chunks but the held one, relative to cf
  float Sh, Uh;              // the held chunk, relative to cf
  int hch;
  float ref, c, cf;          // the lane's largest value; the offset taken from it, and as it was at the last chunk's end
  f32x2 c2;                  // c, twice
  __device__ __forceinline__ void start() {
    acc.clear();
    S = U = Sh = Uh = 0.f;
    ref = kLowestF32;
    hch = 0;
    cf = kNoOffset;
  }
  // before a group with this maximum is summed
  __device__ __forceinline__ void begin_group(float m, bool first) {
    ref = fmaxf(ref, m);
    const float next = offset_of(ref);
    if (!first) {                                     // (the chunk has been summed in part)
      const Shift by(next - c);
#pragma unroll
      for (int i = 0; i < 2; ++i) by.apply(acc.S[i], acc.U[i]);
    }
    c = next;
    c2 = pack2(c, c);
  }
  // what is finished, to another offset
  __device__ __forceinline__ void move_finished(float to) {
    const Shift by(to - cf);
    f32x2 s = pack2(S, Sh), u = pack2(U, Uh);
    by.apply(s, u);
    unpack2(s, S, Sh);
    unpack2(u, U, Uh);
    cf = to;
  }
  __device__ __forceinline__ void end_chunk(bool best, int ch) {       // best: the chunk raised the lane's largest value
    move_finished(c);
    float s, u;
    acc.totals(s, u);
    acc.clear();
    S += best ? Sh : s;
    U += best ? Uh : u;
    Sh = best ? s : Sh;
    Uh = best ? u : Uh;
    hch = best ? ch : hch;
  }
};

// The lanes' sums over the warp into a record, relative to the warp's largest value.
__device__ __forceinline__ void write_record(SumRecord *rec, LaneSums &ls) {
  const int lane = threadIdx.x & 31;
  const uint32_t ord = f32_orderable(__float_as_uint(ls.ref)), top = __reduce_max_sync(kFull, ord);
  const float m = __uint_as_float(f32_from_orderable(top));
  ls.move_finished(offset_of(m));
  const int t = __ffs(__ballot_sync(kFull, ord == top)) - 1;
  float s = ls.S, u = ls.U;
  if (lane == t) {
    rec->held = make_float4(ls.Sh, ls.Uh, __int_as_float(t), __int_as_float(ls.hch));
  } else {
    s += ls.Sh;
    u += ls.Uh;
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    s += __shfl_xor_sync(kFull, s, o);
    u += __shfl_xor_sync(kFull, u, o);
  }
  if (lane == 0) rec->rest = make_float4(s, u, ls.cf, m);
}

// ---------------------------------------------------------------- rows and chunks

template <bool BF16>
struct RowShape {
  int vpr, v_full, nc, words;  // vectors of a row (the last may be ragged), whole ones, chunks, words of two cells per lane
  __device__ __forceinline__ explicit RowShape(int V) {
    vpr = (V + Vec<BF16>::N - 1) / Vec<BF16>::N;
    v_full = V / Vec<BF16>::N;
    nc = (vpr + kChunkVecs - 1) / kChunkVecs;
    words = (nc + 1) / 2;
  }
};

__device__ __forceinline__ const char *row_pointer(const PassParams &p, int b, int j, size_t esz) {
  return reinterpret_cast<const char *>(p.logits) + ((size_t)b * p.seq_stride + (size_t)j * p.row_stride) * esz;
}

// Requests group g of a chunk: src points at the lane's first vector of the chunk, nv counts the whole vectors from the
// chunk's start on.  Vectors past them become the lowest value, which adds exactly 0 to the sums.
template <bool BF16>
__device__ __forceinline__ void load_group(uint4 (&q)[4], const uint4 *src, int g, int nv, int lane) {
  const uint32_t lo = BF16 ? kLowestBf16x2 : __float_as_uint(kLowestF32);
  if (nv >= (g + 1) * 128) {
#pragma unroll
    for (int k = 0; k < 4; ++k) q[k] = ldg_stream(src + g * 128 + k * 32);
  } else {
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      q[k] = make_uint4(lo, lo, lo, lo);
      if (g * 128 + k * 32 + lane < nv) q[k] = ldg_stream(src + g * 128 + k * 32);
    }
  }
}

// Cells are bf16, fp32 maxima rounded towards -inf: the floor taken from them is still reached by K elements, and a cell
// with an element that reaches the floor still reaches it.  The lower halves of fp32 maxima are kept apart, for select_in_order.
__device__ __forceinline__ uint32_t cell_bits(float x, bool exact) {
  uint32_t b = __float_as_uint(x);
  if (!exact && (b & 0x80000000u)) b += 0xFFFFu;      // (a negative value: towards the larger magnitude)
  return b >> 16;
}

// the maximum of an fp32 cell from its rounded and its lower half
__device__ __forceinline__ float whole_cell(uint32_t cell, uint32_t low) {
  return __uint_as_float(((cell & 0x8000u) && low ? cell - 1u : cell) << 16 | low);
}

// How the launch cut the rows, as one CTA sees it.  CTA i has chunks [i per_cta, (i + 1) per_cta) of the rows laid end to end.
// Its tasks are its part of its last row, if it shares that row with the next CTA, its part of its first row, if it shares
// that one, and the rows inside.  It streams them in this order, so that shared rows are complete early.
//   TOPM: the CTA's range in natural order, an equal contiguous part per warp (a part's floor serves all its chunks).
template <bool TOPM>
struct CtaRange {
  int nc, per_cta, u0, u1;     // chunks per row and per CTA; this CTA's chunks
  int in0, in1;                // the rows inside
  int tail, head;              // chunks of the shared last row (if it is not the first as well) and of the shared first row
  int part, busy;              // TOPM: chunks of a warp; warps of the grid with chunks, as if every CTA had per_cta
  __device__ __forceinline__ CtaRange(int nc_, int total) : nc(nc_) {
    per_cta = (total + (int)gridDim.x - 1) / (int)gridDim.x;
    part = (per_cta + kStreamWarps - 1) / kStreamWarps;
    u0 = (int)blockIdx.x * per_cta;
    u1 = u0 + per_cta < total ? u0 + per_cta : total;
    const int a0 = u0 / nc, a1 = u1 > u0 ? (u1 - 1) / nc : a0;
    in0 = a0 * nc < u0 ? a0 + 1 : a0;
    in1 = (a1 + 1) * nc > u1 ? a1 : a1 + 1;
    head = in0 > a0 ? (in0 * nc < u1 ? in0 * nc : u1) - u0 : 0;
    if (in0 == a0 && in1 == a0) { head = u1 - u0; in0 = in1 = a0 + 1; }     // a row begins here and ends beyond
    tail = in1 <= a1 && in1 >= in0 && a1 > a0 ? u1 - a1 * nc : 0;
    if (in1 < in0) in1 = in0;
    busy = 0;
    if (TOPM && per_cta > 0) busy = (total + per_cta - 1) / per_cta * ((per_cta + part - 1) / part);
  }
  __device__ __forceinline__ int chunk_at(int i) const {              // the i-th chunk of the work order
    if (TOPM) return u0 + i;
    return i < tail ? u1 - tail + i : u0 + i - tail;                  // (the first row's part lies before the rows inside)
  }
  __device__ __forceinline__ int n_tasks() const { return (tail > 0) + (head > 0) + in1 - in0; }
  __device__ __forceinline__ int task_row(int k) const {
    if (tail > 0 && k-- == 0) return in1;
    if (head > 0 && k-- == 0) return in0 - 1;
    return in0 + k;
  }
  __device__ __forceinline__ int row_task(int a) const {
    if (a < in0) return tail > 0;
    if (a >= in1) return 0;
    return (tail > 0) + (head > 0) + a - in0;
  }
  __device__ __forceinline__ int task_chunks(int a) const { return a < in0 ? head : (a >= in1 ? tail : nc); }
  // records that the CTA's warps write for row a
  __device__ __forceinline__ int task_records(int a) const {
    const int n = task_chunks(a);
    if (!TOPM) return n < kStreamWarps ? n : kStreamWarps;
    const int from = (a * nc > u0 ? a * nc : u0) - u0;
    return (from + n - 1) / part - from / part + 1;
  }
  // does the warp that streams chunk u of row a write its record after it?
  __device__ __forceinline__ bool ends_record(int u, int a) const {
    const int cta = u / per_cta, row_end = (a + 1) * nc, cta_end = (cta + 1) * per_cta, end = row_end < cta_end ? row_end : cta_end;
    if (!TOPM) return end - u <= kStreamWarps;
    return u + 1 == end || (u - cta * per_cta + 1) % part == 0;
  }
};

// NEAR: the cells of a row inside the CTA's range are in shared memory, those of a row that it shares in the workspace.  For fp32 rows of
// kNearChunks chunks or more, where a CTA has two rows or more.  Shorter rows lose by it (steps of five levels and the acceptance, cells in
// shared memory against the workspace: 400 rows of 32000 tokens 145.4 : 143.4 us, of 48000 180.4 : 178.4, of 64000 211.9 : 210.0, of 96000
// 282.2 : 281.9), long ones gain where a CTA has few (eight levels of 320 rows of 128256 391 : 395, five 295.8 : 296.5, of 480 rows 401.0 : 400.7).
// With less than two rows a CTA nearly all rows are shared (90 rows of 23862 92.9 : 92.0, 200 of 128256 224 : 221).  The bf16 stream, which has
// no time to spare, loses by the other kind of store (640 rows 465 -> 468).
constexpr int kNearChunks = 96;
template <bool BF16, bool TOPM>
__device__ __forceinline__ uint32_t *cells_of_row(const PassParams &p, uint32_t *near, const CtaRange<TOPM> &cr, const RowShape<BF16> &rs, int a) {
  return a >= cr.in0 && a < cr.in1 ? near + (size_t)(a - cr.in0) * rs.words * 32 : p.cells + (size_t)a * rs.words * 32;
}

// ---------------------------------------------------------------- completing a row

// vector k of the lane's 8 in a chunk
__device__ __forceinline__ int cell_vector(int chunk, int lane, int k) { return chunk * kChunkVecs + lane + 32 * k; }

template <bool BF16>
__device__ __forceinline__ float element(const char *row, int tok) {    // -inf as the lowest finite value
  const float x = BF16 ? __uint_as_float((uint32_t)__ldg(reinterpret_cast<const unsigned short *>(row) + tok) << 16)
                       : __ldg(reinterpret_cast<const float *>(row) + tok);
  return x < kLowestF32 ? kLowestF32 : x;
}

// N vectors of a row, clamped; the lowest value past the row's end
template <bool BF16, int N>
__device__ __forceinline__ void load_vectors(uint4 (&q)[N], const char *row, const int (&v)[N], const RowShape<BF16> &rs, int V) {
  const uint32_t lo = BF16 ? kLowestBf16x2 : __float_as_uint(kLowestF32);
#pragma unroll
  for (int u = 0; u < N; ++u) {
    q[u] = make_uint4(lo, lo, lo, lo);
    if (v[u] < rs.v_full) q[u] = __ldg(reinterpret_cast<const uint4 *>(row) + v[u]);
  }
  if (rs.vpr != rs.v_full) {
#pragma unroll
    for (int u = 0; u < N; ++u)
      if (v[u] == rs.v_full) q[u] = load_ragged<BF16>(row, rs.v_full, rs.v_full, V);
  }
#pragma unroll
  for (int u = 0; u < N; ++u) Vec<BF16>::clamp(q[u]);
}

// Which of N values of a lane reach x in any lane, as bits.
template <int N>
__device__ __forceinline__ unsigned reached(const float (&v)[N], float x) {
  unsigned bits = 0u;
#pragma unroll
  for (int i = 0; i < N; ++i) bits |= (unsigned)__any_sync(kFull, v[i] >= x) << i;
  return bits;
}

// Rows whose K largest do not come out of a short list (many equal values, few values, most of the row masked): the chunks whose
// maxima reach a filter, in order, elements in token order 32 at a time; the filter rises to just above the K-th value.  The maxima are
// taken whole here: with the rounded ones every chunk of a masked fp32 row stays in question (four levels of 320 rows of
// 128256 values, six of them finite: 2085 us, so 223).
template <bool BF16, bool NEAR>
__device__ __noinline__ int select_in_order(const PassParams &p, PairShared *ws, const char *row, const uint32_t *cells, int a, float floor) {
  constexpr int kWords = 8;                         // words of cells of a lane at a time
  constexpr int kBatch = 16;                        // elements of a lane in flight
  const RowShape<BF16> rs(p.V);
  const int lane = threadIdx.x & 31, K = p.K;
  int have = 0;                                     // keys kept in pool[0 .. K)
  float thr = floor;
  for (int w0 = 0; w0 < rs.words; w0 += kWords) {
    uint32_t two[kWords], low[kWords];
    float most[kWords];
#pragma unroll
    for (int i = 0; i < kWords; ++i) {
      const size_t at = ((size_t)a * rs.words + w0 + i) * 32 + lane;
      two[i] = w0 + i < rs.words ? (NEAR ? cells[(w0 + i) * 32 + lane] : p.cells[at]) : 0xFF80FF80u;
      low[i] = !BF16 && w0 + i < rs.words ? p.cell_low[at] : 0u;
    }
#pragma unroll
    for (int i = 0; i < kWords; ++i) most[i] = fmaxf(whole_cell(two[i] & 0xFFFFu, low[i] & 0xFFFFu), whole_cell(two[i] >> 16, low[i] >> 16));
    unsigned left = (1u << kWords) - 1u;
    for (unsigned hit; (hit = reached(most, thr) & left) != 0u;) {
      const int w = w0 + __ffs(hit) - 1;
      left &= ~((2u << (w - w0)) - 1u);
      const int t1 = (w + 1) * 2 * kChunkVecs * Vec<BF16>::N, end = t1 < p.V ? t1 : p.V;
      for (int t0 = w * 2 * kChunkVecs * Vec<BF16>::N; t0 < end; t0 += 32 * kBatch) {
        float x[kBatch];
        bool any = false;
#pragma unroll
        for (int i = 0; i < kBatch; ++i) {
          const int tok = t0 + i * 32 + lane;
          x[i] = tok < end ? element<BF16>(row, tok) : -INFINITY;
          any = any || x[i] >= thr;
        }
        if (!__any_sync(kFull, any)) continue;
#pragma unroll
        for (int i = 0; i < kBatch; ++i) {
          const unsigned long long key = x[i] >= thr ? make_key(x[i], (uint32_t)(t0 + i * 32 + lane)) : 0ull;
          const bool in = key != 0ull && (have < K || key > ws->pool[K - 1]);
          const unsigned mask = __ballot_sync(kFull, in);
          if (mask) {
            __syncwarp();
            if (in) ws->pool[have + __popc(mask & ((1u << lane) - 1u))] = key;
            __syncwarp();
            have = rank_pool(ws->pool, have + __popc(mask), K);
            if (have == K) thr = just_above(key_value(ws->pool[K - 1]));   // later tokens of the K-th value lose the tie
          }
        }
      }
    }
  }
  if (lane == 0)
    for (int r = have; r < K; ++r) ws->pool[r] = 0ull;
  __syncwarp();
  return have;
}

// The elements at or above the floor, out of the listed cells, as keys in the pool.  Returns how many there are, or -1 if
// something overflowed.
template <bool BF16>
__device__ __forceinline__ int gather_keys(PairShared *ws, const char *row, const RowShape<BF16> &rs, int V, float floor, int n_list) {
  constexpr int EPV = Vec<BF16>::N;
  constexpr int kBatch = 4;                         // 16-byte loads of a lane in flight: 16 cells
  const int lane = threadIdx.x & 31;
  const unsigned lt_mask = (1u << lane) - 1u;
  int n_vec = 0;                                    // vectors with such an element
  for (int i0 = 0; i0 < n_list * 8; i0 += 32 * kBatch) {
    uint4 q[kBatch];
    int v[kBatch];
#pragma unroll
    for (int u = 0; u < kBatch; ++u) {
      const int i = i0 + u * 32 + lane, cell = i < n_list * 8 ? ws->list[i >> 3] : -1;
      v[u] = cell < 0 ? rs.vpr : cell_vector(cell >> 5, cell & 31, i & 7);
    }
    load_vectors<BF16, kBatch>(q, row, v, rs, V);
#pragma unroll
    for (int u = 0; u < kBatch; ++u) {
      const bool hit = v[u] < rs.vpr && Vec<BF16>::vmax(q[u]) >= floor;
      const unsigned hm = __ballot_sync(kFull, hit);
      const int pos = n_vec + __popc(hm & lt_mask);
      if (hit && pos < kListCap) { ws->vecs[pos] = v[u]; ws->data[pos] = q[u]; }
      n_vec += __popc(hm);
    }
  }
  if (n_vec > kListCap) return -1;
  __syncwarp();
  int n = 0;
#pragma unroll 4
  for (int i0 = 0; i0 < n_vec * EPV; i0 += 32) {
    const int i = i0 + lane;
    float x = -INFINITY;
    int tok = V;
    if (i < n_vec * EPV) {
      tok = ws->vecs[i / EPV] * EPV + i % EPV;
      if (BF16) x = __uint_as_float((uint32_t)reinterpret_cast<const unsigned short *>(ws->data)[i] << 16);
      else x = reinterpret_cast<const float *>(ws->data)[i];
    }
    const bool hit = x >= floor && tok < V;
    const unsigned hm = __ballot_sync(kFull, hit);
    const int pos = n + __popc(hm & lt_mask);
    if (hit && pos < kPoolCap) ws->pool[pos] = make_key(x, (uint32_t)tok);
    n += __popc(hm);
  }
  __syncwarp();
  return n <= kPoolCap ? n : -1;
}

// A row is completed, all its partial results being in place, in two independent halves, by the two warps of a pair.  Each
// is a chain of dependent steps, so loads are issued in batches, as early as their addresses are known.

// The K largest.
template <bool BF16, bool NEAR>
__device__ __forceinline__ void complete_keys(const PassParams &p, PairShared *ws, const uint32_t *row_cells, int a, int b, int j) {
  constexpr int kBatch = 32;                        // words of its column that a lane holds at a time: 64 chunks
  const RowShape<BF16> rs(p.V);
  const int lane = threadIdx.x & 31, K = p.K;
  const char *row = row_pointer(p, b, j, BF16 ? 2 : 4);
  const uint32_t *cells = (NEAR ? row_cells : p.cells + (size_t)a * rs.words * 32) + lane;
  uint32_t v[kBatch], cm2 = kLowestBf16x2;
#pragma unroll
  for (int i = 0; i < kBatch; ++i) v[i] = i < rs.words ? cells[i * 32] : kLowestBf16x2;
#pragma unroll
  for (int i = 0; i < kBatch; ++i) cm2 = max_bf16x2(cm2, v[i]);
  for (int c0 = kBatch; c0 < rs.words; c0 += kBatch) {
#pragma unroll
    for (int i = 0; i < kBatch; ++i) v[i] = c0 + i < rs.words ? cells[(c0 + i) * 32] : kLowestBf16x2;
#pragma unroll
    for (int i = 0; i < kBatch; ++i) cm2 = max_bf16x2(cm2, v[i]);
  }
  // 32 columns, or for a large K 64 half columns, and their places under (maximum desc, index asc): at least K elements
  // reach the K-th largest column maximum (if that many columns have data)
  const float lo = __uint_as_float(cm2 << 16), hi = __uint_as_float(cm2 & 0xFFFF0000u);
  float floor;
  if (K <= 16) {
    const float cm = fmaxf(lo, hi);
    ws->colmax[lane] = cm;
    __syncwarp();
    int place = 0;
#pragma unroll
    for (int i = 0; i < 32; i += 4) {
      const float4 o = *reinterpret_cast<const float4 *>(&ws->colmax[i]);
      place += o.x > cm || (o.x == cm && i < lane);
      place += o.y > cm || (o.y == cm && i + 1 < lane);
      place += o.z > cm || (o.z == cm && i + 2 < lane);
      place += o.w > cm || (o.w == cm && i + 3 < lane);
    }
    floor = __shfl_sync(kFull, cm, __ffs(__ballot_sync(kFull, place == K - 1)) - 1);
  } else {
    ws->colmax[lane] = lo;
    ws->colmax[32 + lane] = hi;
    __syncwarp();
    int p0 = 0, p1 = 0;
#pragma unroll 8
    for (int i = 0; i < 64; ++i) {
      const float o = ws->colmax[i];
      p0 += o > lo || (o == lo && i < lane);
      p1 += o > hi || (o == hi && i < 32 + lane);
    }
    const unsigned b0 = __ballot_sync(kFull, p0 == K - 1), b1 = __ballot_sync(kFull, p1 == K - 1);
    floor = b0 ? __shfl_sync(kFull, lo, __ffs(b0) - 1) : __shfl_sync(kFull, hi, __ffs(b1) - 1);
  }
  const uint32_t fb = __float_as_uint(floor), floor2 = fb | (fb >> 16);

  // ---- the cells that reach it
  int n_list = 0;
  for (int c0 = 0; c0 < rs.words && n_list <= kListCap; c0 += kBatch) {
    if (rs.words > kBatch) {
#pragma unroll
      for (int i = 0; i < kBatch; ++i) v[i] = c0 + i < rs.words ? cells[(c0 + i) * 32] : kLowestBf16x2;
    }
    unsigned long long mask = 0ull;                 // 16 words: bits of their first cells, then of their second ones; twice
#pragma unroll
    for (int h = 0; h < kBatch / 16; ++h) {
      uint32_t m = 0u;
#pragma unroll
      for (int i = 0; i < 16; ++i) {
        uint32_t ge;
        asm("set.ge.u32.bf16x2 %0, %1, %2;" : "=r"(ge) : "r"(v[h * 16 + i]), "r"(floor2));
        m |= (ge & 0x00010001u) << i;
      }
      mask |= (unsigned long long)m << (32 * h);
    }
    const int mine = __popcll(mask);
    int upto = mine;                                // places in lane order
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int v = __shfl_up_sync(kFull, upto, o);
      if (lane >= o) upto += v;
    }
    int pos = n_list + upto - mine;
    n_list += __shfl_sync(kFull, upto, 31);
    while (mask) {
      const int bit = __ffsll((long long)mask) - 1, chunk = 2 * (c0 + ((bit & 32) >> 1) + (bit & 15)) + ((bit >> 4) & 1);
      if (pos < kListCap) ws->list[pos] = chunk < rs.nc ? chunk * 32 + lane : -1;
      ++pos;
      mask &= mask - 1ull;
    }
  }
  __syncwarp();
  const int n_keys = n_list <= kListCap ? gather_keys<BF16>(ws, row, rs, p.V, floor, n_list) : -1;
  const int n_valid = n_keys >= 0 ? rank_pool(ws->pool, n_keys, K) : select_in_order<BF16, NEAR>(p, ws, row, row_cells, a, floor);
  const size_t slot = (size_t)b * p.rows_per_seq_max + j;
  for (int i = lane; i < K; i += 32) p.row_keys[slot * K + i] = ws->pool[i];
  if (lane == 0) {
    p.rows[slot].top = ws->pool[0];
    p.rows[slot].n_valid = n_valid;
  }
  __syncwarp();
}

// The maximum and the merged sums.
template <bool BF16, bool TOPM>
__device__ __forceinline__ void complete_sums(const PassParams &p, const CtaRange<TOPM> &cr, int a, int b, int j) {
  constexpr int kBatch = 2;                         // chunks of a lane at a time: 64 of the row
  const RowShape<BF16> rs(p.V);
  const int lane = threadIdx.x & 31, first = a * rs.nc;
  const char *row = row_pointer(p, b, j, BF16 ? 2 : 4);
  float4 rest[kBatch], held[kBatch];
  // ---- the row maximum and where it is
  float m = kLowestF32;
  int at = 0, tl = 0, tc = 0;                        // the record, its lane and chunk
  for (int c0 = 0; c0 < rs.nc; c0 += 32 * kBatch) {
#pragma unroll
    for (int i = 0; i < kBatch; ++i) {
      const int ch = c0 + i * 32 + lane;
      rest[i] = make_float4(0.f, 0.f, kNoOffset, kLowestF32);
      held[i] = make_float4(0.f, 0.f, 0.f, 0.f);
      if (ch < rs.nc && cr.ends_record(first + ch, a)) {
        const SumRecord *r = p.sums + first + ch;
        rest[i] = r->rest;
        held[i] = r->held;
      }
    }
#pragma unroll
    for (int i = 0; i < kBatch; ++i)
      if (rest[i].w > m) { m = rest[i].w; at = c0 + i * 32 + lane; tl = __float_as_int(held[i].z); tc = __float_as_int(held[i].w); }
  }
  const uint32_t ord = f32_orderable(__float_as_uint(m)), top = __reduce_max_sync(kFull, ord);
  const int owner = __ffs(__ballot_sync(kFull, ord == top)) - 1;
  const float Mf = __shfl_sync(kFull, m, owner);
  const int trec = __shfl_sync(kFull, at, owner), tlane = __shfl_sync(kFull, tl, owner), tch = __shfl_sync(kFull, tc, owner);

  // ---- that lane's vectors of the chunk summed again without the maximum (and without its equals, which are counted)
  const float cM = offset_of(Mf);                                    // the reference of the merge
  float s_own, u_own;
  int equals = 0;
  {
    uint4 q[1];
    const int vec[1] = {lane < kChunkVecs / 32 ? cell_vector(tch, tlane, lane) : rs.vpr};
    load_vectors<BF16, 1>(q, row, vec, rs, p.V);
    float x[Vec<BF16>::N];
    Vec<BF16>::unpack(q[0], x);
    Acc acc;
    acc.clear();
#pragma unroll
    for (int e = 0; e < Vec<BF16>::N; ++e)
      if (x[e] == Mf && lane < kChunkVecs / 32) { x[e] = kLowestF32; ++equals; }
#pragma unroll
    for (int e = 0; e < Vec<BF16>::N; e += 2) acc_pair(acc, (e >> 1) & 1, x[e], x[e + 1], pack2(kLog2e, kLog2e), pack2(cM, cM));
    acc.totals(s_own, u_own);
  }
  // ---- merge: all records brought to the reference of the maximum
  double S = (double)s_own, U = (double)u_own;
  for (int c0 = 0; c0 < rs.nc; c0 += 32 * kBatch) {
#pragma unroll
    for (int i = 0; i < kBatch; ++i) {
      const int ch = c0 + i * 32 + lane;
      const bool have = ch < rs.nc && cr.ends_record(first + ch, a);
      if (rs.nc > 32 * kBatch && have) {
        const SumRecord *r = p.sums + first + ch;
        rest[i] = r->rest;
        held[i] = r->held;
      }
      if (have) {
        const double s = (double)rest[i].x + (ch == trec ? 0.0 : (double)held[i].x);
        const double u = (double)rest[i].y + (ch == trec ? 0.0 : (double)held[i].y);
        const float d = fmaxf(cM - rest[i].z, -2000.f);               // (never positive)
        const double f = pow2_f64(d);
        S += f * s;
        U += f * (u + (double)d * s);
      }
    }
  }
  S = warp_sum(S);
  U = warp_sum(U);
  equals = __reduce_add_sync(kFull, equals);
  if (lane == 0) write_sums(p.rows + (size_t)b * p.rows_per_seq_max + j, Mf, cM, S, U, equals);
  __syncwarp();
}

// What becomes of a row once a CTA has done its part of it, or given up waiting for that part.
enum RowState { kRowWaits, kRowComplete, kRowBroken };

// The CTA's part of a row shared with others: is it the last?  (By one lane; the others' records are visible to it afterwards.)
// A part that was given up is counted too, so that the count comes back to zero and the row is known to be broken.
constexpr unsigned kBrokenPart = 1u << 23;           // above any row's chunks; the parts of a row are at most a grid's 256 CTAs
__device__ __forceinline__ RowState count_shared(const PassParams &p, int a, int chunks, int nc, bool ok) {
  __threadfence();                                   // the CTA's records, before its count
  const unsigned part = (unsigned)chunks + (ok ? 0u : kBrokenPart);
  const unsigned total = atomicAdd(reinterpret_cast<unsigned *>(&p.row_done[a]), part) + part;
  if ((total & (kBrokenPart - 1u)) != (unsigned)nc) return kRowWaits;
  p.row_done[a] = 0;                                 // for the next launch
  __threadfence();                                   // the other CTAs' records, after their counts
  return total == (unsigned)nc ? kRowComplete : kRowBroken;
}

// ---------------------------------------------------------------- truncated entropy (Eq. 3): setting candidates aside

// Where a warp puts the vectors whose largest element reaches its segment's floor (ballot-ranked places in stream
// order, so the result does not depend on timing).
struct TopmState {
  uint4 *region;              // the warp's part of the pool
  int cap, n, first;          // its size in vectors; vectors set aside by the warp so far (may pass cap: then nothing more is stored); n when the segment began
  float floor;
  unsigned long long keep;    // L2 policy of the stores: the vectors are read back right after the pass, the rows never again
};

__device__ __forceinline__ void store_keep_in_l2(uint4 *dst, const uint4 &q, unsigned long long policy) {
  asm volatile("st.global.L2::cache_hint.v4.u32 [%0], {%1, %2, %3, %4}, %5;"
               ::"l"(dst), "r"(q.x), "r"(q.y), "r"(q.z), "r"(q.w), "l"(policy) : "memory");
}

// the collection floor of a segment from the lane maxima over its first two groups
__device__ __forceinline__ float collection_floor(float lmax, int place) {
  const int lane = threadIdx.x & 31;
  uint32_t live = f32_orderable(__float_as_uint(lmax)), low = 0;
  for (int r = 0; r < place; ++r) {
    low = __reduce_max_sync(kFull, live);
    if (lane == __ffs(__ballot_sync(kFull, live == low)) - 1) live = 0;
  }
  return fmaxf(__uint_as_float(f32_from_orderable(low)), kTopmLowestFloor);
}

// ---------------------------------------------------------------- the kernel

// Sums and maximum of the chunk in q, each group of which is requested for the next chunk as soon as it is consumed.
template <bool BF16, bool TOPM>
__device__ __forceinline__ float stream_chunk(uint4 (&q)[kGroups][4], const uint4 *src, int nnv, LaneSums &ls, f32x2 scale, TopmState &ts,
                                              int lane) {
  RunMax<BF16> m;
  m.clear();
#pragma unroll
  for (int g = 0; g < kGroups; ++g) {
    RunMax<BF16> head;
    head.clear();
#pragma unroll
    for (int k = 0; k < 4; ++k) head.take(q[g][k]);
    m.take(head);
    ls.begin_group(head.value(), g == 0);
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      if (TOPM) {
        RunMax<BF16> one;
        one.clear();
        one.take(q[g][k]);
        const bool hit = one.value() >= ts.floor;              // (false for a vector of NaNs; such a row is reported anyway)
        const unsigned hm = __ballot_sync(kFull, hit);
        const int pos = ts.n + __popc(hm & ((1u << lane) - 1u));
        if (hit && pos < ts.cap) store_keep_in_l2(ts.region + pos, q[g][k], ts.keep);
        ts.n += __popc(hm);
      }
      Vec<BF16>::clamp(q[g][k]);
    }
#pragma unroll
    for (int k = 0; k < 4; ++k) acc_vector<BF16>(ls.acc, q[g][k], scale, ls.c2);
    load_group<BF16>(q[g], src, g, nnv, lane);
  }
  return m.value();
}

// One warp's stream: every kStreamWarps-th chunk of the CTA's work order (TOPM: a contiguous part of it).
template <bool BF16, bool TOPM, bool NEAR>
__device__ __forceinline__ void stream(const PassParams &p, CtaShared *cs, const int *s_off, uint32_t *near, const RowShape<BF16> &rs, const CtaRange<TOPM> &cr) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int n = cr.u1 - cr.u0, step = TOPM ? 1 : kStreamWarps;
  int i = TOPM ? warp * cr.part : warp;
  const int end = TOPM ? (i + cr.part < n ? i + cr.part : n) : n;
  if (i >= end) {
    __syncthreads();
    return;
  }
  const size_t esz = BF16 ? 2 : 4;
  const f32x2 scale = pack2(kLog2e, kLog2e);
  const int u_first = cr.chunk_at(i);
  int a = u_first / rs.nc, ch = u_first - a * rs.nc, b = find_sequence(s_off, p.B, a);
  const char *row = row_pointer(p, b, a - s_off[b], esz);
  uint4 q[kGroups][4];
  {
    const uint4 *src = reinterpret_cast<const uint4 *>(row) + ch * kChunkVecs + lane;
#pragma unroll
    for (int g = 0; g < kGroups; ++g) load_group<BF16>(q[g], src, g, rs.v_full - ch * kChunkVecs, lane);
  }
  __syncthreads();                                   // the tasks' barriers are set up
  TopmState ts;
  ts.region = nullptr; ts.cap = 0; ts.n = 0; ts.first = 0; ts.floor = INFINITY; ts.keep = 0ull;
  int region = 0;
  if (TOPM) {
    asm("createpolicy.fractional.L2::evict_last.b64 %0, 1.0;" : "=l"(ts.keep));
    const long long cap = p.topm_pool_vecs / cr.busy;          // an equal part of the pool for every warp with chunks
    ts.cap = (int)(cap < 0x3FFFFFFF ? cap : 0x3FFFFFFF);
    region = (int)((long long)((int)blockIdx.x * ((cr.per_cta + cr.part - 1) / cr.part) + warp) * ts.cap);
    ts.region = p.topm_pool + region;
  }
  LaneSums ls;
  bool fresh = true;                                 // the chunk is the warp's first of its row
  for (;;) {
    // ---- the warp's next chunk
    const bool more = i + step < end;
    int na = a, nch = 0, nb = b;
    const char *nrow = row;
    if (more) {
      const int nu = cr.chunk_at(i + step);
      na = nu / rs.nc;
      nch = nu - na * rs.nc;
      if (na != a) {
        if (na < a) nb = find_sequence(s_off, p.B, na);
        else while (s_off[nb + 1] <= na) ++nb;
        nrow = row_pointer(p, nb, na - s_off[nb], esz);
      }
    }
    const uint4 *src = reinterpret_cast<const uint4 *>(nrow) + nch * kChunkVecs + lane;
    const int nnv = more ? rs.v_full - nch * kChunkVecs : 0;
    const int nvec = rs.vpr - ch * kChunkVecs;       // vectors from the chunk's start to the row's end
    if (nvec <= kChunkVecs && rs.vpr != rs.v_full) { // the row's ragged last vector is in this chunk
      const uint4 t = load_ragged<BF16>(row, rs.v_full, rs.v_full, p.V);
#pragma unroll
      for (int g = 0; g < kGroups; ++g)
#pragma unroll
        for (int k = 0; k < 4; ++k)
          if (g * 128 + k * 32 + lane == nvec - 1) q[g][k] = t;
    }
    if (fresh) {
      ls.start();
      if (TOPM) {
        RunMax<BF16> head;
        head.clear();
#pragma unroll
        for (int g = 0; g < 2; ++g)
#pragma unroll
          for (int k = 0; k < 4; ++k) head.take(q[g][k]);
        ts.floor = collection_floor(head.value(), p.topm_place);
        ts.first = ts.n;
      }
    }
    const float before = ls.ref;
    const float cv = stream_chunk<BF16, TOPM>(q, src, nnv, ls, scale, ts, lane);
    // ---- the chunk's cells; at the end of the warp's part of the row the record
    ls.end_chunk(ls.ref > before, ch);
    const int u = a * rs.nc + ch;
    fresh = !more || na != a;
    if (C2T_IN_BOUNDS(u, p.n_chunks, p.status)) {
      uint32_t *word = p.cells + ((size_t)a * rs.words + (ch >> 1)) * 32 + lane;
      uint32_t *low = BF16 ? nullptr : p.cell_low + (word - p.cells);
      if (NEAR) word = cells_of_row(p, near, cr, rs, a) + (ch >> 1) * 32 + lane;
      if (ch + 1 == rs.nc && !(ch & 1)) {            // (no second cell)
        *word = cell_bits(cv, BF16) | (kLowestBf16x2 & 0xFFFF0000u);
        if (!BF16) *low = __float_as_uint(cv) & 0xFFFFu;
      } else {
        reinterpret_cast<unsigned short *>(word)[ch & 1] = (unsigned short)cell_bits(cv, BF16);
        if (!BF16) reinterpret_cast<unsigned short *>(low)[ch & 1] = (unsigned short)__float_as_uint(cv);
      }
      if (fresh) write_record(p.sums + u, ls);
    }
    if (fresh) {
      if (TOPM) {
        const int seg = (int)blockIdx.x * kStreamWarps + warp + a;    // (both only grow along the parts: unique)
        if (lane == 0 && C2T_IN_BOUNDS(seg, p.n_segs, p.status)) {
          TopmSegment set;
          set.first = region + ts.first;
          set.n = ts.n > ts.cap ? -1 : ts.n - ts.first;
          set.floor = ts.floor;
          set.pad = 0;
          p.topm_seg[seg] = set;
        }
      }
      __syncwarp();
      if (lane == 0) {
        const uint32_t bar = (uint32_t)__cvta_generic_to_shared(cs->bars() + cr.row_task(a));
        asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
      }
    }
    if (!more) break;
    i += step; a = na; ch = nch; b = nb; row = nrow;
  }
}

// the two warps of a pair wait for each other
__device__ __forceinline__ void pair_barrier(int pair) { asm volatile("bar.sync %0, 64;" ::"r"(1 + pair) : "memory"); }

// Until all records of a task are written; false if the wait ran out.
__device__ __forceinline__ bool wait_task(unsigned long long *bar_ptr, int limit) {
  const uint32_t bar = (uint32_t)__cvta_generic_to_shared(bar_ptr);
  uint32_t done = 0u;
  for (int i = 0; i < limit && !done; ++i)
    asm volatile("{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], 0;\n\tselp.u32 %0, 1, 0, p;\n\t}"
                 : "=r"(done) : "r"(bar) : "memory");
  return done != 0u;
}

// A pair's work: the CTA's tasks, one after the other.  A row inside the range is complete when its records are; a
// shared one if this CTA's part of it was the last.  A row whose records do not come in time is given up: it gets a result
// that faults its sequence, and nothing of it stays behind for later rows or launches.
template <bool BF16, bool TOPM, bool NEAR>
__device__ __forceinline__ void complete(const PassParams &p, CtaShared *cs, const int *s_off, uint32_t *near, const RowShape<BF16> &rs, const CtaRange<TOPM> &cr) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, pair = warp >> 1, role = warp & 1;
  const int n_tasks = cr.n_tasks();
  pair_barrier(pair);                                // (both have done with streaming)
  for (;;) {
    if (role == 0 && lane == 0) {
      const int k = atomicAdd(&cs->task, 1);
      RowState go = kRowWaits;
      if (k < n_tasks) {
        const int a = cr.task_row(k);
        const bool ok = wait_task(cs->bars() + k, p.wait_limit);
        if (a >= cr.in0 && a < cr.in1) go = ok ? kRowComplete : kRowBroken;
        else go = count_shared(p, a, cr.task_chunks(a), rs.nc, ok);
      }
      cs->task_of[pair] = k;
      cs->flag[pair] = go;
    }
    pair_barrier(pair);
    const int k = cs->task_of[pair], go = cs->flag[pair];
    pair_barrier(pair);
    if (k >= n_tasks) break;
    if (go == kRowWaits) continue;
    const int a = cr.task_row(k), b = find_sequence(s_off, p.B, a);
    if (go == kRowBroken) {
      if (role == 0) give_up_row(p, b, a - s_off[b]);
    } else if (role == 0) complete_keys<BF16, NEAR>(p, &cs->scratch[pair], NEAR ? cells_of_row(p, near, cr, rs, a) : nullptr, a, b, a - s_off[b]);
    else complete_sums<BF16, TOPM>(p, cr, a, b, a - s_off[b]);
  }
}

// The pass itself: what every warp of the grid does.
template <bool BF16, bool TOPM, bool NEAR>
__device__ __forceinline__ void expand_pass_body(const PassParams &p, unsigned char *s_dyn) {
  CtaShared *cs = reinterpret_cast<CtaShared *>(s_dyn);
  int *s_off = reinterpret_cast<int *>(cs->bars() + p.cta_tasks);
  uint32_t *near = NEAR ? reinterpret_cast<uint32_t *>(s_dyn + p.near_cells) : nullptr;
  const int n_rows = build_row_offsets(p.counts, p.B, p.rows_per_seq_max, s_off);
  const RowShape<BF16> rs(p.V);
  const CtaRange<TOPM> cr(rs.nc, n_rows * rs.nc);
  if (TOPM) {                                        // the selection kernels find a row's segments with these
    if (blockIdx.x == 0)
      for (int i = threadIdx.x; i <= p.B; i += kExpandThreads) p.row_off[i] = s_off[i];
    if (blockIdx.x == 0 && threadIdx.x == 0) {
      p.info->n_rows = n_rows;
      p.info->row_chunks = rs.nc;
      p.info->cta_chunks = cr.per_cta;
    }
  }
  if (cr.u0 >= cr.u1) return;
  for (int k = kExpandThreads - 1 - (int)threadIdx.x; k < cr.n_tasks(); k += kExpandThreads) {   // (the last warps first: they do not stream)
    const uint32_t bar = (uint32_t)__cvta_generic_to_shared(cs->bars() + k);
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(cr.task_records(cr.task_row(k))) : "memory");
  }
  if (threadIdx.x == kExpandThreads - 1) cs->task = 0;
  if (threadIdx.x < kStreamWarps * 32) stream<BF16, TOPM, NEAR>(p, cs, s_off, near, rs, cr);
  else __syncthreads();
  complete<BF16, TOPM, NEAR>(p, cs, s_off, near, rs, cr);
}

template <bool BF16, bool TOPM, bool NEAR>
__global__ void __launch_bounds__(kExpandThreads, 1) expand_pass_kernel(const __grid_constant__ PassParams p) {
  extern __shared__ __align__(16) unsigned char s_dyn[];
  chain_enter();
  expand_pass_body<BF16, TOPM, NEAR>(p, s_dyn);
}

// Expand and prune of a level in one launch, for small batches: the CTA that finishes last (an atomic ticket, nobody
// waits) has every row's result in front of it and does the per-sequence work of c2t_prune for all sequences, one
// after the other.
template <bool BF16>
__global__ void __launch_bounds__(kExpandThreads, 1) expand_prune_kernel(const __grid_constant__ PassParams p,
                                                                         const __grid_constant__ TreeState t, int level,
                                                                         c2t_frontier out) {
  extern __shared__ __align__(16) unsigned char s_dyn[];
  __shared__ unsigned s_ticket;
  __shared__ __align__(16) double s_w[kWCount];
  if (threadIdx.x >= kStreamWarps * 32) stage_classifier(t, s_w, threadIdx.x - kStreamWarps * 32, kExpandThreads - kStreamWarps * 32);   // (written at init)
  chain_enter();
  expand_pass_body<BF16, false, false>(p, s_dyn);
  __syncthreads();
  if (threadIdx.x == 0) {
    __threadfence();                                 // this CTA's row results (seen at the barrier), before its ticket
    s_ticket = atomicAdd(t.ticket, 1u);
    __threadfence();                                 // the other CTAs' results, after their tickets
  }
  __syncthreads();
  if (s_ticket != gridDim.x - 1) return;
  if (threadIdx.x == 0) *t.ticket = 0u;              // for the next launch
  // the pass's shared memory is free now
  PruneShared &sh = *reinterpret_cast<PruneShared *>(s_dyn);
#pragma unroll 1
  for (int b = 0; b < t.B; ++b) prune_level_body<kExpandThreads, kMaxCand / kExpandThreads, false>(t, level, out, nullptr, 0, b, sh, s_w, nullptr);
}

}  // namespace

size_t topm_pool_vectors(size_t batch, size_t rows_per_seq, int vocab, int elem_bytes) {
  const size_t vec = 16 / elem_bytes;
  const size_t n = batch * rows_per_seq * ((vocab + vec - 1) / vec) / kTopmPoolDivisor + 4096;
  return n < 0x7FFFFFFFu ? n : 0x7FFFFFFFu;          // records hold 32-bit positions
}

// A row's floor is the highest of its segments' (up to some forty), and a low place among 32 lane maxima scatters widely: with
// M = 500 of 128256 the place for 3 M elements is the 11th and most rows were read again (1320 us per eight levels of 40 rows
// of fp32; at the 24th or beyond 369).
constexpr int kTopmLeastPlace = 24;
int topm_floor_place(int vocab, int elem_bytes, int M) {
  const int vec = 16 / elem_bytes;
  const int vec_per_row = (vocab + vec - 1) / vec, head = vec_per_row < 256 ? vec_per_row : 256;
  const double per_lane = (double)head * vec / 32.0, share = 3.0 * M / vocab;
  // The lowest place reaches a share 1 - (1 / 32)^(1 / per_lane) of the row (5 % for bf16, 10 % for fp32).  Where that is hardly M
  // elements nothing is set aside, and the rows are read again at once: 8192 bf16 tokens with M = 1000, say.
  if ((1.0 - pow(1.0 / 32.0, 1.0 / per_lane)) * vocab < 1.5 * M) return 0;
  const int place = share >= 1.0 ? 31 : (int)ceil(32.0 * (1.0 - pow(1.0 - share, per_lane)));
  return place < kTopmLeastPlace ? kTopmLeastPlace : (place > 31 ? 31 : place);
}

int row_chunks(int vocab, int elem_bytes) {
  const int vec = 16 / elem_bytes;
  return ((vocab + vec - 1) / vec + kChunkVecs - 1) / kChunkVecs;
}

#ifdef C2T_DEBUG_BOUNDS
extern "C" {
int c2t_debug_task_wait_limit = kTaskWaitLimit;
// blocks of a row in registers, 0 where the level is streamed: for tests that are about one of the two
int c2t_debug_row_cluster(int vocab, int elem_bytes, long long rows, int K, int sms) {
  return c2t::row_pass_plan(vocab, elem_bytes, rows, K, sms).cluster;
}
}
#endif

// the launch's shared memory and limits
constexpr size_t kPassSharedBytes = 100 * 1024;        // more than plan_shared's fixed part at the limits of a configuration
static size_t plan_shared(PassParams &p, int elem_bytes, int grid, bool near) {
  p.wait_limit = C2T_TASK_WAIT_LIMIT;
  p.cta_tasks = (int)((long long)p.B * p.rows_per_seq_max / grid) + 4;       // rows inside a CTA's range, and the two it shares
  const size_t fixed = sizeof(CtaShared) + (size_t)p.cta_tasks * sizeof(unsigned long long) + ((size_t)p.B + 1) * sizeof(int);
  const long long nc = row_chunks(p.V, elem_bytes), per_cta = ((long long)p.B * p.rows_per_seq_max * nc + grid - 1) / grid;
  const size_t at = (fixed + 127) & ~(size_t)127, cells = (size_t)(per_cta / nc + 1) * ((nc + 1) / 2) * 128;
  p.near_cells = near && elem_bytes == 4 && nc >= kNearChunks && per_cta >= 2 * nc && at + cells <= kPassSharedBytes ? (int)at : 0;
  return p.near_cells ? at + cells : fixed;
}

cudaError_t prepare_expand_pass() {
  const int bytes = (int)kPassSharedBytes;
  cudaError_t e = cudaFuncSetAttribute(expand_pass_kernel<true, false, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
  if (e == cudaSuccess) e = cudaFuncSetAttribute(expand_pass_kernel<false, false, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
  if (e == cudaSuccess) e = cudaFuncSetAttribute(expand_pass_kernel<true, true, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
  if (e == cudaSuccess) e = cudaFuncSetAttribute(expand_pass_kernel<false, true, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
  if (e == cudaSuccess) e = cudaFuncSetAttribute(expand_pass_kernel<false, false, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
  if (e == cudaSuccess) e = cudaFuncSetAttribute(expand_prune_kernel<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
  if (e == cudaSuccess) e = cudaFuncSetAttribute(expand_prune_kernel<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
  return e;
}

// How the pass in registers (row_pass.cu) takes the level, if it does.
static RowPlan rows_in_registers(const PassParams &p, int dtype, int sms) {
  if (p.topm_pool) return RowPlan{0, 0};
  return row_pass_plan(p.V, dtype == C2T_BF16 ? 2 : 4, (long long)p.B * p.rows_bound, p.K, sms);
}

cudaError_t launch_expand_prune(PassParams p, const TreeState &t, int level, const c2t_frontier *out, int dtype, int grid, cudaStream_t s) {
  c2t_frontier o = {nullptr, nullptr, nullptr, nullptr};
  if (out) o = *out;
  const RowPlan plan = rows_in_registers(p, dtype, grid);
  if (plan.cluster) return launch_expand_rows_prune(p, t, level, o, dtype, plan, s);
  size_t smem = plan_shared(p, dtype == C2T_BF16 ? 2 : 4, grid, false);
  if (smem < sizeof(PruneShared)) smem = sizeof(PruneShared);
  if (dtype == C2T_BF16)
    return launch_chained(expand_prune_kernel<true>, dim3(grid), dim3(kExpandThreads), smem, s, p, t, level, o);
  return launch_chained(expand_prune_kernel<false>, dim3(grid), dim3(kExpandThreads), smem, s, p, t, level, o);
}

cudaError_t launch_expand_pass(PassParams p, int dtype, int grid, cudaStream_t s) {
  const RowPlan plan = rows_in_registers(p, dtype, grid);
  if (plan.cluster) return launch_expand_rows(p, dtype, plan, s);
  const size_t smem = plan_shared(p, dtype == C2T_BF16 ? 2 : 4, grid, !p.topm_pool);
  const bool bf16 = dtype == C2T_BF16;
  if (p.topm_pool) {                                 // also sets the candidates of Eq. 3 aside
    if (bf16) return launch_chained(expand_pass_kernel<true, true, false>, dim3(grid), dim3(kExpandThreads), smem, s, p);
    return launch_chained(expand_pass_kernel<false, true, false>, dim3(grid), dim3(kExpandThreads), smem, s, p);
  }
  if (p.near_cells) return launch_chained(expand_pass_kernel<false, false, true>, dim3(grid), dim3(kExpandThreads), smem, s, p);
  if (bf16) return launch_chained(expand_pass_kernel<true, false, false>, dim3(grid), dim3(kExpandThreads), smem, s, p);
  return launch_chained(expand_pass_kernel<false, false, false>, dim3(grid), dim3(kExpandThreads), smem, s, p);
}

}  // namespace c2t

// Arg-max over rows of logits, per row the largest logit, ties to the lower token id.
//   argmax_pass_kernel: the rows of all final nodes, for the greedy acceptance walk (Sec. 5 Metrics).
//   row_argmax_kernel: the rows of a matrix, from the logits to the token ids in one launch.
//   accept_lazy_kernel: the acceptance walk that reads only the rows it visits, in one launch.
// argmax_pass_kernel lays the rows end to end and cuts them into equal spans, one per CTA.  The warps of a CTA take groups of
// 128 or 256 vectors (four or eight 16-byte loads per lane, all in flight) in turn, through rows and across them, and a warp brings its
// best key of a row to the row's place by an atomic maximum: nothing waits at a row's end.  (With one key per CTA and row, two
// barriers at every row's end cost more than a short row's loads: 3840 rows of 16032 bf16 values took 54.8 us.  With
// a span per warp a CTA reads 16 places at once: 1 % slower on long rows.)
#include "vocab_common.cuh"

namespace c2t {
namespace {

// A thread's largest vector so far: its maximum (NaN ignored), place and contents.
template <bool BF16>
struct BestVector {
  float m;
  int v;
  uint4 q;
  __device__ __forceinline__ void clear() { m = -INFINITY; v = -1; q = make_uint4(0u, 0u, 0u, 0u); }   // (clamped values are finite)
  // (-inf counts as -2^127 here as everywhere: applied to the maximum, it costs one select per vector)
  __device__ __forceinline__ void take(const uint4 &x, int at) {
    float vm = Vec<BF16>::vmax(x);
    vm = vm < kLowestF32 ? kLowestF32 : vm;
    if (vm > m) { m = vm; v = at; q = x; }
  }
  // the key of its largest element, the lowest token among equals (0: only NaN so far); V: length of the row
  __device__ __forceinline__ unsigned long long key(int V) const {
    unsigned long long best = 0ull;
    if (v >= 0) {
      float x[Vec<BF16>::N];
      Vec<BF16>::unpack(q, x);
#pragma unroll
      for (int i = Vec<BF16>::N - 1; i >= 0; --i)
        if ((x[i] < kLowestF32 ? kLowestF32 : x[i]) == m && v * Vec<BF16>::N + i < V) best = make_key(m, (uint32_t)(v * Vec<BF16>::N + i));
    }
    return best;
  }
};

__device__ __forceinline__ unsigned long long warp_best(unsigned long long best) {      // in lane 0
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const unsigned long long other = __shfl_down_sync(kFull, best, o);
    best = other > best ? other : best;
  }
  return best;
}

constexpr int kMinPassSpan = 1024;     // a CTA of the pass never gets fewer vectors than this
// Loads of a lane per group.  Small groups keep a CTA's reads closer together (rows of 16032 vectors: 156.7 -> 145.7 us for
// 985 MB of bf16; 32064: 105.6 -> 98.5 us for 657 MB of fp32), large ones leave fewer row ends to a warp (rows of 2004 vectors:
// 33.8 -> 27.1 us for 123 MB; 835 vectors: 13.4 -> 11.6 us); rows of 4000 to 8000 vectors do not care.
constexpr int kLongRow = 4096;

template <bool BF16, int kGroupLoads>
__global__ void __launch_bounds__(kPassThreads, kPassCtasPerSm) argmax_pass_kernel(PassParams p) {
  using VT = Vec<BF16>;
  constexpr int kGroup = 32 * kGroupLoads;
  __shared__ int s_off[C2T_MAX_BATCH + 1];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  chain_enter();
  const int n_rows = build_row_offsets(p.counts, p.B, p.rows_per_seq_max, s_off);
  const int vpr = (p.V + VT::N - 1) / VT::N, v_full = p.V / VT::N;
  const long long total = (long long)n_rows * vpr;
  long long span = (total + gridDim.x - 1) / gridDim.x;
  if (span < kMinPassSpan) span = kMinPassSpan;
  long long pos = (long long)blockIdx.x * span;
  const long long end = pos + span < total ? pos + span : total;
  if (pos >= end) return;
  const size_t esz = BF16 ? 2 : 4;
  int a = (int)(pos / vpr), v0 = (int)(pos - (long long)a * vpr);
  int turn = warp;                                   // groups until this warp's next
  for (; pos < end; ++a, v0 = 0) {
    const long long left = end - pos;
    const int seg = left < (long long)(vpr - v0) ? (int)left : vpr - v0;
    const int v1 = v0 + seg, groups = (seg + kGroup - 1) / kGroup;
    pos += seg;
    if (turn < groups) {
      const int b = find_sequence(s_off, p.B, a), i = a - s_off[b], j = p.row_sel ? p.row_sel[b] : i;
      const char *row = reinterpret_cast<const char *>(p.logits) + ((size_t)b * p.seq_stride + (size_t)j * p.row_stride) * esz;
      const int whole = v1 < v_full ? v1 : v_full;   // (only the last vector of a ragged row is not whole)
      BestVector<BF16> bv;
      bv.clear();
      do {
        const int v = v0 + turn * kGroup + lane;
        uint4 q[kGroupLoads];
        if (v0 + (turn + 1) * kGroup <= whole) {
#pragma unroll
          for (int k = 0; k < kGroupLoads; ++k) q[k] = ldg_stream(reinterpret_cast<const uint4 *>(row) + v + k * 32);
#pragma unroll
          for (int k = 0; k < kGroupLoads; ++k) bv.take(q[k], v + k * 32);
        } else {
#pragma unroll
          for (int k = 0; k < kGroupLoads; ++k)
            if (v + k * 32 < whole) q[k] = ldg_stream(reinterpret_cast<const uint4 *>(row) + v + k * 32);
#pragma unroll
          for (int k = 0; k < kGroupLoads; ++k)
            if (v + k * 32 < whole) bv.take(q[k], v + k * 32);
          if (v1 > v_full && (v_full - v0) / kGroup == turn && lane == ((v_full - v0) & 31)) bv.take(VT::load(row, v_full, v_full, p.V), v_full);
        }
        turn += kWarps;
      } while (turn < groups);
      const unsigned long long best = warp_best(bv.key(p.V));
      const size_t slot = (size_t)b * p.rows_per_seq_max + i;
      if (lane == 0 && best && C2T_IN_BOUNDS(slot, p.n_slots, p.status)) atomicMax(&p.best[slot], best);
    }
    turn -= groups;
  }
}

// Rows a * row_stride of a matrix, in equal spans, one per CTA.  A row that lies in one span is answered by that CTA; of a row
// cut between CTAs each leaves its best key, and the CTA that finishes last answers those rows: no launch before this one to
// clear anything, none after it to gather.  The keys are written before they are read in every call.  What one call leaves for the
// next is the ticket: it counts modulo the grid, which is the same for all calls of a device, so that it is 0 after any number of
// whole calls, also when some of them overlapped.  256 rows of 128256 bf16 values (66 MB): 15.1 us;
// with keys and counts per row that the last CTA of a row puts back to zero 14.8, with a launch to clear and one to gather 23.9.
constexpr int kMinSpanVectors = 1024;  // a CTA never gets fewer 16-byte vectors than this
template <bool BF16>
__global__ void __launch_bounds__(kPassThreads, kPassCtasPerSm) row_argmax_kernel(const char *logits, long long row_bytes, int rows, int V,
                                                                                 ArgmaxPieces *pieces, unsigned *ticket, int32_t *out) {
  using VT = Vec<BF16>;
  __shared__ unsigned long long s_best[kWarps], s_key[kMaxArgmaxCtas];
  __shared__ bool s_last;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  static_assert(kMaxArgmaxCtas <= kPassThreads, "a thread per CTA");
  chain_enter();
  const int vpr = (V + VT::N - 1) / VT::N, v_full = V / VT::N;
  const int total = rows * vpr;                      // (at most 4096 * 65536)
  int span = (total + (int)gridDim.x - 1) / (int)gridDim.x;
  if (span < kMinSpanVectors) span = kMinSpanVectors;
  int pos = (int)blockIdx.x * span;
  const int end = pos + span < total ? pos + span : total;
  int a = pos / vpr, v0 = pos - a * vpr;
  ArgmaxPieces mine = {0ull, 0ull};                  // (thread 0)
  for (; pos < end; ++a, v0 = 0) {
    const int seg = end - pos < vpr - v0 ? end - pos : vpr - v0, v1 = v0 + seg;
    const char *row = logits + (size_t)a * row_bytes;
    BestVector<BF16> bv;
    bv.clear();
    int v = v0 + tid;
    for (; v + 3 * kPassThreads < v1; v += 4 * kPassThreads) {
      uint4 q[4];
#pragma unroll
      for (int i = 0; i < 4; ++i) q[i] = VT::load(row, v + i * kPassThreads, v_full, V);
#pragma unroll
      for (int i = 0; i < 4; ++i) bv.take(q[i], v + i * kPassThreads);
    }
    for (; v < v1; v += kPassThreads) bv.take(VT::load(row, v, v_full, V), v);
    unsigned long long key = warp_best(bv.key(V));
    if (lane == 0) s_best[warp] = key;
    __syncthreads();
    if (warp == 0) key = warp_best(lane < kWarps ? s_best[lane] : 0ull);
    __syncthreads();
    if (seg == vpr) {
      if (tid == 0) out[a] = key ? key_token(key) : -1;
    } else if (v0 > 0) {
      mine.first = key;                              // (the row began in another CTA's span)
    } else {
      mine.last = key;
    }
    pos += seg;
  }
  if (tid == 0) {
    pieces[blockIdx.x] = mine;
    unsigned turn;                                   // released: this CTA's pieces; acquired: those of the CTAs before it
    asm volatile("atom.acq_rel.gpu.global.inc.u32 %0, [%1], %2;" : "=r"(turn) : "l"(ticket), "r"(gridDim.x - 1) : "memory");
    s_last = turn == gridDim.x - 1;
  }
  // CTA c = tid, meanwhile: the row that begins in its span and goes on behind it; the CTA in which the row of its first vector begins
  const int c0 = tid * span, c1 = c0 + span < total ? c0 + span : total;
  const bool live = tid < (int)gridDim.x && c0 < total;
  int cut = -1, owner = -1;
  if (live) {
    const int r0 = (c1 - 1) / vpr, f0 = c0 / vpr * vpr;
    if (r0 * vpr >= c0 && (r0 + 1) * vpr > c1) cut = r0;
    if (f0 < c0) owner = f0 / span;
  }
  __syncthreads();
  if (!s_last) return;
  ArgmaxPieces p = {0ull, 0ull};
  if (live) { p.first = __ldcg(&pieces[tid].first); p.last = __ldcg(&pieces[tid].last); }
  s_key[tid] = p.last;
  __syncthreads();
  if (owner >= 0) atomicMax(&s_key[owner], p.first);
  __syncthreads();
  if (cut >= 0) out[cut] = s_key[tid] ? key_token(s_key[tid]) : -1;
}

// ---------------------------------------------------------------- lazy acceptance

__device__ __forceinline__ uint32_t cluster_rank() {
  uint32_t r;
  asm("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}
__device__ __forceinline__ void cluster_barrier() {
  asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
__device__ __forceinline__ void store_to_cta(unsigned long long *slot, uint32_t rank, unsigned long long v) {
  uint32_t at;
  asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(at) : "r"((uint32_t)__cvta_generic_to_shared(slot)), "r"(rank));
  asm volatile("st.shared::cluster.u64 [%0], %1;" ::"r"(at), "l"(v) : "memory");
}

// The greedy walk of one sequence per cluster (Sec. 5 Metrics), reading only the rows it visits.  Per round every CTA of
// the cluster takes the arg-max over its part of the current node's row, its warps put their best keys into all
// CTAs' shared memory, and after one cluster barrier every CTA finds the child that carries the token by itself (the tree is
// in its shared memory).  No sequence waits for another and no round for a launch (two launches per round and one more:
// 555 us per step of 64 x 128256 bf16, so 358).  CTAs: a row split over as many CTAs of the cluster as leaves the whole batch resident.
constexpr int kMaxCluster = 8;
constexpr int kLazyBatch = 8;          // 16-byte loads of a thread in flight
template <bool BF16>
__global__ void __launch_bounds__(kPassThreads, kPassCtasPerSm) accept_lazy_kernel(TreeState t, const char *logits, long long seq_stride,
                                                                                  long long row_stride, int V, int cluster, c2t_accept_out out) {
  using VT = Vec<BF16>;
  extern __shared__ int s_tree[];                    // [2, Nw] parents and tokens
  __shared__ unsigned long long s_keys[2][kMaxCluster * kWarps];
  __shared__ int s_found;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int b = (int)blockIdx.x / cluster, rank = (int)cluster_rank();
  const int Nw = t.Nw, width = t.D + 1;
  const size_t fb = (size_t)b * Nw, esz = BF16 ? 2 : 4;
  int *parent = s_tree, *token = s_tree + Nw;
  chain_enter();
  const int n = t.final_n[b];
  for (int i = tid; i < Nw; i += kPassThreads) {
    parent[i] = t.final_parent[fb + i];
    token[i] = t.final_token[fb + i];
    if (rank == 0) t.node_argmax[fb + i] = -1;
  }
  if (rank == 0 && out.path)
    for (int w = tid; w < width; w += kPassThreads) out.path[(size_t)b * width + w] = w == 0 ? 0 : -1;
  if (tid == 0) s_found = 0x7FFFFFFF;
  cluster_barrier();                                 // (all CTAs of the cluster run; and this CTA's shared memory is set up)
  const int vpr = (V + VT::N - 1) / VT::N, v_full = V / VT::N;
  const int part = (vpr + cluster - 1) / cluster, v_begin = rank * part, v_end = v_begin + part < vpr ? v_begin + part : vpr;
  int cur = 0, len = 0, want = -1;
  for (int round = 0; n > 0; ++round) {
    const char *row = logits + ((size_t)b * seq_stride + (size_t)cur * row_stride) * esz;
    BestVector<BF16> bv;
    bv.clear();
    for (int v0 = v_begin + tid; v0 < v_end; v0 += kPassThreads * kLazyBatch) {
      uint4 q[kLazyBatch];
#pragma unroll
      for (int i = 0; i < kLazyBatch; ++i)
        if (v0 + i * kPassThreads < v_end) q[i] = VT::load(row, v0 + i * kPassThreads, v_full, V);
#pragma unroll
      for (int i = 0; i < kLazyBatch; ++i)
        if (v0 + i * kPassThreads < v_end) bv.take(q[i], v0 + i * kPassThreads);
    }
    unsigned long long *keys = s_keys[round & 1];
    unsigned long long best = warp_best(bv.key(V));
    best = __shfl_sync(kFull, best, 0);
    if (lane < cluster) store_to_cta(&keys[rank * kWarps + warp], (uint32_t)lane, best);
    cluster_barrier();
    best = 0ull;
    for (int i = lane; i < cluster * kWarps; i += 32) best = keys[i] > best ? keys[i] : best;
    best = __shfl_sync(kFull, warp_best(best), 0);
    want = best ? key_token(best) : -1;
    if (rank == 0 && tid == 0) t.node_argmax[fb + cur] = want;
    // the first child that carries it
    int found = 0x7FFFFFFF;
    if (len + 1 < width)
      for (int c = cur + 1 + tid; c < n; c += kPassThreads)
        if (parent[c] == cur && token[c] == want) { found = c; break; }
    found = (int)__reduce_min_sync(kFull, (unsigned)found);
    if (lane == 0 && found != 0x7FFFFFFF) atomicMin(&s_found, found);
    __syncthreads();
    found = s_found;
    __syncthreads();
    if (found == 0x7FFFFFFF) break;                  // (the same in every CTA of the cluster)
    if (tid == 0) s_found = 0x7FFFFFFF;
    cur = found;
    ++len;
    if (rank == 0 && tid == 0 && out.path) out.path[(size_t)b * width + len] = cur;
  }
  if (rank == 0 && tid == 0) {
    if (out.accept_len) out.accept_len[b] = len;
    if (out.next_token) out.next_token[b] = want;
  }
}

}  // namespace

cudaError_t launch_argmax_pass(const PassParams &p, int dtype, int grid, cudaStream_t s) {
  const int vec = dtype == C2T_BF16 ? 8 : 4;
  const bool long_rows = (p.V + vec - 1) / vec >= kLongRow;
  if (dtype == C2T_BF16)
    return launch_chained(long_rows ? argmax_pass_kernel<true, 4> : argmax_pass_kernel<true, 8>, dim3(grid), dim3(kPassThreads), 0, s, p);
  return launch_chained(long_rows ? argmax_pass_kernel<false, 4> : argmax_pass_kernel<false, 8>, dim3(grid), dim3(kPassThreads), 0, s, p);
}

cudaError_t launch_row_argmax(const void *logits, int64_t row_stride, int rows, int V, int dtype, ArgmaxPieces *pieces, unsigned *ticket,
                              int32_t *out, int grid, cudaStream_t s) {
  const char *base = reinterpret_cast<const char *>(logits);
  if (dtype == C2T_BF16)
    return launch_chained(row_argmax_kernel<true>, dim3(grid), dim3(kPassThreads), 0, s, base, (long long)row_stride * 2, rows, V, pieces, ticket, out);
  return launch_chained(row_argmax_kernel<false>, dim3(grid), dim3(kPassThreads), 0, s, base, (long long)row_stride * 4, rows, V, pieces, ticket, out);
}

static size_t lazy_smem(int Nw) { return 2 * (size_t)Nw * sizeof(int); }

cudaError_t prepare_accept_lazy() {
  const int bytes = (int)lazy_smem(C2T_MAX_TREE);
  cudaError_t e = cudaFuncSetAttribute(accept_lazy_kernel<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
  if (e == cudaSuccess) e = cudaFuncSetAttribute(accept_lazy_kernel<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
  return e;
}

cudaError_t launch_accept_lazy(const TreeState &t, const void *logits, int64_t seq_stride, int64_t row_stride, const c2t_accept_out *out,
                               int dtype, int grid, cudaStream_t s) {
  c2t_accept_out o = {nullptr, nullptr, nullptr};
  if (out) o = *out;
  int cluster = 1;                                   // a power of two, while all clusters fit the chip at once
  while (cluster < kMaxCluster && 2 * cluster * t.B <= grid) cluster *= 2;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(t.B * cluster);
  cfg.blockDim = dim3(kPassThreads);
  cfg.dynamicSmemBytes = lazy_smem(t.Nw);
  cfg.stream = s;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  attr[1].id = cudaLaunchAttributeClusterDimension;
  attr[1].val.clusterDim.x = cluster;
  attr[1].val.clusterDim.y = attr[1].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 2;
  const char *base = reinterpret_cast<const char *>(logits);
  if (dtype == C2T_BF16)
    return cudaLaunchKernelEx(&cfg, accept_lazy_kernel<true>, t, base, (long long)seq_stride, (long long)row_stride, (int)t.V, cluster, o);
  return cudaLaunchKernelEx(&cfg, accept_lazy_kernel<false>, t, base, (long long)seq_stride, (long long)row_stride, (int)t.V, cluster, o);
}

}  // namespace c2t

// The expand pass for levels of few rows: every row in the registers of one thread block, or of a cluster of up to eight, per row
// the softmax normaliser and entropy sums and the K largest logits (ties to the lower token id), as expand_pass.cu leaves them
//                                                        (Sec. 4.2.1, Eq. 2, Sec. 4.2.2).
//
// Such a level is a chain of latencies, not a stream: its rows arrive in one round of loads, all in flight at once.  A thread holds
// up to 8 vectors of 16 bytes.  Nothing goes through global memory but the logits and the row's result, nothing is read twice, no row
// waits for another, and there is no list of rows to build: block (b, j) looks at one count.
//   Maxima of 64 groups of the row or more go to every block of the cluster; the K-th largest of them is a floor that at least K elements
// reach, and hardly more do.  While they travel the sums are taken, base 2 as in expand_pass.cu, a lane's relative to an offset from
// its own largest value.  The row's maximum is left out of them afterwards: the lane that holds it is summed again without it, its
// elements dealt out to the warp.  So the sums keep fp32 relative accuracy with respect to "everything but the maximum" however peaked the
// row is.  The threads whose maximum reaches the floor hand their elements over, the leading block ranks the keys and
// merges the warps' sums in double precision, in a fixed order.
//   What bounds it: latencies.  Of a level of 10 rows of 32000 fp32 tokens (clock reads in the kernel, taken once and not kept, when it took 9.9 us)
// the wait for the predecessor takes 0.9 us, the count 0.35, the loads 0.6, maxima 0.4, sums 0.35, the floor 0.6, what goes between the
// blocks 0.7, the result 1.4, the count of finished rows 0.7, the pruning 2.6; the other 1.3 lie outside the block that was read.  Against
// the streaming pass with the pruning of its time, a step: 1 x 32000 fp32 93 -> 67 us, 1 x 128256 bf16 158 -> 125, 8 x 32000 bf16 142 -> 107,
// 5 x 32003 fp32 107 -> 81.
#include "row_sums.cuh"

namespace c2t {
namespace {

constexpr int kMaxRowWarps = kRowThreads / 32;
constexpr int kRowLoads = kRowPart / kRowThreads;     // vectors of a thread
constexpr int kRowGroups = 64;                        // at least (and at least the largest K)
constexpr int kMaxRowGroups = kRowCluster * kMaxRowWarps;
constexpr int kCtaKeys = 64;                          // keys that a block hands over
constexpr int kTooMany = 1 << 20, kGivenUp = 1 << 24;  // instead of a count: not handed over; the block gives the row up
constexpr unsigned long long kNotPut = ~0ull;         // no block's best key
static_assert(kRowGroups >= C2T_MAX_TOPK && kMaxRowGroups >= kRowGroups, "");

// A warp's sums, relative to an integer offset, and how often it holds the row's maximum.
struct alignas(16) RowSums {
  double S, U;
  float offset;
  int equals;
};

struct RowShared {
  unsigned long long maxima_in, results_in;           // transaction barriers: all groups' maxima; everything for the row's result
  __align__(16) float group[kMaxRowGroups];           // the maxima of the row's groups
  RowSums sums[kRowCluster * kMaxRowWarps];           // in the leading block
  unsigned long long keys[kRowCluster][kCtaKeys];     // in the leading block: what every block hands over
  __align__(16) int counts[kRowCluster];              // how many
  unsigned long long pool[kPoolCap];                  // this block's keys; in the leading one then the row's
  __align__(16) uint4 again[kMaxRowWarps][kRowLoads]; // per warp: the vectors of a lane that is summed again
  unsigned long long best[2][kRowCluster], warp_best[kMaxRowWarps];
  unsigned floor;                                     // (orderable)
  int n, lost;
};

// ---------------------------------------------------------------- clusters

__device__ __forceinline__ int cluster_rank() {
  uint32_t r;
  asm("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return (int)r;
}
__device__ __forceinline__ void cluster_arrive() { asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory"); }
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory"); }
// the address of a place in this block's shared memory as block r of the cluster has it
__device__ __forceinline__ uint32_t place_in(const void *at, int r) {
  uint32_t to;
  asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(to) : "r"((uint32_t)__cvta_generic_to_shared(at)), "r"(r));
  return to;
}
__device__ __forceinline__ void put(uint32_t at, unsigned long long v) { asm volatile("st.shared::cluster.u64 [%0], %1;" ::"r"(at), "l"(v) : "memory"); }
// The same with its bytes counted by a transaction barrier of the block that it goes to: the receiver waits for the data, and nobody for
// the stores to be acknowledged (a cluster barrier with release semantics did: 0.5 us after the maxima, 0.7 us before the result).
__device__ __forceinline__ void send(uint32_t at, uint32_t v, uint32_t bar) {
  asm volatile("st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.b32 [%0], %1, [%2];" ::"r"(at), "r"(v), "r"(bar) : "memory");
}
__device__ __forceinline__ void send(uint32_t at, unsigned long long v, uint32_t bar) {
  asm volatile("st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.b64 [%0], %1, [%2];" ::"r"(at), "l"(v), "r"(bar) : "memory");
}
__device__ __forceinline__ void send(uint32_t at, unsigned long long a, unsigned long long b, uint32_t bar) {
  asm volatile("st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.v2.b64 [%0], {%1, %2}, [%3];" ::"r"(at), "l"(a), "l"(b), "r"(bar) : "memory");
}
// an arrival at a block's barrier that announces bytes to it
__device__ __forceinline__ void announce(uint32_t bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.relaxed.cluster.shared::cluster.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}
// false if the wait ran out
__device__ __forceinline__ bool wait_bar(const unsigned long long *bar, int limit) {
  const uint32_t at = (uint32_t)__cvta_generic_to_shared(bar);
  uint32_t done = 0u;
  for (int i = 0; i < limit && !done; ++i)
    asm volatile("{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], 0;\n\tselp.u32 %0, 1, 0, p;\n\t}"
                 : "=r"(done) : "r"(at) : "memory");
  return done != 0u;
}

__device__ __forceinline__ float warp_max(float v) {
  float m;
  asm("redux.sync.max.f32 %0, %1, 0xFFFFFFFF;" : "=f"(m) : "f"(v));
  return m;
}

// ---------------------------------------------------------------- a block's part of a row

template <bool BF16, int NT>
struct RowPart {
  const char *row;
  int vpr, v_full, part, v0, v1;                      // vectors of the row, whole ones, of a block; this block's range
  __device__ __forceinline__ void load(uint4 (&q)[kRowLoads], int V) const {
    const uint32_t lo = BF16 ? kLowestBf16x2 : __float_as_uint(kLowestF32);
    const int whole = v1 < v_full ? v1 : v_full;
#pragma unroll
    for (int k = 0; k < kRowLoads; ++k) {
      const int v = v0 + k * NT + (int)threadIdx.x;
      q[k] = make_uint4(lo, lo, lo, lo);
      if (v < whole) q[k] = ldg_stream(reinterpret_cast<const uint4 *>(row) + v);
    }
    if (v1 > v_full) {                                // (uniform) the row's ragged last vector
#pragma unroll
      for (int k = 0; k < kRowLoads; ++k)
        if (v0 + k * NT + (int)threadIdx.x == v_full) q[k] = load_ragged<BF16>(row, v_full, v_full, V);
    }
#pragma unroll
    for (int k = 0; k < kRowLoads; ++k) Vec<BF16>::clamp(q[k]);
  }
};

// one of a thread's vectors, by a number that is only known at run time
__device__ __forceinline__ uint4 pick(const uint4 (&q)[kRowLoads], int at) {
  uint4 t = q[0];
#pragma unroll
  for (int k = 1; k < kRowLoads; ++k)
    if (k == at) t = q[k];
  return t;
}

template <bool BF16>
__device__ __forceinline__ float element_of(const uint4 &q, int i) {
  const uint32_t w = BF16 ? ((i >> 1) == 0 ? q.x : (i >> 1) == 1 ? q.y : (i >> 1) == 2 ? q.z : q.w) : (i == 0 ? q.x : i == 1 ? q.y : i == 2 ? q.z : q.w);
  return BF16 ? __uint_as_float((i & 1) ? w & 0xFFFF0000u : w << 16) : __uint_as_float(w);
}

// The elements of vector v at or above a floor (which padding does not reach) as keys into the block's pool.  The count in shared
// memory keeps rising when the pool is full.
template <bool BF16>
__device__ __forceinline__ void hand_over(RowShared &sh, const uint4 &q, float floor, int v) {
  constexpr int N = Vec<BF16>::N;
  int c = 0;
#pragma unroll
  for (int i = 0; i < N; ++i) c += element_of<BF16>(q, i) >= floor;
  int pos = atomicAdd(&sh.n, c);
#pragma unroll
  for (int i = 0; i < N; ++i) {
    const float x = element_of<BF16>(q, i);
    if (x >= floor) {
      if (pos < kPoolCap) sh.pool[pos] = make_key(x, (uint32_t)(v * N + i));
      ++pos;
    }
  }
}

// Rows whose K largest do not come out of a short list (many equal values, few values, most of the row masked, very short rows): K rounds
// of "the largest key below the last one" over all blocks of the cluster.  Returns the number of keys, in the leading block's pool, or
// (in every block that is here) -1 if a block has given the row up: it does not put a key in the first round.
template <bool BF16, int NT>
__device__ __noinline__ int select_by_rounds(RowShared &sh, const RowPart<BF16, NT> &rp, int V, int K, int cluster, int rank) {
  constexpr int N = Vec<BF16>::N;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  uint4 q[kRowLoads];
  rp.load(q, V);
  unsigned long long last = ~0ull, best = 0ull;
  int r = 0;
  for (; r < K; ++r) {
    best = 0ull;
#pragma unroll
    for (int k = 0; k < kRowLoads; ++k) {
      const int v = rp.v0 + k * NT + tid;
      if (v >= rp.v1) continue;
      float x[N];
      Vec<BF16>::unpack(q[k], x);
#pragma unroll
      for (int i = 0; i < N; ++i) {
        const unsigned long long key = make_key(x[i], (uint32_t)(v * N + i));
        if (x[i] == x[i] && v * N + i < V && key < last && key > best) best = key;
      }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      const unsigned long long other = __shfl_xor_sync(kFull, best, o);
      best = other > best ? other : best;
    }
    if (lane == 0) sh.warp_best[warp] = best;
    __syncthreads();
    if (warp == 0) {
      best = 0ull;
      for (int w = 0; w < NT / 32; ++w) best = sh.warp_best[w] > best ? sh.warp_best[w] : best;
      if (lane < cluster) put(place_in(&sh.best[r & 1][rank], lane), best);
    }
    __syncwarp();
    cluster_arrive();
    cluster_wait();
    best = 0ull;
    for (int i = 0; i < cluster; ++i) best = sh.best[r & 1][i] > best ? sh.best[r & 1][i] : best;
    if (best + 1ull <= 1ull) break;                   // nothing left, or not put (the same in every block that is here)
    if (tid == 0) sh.pool[r] = best;
    last = best;
  }
  if (best == kNotPut) return -1;                     // (that was the first round)
  __syncthreads();
  for (int i = r + tid; i < K; i += NT) sh.pool[i] = 0ull;
  __syncthreads();
  return r;
}

// Sums (s, u) relative to an offset c, onto a warp's, which have an offset of at most that.  In double precision, as all sums over lanes
// are: a row's sums are mostly a few large elements, which fp32 would round five more times (32000 tokens, scale 4: 1.1e-8 r.m.s. in a
// probability, so rounded 1.6e-8).
__device__ __forceinline__ void add_sums(RowSums &r, float s, float u, float c) {
  const float by = fmaxf(r.offset - c, -2000.f);      // (never positive)
  const double f = pow2_f64(by);
  r.S += f * (double)s;
  r.U += f * ((double)u + (double)by * (double)s);
}

__device__ __forceinline__ void sum_lanes(RowSums &r) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    r.S += __shfl_xor_sync(kFull, r.S, o);
    r.U += __shfl_xor_sync(kFull, r.U, o);
  }
}

// One lane's vectors, in sh.again, summed again without the row's maximum and its equals: a word by every lane of the warp.
template <bool BF16>
__device__ __forceinline__ void sum_again(RowShared &sh, float Mf, RowSums &r) {
  const uint32_t word = reinterpret_cast<const uint32_t *>(sh.again[threadIdx.x >> 5])[threadIdx.x & 31];
  float x0 = BF16 ? __uint_as_float(word << 16) : __uint_as_float(word), x1 = BF16 ? __uint_as_float(word & 0xFFFF0000u) : kLowestF32;
  r.equals += (x0 == Mf) + (x1 == Mf);
  x0 = x0 == Mf ? kLowestF32 : x0;
  x1 = x1 == Mf ? kLowestF32 : x1;
  const float c = offset_of(warp_max(fmaxf(x0, x1)));
  const float t0 = fmaf(x0, kLog2e, c), t1 = fmaf(x1, kLog2e, c), e0 = ex2f(t0), e1 = ex2f(t1);
  add_sums(r, BF16 ? e0 + e1 : e0, BF16 ? fmaf(e0, t0, e1 * t1) : e0 * t0, c);
}

// The warps' sums, merged by one warp of the leading block.
__device__ __forceinline__ void merge_sums(RowShared &sh, RowResult *out, float Mf, int warps) {
  constexpr int kPer = kRowCluster * kMaxRowWarps / 32;
  const int lane = threadIdx.x & 31;
  const float cM = offset_of(Mf);
  double S = 0.0, U = 0.0;
  int equals = 0;
#pragma unroll
  for (int i = 0; i < kPer; ++i) {
    if (i * 32 + lane < warps) {
      const RowSums r = sh.sums[i * 32 + lane];
      const float d = fmaxf(cM - r.offset, -2000.f);  // (never positive)
      const double f = pow2_f64(d);
      S += f * r.S;
      U += f * (r.U + (double)d * r.S);
      equals += r.equals;
    }
  }
  S = warp_sum(S);
  U = warp_sum(U);
  equals = __reduce_add_sync(kFull, equals);
  if (lane == 0) write_sums(out, Mf, cM, S, U, equals);
}

// ---------------------------------------------------------------- a row

// A block whose wait for the row's result ran out: it knows neither what the others handed over nor what they do now.  They are done, or
// in the first round of select_by_rounds, or here.  Either way the next cluster barrier is reached by all of them (those that have
// ended count), and behind it all that they send to this block is on its way: it stays until that has arrived.
__device__ __noinline__ void leave_row(const RowShared &sh) {
  cluster_arrive();
  cluster_wait();
  wait_bar(&sh.maxima_in, kTaskWaitLimit);
  wait_bar(&sh.results_in, kTaskWaitLimit);
  __syncthreads();
}

// Before the kernel waits for its predecessor: this block's shared memory can be written once the block runs.
__device__ __forceinline__ void open_row(RowShared &sh, int cluster) {
  if (threadIdx.x < kRowCluster) sh.best[0][threadIdx.x] = (int)threadIdx.x < cluster ? kNotPut : 0ull;
  if (threadIdx.x == 0) {
    sh.floor = 0u;
    sh.n = sh.lost = 0;
    if (cluster > 1) {
      const uint32_t maxima = (uint32_t)__cvta_generic_to_shared(&sh.maxima_in), results = (uint32_t)__cvta_generic_to_shared(&sh.results_in);
      const int warps = cluster * (int)(blockDim.x >> 5), groups = warps > kRowGroups ? warps : kRowGroups;
      asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;\n\tmbarrier.init.shared::cta.b64 [%1], %2;\n\tfence.mbarrier_init.release.cluster;"
                   ::"r"(maxima), "r"(results), "r"(cluster) : "memory");
      asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(maxima), "r"(groups * 4) : "memory");
    }
  }
  __syncwarp();
  if (cluster > 1) cluster_arrive();
}

// Row (b, j) by the blocks of a cluster, after open_row and the wait for it.  True in the leading block, after the row's result is written (by its first two warps).
template <bool BF16, int NT>
__device__ __forceinline__ bool expand_row(const PassParams &p, RowShared &sh, int b, int j, int cluster, int rank) {
  constexpr int kW = NT / 32;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, K = p.K, warps = cluster * kW;
  RowPart<BF16, NT> rp;
  rp.vpr = (p.V + Vec<BF16>::N - 1) / Vec<BF16>::N;
  rp.v_full = p.V / Vec<BF16>::N;
  rp.part = (rp.vpr + cluster - 1) / cluster;
  rp.v0 = rank * rp.part;
  rp.v1 = rp.v0 + rp.part < rp.vpr ? rp.v0 + rp.part : rp.vpr;
  rp.row = reinterpret_cast<const char *>(p.logits) + ((size_t)b * p.seq_stride + (size_t)j * p.row_stride) * (BF16 ? 2 : 4);
  uint4 q[kRowLoads];
  rp.load(q, p.V);

  // ---- maxima: the thread's, and those of groups of `width` lanes to every block, one of them from each lane of the group
  RunMax<BF16> run;
  run.clear();
#pragma unroll
  for (int k = 0; k < kRowLoads; ++k) run.take(q[k]);
  const float mt = run.value();
  const int groups = warps > kRowGroups ? warps : kRowGroups, width = 32 * warps / groups;
  float g = mt;
  for (int o = 1; o < width; o <<= 1) g = fmaxf(g, __shfl_xor_sync(kFull, g, o));
  const int to = lane & (width - 1), at = (rank * kW + warp) * (32 / width) + lane / width;
  if (cluster > 1) {
    if (to < cluster && C2T_IN_BOUNDS(at, groups, p.status)) send(place_in(&sh.group[at], to), __float_as_uint(g), place_in(&sh.maxima_in, to));
  } else if (to == 0 && C2T_IN_BOUNDS(at, groups, p.status)) {
    sh.group[at] = g;
  }

  // ---- the sums
  const float c = offset_of(mt);
  float s, u;
  {
    const f32x2 scale = pack2(kLog2e, kLog2e), c2 = pack2(c, c);
    Acc acc;
    acc.clear();
#pragma unroll
    for (int k = 0; k < kRowLoads; ++k)
      if (k * NT < rp.part) acc_vector<BF16>(acc, q[k], scale, c2);      // (uniform)
    acc.totals(s, u);
  }
  RowSums sums = {0.0, 0.0, offset_of(warp_max(mt)), 0};
  add_sums(sums, s, u, c);
  sum_lanes(sums);
  if (cluster > 1) {
    if (!wait_bar(&sh.maxima_in, p.wait_limit)) sh.lost = 1;       // (nothing of the kind is expected) the block gives the row up
  } else {
    __syncthreads();
  }

  // ---- the row's maximum, which stays out of them; the floor: the K-th largest of the groups' maxima, the largest value that K of them reach
  float Mf = fmaxf(sh.group[lane], sh.group[32 + lane]);
  if (groups > 64) Mf = fmaxf(Mf, fmaxf(sh.group[64 + lane], sh.group[96 + lane]));
  Mf = warp_max(Mf);
  {
    const int team = NT / groups, member = tid & (team - 1);      // threads of a group: 2 to 8
    const float mine = sh.group[tid / team];
    int reach = 0;
    for (int i = member * 4; i < groups; i += team * 4) {
      const float4 o = *reinterpret_cast<const float4 *>(&sh.group[i]);
      reach += (o.x >= mine) + (o.y >= mine) + (o.z >= mine) + (o.w >= mine);
    }
    for (int o = 1; o < team; o <<= 1) reach += __shfl_xor_sync(kFull, reach, o);
    const unsigned top = __reduce_max_sync(kFull, reach >= K ? f32_orderable(__float_as_uint(mine)) : 0u);
    if (lane == 0 && top) atomicMax(&sh.floor, top);
  }
  __syncthreads();
  const float floor = __uint_as_float(f32_from_orderable(sh.floor));
  const bool live = floor > kLowestF32;               // (uniform; else fewer than K groups have data)

  // ---- the elements that reach it
  if (live && mt >= floor) {
    unsigned hit = 0u;
#pragma unroll
    for (int k = 0; k < kRowLoads; ++k) hit |= (unsigned)(Vec<BF16>::vmax(q[k]) >= floor) << k;
    while (hit) {
      const int k = __ffs(hit) - 1;
      hit &= hit - 1u;
      hand_over<BF16>(sh, pick(q, k), floor, rp.v0 + k * NT + tid);
    }
  }
  __syncthreads();
  if (warp == 0) {
    const int n = sh.n, most = cluster > 1 ? kCtaKeys : kPoolCap, c_n = sh.lost ? kGivenUp : !live || n > most ? kTooMany : n;
    const int handed = c_n < kTooMany ? c_n : 0;
    if (cluster > 1) {
      if (lane < cluster) {
        const uint32_t bar = place_in(&sh.results_in, lane);
        announce(bar, lane == 0 ? (uint32_t)(4 + kW * 24 + handed * 8) : 4u);
        send(place_in(&sh.counts[rank], lane), (uint32_t)c_n, bar);
      }
      const uint32_t bar = place_in(&sh.results_in, 0);
      for (int i = lane; i < handed; i += 32)
        if (C2T_IN_BOUNDS(i, kCtaKeys, p.status)) send(place_in(&sh.keys[rank][i], 0), sh.pool[i], bar);
    } else if (lane == 0) {
      sh.counts[0] = c_n;                             // (the keys are where they are ranked)
    }
    __syncwarp();
  }

  // ---- the warps' sums; the warp that holds the maximum: such lanes again without it
  if (unsigned left = __ballot_sync(kFull, mt == Mf)) {
    sums = {0.0, 0.0, offset_of(Mf), 0};
    if (mt != Mf) add_sums(sums, s, u, c);
    for (; left; left &= left - 1u) {
      __syncwarp();
      if (lane == __ffs(left) - 1) {
#pragma unroll
        for (int k = 0; k < kRowLoads; ++k) sh.again[warp][k] = q[k];
      }
      __syncwarp();
      sum_again<BF16>(sh, Mf, sums);
    }
    sum_lanes(sums);
    sums.equals = __reduce_add_sync(kFull, sums.equals);
  }
  if (lane == 0 && C2T_IN_BOUNDS(rank * kW + warp, kRowCluster * kMaxRowWarps, p.status)) {
    RowSums *record = &sh.sums[rank * kW + warp];
    if (cluster > 1) {
      const uint32_t bar = place_in(&sh.results_in, 0);
      send(place_in(record, 0), (unsigned long long)__double_as_longlong(sums.S), (unsigned long long)__double_as_longlong(sums.U), bar);
      send(place_in(&record->offset, 0), (unsigned long long)(uint32_t)sums.equals << 32 | __float_as_uint(sums.offset), bar);
    } else {
      *record = sums;
    }
  }
  __syncwarp();
  if (cluster > 1) {
    if (__syncthreads_or(!wait_bar(&sh.results_in, p.wait_limit))) {
      leave_row(sh);
      if (rank == 0 && warp == 0) give_up_row(p, b, j);
      return rank == 0;
    }
  } else {
    __syncthreads();
  }

  // ---- the row's result
  int upto[kRowCluster], total = 0;                   // keys up to and with block r
#pragma unroll
  for (int r = 0; r < kRowCluster; ++r) {
    if (r < cluster) total += sh.counts[r];
    upto[r] = total;
  }
  const bool listed = total <= kPoolCap;              // (the same in every block that is here)
  int n_valid = 0;
  if (!listed) {
    n_valid = -1;
    if (total < kGivenUp) n_valid = select_by_rounds<BF16, NT>(sh, rp, p.V, K, cluster, rank);
    else wait_bar(&sh.maxima_in, kTaskWaitLimit);     // (what is on its way to a block arrives before it ends)
    if (n_valid < 0) {
      if (rank == 0 && warp == 0) give_up_row(p, b, j);
      return rank == 0;
    }
  }
  if (rank != 0) return false;
  const size_t slot = (size_t)b * p.rows_per_seq_max + j;
  if (!C2T_IN_BOUNDS(slot, (size_t)p.B * p.rows_per_seq_max, p.status)) return true;
  if (warp == 0) {
    if (listed) {
      for (int i = lane; cluster > 1 && i < total; i += 32) {
        int r = 0, before = 0;
#pragma unroll
        for (int k = 0; k < kRowCluster; ++k)
          if (upto[k] <= i) { r = k + 1; before = upto[k]; }
        if (C2T_IN_BOUNDS(r, cluster, p.status) && C2T_IN_BOUNDS(i - before, kCtaKeys, p.status)) sh.pool[i] = sh.keys[r][i - before];
      }
      __syncwarp();
      n_valid = rank_pool(sh.pool, total, K);
    }
    for (int i = lane; i < K; i += 32) p.row_keys[slot * K + i] = sh.pool[i];
    if (lane == 0) {
      p.rows[slot].top = sh.pool[0];
      p.rows[slot].n_valid = n_valid;
    }
  } else if (warp == 1) {
    merge_sums(sh, p.rows + slot, Mf, warps);
  }
  return true;
}

// ---------------------------------------------------------------- kernels

// Block x = (row slot, place in the cluster), y = sequence.  (row_pass_plan leaves an SM 512 threads of them; with the 64 registers that 1024
// would allow, code spills: 28 sequences of 16000 bf16 tokens 13.3 us a level, so 10.8, 3 of 32000 9.6, so 8.7.)
template <bool BF16, int NT>
__global__ void __launch_bounds__(NT, 512 / NT) expand_rows_kernel(const __grid_constant__ PassParams p, int cluster) {
  __shared__ RowShared sh;
  chain_release();
  open_row(sh, cluster);
  const int b = blockIdx.y, j = (int)blockIdx.x / cluster;
  chain_wait();
  const int n = p.counts[b];
  if (cluster > 1) cluster_wait();
  if (j >= n) return;
  expand_row<BF16, NT>(p, sh, b, j, cluster, cluster > 1 ? cluster_rank() : 0);
}

// Expand and prune of a level in one launch: the cluster that finishes a sequence's last row (a count, nobody
// waits) does the sequence's part of c2t_prune.
template <bool BF16, int NT, int ROUNDS>
__global__ void __launch_bounds__(NT, 512 / NT) expand_rows_prune_kernel(const __grid_constant__ PassParams p, const __grid_constant__ TreeState t,
                                                                           int level, c2t_frontier out, int cluster) {
  __shared__ union {
    RowShared row;
    struct { unsigned long long barriers[2]; PruneShared prune; } then;       // (barriers keep their place)
  } sh;
  __shared__ __align__(16) double s_w[kWCount];
  __shared__ int s_last;
  const int rank = cluster > 1 ? cluster_rank() : 0;
  chain_release();
  open_row(sh.row, cluster);
  if (rank == 0) stage_classifier(t, s_w, threadIdx.x, NT);           // (written at init)
  const int b = blockIdx.y, j = (int)blockIdx.x / cluster;
  chain_wait();
  int n = p.counts[b];
  if (cluster > 1) cluster_wait();
  n = n < p.rows_per_seq_max ? n : p.rows_per_seq_max;
  if (n > 0 && !C2T_IN_BOUNDS(n - 1, p.rows_bound, p.status)) n = p.rows_bound;      // (or its last row would never be counted)
  if (j >= n && !(n <= 0 && j == 0)) return;
  if (n > 0) {
    if (!expand_row<BF16, NT>(p, sh.row, b, j, cluster, rank)) return;
    __syncthreads();                                 // the row's result, before its count
    if (threadIdx.x == 0) {
      int done;                                      // released: this row's result; acquired: those of the rows before it
      asm volatile("atom.acq_rel.gpu.global.inc.u32 %0, [%1], %2;" : "=r"(done) : "l"(p.row_done + (size_t)b * p.rows_per_seq_max), "r"(n - 1) : "memory");
      s_last = done == n - 1;                        // (and the count is back at 0)
    }
    __syncthreads();
    if (!s_last) return;
  } else if (rank != 0) {
    return;
  }
  prune_level_body<NT, ROUNDS, false>(t, level, out, nullptr, 0, b, sh.then.prune, s_w, nullptr);
}

template <typename... KArgs, typename... Args>
cudaError_t launch_rows(void (*kernel)(KArgs...), dim3 grid, int threads, int cluster, cudaStream_t s, Args &&...args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = dim3(threads);
  cfg.stream = s;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  attr[1].id = cudaLaunchAttributeClusterDimension;
  attr[1].val.clusterDim.x = cluster;
  attr[1].val.clusterDim.y = attr[1].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = cluster > 1 ? 2 : 1;
  return cudaLaunchKernelEx(&cfg, kernel, KArgs(args)...);
}

}  // namespace

cudaError_t launch_expand_rows(PassParams p, int dtype, RowPlan plan, cudaStream_t s) {
  p.wait_limit = C2T_TASK_WAIT_LIMIT;
  const dim3 grid(p.rows_bound * plan.cluster, p.B);
  const bool bf16 = dtype == C2T_BF16;
  if (plan.threads == 256) return launch_rows(bf16 ? expand_rows_kernel<true, 256> : expand_rows_kernel<false, 256>, grid, 256, plan.cluster, s, p, plan.cluster);
  return launch_rows(bf16 ? expand_rows_kernel<true, 512> : expand_rows_kernel<false, 512>, grid, 512, plan.cluster, s, p, plan.cluster);
}

cudaError_t launch_expand_rows_prune(PassParams p, const TreeState &t, int level, const c2t_frontier &out, int dtype, RowPlan plan, cudaStream_t s) {
  p.wait_limit = C2T_TASK_WAIT_LIMIT;
  const dim3 grid(p.rows_bound * plan.cluster, p.B);
  const bool bf16 = dtype == C2T_BF16;
  const bool small = t.F * t.K <= plan.threads;       // a candidate per thread
  constexpr int k256 = kMaxCand / 256, k512 = kMaxCand / 512;
  const auto kernel = plan.threads == 256
                          ? (bf16 ? (small ? expand_rows_prune_kernel<true, 256, 1> : expand_rows_prune_kernel<true, 256, k256>)
                                  : (small ? expand_rows_prune_kernel<false, 256, 1> : expand_rows_prune_kernel<false, 256, k256>))
                          : (bf16 ? (small ? expand_rows_prune_kernel<true, 512, 1> : expand_rows_prune_kernel<true, 512, k512>)
                                  : (small ? expand_rows_prune_kernel<false, 512, 1> : expand_rows_prune_kernel<false, 512, k512>));
  return launch_rows(kernel, grid, plan.threads, plan.cluster, s, p, t, level, out, plan.cluster);
}

}  // namespace c2t

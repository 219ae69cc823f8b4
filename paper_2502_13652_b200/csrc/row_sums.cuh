// What the two forms of the expand pass share (expand_pass.cu: rows in a stream; row_pass.cu: rows in registers): packed base-2 sums,
// running maxima, and a row's result from its merged sums.
#pragma once

#include <math.h>

#include "vocab_common.cuh"
#include "level_prune.cuh"

namespace c2t {
namespace {

// ---------------------------------------------------------------- packed sums

typedef unsigned long long f32x2;

__device__ __forceinline__ f32x2 pack2(float lo, float hi) {
  f32x2 d;
  asm("mov.b64 %0, {%1, %2};" : "=l"(d) : "f"(lo), "f"(hi));
  return d;
}
__device__ __forceinline__ void unpack2(f32x2 a, float &lo, float &hi) { asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(a)); }
__device__ __forceinline__ f32x2 fma2(f32x2 a, f32x2 b, f32x2 c) {
  f32x2 d;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
  return d;
}
__device__ __forceinline__ f32x2 add2(f32x2 a, f32x2 b) {
  f32x2 d;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
  return d;
}

__device__ __forceinline__ f32x2 mul2(f32x2 a, f32x2 b) {
  f32x2 d;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
  return d;
}

// S and U of a lane: two packed accumulators each, so that consecutive additions do not wait for each other.
struct Acc {
  f32x2 S[2], U[2];
  __device__ __forceinline__ void clear() { S[0] = S[1] = U[0] = U[1] = 0ull; }
  __device__ __forceinline__ void totals(float &s, float &u) const {
    float a, b, c, d;
    unpack2(add2(S[0], S[1]), a, b);
    unpack2(add2(U[0], U[1]), c, d);
    s = a + b;
    u = c + d;
  }
};

__device__ __forceinline__ void acc_pair(Acc &a, int i, float x0, float x1, f32x2 scale, f32x2 c) {
  const f32x2 t = fma2(pack2(x0, x1), scale, c);
  float t0, t1;
  unpack2(t, t0, t1);
  const f32x2 e = pack2(ex2f(t0), ex2f(t1));
  a.S[i] = add2(a.S[i], e);
  a.U[i] = fma2(e, t, a.U[i]);
}

template <bool BF16>
__device__ __forceinline__ void acc_vector(Acc &a, const uint4 &q, f32x2 scale, f32x2 c) {
  float x[Vec<BF16>::N];
  Vec<BF16>::unpack(q, x);
#pragma unroll
  for (int i = 0; i < Vec<BF16>::N; i += 2) acc_pair(a, (i >> 1) & 1, x[i], x[i + 1], scale, c);
}

// ---------------------------------------------------------------- maxima

// A running maximum of whole vectors (NaN ignored): packed for bf16, plain for fp32.
template <bool BF16>
struct RunMax {
  uint32_t v;
  __device__ __forceinline__ void clear() { v = BF16 ? kLowestBf16x2 : __float_as_uint(kLowestF32); }
  __device__ __forceinline__ void take(const uint4 &q) {
    if (BF16) v = max_bf16x2(v, max_bf16x2(max_bf16x2(q.x, q.y), max_bf16x2(q.z, q.w)));
    else v = __float_as_uint(fmaxf(__uint_as_float(v), fmaxf(fmaxf(__uint_as_float(q.x), __uint_as_float(q.y)),
                                                             fmaxf(__uint_as_float(q.z), __uint_as_float(q.w)))));
  }
  __device__ __forceinline__ void take(const RunMax &o) {
    v = BF16 ? max_bf16x2(v, o.v) : __float_as_uint(fmaxf(__uint_as_float(v), __uint_as_float(o.v)));
  }
  __device__ __forceinline__ float value() const {
    return BF16 ? fmaxf(__uint_as_float(v << 16), __uint_as_float(v & 0xFFFF0000u)) : __uint_as_float(v);
  }
};

// ---------------------------------------------------------------- offsets

// The offset of a reference m: an integer at or below -m log2(e), and monotone, so that no value up to m has a positive t.
__device__ __forceinline__ float offset_of(float m) { return floorf(__fmul_rd(fminf(m, 2e38f), -kLog2e)); }
constexpr float kNoOffset = 3e38f;                    // no data yet: behind every real offset

// Sums follow their offset down by d, an integer <= 0: every t by d, every weight by 2^d (0 from d = -127 on).
struct Shift {
  f32x2 d, f;
  __device__ __forceinline__ explicit Shift(float by) {
    by = fmaxf(by, -127.f);
    const float two = __int_as_float((__float_as_int(by + 12582912.f) << 23) + 0x3F800000);      // 2^by
    d = pack2(by, by);
    f = pack2(two, two);
  }
  __device__ __forceinline__ void apply(f32x2 &S, f32x2 &U) const {
    U = mul2(f, fma2(d, S, U));
    S = mul2(f, S);
  }
};

// 2^d for an integer d <= 0
__device__ __forceinline__ double pow2_f64(float d) { return d < -1000.f ? 0.0 : __hiloint2double((1023 + (int)d) << 20, 0); }

// the ragged last vector of a row, assembled from scalar loads
template <bool BF16>
__device__ __noinline__ uint4 load_ragged(const void *row, int v, int v_full, int V) { return Vec<BF16>::load(row, v, v_full, V); }

// ---------------------------------------------------------------- a row's result

// A row's maximum and its sums S, U relative to cM = offset_of(Mf), over all elements but the `equals` ones with the maximum's value, into
// its result, by one thread.  t = x kLog2e + cM with the fp32 constant, so x - M = t kBack + g, exactly that constant's inverse: its error
// of 1.3e-8 of x must not meet the exact M.  What is left is that 2^t is not e^(t kBack) but short of it by kShort t, small where the
// weight is.
__device__ __forceinline__ void write_sums(RowResult *r, float Mf, float cM, double S, double U, int equals) {
  const double kBack = 1.0 / (double)kLog2e, kShort = kBack - 0.69314718055994530942;
  const double M = (double)Mf, g = -(double)cM * kBack - M, scale = exp_shared(g);
  // sums of e^(t kBack) from those of 2^t, to first order (sum 2^t t^2 taken as U^2 / S: the weight lies close together)
  if (S > 1e-30) {
    const double short_of = kShort * U;
    U += short_of * (double)__fdividef((float)U, (float)S);
    S += short_of;
  }
  const double Sn = S * scale + (double)(equals - 1), Tn = scale * (kBack * U + g * S);
  r->M = M; r->S = Sn; r->T = Tn;
  const double L = log1p(Sn);                       // ln sum_v e^(x_v - M); the maximum contributes the 1
  r->L = L;
  r->H = L - Tn / (1.0 + Sn);                       // Eq. 2 with natural log
  r->fault = row_fault_bits(Mf, Sn, Tn);
}

// The result of a row that was given up: no candidates, and the fault that says so.
__device__ __forceinline__ void give_up_row(const PassParams &p, int b, int j) {
  const int lane = threadIdx.x & 31;
  const size_t slot = (size_t)b * p.rows_per_seq_max + j;
  for (int i = lane; i < p.K; i += 32) p.row_keys[slot * p.K + i] = 0ull;
  if (lane == 0) {
    RowResult r;
    r.M = r.S = r.T = r.L = r.H = 0.0;
    r.top = 0ull;
    r.n_valid = 0;
    r.fault = C2T_ST_INTERNAL;
    p.rows[slot] = r;
  }
  __syncwarp();
}

constexpr int kPoolCap = 128;                       // keys ranked at a time

// Ranks the first n keys of the pool: the K largest move to pool[0 .. K), sorted, 0-padded.  Returns how many there are.
__device__ __noinline__ int rank_pool(unsigned long long *pool, int n, int K) {
  const int lane = threadIdx.x & 31;
  if (n <= 32) {                                     // the usual case: a key per lane
    const unsigned long long key = lane < n ? pool[lane] : 0ull;
    int place = 0;
#pragma unroll 8
    for (int r = 0; r < n; ++r) place += pool[r] > key;
    if (lane >= n) place = lane;                     // (the zeros behind the keys)
    __syncwarp();
    pool[place] = key;
    __syncwarp();
    return n < K ? n : K;
  }
  unsigned long long mine[kPoolCap / 32];
  int rank[kPoolCap / 32];
#pragma unroll
  for (int i = 0; i < kPoolCap / 32; ++i) {
    mine[i] = i * 32 + lane < n ? pool[i * 32 + lane] : 0ull;
    rank[i] = 0;
  }
  for (int r = 0; r < n; ++r) {
    const unsigned long long k = pool[r];
#pragma unroll
    for (int i = 0; i < kPoolCap / 32; ++i) rank[i] += k > mine[i];
  }
  __syncwarp();
#pragma unroll
  for (int i = 0; i < kPoolCap / 32; ++i)
    if (mine[i] != 0ull && rank[i] < K) pool[rank[i]] = mine[i];     // (K <= 32 < n: all K places are taken)
  __syncwarp();
  return K;
}

}  // namespace
}  // namespace c2t

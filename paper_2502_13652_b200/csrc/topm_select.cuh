// The last step of the truncated entropy (Eq. 3), shared by its kernels: from the keys of a candidate set to the sums over the M largest.
#pragma once

#include "vocab_common.cuh"

namespace c2t {
namespace {

// the keys of one array, dealt out to NT threads
template <int NT>
struct FlatKeys {
  const uint32_t *keys;
  unsigned n;
  template <typename F>
  __device__ __forceinline__ void operator()(F f) const {
    for (unsigned i = threadIdx.x; i < n; i += NT) f(keys[i]);
  }
};
template <int NT>
__device__ __forceinline__ FlatKeys<NT> flat_keys(const uint32_t *keys, unsigned n) { return FlatKeys<NT>{keys, n}; }

// Eq. 3's sums from a candidate set in shared memory that is known to hold the M largest elements of the row
// (at least M keys, the order-preserving images of the values; each(f) calls f(key) for a thread's share of them): the M-th largest key, then the terms above it and as
// many copies of the term at it as are still missing.  Called by all NT threads of the CTA; thread 0 writes the
// result.
//   The candidates lie close together (between a floor and the row maximum), so a histogram over fixed key bytes
// would put nearly all of them in one bin, one shared-memory atomic after the other.  The bins follow the data
// instead: kSelBins equal steps between the smallest and the largest key still in play, refined until a step is
// one key wide (one round for bf16 rows as a rule, two or three for fp32).
constexpr int kSelBins = 2048;

// key_lo, key_hi: keys that bound the set from below and from above (the floor it was collected with, the row maximum).
template <bool BF16, int NT, typename Each>
__device__ __forceinline__ void select_and_sum(Each each, int M, float mf, uint32_t key_lo,
                                               uint32_t key_hi, double *s_sum, unsigned *s_need, double2 *out) {
  __shared__ unsigned s_bins[kSelBins];
  __shared__ unsigned s_wsum[NT / 32], s_lo, s_hi;
  __shared__ double s_tail[2];
  constexpr int BPT = kSelBins / NT;               // bins a thread owns when the bin with the M-th largest is looked for
  static_assert(kSelBins % NT == 0, "whole bins per thread");
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  constexpr int KS = BF16 ? 16 : 0;                // bf16 images are told apart by their upper halves
  if (key_lo == 0x80000000u) key_lo = 0x7FFFFFFFu; // a floor of +0 also admits -0, whose key is one lower
  if (tid == 0) { s_lo = key_lo >> KS; s_hi = key_hi >> KS; *s_need = (unsigned)M; }
  __syncthreads();
  // ---- refine [lo, hi] around the M-th largest key
  for (int round = 0; round < 4; ++round) {          // (32 key bits, 11 per round: three at most)
    const uint32_t lo = s_lo, hi = s_hi;
    const unsigned need = *s_need;
    if (lo == hi) break;                             // (uniform) one key left: `need` copies of it are still missing
    const uint32_t range = hi - lo;
    const int shift = range < (uint32_t)kSelBins ? 0 : 32 - __clz(range) - 11;     // range >> shift < kSelBins
    for (int i = tid; i < kSelBins; i += NT) s_bins[i] = 0u;
    __syncthreads();
    each([&](uint32_t key) {
      const uint32_t k = key >> KS;
      if (k >= lo && k <= hi) atomicAdd(&s_bins[(k - lo) >> shift], 1u);
    });
    __syncthreads();
    // the bin, from the top, that holds the need-th largest: thread t owns bins [t BPT, (t + 1) BPT)
    unsigned h[BPT], mine = 0u;
#pragma unroll
    for (int i = 0; i < BPT; ++i) { h[i] = s_bins[tid * BPT + i]; mine += h[i]; }
    unsigned suf = mine;                             // inclusive suffix sum over the lanes of the warp
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const unsigned v = __shfl_down_sync(kFull, suf, o);
      if (lane + o < 32) suf += v;
    }
    if (lane == 0) s_wsum[warp] = suf;
    __syncthreads();
    unsigned higher = suf - mine;                    // keys in the bins of higher threads
    for (int w = warp + 1; w < NT / 32; ++w) higher += s_wsum[w];
    if (higher < need && higher + mine >= need) {    // exactly one thread (at least `need` keys are in play)
      unsigned acc = higher;
      int d = tid * BPT;
#pragma unroll
      for (int i = BPT - 1; i >= 0; --i) {
        if (acc + h[i] >= need) { d = tid * BPT + i; break; }
        acc += h[i];
      }
      const uint32_t new_lo = lo + ((uint32_t)d << shift);
      const uint32_t step_top = new_lo + ((1u << shift) - 1u);
      s_lo = new_lo;
      s_hi = step_top < hi ? step_top : hi;
      *s_need = need - acc;
    }
    __syncthreads();
    if (shift == 0) break;                           // (uniform) the bin was one key
  }
  // keys above tau are all taken; of the keys equal to tau, *s_need are
  const uint32_t tau = s_lo;
  double Sd = 0.0, Td = 0.0;
  each([&](uint32_t key) {
    if ((key >> KS) > tau) {
      const float d = __uint_as_float(f32_from_orderable(key)) - mf;
      const float e = ex2f(d * kLog2e);            // (the expand pass takes its exponentials the same way)
      Sd += (double)e;
      Td += (double)(e * d);
    }
  });
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    Sd += __shfl_xor_sync(kFull, Sd, o);
    Td += __shfl_xor_sync(kFull, Td, o);
  }
  if (lane == 0) { s_sum[warp] = Sd; s_sum[NT / 32 + warp] = Td; }
  if (tid == NT - 1) {                               // meanwhile: the term at tau (its double-precision exp is long)
    // the key's value (a bf16 image's lower half is all ones for a negative value)
    const uint32_t tk = BF16 ? (tau << 16) | ((tau >> 15) ? 0u : 0xFFFFu) : tau;
    const double d = (double)__uint_as_float(f32_from_orderable(tk)) - (double)mf;
    const double e = exp(d);
    s_tail[0] = e;
    s_tail[1] = e * d;
  }
  __syncthreads();
  if (tid == 0) {
    double St = 0.0, Tt = 0.0;
    for (int w = 0; w < NT / 32; ++w) { St += s_sum[w]; Tt += s_sum[NT / 32 + w]; }
    const unsigned need = *s_need;
    St += (double)need * s_tail[0];
    Tt += (double)need * s_tail[1];
    *out = make_double2(St, Tt);
  }
}

}  // namespace
}  // namespace c2t

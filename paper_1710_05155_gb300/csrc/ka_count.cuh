// ka_count.cuh -- bit-sliced counters: 64 replicas counted at once, one uint64
// per binary digit.
#pragma once

#include "ka_internal.cuh"

namespace ka {
namespace {

__device__ __forceinline__ uint64_t maj(uint64_t a, uint64_t b, uint64_t c) {
  return (a & b) | (c & (a | b));
}

// full adder: s += x + y, returns the carry word
__device__ __forceinline__ uint64_t add2(uint64_t& s, uint64_t x, uint64_t y) {
  const uint64_t k = maj(s, x, y);
  s ^= x ^ y;
  return k;
}

// the first two digits of c += x[0] + .. + x[3]; returns the carry of weight four
template <int S>
__device__ __forceinline__ uint64_t add4(uint64_t (&c)[S], const uint64_t (&x)[4]) {
  const uint64_t t0 = add2(c[0], x[0], x[1]), t1 = add2(c[0], x[2], x[3]);
  return add2(c[1], t0, t1);
}

// the digits from weight four on: c += 4 (f0 + f1)
template <int S>
__device__ __forceinline__ void carry8(uint64_t (&c)[S], uint64_t f0, uint64_t f1) {
  uint64_t k = add2(c[2], f0, f1);
#pragma unroll
  for (int s = 3; s < S; ++s) {
    const uint64_t n = c[s] & k;
    c[s] ^= k;
    k = n;
  }
}

// c += x[0] + .. + x[7]
template <int S>
__device__ __forceinline__ void add8(uint64_t (&c)[S], const uint64_t (&x)[8]) {
  const uint64_t lo[4] = {x[0], x[1], x[2], x[3]}, hi[4] = {x[4], x[5], x[6], x[7]};
  const uint64_t f0 = add4(c, lo), f1 = add4(c, hi);
  carry8(c, f0, f1);
}

// The warp total of one counter set, one integer per replica times weight, added
// to acc (shared memory, word position major).  Lanes of the same position are V
// apart.
template <int V, int S>
__device__ __forceinline__ void reduce(const uint64_t (&c)[S], unsigned int* acc,
                                       unsigned int weight = 1u) {
  constexpr int kWide = S + 5;  // digits after summing 32 lanes
  const int lane = threadIdx.x & 31;
  const bool upper = lane & 16;
  uint32_t w[kWide];
  uint32_t carry = 0;
  // lanes 0-15 go on with replicas 0-31 of both lanes, lanes 16-31 with 32-63
#pragma unroll
  for (int s = 0; s < S; ++s) {
    const uint32_t lo = (uint32_t)c[s], hi = (uint32_t)(c[s] >> 32);
    const uint32_t o = __shfl_xor_sync(0xffffffffu, upper ? lo : hi, 16), m = upper ? hi : lo;
    w[s] = m ^ o ^ carry;
    carry = (m & o) | (carry & (m | o));
  }
  w[S] = carry;
  int wide = S + 1;
#pragma unroll
  for (int off = 8; off >= V; off >>= 1) {
    carry = 0;
#pragma unroll
    for (int s = 0; s < kWide; ++s) {
      if (s < wide) {
        const uint32_t o = __shfl_xor_sync(0xffffffffu, w[s], off), m = w[s];
        w[s] = m ^ o ^ carry;
        carry = (m & o) | (carry & (m | o));
      }
    }
    w[wide++] = carry;
  }
  // lanes hh and 16 + hh hold the totals of word position hh
#pragma unroll
  for (int hh = 0; hh < V; ++hh)
#pragma unroll
    for (int half = 0; half < 2; ++half) {
      unsigned int v = 0;
#pragma unroll
      for (int s = 0; s < kWide; ++s)
        if (s < wide) v |= ((__shfl_sync(0xffffffffu, w[s], 16 * half + hh) >> lane) & 1u) << s;
      if (v) atomicAdd(&acc[hh * 64 + 32 * half + lane], v * weight);
    }
}

}  // namespace
}  // namespace ka

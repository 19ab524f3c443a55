// Fixed-point numbers of up to 63 bits for the setup's sums: a double becomes an integer relative to a power of
// two, an integer a pair of words whose products are summed by 32 x 32 + 64 bit multiply-adds (a sixteenth of the
// time of an FP64 one).
#pragma once

#include "amg_internal.cuh"

namespace amgfix {

// (-1)^neg v 2^(BITS - e) cut to an integer, for |v| < 2^e, BITS <= 63; neg: the sign bit's mask
template <int BITS>
__device__ __forceinline__ long long fixed(double v, int e, int neg = 0) {
  const int hi = __double2hiint(v), lo = __double2loint(v), f = (hi >> 20) & 0x7FF;
  const unsigned mh = (((unsigned)hi << 10) & 0x3FFFFFFFu) | 0x40000000u | (unsigned)lo >> 22;  // mantissa 2^10
  const unsigned long long m = (unsigned long long)mh << 32 | (unsigned)lo << 10;
  const long long x = (long long)(m >> min(1085 - BITS + e - f, 63)), s = (hi ^ neg) >> 31;
  return (x ^ s) - s;
}
// words of x = h 2^31 + l, |l| <= 2^30
__device__ __forceinline__ int2 words31(long long x) {
  x += 1 << 30;
  return make_int2((int)(x >> 31), (int)((unsigned)x & 0x7FFFFFFFu) - (1 << 30));
}
__device__ __forceinline__ long long joined(int2 w) { return ((long long)w.x << 31) + w.y; }
__device__ __forceinline__ int2 minus(int2 w) { return make_int2(-w.x, -w.y); }
// h 2^62 + l 2^31 += a b without the product of the low words
__device__ __forceinline__ void mac(long long& h, long long& l, int2 a, int2 b) {
  h += (long long)a.x * b.x;
  l += (long long)a.x * b.y;
  l += (long long)a.y * b.x;
}

}  // namespace amgfix

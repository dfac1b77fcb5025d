// detsum.cuh -- sums of non-negative floating-point values across a warp in integer arithmetic
// (internal). A double-precision add takes 64 cycles on this part (one warp, measured; a five-step
// butterfly with its shuffles about 570), and the sum of c^{i+1} sits on the critical path of
// every iteration of a single-instance solve. Here the lanes agree on the largest exponent, shift
// their significands to it and add them as integers (redux.sync on limbs): no FP64 instruction,
// and a result that does not depend on the order of the lanes. What the shifts cut off of a summand is
// below 2^-53 of the largest value's leading bit for floats (limbs.cuh), 2^-57 for doubles and for the
// sums of warps: no more than a double addition may round off, and nothing where the values are within
// 2^30 of each other.
#pragma once
#include <cuda_runtime.h>

#include "limbs.cuh"

namespace pimpc {
namespace detsum {

constexpr int kSpecial = 1 << 20;   // exponent of infinity (sig 0) and NaN (sig 1)
constexpr int kZero = -(1 << 20);   // exponent of zero
constexpr int kBias = 1080;

// A non-negative value sig 2^(e - kBias).
struct Fx {
  unsigned long long sig;
  int e;
};

__device__ __forceinline__ Fx special_sum(Fx t) {
  return Fx{__any_sync(0xffffffffu, t.e == kSpecial && t.sig != 0) ? 1ull : 0ull, kSpecial};
}

// Sum over the warp of one float per lane (the same Fx in every lane).
__device__ __forceinline__ Fx warp_sum(float v) {
  const unsigned b = __float_as_uint(v) & 0x7fffffffu;
  const int x = (int)(b >> 23);
  const unsigned m = b & 0x7fffffu;
  const int e = x == 0xff ? 1 << 10 : (x ? x : 1);
  const int em = __reduce_max_sync(0xffffffffu, e);
  if (em == 1 << 10) return special_sum(Fx{m ? 1ull : 0ull, x == 0xff ? kSpecial : 0});
  const Limbs q = split(x ? m | 0x800000u : m, em - e);
  const unsigned l0 = __reduce_add_sync(0xffffffffu, q.lo);
  const unsigned l1 = __reduce_add_sync(0xffffffffu, q.hi);
  return Fx{join(l0, l1), exponent(em) + kBias};
}

__device__ __forceinline__ Fx add_limbs(unsigned long long q, int e) {
  const unsigned l0 = __reduce_add_sync(0xffffffffu, (unsigned)q & 0x3fffffu);
  const unsigned l1 = __reduce_add_sync(0xffffffffu, (unsigned)(q >> 22) & 0x3fffffu);
  const unsigned l2 = __reduce_add_sync(0xffffffffu, (unsigned)(q >> 44));
  return Fx{(unsigned long long)l0 + ((unsigned long long)l1 << 22) + ((unsigned long long)l2 << 44),
            e};
}

// Sum over the warp of one double per lane.
__device__ __forceinline__ Fx warp_sum(double v) {
  const unsigned long long b = (unsigned long long)__double_as_longlong(v) & 0x7fffffffffffffffull;
  const int x = (int)(b >> 52);
  const unsigned long long m = b & 0xfffffffffffffull;
  const int e = x == 0x7ff ? 1 << 12 : (x ? x : 1);
  const int em = __reduce_max_sync(0xffffffffu, e);
  if (em == 1 << 12) return special_sum(Fx{m ? 1ull : 0ull, x == 0x7ff ? kSpecial : 0});
  const int sh = em - e;
  const unsigned long long q = sh < 64 ? ((x ? m | (1ull << 52) : m) << 5) >> sh : 0ull;
  return add_limbs(q, em - 1080 + kBias);  // v = m 2^(x - 1075), q = m 2^5
}

// Sum over the warp of one Fx per lane ({0, kZero} where a lane has none).
__device__ __forceinline__ Fx warp_sum(Fx t) {
  if (t.e != kSpecial) {
    if (t.sig == 0) {
      t.e = kZero;
    } else {
      const int lz = __clzll((long long)t.sig);
      t.sig <<= lz;
      t.e -= lz;
    }
  }
  const int em = __reduce_max_sync(0xffffffffu, t.e);
  if (em == kSpecial) return special_sum(t);
  const int sh = em - t.e;
  return add_limbs(sh < 57 ? (t.sig >> 6) >> sh : 0ull, em + 6);
}

__device__ __forceinline__ double to_double(Fx t) {
  if (t.e == kSpecial)
    return __longlong_as_double(t.sig ? 0x7ff8000000000000ll : 0x7ff0000000000000ll);
  if (t.sig == 0) return 0.0;
  // normalise to bit 63, round to nearest (ties away) at 53 bits
  const int lz = __clzll((long long)t.sig);
  const unsigned long long m = t.sig << lz;
  const int ef = t.e - kBias + 63 - lz + 1023;  // biased exponent
  if (ef <= 0) {                                // below the normal range: truncate
    const int sh = 12 - ef;
    return __longlong_as_double((long long)(sh < 64 ? m >> sh : 0ull));
  }
  const unsigned long long r = (m >> 11) + ((m >> 10) & 1ull);  // may carry into the exponent
  const unsigned long long bits = ((unsigned long long)ef << 52) + (r - (1ull << 52));
  return __longlong_as_double((long long)(bits < 0x7ff0000000000000ull ? bits : 0x7ff0000000000000ull));
}

// a <= b for a >= 0 (not NaN) and any b but -0 and NaN: bit patterns of non-negative doubles are
// ordered, and a negative b compares below all of them.
__device__ __forceinline__ bool le_nonneg(double a, double b) {
  return __double_as_longlong(a) <= __double_as_longlong(b);
}

__device__ __forceinline__ bool finite(double v) {
  return ((unsigned)__double2hiint(v) & 0x7ff00000u) != 0x7ff00000u;
}

__device__ __forceinline__ bool finite(float v) {
  return (__float_as_uint(v) & 0x7f800000u) != 0x7f800000u;
}

// Whether a sum of squares of differences of such values may leave the finite range (NaN and infinity
// included): some magnitude of 2^59 (FP32) or 2^500 (FP64) and more.
__device__ __forceinline__ bool large(double a, double b, double c, double d) {
  const unsigned m = max(max((unsigned)__double2hiint(a) & 0x7ff00000u, (unsigned)__double2hiint(b) & 0x7ff00000u),
                         max((unsigned)__double2hiint(c) & 0x7ff00000u, (unsigned)__double2hiint(d) & 0x7ff00000u));
  return m >= (1023u + 500u) << 20;
}
__device__ __forceinline__ bool large(float a, float b, float c, float d) {
  const unsigned m = max(max(__float_as_uint(a) & 0x7f800000u, __float_as_uint(b) & 0x7f800000u),
                         max(__float_as_uint(c) & 0x7f800000u, __float_as_uint(d) & 0x7f800000u));
  return m >= (127u + 59u) << 23;
}

}  // namespace detsum
}  // namespace pimpc

// detsum.cuh -- sums of non-negative floating-point values across a warp in integer arithmetic
// (internal). A double-precision add takes 64 cycles on this part (one warp, measured; a
// five-step butterfly with its shuffles about 570), and the sum of c^{i+1} sits on the critical
// path of every iteration of a single-instance solve. Here the lanes agree on the largest
// exponent, shift their significands to it and add them as integers (redux.sync on 22-bit limbs):
// no FP64 instruction, and a result that does not depend on the order of the lanes. What is cut
// off by the shifts is at most 2^-55 of the largest value per summand, below the rounding of a
// chain of double additions.
#pragma once
#include <cuda_runtime.h>

namespace pimpc {
namespace detsum {

// A non-negative value as significand and exponent: v = sig 2^e up to a constant of the format.
// Infinities and NaN carry e = kSpecial, with sig = 0 for infinity.
constexpr int kSpecial = 1 << 20;

struct Term {
  unsigned long long sig;  // 53 significant bits at most
  int e;
};

__device__ __forceinline__ Term term(double v) {
  const unsigned long long b = (unsigned long long)__double_as_longlong(v);
  const int e = (int)(b >> 52) & 0x7ff;
  const unsigned long long m = b & 0xfffffffffffffull;
  Term t;
  t.sig = e ? (e == 0x7ff ? (m ? 1ull : 0ull) : (m | (1ull << 52))) : m;
  t.e = e == 0x7ff ? kSpecial : (e ? e : 1);
  return t;
}

// A float, in the scale of the doubles: its 24-bit significand moved up by 29 bits.
__device__ __forceinline__ Term term(float v) {
  const unsigned b = __float_as_uint(v);
  const int e = (int)(b >> 23) & 0xff;
  const unsigned m = b & 0x7fffffu;
  Term t;
  t.sig = e == 0xff ? (m ? 1ull : 0ull) : ((unsigned long long)(e ? (m | 0x800000u) : m) << 29);
  t.e = e == 0xff ? kSpecial : (e ? e : 1) + 1023 - 127;
  return t;
}

// The sum over the warp of every lane's cnt terms (cnt <= kMax <= 4, compile-time unrolled), the
// same double in every lane.
template <int kMax>
__device__ __forceinline__ double warp_sum(const Term (&t)[kMax]) {
  int e = t[0].e;
#pragma unroll
  for (int i = 1; i < kMax; ++i) e = max(e, t[i].e);
  const int em = (int)__reduce_max_sync(0xffffffffu, (unsigned)e);
  if (em == kSpecial) {
    bool nan = false;
#pragma unroll
    for (int i = 0; i < kMax; ++i) nan |= t[i].e == kSpecial && t[i].sig != 0;
    return __any_sync(0xffffffffu, nan) ? __longlong_as_double(0x7ff8000000000000ll)
                                        : __longlong_as_double(0x7ff0000000000000ll);
  }
  unsigned l0 = 0, l1 = 0, l2 = 0;
#pragma unroll
  for (int i = 0; i < kMax; ++i) {
    const int sh = em - t[i].e;
    const unsigned long long q = sh < 64 ? (t[i].sig << 3) >> sh : 0ull;
    l0 += (unsigned)q & 0x3fffffu;
    l1 += (unsigned)(q >> 22) & 0x3fffffu;
    l2 += (unsigned)(q >> 44);
  }
  l0 = __reduce_add_sync(0xffffffffu, l0);
  l1 = __reduce_add_sync(0xffffffffu, l1);
  l2 = __reduce_add_sync(0xffffffffu, l2);
  // 56-bit terms, at most 128 of them: the total fits 63 bits
  const unsigned long long tot =
      (unsigned long long)l0 + ((unsigned long long)l1 << 22) + ((unsigned long long)l2 << 44);
  if (tot == 0) return 0.0;
  // normalise to bit 63, round to nearest (ties away) at 53 bits
  const int lz = __clzll((long long)tot);
  const unsigned long long m = tot << lz;
  const int ef = em - 3 + 11 - lz;  // biased exponent of the result
  if (ef <= 0) {                    // below the normal range: truncate
    const int sh = 12 - ef;
    return __longlong_as_double((long long)(sh < 64 ? m >> sh : 0ull));
  }
  const unsigned long long r = (m >> 11) + ((m >> 10) & 1ull);  // may carry into the exponent
  const unsigned long long bits = ((unsigned long long)ef << 52) + (r - (1ull << 52));
  if (bits >= 0x7ff0000000000000ull) return __longlong_as_double(0x7ff0000000000000ll);
  return __longlong_as_double((long long)bits);
}

template <typename T>
__device__ __forceinline__ double warp_sum1(T v) {
  const Term t[1] = {term(v)};
  return warp_sum<1>(t);
}

// a <= b for doubles that are non-negative or whose right side may be negative (eps < 0 never
// holds); both not NaN. Integer comparison: the bit patterns of non-negative doubles are ordered.
__device__ __forceinline__ bool le_nonneg(double a, double b) {
  return __double_as_longlong(a) <= __double_as_longlong(b);
}

__device__ __forceinline__ bool finite(double v) {
  return ((unsigned)__double2hiint(v) & 0x7ff00000u) != 0x7ff00000u;
}

}  // namespace detsum
}  // namespace pimpc

// limbs.cuh -- the integer form in which detsum.cuh adds the floats of a warp (internal; host-callable,
// so that it is checked on the CPU).
#pragma once

#if defined(__CUDACC__)
#define PIMPC_HD __host__ __device__ __forceinline__
#else
#define PIMPC_HD inline
#endif

namespace pimpc {
namespace detsum {

// Two 27-bit limbs of a non-negative finite float with the 24-bit significand sig, whose exponent is
// `below` under the warp's largest, in units of 2^-53 of that one's leading bit: 24 bits with 30 below
// them; what lies below the unit is cut off. 27 bits, so that the sum of 32 lanes fits 32.
struct Limbs {
  unsigned lo, hi;
};
constexpr unsigned kLimb = (1u << 27) - 1u;

PIMPC_HD Limbs split(unsigned sig, int below) {
  const unsigned long long q = below < 64 ? ((unsigned long long)sig << 30) >> below : 0ull;
  return Limbs{(unsigned)q & kLimb, (unsigned)(q >> 27)};
}

// The sum of the limbs' sums as sig 2^e, em the largest exponent field (at least 1): a significand is
// sig 2^(field - 150), a limb pair sig 2^30.
PIMPC_HD unsigned long long join(unsigned lo, unsigned hi) {
  return (unsigned long long)lo + ((unsigned long long)hi << 27);
}
PIMPC_HD int exponent(int em) { return em - 180; }

}  // namespace detsum
}  // namespace pimpc

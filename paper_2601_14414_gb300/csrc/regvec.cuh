// regvec.cuh -- products of a register-resident matrix row with a vector in shared memory, x / 3 and
// the clamp, as the kernels that count FP64 instructions use them (internal).
#pragma once
#include <cuda_runtime.h>

namespace pimpc {

// Elements of a vector of n in shared memory: whole 16-byte pieces.
__host__ __device__ inline int reg_nv(int n, int tsize) {
  const int w = tsize == 4 ? 4 : 2;
  return (n + w - 1) / w * w;
}

// init + sum_j m[j] v[j] over j < cnt, v in shared memory (16-byte aligned, zero-padded to whole
// vectors), m in registers with zeros beyond its length. FP64 runs one chain: a warp issues an
// FP64 instruction every 64 cycles, which is also its latency, so a second chain gains nothing.
template <int NM>
__device__ __forceinline__ float dot(const float (&m)[NM], const float *v, int cnt, float init) {
  float a0 = init, a1 = 0.0f, a2 = 0.0f, a3 = 0.0f;
#pragma unroll
  for (int j = 0; j < NM; j += 4)
    if (j < cnt) {
      const float4 q = *reinterpret_cast<const float4 *>(v + j);
      a0 = fmaf(m[j], q.x, a0);
      a1 = fmaf(m[j + 1], q.y, a1);
      a2 = fmaf(m[j + 2], q.z, a2);
      a3 = fmaf(m[j + 3], q.w, a3);
    }
  return (a0 + a1) + (a2 + a3);
}
template <int NM>
__device__ __forceinline__ double dot(const double (&m)[NM], const double *v, int cnt, double init) {
  double a = init;
#pragma unroll
  for (int j = 0; j < NM; j += 2)
    if (j < cnt) {
      const double2 q = *reinterpret_cast<const double2 *>(v + j);
      a = fma(m[j], q.x, a);
      a = fma(m[j + 1], q.y, a);
    }
  return a;
}

// x / 3 to within a rounding of the correctly rounded quotient: 1/3 as the sum of its value rounded
// down and the rounding of what is left (two operations instead of a division; both parts are
// positive, so that infinities pass).
__device__ __forceinline__ float third(float x) {
  constexpr float hi = 0x1.555554p-2f;
  constexpr float lo = (float)(1.0 / 3.0 - (double)hi);
  return fmaf(x, hi, x * lo);
}
__device__ __forceinline__ double third(double x) {
  constexpr double hi = 1.0 / 3.0;         // (1 - 2^-54) / 3
  constexpr double lo = hi * 0x1p-54;      // 1/3 - hi = 2^-54 / 3
  return fma(x, hi, x * lo);
}

// min(max(w, lo), hi), NaN passing through. FP64 by the order of the bit patterns: two FP64
// comparisons would cost 128 cycles.
__device__ __forceinline__ float clamp(float w, float lo, float hi) {
  return w < lo ? lo : (w > hi ? hi : w);
}
__device__ __forceinline__ long long order_key(double v) {
  const long long b = __double_as_longlong(v);
  return b ^ ((b >> 63) & 0x7fffffffffffffffll);
}
__device__ __forceinline__ double clamp(double w, double lo, double hi) {
  const long long k = order_key(w);
  const bool nan = (__double_as_longlong(w) & 0x7fffffffffffffffll) > 0x7ff0000000000000ll;
  const double z = k < order_key(lo) ? lo : (k > order_key(hi) ? hi : w);
  return nan ? w : z;
}

// Steps 2-3 of one component in the reduced form (lambda = -beta): xb = xbar, bd = Bbar du, ax = Abar xbar
// + ebar, th and b the duals' hats. gamma = bd + beta - ax + lambda is bd - ax, without the duals. Summed
// as (beta + bd) - (beta + ax), one operation fewer where beta starts ax's dot product, it carries beta's
// rounding into v: the rms error of x against FP64 then is 1.25 times that of the unreduced iteration
// for the cart-poles (FP32 and FP64 alike), and 0.73 and 0.94 times so.
template <typename T>
struct Step {
  T w, z, v, t, b;
};
template <typename T>
__device__ __forceinline__ Step<T> steps23(T xb, T bd, T ax, T th, T b, T lo, T hi) {
  Step<T> r;
  const T s = xb + th;
  r.w = third((T)2 * (s + b) + (bd + ax));
  r.z = clamp(r.w, lo, hi);
  r.v = (T)0.5 * (r.z + (bd - ax));
  r.t = s - r.z;
  r.b = b + (bd - r.v);  // bd - v enters the share of c too
  return r;
}

// -v without an FP64 instruction.
__device__ __forceinline__ double negated(double v) {
  return __hiloint2double(__double2hiint(v) ^ (int)0x80000000, __double2loint(v));
}

}  // namespace pimpc

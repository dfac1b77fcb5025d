// stage_reg.cuh -- one thread per stage with the stage in its registers (internal): FP32 instances of
// few states and inputs, forward (admm_stage.cu) and reverse (adjoint.cu).
//
// Components are ordered x_0 .. x_{NX-1}, u_0 .. u_{NU-1}; padded ones have zero rows and columns and
// bounds of zero, and stay zero. The vectors that stages exchange are rows of ld = threads + 1 floats in
// shared memory: row c of sg holds component c of Abar_k^T y_k at slot k (zero beyond the horizon, where
// threads compute but do not store), row c of sx that of xbar_{k+1} at slot k + 1 and of xbar_0 at slot 0.
#pragma once
#include <cuda_runtime.h>

#include "regvec.cuh"

namespace pimpc {
namespace stage {

// Sizes served (kStageThreads stages): padded to 2 + 1, 4 + 1 or 4 + 2 components.
inline int size_class(int nx, int nu) { return nx > 4 || nu > 2 ? -1 : nu <= 1 ? (nx <= 2 ? 0 : 1) : 2; }
inline int padded(int cls) { return cls == 0 ? 3 : cls == 1 ? 5 : 6; }

// The instance's component of a padded one, -1 for none.
template <int NX, int NU>
__device__ __forceinline__ int component(int p, int nx, int nu) {
  return p < NX ? (p < nx ? p : -1) : (p - NX < nu ? nx + p - NX : -1);
}

template <int NX, int NU>
struct Mats {
  static constexpr int NN = NX + NU, NT = NN * (NN + 1) / 2;
  float G[NX][NN];     // [A | B]
  float H[NT], P[NT];  // lower triangles, row by row; P = Bbar M Bbar^T
  float rho;

  static __device__ __forceinline__ constexpr int tri(int r, int c) {
    return r >= c ? r * (r + 1) / 2 + c : c * (c + 1) / 2 + r;
  }

  // g(r, c) of [A | B], h(r, c) of H_k, m(q, i) of M_k, by the instance's own components.
  template <typename FG, typename FH, typename FM>
  __device__ __forceinline__ void setup(int nx, int nu, bool on, float rho_, FG g, FH h, FM m) {
    rho = rho_;
    auto comp = [&](int p) { return on ? component<NX, NU>(p, nx, nu) : -1; };
#pragma unroll
    for (int r = 0; r < NX; ++r)
#pragma unroll
      for (int c = 0; c < NN; ++c) G[r][c] = comp(r) >= 0 && comp(c) >= 0 ? g(r, comp(c)) : 0.0f;
    float J[NU][NN];  // M Bbar^T
#pragma unroll
    for (int q = 0; q < NU; ++q)
#pragma unroll
      for (int c = 0; c < NN; ++c) {
        float s = 0.0f;
#pragma unroll
        for (int i = 0; i < NU; ++i)
          s += (on && q < nu && i < nu ? m(q, i) : 0.0f) * (c < NX ? G[c < NX ? c : 0][NX + i] : (c - NX == i ? 1.0f : 0.0f));
        J[q][c] = s;
      }
#pragma unroll
    for (int r = 0; r < NN; ++r)
#pragma unroll
      for (int c = 0; c <= r; ++c) {
        H[tri(r, c)] = comp(r) >= 0 && comp(c) >= 0 ? h(comp(r), comp(c)) : 0.0f;
        float s = 0.0f;
#pragma unroll
        for (int q = 0; q < NU; ++q) s += (r < NX ? G[r < NX ? r : 0][NX + q] : (r - NX == q ? 1.0f : 0.0f)) * J[q][c];
        P[tri(r, c)] = s;
      }
  }

  // out_r = sum_c S(r, c) x_c, S a packed triangle.
  static __device__ __forceinline__ void sym(const float (&S)[NT], const float (&x)[NN], float (&out)[NN]) {
#pragma unroll
    for (int r = 0; r < NN; ++r) {
      float s = S[tri(r, 0)] * x[0];
#pragma unroll
      for (int c = 1; c < NN; ++c) s = fmaf(S[tri(r, c)], x[c], s);
      out[r] = s;
    }
  }
  // Abar^T y = G^T y_x + (0, y_u), component c.
  __device__ __forceinline__ float abar_t(const float (&y)[NN], int c) const {
    float s = c < NX ? 0.0f : y[c];
#pragma unroll
    for (int r = 0; r < NX; ++r) s = fmaf(G[r][c], y[r], s);
    return s;
  }
  // init + Abar x = init + (G x, x_u), component r.
  __device__ __forceinline__ float abar(const float (&x)[NN], int r, float init) const {
    if (r >= NX) return init + x[r];
#pragma unroll
    for (int c = 0; c < NN; ++c) init = fmaf(G[r < NX ? r : 0][c], x[c], init);
    return init;
  }
};

// A stage's vectors and one plain iteration on them.
template <int NX, int NU>
struct Iter {
  using M = Mats<NX, NU>;
  static constexpr int NN = NX + NU;
  float e[NX], qref[NN], lo[NN], hi[NN], z[NN], v[NN], t[NN], b[NN];

  // ev(r), q(c) = Qbar ref, l(c), h(c) by the instance's own components; the iterate stays.
  template <typename FE, typename FQ, typename FL, typename FH>
  __device__ __forceinline__ void inputs(int nx, int nu, bool on, FE ev, FQ q, FL l, FH h) {
#pragma unroll
    for (int p = 0; p < NN; ++p) {
      const int c = on ? component<NX, NU>(p, nx, nu) : -1;
      if (p < NX) e[p < NX ? p : 0] = c >= 0 ? ev(c) : 0.0f;
      qref[p] = c >= 0 ? q(c) : 0.0f;
      lo[p] = c >= 0 ? l(c) : 0.0f;
      hi[p] = c >= 0 ? h(c) : 0.0f;
    }
  }

  // xb: xbar_{k+1}; kSide: side, bit c set where w_c <= lo_c, bit NN + c where w_c >= hi_c; kShare:
  // share, the stage's share of c / rho (`on`: a stage of the instance), and the iteration is left with true, nothing changed, if `bad`
  // of any thread of the CTA is set.
  template <bool kShare, bool kSide>
  __device__ __forceinline__ bool step(const M &m, float *sg, float *sx, int ld, int k, bool on, bool bad, float (&xb)[NN],
                                       unsigned &side, float &share) {
    float bd[NN];
    {
      float w[NN], y[NN];
#pragma unroll
      for (int c = 0; c < NN; ++c) {
        const float be = c < NX ? b[c] + e[c < NX ? c : 0] : b[c];  // ebar - lambda
        w[c] = v[c] - b[c];
        y[c] = (z[c] - v[c]) - be;
      }
#pragma unroll
      for (int c = 0; c < NN; ++c) {
        const float g = m.abar_t(y, c);
        if (on) sg[c * ld + k] = g;
      }
      M::sym(m.P, w, bd);
    }
    if (kShare) {
      if (__syncthreads_or(bad)) return true;
    } else {
      __syncthreads();
    }
    {
      float h[NN];
#pragma unroll
      for (int c = 0; c < NN; ++c) h[c] = fmaf(m.rho, (z[c] - t[c]) + sg[c * ld + k + 1], qref[c]);
      M::sym(m.H, h, xb);
#pragma unroll
      for (int c = 0; c < NN; ++c) sx[c * ld + k + 1] = xb[c];
    }
    __syncthreads();
    float xp[NN];
#pragma unroll
    for (int c = 0; c < NN; ++c) xp[c] = sx[c * ld + k];
    float g = 0.0f, d = 0.0f;
    side = 0u;
#pragma unroll
    for (int r = 0; r < NN; ++r) {
      const float ax = m.abar(xp, r, r < NX ? e[r < NX ? r : 0] : 0.0f);  // Abar xbar + ebar
      const Step<float> o = steps23(xb[r], bd[r], ax, t[r], b[r], lo[r], hi[r]);
      if (kSide) side |= o.w <= lo[r] ? 1u << r : (o.w >= hi[r] ? 1u << (NN + r) : 0u);
      if (kShare) {  // the duals' differences without their own rounding, as in admm_reg.cuh
        const float d1 = xb[r] - o.z, d2 = bd[r] - o.v, d4 = o.z - z[r], d5 = o.v - v[r];
        g += d2 * d2 + (d4 * d4 + d5 * (d5 - d4));
        d += d1 * d1;
      }
      z[r] = o.z;
      v[r] = o.v;
      t[r] = o.t;
      b[r] = o.b;
    }
    if (kShare) share = on ? 2.0f * g + d : 0.0f;
    return false;
  }
};

}  // namespace stage
}  // namespace pimpc

// admm_stage.cu -- the resident schedule (family 3) with one thread per stage: FP32 instances of
// nx <= 4, nu <= 2 and up to 256 stages, a fixed number of plain iterations.
//
// What bounds a batch of these is instruction issue, and a single one the latency of an iteration.
// With a thread per component (admm_reg.cuh) every component loads each vector that it multiplies
// from shared memory, and a CTA meets four times per iteration. A thread that owns a whole stage of n <= 6 components keeps G_k, the packed lower
// triangles of H_k and P_k = Bbar_k M_k Bbar_k^T and the iterate in registers, multiplies without
// loads, and exchanges two n-vectors with its neighbours: Abar_k^T y_k, formed by the thread that
// holds G_k, to stage k - 1, and xbar_{k+1} to stage k + 1, two barriers in all. The iteration is the
// reduced one of admm_reg.cuh (lambda = -beta throughout). What limits the warps of an SM is the
// registers of a thread: 72 at 2 + 1 components, 128 at 4 + 1, 178 at 4 + 2.
// Per solve of 150 iterations, against a thread per component: 1024 instances of n 5, N 100 629 -> 234
// us, N 20 139 -> 86, N 150 (more components than a CTA has threads: clusters of two CTAs) 3.68 -> 0.34
// ms; 153 instances of N 100 176 -> 87; one instance of n 5, N 60 82 -> 62, N 256 160 -> 90; n 3, N 20
// 59 -> 33; slower by 4 % at most (n 5, one stage, 53 -> 55), so that the batch does not matter.
#include <math.h>

#include "detsum.cuh"
#include "lockstep.cuh"
#include "regvec.cuh"

namespace pimpc {

namespace {

using Args = ls::Args<float>;

__device__ __forceinline__ float wrapped_at(const float *Wp, int m, int r, int c) {
  int d = c - r;
  if (d < 0) d += m;
  return (2 * d <= m) ? Wp[d * m + r] : Wp[(m - d) * m + c];
}

// Components are ordered x_0 .. x_{NX-1}, u_0 .. u_{NU-1}; padded ones have zero rows and columns and
// bounds of zero, and stay zero.
template <int NX, int NU>
struct Stage {
  static constexpr int NN = NX + NU, NT = NN * (NN + 1) / 2;
  float G[NX][NN];  // [A | B]
  float H[NT], P[NT];  // lower triangles, row by row
  float e[NX], qref[NN], lo[NN], hi[NN], rho;
  float z[NN], v[NN], t[NN], b[NN];
  bool on, more;  // a stage of the instance; one with a successor

  static __device__ __forceinline__ constexpr int tri(int r, int c) {
    return r >= c ? r * (r + 1) / 2 + c : c * (c + 1) / 2 + r;
  }

  __device__ __forceinline__ void setup(const Args &a, int warm, int j, int k) {
    const int nx = a.L.nx[j], nu = a.L.nu[j], n = nx + nu, N = a.L.N[j];
    on = k < N;
    more = k + 1 < N;
    rho = (float)a.rho;
    const int lti = a.L.lti, W = a.L.W[j], ldg = odd_ld(n);
    const int oE = nx * ldg, oH = oE + nx, oM = oH + wrapped_size(n);
    const float *blk = a.blk + a.L.blk[j];
    const float *Gk = blk + (lti || !on ? 0 : (int64_t)k * W);
    const float *Hk = (lti ? blk + (more ? 0 : W) : Gk) + oH, *M = Gk + oM;
    const float *ref = a.ref ? a.ref + (a.ref_per_stage ? a.L.Nn[j] + (int64_t)(on ? k : 0) * n : a.L.off_n[j]) : nullptr;
    const float *git = a.it[a.base[j]] + a.L.Ni[j] +
                       (int64_t)(on ? (warm == 2 && more ? k + 1 : k) : 0) * ls::iter_stride_plain(n, 4);
    // the instance's component of a padded one, -1 for none
    auto comp = [&](int p) { return !on ? -1 : p < NX ? (p < nx ? p : -1) : (p - NX < nu ? nx + p - NX : -1); };
#pragma unroll
    for (int p = 0; p < NN; ++p) {
      const int c = comp(p);
      z[p] = v[p] = t[p] = b[p] = qref[p] = lo[p] = hi[p] = 0.0f;
      if (c < 0) continue;
      lo[p] = a.lo[a.L.off_n[j] + c];
      hi[p] = a.hi[a.L.off_n[j] + c];
      if (ref) qref[p] = a.qd[a.L.off_n[j] + c] * ref[c];
      if (warm != 0) {  // the previous solve's iterate, shifted by a stage for warm == 2
        z[p] = git[c];
        v[p] = git[n + c];
        t[p] = git[2 * n + c];
        b[p] = git[3 * n + c];
      }
    }
#pragma unroll
    for (int r = 0; r < NX; ++r) {
      e[r] = on && r < nx ? Gk[oE + r] : 0.0f;
#pragma unroll
      for (int c = 0; c < NN; ++c) G[r][c] = r < nx && comp(c) >= 0 ? Gk[r * ldg + comp(c)] : 0.0f;
    }
    float J[NU][NN];  // M Bbar^T
#pragma unroll
    for (int q = 0; q < NU; ++q)
#pragma unroll
      for (int c = 0; c < NN; ++c) {
        float s = 0.0f;
#pragma unroll
        for (int i = 0; i < NU; ++i)
          s += (on && q < nu && i < nu ? wrapped_at(M, nu, q, i) : 0.0f) *
               (c < NX ? G[c < NX ? c : 0][NX + i] : (c - NX == i ? 1.0f : 0.0f));
        J[q][c] = s;
      }
#pragma unroll
    for (int r = 0; r < NN; ++r)
#pragma unroll
      for (int c = 0; c <= r; ++c) {
        H[tri(r, c)] = comp(r) >= 0 && comp(c) >= 0 ? wrapped_at(Hk, n, comp(r), comp(c)) : 0.0f;
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

  // One plain iteration; share: the stage's share of c / rho. sg, sx: NN rows of ld floats (ld threads);
  // x0: xbar_0 (stage 0's). True, and no more than that, if `bad` of any thread says that the iteration
  // before was the last.
  __device__ __forceinline__ bool iterate(float *sg, float *sx, int ld, int k, const float (&x0)[NN], bool bad,
                                          float &share) {
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
      for (int c = 0; c < NN; ++c) {  // Abar^T y
        float s = c < NX ? 0.0f : y[c];
#pragma unroll
        for (int r = 0; r < NX; ++r) s = fmaf(G[r][c], y[r], s);
        sg[c * ld + k] = s;
      }
      sym(P, w, bd);
    }
    if (__syncthreads_or(bad)) return true;
    float xb[NN];
    {
      float h[NN];
#pragma unroll
      for (int c = 0; c < NN; ++c)
        h[c] = fmaf(rho, (z[c] - t[c]) + (more ? sg[c * ld + k + 1] : 0.0f), qref[c]);
      sym(H, h, xb);
#pragma unroll
      for (int c = 0; c < NN; ++c) sx[c * ld + k] = xb[c];
    }
    __syncthreads();
    float xp[NN];
#pragma unroll
    for (int c = 0; c < NN; ++c) xp[c] = k > 0 ? sx[c * ld + k - 1] : x0[c];
    float g = 0.0f, d = 0.0f;
#pragma unroll
    for (int r = 0; r < NN; ++r) {
      float q = r < NX ? b[r] + e[r < NX ? r : 0] : b[r] + xp[r];  // Abar xbar + ebar - lambda
      if (r < NX) {
#pragma unroll
        for (int c = 0; c < NN; ++c) q = fmaf(G[r < NX ? r : 0][c], xp[c], q);
      }
      const float s = xb[r] + t[r], p = b[r] + bd[r];
      const float w = third(2.0f * s + (p + q));
      const float zn = clamp(w, lo[r], hi[r]);
      const float vn = 0.5f * (zn + (p - q));
      // the duals' differences without their own rounding, as in admm_reg.cuh
      const float d1 = xb[r] - zn, d2 = bd[r] - vn, d4 = zn - z[r], d5 = vn - v[r];
      g += d2 * d2 + (d4 * d4 + d5 * (d5 - d4));
      d += d1 * d1;
      z[r] = zn;
      v[r] = vn;
      t[r] = s - zn;
      b[r] = p - vn;
    }
    share = on ? 2.0f * g + d : 0.0f;
    return false;
  }
};

template <int NX, int NU, int kMinCtas>
__global__ void __launch_bounds__(kStageThreads, kMinCtas)
    stage_kernel(Args a, int warm, double *u_out, double *x_out) {
  using S = Stage<NX, NU>;
  constexpr int NN = S::NN;
  extern __shared__ float vecs[];  // two vectors per stage, and one past the last
  __shared__ ulonglong2 sums[kStageThreads / 32];
  const int j = blockIdx.x, k = threadIdx.x, ld = blockDim.x;
  const int nx = a.L.nx[j], nu = a.L.nu[j], n = nx + nu;
  float *sg = vecs, *sx = vecs + NN * ld;
  S s;
  s.setup(a, warm, j, k);
  float x0[NN];
#pragma unroll
  for (int p = 0; p < NN; ++p) {
    const int c = p < NX ? (p < nx ? p : -1) : (p - NX < nu ? nx + p - NX : -1);
    x0[p] = k == 0 && c >= 0 ? a.xb0[a.L.off_n[j] + c] : 0.0f;
  }
  float share = 0.0f;
  int iters = 0;
  for (; iters < a.max_iters; ++iters)
    if (s.iterate(sg, sx, ld, k, x0, !detsum::finite(share), share)) break;
  // c^{i+1} of the last iteration, independent of the order of its shares
  const int lane = k & 31, warp = k >> 5;
  detsum::Fx sum = detsum::warp_sum(share);
  if (lane == 0) sums[warp] = make_ulonglong2(sum.sig, (unsigned long long)(long long)sum.e);
  __syncthreads();
  if (warp == 0) {
    sum = lane < ld / 32 ? detsum::Fx{sums[lane].x, (int)sums[lane].y} : detsum::Fx{0ull, detsum::kZero};
    sum = detsum::warp_sum(sum);
    if (lane == 0) {
      const double cn = detsum::to_double(sum);
      InstState o;
      o.c = a.rho == 1.0 ? cn : cn * a.rho;
      o.iters = iters;
      o.status = a.ferr && a.ferr[j] ? kFactorFailed : detsum::finite(o.c) ? kMaxIter : kNonFinite;
      o.momentum = 0;
      o.pad = 0;
      a.st[j] = o;
      a.stop[j] = 1;
    }
  }
  if (!s.on) return;
  float *git = a.it[a.base[j]] + a.L.Ni[j] + (int64_t)k * ls::iter_stride_plain(n, 4);
#pragma unroll
  for (int p = 0; p < NN; ++p) {
    const int c = p < NX ? (p < nx ? p : -1) : (p - NX < nu ? nx + p - NX : -1);
    if (c < 0) continue;
    git[c] = s.z[p];
    git[n + c] = s.v[p];
    git[2 * n + c] = s.t[p];
    git[3 * n + c] = s.b[p];
    git[4 * n + c] = -s.b[p];
    if (c < nx) {
      if (x_out) x_out[a.L.Nnx[j] + (int64_t)k * nx + c] = (double)s.z[p];
    } else if (u_out) {
      u_out[a.L.Nnu[j] + (int64_t)k * nu + (c - nx)] = (double)s.z[p];
    }
  }
}

}  // namespace

cudaError_t launch_stage(const AdmmLaunch &s, int size_class, int threads, cudaStream_t stream) {
  const Args a = ls::make_args<float>(s);
  const int nn = size_class == 0 ? 3 : size_class == 1 ? 5 : 6;
  const size_t smem = sizeof(float) * 2 * nn * threads;
  auto kernel = size_class == 0 ? stage_kernel<2, 1, 3> : size_class == 1 ? stage_kernel<4, 1, 2> : stage_kernel<4, 2, 1>;
  kernel<<<s.L.batch, threads, smem, stream>>>(a, s.warm, s.u_out, s.x_out);
  return cudaGetLastError();
}

}  // namespace pimpc

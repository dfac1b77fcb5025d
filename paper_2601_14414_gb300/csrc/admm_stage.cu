// admm_stage.cu -- the resident schedule (family 3) with one thread per stage: FP32 instances of
// nx <= 4, nu <= 2 and up to 256 stages, a fixed number of plain iterations.
//
// What bounds a batch of these is instruction issue, and a single one the latency of an iteration.
// With a thread per component (admm_reg.cuh) every component loads each vector that it multiplies
// from shared memory, and a CTA meets four times per iteration. A thread that owns a whole stage of
// n <= 6 components keeps G_k, the packed lower triangles of H_k and P_k = Bbar_k M_k Bbar_k^T and the
// iterate in registers, multiplies without loads, and exchanges two n-vectors with its neighbours:
// Abar_k^T y_k, formed by the thread that holds G_k, to stage k - 1, and xbar_{k+1} to stage k + 1, two
// barriers in all. The iteration is the reduced one of admm_reg.cuh (lambda = -beta throughout). What limits the warps of an SM is the
// registers of a thread: 69 at 2 + 1 components, 125 at 4 + 1, 167 at 4 + 2.
// Per solve of 150 iterations, against a thread per component: 1024 instances of n 5, N 100 629 -> 217
// us, N 20 139 -> 76, N 150 (more components than a CTA has threads: clusters of two CTAs) 3.68 -> 0.32
// ms; 153 instances of N 100 176 -> 76; one instance of n 5, N 60 82 -> 55, N 256 160 -> 79; n 3, N 20
// 59 -> 37; slower by 4 % at most (n 5, one stage, 53 -> 55), so that the batch does not matter.
#include <math.h>

#include "detsum.cuh"
#include "lockstep.cuh"
#include "stage_reg.cuh"

namespace pimpc {

namespace {

using Args = ls::Args<float>;

__device__ __forceinline__ float wrapped_at(const float *Wp, int m, int r, int c) {
  int d = c - r;
  if (d < 0) d += m;
  return (2 * d <= m) ? Wp[d * m + r] : Wp[(m - d) * m + c];
}

template <int NX, int NU, int kMinCtas>
__global__ void __launch_bounds__(kStageThreads, kMinCtas)
    stage_kernel(Args a, int warm, double *u_out, double *x_out) {
  constexpr int NN = NX + NU;
  extern __shared__ float vecs[];  // sg, sx
  __shared__ ulonglong2 sums[kStageThreads / 32];
  const int j = blockIdx.x, k = threadIdx.x, ld = blockDim.x + 1;
  const int nx = a.L.nx[j], nu = a.L.nu[j], n = nx + nu, N = a.L.N[j], in = a.L.off_n[j];
  float *sg = vecs, *sx = vecs + NN * ld;
  const bool on = k < N;
  stage::Mats<NX, NU> m;
  stage::Iter<NX, NU> s;
  {
    const int lti = a.L.lti, W = a.L.W[j], ldg = odd_ld(n), ks = on ? k : 0;
    const int oE = nx * ldg, oH = oE + nx, oM = oH + wrapped_size(n);
    const float *blk = a.blk + a.L.blk[j];
    const float *Gk = blk + (lti ? 0 : (int64_t)ks * W);
    const float *Hk = (lti ? blk + (k + 1 < N ? 0 : W) : Gk) + oH, *Mk = Gk + oM;
    const float *ref = a.ref ? a.ref + (a.ref_per_stage ? a.L.Nn[j] + (int64_t)ks * n : in) : nullptr;
    // the previous solve's iterate, shifted by a stage for warm == 2
    const float *git = a.it[a.base[j]] + a.L.Ni[j] + (int64_t)(warm == 2 && k + 1 < N ? ks + 1 : ks) * ls::iter_stride_plain(n, 4);
    m.setup(
        nx, nu, on, (float)a.rho, [&](int r, int c) { return Gk[r * ldg + c]; },
        [&](int r, int c) { return wrapped_at(Hk, n, r, c); }, [&](int q, int i) { return wrapped_at(Mk, nu, q, i); });
    s.inputs(
        nx, nu, on, [&](int r) { return Gk[oE + r]; }, [&](int c) { return ref ? a.qd[in + c] * ref[c] : 0.0f; },
        [&](int c) { return a.lo[in + c]; }, [&](int c) { return a.hi[in + c]; });
#pragma unroll
    for (int p = 0; p < NN; ++p) {
      const int c = stage::component<NX, NU>(p, nx, nu);
      const bool have = warm != 0 && on && c >= 0;
      s.z[p] = have ? git[c] : 0.0f;
      s.v[p] = have ? git[n + c] : 0.0f;
      s.t[p] = have ? git[2 * n + c] : 0.0f;
      s.b[p] = have ? git[3 * n + c] : 0.0f;
      // read behind the first iteration's barriers
      if (!on) sg[p * ld + k] = 0.0f;
      if (k == 0) {
        sg[p * ld + ld - 1] = 0.0f;
        sx[p * ld] = c >= 0 ? a.xb0[in + c] : 0.0f;
      }
    }
  }
  float xb[NN], share = 0.0f;
  unsigned side;
  int iters = 0;
  for (; iters < a.max_iters; ++iters)
    if (s.template step<true, false>(m, sg, sx, ld, k, on, !detsum::finite(share), xb, side, share)) break;
  // c^{i+1} of the last iteration, independent of the order of its shares
  const int lane = k & 31, warp = k >> 5;
  detsum::Fx sum = detsum::warp_sum(share);
  if (lane == 0) sums[warp] = make_ulonglong2(sum.sig, (unsigned long long)(long long)sum.e);
  __syncthreads();
  if (warp == 0) {
    sum = lane < (int)blockDim.x / 32 ? detsum::Fx{sums[lane].x, (int)sums[lane].y} : detsum::Fx{0ull, detsum::kZero};
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
  if (!on) return;
  float *git = a.it[a.base[j]] + a.L.Ni[j] + (int64_t)k * ls::iter_stride_plain(n, 4);
#pragma unroll
  for (int p = 0; p < NN; ++p) {
    const int c = stage::component<NX, NU>(p, nx, nu);
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
  const size_t smem = sizeof(float) * 2 * stage::padded(size_class) * (threads + 1);
  auto kernel = size_class == 0 ? stage_kernel<2, 1, 3> : size_class == 1 ? stage_kernel<4, 1, 2> : stage_kernel<4, 2, 1>;
  kernel<<<s.L.batch, threads, smem, stream>>>(a, s.warm, s.u_out, s.x_out);
  return cudaGetLastError();
}

}  // namespace pimpc

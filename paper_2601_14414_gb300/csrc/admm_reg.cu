// admm_reg.cu -- the resident schedule (family 3) for instances with n <= 16: the stage matrices
// and the iterates of an instance live in the registers of one CTA, or of a cluster of C CTAs.
//
// What bounds a resident solve is the latency of one iteration: a few hundred multiply-adds per
// stage between synchronisations, the cross-CTA exchange, and the FP64 decision of steps 5-7.
// Thread (slot, c) owns component c of one stage, so that a CTA's warps are full whatever n is,
// and holds in registers its column of G_{k+1}, its rows of G_k, of H_k and of
//   P_k = Bbar_k M_k Bbar_k^T   (du is only ever used as Bbar_k du_k = P_k (v - beta)),
// so that an iteration loads only vectors from shared memory (broadcast 16-byte reads). The
// lambda of Algorithm 1 needs no state of its own: steps 2-3 give
//   v = (z + gamma) / 2 with gamma = Bbar du + beta - Abar xbar - ebar + lambda, hence
//   beta' + lambda' = gamma + z - 2 v = 0,
// and the hats are linear, so lambda = -beta throughout (the zero start included).
// One iteration: hats, y and w | Abar^T y, h, P w | xbar = H h | Abar xbar, steps 2-4 | one
// exchange. The slots of a CTA are its stages and the two neighbouring ones, whose x-update it
// repeats, so that the CTAs of a cluster meet once per iteration: each pushes its share of c and
// its boundary iterates into the others' shared memory, a cluster barrier follows, and every warp
// sums the shares and takes the decision of steps 5-7 by itself (identical inputs, fixed order),
// in integer arithmetic (detsum.cuh) off the 64-cycle FP64 pipe.
// Measured per pass, against the shared-memory kernel of admm_res.cu (which keeps the instances
// with n > 16 and those too long for a cluster's registers): plain LTI nx 4, nu 2, N 20, FP64, 200
// iterations 1579 -> 758 us; quadrotor sample (n 16, N 200, 100 iterations, with its linearisation
// and factorisation) FP32 907 -> 656 us, FP64 2067 -> 1257 us; CSTR sample (n 3, N 5000, 1000
// iterations, FP32) 22.9 -> 4.76 ms; AFTI-16 solve to 1e-6 (n 6, N 5, FP64) 39.8 -> 17.7 ms.
#include <cooperative_groups.h>
#include <algorithm>
#include <math.h>

#include "detsum.cuh"
#include "lockstep.cuh"

namespace cg = cooperative_groups;

namespace pimpc {

namespace {

template <typename T>
using Args = ls::Args<T>;

constexpr int kMaxN = 16;

// Threads of one CTA by the register bound: 4 n-vectors of matrix rows per thread.
__host__ __device__ constexpr int reg_max_threads(int tsize, int NM) {
  return tsize == 4 ? (NM <= 4 ? 1024 : 512) : (NM <= 4 ? 512 : (NM <= 8 ? 512 : 256));
}

struct RegPlan {
  int C;        // CTAs per instance
  int region;   // elements of each of the four vector regions
};

template <typename T>
struct Vec;
template <>
struct Vec<float> {
  static constexpr int W = 4;
};
template <>
struct Vec<double> {
  static constexpr int W = 2;
};

__host__ __device__ inline int reg_nv(int n, int tsize) {
  const int w = tsize == 4 ? 4 : 2;
  return (n + w - 1) / w * w;
}

// sum_j m[j] v[j] over j < cnt, v in shared memory (16-byte aligned, zero-padded to whole
// vectors), m in registers with zeros beyond its length.
template <int NM>
__device__ __forceinline__ float dot(const float (&m)[NM], const float *v, int cnt) {
  float a0 = 0.0f, a1 = 0.0f, a2 = 0.0f, a3 = 0.0f;
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
__device__ __forceinline__ double dot(const double (&m)[NM], const double *v, int cnt) {
  double a0 = 0.0, a1 = 0.0;
#pragma unroll
  for (int j = 0; j < NM; j += 2)
    if (j < cnt) {
      const double2 q = *reinterpret_cast<const double2 *>(v + j);
      a0 = j ? fma(m[j], q.x, a0) : m[j] * q.x;
      a1 = j ? fma(m[j + 1], q.y, a1) : m[j + 1] * q.y;
    }
  return a0 + a1;
}

// x / 3 to within a rounding of the correctly rounded quotient: 1/3 as the sum of its rounding
// and the rounding of what is left (two operations instead of a division; infinities pass).
__device__ __forceinline__ float third(float x) {
  constexpr float hi = 1.0f / 3.0f;
  constexpr float lo = (float)(1.0 / 3.0 - (double)hi);
  return fmaf(x, hi, x * lo);
}
__device__ __forceinline__ double third(double x) {
  constexpr double hi = 1.0 / 3.0;         // (1 - 2^-54) / 3
  constexpr double lo = hi * 0x1p-54;      // 1/3 - hi = 2^-54 / 3
  return fma(x, hi, x * lo);
}

template <typename T>
__device__ __forceinline__ T sym_at(const T *Wp, int m, int r, int c) {
  int d = c - r;
  if (d < 0) d += m;
  return (2 * d <= m) ? Wp[d * m + r] : Wp[(m - d) * m + c];
}

template <typename T, int NM, int kMinCtas>
__global__ void __launch_bounds__(reg_max_threads((int)sizeof(T), NM), kMinCtas)
    reg_kernel(Args<T> a, RegPlan pl) {
  extern __shared__ __align__(128) unsigned char smem_raw[];
  __shared__ double sShare[2][128];          // shares of c by parity
  __shared__ double sWarp[32];               // warp sums (two-stage exchange)
  __shared__ T sLand[2][2][4][kMaxN];        // boundary iterates: parity, side, vector
  cg::cluster_group cl = cg::this_cluster();
  const int C = pl.C;
  const int r = C > 1 ? (int)cl.block_rank() : 0;
  const int j = blockIdx.x / C;
  const int tid = threadIdx.x, nthreads = blockDim.x, lane = tid & 31, warp = tid >> 5;
  const int nw = nthreads >> 5;
  const int nx = a.L.nx[j], nu = a.L.nu[j], N = a.L.N[j], n = nx + nu;
  const int nv = reg_nv(n, (int)sizeof(T));
  const int k0 = (int)((int64_t)r * N / C), k1 = (int)((int64_t)(r + 1) * N / C);
  const int kb = k0 - (r > 0 ? 1 : 0);                       // stage of slot 0
  const int ke = k1 + (k1 < N ? 1 : 0);                      // one past the last slot's stage
  const int slot = tid / n, c = tid - slot * n, k = kb + slot;
  const bool active = k < ke;
  const bool owned = active && k >= k0 && k < k1;
  const bool has_h = active && k < k1;                       // owned, or the stage before them
  const bool more = k + 1 < N;
  T *sW = reinterpret_cast<T *>(smem_raw), *sY = sW + pl.region, *sH = sY + pl.region,
    *sX = sH + pl.region;                                    // sX: row q = xbar_{kb + q}
  for (int i = tid; i < 4 * pl.region; i += nthreads) sW[i] = (T)0;
  for (int i = tid; i < 256; i += nthreads) (&sShare[0][0])[i] = 0.0;

  // ---- the thread's rows and columns, once ----
  T Gn[NM], Gr[NM], Hr[NM], Pr[NM];
#pragma unroll
  for (int q = 0; q < NM; ++q) Gn[q] = Gr[q] = Hr[q] = Pr[q] = (T)0;
  T zc = 0, vc = 0, tc = 0, bc = 0, zp = 0, vp = 0, tp = 0, bp = 0;  // iterate, and the one before
  T ee = 0, qref = 0, lo = 0, hi = 0;
  const T rho = (T)a.rho;
  const int n5p = ls::iter_stride_plain(n, (int)sizeof(T));
  if (active) {
    const int lti = a.L.lti, W = a.L.W[j], ldg = odd_ld(n);
    const int oE = nx * ldg, oH = oE + nx, oM = oH + wrapped_size(n);
    const T *blk = a.blk + a.L.blk[j];
    const T *Gk = blk + (lti ? 0 : (int64_t)k * W);
    const T *Gk1 = lti ? blk : Gk + W;
    const T *Hk = (lti ? blk + (more ? 0 : W) : Gk) + oH;
    const T *git = a.it[a.base[j]] + a.L.Ni[j] + (int64_t)k * n5p;
    zc = git[c];
    vc = git[n + c];
    tc = git[2 * n + c];
    bc = git[3 * n + c];
    zp = zc; vp = vc; tp = tc; bp = bc;
    ee = c < nx ? Gk[oE + c] : (T)0;
    lo = a.lo[a.L.off_n[j] + c];
    hi = a.hi[a.L.off_n[j] + c];
    if (a.ref) {
      const T *ref = a.ref + (a.ref_per_stage ? a.L.Nn[j] + (int64_t)k * n : a.L.off_n[j]);
      qref = a.qd[a.L.off_n[j] + c] * ref[c];
    }
    if (has_h) {
#pragma unroll
      for (int q = 0; q < NM; ++q) {
        if (q < n) Hr[q] = sym_at(Hk, n, c, q);
        if (q < nx && more) Gn[q] = Gk1[q * ldg + c];
      }
    }
    if (owned) {
#pragma unroll
      for (int q = 0; q < NM; ++q)
        if (q < n) Gr[q] = c < nx ? Gk[c * ldg + q] : (q == c ? (T)1 : (T)0);
      // P row c: sum_i (sum_q Bbar[c][q] M[q][i]) Bbar[q'][i], Bbar = [B; I]
      const T *M = Gk + oM;
      for (int i = 0; i < nu; ++i) {
        T t = (T)0;
        if (c < nx) {
          for (int q = 0; q < nu; ++q) t += Gk[c * ldg + nx + q] * sym_at(M, nu, q, i);
        } else {
          t = sym_at(M, nu, c - nx, i);
        }
#pragma unroll
        for (int q = 0; q < NM; ++q)
          if (q < n) Pr[q] += t * (q < nx ? Gk[q * ldg + nx + i] : (q - nx == i ? (T)1 : (T)0));
      }
    }
  }
  double cprev = 1.0, cval = 0.0, cbest = INFINITY;
  double etac = a.eta;  // eta cprev, formed off the critical path
  int itbest = 0, itfirst = -1, streak = 0, momentum = 0, status = kMaxIter, iters = 0;
  T f = (T)0;
  bool use_prev = false;
  const bool two_stage = C > 1 && C * nw > 128;
  const double eps = a.eps;
  __syncthreads();  // the zero fill, before xbar_0 goes to row 0
  if (r == 0 && tid < n) sX[tid] = a.xb0[a.L.off_n[j] + tid];
  if (C > 1) cl.sync();
  else __syncthreads();

  for (int it = 0; it < a.max_iters; ++it) {
    const int par = it & 1;
    // the momentum factor this iteration's decision would take, fetched ahead
    const double ctab = a.accel ? a.coef_tab[streak] : 0.0;
    const T fnext = (T)ctab;
    // ---- hats, y, w ----
    T zh = zc, vh = vc, th = tc, bh = bc;
    if (use_prev) {
      zh = zc + f * (zc - zp);
      vh = vc + f * (vc - vp);
      th = tc + f * (tc - tp);
      bh = bc + f * (bc - bp);
    }
    if (active) {
      sW[slot * nv + c] = vh - bh;
      sY[slot * nv + c] = (zh - vh) - (bh + ee);
    }
    __syncthreads();
    // ---- Abar_{k+1}^T y_{k+1}, h_k; P_k w_k ----
    T bd = (T)0;
    if (has_h) {
      const T *y = sY + (slot + 1) * nv;
      T acc = (T)0;
      if (more) {
        acc = dot(Gn, y, nx);
        if (c >= nx) acc += y[c];
      }
      sH[slot * nv + c] = qref + rho * ((zh - th) + acc);
    }
    if (owned) bd = dot(Pr, sW + slot * nv, n);
    __syncthreads();
    // ---- xbar_{k+1} = H_k h_k ----
    T xb = (T)0;
    if (has_h) {
      xb = dot(Hr, sH + slot * nv, n);
      sX[(slot + 1) * nv + c] = xb;
    }
    __syncthreads();
    // ---- steps 2-4 ----
    T cacc = (T)0;
    T zn = (T)0, vn = (T)0, tn = (T)0, bn = (T)0;
    if (owned) {
      const T ax = dot(Gr, sX + slot * nv, n);
      const T p = bh + bd;
      const T q = -bh - (ax + ee);  // lambda - Abar xbar - ebar
      const T s = xb + th;
      const T w = third((T)2 * s + (p - q));
      zn = w < lo ? lo : (w > hi ? hi : w);
      vn = (T)0.5 * (zn + (p + q));
      tn = s - zn;
      bn = p - vn;
      const T d1 = tn - th, d2 = bn - bh, d4 = zn - zh, d5 = vn - vh, d6 = d4 - d5;
      cacc = d1 * d1 + ((T)2 * d2) * d2 + d4 * d4 + d5 * d5 + d6 * d6;
      if (C > 1) {  // boundary iterates: the first stage to CTA r - 1, the last to CTA r + 1
        if (k == k0 && r > 0) {
          T *d = cl.map_shared_rank(&sLand[par][1][0][0], r - 1) + c;
          d[0] = zn;
          d[kMaxN] = vn;
          d[3 * kMaxN] = bn;
        }
        if (k == k1 - 1 && k1 < N) {
          T *d = cl.map_shared_rank(&sLand[par][0][0][0], r + 1) + c;
          d[0] = zn;
          d[2 * kMaxN] = tn;
        }
      }
    }
    // ---- the exchange: shares of c ----
    double share = detsum::warp_sum1(cacc);
    double sum;
    if (C == 1) {
      if (lane == 0) sShare[par][warp] = share;
      __syncthreads();
      sum = detsum::warp_sum1(lane < nw ? sShare[par][lane] : 0.0);
    } else if (!two_stage) {
      if (lane < C) *cl.map_shared_rank(&sShare[par][r * nw + warp], lane) = share;
      cl.sync();
      detsum::Term t[4];
#pragma unroll
      for (int i = 0; i < 4; ++i) t[i] = detsum::term(sShare[par][lane + 32 * i]);
      sum = detsum::warp_sum<4>(t);
    } else {
      if (lane == 0) sWarp[warp] = share;
      __syncthreads();
      if (warp == 0) {
        share = detsum::warp_sum1(lane < nw ? sWarp[lane] : 0.0);
        if (lane < C) *cl.map_shared_rank(&sShare[par][r], lane) = share;
      }
      cl.sync();
      sum = detsum::warp_sum1(lane < C ? sShare[par][lane] : 0.0);
    }
    // ---- steps 5-7, by every thread alike ----
    const double cn = a.rho == 1.0 ? sum : a.rho * sum;
    cval = cn;
    iters = it + 1;
    bool stop = true;
    f = (T)0;
    use_prev = false;
    if (!detsum::finite(cn)) {
      status = kNonFinite;
    } else if (detsum::le_nonneg(cn, eps)) {
      status = kConverged;
    } else if (a.stall_win > 0 && cn <= a.stall_below && !(cn < a.stall_fac * cbest) &&
               (double)(it - itbest) >=
                   fmax((double)a.stall_win, a.stall_rel * (double)(itfirst < 0 ? it : itfirst))) {
      status = kStalled;
    } else if (it + 1 >= a.max_iters) {
      status = kMaxIter;
    } else {
      stop = false;
      bool take = false;
      if (a.accel) {
        if (a.mask && it < a.mask_len) take = a.mask[(int64_t)j * a.mask_len + it] != 0;
        else take = detsum::le_nonneg(cn, etac);
      }
      if (take) {  // (alpha_m - 1) / alpha_{m+1}, alpha_0 = 1, from the precomputed table
        f = fnext;
        use_prev = streak > 0;
        momentum += streak > 0;
        ++streak;
      } else {
        streak = 0;
      }
      cprev = cn;
      etac = a.eta * cprev;
    }
    if (a.stall_win > 0 && cn <= a.stall_below) {
      if (itfirst < 0) itfirst = it;
      if (cn < a.stall_fac * cbest) {
        cbest = cn;
        itbest = it;
      }
    }
    // ---- the new iterate becomes the current one; halo slots take theirs from the landing ----
    if (C > 1 && active && !owned) {
      const T *d = &sLand[par][k < k0 ? 0 : 1][0][0] + c;
      zn = d[0];
      if (k < k0) {
        tn = d[2 * kMaxN];
      } else {
        vn = d[kMaxN];
        bn = d[3 * kMaxN];
      }
    }
    zp = zc; vp = vc; tp = tc; bp = bc;
    zc = zn; vc = vn; tc = tn; bc = bn;
    if (stop) break;
  }
  if (owned) {
    T *git = a.it[a.base[j]] + a.L.Ni[j] + (int64_t)k * n5p;
    git[c] = zc;
    git[n + c] = vc;
    git[2 * n + c] = tc;
    git[3 * n + c] = bc;
    git[4 * n + c] = -bc;
  }
  if (r == 0 && tid == 0) {
    InstState s;
    s.iters = iters;
    s.status = status;
    s.momentum = momentum;
    s.pad = 0;
    s.c = cval;
    a.st[j] = s;
    a.stop[j] = 1;
  }
}

template <typename T>
const void *pick_kernel(int NM, bool crowded) {
  if constexpr (sizeof(T) == 4)
    if (crowded && NM == 8) return (const void *)reg_kernel<T, 8, 2>;
  return NM == 4   ? (const void *)reg_kernel<T, 4, 1>
         : NM == 8 ? (const void *)reg_kernel<T, 8, 1>
                   : (const void *)reg_kernel<T, 16, 1>;
}

int reg_class(int n) { return n <= 4 ? 4 : (n <= 8 ? 8 : 16); }

}  // namespace

// Threads and shared memory of one CTA for C CTAs per instance; 0 threads: the batch does not fit
// (an n above 16, fewer stages than CTAs, or more stages per CTA than its threads hold).
void reg_plan(int batch, const int *nx, const int *nu, const int *N, int precision, int C,
              int *threads, int *region, int *nmax) {
  const int ts = precision == 0 ? 4 : 8;
  int thr = 0, reg = 0, nm = 1;
  for (int j = 0; j < batch; ++j) nm = std::max(nm, nx[j] + nu[j]);
  *threads = 0;
  if (nm > kMaxN) return;
  const int cap = reg_max_threads(ts, reg_class(nm));
  for (int j = 0; j < batch; ++j) {
    const int n = nx[j] + nu[j];
    if (N[j] < C) return;
    const int slots = (N[j] + C - 1) / C + (C > 1 ? 2 : 0);
    if ((int64_t)slots * n > cap) return;
    thr = std::max(thr, slots * n);
    reg = std::max(reg, (slots + 1) * reg_nv(n, ts));
  }
  *threads = (thr + 31) / 32 * 32;
  *region = (reg + 3) / 4 * 4;
  *nmax = nm;
}

template <typename T>
static cudaError_t reg_launch_t(const AdmmLaunch &s, const RegLaunch &rl, cudaStream_t stream) {
  Args<T> a = ls::make_args<T>(s);
  a.eps = s.eps + 0.0;  // -0 becomes +0: the stop test compares bit patterns
  cudaError_t rc = cudaMemcpyAsync(s.old_base, s.base, sizeof(int) * s.L.batch,
                                   cudaMemcpyDeviceToDevice, stream);
  if (rc != cudaSuccess) return rc;
  const int n_init = s.L.batch > s.nitems ? s.L.batch : s.nitems;
  ls::solve_init_kernel<T><<<(n_init + 255) / 256, 256, 0, stream>>>(a, s.warm);
  if ((rc = cudaGetLastError()) != cudaSuccess) return rc;
  if (s.warm != 1) {
    ls::prepare_kernel<T><<<dim3(8, s.L.batch), 256, 0, stream>>>(a, s.warm, s.old_base);
    if ((rc = cudaGetLastError()) != cudaSuccess) return rc;
  }
  if (s.max_iters > 0) {
    int dev = 0, nsm = 0;
    if ((rc = cudaGetDevice(&dev)) != cudaSuccess) return rc;
    if ((rc = cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess) return rc;
    const void *kernel = pick_kernel<T>(reg_class(rl.nmax), (int64_t)s.L.batch * rl.C > nsm);
    const size_t smem = (size_t)4 * rl.region * sizeof(T);
    rc = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (rc != cudaSuccess) return rc;
    if (rl.C > 8) {
      rc = cudaFuncSetAttribute(kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
      if (rc != cudaSuccess) return rc;
    }
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(s.L.batch * rl.C);
    cfg.blockDim = dim3(rl.threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = stream;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = rl.C;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    RegPlan pl{rl.C, rl.region};
    void *params[] = {&a, &pl};
    rc = cudaLaunchKernelExC(&cfg, kernel, params);
    if (rc != cudaSuccess) return rc;
  }
  ls::output_kernel<T><<<dim3(4, s.L.batch), 256, 0, stream>>>(a, s.u_out, s.x_out);
  return cudaGetLastError();
}

cudaError_t launch_reg(const AdmmLaunch &s, int precision, const RegLaunch &rl, cudaStream_t stream) {
  return precision == 0 ? reg_launch_t<float>(s, rl, stream) : reg_launch_t<double>(s, rl, stream);
}

}  // namespace pimpc

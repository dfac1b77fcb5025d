// admm_reg.cuh -- the resident schedule (family 3) for instances with n <= 16: the stage matrices
// and the iterates of an instance live in the registers of one CTA, or of C CTAs: a cluster of
// up to 16, or up to 144 that meet through global memory.
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
// repeats, so that the CTAs of an instance meet once per iteration: each sends its share of c to
// all and its boundary iterates to its neighbours, and every CTA sums the shares and takes the
// decision of steps 5-7 by itself (identical inputs, a sum that has no order), in integer
// arithmetic (detsum.cuh) off the 64-cycle FP64 pipe. Within a cluster the data go by st.async
// into the others' shared memory and complete on their mbarriers (520-660 cycles per exchange,
// measured; remote stores and a cluster barrier 890 and more); beyond 16 CTAs they go through
// global memory as 16-byte records that carry their iteration number (1400-1600 cycles, measured with
// 16 to 96 CTAs; a barrier on an atomic counter takes 2500 before any data are read).
// The launch also makes the starting iterates and the outputs: one kernel per solve.
// FP64 is bound by its pipe (a warp issues one FP64 instruction per 64 cycles, an SM one per 19),
// so the FP64 code counts instructions: one chain per dot product, with the sums around it folded
// into its start; x / 3 as two operations; the clamp on bit patterns.
// What is left of an exchange and a decision (about 2000 cycles in a cluster of 16, half of an FP32
// iteration) runs beside the next iteration, in a warp of its own (spec_kernel).
// Per iteration, measured, against the shared-memory kernel of admm_res.cu (which keeps the
// instances with n > 16) and, in brackets, without the deciding warp: plain LTI n 6, N 20, FP64
// 7.9 -> 3.0 us (3.2); quadrotor n 16, N 200 FP32 6.8 -> 1.26 us (1.80), FP64 18.6 -> 4.7 us (5.6);
// CSTR n 3, N 5000 FP32 22.8 -> 1.80 us (2.59), FP64 102 -> 3.65 us (5.9).
#pragma once
#include <cooperative_groups.h>
#include <algorithm>
#include <math.h>

#include "detsum.cuh"
#include "lockstep.cuh"
#include "regvec.cuh"

namespace cg = cooperative_groups;

namespace pimpc {

namespace {

template <typename T>
using Args = ls::Args<T>;

constexpr int kMaxN = 16;
constexpr int kMaxC = 144;           // CTAs of one instance (grid scope)
constexpr int kLaneShares = (kMaxC + 31) / 32;
constexpr int kWaitPolls = 1 << 22;  // bounded waits: polls of a record in global memory ...
constexpr long long kWaitCycles = 1ll << 31;  // ... and cycles at an mbarrier (about a second)

// Who runs an instance: one CTA, a cluster of up to 16, or up to kMaxC CTAs of a cooperative
// launch that exchange through global memory.
enum { kCta = 0, kCluster = 1, kGrid = 2 };

// kSpec: a warp of its own finds c and takes the decisions while the others run the next iteration
// on the hats that a momentum step would give (latency: CTAs that have an SM each). kSolo: warp 0
// finds c between two iterations (batches that crowd the SMs). kLazy: c is not formed before the last
// iteration (the plain iteration with a fixed count, where no decision depends on it but that a
// non-finite c ends the solve, so an iterate that is not finite or so large that its squares may not
// be has it formed).
enum { kSpec = 0, kSolo = 1, kLazy = 2 };

// Threads of one CTA by the register bound: 4 n-vectors of matrix rows per thread.
__host__ __device__ constexpr int reg_max_threads(int tsize, int NM) {
  return tsize == 4 ? (NM <= 4 ? 1024 : 512) : (NM <= 4 ? 512 : (NM <= 8 ? 512 : 256));
}

// With the deciding warp (kSpec), whose iterations have an SM to themselves: FP64 keeps more registers.
__host__ __device__ constexpr int spec_max_threads(int tsize, int NM) {
  return tsize == 4 ? reg_max_threads(tsize, NM) : 256;
}

struct RegPlan {
  int C;              // CTAs per instance
  int region;         // elements of each of the four vector regions
  ulonglong2 *xch;    // grid scope: the exchange records
  double *u_out, *x_out;
  int warm;
};

// Exchange records of one instance (grid scope): by parity, C shares, then per CTA two sides of
// kHaloRecs halo records. Every record carries the iteration in its upper 32 bits and is written
// and read as one 16-byte access, so a reader that sees the iteration sees the payload.
constexpr int kHaloRecs = 3 * kMaxN;
__host__ __device__ inline size_t xch_records(int C) { return (size_t)2 * C * (1 + 2 * kHaloRecs); }

template <typename T>
__device__ __forceinline__ T sym_at(const T *Wp, int m, int r, int c) {
  int d = c - r;
  if (d < 0) d += m;
  return (2 * d <= m) ? Wp[d * m + r] : Wp[(m - d) * m + c];
}

// ---- exchange primitives ---------------------------------------------------------------------

__device__ __forceinline__ unsigned smem_addr(const void *p) {
  return (unsigned)__cvta_generic_to_shared(p);
}
__device__ __forceinline__ unsigned remote(unsigned addr, int rank) {
  unsigned r;
  asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(rank));
  return r;
}
// Store to a CTA of the cluster that counts its bytes on that CTA's mbarrier.
__device__ __forceinline__ void push(unsigned dst, unsigned bar, float v) {
  asm volatile("st.async.shared::cluster.mbarrier::complete_tx::bytes.b32 [%0], %1, [%2];" ::"r"(dst),
               "r"(__float_as_uint(v)), "r"(bar)
               : "memory");
}
__device__ __forceinline__ void push(unsigned dst, unsigned bar, double v) {
  asm volatile("st.async.shared::cluster.mbarrier::complete_tx::bytes.b64 [%0], %1, [%2];" ::"r"(dst),
               "l"(__double_as_longlong(v)), "r"(bar)
               : "memory");
}
__device__ __forceinline__ void push(unsigned dst, unsigned bar, detsum::Fx v) {
  asm volatile("st.async.shared::cluster.mbarrier::complete_tx::bytes.v2.b64 [%0], {%1, %2}, [%3];" ::"r"(
                   dst),
               "l"(v.sig), "l"((long long)v.e), "r"(bar)
               : "memory");
}
__device__ __forceinline__ bool bar_wait(unsigned bar, unsigned parity) {
  const long long t0 = clock64();
  do {
    unsigned ok;
    asm volatile(
        "{\n\t.reg .pred q;\n\t"
        "mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 q, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, q;\n\t}"
        : "=r"(ok)
        : "r"(bar), "r"(parity)
        : "memory");
    if (ok) return true;
  } while (clock64() - t0 < kWaitCycles);
  return false;
}
// One 16-byte record, written and read in a single access.
__device__ __forceinline__ void put_rec(ulonglong2 *p, unsigned long long a, unsigned long long b) {
  asm volatile("{\n\t.reg .b128 t;\n\tmov.b128 t, {%1, %2};\n\t"
               "st.relaxed.gpu.global.b128 [%0], t;\n\t}" ::"l"(p),
               "l"(a), "l"(b)
               : "memory");
}
__device__ __forceinline__ void get_rec(const ulonglong2 *p, unsigned long long &a,
                                        unsigned long long &b) {
  asm volatile("{\n\t.reg .b128 t;\n\tld.relaxed.gpu.global.b128 t, [%2];\n\t"
               "mov.b128 {%0, %1}, t;\n\t}"
               : "=l"(a), "=l"(b)
               : "l"(p)
               : "memory");
}
__device__ __forceinline__ unsigned long long with_tag(unsigned lo, unsigned tag) {
  return (unsigned long long)lo | ((unsigned long long)tag << 32);
}
// Boundary values through global memory. FP32: one record of up to three values per component;
// FP64: one record per value.
__device__ __forceinline__ void put_halo(ulonglong2 *p, int n, int c, unsigned tag, float x, float y,
                                         float w) {
  put_rec(p + c, (unsigned long long)__float_as_uint(x) | ((unsigned long long)__float_as_uint(y) << 32),
          with_tag(__float_as_uint(w), tag));
}
__device__ __forceinline__ void put_halo(ulonglong2 *p, int n, int c, unsigned tag, double x, double y,
                                         double w) {
  put_rec(p + c, (unsigned long long)__double_as_longlong(x), with_tag(0, tag));
  put_rec(p + n + c, (unsigned long long)__double_as_longlong(y), with_tag(0, tag));
  put_rec(p + 2 * n + c, (unsigned long long)__double_as_longlong(w), with_tag(0, tag));
}
__device__ __forceinline__ bool get_halo(const ulonglong2 *p, int n, int c, unsigned tag, float &x,
                                         float &y, float &w) {
  unsigned long long a, b;
  for (int i = 0; i < kWaitPolls; ++i) {
    get_rec(p + c, a, b);
    if ((unsigned)(b >> 32) != tag) continue;
    x = __uint_as_float((unsigned)a);
    y = __uint_as_float((unsigned)(a >> 32));
    w = __uint_as_float((unsigned)b);
    return true;
  }
  return false;
}
__device__ __forceinline__ bool get_halo(const ulonglong2 *p, int n, int c, unsigned tag, double &x,
                                         double &y, double &w) {
  unsigned long long a[3], b[3];
  for (int i = 0; i < kWaitPolls; ++i) {
#pragma unroll
    for (int q = 0; q < 3; ++q) get_rec(p + q * n + c, a[q], b[q]);
    if ((unsigned)(b[0] >> 32) != tag || (unsigned)(b[1] >> 32) != tag || (unsigned)(b[2] >> 32) != tag)
      continue;
    x = __longlong_as_double((long long)a[0]);
    y = __longlong_as_double((long long)a[1]);
    w = __longlong_as_double((long long)a[2]);
    return true;
  }
  return false;
}

// Data of the exchanges in shared memory.
template <typename T>
struct Shared {
  ulonglong2 share[2][16];      // cluster: shares of c by parity (sig, e)
  ulonglong2 warp[32];          // warp sums (sig, e)
  T land[2][2][3][kMaxN];       // cluster: boundary iterates by parity and side
  unsigned long long bar[2];    // cluster: mbarriers by parity: boundary iterates (and shares)
  unsigned long long sbar[2];   // cluster, kSpec: mbarriers by parity: shares
  double cn;                    // kSolo: c / rho, as found by warp 0
  T fnext;                      // kSpec: the decision: momentum factor of the iteration after the
  int stop, take, use_next;     // next, stop, momentum step (else restart), whether fnext applies
  int fail;                     // a wait gave up
};

// One thread's component of one stage: its matrix rows, its iterate and the one before.
template <typename T, int NM>
struct Lane {
  T Gn[NM], Gr[NM], Hr[NM], Pr[NM];
  T zc, vc, tc, bc, zp, vp, tp, bp;
  T ee, qref, lo, hi, rho;
  int nx, n, nv, slot, c, k, k0, k1;
  bool active, owned, has_h, more, below, above;  // below / above: a CTA of the instance on that side

  __device__ __forceinline__ void setup(const Args<T> &a, int warm, int j, int r, int C, int tid) {
    const int nu = a.L.nu[j], N = a.L.N[j];
    nx = a.L.nx[j];
    n = nx + nu;
    nv = reg_nv(n, (int)sizeof(T));
    k0 = (int)((int64_t)r * N / C);
    k1 = (int)((int64_t)(r + 1) * N / C);
    below = r > 0;
    above = k1 < N;
    slot = tid / n;
    c = tid - slot * n;
    k = k0 - (below ? 1 : 0) + slot;            // slot 0 is the stage before the CTA's, if any
    active = k < k1 + (above ? 1 : 0);          // the last slot the stage after them
    owned = active && k >= k0 && k < k1;
    has_h = active && k < k1;                   // owned, or the stage before them
    more = k + 1 < N;
#pragma unroll
    for (int q = 0; q < NM; ++q) Gn[q] = Gr[q] = Hr[q] = Pr[q] = (T)0;
    zc = vc = tc = bc = zp = vp = tp = bp = (T)0;
    ee = qref = lo = hi = (T)0;
    rho = (T)a.rho;
    if (!active) return;
    const int lti = a.L.lti, W = a.L.W[j], ldg = odd_ld(n);
    const int oE = nx * ldg, oH = oE + nx, oM = oH + wrapped_size(n);
    const T *blk = a.blk + a.L.blk[j];
    const T *Gk = blk + (lti ? 0 : (int64_t)k * W);
    const T *Gk1 = lti ? blk : Gk + W;
    const T *Hk = (lti ? blk + (more ? 0 : W) : Gk) + oH;
    if (warm != 0) {  // the previous solve's iterate, shifted by a stage for warm == 2
      const T *git = iterates(a, j) + (int64_t)(warm == 2 && more ? k + 1 : k) * stride();
      zc = git[c];
      vc = git[n + c];
      tc = git[2 * n + c];
      bc = git[3 * n + c];
    }
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

  __device__ __forceinline__ int stride() const { return ls::iter_stride_plain(n, (int)sizeof(T)); }
  __device__ __forceinline__ T *iterates(const Args<T> &a, int j) const {
    return a.it[a.base[j]] + a.L.Ni[j];
  }

  // Steps 1-4 with hats cur + f (cur - prev) (momentum) or cur: the new iterate of an owned component
  // and its share of c. sW, sY, sH, sX: the CTA's vectors (sX: row q = xbar of slot q); sync: a barrier
  // of its threads, after which earlier reads of the vectors are over.
  // kShare: whether the share is formed.
  template <bool kShare, typename Sync>
  __device__ __forceinline__ void iterate(T *sW, T *sY, T *sH, T *sX, T f, bool momentum, Sync sync, T &zn,
                                          T &vn, T &tn, T &bn, T &cacc) {
    // ---- hats, y, w ----
    T zh = zc, vh = vc, th = tc, bh = bc;
    if (momentum) {
      zh = zc + f * (zc - zp);
      vh = vc + f * (vc - vp);
      th = tc + f * (tc - tp);
      bh = bc + f * (bc - bp);
    }
    if (active) {
      sW[slot * nv + c] = vh - bh;
      sY[slot * nv + c] = (zh - vh) - (bh + ee);
    }
    sync();
    // ---- Abar_{k+1}^T y_{k+1}, h_k; Bbar du = P_k w_k ----
    T bd = (T)0;
    if (has_h) {
      const T *y = sY + (slot + 1) * nv;
      T acc = zh - th;
      if (more) {
        if (c >= nx) acc += y[c];
        acc = dot(Gn, y, nx, acc);
      }
      sH[slot * nv + c] = qref + rho * acc;
    }
    if (owned) bd = dot(Pr, sW + slot * nv, n, (T)0);
    sync();
    // ---- xbar_{k+1} = H_k h_k ----
    T xb = (T)0;
    if (has_h) {
      xb = dot(Hr, sH + slot * nv, n, (T)0);
      sX[(slot + 1) * nv + c] = xb;
    }
    sync();
    // ---- steps 2-4 ----
    cacc = (T)0;
    zn = vn = tn = bn = (T)0;
    if (owned) {
      const Step<T> r = steps23(xb, bd, dot(Gr, sX + slot * nv, n, ee), th, bh, lo, hi);
      zn = r.z;
      vn = r.v;
      tn = r.t;
      bn = r.b;
      // theta' - theta = xbar - z' and beta' - beta = Bbar du - v', without the duals' own rounding
      if constexpr (kShare) cacc = share(xb - zn, bd - vn, zn - zh, vn - vh);
    }
  }

  // d1^2 + d2^2 + d3^2 + d4^2 + d5^2 + (d4 - d5)^2 with d3 = -d2.
  static __device__ __forceinline__ T share(T d1, T d2, T d4, T d5) {
    const T g = d2 * d2 + (d4 * d4 + d5 * (d5 - d4));
    return (T)2 * g + d1 * d1;
  }

  // Cluster: the first stage's new iterate to CTA r - 1, the last one's to CTA r + 1.
  __device__ __forceinline__ void push_boundary(Shared<T> &sh, int par, int r, T zn, T vn, T tn, T bn) const {
    if (owned && k == k0 && below) {
      const unsigned bar = remote(smem_addr(&sh.bar[par]), r - 1);
      const unsigned d = remote(smem_addr(&sh.land[par][1][0][c]), r - 1);
      push(d, bar, zn);
      push(d + kMaxN * sizeof(T), bar, vn);
      push(d + 2 * kMaxN * sizeof(T), bar, bn);
    }
    if (owned && k == k1 - 1 && above) {
      const unsigned bar = remote(smem_addr(&sh.bar[par]), r + 1);
      const unsigned d = remote(smem_addr(&sh.land[par][0][0][c]), r + 1);
      push(d, bar, zn);
      push(d + kMaxN * sizeof(T), bar, tn);
    }
  }
  __device__ __forceinline__ unsigned boundary_bytes() const {
    return (unsigned)((int)sizeof(T) * n * ((below ? 2 : 0) + (above ? 3 : 0)));
  }
  // Cluster: what the neighbours pushed, for the slots of their stages.
  __device__ __forceinline__ void land(const Shared<T> &sh, int par, T &zn, T &vn, T &tn, T &bn) const {
    const T *d = &sh.land[par][k < k0 ? 0 : 1][0][c];
    zn = d[0];
    if (k < k0) {
      tn = d[kMaxN];
    } else {
      vn = d[kMaxN];
      bn = d[2 * kMaxN];
    }
  }

  // The current iterate to the solver's buffer, and the outputs.
  __device__ __forceinline__ void store(const Args<T> &a, const RegPlan &pl, int j) const {
    if (!owned) return;
    T *git = iterates(a, j) + (int64_t)k * stride();
    git[c] = zc;
    git[n + c] = vc;
    git[2 * n + c] = tc;
    git[3 * n + c] = bc;
    git[4 * n + c] = -bc;
    if (c < nx) {
      if (pl.x_out) pl.x_out[a.L.Nnx[j] + (int64_t)k * nx + c] = (double)zc;
    } else if (pl.u_out) {
      pl.u_out[a.L.Nnu[j] + (int64_t)k * (n - nx) + (c - nx)] = (double)zc;
    }
  }
};

// Steps 5-7 of one instance: the stop tests and the momentum decision, from c^{i+1}.
struct Decider {
  double cval = 0.0, cbest = INFINITY, etac;  // etac: eta times the last c (1 at the start)
  double eps, rho;
  int itbest = 0, itfirst = -1, streak = 0, momentum = 0, status = kMaxIter, iters = 0;
  bool unit_rho, watch;

  template <typename T>
  __device__ __forceinline__ explicit Decider(const Args<T> &a)
      : etac(a.eta), eps(a.eps), rho(a.rho), unit_rho(a.rho == 1.0),
        watch(a.stall_win > 0 || a.mask != nullptr) {}

  // c from the sum of the shares: the stop flag, and whether the next hats take the momentum step.
  template <typename T>
  __device__ __forceinline__ bool step(const Args<T> &a, int j, int it, double cn, bool &take) {
    if (!unit_rho) cn *= rho;
    cval = cn;
    iters = it + 1;
    bool stop = false;
    if (detsum::le_nonneg(cn, eps) || !detsum::finite(cn) || it + 1 >= a.max_iters || watch) {
      take = false;
      if (!detsum::finite(cn)) {
        status = kNonFinite; stop = true;
      } else if (detsum::le_nonneg(cn, eps)) {
        status = kConverged; stop = true;
      } else if (a.stall_win > 0 && cn <= a.stall_below && !(cn < a.stall_fac * cbest) &&
                 (double)(it - itbest) >=
                     fmax((double)a.stall_win, a.stall_rel * (double)(itfirst < 0 ? it : itfirst))) {
        status = kStalled; stop = true;
      } else if (it + 1 >= a.max_iters) {
        status = kMaxIter; stop = true;
      } else if (a.accel) {
        if (a.mask && it < a.mask_len) take = a.mask[(int64_t)j * a.mask_len + it] != 0;
        else take = detsum::le_nonneg(cn, etac);
      }
      if (a.stall_win > 0 && cn <= a.stall_below) {
        if (itfirst < 0) itfirst = it;
        if (cn < a.stall_fac * cbest) {
          cbest = cn;
          itbest = it;
        }
      }
    } else {
      take = a.accel && detsum::le_nonneg(cn, etac);
    }
    etac = a.eta * cn;
    momentum += take && streak > 0;
    streak = take ? streak + 1 : 0;
    return stop;
  }

  // The momentum factor (alpha_m - 1) / alpha_{m+1}, alpha_0 = 1, after m momentum steps in a row,
  // from the precomputed table: loaded here and not where it is used.
  template <typename T>
  __device__ __forceinline__ double factor(const Args<T> &a, int m) const {
    double v;
    asm volatile("ld.global.f64 %0, [%1];" : "=d"(v) : "l"(a.coef_tab + (a.accel ? m : 0)));
    return v;
  }

  template <typename T>
  __device__ __forceinline__ void store(const Args<T> &a, int j) const {
    InstState s;
    s.iters = iters;
    s.status = a.ferr && a.ferr[j] ? kFactorFailed : status;
    s.momentum = momentum;
    s.pad = 0;
    s.c = cval;
    a.st[j] = s;
    a.stop[j] = 1;
  }
};

__device__ __forceinline__ ulonglong2 packed(detsum::Fx t) {
  return make_ulonglong2(t.sig, (unsigned long long)(long long)t.e);
}
__device__ __forceinline__ detsum::Fx unpacked(ulonglong2 q) { return detsum::Fx{q.x, (int)q.y}; }

// Zeroes the vectors, sets up the mbarriers and xbar_0 (every thread of the CTA).
template <typename T, int SC>
__device__ __forceinline__ void start_cta(const Args<T> &a, const RegPlan &pl, Shared<T> &sh, T *vec, T *sX,
                                          int j, int r, int n) {
  const int tid = threadIdx.x;
  for (int i = tid; i < 4 * pl.region; i += blockDim.x) vec[i] = (T)0;
  if (tid < 32) sh.warp[tid] = make_ulonglong2(0, (unsigned long long)(long long)detsum::kZero);
  if (tid == 0) {
    sh.fail = 0;
    if (SC == kCluster) {
      for (int p = 0; p < 2; ++p) {
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_addr(&sh.bar[p])));
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_addr(&sh.sbar[p])));
      }
      asm volatile("fence.mbarrier_init.release.cluster;");
    }
  }
  __syncthreads();
  if (r == 0 && tid < n) sX[tid] = a.xb0[a.L.off_n[j] + tid];
  if (SC == kCluster) cg::this_cluster().sync();  // every mbarrier is ready
  else __syncthreads();
}

__device__ __forceinline__ void expect(unsigned long long *bar, unsigned bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_addr(bar)), "r"(bytes)
               : "memory");
}
template <int kId>
__device__ __forceinline__ void named_sync(int threads) {
  asm volatile("bar.sync %0, %1;" ::"n"(kId), "r"(threads) : "memory");
}
template <int kId>
__device__ __forceinline__ void named_arrive(int threads) {
  asm volatile("bar.arrive %0, %1;" ::"n"(kId), "r"(threads) : "memory");
}

// kSpec. The last warp of the CTA decides, the others iterate. Iteration i's warp sums are handed to the
// decider, which sums them, exchanges shares with the other CTAs, takes the decision and hands it
// back; meanwhile the others run iteration i + 1 on the hats that a momentum step would give, the
// factor of which is known an iteration ahead. At its end they learn the decision of i: stop (the
// iteration in hand is dropped), momentum (it stands), restart (it is run again on hats equal to the
// iterates, unless it was without momentum anyway). Only then its boundary iterates and sums leave
// the CTA, so a CTA is never more than one iteration ahead of another, which two buffers by parity
// allow for.
template <typename T, int NM, int SC>
__global__ void __launch_bounds__(spec_max_threads((int)sizeof(T), NM), 1) spec_kernel(Args<T> a, RegPlan pl) {
  extern __shared__ __align__(128) unsigned char smem_raw[];
  __shared__ Shared<T> sh;
  const int C = SC == kCta ? 1 : pl.C;
  const int r = SC == kCta ? 0 : (int)(blockIdx.x % C);  // the rank in the cluster: C divides grid
  const int j = blockIdx.x / C;
  const int all = blockDim.x, nct = all - 32;            // threads, and those that iterate
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nw = nct >> 5;
  const bool decides = warp == nw;
  T *sW = reinterpret_cast<T *>(smem_raw), *sY = sW + pl.region, *sH = sY + pl.region, *sX = sH + pl.region;
  ulonglong2 *xs = nullptr, *xh = nullptr;  // grid: this instance's share and halo records
  if (SC == kGrid) {
    xs = pl.xch + (size_t)j * xch_records(C);
    xh = xs + 2 * C;
  }
  start_cta<T, SC>(a, pl, sh, sW, sX, j, r, a.L.nx[j] + a.L.nu[j]);

  if (decides) {
    Decider d(a);
    for (int it = 0;; ++it) {
      const int par = it & 1;
      const unsigned tag = (unsigned)it + 1;
      if (SC == kCluster && lane == 0) expect(&sh.sbar[par], (unsigned)(16 * C));
      const T fmore = (T)d.factor(a, d.streak + 1);
      named_sync<2>(all);  // the warp sums of iteration it
      bool ok = SC == kCta || *(volatile int *)&sh.fail == 0;
      detsum::Fx sum = unpacked(sh.warp[nw == 1 ? 0 : lane]);  // {0, kZero} beyond the CTA's warps
      if (nw > 1) sum = detsum::warp_sum(sum);
      if (SC == kCluster && ok) {
        if (lane < C)
          push(remote(smem_addr(&sh.share[par][r]), lane), remote(smem_addr(&sh.sbar[par]), lane), sum);
        ok = __all_sync(0xffffffffu, bar_wait(smem_addr(&sh.sbar[par]), (unsigned)(it >> 1) & 1u));
        sum = detsum::warp_sum(lane < C ? unpacked(sh.share[par][lane]) : detsum::Fx{0ull, detsum::kZero});
      }
      if (SC == kGrid && ok) {
        if (lane == 0) put_rec(xs + par * C + r, sum.sig, with_tag((unsigned)sum.e, tag));
        detsum::Fx t[kLaneShares];  // the lane's shares, all in flight
        ok = false;
        for (int n_ = 0; n_ < kWaitPolls && !ok; ++n_) {
          bool mine = true;
#pragma unroll
          for (int q = 0; q < kLaneShares; ++q) {
            unsigned long long b = with_tag((unsigned)detsum::kZero, tag);
            t[q].sig = 0;
            if (lane + 32 * q < C) get_rec(xs + par * C + lane + 32 * q, t[q].sig, b);
            t[q].e = (int)(unsigned)b;
            mine = mine && (unsigned)(b >> 32) == tag;
          }
          ok = __all_sync(0xffffffffu, mine);
        }
        sum = detsum::warp_sum(t[0]);
        if (C > 32) {  // the sums of each round of 32, on lanes 0, 1, ..
          detsum::Fx mine = lane == 0 ? sum : detsum::Fx{0ull, detsum::kZero};
#pragma unroll
          for (int q = 1; q < kLaneShares; ++q) {
            const detsum::Fx sq = detsum::warp_sum(t[q]);
            if (lane == q) mine = sq;
          }
          sum = detsum::warp_sum(mine);
        }
      }
      bool take = false;
      bool stop = d.step(a, j, it, detsum::to_double(sum), take);
      if (!ok) {  // a wait gave up, here or at a boundary: nothing leaves this CTA any more
        stop = true;
        d.status = kTimeout;
      }
      if (lane == 0) {
        sh.stop = stop;
        sh.take = take;
        sh.fnext = take ? fmore : (T)0;
        sh.use_next = take;  // after a restart the next factor is 0
        if (!ok) sh.fail = 1;
      }
      __syncwarp();
      named_arrive<3>(all);  // the decision of iteration it
      if (stop) break;
    }
    if (r == 0 && lane == 0) d.store(a, j);
  } else {
    Lane<T, NM> L;
    L.setup(a, pl.warm, j, r, C, tid);
    auto sync = [&]() { named_sync<1>(nct); };
    sync();
    T f = (T)0;
    bool momentum = false;
    for (int it = 0;; ++it) {
      const int par = it & 1, last = par ^ 1;
      const unsigned tag = (unsigned)it + 1;
      if (SC == kCluster && tid == 0) expect(&sh.bar[par], L.boundary_bytes());
      if (SC != kCta && it > 0 && L.active && !L.owned) {  // the neighbours' iterate of it - 1
        T zn = (T)0, vn = (T)0, tn = (T)0, bn = (T)0;
        if (SC == kCluster) {
          if (!bar_wait(smem_addr(&sh.bar[last]), (unsigned)((it - 1) >> 1) & 1u)) sh.fail = 1;
          L.land(sh, last, zn, vn, tn, bn);
        } else {
          T x, y, w;
          const bool before = L.k < L.k0;
          if (!get_halo(xh + ((size_t)(last * C + r) * 2 + (before ? 0 : 1)) * kHaloRecs, L.n, L.c, tag - 1, x, y, w)) {
            sh.fail = 1;
            x = y = w = (T)0;
          }
          zn = x;
          if (before) {
            tn = y;
          } else {
            vn = y;
            bn = w;
          }
        }
        L.zp = L.zc; L.vp = L.vc; L.tp = L.tc; L.bp = L.bc;
        L.zc = zn; L.vc = vn; L.tc = tn; L.bc = bn;
      }
      T zn, vn, tn, bn, cacc;
      T fnext = (T)0;
      bool mnext = false;
      if (it < a.max_iters) {
        L.template iterate<true>(sW, sY, sH, sX, f, momentum, sync, zn, vn, tn, bn, cacc);
      }
      if (it > 0) {
        named_sync<3>(all);  // the decision of it - 1
        if (*(volatile int *)&sh.stop) break;
        fnext = *(volatile T *)&sh.fnext;
        mnext = *(volatile int *)&sh.use_next != 0;
        if (momentum && !*(volatile int *)&sh.take)
          L.template iterate<true>(sW, sY, sH, sX, (T)0, false, sync, zn, vn, tn, bn, cacc);
      }
      if (SC == kCta || *(volatile int *)&sh.fail == 0) {
        if (SC == kCluster) L.push_boundary(sh, par, r, zn, vn, tn, bn);
        if (SC == kGrid && L.owned) {
          if (L.k == L.k0 && L.below)
            put_halo(xh + ((size_t)(par * C + r - 1) * 2 + 1) * kHaloRecs, L.n, L.c, tag, zn, vn, bn);
          if (L.k == L.k1 - 1 && L.above)
            put_halo(xh + (size_t)(par * C + r + 1) * 2 * kHaloRecs, L.n, L.c, tag, zn, tn, (T)0);
        }
      }
      const detsum::Fx sum = detsum::warp_sum(cacc);
      if (lane == 0) sh.warp[warp] = packed(sum);
      named_arrive<2>(all);
      if (L.owned) {
        L.zp = L.zc; L.vp = L.vc; L.tp = L.tc; L.bp = L.bc;
        L.zc = zn; L.vc = vn; L.tc = tn; L.bc = bn;
      }
      f = fnext;
      momentum = mnext;
    }
    L.store(a, pl, j);
  }
  if (SC == kCluster) cg::this_cluster().sync();  // no CTA leaves with a push to it in flight
}

// kSolo and kLazy: one iteration after the other.
template <typename T, int NM, int SC, int kMode, int kMinCtas>
__global__ void __launch_bounds__(reg_max_threads((int)sizeof(T), NM), kMinCtas)
    reg_kernel(Args<T> a, RegPlan pl) {
  extern __shared__ __align__(128) unsigned char smem_raw[];
  __shared__ Shared<T> sh;
  constexpr bool lazy = kMode == kLazy;
  const int C = SC == kCta ? 1 : pl.C;
  const int r = SC == kCta ? 0 : (int)(blockIdx.x % C);  // the rank in the cluster: C divides grid
  const int j = blockIdx.x / C;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  T *sW = reinterpret_cast<T *>(smem_raw), *sY = sW + pl.region, *sH = sY + pl.region, *sX = sH + pl.region;
  start_cta<T, SC>(a, pl, sh, sW, sX, j, r, a.L.nx[j] + a.L.nu[j]);
  Lane<T, NM> L;
  L.setup(a, pl.warm, j, r, C, tid);
  Decider d(a);
  auto sync = [&]() { __syncthreads(); };
  sync();
  T f = (T)0;
  bool momentum = false;
  for (int it = 0; it < a.max_iters; ++it) {
    const int par = it & 1;
    if (SC == kCluster && tid == 0) expect(&sh.bar[par], (unsigned)(16 * C) + L.boundary_bytes());
    // the momentum factor this iteration's decision would take, fetched ahead
    const T fnext = lazy ? (T)0 : (T)d.factor(a, d.streak);
    T zn, vn, tn, bn, cacc;
    L.template iterate<!lazy>(sW, sY, sH, sX, f, !lazy && momentum, sync, zn, vn, tn, bn, cacc);
    if (SC != kCta && sh.fail) break;  // set before the iteration's first barrier, if at all: uniform
    if (SC == kCluster) L.push_boundary(sh, par, r, zn, vn, tn, bn);
    if (lazy) {
      if (it + 1 < a.max_iters && !__syncthreads_or(detsum::large(zn, vn, tn, bn))) {
        L.zc = zn; L.vc = vn; L.tc = tn; L.bc = bn;
        continue;
      }
      cacc = L.owned ? L.share(tn - L.tc, bn - L.bc, zn - L.zc, vn - L.vc) : (T)0;
    }
    // ---- c: by warp 0, the others read it (their integer sums take longer than one more barrier) ----
    detsum::Fx sum = detsum::warp_sum(cacc);
    if (lane == 0) sh.warp[warp] = packed(sum);
    __syncthreads();
    if (warp == 0) {
      sum = detsum::warp_sum(unpacked(sh.warp[lane]));  // {0, kZero} beyond the CTA's warps
      if (SC == kCluster) {
        if (lane < C)
          push(remote(smem_addr(&sh.share[par][r]), lane), remote(smem_addr(&sh.bar[par]), lane), sum);
        if (!bar_wait(smem_addr(&sh.bar[par]), (unsigned)(it >> 1) & 1u)) sh.fail = 1;
        sum = detsum::warp_sum(lane < C ? unpacked(sh.share[par][lane]) : detsum::Fx{0ull, detsum::kZero});
      }
      const double cn = detsum::to_double(sum);
      if (lane == 0) sh.cn = cn;
    }
    __syncthreads();
    const double cn = sh.cn;
    bool take = false, stop;
    if (lazy) {  // here on the last iteration, or for a c that may not be finite
      d.cval = d.unit_rho ? cn : cn * d.rho;
      d.iters = it + 1;
      stop = it + 1 >= a.max_iters;
      if (!detsum::finite(d.cval)) {
        d.status = kNonFinite; stop = true;
      }
    } else {
      const bool high = d.streak > 0;
      stop = d.step(a, j, it, cn, take);
      momentum = take && high;
      f = take ? fnext : (T)0;
    }
    // ---- the new iterate becomes the current one; halo slots take theirs from the landing ----
    if (SC == kCluster && L.active && !L.owned) L.land(sh, par, zn, vn, tn, bn);
    if (!lazy) {
      L.zp = L.zc; L.vp = L.vc; L.tp = L.tc; L.bp = L.bc;
    }
    L.zc = zn; L.vc = vn; L.tc = tn; L.bc = bn;
    if (stop) break;
  }
  if (SC != kCta) {
    __syncthreads();
    if (sh.fail) d.status = kTimeout;
  }
  L.store(a, pl, j);
  if (r == 0 && tid == 0) d.store(a, j);
  if (SC == kCluster) cg::this_cluster().sync();  // no CTA leaves with a push to it in flight
}

inline int reg_class(int n) { return n <= 4 ? 4 : (n <= 8 ? 8 : 16); }

template <typename T, int SC, int kMode>
const void *pick_kernel(int NM, bool crowded) {
  if constexpr (sizeof(T) == 4 && SC == kCta)
    if (crowded && NM == 8) return (const void *)reg_kernel<T, 8, SC, kMode, 2>;
  return NM == 4   ? (const void *)reg_kernel<T, 4, SC, kMode, 1>
         : NM == 8 ? (const void *)reg_kernel<T, 8, SC, kMode, 1>
                   : (const void *)reg_kernel<T, 16, SC, kMode, 1>;
}

template <typename T, int SC>
const void *pick_spec(int NM) {
  return NM == 4   ? (const void *)spec_kernel<T, 4, SC>
         : NM == 8 ? (const void *)spec_kernel<T, 8, SC>
                   : (const void *)spec_kernel<T, 16, SC>;
}

// The launch of one solve.
template <typename T>
cudaError_t reg_launch_t(const AdmmLaunch &s, const RegLaunch &rl, cudaStream_t stream) {
  Args<T> a = ls::make_args<T>(s);
  a.eps = s.eps + 0.0;  // -0 becomes +0: the stop test compares bit patterns
  cudaError_t rc;
  if (s.max_iters <= 0) {  // nothing to iterate: the starting iterates are the result
    rc = cudaMemcpyAsync(s.old_base, s.base, sizeof(int) * s.L.batch, cudaMemcpyDeviceToDevice, stream);
    if (rc != cudaSuccess) return rc;
    const int n_init = s.L.batch > s.nitems ? s.L.batch : s.nitems;
    ls::solve_init_kernel<T><<<(n_init + 255) / 256, 256, 0, stream>>>(a, s.warm);
    if ((rc = cudaGetLastError()) != cudaSuccess) return rc;
    if (s.warm != 1) {
      ls::prepare_kernel<T><<<dim3(8, s.L.batch), 256, 0, stream>>>(a, s.warm, s.old_base);
      if ((rc = cudaGetLastError()) != cudaSuccess) return rc;
    }
    ls::output_kernel<T><<<dim3(4, s.L.batch), 256, 0, stream>>>(a, s.u_out, s.x_out);
    return cudaGetLastError();
  }
  int dev = 0, nsm = 0;
  if ((rc = cudaGetDevice(&dev)) != cudaSuccess) return rc;
  if ((rc = cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess) return rc;
  const int cls = reg_class(rl.nmax);
  // A batch that leaves every CTA an SM runs the deciding warp beside the others; one that does not
  // has other CTAs to run meanwhile.
  const bool watch = s.stall_win > 0 || s.mask != nullptr;
  const bool lazy = !s.accel && s.eps < 0.0 && !watch;
  if constexpr (sizeof(T) == 4)  // a thread per stage is the faster one at every batch and horizon
    if (lazy && rl.stage_class >= 0)
      return launch_stage(s, rl.stage_class, rl.stage_threads, stream);
  const bool crowded = (int64_t)s.L.batch * rl.C > nsm || rl.threads + 32 > spec_max_threads((int)sizeof(T), cls);
  const bool spec = rl.C > 16 || (!crowded && !(lazy && rl.C == 1));
  const void *kernel = spec ? (rl.C == 1    ? pick_spec<T, kCta>(cls)
                               : rl.C <= 16 ? pick_spec<T, kCluster>(cls)
                                            : pick_spec<T, kGrid>(cls))
                       : rl.C > 1 ? pick_kernel<T, kCluster, kSolo>(cls, false)
                       : lazy     ? pick_kernel<T, kCta, kLazy>(cls, crowded)
                                  : pick_kernel<T, kCta, kSolo>(cls, crowded);
  const size_t smem = (size_t)4 * rl.region * sizeof(T);
  rc = allow_smem(kernel, smem);
  if (rc != cudaSuccess) return rc;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(s.L.batch * rl.C);
  cfg.blockDim = dim3(rl.threads + (spec ? 32 : 0));
  cfg.dynamicSmemBytes = smem;
  cfg.stream = stream;
  cudaLaunchAttribute attr[1];
  cfg.attrs = attr;
  cfg.numAttrs = rl.C > 1 ? 1 : 0;
  if (rl.C > 16) {  // all CTAs resident at once; records of an earlier solve are cleared
    rc = cudaMemsetAsync(rl.xch, 0, rl.xch_bytes, stream);
    if (rc != cudaSuccess) return rc;
    attr[0].id = cudaLaunchAttributeCooperative;
    attr[0].val.cooperative = 1;
  } else if (rl.C > 1) {
    if (rl.C > 8) {
      rc = cudaFuncSetAttribute(kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
      if (rc != cudaSuccess) return rc;
    }
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = rl.C;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
  }
  RegPlan pl{rl.C, rl.region, (ulonglong2 *)rl.xch, s.u_out, s.x_out, s.warm};
  void *params[] = {&a, &pl};
  return cudaLaunchKernelExC(&cfg, kernel, params);
}

}  // namespace

}  // namespace pimpc

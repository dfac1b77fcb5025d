// admm_dense.cu -- Algorithm 1 in FP64 on plain stage blocks with every lane of a warp at work
// (schedule family 0, FP64 iterations on box constraints; the lane-group kernel of admm.cu keeps
// FP32 iterations and non-box input sets).
//
// The FP64 pipe bounds FP64 iterations: it takes a warp-wide instruction every 19 cycles per SM
// (measured) whatever the number of active lanes, so a warp that gives a stage of n = 19 components
// 32 lanes pays for 13 idle ones, and each of the few dozen elementwise operations of steps 2-4
// costs as much as a multiply-add of the products. Here thread t owns component t mod n of stage
// t / n of a sub-chunk (a CTA of 256 threads holds 256 / n slots: S stages and the next one), the
// short products with nu outputs run on cnt * nu consecutive threads, and the elementwise part is
// the reduced form of admm_reg.cuh: lambda = -beta (steps 2-3 give beta' + lambda' = 0, and the
// hats are linear), sums folded into the starts of the dot products, x / 3 in two operations,
// clamps on bit patterns, and the share of c summed in integers (detsum.cuh). About 104 FP64
// instructions per component at n = 19 instead of 150, on full warps: 256 uneven instances (70k
// stages) take 0.35 ms per iteration instead of 0.70.
//
// Items, the halo stage before an item, the queue, the grid barrier and the pass over the instances
// are those of admm.cu. Stage blocks arrive by cp.async.bulk (one buffer; the other CTAs of the SM
// compute meanwhile), the iterates go from L2 straight into their threads' registers.
#include <algorithm>

#include "bulk.cuh"
#include "detsum.cuh"
#include "lockstep.cuh"
#include "regvec.cuh"

namespace pimpc {

namespace {

using ls::kWaitLimit;
using namespace bulk;

constexpr int kThreads = 256;

struct Plan {
  int blk, halo, vec;  // doubles: stage blocks, halo (or LTI) blocks, one vector region
};

// Words of a stage's G and e, rounded to 16 bytes (what the next stage contributes to a sub-chunk).
__host__ __device__ inline int ge_words(int nx, int n) { return (nx * odd_ld(n) + nx + 1) & ~1; }

// sum_r m[r * ld] v[r], r < cnt, from init: v 16-byte aligned in shared memory, broadcast reads.
__device__ __forceinline__ double dot_strided(const double *m, int ld, const double *v, int cnt, double init) {
  double a = init;
  int r = 0;
  for (; r + 1 < cnt; r += 2) {
    const double2 q = *reinterpret_cast<const double2 *>(v + r);
    a = fma(m[r * ld], q.x, a);
    a = fma(m[(r + 1) * ld], q.y, a);
  }
  if (r < cnt) a = fma(m[r * ld], v[r], a);
  return a;
}

// (S x)_c for a symmetric m x m matrix stored as wrapped diagonals (see products.cuh), one chain.
__device__ __forceinline__ double sym_dot(const double *D, const double *x, int m, int c) {
  double a = D[c] * x[c];
  const int half = (m - 1) / 2;
  int ip = c, im = c;
  const double *row = D;
  for (int d = 1; d <= half; ++d) {
    row += m;
    ip = (ip + 1 == m) ? 0 : ip + 1;
    im = (im == 0) ? m - 1 : im - 1;
    a = fma(row[c], x[ip], a);
    a = fma(row[im], x[im], a);
  }
  if ((m & 1) == 0) {
    row += m;
    a = fma(row[c], x[c + m / 2 < m ? c + m / 2 : c - m / 2], a);
  }
  return a;
}

__global__ void __launch_bounds__(kThreads, 3) dense_kernel(ls::Args<double> a, Plan pl) {
  extern __shared__ __align__(128) unsigned char smem_raw[];
  __shared__ __align__(8) uint64_t mbar;
  __shared__ int sItem, sOk, sArr, sRed[kThreads / 32];
  __shared__ ulonglong2 sSum[32];
  double *sm = reinterpret_cast<double *>(smem_raw);
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const unsigned nblocks = gridDim.x;
  Ctl *ctl = a.ctl;
  const int lti = a.L.lti;
  double *rB = sm, *rHalo = rB + pl.blk;
  double *sW = rHalo + pl.halo, *sY = sW + pl.vec, *sH = sY + pl.vec, *sX = sH + pl.vec,
         *sT = sX + pl.vec, *sD = sT + pl.vec;

  if (tid == 0) {
    mbar_init(&mbar, 1);
    fence_mbar_init();
  }
  if (tid < 32) sSum[tid] = make_ulonglong2(0, (unsigned long long)(long long)detsum::kZero);
  __syncthreads();
  uint32_t parity = 0u;
  bool pend = false;

  int cl = 0;
  for (int it = 0; it < a.max_iters; ++it) {
    const int nact = *(volatile int *)&ctl->nlist[cl];
    bool ok = true;
    for (;;) {
      if (tid == 0) sItem = atomicAdd(&ctl->queue[it & 1], 1);
      __syncthreads();
      const int q = sItem;
      __syncthreads();
      if (q >= nact) break;
      const int item = a.list[cl][q];
      if (item < 0) continue;  // an entry of an instance that has stopped
      const int j = a.item_inst[item];
      if (*(volatile int *)&a.stop[j]) continue;
      const int ka = a.item_a[item], kb = a.item_b[item];
      const int nx = a.L.nx[j], nu = a.L.nu[j], N = a.L.N[j], n = nx + nu;
      const int S = a.grp[j] - 1;  // stages per sub-chunk; slot S serves the halo
      const int nv = (n + 1) & ~1, nuv = (nu + 1) & ~1;
      const int n5p = ls::iter_stride_plain(n, 8);
      const int W = a.L.W[j], ldg = odd_ld(n);
      const int oE = nx * ldg, oH = oE + nx, oM = oH + wrapped_size(n);
      const int bse = a.base[j];
      const int64_t ib = a.L.Ni[j];
      const double *Ic = a.it[(bse + it) % 3] + ib;
      const double *Ip = a.it[(bse + it + 2) % 3] + ib;
      double *In = a.it[(bse + it + 1) % 3] + ib;
      const double *blk = a.blk + a.L.blk[j];
      const double f = *(volatile double *)&a.coef[j];
      const bool use_prev = f != 0.0;
      const double rho = a.rho;
      const double *ref = a.ref ? (a.ref + (a.ref_per_stage ? a.L.Nn[j] : a.L.off_n[j])) : nullptr;
      const int refstride = a.ref_per_stage ? n : 0;
      const int slot = tid / n, c = tid - slot * n;
      const bool lane_ok = slot <= S;
      const int ts = tid / nu, tq = tid - ts * nu;  // the products with nu outputs: stage, input
      double lo = 0.0, hi = 0.0, qd = 0.0;
      if (lane_ok) {
        lo = a.lo[a.L.off_n[j] + c];
        hi = a.hi[a.L.off_n[j] + c];
        if (ref) qd = a.qd[a.L.off_n[j] + c];
      }
      double cacc = 0.0;

      // Copies of the sub-chunk that starts at stage k0 (thread 0 issues).
      auto issue = [&](int k0, bool first) {
        const int cnt = min(S, kb - k0);
        const int la = (k0 + cnt < N) ? 1 : 0;  // the next stage: its G and e only
        const uint32_t bytes = (uint32_t)((cnt * W + la * ge_words(nx, n)) * sizeof(double));
        const bool halo = first && ka > 0 && !lti;
        const uint32_t extra = halo ? (uint32_t)(W * sizeof(double))
                                    : (lti && first ? (uint32_t)(2 * W * sizeof(double)) : 0u);
        const uint32_t all = (lti ? 0u : bytes) + extra;
        mbar_expect_tx(&mbar, all);
        if (!lti) bulk_load(rB, blk + (int64_t)k0 * W, bytes, &mbar);
        if (halo) bulk_load(rHalo, blk + (int64_t)(ka - 1) * W, extra, &mbar);
        if (lti && first) bulk_load(rHalo, blk, extra, &mbar);
      };

      const int nsub = (kb - ka + S - 1) / S;
      for (int sc = 0; sc < nsub; ++sc) {
        const int k0 = ka + sc * S;
        const int cnt = min(S, kb - k0);
        const int la = (k0 + cnt < N) ? 1 : 0;
        const bool copies = !lti || sc == 0;
        if (copies) {  // the buffer is free: the barrier that ended the last sub-chunk
          if (tid == 0) issue(k0, sc == 0);
          pend = true;
        }
        if (!lti && sc + 1 < nsub && tid == 0) {  // the next sub-chunk's blocks into L2
          const int k1 = k0 + S, c1 = min(S, kb - k1);
          bulk_prefetch_l2(blk + (int64_t)k1 * W, (uint32_t)(c1 * W * sizeof(double)));
        }
        // Hats of this thread's component, from L2, while the copies fly: stages k0 .. k0 + cnt
        // (the next one included), and the stage before the item on slot S.
        const bool halo = sc == 0 && ka > 0;
        const bool owned = lane_ok && slot < cnt;
        const bool next = la && slot == cnt && slot <= S;
        const bool before = halo && slot == S;
        const int k = k0 + slot;
        double zh = 0.0, vh = 0.0, th = 0.0, bh = 0.0;
        if (owned || next) {
          const double *h = Ic + (int64_t)k * n5p + c;
          zh = __ldcg(h);
          vh = __ldcg(h + n);
          th = __ldcg(h + 2 * n);
          bh = __ldcg(h + 3 * n);
          if (use_prev) {
            const double *p = Ip + (int64_t)k * n5p + c;
            zh += f * (zh - __ldcg(p));
            vh += f * (vh - __ldcg(p + n));
            th += f * (th - __ldcg(p + 2 * n));
            bh += f * (bh - __ldcg(p + 3 * n));
          }
        }
        double zm = 0.0;  // slot S: z - theta of stage ka - 1
        if (before) {
          const double *h = Ic + (int64_t)(ka - 1) * n5p + c;
          double z = __ldcg(h), t = __ldcg(h + 2 * n);
          if (use_prev) {
            const double *p = Ip + (int64_t)(ka - 1) * n5p + c;
            z += f * (z - __ldcg(p));
            t += f * (t - __ldcg(p + 2 * n));
          }
          zm = z - t;
        }
        double qr = 0.0, qrm = 0.0;
        if (ref && owned) qr = qd * ref[(int64_t)k * refstride + c];
        if (ref && before) qrm = qd * ref[(int64_t)(ka - 1) * refstride + c];
        if (copies) {
          // One thread waits on the copies; the others wait at the barrier without issuing.
          if (tid == 0) sArr = mbar_wait(&mbar, parity, ctl) ? 1 : 0;
          __syncthreads();
          if (!sArr) { ok = false; break; }  // may still be in flight: pending for the exit wait
          parity ^= 1u;
          pend = false;
        }
        const double *Gk = lti ? rHalo : rB + slot * W;              // G_k, e_k, M_k of the thread's stage
        const double *Gk1 = lti ? rHalo : rB + (slot + 1) * W;       // G_{k+1}
        const double *Hk = (lti ? rHalo + ((k < N - 1) ? 0 : W) : Gk) + oH;
        // ---- w = v - beta, y = z - v - beta - ebar ----
        if (owned || next) {
          if (owned) sW[slot * nv + c] = vh - bh;
          sY[slot * nv + c] = (zh - vh) - (bh + (c < nx ? Gk[oE + c] : 0.0));
        }
        if (tid < n) sX[tid] = sc > 0 ? sX[S * nv + tid] : (ka == 0 ? a.xb0[a.L.off_n[j] + tid] : 0.0);
        __syncthreads();
        // ---- t = B^T w_x + w_u; h = Qbar ref + rho (z - theta + Abar_{k+1}^T y_{k+1}) ----
        if (ts < cnt) {
          const double *G = lti ? rHalo : rB + ts * W;
          sT[ts * nuv + tq] = dot_strided(G + nx + tq, ldg, sW + ts * nv, nx, sW[ts * nv + nx + tq]);
        }
        if (owned || before) {
          const bool more = before || k + 1 < N;
          const double *y = sY + (before ? 0 : slot + 1) * nv;
          const double *G = before ? (lti ? rHalo : rB) : Gk1;
          double acc = before ? zm : zh - th;
          if (more) {
            if (c >= nx) acc += y[c];
            acc = dot_strided(G + c, ldg, y, nx, acc);
          }
          sH[slot * nv + c] = (before ? qrm : qr) + rho * acc;
        }
        __syncthreads();
        // ---- du = M t; xbar_{k+1} = H h ----
        if (ts < cnt) {
          const double *M = (lti ? rHalo : rB + ts * W) + oM;
          sD[ts * nuv + tq] = sym_dot(M, sT + ts * nuv, nu, tq);
        }
        double xb = 0.0;
        if (owned) {
          xb = sym_dot(Hk, sH + slot * nv, n, c);
          sX[(slot + 1) * nv + c] = xb;
        } else if (before) {  // xbar_ka = H_{ka-1} h_{ka-1}
          sX[c] = sym_dot(rHalo + oH, sH + slot * nv, n, c);
        }
        __syncthreads();
        // ---- steps 2-4 ----
        if (owned) {
          const double *xk = sX + slot * nv, *du = sD + slot * nuv;
          double bd, ax;  // Bbar du, Abar xbar + ebar
          if (c < nx) {
            const double *row = Gk + c * ldg;  // odd stride: the lanes' rows hit distinct banks
            ax = dot_strided(row, 1, xk, n, Gk[oE + c]);
            bd = dot_strided(row + nx, 1, du, nu, 0.0);
          } else {
            ax = xk[c];
            bd = du[c - nx];
          }
          const Step<double> r = steps23(xb, bd, ax, th, bh, lo, hi);
          double *o = In + (int64_t)k * n5p + c;
          o[0] = r.z;
          o[n] = r.v;
          o[2 * n] = r.t;
          o[3 * n] = r.b;
          o[4 * n] = negated(r.b);
          // theta' - theta = xbar - z' and beta' - beta = Bbar du - v', without the duals' own rounding
          const double d1 = xb - r.z, d2 = bd - r.v, d4 = r.z - zh, d5 = r.v - vh;
          // d1^2 + d2^2 + d3^2 + d4^2 + d5^2 + (d4 - d5)^2 with d3 = -d2
          const double g = d2 * d2 + (d4 * d4 + d5 * (d5 - d4));
          cacc = fma(d1, d1, fma(2.0, g, cacc));
        }
        __syncthreads();
      }
      if (!ok) break;
      // ---- step 4: this item's share of c (steps 5-7 follow in the pass after the barrier) ----
      detsum::Fx sum = detsum::warp_sum(cacc);
      if (lane == 0) sSum[warp] = make_ulonglong2(sum.sig, (unsigned long long)(long long)sum.e);
      __syncthreads();
      if (warp == 0) {
        const ulonglong2 t = sSum[lane];  // {0, kZero} beyond the CTA's warps
        sum = detsum::warp_sum(detsum::Fx{t.x, (int)t.y});
        if (lane == 0) a.cpart[item] = detsum::to_double(sum);
      }
    }
    if (blockIdx.x == 0 && tid == 0) ctl->queue[(it + 1) & 1] = 0;
    if (!ls::grid_sync(ctl, nblocks, &sOk)) break;
    if (!ls::finish_pass(a, it, cl, nblocks, &sOk)) break;
    if (*(volatile int *)&ctl->active <= 0) break;
    if (!ls::compact(a, cl, nact, &sOk, sRed)) break;
  }
  // Never leave a bulk copy in flight into shared memory: wait (bounded) for a pending phase.
  if (pend) {
    long long k = 0;
    while (!mbar_try_wait(&mbar, parity) && ++k < kWaitLimit) {
    }
  }
}

}  // namespace

// Slots of a sub-chunk (S stages and one more) for an instance, and the plan's regions in doubles.
static int64_t dense_words(int nx, int nu, int W, int lti, int SL, int *blk, int *halo, int *vec) {
  const int n = nx + nu, nv = (n + 1) & ~1;
  *blk = lti ? 0 : (SL - 1) * W + ge_words(nx, n);
  *halo = lti ? 2 * W : W;
  *vec = (SL + 1) * nv;
  auto up = [](int v) { return (v + 15) & ~15; };
  *blk = up(*blk);
  *halo = up(*halo);
  *vec = up(*vec);
  return (int64_t)*blk + *halo + 6 * (int64_t)*vec;
}

// Slots per sub-chunk of each instance, at least two stages' worth, within a third of an SM's shared
// memory, and the launch's regions. Each region is the largest over the instances, so that a batch of
// one size runs three CTAs per SM, as the kernel is compiled for, and one of many sizes may run two (the
// 256 uneven instances: 82,688 bytes, two CTAs). False if an instance does not fit, or if a CTA's
// threads give one fewer than five slots (n > 51): with four a quarter of them hold the next stage,
// and the lane groups win (304 stage-invariant instances, N 200: n 48, five slots, 1.70 ms per
// iteration in lane groups, 1.12 here; n 56 1.95 and 2.63; 256 of n 64, N 1000 11.9 and 13.7).
bool dense_plan(int batch, const int *nx, const int *nu, const int *W, int lti, int64_t smem_sm,
                int64_t optin, int *slots, int *plan, size_t *smem) {
  plan[0] = plan[1] = plan[2] = 0;
  for (int j = 0; j < batch; ++j) {
    int SL = kThreads / (nx[j] + nu[j]), b, h, v;
    if (SL < 5) return false;
    while (SL > 2 && dense_words(nx[j], nu[j], W[j], lti, SL, &b, &h, &v) * 8 > smem_sm / 3 - 2048) --SL;
    dense_words(nx[j], nu[j], W[j], lti, SL, &b, &h, &v);
    slots[j] = SL;
    plan[0] = std::max(plan[0], b);
    plan[1] = std::max(plan[1], h);
    plan[2] = std::max(plan[2], v);
  }
  *smem = sizeof(double) * ((size_t)plan[0] + plan[1] + 6 * (size_t)plan[2]);
  return (int64_t)*smem + 4096 <= optin;
}

int dense_threads() { return kThreads; }

cudaError_t dense_configure(size_t smem, int *blocks_per_sm) {
  const cudaError_t rc = allow_smem((const void *)dense_kernel, smem);
  if (rc != cudaSuccess) return rc;
  return cudaOccupancyMaxActiveBlocksPerMultiprocessor(blocks_per_sm, dense_kernel, kThreads, smem);
}

cudaError_t launch_dense(const AdmmLaunch &s, const int *plan, size_t smem, cudaStream_t stream) {
  ls::Args<double> a = ls::make_args<double>(s);
  Plan pl{plan[0], plan[1], plan[2]};
  void *params[] = {&a, &pl};
  return ls::launch_sequence<double>(s, a, (const void *)dense_kernel, params, smem, stream);
}

}  // namespace pimpc

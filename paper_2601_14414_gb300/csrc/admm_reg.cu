// admm_reg.cu -- planning of the register-resident schedule and its FP32 kernels (admm_reg.cuh).
#include "admm_reg.cuh"
#include "stage_reg.cuh"

namespace pimpc {

cudaError_t launch_reg64(const AdmmLaunch &s, const RegLaunch &rl, cudaStream_t stream);

// Threads and shared memory of one CTA for C CTAs per instance; 0 threads: the batch does not fit
// (an n above 16, fewer stages than CTAs, or more stages per CTA than its threads hold).
void reg_plan(int batch, const int *nx, const int *nu, const int *N, int precision, RegLaunch *rl) {
  const int ts = precision == 0 ? 4 : 8, C = rl->C;
  int thr = 0, reg = 0, nm = 1;
  for (int j = 0; j < batch; ++j) nm = std::max(nm, nx[j] + nu[j]);
  rl->threads = 0;
  if (nm > kMaxN || C > kMaxC) return;
  const int cls = reg_class(nm);  // more CTAs than a cluster: with the deciding warp
  const int cap = C > 16 ? spec_max_threads(ts, cls) - 32 : reg_max_threads(ts, cls);
  for (int j = 0; j < batch; ++j) {
    const int n = nx[j] + nu[j];
    if (N[j] < C) return;
    const int slots = (N[j] + C - 1) / C + (C > 1 ? 2 : 0);
    if ((int64_t)slots * n > cap) return;
    thr = std::max(thr, slots * n);
    reg = std::max(reg, (slots + 1) * reg_nv(n, ts));
  }
  rl->threads = (thr + 31) / 32 * 32;
  rl->region = (reg + 3) / 4 * 4;
  rl->nmax = nm;
  rl->xch_bytes = C > 16 ? sizeof(ulonglong2) * xch_records(C) * (size_t)batch : 0;
}

// The resident schedule in registers (n <= 16): CTAs per instance, 0 threads if it does not fit.
// With item_scale = 0 one CTA as long as its threads stay within `one`: in FP32 what the kernel with a
// deciding warp holds (n 6, N 60: 0.83 us per iteration on one CTA of 384 threads, 1.13 on two), in
// FP64 four warps, one per scheduler, because a fifth queues for the FP64 pipe (n 6, N 60: 8.0 us on
// one CTA, 3.3 on four; N 20, four warps: 3.03 on one and on two). Else the smallest cluster whose CTAs
// stay within `few` threads (FP32, n 16, N 50: 1.25 us with 256 threads, 1.19 with 160, 1.18 with 96),
// the cluster of 16 within `most`, and beyond that (FP64, whose iterations are long enough to pay for
// an exchange through global memory, or instances that no cluster holds) the fewest CTAs within
// `grid` (n 16, N 200, FP64: 7.15 us on a cluster of 16, 4.93 on 32 CTAs of 160 threads, 4.73 on 40 of
// 128, 4.72 on 64; n 3, N 5000: 4.12 on 96, 3.65 on 128; n 16, N 100: 4.67 on the cluster and on 32).
// Batches larger than the SMs take the fewest CTAs that hold an instance; clusters of 5 and 6 only where
// they make two and a half rounds of CTAs or more, because the GPCs hold them unevenly (FP64, n 16, 30
// iterations, the shared-memory kernel / 8 / 5 or 6 CTAs: N 60, 76 instances 908 / 1051 / 667 us, 304 3557 /
// 3664 / 2425; N 80, 76 1120 / 1176 / 981; FP32, n 16, N 121, 76 369 / 389 / 215; N 70, 60 instances 1102 /
// 709 / 737).
static RegLaunch choose_reg(int item_scale, int batch, const int *nx, const int *nu, const int *N,
                            int precision, int nsm) {
  const bool f32 = precision == 0;
  const int one = f32 ? 480 : 128, few = f32 ? 160 : 128, most = f32 ? 1024 : 160, grid = f32 ? 512 : 128;
  RegLaunch best;
  for (int cand : {1, 2, 4, 5, 6, 8, 16, 24, 32, 40, 48, 64, 80, 96, 112, 128, 144}) {
    if (item_scale > 0 && cand != item_scale) continue;
    if ((cand == 5 || cand == 6) && (item_scale > 0 || 2 * (int64_t)batch * cand < 5 * (int64_t)nsm)) continue;
    RegLaunch t;
    t.C = cand;
    reg_plan(batch, nx, nu, N, precision, &t);
    if (t.threads == 0) continue;
    if ((best.threads > 0 || cand > 16) && (int64_t)batch * cand > nsm) break;
    best = t;
    if (t.threads <= (cand == 1 ? one : cand < 16 ? few : cand == 16 ? most : grid)) break;
  }
  return best;
}

// Plans the resident schedule (family 3): the shared-memory kernel's cluster size, regions and
// bytes per CTA, and the register kernel's launch where every instance has n <= 16. False if the
// instances do not fit the shared memory of a cluster (of item_scale CTAs, if that is not 0), or
// one has fewer stages than its CTAs.
// With item_scale = 0: the fewest CTAs that fit, or, when the whole batch occupies few SMs (latency,
// not throughput, is what a small batch needs), the most CTAs (up to 16) that still give every
// CTA four stages or more.
bool plan_resident(int item_scale, int batch, const int *nx, const int *nu, const int *N,
                   const int *W, int lti, int precision, int nsm, size_t optin, int *res,
                   size_t *smem, RegLaunch *reg) {
  const int thr = res_threads(precision), ts = precision == 0 ? 4 : 8;
  const int nmin = *std::min_element(N, N + batch);
  int fewest = 0, most = 0, plan[6], p_few[6], p_most[6];
  size_t b_few = 0, b_most = 0;
  for (int cand : {1, 2, 4, 8, 16}) {
    if (item_scale > 0 && cand != item_scale) continue;
    const size_t b = res_plan(batch, nx, nu, N, W, lti, precision, thr, cand, plan);
    if (b == 0 || b + 1024 > optin - 256) continue;
    if (fewest == 0) { fewest = cand; b_few = b; std::copy(plan, plan + 6, p_few); }
    if (item_scale > 0 || (nmin >= 4 * cand && (int64_t)batch * cand <= nsm)) {
      most = cand; b_most = b; std::copy(plan, plan + 6, p_most);
    }
  }
  if (fewest == 0) return false;
  const bool wide = most >= fewest;
  std::copy(wide ? p_most : p_few, (wide ? p_most : p_few) + 6, res);
  *smem = wide ? b_most : b_few;
  // what the shared-memory kernel accepts, in registers where n <= 16 allows it
  *reg = choose_reg(item_scale, batch, nx, nu, N, precision, nsm);
  if (reg->threads > 0) *smem = (size_t)4 * reg->region * ts;
  if (reg->threads > 0 && precision == 0 && item_scale <= 1) {
    const int mx = *std::max_element(nx, nx + batch), mu = *std::max_element(nu, nu + batch);
    const int mN = *std::max_element(N, N + batch);
    if (stage::size_class(mx, mu) >= 0 && mN <= kStageThreads) {
      reg->stage_class = stage::size_class(mx, mu);
      reg->stage_threads = (mN + 31) / 32 * 32;
    }
  }
  return true;
}

cudaError_t launch_reg(const AdmmLaunch &s, int precision, const RegLaunch &rl, cudaStream_t stream) {
  return precision == 0 ? reg_launch_t<float>(s, rl, stream) : launch_reg64(s, rl, stream);
}

}  // namespace pimpc

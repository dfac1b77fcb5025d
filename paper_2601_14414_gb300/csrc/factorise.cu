// factorise.cu -- the per-stage cache of Algorithm 1 ("cache J_k and H_k"), computed in FP64.
//
// For stage k (LTV) the warp forms
//   K = Qbar + rho I + rho Abar_{k+1}^T Abar_{k+1}   (k < N-1),   K = Qbar + rho I   (k = N-1),
// where Abar^T Abar = G^T G + diag(0, I_nu) with G = [A | B] (Theorem 2's velocity form), and
// writes H_k = K^{-1}, inverted by sweeps of the symmetric matrix (Gauss-Jordan elimination in
// pivot order, which needs no pivoting for a positive definite K). It also writes
// M_k = (B_k^T B_k + I + Wdu / rho)^{-1}, so that the du update of Algorithm 1 step 1,
// J_k (v - beta) with J_k = (Bbar^T Bbar)^{-1} Bbar^T, is M_k (B_k^T (v - beta)_x + (v - beta)_u);
// and it copies G_k and e_k into the stage block.
// Outputs are converted to the iteration precision T. LTI instances have two blocks: block 0
// with H = (Qbar + rho I + rho Abar^T Abar)^{-1} and block 1 with the terminal H_{N-1}.
//
// Bound by the FP64 pipe, which takes a warp-wide instruction every 19 cycles per SM (64 per
// scheduler, and 64 cycles of latency), whatever the number of active lanes: everything but the
// multiply-adds of the Gram matrix and of the sweeps is kept off it. The reciprocal of a pivot
// starts from the FP32 one and takes three FP64 instructions instead of a division's dozen or
// so, signs and pivot tests work on bit patterns, and kLanes lanes work on one stage, so that a
// warp's per-pivot instructions (reciprocal, scaled column) serve 32 / kLanes stages at once. A
// small batch, which leaves schedulers idle, takes two whole warps per stage instead, one for H and
// one for M and the copies, with all rows of G at once: there the chain of one stage is what counts.
// 1.13M stages of the batched workload (nx 4 .. 24, nu 2 .. 8): 56.5 ms with a warp per stage,
// divisions and all of G in shared memory, 26.4 ms so (the FP64 pipe busy 83 % of its nominal
// rate, which is what it sustains; the multiply-adds alone would take 17). 5000 stages of n = 3:
// 27.9 and 9.6 us.
#include <algorithm>

#include "bl_slot.cuh"
#include "launch.h"

namespace pimpc {

namespace {

struct FactArgs {
  Layout L;
  const double *A, *B, *e;   // FP64 dynamics, user layout
  const double *qd;          // [sum n] Qbar diagonal in FP64
  const double *rdu;         // [sum n] with the W_du diagonal at the input slots (or null)
  double rho;
  const int *binst;          // instance of each global block
  const int64_t *bbase;      // first global block of each instance
  int64_t nblocks;
  int words_per_stage;       // shared-memory doubles per stage (per part of one, kParts == 2)
  int rows;                  // rows of G held at a time
  int tab_len, tab_words;    // entries of the triangle table, and its doubles
  int *err;                  // [batch]: set to 1 for an instance with a non-positive pivot
};

// Row i and column c <= i of the t-th lower-triangle entry in row-major order
// (t = i (i + 1) / 2 + c). The CTA tabulates them (i << 8 | c) once: every size enumerates its
// triangle in the same order, and a warp that stepped the indices entry by entry diverged.
__device__ __forceinline__ unsigned short tri_entry(int t) {
  int i = (int)((sqrtf(8.0f * (float)t + 1.0f) - 1.0f) * 0.5f);
  while (i * (i + 1) / 2 > t) --i;
  while ((i + 1) * (i + 2) / 2 <= t) ++i;
  return (unsigned short)(i << 8 | (t - i * (i + 1) / 2));
}

__device__ __noinline__ double divided(double a) { return 1.0 / a; }

// 1 / a for a normal positive a away from the ends of the exponent range (else the division): the
// FP32 reciprocal r of a's significand (relative error e0 <= 2^-22) scaled by a's exponent, then
// one third-order Newton step x = r (1 + e + e^2), e = 1 - a r, whose error is e0^3 and a rounding.
__device__ __forceinline__ double reciprocal(double a) {
  const unsigned long long bits = (unsigned long long)__double_as_longlong(a);
  const int ex = (int)(bits >> 52);
  if (ex < 4 || ex > 2040) return divided(a);  // a NaN, infinite, tiny, huge or negative
  const float m = __uint_as_float(0x3f800000u | ((unsigned)(bits >> 29) & 0x7fffffu));  // [1, 2)
  const unsigned rb = __float_as_uint(__frcp_rn(m));                                    // (1/2, 1]
  const long long x0 = ((long long)(rb >> 23) - 127 + 1023 - (ex - 1023)) << 52 |
                       (long long)(rb & 0x7fffffu) << 29;
  const double x = __longlong_as_double(x0);
  const double e = fma(-a, x, 1.0);
  return fma(x, fma(e, e, e), x);
}

// A value, or its negative, in the iteration precision: the sign is flipped as a bit of the
// stored word (a negation of a double is an FP64 instruction).
__device__ __forceinline__ void store(float *p, double v, bool neg) {
  *reinterpret_cast<unsigned *>(p) = __float_as_uint((float)v) ^ (neg ? 0x80000000u : 0u);
}
__device__ __forceinline__ void store(double *p, double v, bool neg) {
  *reinterpret_cast<long long *>(p) =
      __double_as_longlong(v) ^ (neg ? (long long)0x8000000000000000ull : 0ll);
}

// Rounds of kLanes lanes over cnt entries. Every lane runs all of them (lanes that leave a loop a
// round early run its unrolled remainder by themselves; the
// triangle, its table and the rows of G are padded so that the last round may run past the end).
template <int kLanes>
__device__ __forceinline__ int rounds(int cnt) {
  return (cnt + kLanes - 1) / kLanes;
}

// Slot of element (r, c) in a packed lower triangle.
__device__ __forceinline__ int tri_slot(int r, int c) {
  const int i = r > c ? r : c, j = r > c ? c : r;
  return i * (i + 1) / 2 + j;
}

// The negative inverse of the symmetric positive definite m x m matrix whose lower triangle is
// packed in S, by m sweeps of the symmetric matrix (Gauss-Jordan elimination with the pivots in
// order; for a positive definite matrix every pivot is positive, and a pivot that is not flags
// err): sweeping pivot k with d = 1 / a_kk sets a_ij -= a_ik a_kj d for i, j != k, a_ik = a_ik d,
// a_kk = -d; after all m sweeps the matrix holds -S^{-1}. kLanes lanes (gl = 0 .. kLanes - 1) share the
// entries (t = gl, gl + kLanes, ... in row-major order). col (2 m values) holds the pivot column
// and the column times d. mmax: the largest m of the stages of this warp, so that the warp stays
// together.
template <int kLanes>
__device__ void sweep_inverse(double *S, double *col, const unsigned short *tab, int m, int mmax,
                              int gl, int *err) {
  double *cold = col + m;
  const int tr = rounds<kLanes>(m * (m + 1) / 2), cr = rounds<kLanes>(m);
  for (int k = 0; k < mmax; ++k) {
    __syncwarp();
    double d = 1.0;
    if (k < m) {
      double akk = S[tri_slot(k, k)];
      const long long b = __double_as_longlong(akk);
      if (!(b > 0 && b <= 0x7ff0000000000000ll)) {  // not > 0, or NaN
        if (gl == 0) *err = 1;
        akk = 1.0;
      }
      d = reciprocal(akk);
      for (int q = 0, i = gl; q < cr; ++q, i += kLanes)
        if (i < m) {
          const double c = S[tri_slot(i, k)];
          col[i] = c;
          cold[i] = c * d;
        }
    }
    __syncwarp();
    if (k < m) {
      const double nd = __hiloint2double(__double2hiint(d) | (int)0x80000000, __double2loint(d));
      for (int q = 0, t = gl; q < tr; ++q, t += kLanes) {
        const int i = tab[t] >> 8, j = tab[t] & 0xff;
        // entry (i, j), j <= i: every lane runs the multiply-add, the pivot's row and column
        // select their values
        double v = fma(-col[i], cold[j], S[t]);
        if (i == k) v = (j == k) ? nd : cold[j];
        else if (j == k) v = cold[i];
        S[t] = v;
      }
    }
  }
  __syncwarp();
}

// Rows of G held at a time by large batches: with all of G, or with 8 rows, an SM holds too few warps
// to fill the FP64 pipe (batched workload: 8 warps 68 % busy, 12 warps 75 %, 16 warps 83 %, which is
// its limit at 19 cycles per instruction).
constexpr int kRows = 6;
constexpr int kPad = 8;  // rows of G and columns: entries a last round may read past their end

// kParts: 1, a group of lanes does all of a stage; 2, consecutive groups do H, and M and the copies.
template <typename T, int kLanes, int kParts>
__global__ void __launch_bounds__(128) factorise_kernel(FactArgs a, T *blk) {
  extern __shared__ double smem[];
  const int gl = threadIdx.x & (kLanes - 1);
  const int group = threadIdx.x / kLanes;
  const bool do_H = kParts == 1 || (group & 1) == 0, do_M = kParts == 1 || (group & 1) == 1;
  const int rows_max = a.rows;
  const int64_t b0 = ((int64_t)blockIdx.x * (blockDim.x / kLanes) + group) / kParts;
  const bool valid = b0 < a.nblocks;  // the groups of a warp stay together: the last ones idle
  const int64_t b = valid ? b0 : a.nblocks - 1;
  unsigned short *tab = reinterpret_cast<unsigned short *>(smem);
  for (int t = threadIdx.x; t < a.tab_len; t += blockDim.x) tab[t] = tri_entry(t);
  __syncthreads();
  double *sh = smem + a.tab_words + (size_t)group * a.words_per_stage;
  const int j = a.binst[b];
  const int kb = (int)(b - a.bbase[j]);
  const int nx = a.L.nx[j], nu = a.L.nu[j], N = a.L.N[j], n = nx + nu;
  double *G = sh;                          // up to rows_max rows of n
  double *S = G + rows_max * n + kPad;       // lower triangle, packed
  double *col = S + n * (n + 1) / 2 + kLanes;  // 2 n
  const bool lti = a.L.lti != 0;
  const bool terminal = lti ? (kb == 1) : (kb == N - 1);
  const double rho = a.rho;
  const double *qd = a.qd + a.L.off_n[j];
  const int nmax = (int)__reduce_max_sync(0xffffffffu, (unsigned)n);
  const int numax = (int)__reduce_max_sync(0xffffffffu, (unsigned)nu);

  // Dynamics of the stage whose Abar enters H (k+1), and of the stage itself (k).
  const int kH = lti ? 0 : kb + 1;
  const int kS = lti ? 0 : kb;
  const double *A = a.A + a.L.offA[j];
  const double *B = a.B + a.L.offB[j];
  const double *e = a.e ? a.e + a.L.offe[j] : nullptr;

  const int nxmax = (int)__reduce_max_sync(0xffffffffu, (unsigned)nx);
  if (do_H) {
    // K = Qbar + rho I (+ rho (G^T G + diag(0, I))), lower triangle, rows_max rows of G at a time.
    const int tr = rounds<kLanes>(n * (n + 1) / 2);
    for (int r0 = 0; r0 < nxmax; r0 += rows_max) {
      const int rows = terminal ? 0 : min(rows_max, nx - r0);  // <= 0: this stage is done
      const double *Ak = A + (size_t)kH * nx * nx, *Bk = B + (size_t)kH * nx * nu;
      __syncwarp();
      for (int w = gl; w < rows * n; w += kLanes) {
        const int r = w / n, c = w - r * n;
        G[w] = c < nx ? Ak[(r0 + r) * nx + c] : Bk[(r0 + r) * nu + (c - nx)];
      }
      __syncwarp();
      if (r0 == 0 || rows > 0)
        for (int q = 0, t = gl; q < tr; ++q, t += kLanes) {  // every lane its own (i, c), c <= i
          const int i = tab[t] >> 8, c = tab[t] & 0xff;
          double s = r0 ? S[t] : 0.0;
          for (int r = 0; r < rows; ++r) s = fma(G[r * n + i], G[r * n + c], s);
          S[t] = s;
        }
    }
    __syncwarp();
    if (rho != 1.0) {  // the off-diagonal entries; the diagonal follows
      for (int t = gl; t < n * (n + 1) / 2; t += kLanes)
        if (tab[t] >> 8 != (tab[t] & 0xff)) S[t] *= rho;
      __syncwarp();
    }
    for (int i = gl; i < n; i += kLanes) {  // the diagonal's own terms
      double s = S[tri_slot(i, i)];
      if (!terminal && i >= nx) s += 1.0;
      s *= rho;
      S[tri_slot(i, i)] = s + (qd[i] + rho);
    }
    sweep_inverse<kLanes>(S, col, tab, n, nmax, gl, a.err + j);
  }

  const int W = a.L.W[j];
  const int lay = a.L.tiled;
  const bool packed = lay == 1 || lay == 2;  // symmetric matrices packed lower
  const bool blocked = lay == 3;
  const int ts = (int)sizeof(T);
  const int ldg = blocked ? bl_ldg(n, ts) : (packed ? n : odd_ld(n));
  const int oE = nx * ldg;
  const int oH = blocked ? bl_oH(nx, nu, ts) : oE + nx;
  const int oM = blocked ? bl_oM(nx, nu, ts) : oH + (packed ? packed_size(n) : wrapped_size(n));
  // Element e of this block: tiled stage-varying data interleaves 32 stages element-major;
  // halo tiles interleave tw slots and hold the stage up to three times (its own slot and the
  // halo slots of the neighbouring tiles); everything else is a plain block.
  T *bases[3];
  int nb = 1, es;
  if (a.L.tiled == 2) {
    const int tw = a.L.tw[j];
    int t, sl, tt[2], ss[2];
    halo_slot(tw, kb, t, sl);
    es = tw;
    bases[0] = blk + a.L.blk[j] + (int64_t)t * W + sl;
    const int m = halo_copies(tw, N, kb, tt, ss);
    for (int q = 0; q < m; ++q) bases[1 + q] = blk + a.L.blk[j] + (int64_t)tt[q] * W + ss[q];
    nb = 1 + m;
  } else if (lay == 1 && !lti) {
    bases[0] = blk + a.L.blk[j] + (int64_t)(kb >> 5) * 32 * W + (kb & 31);
    es = 32;
  } else {
    bases[0] = blk + a.L.blk[j] + (int64_t)kb * W;
    es = 1;
  }
  auto put = [&](int e, double v, bool neg = false) {
    if (valid)
      for (int q = 0; q < nb; ++q) store(bases[q] + (int64_t)e * es, v, neg);
  };
  // Symmetric matrices (Xs: the negated lower triangle): packed lower row-major
  // (one-thread-per-stage kernels) or wrapped diagonals, row d holding S[c][(c + d) mod m]
  // (lane-group kernels); H of the blocked layout as wrapped 4 x 4 block diagonals (slot w is
  // element (a, b) of block (d, I), see bl_sym_index).
  auto put_sym_blocks = [&](int o, int m, const double *Xs) {
    const int nbm = bl_nb(m);
    for (int w = gl; w < bl_sym_words(m); w += kLanes) {
      int d, I, a4, b;
      if (!bl_sym_slot(nbm, w, d, I, a4, b)) {  // padding of the diagonal-block region
        put(o + w, 0.0);
        continue;
      }
      const int r = 4 * I + a4, c = 4 * ((I + d) % nbm) + b;
      const bool in = r < m && c < m;
      put(o + w, in ? Xs[tri_slot(r, c)] : 0.0, in);
    }
  };
  auto put_sym = [&](int o, int m, const double *Xs) {
    if (packed) {
      for (int t = gl; t < m * (m + 1) / 2; t += kLanes) put(o + t, Xs[t], true);
    } else {
      const int words = wrapped_size(m);
      for (int w = gl; w < words; w += kLanes) {
        const int d = w / m, c = w - d * m;
        put(o + w, Xs[tri_slot(c, (c + d) % m)], true);
      }
    }
  };
  if (do_H) {
    if (blocked) put_sym_blocks(oH, n, S);
    else put_sym(oH, n, S);
    __syncwarp();
  }
  if (!do_M) return;

  // Own-stage G_k, e_k and M_k = (B_k^T B_k + I + Wdu/rho)^{-1}.
  const double *Ak = A + (size_t)kS * nx * nx, *Bk = B + (size_t)kS * nx * nu;
  for (int w = gl; w < nx * n; w += kLanes) {
    const int r = w / n, c = w - r * n;
    put(r * ldg + c, c < nx ? Ak[r * nx + c] : Bk[r * nu + (c - nx)]);
  }
  for (int w = gl; w < nx * (ldg - n); w += kLanes) {  // row padding
    const int r = w / (ldg - n);
    put(r * ldg + n + (w - r * (ldg - n)), 0.0);
  }
  for (int r = gl; r < nx; r += kLanes) put(oE + r, e ? e[(size_t)kS * nx + r] : 0.0);
  if (blocked)
    for (int r = nx + gl; r < bl_pad4(nx); r += kLanes) put(oE + r, 0.0);
  const double *rdu = a.rdu ? a.rdu + a.L.off_n[j] + nx : nullptr;
  const int tru = rounds<kLanes>(nu * (nu + 1) / 2);
  for (int r0 = 0; r0 < nxmax; r0 += rows_max) {
    const int rows = min(rows_max, nx - r0);
    __syncwarp();
    for (int w = gl; w < rows * nu; w += kLanes) G[w] = Bk[r0 * nu + w];
    __syncwarp();
    for (int q = 0, t = gl; q < tru; ++q, t += kLanes) {
      const int i = tab[t] >> 8, c = tab[t] & 0xff;
      double s = r0 ? S[t] : 0.0;
      for (int r = 0; r < rows; ++r) s = fma(G[r * nu + i], G[r * nu + c], s);
      S[t] = s;
    }
  }
  __syncwarp();
  for (int i = gl; i < nu; i += kLanes) S[tri_slot(i, i)] += 1.0 + (rdu ? rdu[i] / rho : 0.0);
  sweep_inverse<kLanes>(S, col, tab, nu, numax, gl, a.err + j);
  put_sym(oM, nu, S);
  if (!packed) {  // padding of a plain or blocked block
    const int end = oM + wrapped_size(nu);
    for (int w = end + gl; w < W; w += kLanes) put(w, 0.0);
  }
}

template <typename T, int kLanes, int kParts>
cudaError_t launch_lanes(const FactArgs &a, T *blk, int warps, size_t per_group, cudaStream_t stream) {
  const int groups = warps * 32 / kLanes, stages = groups / kParts;
  const size_t smem = per_group * groups + sizeof(double) * a.tab_words;
  cudaError_t rc = allow_smem((const void *)factorise_kernel<T, kLanes, kParts>, smem);
  if (rc != cudaSuccess) return rc;
  factorise_kernel<T, kLanes, kParts>
      <<<(unsigned)((a.nblocks + stages - 1) / stages), 32 * warps, smem, stream>>>(a, blk);
  return cudaGetLastError();
}

template <typename T>
cudaError_t launch_t(const FactArgs &a, T *blk, int lanes, int parts, int warps, size_t per_group,
                     cudaStream_t stream) {
  return lanes == 8    ? launch_lanes<T, 8, 1>(a, blk, warps, per_group, stream)
         : lanes == 16 ? launch_lanes<T, 16, 1>(a, blk, warps, per_group, stream)
         : parts == 1  ? launch_lanes<T, 32, 1>(a, blk, warps, per_group, stream)
                       : launch_lanes<T, 32, 2>(a, blk, warps, per_group, stream);
}

}  // namespace

// Shared-memory doubles of one stage: `rows` rows of G, the packed lower triangle, the pivot
// column twice.
static int factorise_stage_words(int max_n, int lanes, int rows) {
  return rows * max_n + kPad + max_n * (max_n + 1) / 2 + lanes + 2 * max_n + kPad;
}

cudaError_t launch_factorise(const Layout &L, const double *A, const double *B, const double *e,
                             const double *qd, const double *rdu, double rho, const int *binst,
                             const int64_t *bbase, int64_t nblocks, int max_nx, int max_n,
                             int precision, void *blk, int *err, cudaStream_t stream) {
  FactArgs a;
  a.L = L; a.A = A; a.B = B; a.e = e; a.qd = qd; a.rdu = rdu; a.rho = rho;
  a.binst = binst; a.bbase = bbase; a.nblocks = nblocks; a.err = err;
  cudaError_t rc = cudaMemsetAsync(err, 0, sizeof(int) * (size_t)L.batch, stream);
  if (rc != cudaSuccess) return rc;
  if (nblocks == 0) return cudaSuccess;
  int dev = 0, nsm = 0;
  if ((rc = cudaGetDevice(&dev)) != cudaSuccess) return rc;
  if ((rc = cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess) return rc;
  // Few stages (up to two per SM): two warps each, spread over the schedulers (200 stages of n = 16:
  // 31 us with a warp each, 24 with two). Up to eight per SM: a warp each. Many: 8 or 16 lanes each.
  const int parts = nblocks <= 2 * (int64_t)nsm ? 2 : 1;
  int lanes = nblocks <= 8 * (int64_t)nsm ? 32 : (max_n <= 8 ? 8 : 16);
  int warps = parts == 2 ? 2 : (nblocks <= 4 * (int64_t)nsm ? 1 : 4);
  a.rows = parts == 2 ? max_nx : std::min(kRows, max_nx);
  auto bytes = [&](int l, int w) { return sizeof(double) * factorise_stage_words(max_n, l, a.rows) * (32 / l) * w; };
  while (lanes < 32 && bytes(lanes, warps) > 100 * 1024) lanes *= 2;
  while (warps > parts && bytes(lanes, warps) > 200 * 1024) warps >>= 1;
  a.words_per_stage = factorise_stage_words(max_n, lanes, a.rows);
  a.tab_len = max_n * (max_n + 1) / 2 + lanes;
  a.tab_words = (a.tab_len + 3) / 4;
  const size_t per_stage = sizeof(double) * a.words_per_stage;
  return precision == 0 ? launch_t<float>(a, (float *)blk, lanes, parts, warps, per_stage, stream)
                        : launch_t<double>(a, (double *)blk, lanes, parts, warps, per_stage, stream);
}

}  // namespace pimpc

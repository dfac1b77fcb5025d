// models.cu -- built-in nonlinear models, explicit-Euler relinearisation and the plant step.
//
// Real-time iteration (the NMPC scheme the paper's LTV formulation generalises, Sec. I-II): at
// every sample the model x_{k+1} = F(x_k, u_k) = x_k + dt f(x_k, u_k) is linearised along a
// trajectory, A_k = dF/dx, B_k = dF/du, e_k = F(xbar_k, ubar_k) - A_k xbar_k - B_k ubar_k,
// and the solver runs on the resulting stage matrices without building a QP. Jacobians come
// from forward-mode dual numbers, all in FP64, a group of lanes per linearisation point and a lane
// per seed direction: an FP64 instruction takes a warp 64 cycles whatever its active lanes, so a
// thread that walked the 16 directions of the quadrotor by itself took 301 us for 200 points.
// Lane q of a group evaluates the sine and cosine of angle q once and the others read them.
#include <math.h>

#include "launch.h"

namespace pimpc {

namespace {

// First-order dual number v + d eps.
struct Dual {
  double v, d;
  __device__ Dual() {}
  __device__ Dual(double a, double b = 0.0) : v(a), d(b) {}
};
__device__ inline Dual mk(double v, double d) { return Dual(v, d); }
__device__ inline Dual operator+(Dual a, Dual b) { return Dual{a.v + b.v, a.d + b.d}; }
__device__ inline Dual operator-(Dual a, Dual b) { return Dual{a.v - b.v, a.d - b.d}; }
__device__ inline Dual operator*(Dual a, Dual b) { return Dual{a.v * b.v, a.d * b.v + a.v * b.d}; }
__device__ inline Dual operator/(Dual a, Dual b) {
  return Dual{a.v / b.v, (a.d * b.v - a.v * b.d) / (b.v * b.v)};
}
__device__ inline Dual operator*(double s, Dual a) { return Dual{s * a.v, s * a.d}; }
__device__ inline Dual operator+(double s, Dual a) { return Dual{s + a.v, a.d}; }
__device__ inline Dual operator-(double s, Dual a) { return Dual{s - a.v, -a.d}; }
__device__ inline Dual exp(Dual a) {
  double e = ::exp(a.v);
  return Dual{e, e * a.d};
}
__device__ inline double dexp(double a) { return ::exp(a); }
__device__ inline Dual dexp(Dual a) { return exp(a); }

// Sines and cosines of a model's angles: from the values, and with the angles' derivatives.
constexpr int kMaxAngles = 3;
struct Angles {
  double s[kMaxAngles], c[kMaxAngles];
};
__device__ inline double sine(const Angles &t, int i, double) { return t.s[i]; }
__device__ inline double cosine(const Angles &t, int i, double) { return t.c[i]; }
__device__ inline Dual sine(const Angles &t, int i, Dual a) { return Dual{t.s[i], t.c[i] * a.d}; }
__device__ inline Dual cosine(const Angles &t, int i, Dual a) { return Dual{t.c[i], -t.s[i] * a.d}; }

// Quadrotor, "+" layout: x = (position, velocity, roll, pitch, yaw, body rates), u = rotor
// thrusts; p = (m, g, Jx, Jy, Jz, arm, yaw coefficient). Rotation R = Rz(yaw) Ry(pitch) Rx(roll).
template <typename S>
__device__ void quadrotor(const double *p, const Angles &t, const S *x, const S *u, S *f) {
  const double m = p[0], g = p[1], Jx = p[2], Jy = p[3], Jz = p[4], arm = p[5], kq = p[6];
  const S thrust = u[0] + u[1] + u[2] + u[3];
  const S tau_x = arm * (u[1] - u[3]);
  const S tau_y = arm * (u[2] - u[0]);
  const S tau_z = kq * ((u[0] + u[2]) - (u[1] + u[3]));
  const S sr = sine(t, 0, x[6]), cr = cosine(t, 0, x[6]);
  const S sp = sine(t, 1, x[7]), cp = cosine(t, 1, x[7]);
  const S sy = sine(t, 2, x[8]), cy = cosine(t, 2, x[8]);
  const S wx = x[9], wy = x[10], wz = x[11];
  const S acc = (1.0 / m) * thrust;
  for (int i = 0; i < 3; ++i) f[i] = x[3 + i];
  f[3] = acc * (cy * sp * cr + sy * sr);
  f[4] = acc * (sy * sp * cr - cy * sr);
  f[5] = acc * (cp * cr) - S(g);
  // roll/pitch/yaw rates from body rates
  f[6] = wx + (sr * wy + cr * wz) * (sp / cp);
  f[7] = cr * wy - sr * wz;
  f[8] = (sr * wy + cr * wz) / cp;
  // J dw/dt = tau - w x (J w), J diagonal
  f[9] = (1.0 / Jx) * (tau_x - (Jz - Jy) * (wy * wz));
  f[10] = (1.0 / Jy) * (tau_y - (Jx - Jz) * (wz * wx));
  f[11] = (1.0 / Jz) * (tau_z - (Jy - Jx) * (wx * wy));
}

// Cart-pole with a uniform pole (half-length l), upright at angle 0:
// x = (cart position, cart velocity, angle, angular rate), u = force; p = (mc, mp, l, g).
template <typename S>
__device__ void cartpole(const double *p, const Angles &t, const S *x, const S *u, S *f) {
  const double mc = p[0], mp = p[1], l = p[2], g = p[3], mt = mc + mp;
  const S s = sine(t, 0, x[2]), c = cosine(t, 0, x[2]);
  const S w = x[3];
  const S b = (1.0 / mt) * (u[0] + (mp * l) * (w * w) * s);
  const S ang = (g * s - c * b) / (l * (4.0 / 3.0 - (mp / mt) * (c * c)));
  f[0] = x[1];
  f[1] = b - ((mp * l) / mt) * (ang * c);
  f[2] = w;
  f[3] = ang;
}

// CSTR of the paper's example (Sec. V): x = (C_A, T), u = T_c; p = (C_Ai, k0, EaR, T_i).
template <typename S>
__device__ void cstr(const double *p, const S *x, const S *u, S *f) {
  const S rate = p[1] * (dexp(-p[2] / x[1]) * x[0]);
  f[0] = (p[0] - x[0]) - rate;
  f[1] = (p[3] + 0.3 * u[0]) - 1.3 * x[1] + 11.92 * rate;
}

// Sizes of a model: states, inputs, angles (at states first_angle ..), lanes per point (the power
// of two that holds the nx + nu directions).
template <int kModel>
struct Sizes;
template <>
struct Sizes<0> {
  static constexpr int nx = 12, nu = 4, angles = 3, first_angle = 6, lanes = 16;
};
template <>
struct Sizes<1> {
  static constexpr int nx = 4, nu = 1, angles = 1, first_angle = 2, lanes = 8;
};
template <>
struct Sizes<2> {
  static constexpr int nx = 2, nu = 1, angles = 0, first_angle = 0, lanes = 4;
};

template <int kModel, typename S>
__device__ __forceinline__ void eval_model(const double *p, const Angles &t, const S *x, const S *u, S *f) {
  if constexpr (kModel == 0) quadrotor(p, t, x, u, f);
  else if constexpr (kModel == 1) cartpole(p, t, x, u, f);
  else cstr(p, x, u, f);
}

__device__ __host__ inline int nparams(int model) { return model == 0 ? 7 : 4; }

// The angles of a point: lane q of its group evaluates angle q, the whole warp takes part.
template <int kModel>
__device__ __forceinline__ void find_angles(const double *xv, int gl, Angles &t) {
  using Z = Sizes<kModel>;
  if constexpr (Z::angles > 0) {
    double a = xv[Z::first_angle];
#pragma unroll
    for (int q = 1; q < Z::angles; ++q)
      if (gl == q) a = xv[Z::first_angle + q];
    double s, c;
    sincos(a, &s, &c);
#pragma unroll
    for (int q = 0; q < Z::angles; ++q) {
      t.s[q] = __shfl_sync(0xffffffffu, s, q, Z::lanes);
      t.c[q] = __shfl_sync(0xffffffffu, c, q, Z::lanes);
    }
  }
}

constexpr int kModelThreads = 64;

// A group of lanes per linearisation point (stage k of instance j, or instance j for LTI data):
// lane dir evaluates direction dir, then lane i forms component i of e.
template <int kModel>
__global__ void __launch_bounds__(kModelThreads)
    linearise_kernel(Layout L, const double *params, double dt, const double *xbar,
                     const double *ubar, double *A, double *B, double *e, int64_t total,
                     const int *pinst, const int64_t *pbase) {
  using Z = Sizes<kModel>;
  constexpr int nx = Z::nx, nu = Z::nu, n = nx + nu, g = Z::lanes;
  __shared__ double rows[kModelThreads / g][nx][g + 1];
  const int gl = threadIdx.x % g, grp = threadIdx.x / g;
  const int64_t at = (int64_t)blockIdx.x * (kModelThreads / g) + grp;
  const bool valid = at < total;  // the last groups repeat the last point and write nothing
  const int64_t pt = valid ? at : total - 1;
  const int j = pinst ? pinst[pt] : (int)pt;
  const int k = pinst ? (int)(pt - pbase[j]) : 0;
  const double *p = params + (int64_t)j * nparams(kModel);
  const int64_t sx = (L.lti ? L.off_nx[j] : L.Nnx[j]) + (int64_t)k * nx;
  const int64_t su = (L.lti ? L.off_nu[j] : L.Nnu[j]) + (int64_t)k * nu;
  double xv[nx], uv[nu];
#pragma unroll
  for (int i = 0; i < nx; ++i) xv[i] = xbar[sx + i];
#pragma unroll
  for (int i = 0; i < nu; ++i) uv[i] = ubar[su + i];
  Angles t;
  find_angles<kModel>(xv, gl, t);
  Dual xd[nx], ud[nu], fd[nx];
#pragma unroll
  for (int i = 0; i < nx; ++i) xd[i] = mk(xv[i], i == gl ? 1.0 : 0.0);
#pragma unroll
  for (int i = 0; i < nu; ++i) ud[i] = mk(uv[i], nx + i == gl ? 1.0 : 0.0);
  eval_model<kModel>(p, t, xd, ud, fd);
  double *Ak = A + L.offA[j] + (int64_t)k * nx * nx;
  double *Bk = B + L.offB[j] + (int64_t)k * nx * nu;
  double f = 0.0, x = 0.0;  // of component gl
#pragma unroll
  for (int i = 0; i < nx; ++i) {
    const double v = gl < nx ? (i == gl ? 1.0 : 0.0) + dt * fd[i].d : dt * fd[i].d;
    if (i == gl) {
      f = fd[i].v;
      x = xv[i];
    }
    rows[grp][i][gl] = v;
    if (valid && gl < nx) Ak[i * nx + gl] = v;
    else if (valid && gl < n) Bk[i * nu + (gl - nx)] = v;
  }
  __syncwarp();
  if (valid && gl < nx) {
    double s = x + dt * f;
#pragma unroll
    for (int c = 0; c < nx; ++c) s -= rows[grp][gl][c] * xv[c];
#pragma unroll
    for (int c = 0; c < nu; ++c) s -= rows[grp][gl][nx + c] * uv[c];
    e[L.offe[j] + (int64_t)k * nx + gl] = s;
  }
}

template <int kModel>
__global__ void __launch_bounds__(kModelThreads)
    plant_kernel(Layout L, const double *params, double dt, const double *x, const double *u,
                 double *x_next) {
  using Z = Sizes<kModel>;
  constexpr int nx = Z::nx, nu = Z::nu;
  const int gl = threadIdx.x % Z::lanes;
  const int at = (int)((blockIdx.x * kModelThreads + threadIdx.x) / Z::lanes);
  const int j = at < L.batch ? at : L.batch - 1;
  double xv[nx], uv[nu], f[nx];
#pragma unroll
  for (int i = 0; i < nx; ++i) xv[i] = x[L.off_nx[j] + i];
#pragma unroll
  for (int i = 0; i < nu; ++i) uv[i] = u[L.off_nu[j] + i];
  Angles t;
  find_angles<kModel>(xv, gl, t);
  eval_model<kModel>(params + (int64_t)j * nparams(kModel), t, xv, uv, f);
  // x_next may be x itself: every lane of the group has read its point by now (the shuffles
  // above, or this barrier)
  __syncwarp();
  if (at < L.batch && gl == 0) {
#pragma unroll
    for (int i = 0; i < nx; ++i) x_next[L.off_nx[j] + i] = xv[i] + dt * f[i];
  }
}

}  // namespace

int model_nparams(int model) { return nparams(model); }

int model_dims(int model, int *nx, int *nu) {
  switch (model) {
    case 0: *nx = 12; *nu = 4; return 0;
    case 1: *nx = 4; *nu = 1; return 0;
    case 2: *nx = 2; *nu = 1; return 0;
    default: return -1;
  }
}

cudaError_t launch_linearise(const Layout &L, int model, const double *params, double dt,
                             const double *xbar, const double *ubar, double *A, double *B,
                             double *e, int64_t total_points, const int *pinst,
                             const int64_t *pbase, cudaStream_t stream) {
  if (total_points == 0) return cudaSuccess;
  auto run = [&](auto kernel, int lanes) {
    const int64_t per = kModelThreads / lanes;
    kernel<<<(unsigned)((total_points + per - 1) / per), kModelThreads, 0, stream>>>(
        L, params, dt, xbar, ubar, A, B, e, total_points, pinst, pbase);
    return cudaGetLastError();
  };
  return model == 0   ? run(linearise_kernel<0>, Sizes<0>::lanes)
         : model == 1 ? run(linearise_kernel<1>, Sizes<1>::lanes)
                      : run(linearise_kernel<2>, Sizes<2>::lanes);
}

cudaError_t launch_plant_step(const Layout &L, int model, const double *params, double dt,
                              const double *x, const double *u, double *x_next,
                              cudaStream_t stream) {
  auto run = [&](auto kernel, int lanes) {
    const int per = kModelThreads / lanes;
    kernel<<<(L.batch + per - 1) / per, kModelThreads, 0, stream>>>(L, params, dt, x, u, x_next);
    return cudaGetLastError();
  };
  return model == 0   ? run(plant_kernel<0>, Sizes<0>::lanes)
         : model == 1 ? run(plant_kernel<1>, Sizes<1>::lanes)
                      : run(plant_kernel<2>, Sizes<2>::lanes);
}

}  // namespace pimpc

"""Performance cases: the calls a user of this library makes, over the range of sizes it serves.

Every case goes through the public entry points of ``paper_2601_14414_gb300.pimpc`` (and
``autograd``) with device memory on the current stream, except the AFTI-16 controller, which calls
the solver with host buffers as a control loop does. ``prepare`` makes what such a program holds
before the call (the solver object, its schedule, inputs drawn from the seed); ``run`` is one pass.

The C ABI hands results over as FP64 arrays. A solver with FP32 iterations computes them in FP32,
so its user keeps them in FP32 tensors (``_kept``); results of FP64 iterations stay FP64. Solves of
a fixed number of iterations return (u, x); solves to a tolerance also return iters, c and status.

``exact`` is Algorithm 1 in plain torch, FP64, on the instances padded to common sizes.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2601_14414_gb300 import autograd, pimpc
from paper_2601_14414_gb300 import workloads as W

F64 = torch.float64


def _dev():
    return torch.device("cuda", torch.cuda.current_device())


# ---- the cases -------------------------------------------------------------------------------

def listed():
    return [
        # The smallest call: plain linear MPC of one instance, 200 iterations in FP64, the
        # controller that solves one small problem over and over.
        dict(name="lti_single_f64", kind="lti", nx=4, nu=2, N=20, iters=200, accel=0, f64=True),
        # The paper's AFTI-16 tracking controller: one host-memory solve to c <= 1e-6.
        dict(name="afti16_host_f64", kind="afti16", N=5, rho=10.0, f64=True),
        # Real-time iteration of the quadrotor NMPC: linearise along the trajectory, factorise,
        # 100 accelerated iterations, plant step; the latency of one control sample.
        dict(name="quadrotor_rti_f32", kind="quadrotor", N=200, iters=100, f64=False),
        dict(name="quadrotor_rti_f64", kind="quadrotor", N=200, iters=100, f64=True),
        # The paper's CSTR NMPC sample at its size: a long horizon of a small model.
        dict(name="cstr_rti_f32", kind="cstr", N=5000, iters=1000, f64=False),
        dict(name="cstr_rti_f64", kind="cstr", N=5000, iters=1000, f64=True),
        # A differentiable-MPC training step: a batch of cart-poles, forward and backward.
        dict(name="cartpole_train_f32", kind="cartpole", batch=1024, N=100, iters=150, every=25,
             f64=False),
        # One entry-point call that allocates nothing, for controllers without allocation.
        dict(name="static_ltv_f32", kind="static", nx=12, nu=4, N=200, iters=100, f64=False),
        # Batches of uneven time-varying instances: the batched-service workload (factorise and
        # a fixed iteration budget), in FP64 to a tolerance, and with non-box input sets.
        dict(name="uneven_f32", kind="uneven", batch=4096, shapes=3, iters=50, eps=-1.0,
             sets=False, f64=False),
        dict(name="uneven_tol_f64", kind="uneven", batch=256, shapes=3, iters=500, eps=1e-6,
             sets=False, f64=True),
        dict(name="uneven_sets_f32", kind="uneven", batch=512, shapes=3, iters=50, eps=-1.0,
             sets=True, f64=False),
        # Stage-invariant instances with a large state, on the tensor cores.
        dict(name="large_lti_f32", kind="large_lti", batch=256, nx=48, nu=16, N=1000, iters=100,
             f64=False),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["lti", "afti16", "quadrotor", "cstr", "cartpole", "static", "uneven",
                       "large_lti"])
    f64 = rng.random() < 0.5
    if kind == "lti":
        return dict(kind=kind, nx=rng.randint(2, 12), nu=rng.randint(1, 4), N=_log(rng, 5, 100),
                    iters=rng.randint(50, 200), accel=rng.randint(0, 1), f64=f64)
    if kind == "afti16":
        return dict(kind=kind, N=rng.randint(4, 12), rho=rng.uniform(5.0, 20.0), f64=True)
    if kind == "quadrotor":
        return dict(kind=kind, N=_log(rng, 20, 300), iters=rng.randint(20, 100), f64=f64)
    if kind == "cstr":
        return dict(kind=kind, N=_log(rng, 100, 5000), iters=_log(rng, 100, 1000), f64=f64)
    if kind == "cartpole":
        return dict(kind=kind, batch=_log(rng, 16, 64 if f64 else 1024), N=rng.randint(20, 150),
                    iters=rng.randint(40, 150), every=rng.randint(5, 30), f64=f64)
    if kind == "static":
        return dict(kind=kind, nx=rng.randint(2, 24), nu=rng.randint(1, 8), N=_log(rng, 20, 400),
                    iters=rng.randint(20, 100), f64=f64)
    if kind == "uneven":
        sets = rng.random() < 0.3
        return dict(kind=kind, batch=_log(rng, 16, 256 if f64 else 2048),
                    shapes=rng.randint(4, 1 << 20), iters=rng.randint(20, 100), eps=-1.0,
                    sets=sets, f64=f64)
    return dict(kind=kind, batch=_log(rng, 16, 200), nx=rng.randint(17, 48),
                nu=rng.randint(2, 16), N=_log(rng, 100, 1000), iters=rng.randint(20, 100),
                f64=False)


# ---- inputs ----------------------------------------------------------------------------------

class _Handle:
    """A solver made through the C ABI, destroyed with the state that holds it."""

    def __init__(self, nx, nu, N, lti, f64):
        self.h = pimpc.pimpc_create(nx, nu, N, lti, pimpc.F64 if f64 else pimpc.F32,
                                    torch.cuda.current_device())

    def __del__(self):
        try:
            pimpc.pimpc_destroy(self.h)
        except Exception:
            pass


def _t(a):
    return torch.from_numpy(np.ascontiguousarray(a, np.float64)).to(_dev())


def _kept(f64, *ts):
    return list(ts) if f64 else [t.float() for t in ts]


def _shape_of(case):
    """(nx, nu, N) arrays of the case's instances."""
    k = case["kind"]
    if k == "uneven":
        return W.batched_dims(case["shapes"], case["batch"])
    nx, nu = {"quadrotor": (12, 4), "cstr": (2, 1), "cartpole": (4, 1),
              "afti16": (4, 2)}.get(k, (case.get("nx"), case.get("nu")))
    b = case.get("batch", 1)
    return np.full(b, nx), np.full(b, nu), np.full(b, case["N"])


def _stages(A, nx):
    """Scales A [..., nx, nx] (Gaussian entries) to spectral radius 1."""
    return A / np.max(np.abs(np.linalg.eigvals(A)), axis=-1)[..., None, None]


def _uneven_inputs(case, seed):
    """The batched uneven recipe of the repository's workloads, drawn on the GPU: per stage a
    signed-permutation similarity of an eigen-analysed Gaussian matrix (here from a pool of 32
    per state size) scaled to a spectral radius in [0.9, 1.05]."""
    nx, nu, N = _shape_of(case)
    dev = _dev()
    g = torch.Generator(device=dev)
    g.manual_seed(seed)
    rng = np.random.default_rng(seed)
    offA = np.concatenate([[0], np.cumsum(N * nx * nx)])
    A = torch.empty(int(offA[-1]), dtype=F64, device=dev)
    for m in np.unique(nx):
        pool = torch.from_numpy(_stages(rng.standard_normal((32, m, m)), m)).to(dev)
        idx = np.flatnonzero(nx == m)
        off = np.concatenate([offA[j] + np.arange(N[j], dtype=np.int64) * m * m for j in idx])
        S = len(off)
        pick = torch.randint(0, 32, (S,), generator=g, device=dev)
        perm = torch.argsort(torch.rand(S, m, generator=g, device=dev), dim=1)
        sign = 2.0 * torch.randint(0, 2, (S, m), generator=g, device=dev).to(F64) - 1.0
        rad = 0.9 + 0.15 * torch.rand(S, 1, 1, generator=g, device=dev, dtype=F64)
        M = pool[pick[:, None, None], perm[:, :, None], perm[:, None, :]]
        M = M * sign[:, :, None] * sign[:, None, :] * rad
        at = torch.from_numpy(off).to(dev)[:, None] + torch.arange(m * m, device=dev)
        A[at.reshape(-1)] = M.reshape(-1)
    d = dict(nx=nx, nu=nu, N=N, lti=False, rho=1.0, A=A)
    d["B"] = torch.randn(int(np.sum(N * nx * nu)), generator=g, device=dev, dtype=F64)
    d["e"] = 0.6 * torch.rand(int(np.sum(N * nx)), generator=g, device=dev, dtype=F64) - 0.3
    d["x0"] = 6.0 * torch.rand(int(np.sum(nx)), generator=g, device=dev, dtype=F64) - 3.0
    tx, tu = int(np.sum(nx)), int(np.sum(nu))
    one = lambda k, v: torch.full((k,), v, dtype=F64, device=dev)
    d.update(q=one(tx, 1.0), r=one(tu, 0.1), rdu=None, xmin=one(tx, -5.0), xmax=one(tx, 5.0),
             umin=one(tu, -1.0), umax=one(tu, 1.0), ref=one(tx + tu, 0.0), u_prev=None)
    if case["sets"]:  # every kind of set, the box among them
        kind = rng.integers(0, 5, len(nx)).astype(np.int32)
        d["uset"] = (kind, rng.uniform(0.5, 2.0, len(nx)), rng.standard_normal(tu))
    return d


def _inputs(case, seed):
    """Concatenated C ABI inputs (device FP64 tensors) of the case's instances."""
    k = case["kind"]
    if k == "uneven":
        return _uneven_inputs(case, seed)
    nx, nu, N = _shape_of(case)
    rng = np.random.default_rng(seed)
    b, mx, mu, n = len(nx), int(nx[0]), int(nu[0]), int(N[0])
    d = dict(nx=nx, nu=nu, N=N, lti=k in ("lti", "afti16", "cartpole", "large_lti"), rho=1.0,
             rdu=None, u_prev=None)
    inf = np.inf
    if k == "lti":
        d.update(A=0.95 * _stages(rng.standard_normal((mx, mx)), mx),
                 B=rng.standard_normal((mx, mu)), e=np.zeros(mx), q=np.ones(mx),
                 r=0.1 * np.ones(mu), x0=rng.uniform(-3, 3, mx), ref=np.zeros(mx + mu),
                 xmin=-5.0 * np.ones(mx), xmax=5.0 * np.ones(mx), umin=-np.ones(mu),
                 umax=np.ones(mu))
    elif k == "static":
        A = _stages(rng.standard_normal((n, mx, mx)), mx)
        d.update(A=A * rng.uniform(0.9, 1.05, (n, 1, 1)), B=rng.standard_normal((n, mx, mu)),
                 e=rng.uniform(-0.3, 0.3, (n, mx)), q=np.ones(mx), r=0.1 * np.ones(mu),
                 x0=rng.uniform(-3, 3, mx), ref=np.zeros(mx + mu), xmin=-5.0 * np.ones(mx),
                 xmax=5.0 * np.ones(mx), umin=-np.ones(mu), umax=np.ones(mu))
    elif k == "large_lti":
        A = 0.95 * _stages(rng.standard_normal((b, mx, mx)), mx)
        d.update(A=A, B=rng.standard_normal((b, mx, mu)), e=rng.uniform(-0.3, 0.3, (b, mx)),
                 q=rng.uniform(0.1, 10.0, b * mx), r=rng.uniform(0.01, 1.0, b * mu),
                 x0=rng.uniform(-3, 3, b * mx), ref=np.zeros(b * (mx + mu)),
                 xmin=-5.0 * np.ones(b * mx), xmax=5.0 * np.ones(b * mx),
                 umin=-W.LARGE_LTI_UMAX * np.ones(b * mu), umax=W.LARGE_LTI_UMAX * np.ones(b * mu))
    elif k == "afti16":
        wl = W.afti16(N=n, rho=case["rho"])
        d.update({key: wl[key] for key in ("A", "B", "e", "q", "r", "rdu", "xmin", "xmax", "umin",
                                           "umax", "rho")})
        # a state on the way to the +10 degree pitch command, the last applied deflections
        d.update(x0=np.array([0.0, 0.0, 0.0, rng.uniform(-10.0, 10.0)]),
                 u_prev=rng.uniform(-5.0, 5.0, mu), ref=W.afti16_reference(wl, 0))
    elif k == "quadrotor":
        wl = W.quadrotor_rti(N=n)
        goal = rng.uniform(-5, 5, 3)
        x0 = np.concatenate([rng.uniform(-1, 1, 3), rng.uniform(-0.5, 0.5, 3),
                             rng.uniform(-0.1, 0.1, 3), rng.uniform(-0.1, 0.1, 3)])
        s = np.linspace(0.0, 1.0, n)[:, None]
        xbar = np.concatenate([x0[:3] + s * (goal - x0[:3]), np.repeat(goal[None] * 0.2, n, 0),
                               rng.uniform(-0.3, 0.3, (n, 3)), rng.uniform(-0.3, 0.3, (n, 3))], 1)
        d.update({key: wl[key] for key in ("q", "r", "xmin", "xmax", "umin", "umax")})
        d.update(model=W.MODEL_QUADROTOR, params=wl["params"], dt=wl["dt"], x0=x0, xbar=xbar,
                 ubar=wl["hover_u"] + rng.uniform(-0.3, 0.3, (n, 4)),
                 ref=np.concatenate([goal, np.zeros(9), wl["hover_u"]]))
    elif k == "cstr":
        wl = W.cstr_nmpc(N=n)
        x0 = np.array([rng.uniform(7.5, 9.0), rng.uniform(308.0, 314.0)])
        d.update({key: wl[key] for key in ("q", "r", "rdu", "xmin", "xmax", "umin", "umax",
                                           "u_prev", "ref")})
        d.update(model=W.MODEL_CSTR, dt=wl["dt"], x0=x0,
                 params=np.append(wl["params"], W.cstr_inlet_temperature(rng.uniform(0, 100))),
                 xbar=x0 + rng.uniform(-0.1, 0.1, (n, 2)), ubar=300.0 + rng.uniform(-5, 5, (n, 1)))
    else:  # cartpole: the trained quantities differ from instance to instance
        x0 = np.zeros((b, 4))
        x0[:, 2] = rng.uniform(-0.3, 0.3, b)
        d.update(model=W.MODEL_CARTPOLE, params=np.tile(W.CARTPOLE_PARAMS, b), dt=0.05, x0=x0,
                 xbar=np.zeros((b, 4)), ubar=np.zeros((b, 1)),
                 q=np.tile([10.0, 1.0, 10.0, 1.0], b) * rng.uniform(0.8, 1.25, 4 * b),
                 r=0.1 * rng.uniform(0.8, 1.25, b), ref=np.zeros(5 * b),
                 xmin=np.full(4 * b, -inf), xmax=np.full(4 * b, inf), umin=np.full(b, -10.0),
                 umax=np.full(b, 10.0), gu=rng.standard_normal(b * n),
                 gx=rng.standard_normal(4 * b * n))
    return {key: _t(v).reshape(-1) if isinstance(v, np.ndarray) and key not in ("nx", "nu", "N")
            else v for key, v in d.items()}


def _accel(case):
    return case.get("accel", 0 if case["kind"] == "cartpole" else 1)


def prepare(case, seed):
    k, f64, dev = case["kind"], case["f64"], _dev()
    d = _inputs(case, seed)
    nx, nu, N = d["nx"], d["nu"], d["N"]
    st = dict(case=case, d=d, f64=f64)
    st["u"] = torch.zeros(int(np.sum(N * nu)), dtype=F64, device=dev)
    st["x"] = torch.zeros(int(np.sum(N * nx)), dtype=F64, device=dev)
    if k == "static":
        return st
    if k == "cartpole":
        cut = lambda a, w: [p.cpu().numpy() for p in a.reshape(-1, w)]
        per = {key: cut(d[key], w) for key, w in (("q", 4), ("r", 1), ("xmin", 4), ("xmax", 4),
                                                  ("umin", 1), ("umax", 1), ("x0", 4), ("ref", 5))}
        insts = [dict({key: v[j] for key, v in per.items()}, nx=4, nu=1, N=int(N[j]), lti=True,
                      rdu=None, u_prev=None, rho=1.0) for j in range(len(nx))]
        s = pimpc.Solver(insts, precision=pimpc.F64 if f64 else pimpc.F32, eps=-1.0,
                         max_iters=case["iters"], accel=0)
        s.set_schedule(pimpc.FAMILY_RESIDENT)
        pimpc.pimpc_linearise(s.h, d["model"], d["params"], d["dt"], d["xbar"], d["ubar"])
        st["solver"] = s
        st["args"] = [d[key].requires_grad_(key != "ref") for key in
                      ("x0", "ref", "q", "r", "xmin", "xmax", "umin", "umax")]
        return st
    s = st["solver"] = _Handle(nx, nu, N, d["lti"], f64)
    if k == "large_lti":
        pimpc.pimpc_set_schedule(s.h, pimpc.FAMILY_TENSOR)
    elif k != "uneven":
        pimpc.pimpc_set_schedule(s.h, pimpc.FAMILY_RESIDENT)
    pimpc.pimpc_set_weights(s.h, d["q"], d["r"], d["rdu"])
    pimpc.pimpc_set_bounds(s.h, d["xmin"], d["xmax"], d["umin"], d["umax"])
    pimpc.pimpc_set_options(s.h, d["rho"], 1e-6 if k == "afti16" else case.get("eps", -1.0),
                            20000 if k == "afti16" else case["iters"], _accel(case))
    if "A" in d:
        pimpc.pimpc_set_dynamics(s.h, d["A"], d["B"], d["e"])
    if "uset" in d:
        pimpc.pimpc_set_input_set(s.h, *d["uset"])
    if k in ("lti", "large_lti"):  # the plant does not change: the cache is part of the setup
        pimpc.pimpc_factorise(s.h, torch.cuda.current_stream().cuda_stream)
    if k == "lti":
        pimpc.pimpc_set_graph(s.h, 1)
    if k == "afti16":
        pimpc.pimpc_factorise(s.h)
        st["host"] = {key: d[key].cpu().numpy() for key in ("x0", "u_prev", "ref")}
        st["hu"], st["hx"] = np.zeros(int(np.sum(N * nu))), np.zeros(int(np.sum(N * nx)))
    if k in ("quadrotor", "cstr"):
        st["x_next"] = torch.zeros(int(nx[0]), dtype=F64, device=dev)
    b = len(nx)
    st["iters"] = torch.zeros(b, dtype=torch.int32, device=dev)
    st["c"] = torch.zeros(b, dtype=F64, device=dev)
    st["status"] = torch.zeros(b, dtype=torch.int32, device=dev)
    torch.cuda.synchronize()
    return st


def run(st):
    case, d, f64, u, x = st["case"], st["d"], st["f64"], st["u"], st["x"]
    k = case["kind"]
    if k == "static":
        nx, nu, N = (int(d[key][0]) for key in ("nx", "nu", "N"))
        pimpc.pimpc_solve_static(nx, nu, N, pimpc.F64 if f64 else pimpc.F32, d["A"], d["B"],
                                 d["e"], d["q"], d["r"], d["xmin"], d["xmax"], d["umin"],
                                 d["umax"], d["x0"], d["ref"], d["rho"], -1.0, case["iters"], 1,
                                 0.999, u, x)
        return _kept(f64, u, x)
    if k == "cartpole":
        uu, xx = autograd.unrolled_solve(st["solver"], case["iters"], *st["args"],
                                         checkpoint_every=case["every"])
        wrt = [a for a in st["args"] if a.requires_grad]
        gs = torch.autograd.grad([uu, xx], wrt, [d["gu"], d["gx"]])
        return _kept(f64, uu.detach(), xx.detach(), *gs)
    h = st["solver"].h
    if k == "afti16":
        it, c, status = np.zeros(1, np.int32), np.zeros(1), np.zeros(1, np.int32)
        pimpc.pimpc_solve(h, st["host"]["x0"], st["host"]["u_prev"], st["host"]["ref"], False, 0,
                          st["hu"], st["hx"], it, c, status)
        return [st["hu"].copy(), st["hx"].copy(), it, c, status]
    if k in ("lti", "large_lti"):
        pimpc.pimpc_solve(h, d["x0"], None, d["ref"], False, 0, u, x)
        return _kept(f64, u, x)
    if k in ("quadrotor", "cstr"):
        pimpc.pimpc_linearise(h, d["model"], d["params"], d["dt"], d["xbar"], d["ubar"])
        pimpc.pimpc_solve(h, d["x0"], d["u_prev"], d["ref"], False, 0, u, x)
        pimpc.pimpc_plant_step(h, d["model"], d["params"], d["dt"], d["x0"], u[:int(d["nu"][0])],
                               st["x_next"])
        return _kept(f64, u, x, st["x_next"])
    pimpc.pimpc_factorise(h, torch.cuda.current_stream().cuda_stream)
    if case["eps"] < 0:
        pimpc.pimpc_solve(h, d["x0"], None, d["ref"], False, 0, u, x)
        return _kept(f64, u, x)
    pimpc.pimpc_solve(h, d["x0"], None, d["ref"], False, 0, u, x, st["iters"], st["c"],
                      st["status"])
    return _kept(f64, u, x) + [st["iters"], st["c"], st["status"]]


def work(case):
    """Inputs read once and outputs written once (FP64, as the C ABI has them), and the
    multiply-adds and elementwise steps of Algorithm 1's iterations (the backward pass: twice the
    forward's); for the calls that factorise, the two inversions and their Gram matrices too."""
    k = case["kind"]
    nx, nu, N = (np.asarray(a, np.float64) for a in _shape_of(case))
    n = nx + nu
    iters = 2700 if k == "afti16" else case["iters"]
    per = 4 * nx * n + 4 * nx * nu + 2 * n * n + 2 * nu * nu + 40 * n
    flops = float(np.sum(N * per)) * iters
    lti = k in ("lti", "afti16", "cartpole", "large_lti")
    mats = float(np.sum((1 if lti else N) * (nx * n + nx)))
    if k == "quadrotor" or k == "cstr":
        mats = float(np.sum(N * n))  # the linearisation points
    nbytes = 8.0 * (mats + float(np.sum(N * n)) + float(np.sum(nx + 6 * n)))
    if k == "cartpole":
        flops *= 3
        nbytes += 8.0 * float(np.sum(N * n) + np.sum(5 * n))
    if k in ("quadrotor", "cstr", "static", "uneven"):
        flops += float(np.sum(N * (nx * n * n + n ** 3 + nx * nu * nu + nu ** 3)))
    return {"bytes": nbytes, "flops": flops}


# ---- the same results in plain torch, FP64 -----------------------------------------------------

def _f_quadrotor(p, x, u):
    m, g, Jx, Jy, Jz, arm, kq = p.unbind()
    thrust = u.sum() / m
    sr, cr, sp, cp, sy, cy = (f(x[i]) for i in (6, 7, 8) for f in (torch.sin, torch.cos))
    wx, wy, wz = x[9], x[10], x[11]
    tx, ty = arm * (u[1] - u[3]), arm * (u[2] - u[0])
    tz = kq * (u[0] + u[2] - u[1] - u[3])
    return torch.stack([x[3], x[4], x[5], thrust * (cy * sp * cr + sy * sr),
                        thrust * (sy * sp * cr - cy * sr), thrust * cp * cr - g,
                        wx + (sr * wy + cr * wz) * sp / cp, cr * wy - sr * wz,
                        (sr * wy + cr * wz) / cp, (tx - (Jz - Jy) * wy * wz) / Jx,
                        (ty - (Jx - Jz) * wz * wx) / Jy, (tz - (Jy - Jx) * wx * wy) / Jz])


def _f_cartpole(p, x, u):
    mc, mp, l, g = p.unbind()
    s, c = torch.sin(x[2]), torch.cos(x[2])
    b = (u[0] + mp * l * x[3] ** 2 * s) / (mc + mp)
    acc = (g * s - c * b) / (l * (4.0 / 3.0 - mp * c * c / (mc + mp)))
    return torch.stack([x[1], b - mp * l * acc * c / (mc + mp), x[3], acc])


def _f_cstr(p, x, u):
    rate = p[1] * torch.exp(-p[2] / x[1]) * x[0]
    return torch.stack([p[0] - x[0] - rate, p[3] + 0.3 * u[0] - 1.3 * x[1] + 11.92 * rate])


_MODELS = {W.MODEL_QUADROTOR: _f_quadrotor, W.MODEL_CARTPOLE: _f_cartpole, W.MODEL_CSTR: _f_cstr}


def _linearised(d, nx, nu):
    f, p = _MODELS[d["model"]], d["params"]
    step = lambda x, u: x + d["dt"] * f(p, x, u)
    if d["lti"]:  # one point, the same for every instance
        p = p[:4]
    xb, ub = d["xbar"].reshape(-1, nx), d["ubar"].reshape(-1, nu)
    A, B = torch.func.vmap(torch.func.jacfwd(step, argnums=(0, 1)))(xb, ub)
    F = torch.func.vmap(step)(xb, ub)
    e = F - (A @ xb[:, :, None])[..., 0] - (B @ ub[:, :, None])[..., 0]
    return A, B, e


def _project(w, kind, r, a):
    """Euclidean projection of w [b, N, nu] on each instance's set, kinds 1..4 (0: unchanged)."""
    out = w.clone()
    r = r[:, None, None]
    nrm = w.norm(dim=-1, keepdim=True)
    ball = torch.where(nrm > r, w * (r / nrm.clamp_min(1e-300)), w)
    aw = w.abs()
    srt = aw.sort(dim=-1, descending=True).values
    cum = srt.cumsum(-1) - r
    cnt = torch.arange(1, w.shape[-1] + 1, device=w.device, dtype=F64)
    last = (srt * cnt > cum).sum(-1, keepdim=True).clamp_min(1)
    tau = torch.gather(cum, -1, last - 1) / last
    l1 = torch.where(aw.sum(-1, keepdim=True) > r, w.sign() * (aw - tau).clamp_min(0), w)
    a = a[:, None]
    nn = (a * a).sum(-1, keepdim=True).clamp_min(1e-300)
    half = w - a * (((a * w).sum(-1, keepdim=True) - r).clamp_min(0) / nn)
    t, y = w[..., :1], w[..., 1:]
    s = y.norm(dim=-1, keepdim=True)
    h = 0.5 * (t + s)
    cone = torch.cat([h, h * y / s.clamp_min(1e-300)], -1)
    cone = torch.where(s <= t, w, torch.where(s <= -t, torch.zeros_like(w), cone))
    for i, v in ((1, ball), (2, l1), (3, half), (4, cone)):
        out = torch.where((kind == i)[:, None, None], v, out)
    return out


def _algorithm(p, rho, eps, iters, accel, eta=0.999):
    """Algorithm 1 on instances padded to common sizes: A [b, N|1, nx, nx], B, e, per-instance
    q, r, rdu, bounds, x0, u_prev, ref [b, n], N [b]. Returns z [b, N, n], iters, c, status."""
    A, B, e, N = p["A"], p["B"], p["e"], p["N"]
    b, nx, nu, S = A.shape[0], A.shape[-1], B.shape[-1], p["S"]
    dev, n = A.device, nx + nu
    G = torch.cat([A, B], -1)
    eye = lambda m: torch.eye(m, dtype=F64, device=dev)
    qd = torch.cat([p["q"], p["r"]], -1)
    K = rho * (G.mT @ G) + torch.diag_embed(qd + rho)[:, None]
    K[..., nx:, nx:] = K[..., nx:, nx:] + rho * eye(nu)
    stage = torch.arange(S, device=dev)
    last = (stage == N[:, None] - 1)[..., None]
    live = (stage < N[:, None])[..., None].to(F64)
    more = (stage < N[:, None] - 1)[..., None].to(F64)
    H = torch.linalg.inv(K)
    if H.shape[1] > 1:  # H_k goes with the next stage's matrices
        H = torch.cat([H[:, 1:], H[:, :1]], 1)
    del K
    end = (1.0 / (qd + rho))[:, None]
    M = torch.linalg.inv(B.mT @ B + eye(nu) + torch.diag_embed(p["rdu"] / rho)[:, None])
    xb0 = torch.cat([p["x0"], p["u_prev"]], -1)[:, None]
    qr, lo, hi = (qd * p["ref"])[:, None], p["lo"][:, None], p["hi"][:, None]
    if A.shape[1] == 1:
        mul = lambda m, v: v @ m[:, 0].mT
    else:
        mul = lambda m, v: (m @ v[..., None])[..., 0]
    eb = torch.cat([e, torch.zeros(e.shape[:-1] + (nu,), dtype=F64, device=dev)], -1)
    cur = [torch.zeros(b, S, n, dtype=F64, device=dev) for _ in range(5)]
    hat, cprev, al = cur, torch.ones(b, dtype=F64, device=dev), torch.ones(b, dtype=F64, device=dev)
    run_ = torch.ones(b, dtype=torch.bool, device=dev)
    its, cs = torch.zeros(b, dtype=torch.int32, device=dev), torch.zeros(b, dtype=F64, device=dev)
    for i in range(iters):
        zh, vh, th, bh, lh = hat
        w = vh - bh
        du = mul(M, mul(B.mT, w[..., :nx]) + w[..., nx:])
        y = zh - vh + lh - eb
        g = mul(G.mT, y[..., :nx])
        g = torch.cat([g[..., :nx], g[..., nx:] + y[..., nx:]], -1)
        g = torch.cat([g[:, 1:], g[:, :1]], 1) * more
        hk = qr + rho * (zh - th + g)
        xb = torch.where(last, end * hk, mul(H, hk))
        xp = torch.cat([xb0, xb[:, :-1]], 1)
        ax = torch.cat([mul(G, xp), xp[..., nx:]], -1)
        bd = torch.cat([mul(B, du), du], -1)
        gam = bd + bh - ax - eb + lh
        wz = (2.0 * (xb + th + ax + eb - lh) + gam) / 3.0
        z = torch.minimum(torch.maximum(wz, lo), hi)
        if p.get("kind") is not None:
            box = (p["kind"] == 0)[:, None, None]
            pu = _project(wz[..., nx:], p["kind"], p["rad"], p["nrm"])
            z = torch.cat([z[..., :nx], torch.where(box, z[..., nx:], pu)], -1)
        v = 0.5 * (z + gam)
        new = [z, v, th + xb - z, bh + bd - v, lh + z - ax - v - eb]
        d1, d2, d3, d4, d5 = new[2] - th, new[3] - bh, new[4] - lh, z - zh, v - vh
        c = None
        if accel or eps >= 0:
            sq = d1 ** 2 + d2 ** 2 + d3 ** 2 + d4 ** 2 + d5 ** 2 + (d4 - d5) ** 2
            c = rho * (sq * live).sum((1, 2))
        if eps >= 0:
            its = torch.where(run_, its + 1, its)
            cs = torch.where(run_, c, cs)
            keep = run_[:, None, None]
            new = [torch.where(keep, a, o) for a, o in zip(new, cur)]
            run_ = run_ & ~(c <= eps)
            if i % 16 == 15 and not bool(run_.any()):
                cur = new
                break
        prev, cur, hat = cur, new, new
        if accel:
            take = c <= eta * cprev
            an = 0.5 + 0.5 * torch.sqrt(1.0 + 4.0 * al * al)
            f = torch.where(take, (al - 1.0) / an, torch.zeros_like(al))[:, None, None]
            al = torch.where(take, an, torch.ones_like(al))
            cprev = c
            hat = [a + f * (a - o) for a, o in zip(cur, prev)]
    return cur[0], its, cs, torch.where(run_, 1, 0).to(torch.int32)


def _padded(d, idx, mx, mu, S):
    """The instances idx of the concatenated inputs, padded with zeros to (mx, mu, S)."""
    nx, nu, N = d["nx"], d["nu"], d["N"]
    dev, lti, b = _dev(), d["lti"], len(idx)
    reps = np.ones(len(nx), np.int64) if lti else N
    off = {key: np.concatenate([[0], np.cumsum(w)]) for key, w in
           (("A", reps * nx * nx), ("B", reps * nx * nu), ("e", reps * nx), ("x", nx), ("u", nu),
            ("n", nx + nu))}
    R = 1 if lti else S
    zero = lambda *s: torch.zeros(*s, dtype=F64, device=dev)
    p = dict(A=zero(b, R, mx, mx), B=zero(b, R, mx, mu), e=zero(b, R, mx), S=S,
             N=torch.from_numpy(np.asarray(N[idx], np.int64)).to(dev))
    for key in ("q", "x0"):
        p[key] = zero(b, mx)
    for key in ("r", "rdu", "u_prev", "nrm"):
        p[key] = zero(b, mu)
    p["ref"] = zero(b, mx + mu)
    p["lo"], p["hi"] = zero(b, mx + mu) - math.inf, zero(b, mx + mu) + math.inf
    cut = lambda key, o, j: d[key][int(off[o][j]):int(off[o][j + 1])]
    for i, j in enumerate(idx):
        a, c, m = int(nx[j]), int(nu[j]), 1 if lti else int(N[j])
        p["A"][i, :m, :a, :a] = cut("A", "A", j).reshape(m, a, a)
        p["B"][i, :m, :a, :c] = cut("B", "B", j).reshape(m, a, c)
        p["e"][i, :m, :a] = cut("e", "e", j).reshape(m, a)
        p["q"][i, :a], p["x0"][i, :a] = cut("q", "x", j), cut("x0", "x", j)
        p["r"][i, :c] = cut("r", "u", j)
        for key in ("rdu", "u_prev"):
            if d[key] is not None:
                p[key][i, :c] = cut(key, "u", j)
        ref = cut("ref", "n", j)
        p["ref"][i, :a], p["ref"][i, mx:mx + c] = ref[:a], ref[a:]
        for side, xk, uk in (("lo", "xmin", "umin"), ("hi", "xmax", "umax")):
            p[side][i, :a], p[side][i, mx:mx + c] = cut(xk, "x", j), cut(uk, "u", j)
    if "uset" in d:
        kind, r, a = d["uset"]
        p["kind"] = torch.from_numpy(kind[idx].astype(np.int64)).to(dev)
        p["rad"] = torch.from_numpy(r[idx]).to(dev)
        for i, j in enumerate(idx):
            if kind[j] == 3:
                p["nrm"][i, :int(nu[j])] = _t(a[int(off["u"][j]):int(off["u"][j + 1])])
    return p


def exact(case, seed):
    k = case["kind"]
    d = _inputs(case, seed)
    nx, nu, N = d["nx"], d["nu"], d["N"]
    eps = 1e-6 if k == "afti16" else case.get("eps", -1.0)
    iters = 20000 if k == "afti16" else case["iters"]
    if "model" in d:
        A, B, e = _linearised(d, int(nx[0]), int(nu[0]))
        d.update(A=A.reshape(-1), B=B.reshape(-1), e=e.reshape(-1))
    if k == "cartpole":
        return _exact_train(case, d)
    order = np.argsort(N, kind="stable")
    u = [None] * len(nx)
    x = [None] * len(nx)
    step = 256 if k == "uneven" else 64
    its = torch.zeros(len(nx), dtype=torch.int32, device=_dev())
    status = its.clone()
    c = torch.zeros(len(nx), dtype=F64, device=_dev())
    for at in range(0, len(nx), step):
        idx = order[at:at + step]
        mx, mu, S = int(nx[idx].max()), int(nu[idx].max()), int(N[idx].max())
        z, i_, c_, s_ = _algorithm(_padded(d, idx, mx, mu, S), d["rho"], eps, iters, _accel(case))
        for r, j in enumerate(idx):
            zj = z[r, :int(N[j])]
            x[j], u[j] = zj[:, :int(nx[j])].reshape(-1), zj[:, mx:mx + int(nu[j])].reshape(-1)
        at_ = torch.from_numpy(idx).to(_dev())
        its[at_], c[at_], status[at_] = i_, c_, s_
    u, x = torch.cat(u), torch.cat(x)
    if k in ("quadrotor", "cstr"):
        f = _MODELS[d["model"]]
        return [u, x, d["x0"] + d["dt"] * f(d["params"], d["x0"], u[:int(nu[0])])]
    if eps < 0:
        return [u, x]
    return [u, x, None, c, None]


def _exact_train(case, d):
    """Forward and gradients of the unrolled plain iteration by torch's autograd."""
    leaf = {key: d[key].detach().clone().requires_grad_(True)
            for key in ("x0", "q", "r", "xmin", "xmax", "umin", "umax")}
    b, S, dev = len(d["nx"]), int(d["N"][0]), _dev()
    two = lambda a, m: a.reshape(b, m)
    p = dict(A=d["A"].reshape(b, 1, 4, 4), B=d["B"].reshape(b, 1, 4, 1),
             e=d["e"].reshape(b, 1, 4), S=S, N=torch.full((b,), S, device=dev),
             q=two(leaf["q"], 4), r=two(leaf["r"], 1), x0=two(leaf["x0"], 4),
             rdu=torch.zeros(b, 1, dtype=F64, device=dev),
             u_prev=torch.zeros(b, 1, dtype=F64, device=dev), ref=two(d["ref"], 5),
             lo=torch.cat([two(leaf["xmin"], 4), two(leaf["umin"], 1)], -1),
             hi=torch.cat([two(leaf["xmax"], 4), two(leaf["umax"], 1)], -1))
    z = _algorithm(p, 1.0, -1.0, case["iters"], 0)[0]
    u, x = z[..., 4:].reshape(-1), z[..., :4].reshape(-1)
    gs = torch.autograd.grad([u, x], [leaf[key] for key in
                                      ("x0", "q", "r", "xmin", "xmax", "umin", "umax")],
                             [d["gu"], d["gx"]])
    return [u.detach(), x.detach(), *gs]

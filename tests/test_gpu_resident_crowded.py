"""The register-resident kernel without a deciding warp (schedule 3, n <= 16: batches of more CTAs than
SMs, or CTAs whose threads are all taken) when decisions are taken: momentum and restarts, stops on the
tolerance at different iterations, replayed masks and the stall test, on one CTA and on clusters, for
the size classes 4, 8 and 16, against the FP64 oracle.

FP64 takes its own decisions: iteration counts and states as the oracle's, iterates to 1e-10 at a fixed
count and 1e-9 at a tolerance. FP32 replays the oracle's restarts: 1e-4 at a fixed count; its c is a sum of m
squared differences of iterates within d of the oracle's, so |dc| <= 4 sqrt(m c) d + 4 m d^2, and a stop at
eps comes between the first iterations at which the oracle's c is below eps plus and minus that, with d
1e-5 of the iterates (their rounding over a hundred contractive iterations)."""
import numpy as np
import pytest
import torch

import oracle
from paper_2601_14414_gb300 import pimpc
from paper_2601_14414_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def relerr(a, b):
    return float(np.max(np.abs(a - b)) / max(np.max(np.abs(b)), 1e-12))


# by size class and CTAs per instance, FP32 then FP64: as many stages as the CTAs hold, and fewer
SIZES = {
    (4, 1): ([(2, 1, 341), (3, 1, 40), (1, 1, 7), (3, 1, 256)], [(2, 1, 170), (3, 1, 33), (1, 1, 7), (3, 1, 128)]),
    (8, 1): ([(5, 2, 36), (6, 2, 64), (4, 1, 3)], [(5, 2, 36), (6, 2, 64), (4, 1, 3)]),
    (16, 1): ([(9, 4, 15), (12, 4, 32), (8, 1, 1)], [(9, 4, 15), (12, 4, 16), (8, 1, 1)]),
    (4, 2): ([(2, 1, 600), (3, 1, 50)], [(2, 1, 300), (3, 1, 50)]),
    (8, 2): ([(6, 2, 110), (5, 1, 9)], [(6, 2, 110), (5, 1, 9)]),
    (16, 4): ([(12, 4, 100), (9, 2, 21)], [(12, 4, 50), (9, 2, 21)]),
}


def crowd(cls, precision, few):
    """The class's sizes in turn, one CTA more than the device has SMs (or, few, just the sizes)."""
    dims = SIZES[cls][0 if precision == pimpc.F32 else 1]
    some = []
    for j in range(len(dims) * (1 if few else 3)):
        i = W.random_ltv(8700 + 17 * cls[0] + j, *dims[j % len(dims)])
        rng = np.random.default_rng(8800 + j)
        i["ref"] = 0.2 * rng.standard_normal(i["nx"] + i["nu"])
        if j % 2:
            i["rdu"] = rng.uniform(0.1, 0.4, i["nu"])
        i["rho"] = 1.3
        some.append(i)
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    count = len(some) if few else max(len(some), sms // cls[1] + 1)
    return some, [some[j % len(some)] for j in range(count)]


def solver(insts, cls, precision, **opts):
    s = pimpc.Solver(insts, precision=precision, accel=1, **opts)
    s.set_schedule(pimpc.FAMILY_RESIDENT, 0, cls[1])
    return s


@pytest.mark.parametrize("cls", list(SIZES))
def test_fp64_decides_as_the_oracle(cls):
    some, insts = crowd(cls, pimpc.F64, False)
    s = solver(insts, cls, pimpc.F64, eps=-1.0, max_iters=80)
    r, its = s.solve(), s.iterates()
    ora = oracle.solve_batch(some, eps=-1.0, max_iters=80, accel=1, history=True)
    assert any(o["mask"][:-1].min() == 0 and o["mask"].max() == 1 for o in ora)  # momentum and restarts
    for j in range(len(insts)):
        o = ora[j % len(some)]
        assert r["iters"][j] == 80 and r["status"][j] == pimpc.MAXITER, j
        for key in ("z", "v", "th", "be", "la"):
            assert relerr(its[j][key], o[key]) <= 1e-10, (j, key)
    s.set_options(1e-6, 1500, 1)
    r = s.solve()
    ora = oracle.solve_batch(some, eps=1e-6, max_iters=1500, accel=1)
    assert len({o["iters"] for o in ora}) > 1
    for j in range(len(insts)):
        o = ora[j % len(some)]
        assert r["iters"][j] == o["iters"] and r["status"][j] == o["status"], j
        assert relerr(r["u"][j], o["u"]) <= 1e-9 and relerr(r["x"][j], o["x"]) <= 1e-9, j
    s.close()


@pytest.mark.parametrize("few", [False, True])
@pytest.mark.parametrize("cls", list(SIZES))
def test_fp32_with_the_oracles_restarts(cls, few):
    some, insts = crowd(cls, pimpc.F32, few)
    K = 100
    ora = oracle.solve_batch(some, eps=-1.0, max_iters=K, accel=1, history=True)
    mask = np.ascontiguousarray(np.stack([ora[j % len(some)]["mask"] for j in range(len(insts))]).astype(np.uint8))
    s = solver(insts, cls, pimpc.F32, eps=-1.0, max_iters=K)
    pimpc.pimpc_set_restart_mask(s.h, mask, K)
    r = s.solve()
    for j in range(len(insts)):
        o = ora[j % len(some)]
        assert r["iters"][j] == K
        assert relerr(r["u"][j], o["u"]) <= 1e-4 and relerr(r["x"][j], o["x"]) <= 1e-4, j
    eps = 1e-2
    s.set_options(eps, K, 1)
    r = s.solve()
    for j in range(len(insts)):
        o = ora[j % len(some)]
        d = 1e-5 * max(np.max(np.abs(o[key])) for key in ("z", "v", "th", "be", "la"))
        m = 6 * o["z"].size * some[j % len(some)]["rho"]
        dc = 4 * np.sqrt(m * eps) * d + 4 * m * d * d

        def first(bound):
            hit = np.flatnonzero(o["c_hist"] <= bound)
            return int(hit[0]) + 1 if len(hit) else K
        assert first(eps + dc) <= r["iters"][j] <= first(eps - dc), j
        assert r["status"][j] == (pimpc.CONVERGED if r["c"][j] <= eps else pimpc.MAXITER), j
    s.close()


@pytest.mark.parametrize("cls", [(4, 1), (8, 1), (16, 4)])
def test_fp32_stall_stop(cls):
    some, insts = crowd(cls, pimpc.F32, False)
    s = solver(insts, cls, pimpc.F32, eps=1e-14, max_iters=20000)
    pimpc.pimpc_set_stall(s.h, 200, 0.5)
    r = s.solve()
    st = np.asarray(r["status"])
    assert np.all((st == pimpc.STALLED) | (st == pimpc.CONVERGED)) and np.any(st == pimpc.STALLED)
    ora = oracle.solve_batch(some, eps=1e-22, max_iters=60000, accel=1)
    for j in range(len(insts)):
        o = ora[j % len(some)]
        scale = max(1.0, np.max(np.abs(o["u"])), np.max(np.abs(o["x"])))
        err = max(np.max(np.abs(r["u"][j] - o["u"])), np.max(np.abs(r["x"][j] - o["x"])))
        assert err <= 1e-4 * scale, j
    s.close()


@pytest.mark.parametrize("precision,dims", [
    (pimpc.F64, [(12, 4, 60), (11, 4, 43)]), (pimpc.F64, [(12, 4, 83), (9, 5, 80)]),
    (pimpc.F32, [(12, 4, 121), (13, 3, 33)]), (pimpc.F32, [(14, 2, 150)]),
])
def test_clusters_of_five_and_six(precision, dims):
    # batches of two and a half rounds of CTAs or more whose largest instance needs more than four CTAs
    some = [W.random_ltv(8900 + j, *dims[j % len(dims)]) for j in range(4)]
    count = torch.cuda.get_device_properties(0).multi_processor_count // 2
    K = 60
    ora = oracle.solve_batch(some, eps=-1.0, max_iters=K, accel=1, history=True)
    mask = np.ascontiguousarray(np.stack([ora[j % 4]["mask"] for j in range(count)]).astype(np.uint8))
    s = pimpc.Solver([some[j % 4] for j in range(count)], precision=precision, eps=-1.0, max_iters=K, accel=1)
    s.set_schedule(pimpc.FAMILY_RESIDENT)
    pimpc.pimpc_set_restart_mask(s.h, mask, K)
    r = s.solve()
    tol = 1e-10 if precision == pimpc.F64 else 1e-4
    for j in range(count):
        o = ora[j % 4]
        assert r["iters"][j] == K
        assert relerr(r["u"][j], o["u"]) <= tol and relerr(r["x"][j], o["x"]) <= tol, j
    s.close()

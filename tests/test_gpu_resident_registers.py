"""The register-resident kernel (schedule 3, n <= 16) against the FP64 oracle at the edges of its
size classes: n at and around 4, 8 and 16, one stage, horizons that fill a CTA's threads or leave
a ragged last CTA, every cluster size, both stage kinds. Tolerances as in the other schedules'
parity tests: 1e-10 in FP64 and 1e-4 in FP32 at a fixed iteration count."""
import numpy as np
import pytest

import oracle
from paper_2601_14414_gb300 import pimpc
from paper_2601_14414_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def relerr(a, b):
    return float(np.max(np.abs(a - b)) / max(np.max(np.abs(b)), 1e-12))


def check(insts, precision, cluster, iters, accel, warm=0):
    s = pimpc.Solver(insts, precision=precision, eps=-1.0, max_iters=iters, accel=accel)
    s.set_schedule(pimpc.FAMILY_RESIDENT, 0, cluster)
    ora = [oracle.solve(i, eps=-1.0, max_iters=iters, accel=accel, history=True) for i in insts]
    if accel:  # the oracle's restart decisions, so that rounding cannot change one
        mask = np.ascontiguousarray(np.stack([o["mask"] for o in ora]).astype(np.uint8))
        pimpc.pimpc_set_restart_mask(s.h, mask, iters)
    r = s.solve()
    its = s.iterates()
    tol = 1e-10 if precision == pimpc.F64 else 1e-4
    for j, o in enumerate(ora):
        assert relerr(r["u"][j], o["u"]) <= tol, j
        assert relerr(r["x"][j], o["x"]) <= tol, j
        if precision == pimpc.F64:
            for key in ("z", "v", "th", "be", "la"):
                assert relerr(its[j][key], o[key]) <= tol, (j, key)
            # c sums 6 N n squared differences of iterates that are each within d of the
            # oracle's: |dc| <= 2 sqrt(6 N n c) 2 d + 6 N n (2 d)^2
            d = tol * max(np.max(np.abs(o[key])) for key in ("z", "v", "th", "be", "la"))
            m = 6 * o["z"].size
            assert abs(r["c"][j] - o["c"]) <= 4 * np.sqrt(m * o["c"]) * d + 4 * m * d * d
    s.close()


DIMS = [(1, 1), (2, 1), (3, 1), (4, 1), (6, 2), (5, 3), (8, 1), (12, 4), (1, 15), (15, 1), (9, 7)]


@pytest.mark.parametrize("precision", [pimpc.F32, pimpc.F64])
@pytest.mark.parametrize("accel", [0, 1])
def test_size_classes(precision, accel):
    for nx, nu in DIMS:
        n = nx + nu
        insts = [W.random_ltv(7000 + 10 * n + N, nx, nu, N) for N in (1, 2, 128 // n + 1)]
        check(insts, precision, 0, 80, accel)


@pytest.mark.parametrize("cluster", [1, 2, 4, 8, 16])
@pytest.mark.parametrize("precision", [pimpc.F32, pimpc.F64])
def test_clusters(precision, cluster):
    # N = C (every CTA one stage and two neighbours), ragged, and two classes in one batch
    check([W.random_ltv(7100, 3, 1, cluster), W.random_ltv(7101, 12, 4, 2 * cluster + 3)],
          precision, cluster, 60, 1)
    check([W.random_ltv(7102, 2, 1, 40 * cluster - 1)], precision, cluster, 60, 1)
    check([W.plain_lti(7103, 4, 2, 17 + cluster)], precision, cluster, 60, 1)


def test_cstr_long_horizon_exchanges_in_two_stages():
    # 945 threads per CTA: more than 128 warps in the cluster
    check([W.random_ltv(7200, 2, 1, 5000)], pimpc.F32, 16, 40, 1)


@pytest.mark.parametrize("precision", [pimpc.F32, pimpc.F64])
@pytest.mark.parametrize("accel", [0, 1])
def test_more_than_a_cluster(precision, accel):
    # FP64 instances too long for a cluster's four warps, and an FP32 one no cluster holds: CTAs
    # of a cooperative launch exchange through global memory (24 to 96 CTAs, ragged last ones)
    for nx, nu, N in ((12, 4, 200), (3, 2, 1009), (7, 5, 331)) if precision == pimpc.F64 else (
            (3, 2, 3001),):
        check([W.random_ltv(7400 + N, nx, nu, N)], precision, 0, 50, accel)
    if precision == pimpc.F64:
        check([W.random_ltv(7450 + j, 12, 4, 160 + j) for j in range(3)], precision, 0, 50, accel)


@pytest.mark.parametrize("mode", [1, 2])
def test_warm_start_of_long_instances(mode):
    inst = W.random_ltv(7460, 6, 3, 400)
    s = pimpc.Solver([inst], precision=pimpc.F64, eps=-1.0, max_iters=40, accel=1)
    s.set_schedule(pimpc.FAMILY_RESIDENT)
    s.solve()
    warm = {k: v.copy() for k, v in s.iterates()[0].items()}
    if mode == 2:
        warm = {k: np.concatenate([v[1:], v[-1:]], axis=0) for k, v in warm.items()}
    s.solve(warm_start=mode)
    got = s.iterates()[0]
    o = oracle.solve(inst, eps=-1.0, max_iters=40, accel=1, warm=warm)
    for key in ("z", "v", "th", "be", "la"):
        assert relerr(got[key], o[key]) <= 1e-10, key
    s.close()


def test_non_finite_dynamics_are_reported():
    inst = W.plain_lti(7300, 4, 2, 20)
    inst["x0"] = np.array([np.inf, 0.0, 0.0, 0.0])
    for precision in (pimpc.F32, pimpc.F64):
        for cluster in (1, 4):
            s = pimpc.Solver([inst], precision=precision, eps=-1.0, max_iters=20, accel=0)
            s.set_schedule(pimpc.FAMILY_RESIDENT, 0, cluster)
            r = s.solve()
            assert r["status"][0] == pimpc.NONFINITE and r["iters"][0] == 1
            s.close()

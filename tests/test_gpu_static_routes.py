"""pimpc_solve_static on each of its routes against the FP64 oracle: registers of one CTA, of a
cluster, of more CTAs than a cluster (FP64), shared memory of a cluster (n > 16), and tiles (too
long for a cluster, or more iterations than the momentum table holds). Tolerances as in the other
parity tests: 1e-10 in FP64, 1e-4 in FP32 at a fixed count of the plain iteration."""
import numpy as np
import pytest

import oracle
from paper_2601_14414_gb300 import pimpc
from paper_2601_14414_gb300 import workloads as W
from test_zz_no_alloc import relerr, run_static

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx,nu,N,iters", [(4, 2, 20, 60), (12, 4, 60, 60), (12, 4, 230, 60),
                                           (20, 6, 60, 60), (17, 2, 3, 60), (24, 8, 900, 20),
                                           (3, 1, 33, 4100)])
@pytest.mark.parametrize("precision", [pimpc.F32, pimpc.F64])
def test_routes(precision, nx, nu, N, iters):
    if precision == pimpc.F64 and N == 900:
        N = 700  # the tiles of 900 stages exceed the static array in FP64
    inst = W.random_ltv(8500 + N, nx, nu, N)
    accel = 1 if precision == pimpc.F64 and iters < 100 else 0
    u, x, its, c, st = run_static(inst, precision, -1.0, iters, accel)
    o = oracle.solve(inst, eps=-1.0, max_iters=iters, accel=accel)
    tol = 1e-10 if precision == pimpc.F64 else 1e-4
    assert its == iters and st == pimpc.MAXITER
    assert relerr(u, o["u"]) <= tol and relerr(x, o["x"]) <= tol


def test_stops_on_the_tolerance():
    inst = W.random_ltv(8600, 6, 2, 40)
    u, x, its, c, st = run_static(inst, pimpc.F64, 1e-9, 3000, 1)
    o = oracle.solve(inst, eps=1e-9, max_iters=3000, accel=1)
    assert st == pimpc.CONVERGED and its == o["iters"] and c <= 1e-9
    assert relerr(u, o["u"]) <= 1e-10

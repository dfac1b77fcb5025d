"""The stage cache at the sizes where its work is split differently: a warp per stage (few
stages), 16 and 8 lanes per stage (many), partial last rounds of the triangle, partial row chunks,
batches whose stages are not a multiple of a warp's, rho != 1, W_du. Checked through two FP64
iterations against the FP64 oracle, which inverts by another method (tolerance 1e-10, as the other
FP64 parity tests)."""
import numpy as np
import pytest

import oracle
from paper_2601_14414_gb300 import pimpc
from paper_2601_14414_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def relerr(a, b):
    return float(np.max(np.abs(a - b)) / max(np.max(np.abs(b)), 1e-12))


def check(insts, sample, rho):
    for i in insts:
        i["rho"] = rho
    s = pimpc.Solver(insts, precision=pimpc.F64, eps=-1.0, max_iters=2, accel=0)
    s.solve()
    its = s.iterates()
    for j in sample:
        o = oracle.solve(insts[j], eps=-1.0, max_iters=2, accel=0)
        for key in ("z", "v", "th", "be", "la"):
            assert relerr(its[j][key], o[key]) <= 1e-10, (j, key)
    s.close()


@pytest.mark.parametrize("rho", [1.0, 0.7])
@pytest.mark.parametrize("nmax,count", [(8, 3), (8, 40), (32, 3), (32, 40)])
def test_lanes_per_stage(nmax, count, rho):
    # 3 instances: a warp per stage; 40: more than 1216 stages, 8 lanes (n <= 8) or 16
    dims = [(nx, nu) for nx, nu in ((1, 1), (2, 1), (5, 3), (7, 1), (6, 2), (12, 4), (13, 5),
                                    (24, 8), (31, 1), (9, 23)) if nx + nu <= nmax]
    insts = []
    for j in range(count):
        nx, nu = dims[j % len(dims)]
        i = W.random_ltv(8000 + 50 * nmax + j, nx, nu, 37)
        if j % 3 == 1:
            i["rdu"] = np.linspace(0.1, 0.4, nu)
        insts.append(i)
    check(insts, range(min(count, 11)), rho)


def test_many_large_stage_invariant_instances():
    insts = [W.plain_lti(8200 + j, 48 if j % 2 else 3, 16 if j % 2 else 2, 3) for j in range(640)]
    check(insts, [0, 1, 638, 639], 1.3)

"""The stage cache in each band of its launch rule, by stages per SM: up to two (two warps a stage, all
rows of G at once), up to four (a warp a stage, one warp a CTA, rows of G in chunks), up to eight (four warps a
CTA), more (8 or 16 lanes a stage). One stage below, at and above each edge, more rows than a chunk, rho 1
and 0.7, W_du. Checked through two FP64 iterations against the FP64 oracle, which inverts by another method
(tolerance 1e-10, as the other FP64 parity tests)."""
import numpy as np
import pytest
import torch

import oracle
from paper_2601_14414_gb300 import pimpc
from paper_2601_14414_gb300 import workloads as W

pytestmark = pytest.mark.gpu

DIMS = {8: [(7, 1), (1, 1), (5, 3), (2, 1)], 32: [(24, 8), (1, 1), (31, 1), (9, 23), (13, 5)]}


def relerr(a, b):
    return float(np.max(np.abs(a - b)) / max(np.max(np.abs(b)), 1e-12))


@pytest.mark.parametrize("rho", [1.0, 0.7])
@pytest.mark.parametrize("nmax", [8, 32])
@pytest.mark.parametrize("per_sm", [2, 4, 8])
@pytest.mark.parametrize("over", [0, 1])
def test_bands(per_sm, over, nmax, rho):
    stages = per_sm * torch.cuda.get_device_properties(0).multi_processor_count + over
    dims, insts = DIMS[nmax], []
    while stages > 0:
        j = len(insts)
        nx, nu = dims[j % len(dims)]
        N = min(stages, (37, 5, 64, 90, 23)[j % 5])
        i = W.random_ltv(8000 + 50 * nmax + j, nx, nu, N, rho=rho)
        if j % 3 == 1:
            i["rdu"] = np.linspace(0.1, 0.4, nu)
        insts.append(i)
        stages -= N
    s = pimpc.Solver(insts, precision=pimpc.F64, eps=-1.0, max_iters=2, accel=0)
    s.solve()
    its = s.iterates()
    for j, o in enumerate(oracle.solve_batch(insts, eps=-1.0, max_iters=2, accel=0)):
        for key in ("z", "v", "th", "be", "la"):
            assert relerr(its[j][key], o[key]) <= 1e-10, (j, key)
    s.close()

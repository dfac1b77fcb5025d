"""The reduced iteration of the resident kernels (lambda = -beta, no state of its own) rounds no worse than
Algorithm 1 with all five vectors, which the lane groups run (schedule 0), in FP32 against the FP64 oracle.

Each instance's rms error of x and of u is compared, and the geometric mean of the ratios over 32 instances
must stay below 1.2. Emulated in numpy beforehand on such instances: 1.3 with beta summed into both
sides of gamma = Bbar du + beta - Abar xbar - ebar + lambda, where it cancels, and 0.8 to 1.1 without; 32
instances leave a scatter of a few per cent."""
import numpy as np
import pytest

import oracle
from paper_2601_14414_gb300 import pimpc
from paper_2601_14414_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx,nu,N", [(6, 2, 40), (4, 2, 40)])  # a thread per component, and per stage
def test_error_against_the_unreduced_iteration(nx, nu, N):
    insts = [W.plain_lti(9000 + j, nx, nu, N) for j in range(32)]
    ora = oracle.solve_batch(insts, eps=-1.0, max_iters=120, accel=0)
    err = {}
    for family in (pimpc.FAMILY_RESIDENT, pimpc.FAMILY_LANES):
        s = pimpc.Solver(insts, precision=pimpc.F32, eps=-1.0, max_iters=120, accel=0)
        s.set_schedule(family)
        r = s.solve()
        err[family] = {k: np.array([np.sqrt(np.mean((a - o[k]) ** 2)) for a, o in zip(r[k], ora)]) for k in ("u", "x")}
        s.close()
    for k in ("u", "x"):
        ratio = err[pimpc.FAMILY_RESIDENT][k] / err[pimpc.FAMILY_LANES][k]
        assert np.exp(np.mean(np.log(ratio))) <= 1.2, (k, ratio)

"""The register sweep of pimpc_backward (every instance with n <= 16 in one CTA's threads) against
the workspace sweep, which a batch takes as soon as one of its instances has n > 16: the same
instances alone and together with such a one. Sizes at the edges of the register classes and of
a CTA's threads (512 components in FP32, 256 for n > 8 in FP64), segments of one iteration, of some
and of all, both reference forms, each stage layout. FP64: both sweeps differentiate the same map
and differ by rounding only (1e-16 through a few dozen iterations: 1e-10 of the gradient allowed);
FP32: 1e-5, as in the other adjoint tests."""
import numpy as np
import pytest

from paper_2601_14414_gb300 import pimpc
from paper_2601_14414_gb300 import workloads as W

pytestmark = pytest.mark.gpu

LARGE = (20, 4, 12)


def instances(dims, per_stage, seed):
    out = []
    for j, (nx, nu, N) in enumerate(dims):
        i = W.random_ltv(seed + j, nx, nu, N, xabs=1.5, uabs=0.4)
        rng = np.random.default_rng(seed + 100 + j)
        i["ref"] = 0.3 * rng.standard_normal((N, nx + nu) if per_stage else nx + nu)
        i["rho"] = 1.2
        if j % 2:
            i["rdu"] = rng.uniform(0.1, 0.4, nu)
        out.append(i)
    return out


def gradients(insts, precision, iters, K, family):
    Wu = [np.random.default_rng(9 + j).standard_normal((i["N"], i["nu"])) for j, i in enumerate(insts)]
    Wx = [np.random.default_rng(59 + j).standard_normal((i["N"], i["nx"])) for j, i in enumerate(insts)]
    s = pimpc.Solver(insts, precision=precision, eps=-1.0, max_iters=iters, accel=0)
    if family is not None:
        s.set_schedule(family)
    s.solve()
    g = s.backward(Wu, Wx, checkpoint_every=K)
    s.close()
    return g


@pytest.mark.parametrize("precision,dims", [
    (pimpc.F64, [(1, 1, 1), (3, 1, 2), (2, 1, 128), (3, 2, 40)]),
    (pimpc.F64, [(5, 3, 64), (4, 2, 85), (7, 1, 3)]),
    (pimpc.F64, [(12, 4, 16), (8, 1, 28), (1, 15, 5)]),
    (pimpc.F32, [(3, 1, 128), (4, 1, 100), (6, 2, 64)]),
    (pimpc.F32, [(12, 4, 32), (15, 1, 31), (9, 2, 46)]),
])
@pytest.mark.parametrize("iters,K,family,per_stage", [
    (33, 5, None, False), (33, 1, None, True), (24, 24, pimpc.FAMILY_RESIDENT, True),
    (7, 100, pimpc.FAMILY_BLOCKED, False),
])
def test_registers_match_the_workspace_sweep(precision, dims, iters, K, family, per_stage):
    small = instances(dims, per_stage, 9000)
    a = gradients(small, precision, iters, K, family)
    b = gradients(small + instances([LARGE], per_stage, 9500), precision, iters, K, family)
    tol = 1e-10 if precision == pimpc.F64 else 1e-5
    for j in range(len(small)):
        for name in ("x0", "q", "r", "ref", "xmin", "xmax", "umin", "umax"):
            want = np.asarray(b[name][j])
            got = np.asarray(a[name][j])
            assert np.max(np.abs(got - want)) <= tol * max(1.0, np.max(np.abs(want))), (j, name)

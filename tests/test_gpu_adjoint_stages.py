"""The backward sweep with one thread per stage (FP32, at most 4 states and 2 inputs, horizons up to
256) against the workspace sweep, which a batch takes as soon as one of its instances is too large:
the same instances alone and together with a large one. (Every batch here has an instance with more
components than a CTA of the kernel with one thread per component holds.) Each size class with exact and padded sizes,
horizons at the edges of a warp and of a CTA, segments of one iteration, of some and of all, both
reference forms, with and without the gradients that need the primal iterates. Both sweeps
differentiate the same map in FP32 (6e-8 per operation through a few dozen contractive iterations):
1e-5, as in the other adjoint tests."""
import numpy as np
import pytest

from paper_2601_14414_gb300 import pimpc
from paper_2601_14414_gb300 import workloads as W

pytestmark = pytest.mark.gpu

NAMES = ("x0", "q", "r", "ref", "xmin", "xmax", "umin", "umax")


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


def gradients(insts, iters, K, family):
    Wu = [np.random.default_rng(9 + j).standard_normal((i["N"], i["nu"])) for j, i in enumerate(insts)]
    Wx = [np.random.default_rng(59 + j).standard_normal((i["N"], i["nx"])) for j, i in enumerate(insts)]
    s = pimpc.Solver(insts, precision=pimpc.F32, eps=-1.0, max_iters=iters, accel=0)
    if family is not None:
        s.set_schedule(family)
    s.solve()
    g = s.backward(Wu, Wx, checkpoint_every=K)
    s.close()
    return g


@pytest.mark.parametrize("dims", [
    [(1, 1, 1), (2, 1, 33), (2, 1, 256)],
    [(4, 1, 20), (3, 1, 31), (4, 1, 32), (1, 1, 2), (4, 1, 129)],
    [(4, 2, 64), (3, 2, 65), (2, 2, 255), (4, 1, 1)], [(4, 2, 256)],
])
@pytest.mark.parametrize("iters,K,family,per_stage", [
    (33, 5, None, False), (33, 1, None, True), (24, 24, None, True), (7, 100, pimpc.FAMILY_BLOCKED, False),
])
def test_stage_threads_match_the_workspace_sweep(dims, iters, K, family, per_stage):
    small = instances(dims, per_stage, 9000)
    a = gradients(small, iters, K, family)
    b = gradients(small + instances([(20, 4, 12)], per_stage, 9500), iters, K, family)
    for j in range(len(small)):
        for name in NAMES:
            want, got = np.asarray(b[name][j]), np.asarray(a[name][j])
            assert np.max(np.abs(got - want)) <= 1e-5 * max(1.0, np.max(np.abs(want))), (j, name)


def test_crowded_batches_match_small_ones():
    # more than two rounds of CTAs of a thread per component: the same instances in a batch of that
    # size (a thread per stage) and in batches small enough for a thread per component
    import torch
    count = 2 * torch.cuda.get_device_properties(0).multi_processor_count + 1
    some = instances([(4, 1, 100), (2, 1, 90), (3, 1, 64)], False, 9200)
    b = gradients(some, 40, 11, pimpc.FAMILY_RESIDENT)
    a = gradients([some[j % 3] for j in range(count)], 40, 11, pimpc.FAMILY_RESIDENT)
    # the weights of the loss are drawn by position, so only the first three compare
    for j in range(3):
        for name in NAMES:
            want, got = np.asarray(b[name][j]), np.asarray(a[name][j])
            assert np.max(np.abs(got - want)) <= 1e-5 * max(1.0, np.max(np.abs(want))), (j, name)

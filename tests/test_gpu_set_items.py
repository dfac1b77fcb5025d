"""FP64 batches on plain stage blocks (schedule 0): each of the two kernels gets items of its own
sub-chunks. Box constraints run CTAs of 256 threads with 256 // n slots, one of them the next stage's;
input sets run lane groups of 8, 16 or 32 lanes in CTAs of 128. The item counts are those of whole
sub-chunks, and solves to a tolerance (instances that stop one after the other, so that the lists are
compacted and the fine items take over) agree with the oracle with the set on, off and on again:
1e-10 at a fixed count, iteration counts equal to the tolerance."""
import numpy as np
import pytest

import oracle
from paper_2601_14414_gb300 import pimpc
from paper_2601_14414_gb300 import workloads as W

pytestmark = pytest.mark.gpu

DIMS = [(4, 2, 60), (12, 4, 45), (14, 5, 33), (2, 1, 131), (16, 1, 24), (9, 3, 7)]


def relerr(a, b):
    return float(np.max(np.abs(a - b)) / max(np.max(np.abs(b)), 1e-12))


def lanes(n):
    return 128 // (8 if n <= 8 else 16 if n <= 16 else 32)


def full(n):
    return 256 // n - 1


def count(stages, scale):
    return sum(-(-N // (stages(nx + nu) * max(scale, 1))) for nx, nu, N in DIMS)


@pytest.mark.parametrize("scale", [0, 2])
def test_each_kernel_has_its_own_items(scale):
    insts = [W.random_ltv(9300 + j, nx, nu, N) for j, (nx, nu, N) in enumerate(DIMS)]
    b, tot = len(insts), sum(i["nu"] for i in insts)
    s = pimpc.Solver(insts, precision=pimpc.F64, eps=-1.0, max_iters=40, accel=1)
    s.set_schedule(pimpc.FAMILY_LANES, 0, scale)
    for on in (False, True, False, True):
        kind = np.full(b, pimpc.USET_BALL2 if on else pimpc.USET_BOX, np.int32)
        pimpc.pimpc_set_input_set(s.h, kind, np.full(b, 0.5), np.zeros(tot))
        got = s.schedule()
        want = count(lanes if on else full, scale)
        assert got["items"] == want and got["threads"] == (128 if on else 256)
        assert got["grid"] == want  # fewer items than the GPU holds CTAs
        cons = [dict(i, uset=dict(kind=pimpc.USET_BALL2, r=0.5)) if on else i for i in insts]
        s.set_options(-1.0, 40, 1)
        r = s.solve()
        for j, o in enumerate(oracle.solve_batch(cons, eps=-1.0, max_iters=40, accel=1)):
            assert relerr(r["u"][j], o["u"]) <= 1e-10 and relerr(r["x"][j], o["x"]) <= 1e-10, (on, j)
        s.set_options(1e-7, 3000, 1)
        r = s.solve()
        for j, o in enumerate(oracle.solve_batch(cons, eps=1e-7, max_iters=3000, accel=1)):
            assert r["iters"][j] == o["iters"] and r["status"][j] == o["status"], (on, j)
    s.close()

"""The resident schedule's kernel with one thread per stage (FP32, nx <= 4, nu <= 2, N <= 256, fixed
plain iterations) against the FP64 oracle: every size class with exact and
padded sizes, horizons at the edges of a warp and of a CTA and just beyond them (another kernel),
both stage kinds, warm starts, references per stage, a non-finite instance among finite ones.
Tolerance as in the other schedules' FP32 parity tests: 1e-4 at a fixed iteration count."""
import numpy as np
import pytest
import torch

import oracle
from paper_2601_14414_gb300 import pimpc
from paper_2601_14414_gb300 import workloads as W

pytestmark = pytest.mark.gpu

TOL = 1e-4


def relerr(a, b):
    return float(np.max(np.abs(a - b)) / max(np.max(np.abs(b)), 1e-12))


def repeated(dims, make):
    """One instance more than the device has SMs, the sizes in turn."""
    count = torch.cuda.get_device_properties(0).multi_processor_count + 1
    return [make(j, *dims[j % len(dims)]) for j in range(count)]


def ltv(j, nx, nu, N):
    i = W.random_ltv(8100 + j, nx, nu, N)
    rng = np.random.default_rng(8600 + j)
    i["ref"] = 0.2 * rng.standard_normal((N, nx + nu))
    i["rho"] = 1.3
    if j % 2:
        i["rdu"] = rng.uniform(0.1, 0.4, nu)
    return i


def solver(insts, iters):
    s = pimpc.Solver(insts, precision=pimpc.F32, eps=-1.0, max_iters=iters, accel=0)
    s.set_schedule(pimpc.FAMILY_RESIDENT)
    return s


def compare(insts, r, its, ora):
    for j, o in enumerate(ora):
        assert relerr(r["u"][j], o["u"]) <= TOL and relerr(r["x"][j], o["x"]) <= TOL, j
        for key in ("z", "v", "th", "be", "la"):
            assert relerr(its[j][key], o[key]) <= TOL, (j, key)
        # c sums 6 N n squared differences of iterates that are each within d of the oracle's
        d = TOL * max(np.max(np.abs(o[key])) for key in ("z", "v", "th", "be", "la"))
        m = 6 * o["z"].size * insts[j].get("rho", 1.0)
        assert abs(r["c"][j] - o["c"]) <= 4 * np.sqrt(m * o["c"]) * d + 4 * m * d * d, j
        assert r["iters"][j] == o["iters"] and r["status"][j] == pimpc.MAXITER, j


@pytest.mark.parametrize("dims", [
    [(2, 1, 1), (1, 1, 31), (2, 1, 33), (2, 1, 256)],
    [(4, 1, 1), (3, 1, 32), (4, 1, 65), (1, 1, 2), (4, 1, 100)],
    [(4, 2, 1), (3, 2, 64), (2, 2, 97), (4, 1, 40), (4, 2, 80)],
    [(3, 1, 256), (4, 1, 255)], [(4, 2, 256), (2, 1, 254)], [(4, 1, 257), (3, 1, 258)],
])
@pytest.mark.parametrize("iters", [1, 2, 61])
def test_fixed_iterations_match_the_oracle(dims, iters):
    insts = repeated(dims, ltv)
    s = solver(insts, iters)
    r = s.solve()
    compare(insts, r, s.iterates(), oracle.solve_batch(insts, eps=-1.0, max_iters=iters, accel=0))
    s.close()


@pytest.mark.parametrize("nx,nu,N", [(2, 1, 40), (4, 1, 100), (4, 2, 20)])
@pytest.mark.parametrize("mode", [1, 2])
def test_stage_invariant_instances_and_warm_starts(nx, nu, N, mode):
    insts = repeated([(nx, nu, N)], lambda j, *d: W.plain_lti(8300 + j, *d))
    s = solver(insts, 30)
    r = s.solve()
    compare(insts, r, s.iterates(), oracle.solve_batch(insts, eps=-1.0, max_iters=30, accel=0))
    warm = s.iterates()
    if mode == 2:
        warm = [{k: np.concatenate([v[1:], v[-1:]], axis=0) for k, v in w.items()} for w in warm]
    r = s.solve(warm_start=mode)
    compare(insts, r, s.iterates(), [oracle.solve(i, eps=-1.0, max_iters=30, accel=0, warm=w)
                                     for i, w in zip(insts, warm)])
    s.close()


def test_a_non_finite_instance_stops_alone():
    insts = repeated([(4, 1, 30)], lambda j, *d: W.plain_lti(8400 + j, *d))
    insts[3]["x0"] = np.array([np.inf, 0.0, 0.0, 0.0])
    s = solver(insts, 20)
    r = s.solve()
    assert r["status"][3] == pimpc.NONFINITE and r["iters"][3] == 1
    good = [j for j in range(len(insts)) if j != 3]
    ora = oracle.solve_batch([insts[j] for j in good], eps=-1.0, max_iters=20, accel=0)
    its = s.iterates()
    compare([insts[j] for j in good], {k: [r[k][j] for j in good] for k in r}, [its[j] for j in good], ora)
    s.close()

"""FP64 iterations on full warps (schedule 0, box constraints) against the FP64 oracle at a fixed
iteration count (1e-10, as the other FP64 parity tests): slots that fill a CTA's 256 threads exactly
or leave some over, sub-chunks cut by the shared-memory budget, items that end inside a sub-chunk,
one stage, many inputs, both stage kinds, per-stage references, warm starts, and the change to the
lane groups and back when an input set is put on and taken off."""
import numpy as np
import pytest

import oracle
from paper_2601_14414_gb300 import pimpc
from paper_2601_14414_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def relerr(a, b):
    return float(np.max(np.abs(a - b)) / max(np.max(np.abs(b)), 1e-12))


def batch(dims, seed, per_stage=False):
    out = []
    for j, (nx, nu, N) in enumerate(dims):
        i = W.random_ltv(seed + j, nx, nu, N)
        i["ref"] = 0.2 * np.random.default_rng(seed + j).standard_normal((N, nx + nu) if per_stage else nx + nu)
        if j % 3 == 1:
            i["rdu"] = np.full(nu, 0.3)
        out.append(i)
    return out


DIMS = [(1, 1, 300), (2, 1, 85), (3, 1, 1), (12, 4, 33), (15, 1, 16), (24, 8, 50), (31, 1, 9),
        (1, 31, 13), (14, 5, 143), (9, 23, 11), (7, 2, 29)]


@pytest.mark.parametrize("items", [0, 1, 3])
@pytest.mark.parametrize("accel", [0, 1])
def test_matches_the_oracle(items, accel):
    insts = batch(DIMS, 9700, per_stage=items == 1)
    s = pimpc.Solver(insts, precision=pimpc.F64, eps=-1.0, max_iters=60, accel=accel)
    s.set_schedule(pimpc.FAMILY_LANES, 0, items)
    assert s.schedule()["threads"] == 256
    r = s.solve()
    its = s.iterates()
    ora = oracle.solve_batch(insts, eps=-1.0, max_iters=60, accel=accel)
    for j, o in enumerate(ora):
        for key in ("z", "v", "th", "be", "la"):
            assert relerr(its[j][key], o[key]) <= 1e-10, (j, key)
        assert r["iters"][j] == 60


@pytest.mark.parametrize("dims", [[(4, 2, 20), (48, 16, 75), (3, 1, 1), (33, 31, 40), (7, 5, 300)]])
def test_stage_invariant(dims):
    insts = [W.plain_lti(9800 + j, nx, nu, N) for j, (nx, nu, N) in enumerate(dims)]
    s = pimpc.Solver(insts, precision=pimpc.F64, eps=-1.0, max_iters=60, accel=1)
    r = s.solve()
    for j, o in enumerate(oracle.solve_batch(insts, eps=-1.0, max_iters=60, accel=1)):
        assert relerr(r["u"][j], o["u"]) <= 1e-10 and relerr(r["x"][j], o["x"]) <= 1e-10, j


@pytest.mark.parametrize("n", [51, 52])
def test_five_slots_and_four(n):
    # the widest instance that gives a CTA five slots, and one more, which the lane groups take
    insts = [W.plain_lti(9850 + j, nx, nu, N) for j, (nx, nu, N) in enumerate([(n - 11, 11, 30), (4, 2, 20)])]
    s = pimpc.Solver(insts, precision=pimpc.F64, eps=-1.0, max_iters=60, accel=1)
    r = s.solve()
    for j, o in enumerate(oracle.solve_batch(insts, eps=-1.0, max_iters=60, accel=1)):
        assert relerr(r["u"][j], o["u"]) <= 1e-10 and relerr(r["x"][j], o["x"]) <= 1e-10, j


def test_stops_warm_starts_and_input_sets():
    insts = batch(DIMS[3:8], 9900)
    s = pimpc.Solver(insts, precision=pimpc.F64, eps=1e-6, max_iters=4000, accel=1)
    r = s.solve()
    ora = oracle.solve_batch(insts, eps=1e-6, max_iters=4000, accel=1)
    for j, o in enumerate(ora):
        assert r["iters"][j] == o["iters"] and relerr(r["u"][j], o["u"]) <= 1e-9, j
    warm = s.iterates()
    s.set_options(-1.0, 15, 1)
    s.solve(warm_start=2)
    its = s.iterates()
    for j, inst in enumerate(insts):
        w = {k: np.concatenate([v[1:], v[-1:]], axis=0) for k, v in warm[j].items()}
        o = oracle.solve(inst, eps=-1.0, max_iters=15, accel=1, warm=w)
        assert relerr(its[j]["z"], o["z"]) <= 1e-10 and relerr(its[j]["la"], o["la"]) <= 1e-9, j
    tot = sum(i["nu"] for i in insts)
    pimpc.pimpc_set_input_set(s.h, np.full(len(insts), pimpc.USET_BALL2, np.int32),
                              np.full(len(insts), 0.5), np.zeros(tot))
    assert s.schedule()["threads"] == 128
    s.solve()
    sets = s.iterates()
    for j, inst in enumerate(insts):
        o = oracle.solve(dict(inst, uset=dict(kind=pimpc.USET_BALL2, r=0.5)), eps=-1.0, max_iters=15, accel=1)
        assert relerr(sets[j]["z"], o["z"]) <= 1e-10, j
    pimpc.pimpc_set_input_set(s.h, np.zeros(len(insts), np.int32), np.zeros(len(insts)), None)
    s.solve()
    box = s.iterates()
    for j, inst in enumerate(insts):
        o = oracle.solve(inst, eps=-1.0, max_iters=15, accel=1)
        assert relerr(box[j]["z"], o["z"]) <= 1e-10, j
    s.close()

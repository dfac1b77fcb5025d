"""The gradient sums of pimpc_backward keep FP64's range and bits with FP32 iterations.

The iteration is positively homogeneous: with x0, e, the reference and the bounds scaled by 2^a every
iterate scales by 2^a, and with the loss's gradient scaled by 2^b every adjoint by 2^b. As long as FP32
iterates and adjoints stay normal, powers of two change no rounding, so the gradients of the scaled
problem equal the others times their power of two exactly: x0's, the reference's and the bounds' 2^b, the
weights' 2^(a + b), whose sums of products leave FP32's range at both ends here (2^135 and 2^-140). Each
sweep: a thread per component, a thread per stage (more components than a CTA has threads, or more than
two rounds of such CTAs), vectors in global memory."""
import numpy as np
import pytest

from paper_2601_14414_gb300 import pimpc
from paper_2601_14414_gb300 import workloads as W

pytestmark = pytest.mark.gpu

POWERS = dict(x0=(0, 1), ref=(0, 1), xmin=(0, 1), xmax=(0, 1), umin=(0, 1), umax=(0, 1), q=(1, 1), r=(1, 1))


def gradients(dims, a, b):
    insts, gu, gx = [], [], []
    for j, (nx, nu, N) in enumerate(dims):
        i = W.random_ltv(9600 + j, nx, nu, N, xabs=1.5, uabs=0.4)
        rng = np.random.default_rng(9700 + j)
        i["ref"] = 0.3 * rng.standard_normal(nx + nu)
        for key in ("x0", "e", "ref", "xmin", "xmax", "umin", "umax"):
            i[key] = np.ldexp(i[key], a)
        insts.append(i)
        gu.append(np.ldexp(rng.standard_normal((N, nu)), b))
        gx.append(np.ldexp(rng.standard_normal((N, nx)), b))
    s = pimpc.Solver(insts, precision=pimpc.F32, eps=-1.0, max_iters=30, accel=0)
    s.solve()
    g = s.backward(gu, gx, checkpoint_every=7)
    s.close()
    return g


@pytest.mark.parametrize("dims", [
    [(3, 1, 15), (6, 2, 40), (12, 4, 9)], [(4, 1, 129), (2, 1, 30)], [(4, 2, 100)], [(20, 4, 12), (4, 1, 10)],
])
@pytest.mark.parametrize("a,b", [(40, 95), (-70, -70)])
def test_gradients_scale_exactly(dims, a, b):
    base, got = gradients(dims, 0, 0), gradients(dims, a, b)
    for name, (pa, pb) in POWERS.items():
        for j in range(len(dims)):
            want = np.ldexp(np.asarray(base[name][j]), pa * a + pb * b)
            assert np.array_equal(np.asarray(got[name][j]), want), (name, j)

"""The FP64 node kernels round alike: which one solves a node does not show in its solution.

The method reads indicators and moments of disks without an eigenvalue as differences of
node solutions that nearly cancel, so a kernel that rounds differently (a quotient formed as
a product with a rounded reciprocal, say) moves them by many times its own error. Nodes in
shared memory (lu_small.cu, lu_resident.cu) therefore give the blocked routines' bits
(lu_core.cuh). Those solve a node that a precision form's refinement gives up: one sweep is
never enough for a remaining error of 1e-15. The warp-per-node kernel takes small orders in
every form, and is compared with pmcim_solve_points_noalloc, whose solve is the same for
orders of one block (a disk with N = 2 and dyadic centre and radius has exact nodes c +- r
and weights +- r / 2: C0 = (r / 2)(X_0 - X_1), one rounding per part).
"""
import numpy as np
import pytest

import workloads as w
from tests.test_gpu_parity import pm  # noqa: F401
from tests.test_zz_no_alloc import _call_noalloc

pytestmark = pytest.mark.gpu


def _problem(n, l):
    rng = np.random.default_rng(31 * n + l)
    A = [rng.random((n, n)) - 0.5 + 1j * (rng.random((n, n)) - 0.5) for _ in range(3)]
    prob = w.Problem(n, [(A[0], w.MONOMIAL, 0, 0.0), (A[1], w.MONOMIAL, 1, 0.0), (A[2], w.EXP_NEG, 0, 0.5)])
    return prob, np.asfortranarray(rng.random((n, l)) - 0.5 + 1j * (rng.random((n, l)) - 0.5))


@pytest.mark.parametrize("n,l", [(1, 3), (2, 16), (5, 1), (17, 5), (24, 1), (32, 16)])
def test_small_kernel_gives_the_blocked_kernels_bits(pm, n, l):  # noqa: F811
    prob, V = _problem(n, l)
    c, r = 0.25 - 0.125j, 0.5
    X = _call_noalloc(pm, prob, np.array([c + r, c - r]), V)
    P = pm.Problem(n, prob.terms)
    C0, _, _, _ = P.moments([w.Region(c, r, 2)], V)
    P.close()
    assert np.array_equal(C0[0], (X[0] - X[1]) * (r / 2))


@pytest.mark.parametrize("n,l", [(3, 17), (32, 33), (33, 1), (33, 8), (40, 9), (63, 16), (64, 64), (65, 7), (96, 8),
                                 (104, 10), (118, 1)])
def test_resident_kernel_gives_the_blocked_kernels_bits(pm, n, l):  # noqa: F811
    prob, V = _problem(n, l)
    P = pm.Problem(n, prob.terms)
    reg = [w.Region(0.3 - 0.1j, 0.6, 8)]
    got = P.moments(reg, V)
    want = P.moments(reg, V, opt=pm.options(precision=pm.PREC_FP32_IR, max_ir_sweeps=1, tol_ir=1e-15))
    P.close()
    for a, b in zip(got, want):
        assert np.array_equal(a, b)

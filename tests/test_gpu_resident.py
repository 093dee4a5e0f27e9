"""FP64 nodes whose matrix stays in shared memory (lu_resident.cu) against the CPU oracle.

Same bound as the other moment tests. The sizes lie at the edges of the kernel's
range (just above the warp-per-node kernel, one to eight CTAs per SM, the largest
orders that fit at l = 1, 10 and 64, and the first that does not) and off its
8-row, 16-column tiles; tiny orders reach it with more than 16 probe columns.
"""
import math

import numpy as np
import pytest

import workloads as w
from tests.test_gpu_parity import _check_moments, pm  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,l", [(1, 17), (2, 64), (33, 1), (33, 16), (47, 3), (64, 8), (73, 16), (104, 10), (110, 10),
                                 (115, 10), (119, 1), (121, 1), (90, 64)])
def test_resident_nodes(pm, n, l):  # noqa: F811
    rng = np.random.default_rng(700 + 100 * n + l)
    A = [w.complex_gaussian(rng, (n, n)) / math.sqrt(n) for _ in range(3)]
    prob = w.Problem(n, [(A[d], w.MONOMIAL, d, 0.0) for d in range(3)])
    _check_moments(pm, prob, [w.Region(0.3 - 0.2j, 0.9, 4)], w.probe_block(rng, n, l))


def test_resident_batch_of_uneven_sizes(pm):  # noqa: F811
    """One call, several launches (by CTAs per SM), against one call per problem."""
    W = w.batched_quadratics([3, 5, 9, 12], l=4, n_lo=34, n_hi=118)
    P = [pm.Problem(x.problem.n, x.problem.terms) for x in W]
    regs = [x.regions[:1] for x in W]
    got = pm.batch_solve(P, regs, [x.V for x in W])
    one = [p.solve(r, x.V) for p, r, x in zip(P, regs, W)]
    assert np.array_equal(got["lam"], np.concatenate([r["lam"] for r in one]))
    for p in P:
        p.close()

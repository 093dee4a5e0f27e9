"""The certificates' bordered step takes any limit of refinement sweeps.

max_ir_sweeps is limited to 1..10 for the precision forms only; with FP64 node solves any
number is accepted, and the bordered step of pmcim_certify (and of pmcim_solve) refines with
it. A step that has converged is not changed by a larger limit.
"""
import numpy as np
import pytest

import workloads as w
from tests.test_gpu_certify import _random_starts, _spectrum, pm  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [20, 40, 200])
def test_more_sweeps_than_the_precision_forms_allow(pm, n):  # noqa: F811
    mu = _spectrum(n, seed=n)
    prob, _ = w.similarity_linear(mu, seed=n + 1)
    lam = mu[:: max(1, n // 24)]
    starts = _random_starts(n, len(lam), seed=5)
    h = pm.Problem(prob.n, prob.terms)
    got = {k: h.certify(lam, starts, opt=pm.options(max_ir_sweeps=k)) for k in (6, 10, 11, 17, 20, 33, 2 ** 31 - 1)}
    h.close()
    cert, acc = got[10]
    assert acc.all() and np.all(cert > 0)
    for k, (c, a) in got.items():
        assert np.array_equal(a, acc), k
        if k > 10:
            assert np.array_equal(c, cert), k

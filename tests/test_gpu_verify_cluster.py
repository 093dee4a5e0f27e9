"""sigma_min of values that share clusters of CTAs (lu_fp64.cu) against NumPy's SVD.

Orders at the edges of the 32-column panels, of the 32-row solve blocks and of the rule for
the cluster's size, with few values (1 to 8 CTAs a value) and more values than SMs.

T(z) = A + z B with sigma_min(A) = 0.05, its other singular values in [0.5, 2] and
|z| ||B|| <= 0.02, so that the inverse iteration (ratio below (0.07 / 0.48)^2 a step) stops
by its 1e-12 rule well before its 30 steps. A backward stable LU moves a singular value by a
modest multiple of n u ||T||, relative to 0.03: 1e-10 leaves a factor of ten at n = 300.
"""
import numpy as np
import pytest

import workloads as w
from tests.test_gpu_parity import pm  # noqa: F401

pytestmark = pytest.mark.gpu


def _problem(n, seed):
    rng = np.random.default_rng(seed)
    q1 = np.linalg.qr(w.complex_gaussian(rng, (n, n)))[0]
    q2 = np.linalg.qr(w.complex_gaussian(rng, (n, n)))[0]
    sv = np.concatenate([np.linspace(2.0, 0.5, n - 1), [0.05]])
    B = w.complex_gaussian(rng, (n, n))
    B *= 0.02 / np.linalg.norm(B, 2)
    return w.Problem(n, [((q1 * sv) @ q2, w.MONOMIAL, 0, 0.0), (B, w.MONOMIAL, 1, 0.0)]), rng


@pytest.mark.parametrize("n,m", [(1, 1), (2, 3), (31, 2), (32, 1), (33, 5), (63, 1), (64, 40), (65, 9), (128, 1),
                                 (130, 3), (257, 1), (300, 20), (48, 400)])
def test_sigma_min(pm, n, m):  # noqa: F811
    prob, rng = _problem(n, 40 + n)
    lam = rng.uniform(0, 1, m) * np.exp(2j * np.pi * rng.uniform(0, 1, m))
    P = pm.Problem(prob.n, prob.terms)
    sig, acc = P.verify(lam)
    P.close()
    A, B = prob.terms[0][0], prob.terms[1][0]
    ref = np.array([np.linalg.svd(A + z * B, compute_uv=False)[-1] for z in lam])
    assert np.max(np.abs(sig - ref) / ref) <= 1e-10
    assert not np.any(acc)


@pytest.mark.parametrize("n", [1, 33, 130])
def test_exact_zero_pivot(pm, n):  # noqa: F811
    """diag(1, 2, ...) - z I at z = n: the last pivot is exactly zero, in every CTA's eyes."""
    P = pm.Problem(n, [(np.diag(np.arange(1.0, n + 1)).astype(complex), w.MONOMIAL, 0, 0.0),
                       (-np.eye(n, dtype=complex), w.MONOMIAL, 1, 0.0)])
    sig, acc = P.verify(np.array([n, n + 0.5], dtype=complex))
    P.close()
    assert sig[0] == 0.0 and acc[0]
    assert abs(sig[1] - 0.5) <= 1e-10

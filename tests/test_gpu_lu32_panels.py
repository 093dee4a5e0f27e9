"""The FP32 LU's register panels and block solves (lu32.cuh) through the precision forms.

One disk of two nodes per case, against LAPACK: the refined solutions end within an
estimated 1e-11 |X_j| in the max norm, so ||dX_j||_F <= sqrt(n l) 1e-11 ||X_j||_F. Orders at
the edges of the panel classes (256, 512, 1024, 2048 rows), where a panel of 2, 4 or 8 rows
per thread and the global-memory panel above 2048 rows take over, last panels of one
column, right-hand sides of 1 to 64 columns, and matrices that make the pivot search work:
equal magnitudes in whole columns (ties), rows that all have to be interchanged, and a
column of zeros at some node.
"""
import math

import numpy as np
import pytest

import oracle as o
import workloads as w
from tests.test_gpu_parity import pm  # noqa: F401

pytestmark = pytest.mark.gpu


def _check(pm, prob, V, forms, reg=w.Region(0.3 - 0.2j, 0.9, 2)):  # noqa: F811
    n, l = V.shape
    z, wt = o.nodes_weights(reg.c, reg.r, reg.N)
    X = [np.linalg.solve(o.assemble_T(prob, zz), V) for zz in z]
    tol = math.sqrt(n * l) * 1e-11 * np.dot(abs(wt), [np.linalg.norm(x) for x in X])
    P = pm.Problem(n, prob.terms)
    for form in forms:
        C0, _, _, _ = P.moments([reg], V, opt=pm.options(precision=form))
        assert np.linalg.norm(C0[0] - sum(a * x for a, x in zip(wt, X))) <= tol, form
    P.close()


@pytest.mark.parametrize("n,l", [(33, 1), (64, 64), (97, 8), (255, 9), (256, 16), (257, 5), (289, 33), (511, 8),
                                 (513, 3), (1023, 4), (1025, 17), (2049, 2)])
def test_panel_classes(pm, n, l):  # noqa: F811
    rng = np.random.default_rng(11 * n + l)
    A = [w.complex_gaussian(rng, (n, n)) / math.sqrt(n) for _ in range(2)]
    prob = w.Problem(n, [(A[d], w.MONOMIAL, d, 0.0) for d in range(2)])
    forms = [pm.PREC_FP32_IR, pm.PREC_TF32X3_IR] + ([pm.PREC_BF16X3_IR] if n < 600 else [])
    _check(pm, prob, w.probe_block(rng, n, l), forms)


@pytest.mark.parametrize("n", [40, 260, 530])
def test_ties_and_interchanges(pm, n):  # noqa: F811
    rng = np.random.default_rng(n)
    V = w.probe_block(rng, n, 6)
    # a row permutation of a diagonally dominant matrix: every step interchanges rows
    D = w.complex_gaussian(rng, (n, n)) * (0.1 / math.sqrt(n)) + np.eye(n)
    prob = w.Problem(n, [(np.asfortranarray(np.roll(D, 7, axis=0)), w.MONOMIAL, 0, 0.0),
                         (0.01 + 0j, w.MONOMIAL, 1, 0.0)])
    _check(pm, prob, V, [pm.PREC_FP32_IR, pm.PREC_TF32X3_IR])
    # entries of one magnitude: the DFT matrix ties in every column
    F = np.exp(-2j * np.pi * np.outer(np.arange(n), np.arange(n)) / n) / math.sqrt(n)
    prob = w.Problem(n, [(np.asfortranarray(F), w.MONOMIAL, 0, 0.0), (3.0 + 0j, w.MONOMIAL, 1, 0.0)])
    _check(pm, prob, V, [pm.PREC_FP32_IR, pm.PREC_TF32X3_IR])


def test_zero_column_is_reported(pm):  # noqa: F811
    """Column 37 of T(z_0) is exactly zero: a singular node, reported and not fatal."""
    n = 96
    rng = np.random.default_rng(5)
    A = w.complex_gaussian(rng, (n, n))
    A[:, 37] = 0.0
    B = np.zeros((n, n), complex)
    B[:, 37] = w.complex_gaussian(rng, (n, 1))[:, 0]
    prob = w.Problem(n, [(np.asfortranarray(A), w.MONOMIAL, 0, 0.0), (np.asfortranarray(B), w.MONOMIAL, 1, 0.0)])
    P = pm.Problem(n, prob.terms)
    res = P.solve([w.Region(-0.5 + 0j, 0.5, 4)], w.probe_block(rng, n, 4), opt=pm.options(precision=pm.PREC_FP32_IR))
    assert res["status"][0] & pm.RS_SINGULAR_NODE
    P.close()

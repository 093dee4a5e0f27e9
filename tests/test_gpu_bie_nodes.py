"""Boundary-integral nodes of the precision forms (bie_nodes.cu, oz_refine.cu) against the oracle.

The refinement stops at an estimated error of 1e-11 |X_j| in the max norm, so that
||dX_j||_F <= sqrt(n l) 1e-11 ||X_j||_F, and the weighted sums carry at most that times
sum_j |w_j| ||X_j||_F. Sizes: just above the small kernel, at and off the 128-row blocks
and 32-wide chunks of the digit tiles, an odd number of column groups and more than a
tile's four; a circle (first column only), a circle with a dense term (the whole matrix)
and an ellipse, alone and in one batch with a coefficient problem.
"""
import math

import numpy as np
import pytest

import oracle as o
import workloads as w
from tests.test_gpu_parity import pm  # noqa: F401

pytestmark = pytest.mark.gpu


def _problem(curve, dense, rng):
    n = curve.samples.shape[1]
    terms = [(0.5 + 0j, w.MONOMIAL, 0, 0.0), (curve, w.HELMHOLTZ_DLP, 0, 0.0)]
    if dense:
        terms.append((w.complex_gaussian(rng, (n, n)) * (0.05 / math.sqrt(n)), w.MONOMIAL, 1, 0.0))
    return w.Problem(n, terms)


@pytest.mark.parametrize("n,l,kind", [(34, 3, "circle"), (34, 17, "ellipse"), (62, 8, "dense"), (128, 9, "circle"),
                                      (130, 40, "ellipse"), (130, 5, "dense"), (258, 12, "circle"),
                                      (258, 8, "ellipse")])
@pytest.mark.parametrize("form", ["fp32", "tf32x3"])
def test_moments(pm, n, l, kind, form):  # noqa: F811
    rng = np.random.default_rng(40 * n + l)
    curve = w.ellipse_curve(n, 1.2, 0.7) if kind == "ellipse" else w.circle_curve(n)
    prob = _problem(curve, kind == "dense", rng)
    V = w.probe_block(rng, n, l)
    P = pm.Problem(n, prob.terms)
    opt = pm.options(precision={"fp32": pm.PREC_FP32_IR, "tf32x3": pm.PREC_TF32X3_IR}[form])
    regs = [w.Region(0.5 - 1.25j, 0.2121, 8), w.Region(2.15 - 1.85j, 0.3, 4)]
    C0, C1, ph, _ = P.moments(regs, V, opt=opt)
    for g, reg in enumerate(regs):
        z, wt = o.nodes_weights(reg.c, reg.r, reg.N)
        X = [np.linalg.solve(o.assemble_T(prob, zz), V) for zz in z]
        nrm = [np.linalg.norm(x) for x in X]
        tol = math.sqrt(n * l) * 1e-11
        assert np.linalg.norm(C0[g] - sum(a * x for a, x in zip(wt, X))) <= tol * np.dot(abs(wt), nrm)
        assert np.linalg.norm(C1[g] - sum(a * b * x for a, b, x in zip(wt, z, X))) <= tol * np.dot(abs(wt * z), nrm)
        h = sum(2 * wt[j] * X[j][:, 0] for j in range(1, reg.N, 2))
        assert np.linalg.norm(ph[g] - h) <= 2 * tol * np.dot(abs(wt), nrm)
    P.close()


def test_batch_with_a_coefficient_problem(pm):  # noqa: F811
    """One launch for both kinds of nodes gives each problem the values of its own call."""
    S = w.scattering_disk(n=64, l=4)
    Q = w.quadratic_small(seed=3, n=48, l=8, N=32)
    E = w.Workload("ellipse", _problem(w.ellipse_curve(48, 1.2, 0.8), False, None), S.regions, S.V[:48, :3])
    opt = pm.options(precision=pm.PREC_FP32_IR)
    P = [pm.Problem(x.problem.n, x.problem.terms) for x in (S, Q, E)]
    regs = [S.regions[6:8], Q.regions[5:7], S.regions[34:37]]
    V = [S.V, Q.V, np.linalg.qr(E.V)[0]]
    got = pm.batch_solve(P, regs, V, opt=opt)
    one = [p.solve(r, v, opt=opt)["lam"] for p, r, v in zip(P, regs, V)]
    assert len(got["lam"]) == sum(len(x) for x in one) > 0
    assert np.max(np.abs(got["lam"] - np.concatenate(one))) <= 1e-10
    for p in P:
        p.close()

"""Nodes that a precision form solves again in FP64: few of them (a cluster of CTAs shares a
node), many (a CTA each), and both against the FP64 form, to the bit.

One refinement sweep is never enough for a remaining error of 1e-15, so every node of these
calls is solved again. Orders give clusters of 2, 4 and 8 CTAs, one column block and several,
a last block of one column, and fewer probe columns than CTAs.
"""
import numpy as np
import pytest

import workloads as w
from tests.test_gpu_parity import pm  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,l,N", [(34, 3, 8), (65, 1, 4), (130, 5, 8), (161, 17, 8), (257, 3, 4), (300, 64, 4),
                                   (34, 3, 256), (130, 5, 128)])
@pytest.mark.parametrize("form", ["fp32", "tf32x3"])
def test_same_solutions_as_the_fp64_form(pm, n, l, N, form):  # noqa: F811
    rng = np.random.default_rng(9 * n + l)
    A = [rng.random((n, n)) - 0.5 + 1j * (rng.random((n, n)) - 0.5) for _ in range(2)]
    V = np.asfortranarray(rng.random((n, l)) - 0.5 + 1j * (rng.random((n, l)) - 0.5))
    P = pm.Problem(n, [(-0.5 + 0.25j, w.MONOMIAL, 2, 0.0), (A[0], w.MONOMIAL, 0, 0.0), (A[1], w.EXP_NEG, 0, 0.5)])
    reg = [w.Region(0.3 - 0.1j, 0.6, N), w.Region(-1.0 + 0.5j, 0.25, N)]
    want = P.moments(reg, V)
    precision = {"fp32": pm.PREC_FP32_IR, "tf32x3": pm.PREC_TF32X3_IR}[form]
    got = P.moments(reg, V, opt=pm.options(precision=precision, max_ir_sweeps=1, tol_ir=1e-15))
    P.close()
    for a, b in zip(got, want):
        assert np.array_equal(a, b)


def test_boundary_integral_nodes(pm):  # noqa: F811
    """The same re-solve with T(z_j) as the assembly left it, circulant and not."""
    for curve in (w.circle_curve(130), w.ellipse_curve(130, 1.2, 0.7)):
        V = w.probe_block(np.random.default_rng(4), 130, 6)
        P = pm.Problem(130, [(0.5 + 0j, w.MONOMIAL, 0, 0.0), (curve, w.HELMHOLTZ_DLP, 0, 0.0)])
        reg = [w.Region(0.5 - 1.25j, 0.2, 8)]
        want = P.moments(reg, V)
        got = P.moments(reg, V, opt=pm.options(precision=pm.PREC_FP32_IR, max_ir_sweeps=1, tol_ir=1e-15))
        P.close()
        # (the assembly kernels add the identity part in another order: rounding of T(z_j), and
        # the solutions' condition is below 100 here)
        for a, b in zip(got, want):
            assert np.linalg.norm(a - b) <= 1e-12 * np.linalg.norm(b)

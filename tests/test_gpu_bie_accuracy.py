"""Boundary-integral nodes in a precision form at the tightest tolerance, against SciPy's Bessel values.

A node refined to the end is limited by T(z_j) and by its residuals, which are no less
accurate than FP64 products when the tolerance asks for more than the default: its error is
then at most that of a plain FP64 LU, whose elimination rounds n times as often (a factor of
two is left for the spread of 16 points). Node solutions are read from pf_abs =
sum_j |w_j| |X_j[:, 0]| of two nodes at nearly the same point.
"""
import numpy as np
import pytest

import workloads as w
from oracle import bie_ref
from tests.test_gpu_parity import pm  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("a,b", [(1.0, 1.0), (0.8, 1.1)])
@pytest.mark.parametrize("n", [34, 64, 128])
def test_tight_refinement_is_as_accurate_as_fp64(pm, n, a, b):  # noqa: F811
    t = 2.0 * np.pi * np.arange(n) / n
    c, s = np.cos(t), np.sin(t)
    cv = np.array([a * c, b * s, -a * s, b * c, -a * c, -b * s])
    curve = w.BoundaryCurve(cv, 0.5)
    rng = np.random.default_rng(n)
    V = np.asfortranarray(rng.standard_normal((n, 2)) + 1j * rng.standard_normal((n, 2)))
    zs = [complex(x, y) for x in (0.4, 1.1, 2.0, 3.0) for y in (-3.0, -2.0, -1.0, -0.3)]
    want = []
    for z in zs:
        T = 0.5 * np.eye(n) + 0.5 * bie_ref.dlp_matrix(cv, z)
        x = np.linalg.solve(T, V[:, 0])
        r = V[:, 0] - (T.astype(np.clongdouble) @ x.astype(np.clongdouble)).astype(complex)
        want.append(np.abs(x + np.linalg.solve(T, r)))
    P = pm.Problem(n, [(0.5 + 0j, w.MONOMIAL, 0, 0.0), (curve, w.HELMHOLTZ_DLP, 0, 0.0)])
    regs = [w.Region(z, 1e-10, 2) for z in zs]

    def error(opt):
        pa = P.moments(regs, V, opt=opt)[3]
        return np.array([np.linalg.norm(p / 1e-10 - x) / np.linalg.norm(x) for p, x in zip(pa, want)])

    plain = error(pm.options())
    for form in (pm.PREC_FP32_IR, pm.PREC_TF32X3_IR):
        tight = error(pm.options(precision=form, tol_ir=1e-15, max_ir_sweeps=10))
        assert np.median(tight) <= 2.0 * np.median(plain), (np.median(tight), np.median(plain))
        assert tight.max() <= 2.0 * plain.max(), (tight.max(), plain.max())
    P.close()

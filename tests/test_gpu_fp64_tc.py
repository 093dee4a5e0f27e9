"""FP64 nodes whose trailing updates run as exact digit products on the tensor cores
(lu_fp64_tc.cuh) against the CPU oracle.

Same bound as the other moment tests. The orders lie around the outer blocks of 64 columns
(with the 32 rows that must remain), the tiles of 128 rows and 16 columns, and the first
orders past the shared-memory-resident kernel; 64 probe columns widen the tiles' last column.
"""
import math

import numpy as np
import pytest

import oracle as o
import workloads as w
from tests.test_gpu_parity import _check_moments, pm  # noqa: F401

pytestmark = pytest.mark.gpu


def _quadratic(rng, n):
    return [w.complex_gaussian(rng, (n, n)) / math.sqrt(n) for _ in range(3)]


@pytest.mark.parametrize("n,l", [(100, 64), (122, 1), (127, 16), (128, 5), (129, 10), (159, 1), (160, 8), (161, 64),
                                 (192, 3), (223, 16), (224, 17), (225, 1), (320, 10), (385, 7), (500, 16)])
def test_moments(pm, n, l):  # noqa: F811
    rng = np.random.default_rng(900 + 100 * n + l)
    prob = w.Problem(n, [(a, w.MONOMIAL, d, 0.0) for d, a in enumerate(_quadratic(rng, n))])
    _check_moments(pm, prob, [w.Region(0.3 - 0.2j, 0.9, 4)], w.probe_block(rng, n, l),
                   opt=pm.options(precision=pm.PREC_FP64))


@pytest.mark.parametrize("rows,cols", [(40, 0), (0, 40), (40, 40), (700, 0)])
def test_scaled_rows_and_columns(pm, rows, cols):  # noqa: F811
    """T' = R T C and V' = R V with powers of two in R and C have C0' = C^{-1} C0. The scales
    change the pivots, so a solve loses some accuracy to them, LAPACK's too: the digits may not
    lose more than a small multiple of that (2^700 is past their range and takes the FMA pipes)."""
    rng = np.random.default_rng(77)
    n, l = 300, 6
    A = _quadratic(rng, n)
    V = w.probe_block(rng, n, l)
    R = 2.0 ** (rng.integers(-rows, rows + 1, n) if rows < 500 else np.full(n, rows))
    C = 2.0 ** rng.integers(-cols, cols + 1, n)
    reg = w.Region(0.1 + 0.1j, 0.4, 4)
    plain = w.Problem(n, [(a, w.MONOMIAL, d, 0.0) for d, a in enumerate(A)])
    scaled = w.Problem(n, [((R[:, None] * a) * C, w.MONOMIAL, d, 0.0) for d, a in enumerate(A)])
    X = o.moments(plain, reg.c, reg.r, reg.N, V).C0
    lapack = o.moments(scaled, reg.c, reg.r, reg.N, R[:, None] * V).C0 * C[:, None]
    P = pm.Problem(n, scaled.terms)
    got = P.moments([reg], R[:, None] * V, pm.options(precision=pm.PREC_FP64))[0][0] * C[:, None]
    P.close()
    assert np.linalg.norm(got - X) <= 4.0 * np.linalg.norm(lapack - X) + 1e-11 * np.linalg.norm(X)


def test_waits_that_run_out(pm):  # noqa: F811
    """With 16-cycle waits the updates end on the FMA pipes: the same bound holds."""
    rng = np.random.default_rng(78)
    prob = w.Problem(200, [(a, w.MONOMIAL, d, 0.0) for d, a in enumerate(_quadratic(rng, 200))])
    try:
        pm.debug_wait_limits(16, 0)
        _check_moments(pm, prob, [w.Region(0.3 - 0.2j, 0.9, 4)], w.probe_block(rng, 200, 10),
                       opt=pm.options(precision=pm.PREC_FP64))
    finally:
        pm.debug_wait_limits(0, 0)

"""A precision-form call of several waves whose nodes need very different workspaces.

The first wave holds some 490 000 small nodes, the second a few large ones with T(z_j) kept in
FP64 (17 MB each). Memory is planned wave by wave: many small nodes at the large ones' size
would be terabytes.
"""
import numpy as np
import pytest

import workloads as w
from tests.test_gpu_parity import pm  # noqa: F401

pytestmark = pytest.mark.gpu


def test_small_nodes_in_one_wave_and_large_ones_in_the_next(pm):  # noqa: F811
    rng = np.random.default_rng(17)
    opt = pm.options(precision=pm.PREC_FP32_IR, residual_fp64=1)
    n, l = 34, 64
    small = pm.Problem(n, [(-1.0 + 0j, w.MONOMIAL, 1, 0.0), (w.complex_gaussian(rng, (n, n)), w.MONOMIAL, 0, 0.0)])
    # no eigenvalue: nothing but the nodes' solutions is computed (16 GB of them, and one disk more)
    disks = [w.Region(50.0 + g, 0.5, 4096) for g in range((16 << 30) // (n * l * 16 * 4096) + 1)]
    n = 1024
    A = w.complex_gaussian(rng, (n, n)) / 32.0
    large = pm.Problem(n, [(-1.0 + 0j, w.MONOMIAL, 1, 0.0), (A, w.MONOMIAL, 0, 0.0), (0.1 * A, w.EXP_NEG, 0, 0.5)])
    reg, V = w.Region(0.2 + 0.1j, 0.03, 16), w.probe_block(rng, n, 8)
    one = large.solve([reg], V, opt=opt)
    got = pm.batch_solve([small, large], [disks, [reg]], [w.probe_block(rng, 34, l), V], opt=opt)
    assert len(one["lam"]) > 0
    assert np.array_equal(got["lam"], one["lam"])
    assert (got["problem_of"] == 1).all()
    small.close()
    large.close()

"""FP64 batches whose problems have different numbers of probe columns.

Nodes that fit shared memory are launched together by how many of them an SM holds. A
problem with few rows and many columns shares a launch with one of many rows and few
columns here, where the largest order and the largest column count together fit no SM.
"""
import math

import numpy as np
import pytest

import workloads as w
from tests.test_gpu_parity import pm  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("sizes", [[(110, 10), (60, 60)], [(118, 1), (100, 16), (33, 64)],
                                   [(115, 10), (90, 64), (47, 3), (52, 40)]])
def test_batch_with_different_probe_columns(pm, sizes):  # noqa: F811
    reg = w.Region(0.3 - 0.2j, 0.25, 16)
    P, V = [], []
    for n, l in sizes:
        rng = np.random.default_rng(50 * n + l)
        P.append(pm.Problem(n, [(w.complex_gaussian(rng, (n, n)) / math.sqrt(n), w.MONOMIAL, d, 0.0)
                                for d in range(3)]))
        V.append(w.probe_block(rng, n, l))
    got = pm.batch_solve(P, [[reg]] * len(P), V)
    one = [p.solve([reg], v) for p, v in zip(P, V)]
    assert np.array_equal(got["lam"], np.concatenate([r["lam"] for r in one]))
    assert len(got["lam"]) > 0
    for p in P:
        p.close()

"""The precision forms' indicators stay the recorded ones where they are sensitive to rounding.

On a disk without an eigenvalue the node solutions cancel in P f, and the indicator (Eq. 3.1)
carries the refinement's error (an estimated 1e-11 |X| at the most) divided by what is left of
the sum, here about 1e-7 of it. The indicator is then a number to within some 1e-6, and yet
users compare it from one version to the next: so an LU, a solve or a residual that rounds
differently must not replace another. The file holds the values that the forms gave when one
kernel solved a node from assembly to refinement. Inputs are uniform random numbers and IEEE
operations on them, the same on every machine.
"""
import json
import math
import os

import numpy as np
import pytest

import workloads as w

pytestmark = pytest.mark.gpu
GOLDEN = os.path.join(os.path.dirname(os.path.abspath(__file__)), "golden", "precision_form_indicators.json")
# orders in each class of panels (rows per thread) and off the tiles, one column and several blocks of them
SIZES = [(33, 4), (100, 10), (161, 17), (300, 8), (520, 33), (1030, 1), (2060, 3)]
FORMS = {"fp32": 1, "tf32x3": 3, "bf16x3": 4}


def indicators(pmcim, form, n, l):
    """Indicator and ||P f|| of two disks right of the spectrum of (A0 + 0.2 A1 e^{-z/2}) - z I."""
    rng = np.random.default_rng(1000 * n + l)
    A = [(rng.random((n, n)) - 0.5 + 1j * (rng.random((n, n)) - 0.5)) * math.sqrt(6.0 / n) for _ in range(2)]
    V = np.asfortranarray(rng.random((n, l)) - 0.5 + 1j * (rng.random((n, l)) - 0.5))
    P = pmcim.Problem(n, [(-1.0 + 0j, w.MONOMIAL, 1, 0.0), (A[0], w.MONOMIAL, 0, 0.0), (0.2 * A[1], w.EXP_NEG, 0, 0.5)])
    ind, _, norm, _ = P.indicator([w.Region(2.5 + 0.25j, 0.5, 16), w.Region(2.25 - 0.5j, 0.375, 16)], V,
                                  opt=pmcim.options(precision=FORMS[form]))
    P.close()
    return np.concatenate([ind, norm])


@pytest.mark.parametrize("n,l", SIZES)
@pytest.mark.parametrize("form", sorted(FORMS))
def test_indicators_where_solutions_cancel(form, n, l):
    import torch
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    from paper_2312_13117_gb300 import build, pmcim
    build.build()
    with open(GOLDEN) as f:
        want = np.array(json.load(f)["%s_n%d_l%d" % (form, n, l)])
    got = indicators(pmcim, form, n, l)
    assert np.all(np.abs(got - want) <= 1e-9 * np.abs(want)), (got, want)

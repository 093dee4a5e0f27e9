"""A precision-form call on a device whose memory is nearly all taken by others.

Chunks then hold few nodes, and the FP64 matrices of nodes that are solved again (here all
of them: one sweep is never enough for a remaining error of 1e-15) no more than the same
share of the free memory. Solutions do not depend on the chunks.
"""
import numpy as np
import pytest

import workloads as w
from tests.test_gpu_parity import pm  # noqa: F401

pytestmark = pytest.mark.gpu


def test_re_solves_within_the_free_memory(pm):  # noqa: F811
    import torch
    n, l = 512, 8
    rng = np.random.default_rng(2)
    # nine dense terms: the digits of f_k X take as much beside a node's FP32 slot as the FP64 matrix
    # takes over it
    A = [w.complex_gaussian(rng, (n, n)) / 64.0 for _ in range(9)]
    V = w.probe_block(rng, n, l)
    terms = [(-1.0 + 0j, w.MONOMIAL, 1, 0.0)] + [(a, w.EXP_NEG, 0, 0.1 * k) for k, a in enumerate(A)]
    reg = [w.Region(0.3 - 0.1j, 0.2, 64), w.Region(-0.4 + 0.1j, 0.3, 64)]
    opt = pm.options(precision=pm.PREC_FP32_IR, max_ir_sweeps=1, tol_ir=1e-15)
    P = pm.Problem(n, terms)
    want = P.moments(reg, V, opt=opt)
    P.close()
    Q = pm.Problem(n, terms)
    Q.moments([w.Region(0.3 - 0.1j, 0.2, 2)], V, opt=opt)  # everything but the large workspaces
    torch.cuda.empty_cache()
    free, _ = torch.cuda.mem_get_info()
    held = torch.empty(free - (400 << 20), dtype=torch.uint8, device="cuda")
    try:
        got = Q.moments(reg, V, opt=opt)
    finally:
        del held
        torch.cuda.empty_cache()
    Q.close()
    for a, b in zip(got, want):
        assert np.array_equal(a, b)

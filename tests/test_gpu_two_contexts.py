"""Two contexts of different degree on one device: what a launch may ask for in shared memory is a
property of the kernel, so factoring a context of low degree must leave a context of high degree, that
was factored before it, all it needs, for launches that it has not made yet (another number of
right-hand sides, gradients) as well.  Results are compared with the same context's own, made before
the second one existed (1e-12 in FP64, 1e-5 in complex64: the bounds of one application elsewhere), or
judged by the residual of the solution (1e-10 where it was found to 1e-12 in the dual variables)."""
import numpy as np
import pytest
import torch

import workloads as W
from paper_1808_04713_gb300 import ddh

pytestmark = pytest.mark.gpu


def _solver(p, **opts):
    w = W.small_uniform(3, p, 9.0, seed=2, eps_range=(1.0, 1.3))
    s = ddh.DDH(0)
    s.set_mesh(w.base_n, w.leaves, w.p)
    s.set_coefficients(w.k, w.eps)
    s.factor(**opts)
    return s


@pytest.mark.parametrize("prec", [ddh.PREC_FP64, ddh.PREC_MIXED_FP32])
def test_smaller_context_leaves_the_larger_one_usable(prec):
    big = _solver(24, precision=prec, tol=1e-12)
    g = torch.Generator(device="cuda").manual_seed(1)
    v = torch.view_as_complex(torch.randn((8, big.info().n_dual, 2), generator=g, device="cuda", dtype=torch.float64))
    one = [big.apply_dual_operator(which, v[:1], prec) for which in (0, 1)]
    small = _solver(4)
    for which in (0, 1):                      # eight at once: a block size the large context has not launched
        y = big.apply_dual_operator(which, v, prec)
        err = ((y[:1] - one[which]).norm() / one[which].norm()).item()
        assert err <= (1e-12 if prec == ddh.PREC_FP64 else 1e-5), err
    b = big.rhs_planewave(np.linspace(0.0, 1.0, 4))
    u, _ = big.solve(b, tol=1e-12)
    assert max(big.primal_residual(b, u)) <= 1e-10
    assert bool(torch.isfinite(big.grad_eps(u, u)).all())
    small.close()
    big.close()

"""The fixed-point dense products of the FP64 operator (csrc/ddh_fixed.cuh) at the sizes where they
can go wrong: column tiles and lane chains of the dense K^-1, short and long rows of the fronts,
every right-hand-side block and its remainder, and vectors that hold an infinity or a NaN.

The dense K^-1 and the nested-dissection factor are two factorisations of one matrix that share no
product kernel, so each checks the other; both are within about cond(K) eps of the exact operator
(cond(K) < 1e4 on these meshes and eps = 2^-53: 1e-12, taken ten times larger for the two sides)."""
import numpy as np
import pytest
import torch

import workloads as W
from paper_1808_04713_gb300 import ddh

pytestmark = pytest.mark.gpu
TOL = 1e-11


def _solver(w, **opts):
    s = ddh.DDH(0)
    s.set_mesh(w.base_n, w.leaves, w.p)
    s.set_coefficients(w.k, w.eps)
    s.factor(**opts)
    return s


def _dual(n_dual, R, seed=3):
    g = torch.Generator(device="cuda").manual_seed(seed)
    x = torch.randn((R, n_dual, 2), generator=g, device="cuda", dtype=torch.float64)
    # right-hand sides of very different size in one block: each has its own scale
    return torch.view_as_complex(x) * 1e3 ** (torch.arange(R, device="cuda", dtype=torch.float64)[:, None] - R / 2)


# n_coarse = (n+1)^2 + 2 n (n+1) (l-1): 9 and 65 (fewer rows than a CTA), 924 and 1729 below and above the 1008
# columns of an eight-vector tile, 3801 above two of either kind
@pytest.mark.parametrize("n,l", [(2, 1), (4, 2), (13, 3), (18, 3), (20, 5)])
@pytest.mark.parametrize("R", [1, 2, 3, 5, 8, 9])
def test_dense_inverse_matches_nested_dissection(n, l, R):
    w = W.small_uniform(n, 8, 1.1 * n, seed=2, eps_range=(1.0, 1.3))
    a = _solver(w, coarse_form=ddh.COARSE_DENSE, l_override=l)
    b = _solver(w, coarse_form=ddh.COARSE_ND_LEVELS, l_override=l)
    v = _dual(a.info().n_dual, R)
    x, y = a.apply_dual_operator(0, v), b.apply_dual_operator(0, v)
    err = ((x - y).norm(dim=1) / y.norm(dim=1)).max().item()
    assert err <= TOL, err
    # a right-hand side's result does not depend on the block it is in
    assert torch.equal(a.apply_dual_operator(0, v[:1]), x[:1])
    assert torch.equal(b.apply_dual_operator(0, v[:1]), y[:1])
    a.close()
    b.close()


@pytest.mark.parametrize("form", [ddh.COARSE_DENSE, ddh.COARSE_ND_LEVELS])
@pytest.mark.parametrize("bad", [float("nan"), float("inf")])
def test_non_finite_values_stay_in_their_right_hand_side(form, bad):
    w = W.small_uniform(6, 8, 9.0, seed=2, eps_range=(1.0, 1.3))
    s = _solver(w, coarse_form=form)
    v = _dual(s.info().n_dual, 3)
    ref = s.apply_dual_operator(0, v)
    v2 = v.clone()
    v2[1, 5] = bad
    y = s.apply_dual_operator(0, v2)
    assert torch.equal(y[0], ref[0]) and torch.equal(y[2], ref[2])
    assert not bool(torch.isfinite(torch.view_as_real(y[1])).all())
    zero = s.apply_dual_operator(0, torch.zeros_like(v))
    assert not bool(zero.abs().any())
    s.close()

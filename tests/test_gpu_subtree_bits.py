"""The subtree launches of the coarse solve (ddh_info.coarse_subtrees > 0) sum a front's rows in another order than
the level launches do.  Where the tree is cut follows from the tree alone, so solves come out with the
same bits whatever the chains of right-hand sides, and a right-hand side with the same bits whatever is
solved beside it, for the complex128 factor and for its complex64 copy."""
import numpy as np
import pytest
import torch

import workloads as W
from paper_1808_04713_gb300 import ddh

pytestmark = pytest.mark.gpu


def _solver(n, l, subtrees, **opts):
    w = W.small_uniform(n, 8, 2.0 * n, seed=2, eps_range=(1.0, 1.3))
    s = ddh.DDH(0)
    s.set_mesh(w.base_n, w.leaves, w.p)
    s.set_coefficients(w.k, w.eps)
    s.factor(l_override=l, coarse_form=ddh.COARSE_ND_LEVELS, **opts)
    assert (s.info().coarse_subtrees > 0) == subtrees
    return s


# 16 subtrees, 64 (the cut at 16 has fronts of 199 entries), none
@pytest.mark.parametrize("n,l,subtrees", [(16, 5, True), (32, 5, True), (6, 3, False)])
@pytest.mark.parametrize("opts", [{"precision": ddh.PREC_FP64}, {"precision": ddh.PREC_MIXED_FP32},
                                  {"precision": ddh.PREC_MIXED_FP32, "coarse_fp32": 1}])
def test_chains_and_contexts_give_the_same_bits(n, l, subtrees, opts):
    outs = []
    for chains in (1, 2, 4, 4):
        s = _solver(n, l, subtrees, nd_chains=chains, **opts)
        u, st = s.solve(s.rhs_planewave(np.linspace(0.0, 2.0, 8)), tol=1e-10)
        outs.append((u.cpu(), [(x.iterations, x.inner_iterations) for x in st]))
        s.close()
    for u, its in outs[1:]:
        assert torch.equal(u, outs[0][0]) and its == outs[0][1]


@pytest.mark.parametrize("n,l", [(16, 5), (32, 5)])
def test_a_right_hand_side_does_not_depend_on_the_others(n, l):
    s = _solver(n, l, True)
    g = torch.Generator(device="cuda").manual_seed(1)
    v = torch.view_as_complex(torch.randn((9, s.info().n_dual, 2), generator=g, device="cuda", dtype=torch.float64))
    all9 = s.apply_dual_operator(0, v)
    for R in (1, 2, 3, 5, 8):
        assert torch.equal(s.apply_dual_operator(0, v[:R].contiguous()), all9[:R])
    s.close()

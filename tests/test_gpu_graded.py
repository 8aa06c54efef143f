"""FP64 products of graded data: entries of a row, or of a vector, that differ by many orders of magnitude keep
their own digits, as in a sum of FP64 products.

One application is compared, component by component, with the superposition of its columns (each the
application to a unit vector, where nothing is graded), summed exactly.  Preconditioner: the sums have
at most 4 p terms and are followed by two roundings, each within 2^-52 of the absolute products, taken
64 times larger.  Interface operator: its coarse matrix, scaled to unit diagonal, has a condition number
below 1e4 on these meshes, so its FP64 form is within about 1e4 2^-53 = 1e-12 of the absolute products,
taken ten times larger as in the comparison of the two coarse forms."""
import math

import numpy as np
import pytest
import torch

import workloads as W
from paper_1808_04713_gb300 import ddh

pytestmark = pytest.mark.gpu


def _two_regions(jump, **opts):
    """Poisson on 8 x 8 squares, p = 4, l = 2, the coefficient `jump` on the right half."""
    n = 8
    leaves = W.uniform_leaves(n)
    s = ddh.DDH(0)
    s.set_mesh(n, leaves, np.full(n * n, 4, np.int32))
    s.set_poisson(np.where(leaves[:, 1] >= n // 2, float(jump), 1.0))
    s.factor(l_override=2, **opts)
    return s


def _columns(s, which):
    n = s.info().n_dual
    eye = torch.eye(n, dtype=torch.complex128, device="cuda")
    return torch.cat([s.apply_dual_operator(which, eye[i:i + 16].contiguous()) for i in range(0, n, 16)]).cpu().numpy().T


def _check(s, which, v, tol):
    A = _columns(s, which)
    y = s.apply_dual_operator(which, torch.tensor(v, device="cuda")).cpu().numpy()
    for r in range(len(v)):
        t = A * v[r][None, :]
        ref = np.array([complex(math.fsum(row.real), math.fsum(row.imag)) for row in t])
        P = np.abs(t).sum(axis=1)
        assert (np.abs(y[r] - ref) <= tol * P).all(), np.max(np.abs(y[r] - ref) / P)


def _graded(rng, R, n, decades):
    v = rng.standard_normal((R, n)) + 1j * rng.standard_normal((R, n))
    return v * 10.0 ** rng.uniform(-decades, 0.0, (R, n))


@pytest.mark.parametrize("decades", [0, 6, 12, 30])
def test_preconditioner(decades):
    w = W.small_uniform(3, 8, 6.0, seed=2, eps_range=(1.0, 1.3))
    s = ddh.DDH(0)
    s.set_mesh(w.base_n, w.leaves, w.p)
    s.set_coefficients(w.k, w.eps)
    s.factor()
    rng = np.random.default_rng(decades)
    for R in (1, 2, 5, 8):
        _check(s, 1, _graded(rng, R, s.info().n_dual, decades), 64 * 2.0 ** -52)
    s.close()


@pytest.mark.parametrize("form", [ddh.COARSE_DENSE, ddh.COARSE_ND_LEVELS, ddh.COARSE_ND])
@pytest.mark.parametrize("jump", [1.0, 1e4, 1e8])
def test_operator_across_a_jump(form, jump):
    s = _two_regions(jump, coarse_form=form)
    rng = np.random.default_rng(7)
    for R in (1, 3, 8):
        _check(s, 0, _graded(rng, R, s.info().n_dual, 0), 1e-11)
    s.close()

"""The Poisson PCG stops where its residual does, whatever the context solved before: the work of a solve
(kernels launched, iterations, result) is the same after a solve that ran into its iteration limit, and
an iteration limit of one is one iteration."""
import numpy as np
import pytest
import torch

import workloads as W
from paper_1808_04713_gb300 import ddh

pytestmark = pytest.mark.gpu


def _solver(**opts):
    w = W.poisson_table2(3, 64, 2)
    s = ddh.DDH(0)
    s.set_mesh(w.base_n, w.leaves, w.p)
    s.set_poisson(w.rho)
    s.factor(l_override=2, **opts)
    return s


def _counted(s, b, tol):
    n = s.kernel_launches()
    u, st = s.solve(b, tol=tol, allow_noconv=True)
    return s.kernel_launches() - n, [x.iterations for x in st], u


@pytest.mark.parametrize("use_graph", [0, 1])
@pytest.mark.parametrize("R", [1, 3])
def test_work_does_not_depend_on_the_solve_before(R, use_graph):
    s = _solver(maxit=60, use_graph=use_graph)
    g = torch.Generator(device="cuda").manual_seed(2)
    b = torch.rand((R, s.n_local), generator=g, device="cuda", dtype=torch.float64).to(torch.complex128)
    _counted(s, b, 1e-8)
    n0, its, u = _counted(s, b, 1e-8)
    assert max(its) < 30
    assert _counted(s, b, 1e-200)[1] == [60] * R          # below any residual that 60 iterations reach
    n1, its1, u1 = _counted(s, b, 1e-8)
    assert (n1, its1) == (n0, its) and torch.equal(u, u1)
    nz = _counted(s, torch.zeros_like(b), 1e-8)
    assert nz[1] == [0] * R and nz[0] < n0 and not bool(nz[2].abs().any())
    s.close()


def test_one_iteration():
    s = _solver(maxit=1)
    b = torch.ones((1, s.n_local), device="cuda", dtype=torch.complex128)
    assert _counted(s, b, 1e-8)[1] == [1]
    assert np.isfinite(s.pcg_spectrum(0)).all()
    s.close()


def test_limit_equal_to_the_iterations_needed():
    s = _solver()
    b = torch.ones((1, s.n_local), device="cuda", dtype=torch.complex128)
    need = _counted(s, b, 1e-8)[1][0]
    s.close()
    s = _solver(maxit=need)
    assert s.solve(b, tol=1e-8)[1][0].iterations == need          # converged: no error raised
    s.close()
    s = _solver(maxit=need - 1)
    with pytest.raises(ddh.DDHError):
        s.solve(b, tol=1e-8)
    s.close()

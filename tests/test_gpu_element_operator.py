"""The element operator in FP64 (k_elem_matvec) at the degrees where its rows have other taps: p = 3 to 5
(rows 0 to 3 and the last two overlap), the largest, and mixed degrees in one launch.

The solves run on factors that the host forms from the matrix entries, so the residual of a solution
found to 1e-12 in the dual variables tests the operator itself; a solution's residual is within about
ten times that on these small meshes.  With twice the solution the residual is -b, relative norm 1."""
import pytest

import workloads as W
from paper_1808_04713_gb300 import ddh

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("p,k,p_range", [(3, 2.0, None), (4, 2.5, None), (5, 3.0, None), (21, 20.0, None),
                                         (32, 25.0, None), (6, 4.0, (4, 17))])
def test_residual_of_a_solution(p, k, p_range):
    w = W.small_uniform(3, p, k, seed=2, eps_range=(1, 2), p_range=p_range)
    s = ddh.DDH(0)
    s.set_mesh(w.base_n, w.leaves, w.p)
    s.set_coefficients(w.k, w.eps)
    s.factor(tol=1e-12)
    b = s.rhs_planewave(w.thetas)
    u, st = s.solve(b, tol=1e-12)
    assert max(s.primal_residual(b, u)) <= 1e-11
    assert max(abs(s.primal_residual(b, 2.0 * u) - 1.0)) <= 1e-11
    s.close()

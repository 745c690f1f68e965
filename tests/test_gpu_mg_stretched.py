"""The multigrid-preconditioned solve on cells longer than wide: from an aspect ratio of 1.91 on the
plain Jacobi factor omega / diagonal amplifies the errors that alternate across the short side, and
the smoother takes another.  Just below and above that ratio, and up to 4, either way; against the
oracle's direct solution (bound of the mixed-precision parity tests).  Iterations: the worst
remaining mode, smooth along the short side, loses 0.85 / 8 of itself per sweep at a ratio of 4, so
a cycle leaves 0.8 of it, a condition number of 5 and a CG factor of 0.38: thirty iterations to
1e-12, three times that allowed for the body, the edges and the restarts."""
import numpy as np
import pytest

from paper_2512_12232_gb300 import workloads as W
from tests.gpu_util import oracle_solution, rel_l2

pytestmark = pytest.mark.gpu

D, N = W.BC_DIRICHLET_UY, W.BC_NATURAL


@pytest.mark.parametrize("bc", [(D, D, D, D), (N, N, D, D)], ids=["dirichlet", "natural"])
@pytest.mark.parametrize("nx,ny", [(200, 190), (190, 201), (256, 256), (201, 403), (256, 64), (129, 257), (300, 38)])
def test_multigrid_on_stretched_cells(nx, ny, bc):
    from paper_2512_12232_gb300 import api
    c = W.Case(-4.0, 4.0, -2.0, 2.0, nx, ny, np.array([[0.13, 0.07, 0.6]]), 6, bc)
    ref = oracle_solution(c, 1.0)[3]
    with api.mesh_build(c.grid, c.bodies, c.sweeps, c.bc) as g:
        res = api.psi_solve(g, U=1.0, tol=1e-12, precision=api.PF_MIXED, preconditioner="mg", k_max=400,
                            raise_on_failure=False)
        assert res.info[0]["status"] == 0 and res.info[0]["rel_true_residual"] <= 1e-12
        assert res.info[0]["iters"] <= 90
        assert rel_l2(res.psi.cpu().numpy(), ref.ravel()) <= 1e-6

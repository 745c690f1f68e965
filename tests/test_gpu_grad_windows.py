"""dJ/dX and dJ/dc against the oracle where the shape-derivative and transposed-smoothing
kernels meet their edges: grids smaller than a tile, ragged last tiles, bodies and smoothing
windows that reach the grid's sides, numbers of sweeps that are no multiple of a launch's
four, rectangular cells.  Tolerance: that of the gradient's parity tests, 1e-8 of the largest
entry (solves to 1e-13, condition numbers up to 1e4)."""
import numpy as np
import pytest

from oracle import grad as OG, mesh as OM
from paper_2512_12232_gb300 import workloads as W

pytestmark = pytest.mark.gpu

BODIES = np.array([[-2.7, -0.62, 0.67], [2.8, 0.73, 0.61]])


@pytest.mark.parametrize("nx,ny,sweeps", [(41, 20, 3), (65, 29, 9), (63, 33, 20), (130, 37, 21), (64, 32, 4)])
def test_gradient_matches_oracle(nx, ny, sweeps):
    from paper_2512_12232_gb300 import api
    case = W.Case(-4.0, 4.0, -2.0, 2.0, nx, ny, BODIES, sweeps)
    m = OM.build_mesh(case.grid, case.bodies, case.sweeps, case.bc)
    J_ref, dX_ref, dc_ref, _ = OG.gradient(m, case.sweeps, 1.0, 0, 1, 0)
    with api.mesh_build(case.grid, case.bodies, case.sweeps, case.bc) as g:
        api.psi_solve(g, U=1.0, tol=1e-13, precision=api.PF_FP64)
        dX, dc, J = api.grad(g, 0, 0, 1, 1.0, 1e-13)
    assert abs(J[0] - J_ref) <= 1e-10 * max(1.0, abs(J_ref))
    assert np.abs(dX.cpu().numpy() - dX_ref).max() <= 1e-8 * np.abs(dX_ref).max()
    assert np.abs(dc - dc_ref).max() <= 1e-8 * np.abs(dc_ref).max()

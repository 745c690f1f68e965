"""The multigrid-preconditioned solve where an odd number of cells meets a natural side, at the
first level and at later ones: the coarse line there must not come to lie ever closer to its
neighbour.  Against the oracle's direct solution; bounds are those of test_gpu_mg_tiles."""
import numpy as np
import pytest

from paper_2512_12232_gb300 import workloads as W
from tests.gpu_util import oracle_solution, rel_l2

pytestmark = pytest.mark.gpu

D, N = W.BC_DIRICHLET_UY, W.BC_NATURAL


def _case(nx, ny, bc, r=0.4, box=(-4.0, 4.0, -2.0, 2.0)):
    return W.Case(*box, nx, ny, np.array([[0.13, 0.07, r]]), 6, bc)


CASES = {"outlet_257x129": [_case(257, 129, (N, N, D, D))], "outlet_257x128": [_case(257, 128, (N, N, D, D))],
         "outlet_129x65": [_case(129, 65, (D, N, D, D))], "top_256x129": [_case(256, 129, (D, D, D, N))],
         "two_sides_193x97": [_case(193, 97, (D, N, D, N))], "inlet_257x129": [_case(257, 129, (N, D, N, D))],
         "odd_at_every_level_511x255": [_case(511, 255, (D, N, N, D))], "one_block_33x17": [_case(33, 17, (N, N, D, D), 0.7)],
         "thin_33x3": [W.Case(-4.0, 4.0, -0.4, 0.4, 33, 3, np.zeros((0, 3)), 0, (D, N, D, N))],
         "batch": [_case(257, 129, (N, N, D, D)), _case(200, 101, (N, N, D, D)), _case(65, 33, (N, N, D, D), 0.5)]}


@pytest.mark.parametrize("name", list(CASES))
def test_multigrid_at_odd_natural_sides(name):
    from paper_2512_12232_gb300 import api
    cases = CASES[name]
    with api.batch_build(cases) as g:
        res = api.psi_solve(g, U=1.0, tol=1e-12, precision=api.PF_MIXED, preconditioner="mg", k_max=400,
                            raise_on_failure=False)
        psi = res.psi.cpu().numpy()
        for v, c in enumerate(cases):
            assert res.info[v]["status"] == 0 and res.info[v]["rel_true_residual"] <= 1e-12
            assert res.info[v]["iters"] <= 60
            ref = oracle_solution(c, 1.0)[3]
            assert rel_l2(psi[g.node_offsets[v]:g.node_offsets[v + 1]], ref.ravel()) <= 1e-6, v


def test_phi_with_an_odd_number_of_rows():
    """phi has natural conditions at the bottom and the top."""
    from paper_2512_12232_gb300 import api
    c = _case(256, 129, (D, D, D, D))
    with api.mesh_build(c.grid, c.bodies, c.sweeps, c.bc) as g:
        phi, info, _ = api.phi_solve(g, U=1.0, tol=1e-12, precision=api.PF_MIXED, preconditioner="mg", k_max=400,
                                     raise_on_failure=False)
        ref, _, _ = api.phi_solve(g, U=1.0, tol=1e-13, precision=api.PF_FP64)
    assert info[0]["status"] == 0 and info[0]["iters"] <= 60
    assert rel_l2(phi.cpu().numpy(), ref.cpu().numpy()) <= 1e-6


@pytest.mark.parametrize("nx,ny,bc", [(2000, 40, (D, N, N, N)), (600, 9, (D, N, N, N)), (40, 600, (N, N, D, N)), (300, 2, (D, N, N, N)),
                                      (3, 300, (N, N, N, D)), (129, 65, (N, D, N, N))])
def test_multigrid_on_thin_domains_between_natural_sides(nx, ny, bc):
    """Halved until one cell is left between two natural sides, that direction becomes one line; phi
    has natural conditions at the bottom and the top of the same grid (and of its transpose)."""
    from paper_2512_12232_gb300 import api
    h = 4.0 * ny / nx
    c = W.Case(-4.0, 4.0, -h, h, nx, ny, np.zeros((0, 3)), 0, bc)
    with api.mesh_build(c.grid, c.bodies, c.sweeps, c.bc) as g:
        res = api.psi_solve(g, U=1.0, tol=1e-10, precision=api.PF_MIXED, preconditioner="mg", k_max=400,
                            raise_on_failure=False)
        phi, info, _ = api.phi_solve(g, U=1.0, tol=1e-10, precision=api.PF_MIXED, preconditioner="mg", k_max=400,
                                     raise_on_failure=False)
    assert res.info[0]["status"] == 0 and res.info[0]["iters"] <= 60
    assert info[0]["status"] == 0 and info[0]["iters"] <= 60
    # without bodies both are linear: phi = U x, and psi = U y up to a constant per unfixed side
    x = np.tile(np.linspace(-4.0, 4.0, nx + 1), ny + 1)
    assert rel_l2(phi.cpu().numpy(), x) <= 1e-4          # tol 1e-10 and a condition number of up to 1e6


@pytest.mark.parametrize("nx,ny,asp", [(2000, 40, 2 / 3), (200, 160, 1.6), (256, 200, 25 / 16), (257, 129, 1.0)])
def test_phi_around_a_body(nx, ny, asp):
    """The natural condition on a body leaves rows of partial cells whose Jacobi factor is damped."""
    from paper_2512_12232_gb300 import api
    h = 4.0 * ny / nx / asp
    c = W.Case(-4.0, 4.0, -h, h, nx, ny, np.array([[0.1 * h, 0.07 * h, 0.35 * h]]), 4, (D, D, D, D))
    with api.mesh_build(c.grid, c.bodies, c.sweeps, c.bc) as g:
        phi, info, _ = api.phi_solve(g, U=1.0, tol=1e-10, precision=api.PF_MIXED, preconditioner="mg", k_max=300,
                                     raise_on_failure=False)
        ref, _, _ = api.phi_solve(g, U=1.0, tol=1e-12, precision=api.PF_FP64)
    assert info[0]["status"] == 0 and info[0]["iters"] <= 60
    assert rel_l2(phi.cpu().numpy(), ref.cpu().numpy()) <= 1e-4      # tol 1e-10 and a condition number of up to 1e6

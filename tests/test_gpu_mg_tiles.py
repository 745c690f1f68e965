"""The multigrid-preconditioned solve against the oracle's direct solution where its tile and
level kernels change path: grids of a few tiles with and without plain ones, even and odd
numbers of cells (odd last lines copy their coarse node), natural sides (FREE nodes on the
grid's edge), several variants.  Tolerance: that of the mixed-precision parity tests, 1e-6 in
relative L2 at a true residual of 1e-12 (condition numbers up to 1e5 leave 1e-7)."""
import numpy as np
import pytest

from paper_2512_12232_gb300 import workloads as W
from tests.gpu_util import oracle_solution, rel_l2

pytestmark = pytest.mark.gpu

D, N = W.BC_DIRICHLET_UY, W.BC_NATURAL


def _case(nx, ny, bc=(D, D, D, D), r=0.4):
    return W.Case(-4.0, 4.0, -2.0, 2.0, nx, ny, np.array([[0.13, 0.07, r]]), 6, bc)


CASES = {"one_tile": [_case(40, 20, r=0.7)], "no_plain_tile": [_case(130, 40)], "even": [_case(320, 160)],
         "odd": [_case(321, 161)], "natural": [_case(256, 129, (N, N, D, D))],
         "natural_odd_tile_edge": [_case(255, 127, (N, N, N, D))], "tile_multiple": [_case(384, 192)],
         "batch": [_case(200, 100), _case(333, 167), _case(96, 48)]}


@pytest.mark.parametrize("name", list(CASES))
def test_multigrid_solve_matches_oracle(name):
    from paper_2512_12232_gb300 import api
    cases = CASES[name]
    with api.batch_build(cases) as g:
        res = api.psi_solve(g, U=1.0, tol=1e-12, precision=api.PF_MIXED, preconditioner="mg", k_max=400)
        psi = res.psi.cpu().numpy()
        for v, c in enumerate(cases):
            assert res.info[v]["status"] == 0 and res.info[v]["rel_true_residual"] <= 1e-12
            assert res.info[v]["iters"] <= 60
            ref = oracle_solution(c, 1.0)[3]
            assert rel_l2(psi[g.node_offsets[v]:g.node_offsets[v + 1]], ref.ravel()) <= 1e-6, v

"""A solve after one that a bounded wait ended, on the same handle: the words that the blocks
exchanged before the wait gave up carry numbers that the next solve uses again, so none of them
may be left to be taken for its own.  Sums are taken in a fixed order, so the repeated solve has
the bits of a first one on a fresh handle; a stale sum (of another U) changes alpha at once."""
import numpy as np
import pytest

from paper_2512_12232_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", ["fp64", "mixed"])
@pytest.mark.parametrize("after", [0, 3])      # solves of the handle before the one that gives up
def test_solve_after_a_wait_that_gave_up(prec, after):
    from paper_2512_12232_gb300 import api
    from paper_2512_12232_gb300._lib import PF_ETIMEOUT
    p, tol = (api.PF_FP64, 1e-12) if prec == "fp64" else (api.PF_MIXED, 1e-8)
    c = W.five_cylinder_case(0.5, 256, 128, 20)
    with api.mesh_build(c.grid, c.bodies, c.sweeps, c.bc) as g:
        first = api.psi_solve(g, U=-0.5, tol=tol, precision=p)
    with api.mesh_build(c.grid, c.bodies, c.sweeps, c.bc) as g:
        for k in range(after):
            api.psi_solve(g, U=1.0 + k, tol=tol, precision=p)
        g.test_wait_timeout(True)
        assert api.psi_solve(g, U=1.0, tol=tol, precision=p, raise_on_failure=False).status == PF_ETIMEOUT
        g.test_wait_timeout(False)
        for _ in range(2):
            again = api.psi_solve(g, U=-0.5, tol=tol, precision=p)
            assert again.status == 0 and again.info[0]["iters"] == first.info[0]["iters"]
            assert np.array_equal(again.psi.cpu().numpy(), first.psi.cpu().numpy())
            assert np.array_equal(again.body_psi, first.body_psi)


def test_restarts_are_bounded_as_in_chunks():
    """A mixed solve whose tolerance cannot be met restarts until its launches are used up: as many
    as the streaming kernel's chunks of 256 iterations, k_max / 256 + 1000, and the last ones a
    launch is queued ahead."""
    from paper_2512_12232_gb300 import api
    D = W.BC_DIRICHLET_UY
    c = W.Case(-4.0, 4.0, -2.0, 2.0, 40, 20, np.array([[0.13, 0.07, 0.6]]), 8, (D, D, D, D))
    k_max = 300_000
    with api.mesh_build(c.grid, c.bodies, c.sweeps, c.bc) as g:
        res = api.psi_solve(g, U=1.0, tol=1e-30, precision=api.PF_MIXED, inner_tol=0.9999, k_max=k_max,
                            raise_on_failure=False)
    assert res.info[0]["status"] == 3 and res.info[0]["iters"] < k_max
    assert res.info[0]["refinements"] >= k_max // 256 + 1000 - 2

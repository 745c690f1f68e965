"""The streaming CG kernel (csrc/solver.cu, k_cg) at the sizes of the solve tests.  Batches whose
CG state fits the chip run another kernel, so the tests of ragged grids, natural sides, uneven
batches, fixed bodies, phi, iteration caps, tuned schedules and bounded waits are run here once
more, with every handle told to stream.  Cases and tolerances are those of the modules they
come from."""
import numpy as np
import pytest

from paper_2512_12232_gb300 import workloads as W
from tests.test_gpu_cutmesh import test_cut_solve_matches_oracle  # noqa: F401
from tests.test_gpu_failure import test_bounded_wait_gives_up_with_etimeout  # noqa: F401
from tests.test_gpu_grad import (test_batched_gradient_equals_single, test_gradient_matches_oracle,  # noqa: F401
                                 test_set_coords_solves_and_differentiates_at_the_given_coordinates)
from tests.test_gpu_invariants import test_solution_satisfies_the_discrete_equations  # noqa: F401
from tests.test_gpu_phi import test_phi_matches_oracle, test_phi_on_an_uneven_batch  # noqa: F401
from tests.test_gpu_resident import (test_resident_iteration_cap, test_resident_solve_matches_oracle,  # noqa: F401
                                     test_resident_solve_with_many_bodies)
from tests.test_gpu_resident_dots import test_small_products_count  # noqa: F401
from tests.test_gpu_shapes import test_kutta_solve_matches_oracle, test_uneven_batch_of_shapes  # noqa: F401
from tests.test_gpu_solve import (test_batched_solve_equals_single_solves, test_k_max_reports_not_converged,  # noqa: F401
                                  test_many_variant_batch, test_mixed_batch_reaches_tolerance_and_matches,
                                  test_paper_stopping_rule_matches_oracle_cg, test_schur_form_matches_oracle_and_mpc,
                                  test_schur_form_on_a_batch, test_solve_is_deterministic, test_solve_matches_oracle,
                                  test_tuned_schedule_matches_untuned)

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def api():
    from paper_2512_12232_gb300 import api
    return api


@pytest.fixture(autouse=True)
def streaming_handles(api, monkeypatch):
    build = api.Mesh.__init__

    def init(self, *args, **kw):
        build(self, *args, **kw)
        self.test_streaming(True)

    monkeypatch.setattr(api.Mesh, "__init__", init)


@pytest.mark.parametrize("prec", ["fp64", "mixed"])
def test_which_kernel_ran(api, prec):
    """A resident solve counts its iterations, a streaming one the launches of whole chunks of 256."""
    p = api.PF_FP64 if prec == "fp64" else api.PF_MIXED
    c = W.five_cylinder_case(0.5, 200, 100, 20)
    with api.mesh_build(c.grid, c.bodies, c.sweeps, c.bc) as g:
        for on in (True, False, True):
            g.test_streaming(on)
            res = api.psi_solve(g, U=1.0, tol=1e-8, precision=p)
            n, it = g.timing()["cg_launches"], res.info[0]["iters"]
            assert (n % 256 == 0 and n >= it) if on else n == it
            assert it % 256                     # (else the counts would not tell the kernels apart)
            assert res.info[0]["rel_true_residual"] <= 1e-8 and np.all(np.isfinite(res.body_psi))


def test_bounded_wait_of_the_streaming_kernel(api):
    """The wait that gives up is the one for a tile's copy, and a later solve on the handle is whole."""
    from paper_2512_12232_gb300 import _lib
    c = W.five_cylinder_case(0.5, 256, 128, 20)
    with api.mesh_build(c.grid, c.bodies, c.sweeps, c.bc) as g:
        first = api.psi_solve(g, U=1.0, tol=1e-8, precision=api.PF_MIXED)
        g.test_wait_timeout(True)
        with pytest.raises(_lib.PfError, match="TMA tile"):
            api.psi_solve(g, U=2.0, tol=1e-8, precision=api.PF_MIXED, chunk=4)
        g.test_wait_timeout(False)
        again = api.psi_solve(g, U=1.0, tol=1e-8, precision=api.PF_MIXED)
        assert np.array_equal(again.psi.cpu().numpy(), first.psi.cpu().numpy())

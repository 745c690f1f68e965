"""The CG with its state on the chip (csrc/resident.cu) against the oracle's direct solves, at
the sizes where its block cut can go wrong: grids of a few nodes, one block, blocks with a
ragged last row and column, half strips of two rows, wide and tall grids, bodies that share a
thread's strip, natural sides (rows without all four cells), batches that queue, and a solve
cut into many launches.  Tolerances are those of the GPU parity tests: at a true residual tol
the error of psi is tol times a condition number of up to 1e5 on these grids, so 1e-10 in
relative L2 for FP64 at 1e-15 x 1e5; 1e-6 in mixed precision at 1e-12."""
import functools

import numpy as np
import pytest

from oracle import mesh as OM, solve as OS, system as OSY
from paper_2512_12232_gb300 import workloads as W
from tests.gpu_util import rel_l2

pytestmark = pytest.mark.gpu

D, N = W.BC_DIRICHLET_UY, W.BC_NATURAL


def _case(nx, ny, bodies, sweeps=8, bc=(D, D, D, D), box=(-4.0, 4.0, -2.0, 2.0)):
    return W.Case(*box, nx, ny, np.asarray(bodies, dtype=np.float64).reshape(-1, 3), sweeps, bc)


ONE = [[0.13, 0.07, 0.6]]
CASES = {
    "3x3_nodes": [_case(2, 2, [])],
    "one_column_of_cells": [_case(33, 2, [])],
    "one_block": [_case(40, 20, ONE)],
    "ragged": [_case(101, 67, ONE)],
    "wide": [_case(603, 37, [[0.13, 0.07, 0.9]])],
    "tall": [_case(31, 301, ONE, box=(-2.0, 2.0, -4.0, 4.0))],
    "natural": [_case(150, 75, ONE, bc=(N, N, D, D))],
    "natural_three_sides": [_case(90, 45, ONE, bc=(D, N, N, N))],
    "close_bodies": [_case(160, 80, [[-0.9, -0.62, 0.5], [-0.87, 0.55, 0.5], [0.6, 0.1, 0.4], [1.9, 0.0, 0.3]])],
    "uneven_batch": [_case(64, 32, ONE), _case(200, 33, ONE), _case(48, 96, ONE, box=(-2.0, 2.0, -4.0, 4.0)),
                     _case(97, 49, [])],
    "queue": [_case(320 + 2 * k, 160 + k, [[0.13 + 0.001 * k, 0.07, 0.6]], 40) for k in range(20)],
}


@functools.lru_cache(maxsize=64)
def _reference(name, v):
    c = CASES[name][v]
    m = OM.build_mesh(c.grid, c.bodies, c.sweeps, c.bc)
    s = OSY.assemble(m, 1.0)
    u, psi = OS.solve_direct(s)
    return psi, u[s.n_free:]


@pytest.fixture(scope="module")
def api():
    from paper_2512_12232_gb300 import api
    return api


@pytest.mark.parametrize("prec,tol,bound", [("fp64", 1e-13, 1e-10), ("mixed", 1e-12, 1e-6)])
@pytest.mark.parametrize("name", list(CASES))
def test_resident_solve_matches_oracle(api, name, prec, tol, bound):
    cases = CASES[name]
    p = api.PF_FP64 if prec == "fp64" else api.PF_MIXED
    with api.batch_build(cases) as g:
        for chunk in (0, 7):               # 7: every launch pauses and the next one goes on
            if chunk and name in ("queue", "wide"):
                continue
            res = api.psi_solve(g, U=1.0, tol=tol, precision=p, chunk=chunk)
            psi = res.psi.cpu().numpy()
            for v in range(len(cases)):
                if name == "queue" and v % 7:
                    continue
                ref, C = _reference(name, v)
                assert res.info[v]["status"] == 0 and res.info[v]["rel_true_residual"] <= tol
                assert rel_l2(psi[g.node_offsets[v]:g.node_offsets[v + 1]], ref) <= bound, (name, v, chunk)
                k = g.body_offsets[v]
                np.testing.assert_allclose(res.body_psi[k:k + len(C)], C, rtol=0, atol=10 * bound)
        again = api.psi_solve(g, U=1.0, tol=tol, precision=p, chunk=chunk if name not in ("queue", "wide") else 0)
    assert np.array_equal(again.psi.cpu().numpy(), psi)   # sums are taken in a fixed order


def test_resident_iteration_cap(api):
    """k_max ends a solve inside a launch with the capped status and a finite iterate."""
    c = CASES["ragged"][0]
    with api.mesh_build(c.grid, c.bodies, c.sweeps, c.bc) as g:
        res = api.psi_solve(g, U=1.0, tol=1e-12, precision=api.PF_MIXED, k_max=11, raise_on_failure=False)
        assert res.info[0]["iters"] == 11 and res.info[0]["status"] == 3   # PF_ENOT_CONVERGED
        assert np.all(np.isfinite(res.psi.cpu().numpy()))


@pytest.mark.parametrize("rows,cols", [(4, 4), (5, 7)])
def test_resident_solve_with_many_bodies(api, rows, cols):
    """The first block sums sixteen bodies' rows at a time: as many, and three rounds of them,
    with bodies in one block and across several."""
    bodies = [[-3.4 + 6.8 * i / (cols - 1) + 0.011, -1.5 + 3.0 * j / (rows - 1) + 0.007, 0.23]
              for j in range(rows) for i in range(cols)]
    c = _case(201, 101, bodies)
    m = OM.build_mesh(c.grid, c.bodies, c.sweeps, c.bc)
    s = OSY.assemble(m, 1.0)
    u, psi = OS.solve_direct(s)
    with api.mesh_build(c.grid, c.bodies, c.sweeps, c.bc) as g:
        for p, tol, bound in ((api.PF_FP64, 1e-13, 1e-10), (api.PF_MIXED, 1e-12, 1e-6)):
            res = api.psi_solve(g, U=1.0, tol=tol, precision=p)
            assert rel_l2(res.psi.cpu().numpy(), psi) <= bound
            np.testing.assert_allclose(res.body_psi, u[s.n_free:], rtol=0, atol=10 * bound)


def test_resident_blocks_join_short_plain_runs(api):
    """Sixteen variants whose rows of undisplaced cells above and below the body are too few for
    blocks of their own: they join the neighbouring blocks, and the batch fits at once."""
    cases = [_case(256, 128, [[0.13 + 0.004 * k, 0.07 - 0.01 * k, 0.25]], 40) for k in range(16)]
    with api.batch_build(cases) as g:
        for p, tol, bound in ((api.PF_FP64, 1e-13, 1e-10), (api.PF_MIXED, 1e-12, 1e-6)):
            res = api.psi_solve(g, U=1.0, tol=tol, precision=p)
            psi = res.psi.cpu().numpy()
            for v in (0, 7, 15):
                c = cases[v]
                m = OM.build_mesh(c.grid, c.bodies, c.sweeps, c.bc)
                _, ref = OS.solve_direct(OSY.assemble(m, 1.0))
                assert rel_l2(psi[g.node_offsets[v]:g.node_offsets[v + 1]], ref) <= bound, v


def test_solve_without_room_for_the_exchange_buffers(api):
    """Each allocation of a handle's first solve is refused in turn.  Where it was one of the eight
    of the exchange between blocks, the streaming kernel solves; the others end in PF_ENOMEM."""
    import torch
    from paper_2512_12232_gb300 import _lib
    lib = _lib.load()
    made, refused = [0], [-1]

    @_lib.ALLOC_FN
    def alloc(nbytes, stream, ctx):
        made[0] += 1
        if made[0] - 1 == refused[0]:
            return None
        return torch.cuda.caching_allocator_alloc(int(nbytes), torch.cuda.current_device(), int(stream or 0))

    @_lib.FREE_FN
    def free(ptr, stream, ctx):
        torch.cuda.caching_allocator_delete(int(ptr))

    c = CASES["ragged"][0]
    ref, _ = _reference("ragged", 0)
    streamed = 0
    assert lib.pf_set_allocator(alloc, free, None) == _lib.PF_OK
    try:
        with api.mesh_build(c.grid, c.bodies, c.sweeps, c.bc) as g:
            built = made[0]
            res = api.psi_solve(g, U=1.0, tol=1e-13, precision=api.PF_FP64)
            total = made[0]
            assert g.timing()["cg_launches"] == res.info[0]["iters"]
        for k in range(built, total):
            made[0], refused[0] = 0, k
            with api.mesh_build(c.grid, c.bodies, c.sweeps, c.bc) as g:
                try:
                    res = api.psi_solve(g, U=1.0, tol=1e-13, precision=api.PF_FP64)
                except _lib.PfError as e:
                    assert "PF_ENOMEM" in str(e)
                    continue
                assert rel_l2(res.psi.cpu().numpy(), ref) <= 1e-10
                # (the streaming kernel runs whole chunks of launches, more than there are iterations)
                streamed += g.timing()["cg_launches"] > res.info[0]["iters"]
    finally:
        lib.pf_set_allocator(_lib.ALLOC_FN(), _lib.FREE_FN(), None)
    assert streamed == 8

"""pf_apply straight on the caller's vectors against the same call in place (which goes through
the padded vectors and k_apply), on grids of a few nodes, with ragged tiles, natural sides,
displaced cells and several variants.  FP32 rows are formed by the same functions: bit for
bit.  FP64 rows of plain tiles sum in another order: each row adds at most 24 products
k (p_m - p_n), each rounded a few times, so they agree to 64 eps max|k| max|p|."""
import ctypes as C

import numpy as np
import pytest
import torch

from paper_2512_12232_gb300 import workloads as W

pytestmark = pytest.mark.gpu

D, N = W.BC_DIRICHLET_UY, W.BC_NATURAL


def _case(nx, ny, bodies, bc=(D, D, D, D)):
    return W.Case(-4.0, 4.0, -2.0, 2.0, nx, ny, np.asarray(bodies, dtype=np.float64).reshape(-1, 3), 8, bc)


ONE = [[0.13, 0.07, 0.6]]
CASES = {"3x3_nodes": [_case(2, 2, [])], "one_tile": [_case(63, 15, [])], "tile_plus_one": [_case(64, 16, [])],
         "ragged": [_case(150, 75, ONE, (N, N, D, D))], "wide": [_case(701, 350, ONE)],
         "batch": [_case(131, 67, ONE), _case(64, 33, ONE), _case(300, 151, ONE)]}


@pytest.mark.parametrize("prec", ["fp64", "mixed"])
@pytest.mark.parametrize("name", list(CASES))
def test_direct_apply_matches_the_padded_path(name, prec):
    from paper_2512_12232_gb300 import _lib as L, api
    p = api.PF_FP64 if prec == "fp64" else api.PF_MIXED
    with api.batch_build(CASES[name]) as g:
        x = torch.from_numpy(W.random_vector(int(g.node_offsets[-1]), 5)).cuda()
        y, sums = api.apply(g, x, p)
        z = x.clone()
        nb = g.body_offsets[-1]
        ref = (C.c_double * max(1, nb))()
        L.check(L.load().pf_apply(g.handle, p, C.c_void_p(z.data_ptr()), C.c_void_p(z.data_ptr()), ref,
                                  C.c_void_p(torch.cuda.current_stream().cuda_stream)))
        if prec == "mixed":
            assert torch.equal(y, z) and np.array_equal(sums, np.array(ref[:nb]))
        else:
            tol = 64 * 2.3e-16 * 4.0 * x.abs().max().item()      # |k| <= 4 on these cells
            assert (y - z).abs().max().item() <= tol
            np.testing.assert_allclose(sums, np.array(ref[:nb]), rtol=0, atol=tol * 400)   # up to 400 nodes a body

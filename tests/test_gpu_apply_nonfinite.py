"""pf_apply with infinities and NaN among its values: straight on the caller's vectors as in
place (which goes through the padded vectors and k_apply), the same rows are infinite, of the
same sign, and the same ones NaN.  Plain tiles, displaced cells, tile edges and ragged tiles; the
values lie apart, next to each other, and at every place of a tile's rows and columns."""
import ctypes as C

import numpy as np
import pytest
import torch

from paper_2512_12232_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", ["fp64", "mixed"])
@pytest.mark.parametrize("box", [(-4.0, 4.0, -2.0, 2.0), (-4.0, 4.0, -0.7, 0.7), (-1.2, 1.2, -2.0, 2.0)])
def test_nonfinite_rows_match_the_padded_path(prec, box):
    from paper_2512_12232_gb300 import _lib as L, api
    p = api.PF_FP64 if prec == "fp64" else api.PF_MIXED
    D = W.BC_DIRICHLET_UY
    c = W.Case(*box, 333, 170, np.array([[0.13, 0.07, 0.4]]), 8, (D, D, D, D))
    with api.mesh_build(c.grid, c.bodies, c.sweeps, c.bc) as g:
        n = int(g.node_offsets[-1])
        x = W.random_vector(n, 7)
        rng = np.random.default_rng(11)
        at = rng.choice(n, n // 60, replace=False)
        x[at] = rng.choice([np.inf, -np.inf, np.nan], len(at))
        x = torch.from_numpy(x).cuda()
        y, _ = api.apply(g, x, p)
        z = x.clone()
        L.check(L.load().pf_apply(g.handle, p, C.c_void_p(z.data_ptr()), C.c_void_p(z.data_ptr()), None,
                                  C.c_void_p(torch.cuda.current_stream().cuda_stream)))
    y, z = y.cpu().numpy(), z.cpu().numpy()
    assert np.isinf(z).any() and np.isnan(z).any()
    assert np.array_equal(np.isnan(y), np.isnan(z))
    assert np.array_equal(np.where(np.isinf(y), y, 0.0), np.where(np.isinf(z), z, 0.0))

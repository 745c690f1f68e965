"""Bits of the FP32 mode's dot products, seen through a solve at a small U.  With U a power of
two every value of the iteration scales exactly, so psi / U is that of U = 1 bit for bit as long
as no product leaves FP32's range (2^-50).  At 2^-66 the products r r are about 2^-142, and only a
sum that keeps every product to FP32's last subnormal bit stays near: each is then off by at
most 2^-150, 2^-8 of itself with random signs, over 4700 nodes 6e-5 of the sum.  Twelve
iterations restated on the CPU: 9.7e-5 in psi with exact products and two-float sums, 2.6e-3 where
the sums are taken on a grid of 2^-143; the bound is their geometric mean."""
import numpy as np
import pytest

from paper_2512_12232_gb300 import workloads as W
from tests.gpu_util import rel_l2

pytestmark = pytest.mark.gpu


def test_small_products_count():
    from paper_2512_12232_gb300 import api
    D = W.BC_DIRICHLET_UY
    c = W.Case(-4.0, 4.0, -2.0, 2.0, 97, 49, np.array([[0.13, 0.07, 0.6]]), 8, (D, D, D, D))
    with api.mesh_build(c.grid, c.bodies, c.sweeps, c.bc) as g:
        psi = []
        for k in (0, 50, 66):
            res = api.psi_solve(g, U=2.0 ** -k, tol=1e-12, precision=api.PF_MIXED, k_max=12, raise_on_failure=False)
            assert res.info[0]["iters"] == 12
            psi.append(res.psi.cpu().numpy() * 2.0 ** k)
    assert np.array_equal(psi[1], psi[0])
    assert rel_l2(psi[2], psi[0]) <= 5e-4

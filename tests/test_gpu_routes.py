"""Which CG kernel a batch takes, where the choice is one of speed: few large FP64 grids that would
run one after the other stream, many small ones and FP32 ones queue on the chip, and so do not
launches of a few iterations, which would carry the state in and out each time.  Either way the
answer is the oracle's (test_gpu_resident, test_gpu_streaming); here both kernels agree to the
solve's tolerance."""
import numpy as np
import pytest

from paper_2512_12232_gb300 import workloads as W
from tests.gpu_util import rel_l2

pytestmark = pytest.mark.gpu

D = W.BC_DIRICHLET_UY


def _case(nx, ny, sweeps=30):
    return W.Case(-4.0, 4.0, -4.0 * ny / nx, 4.0 * ny / nx, nx, ny, np.array([[0.13, 0.07, 0.6]]), sweeps, (D, D, D, D))


@pytest.mark.parametrize("prec,cases,chunk,resident", [
    ("fp64", [_case(842, 411)] * 2, 0, False),
    ("fp64", [_case(453, 234)] * 7, 0, False),
    ("fp64", [_case(155, 66)] * 63, 0, True),
    ("mixed", [_case(1371, 795)] * 2, 0, True),
    ("mixed", [_case(1371, 795)] * 2, 8, False),
    ("mixed", [_case(256, 128)], 1, False),
    ("mixed", [_case(256, 128)], 6, True),
    ("fp64", [_case(256, 128)], 5, False),
    ("fp64", [_case(256, 128)], 16, True),
], ids=["fp64_two_large", "fp64_seven", "fp64_many_small", "fp32_two_large", "fp32_queue_chunk_8", "chunk_1", "chunk_6",
        "fp64_chunk_5", "fp64_chunk_16"])
def test_route(prec, cases, chunk, resident):
    from paper_2512_12232_gb300 import api
    p, state = (api.PF_FP64, 32) if prec == "fp64" else (api.PF_MIXED, 16)
    with api.batch_build(cases) as g:
        free = sum(g.stats(v)["n_free"] for v in range(len(cases)))
        psi = []
        for on in (False, True):
            g.test_streaming(on)
            res = api.psi_solve(g, U=1.0, tol=1e-10, precision=p, chunk=chunk)
            t = g.timing()
            bytes_a_node = t["cg_bytes_per_launch"] * t["cg_launches"] / (free * res.info[0]["iters"])
            assert (bytes_a_node < state) == (resident and not on)      # (streaming: 2 x state a node and iteration)
            psi.append(res.psi.cpu().numpy())
    assert rel_l2(psi[0], psi[1]) <= 1e-5            # tol 1e-10 and a condition number of up to 1e5, both sides

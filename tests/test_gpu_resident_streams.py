"""Handles that solve at the same time, each from a thread and on a stream of its own, on the
resident CG kernel: batches that leave room for each other on the chip and batches that fill it.
A launch's blocks wait for each other only, and it is cooperative: all of them are placed or none.
Sums are taken in a fixed order, so every solve has the bits of the same solve run alone."""
import threading

import numpy as np
import pytest
import torch

from paper_2512_12232_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx,variants", [(128, 1), (400, 5)])
def test_two_handles_solve_at_the_same_time(nx, variants):
    from paper_2512_12232_gb300 import api
    cases = [W.five_cylinder_case(0.25 + 0.1 * k, nx, nx // 2, 20) for k in range(variants)]
    handles = [api.batch_build(cases) for _ in range(2)]
    try:
        alone = {p: api.psi_solve(handles[0], U=1.0, tol=1e-8, precision=p).psi.cpu().numpy()
                 for p in (api.PF_MIXED, api.PF_FP64)}
        torch.cuda.synchronize()
        wrong = []

        def work(k):
            try:
                with torch.cuda.stream(torch.cuda.Stream()):
                    for n in range(6):
                        p = api.PF_FP64 if (n + k) % 2 else api.PF_MIXED
                        r = api.psi_solve(handles[k], U=1.0, tol=1e-8, precision=p)
                        if not np.array_equal(r.psi.cpu().numpy(), alone[p]):
                            wrong.append((k, n))
            except Exception as e:                       # noqa: BLE001 (reported by the test's thread)
                wrong.append((k, repr(e)))

        threads = [threading.Thread(target=work, args=(k,)) for k in range(2)]
        for t in threads:
            t.start()
        for t in threads:
            t.join()
        assert not wrong, wrong
    finally:
        for g in handles:
            g.close()

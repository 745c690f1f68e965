"""What a solve reports of its CG kernel: the bytes of a batch whose state stays on the chip are the
state's way in and out once per inner solve, and bench.py names the kernel that ran."""
import json
import os
import subprocess
import sys

import pytest

from paper_2512_12232_gb300 import workloads as W

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.mark.parametrize("prec,state", [("fp64", 32), ("mixed", 16)])
def test_bytes_follow_the_kernel(prec, state):
    from paper_2512_12232_gb300 import api
    p = api.PF_FP64 if prec == "fp64" else api.PF_MIXED
    c = W.five_cylinder_case(0.5, 200, 100, 20)
    with api.mesh_build(c.grid, c.bodies, c.sweeps, c.bc) as g:
        st = g.stats(0)
        for on in (False, True):
            g.test_streaming(on)
            res = api.psi_solve(g, U=1.0, tol=1e-8, precision=p)
            t, i = g.timing(), res.info[0]
            total = t["cg_bytes_per_launch"] * t["cg_launches"]
            if on:                               # x, r, p, q read and written by every iteration
                assert total >= 2 * state * st["n_free"] * i["iters"]
            else:
                once = 2 * state * st["n_free"] + st["n_nodes"] + 48 * st["n_general_cells"]
                assert 2 * state * st["n_free"] * i["refinements"] <= total <= once * i["refinements"] * (1 + 1e-12)


def test_bench_names_the_kernel_that_ran():
    env = {k: v for k, v in os.environ.items() if k not in ("RANK", "WORLD_SIZE", "LOCAL_RANK")}
    r = subprocess.run([sys.executable, "bench.py", "--config", "c1", "--steps", "1", "--warmup", "3", "--no-e2e",
                        "--no-fp64", "--no-mg", "--no-parity", "--no-cpu-baseline"], cwd=ROOT, env=env,
                       capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stderr[-3000:]
    rf = json.loads([ln for ln in r.stdout.splitlines() if ln.startswith("{")][0])["roofline"]
    assert rf["kernel"].startswith("k_cg_resident<float>") and rf["traffic"] is None
    assert rf["frac"] < 0.05

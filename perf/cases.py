"""Performance cases of the stream-function solver: the calls its users make, with inputs drawn
from a seed, the least work of each call, and the results in 64-bit arithmetic.

A case is a dict of plain values:
  kind       solve  psi_solve on a mesh that is built already (and CoPFI / the velocity field)
             study  mesh build + psi_solve + CoPFI, the handle released again: one pass of a
                    parametric study, every variant's geometry new
             grad   psi_solve + adjoint shape gradient on a mesh that is built already
             design objective(centres) and its backward pass through torch.autograd: one step
                    of a shape optimisation (mesh, solve, adjoint, chain rule to the centres)
             apply  the matrix-free operator alone on a nodal vector of the caller's
  layout     cylinder  one cylinder in [-10,10]x[-5,5]
             five      five jittered cylinders in [-20,20]x[-10,10], one grid size
             sweep     the same on grids of uneven sizes, 256x128 to nx x nx/2
             channel   three cylinders on the axis of a channel and a transverse pair,
                       natural inlet and outlet
             airfoil   a Joukowski airfoil at incidence with the Kutta condition
  nx, variants, sweeps, precision (mixed / fp64), precond (none / mg), tol.

Solves run to a relative true residual of 1e-13 (the tests' for psi itself; the gradient cases
take 1e-12, the default of the adjoint and autograd functions): psi is then settled in its
first nine digits, where at 1e-8 it still moves in the seventh with the place where the
iteration stops.  Iteration counts grow with the tolerance's logarithm; the kernels and their
shares are the same.
"""
from __future__ import annotations

import functools
import math

import numpy as np
import torch

from paper_2512_12232_gb300 import api, autograd
from paper_2512_12232_gb300 import workloads as W


def _tol(kind):
    return 1e-12 if kind in ("grad", "design") else 1e-13


def listed():
    def c(name, kind, layout, nx, variants, sweeps, precision="mixed", precond="none"):
        return {"name": name, "kind": kind, "layout": layout, "nx": nx, "variants": variants, "sweeps": sweeps,
                "precision": precision, "precond": precond, "tol": _tol(kind)}
    return [
        # the validation problem: one cylinder on 128x64 cells in FP64, the smallest solve;
        # a few hundred iterations of almost nothing but latency
        c("cylinder_fp64_128", "solve", "cylinder", 128, 1, 50, "fp64"),
        # one step of a shape optimisation over five cylinder centres through torch.autograd
        c("design_step_256", "design", "five", 256, 1, 64),
        # the gap-ratio table of the paper's channel: five gap ratios in one batch on a
        # ragged 403x201 grid, body values, CoPFI and one velocity field
        c("channel_403", "solve", "channel", 403, 5, 60),
        # an airfoil polar: eight incidences, Kutta condition, so the Schur form of the solve
        c("airfoil_polar_256", "solve", "airfoil", 256, 8, 64),
        # a single five-cylinder solve in plain FP64
        c("five_fp64_1024", "solve", "five", 1024, 1, 200, "fp64"),
        # the five-cylinder study on its own grid, 2048x1024, five gaps in one batch
        c("five_mixed_2048", "solve", "five", 2048, 5, 200),
        # the parametric sweep: 256 jittered layouts on uneven grids, the paper's CG
        c("sweep_mixed_256", "solve", "sweep", 1024, 256, 200),
        # the same sweep as a user runs it when only speed counts: meshes from scratch and
        # the multigrid-preconditioned solve
        c("sweep_study_mg_256", "study", "sweep", 1024, 256, 200, precond="mg"),
        # one very fine grid, 8192x4096, multigrid-preconditioned
        c("fine_mg_8192", "solve", "five", 8192, 1, 200, precond="mg"),
        # the differentiation study: 64 layouts, CoPFI and its gradient with respect to all
        # node coordinates and centres (forward and adjoint solve, shape derivative)
        c("gradient_mg_64", "grad", "five", 1024, 64, 200, precond="mg"),
        # the operator alone, FP32 arithmetic, on the finest grid (a caller's own Krylov
        # method) ...
        c("apply_mixed_8192", "apply", "five", 8192, 1, 200),
        # ... and in FP64 on a small ragged one, where the call itself is most of the time
        c("apply_fp64_403", "apply", "channel", 403, 1, 60, "fp64"),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["solve", "solve", "solve", "study", "grad", "design", "apply", "apply"])
    precision, precond = "mixed", rng.choice(["none", "mg"])
    layout = "five"
    variants = 1
    if kind == "solve":
        layout = rng.choice(["cylinder", "five", "sweep", "channel", "airfoil"])
        if layout in ("cylinder", "five") and rng.random() < 0.3:
            precision, precond = "fp64", "none"
        if layout == "airfoil":
            nx, variants = _log_int(rng, 128, 512), rng.randint(1, 12)
        elif layout == "channel":
            nx, variants = _log_int(rng, 301, 1001), rng.randint(1, 6)
        elif layout == "sweep":
            nx, variants = rng.randrange(320, 1025, 32), _log_int(rng, 4, 192)
        elif precision == "fp64":
            nx = _log_int(rng, 96, 1024)
        elif precond == "mg":
            nx, variants = _log_int(rng, 96, 6000), rng.randint(1, 4)
        else:
            nx, variants = _log_int(rng, 96, 2600), rng.randint(1, 4)
    elif kind == "study":
        layout, nx, variants = "sweep", rng.randrange(320, 1025, 32), _log_int(rng, 2, 192)
    elif kind == "grad":
        nx, variants = _log_int(rng, 256, 1200), _log_int(rng, 1, 24)
    elif kind == "design":
        nx, precond = _log_int(rng, 256, 900), "none"
    else:
        precond, precision = "none", rng.choice(["mixed", "fp64"])
        layout = rng.choice(["cylinder", "five", "channel"])
        nx, variants = _log_int(rng, 128, 6000), rng.randint(1, 3)
        if layout == "channel":
            nx = max(nx, 301)
    nx = max(nx, {"five": 256, "cylinder": 120}.get(layout, 0))   # coarser grids do not resolve the bodies
    sweeps = rng.choice([50, 60, 64, 100, 200])
    return {"kind": kind, "layout": layout, "nx": nx, "variants": variants, "sweeps": sweeps, "precision": precision,
            "precond": precond, "tol": _tol(kind)}


# ------------------------------------------------------------------ inputs


TRIES = 20


def _geometry(case, seed, attempt):
    """(workload cases, polygon lists or None) of a case, from the seed.  A draw whose mesh
    folds (a body grazing a grid node) is drawn again: `attempt` counts."""
    rng = np.random.default_rng([seed % (1 << 31), attempt, 17])
    nx, n, sweeps = case["nx"], case["variants"], case["sweeps"]
    if case["layout"] == "cylinder":
        out = []
        for _ in range(n):
            k = W.single_cylinder(nx, nx // 2, sweeps)
            k.bodies = k.bodies + np.array([[*rng.normal(0.0, 0.05, 2), 0.0]])
            out.append(k)
        return out, None
    if case["layout"] == "channel":
        return [W.paper_channel_case(float(d), nx, nx // 2, sweeps) for d in rng.uniform(0.3, 0.7, n)], None
    if case["layout"] == "airfoil":
        pairs = [W.airfoil_case(nx, float(a), sweeps) for a in rng.uniform(0.0, 10.0, n)]
        return [p[0] for p in pairs], [p[1] for p in pairs]
    sizes = [nx] * n
    if case["layout"] == "sweep":         # the grids belong to the case, the layouts to the seed
        sizes = np.random.default_rng(n).choice(np.arange(256, nx + 1, 32), n).tolist()
    return [W.parametric_sweep(1, seed=int(rng.integers(1 << 31)), nx_choices=(m,), sweeps=sweeps)[0]
            for m in sizes], None


def _precision(case):
    return api.PF_FP64 if case["precision"] == "fp64" else api.PF_MIXED


@functools.cache
def _allocator():
    """Device memory through PyTorch's caching allocator, set once, as a PyTorch program does."""
    api.use_torch_allocator()


def prepare(case, seed):
    _allocator()
    for attempt in range(TRIES):
        geo, polygons = _geometry(case, seed, attempt)
        mesh = api.batch_build(geo, polygons=polygons)
        if mesh.valid:
            break
        mesh.close()
    state = {"case": case, "geo": geo, "polygons": polygons}
    if case["kind"] in ("solve", "grad", "apply"):
        state["mesh"] = mesh
    else:
        mesh.close()                      # these build their own in every pass
    if case["kind"] == "apply":
        total = int(state["mesh"].node_offsets[-1])
        g = torch.Generator(device="cuda").manual_seed(seed % (1 << 62))
        state["p"] = torch.randn(total, dtype=torch.float64, device="cuda", generator=g)
    if case["kind"] == "design":
        state["centres"] = torch.tensor(geo[0].bodies[:, :2], dtype=torch.float64)
    return state


def _solve(mesh, case):
    return api.psi_solve(mesh, U=1.0, tol=case["tol"], precision=_precision(case), preconditioner=case["precond"])


def _copfi(mesh):
    return np.array([api.copfi(mesh, v, 3, 4, 1.0) for v in range(mesh.n_variants)])


def run(state):
    case = state["case"]
    if case["kind"] == "apply":
        y, sums = api.apply(state["mesh"], state["p"], _precision(case))
        return {"y": y, "body_sums": sums}
    if case["kind"] == "design":
        k = state["geo"][0]
        c = state["centres"].clone().requires_grad_()
        J = autograd.objective(c, k.bodies[:, 2], k.grid, k.sweeps, k.bc, tol=case["tol"])
        J.backward()
        return {"J": J.detach(), "dJdc": c.grad}
    if case["kind"] == "study":
        with api.batch_build(state["geo"]) as mesh:
            res = _solve(mesh, case)
            return {"psi": res.psi, "body_psi": res.body_psi, "copfi": _copfi(mesh)}
    mesh = state["mesh"]
    res = _solve(mesh, case)
    out = {"psi": res.psi, "body_psi": res.body_psi}
    if case["kind"] == "grad":
        out["dJdX"], out["dJdc"], out["J"] = api.grad(mesh, api.PF_OBJ_COPFI, 3, 4, 1.0, case["tol"])
    elif case["layout"] == "channel":
        out["copfi"] = _copfi(mesh)
    if case["layout"] in ("channel", "airfoil"):
        out["velocity"] = api.velocity_field(mesh, 0)
    return out


# ------------------------------------------------------------------ least work


def _sizes(case):
    """(nx, ny) of the variants; the mean of the range for uneven grids."""
    nx = case["nx"]
    if case["layout"] == "sweep":
        ks = range(256, nx + 1, 32)
        return [(k, k // 2) for k in ks], case["variants"] / len(ks)
    return [(nx, nx // 2)], case["variants"]


def _iterations(case, nx):
    """CG iterations of one solve, measured on these layouts: proportional to the cells across
    the domain for the plain CG (fewer in FP64), nearly constant for the multigrid one."""
    if case["precond"] == "mg":
        return 45
    if case["precision"] == "fp64":
        return 2.6 * nx
    return {"cylinder": 3.3, "five": 3.6, "sweep": 3.6, "channel": 4.6, "airfoil": 2.6}[case["layout"]] * nx


def work(case):
    """Least bytes and operations of one pass.  The operator: the vector read and written
    once, one tag byte per node.  A CG iteration: x, r and p read and written once.  A
    multigrid iteration: those, and on the fine level the residual, the smoothed vector and
    its correction once each (a third more for the coarser levels).  Operations: 16 per
    node and operator row, 14 for the updates and dot products."""
    sizes, each = _sizes(case)
    size = 8 if case["precision"] == "fp64" else 4
    total_b = total_f = 0.0
    for nx, ny in sizes:
        n = (nx + 1.0) * (ny + 1.0)
        if case["kind"] == "apply":
            total_b += 17.0 * n
            total_f += 16.0 * n
            continue
        its = _iterations(case, nx)
        solves = 2.0 if case["kind"] in ("grad", "design") or case["layout"] == "airfoil" else 1.0
        per_b, per_f = 6.0 * size, 30.0
        if case["precond"] == "mg":
            per_b, per_f = 14.0 * size, 80.0
        total_b += solves * its * n * per_b + 8.0 * n
        total_f += solves * its * n * per_f
        if case["kind"] in ("study", "design"):
            total_b += 16.0 * n
            total_f += 8.0 * n * case["sweeps"]
        if case["kind"] == "grad":
            total_b += 16.0 * n
            total_f += 100.0 * n + 8.0 * n * case["sweeps"]
    return {"bytes": total_b * each, "flops": total_f * each}


# ------------------------------------------------------------------ 64-bit results
#
# The method in plain torch, float64: the body-conforming mesh of circles (a node is inside a
# body when (x-cx)^2 + (y-cy)^2 <= r^2; inside corners of cells with an outside corner move
# radially onto the circle; the displacement is spread by Jacobi sweeps), Q4 element matrices
# by 2x2 Gauss quadrature, their off-diagonal entries summed per pair of neighbouring nodes,
# and CG on the free nodes and one value per body, restarted from the true residual.


class _Exact:
    def __init__(self, geo, differentiable=False):
        dev = "cuda" if torch.cuda.is_available() else "cpu"
        f8 = dict(dtype=torch.float64, device=dev)
        k = geo[0]
        self.bodies = torch.tensor(np.stack([g.bodies for g in geo]), **f8)      # [v, b, 3]
        V, B = self.bodies.shape[:2]
        self.V, self.B, self.ny, self.nx = V, B, k.ny, k.nx
        self.valid = True
        hx, hy = (k.x1 - k.x0) / k.nx, (k.y1 - k.y0) / k.ny
        x = (k.x0 + torch.arange(k.nx + 1, **f8) * hx).expand(k.ny + 1, -1)
        y = (k.y0 + torch.arange(k.ny + 1, **f8) * hy)[:, None].expand(-1, k.nx + 1)
        bid = torch.full((V, k.ny + 1, k.nx + 1), -1, dtype=torch.int64, device=dev)
        for b in range(B):
            cx, cy, r = (self.bodies[:, b, m][:, None, None] for m in range(3))
            bid[(x - cx) ** 2 + (y - cy) ** 2 <= r * r] = b
        out = bid < 0
        self.active = out[:, :-1, :-1] | out[:, :-1, 1:] | out[:, 1:, :-1] | out[:, 1:, 1:]
        touch = torch.zeros_like(out)
        for j in (slice(None, -1), slice(1, None)):
            for i in (slice(None, -1), slice(1, None)):
                touch[:, j, i] |= self.active
        self.body = ~out & touch
        ring = torch.zeros_like(out)
        for side, at in zip(k.bc, ((slice(None), slice(None), 0), (slice(None), slice(None), -1),
                                   (slice(None), 0), (slice(None), -1))):
            if side == W.BC_DIRICHLET_UY:
                ring[at] = True
        self.dirichlet = ring & out
        self.free = out & ~ring
        self.bnode = torch.nonzero(self.body.reshape(-1)).reshape(-1)
        where = bid.reshape(-1)[self.bnode] + B * (self.bnode // ((k.ny + 1) * (k.nx + 1)))
        self.where = where                                                       # v * B + b of each body node
        self.c = self.bodies[:, :, :2].clone()
        if differentiable:
            self.c.requires_grad_()
        # radial projection and Jacobi sweeps of the displacement
        cc = self.c.reshape(-1, 2)[where]
        rr = self.bodies[:, :, 2].reshape(-1)[where]
        gx = x.expand(V, -1, -1).reshape(-1)[self.bnode]
        gy = y.expand(V, -1, -1).reshape(-1)[self.bnode]
        ex, ey = gx - cc[:, 0], gy - cc[:, 1]
        rho = torch.sqrt(ex * ex + ey * ey)
        N = V * (k.ny + 1) * (k.nx + 1)
        inner = out[:, 1:-1, 1:-1]
        coords = []
        for g, ctr, e, base in ((gx, cc[:, 0], ex, x), (gy, cc[:, 1], ey, y)):
            d = torch.zeros(N, **f8).index_put((self.bnode,), ctr + rr * e / rho - g).reshape(V, k.ny + 1, k.nx + 1)
            for _ in range(k.sweeps):
                s = 0.25 * (d[:, 1:-1, :-2] + d[:, 1:-1, 2:] + d[:, :-2, 1:-1] + d[:, 2:, 1:-1])
                d = torch.nn.functional.pad(torch.where(inner, s, d[:, 1:-1, 1:-1]), (1, 1, 1, 1))
            coords.append(base + d)
        self.X, self.Y = coords
        self.g = torch.where(self.dirichlet, self.Y.detach(), 0.0)               # psi = U y, U = 1

    def weights(self, X, Y):
        """Off-diagonal entries of the assembled operator towards E, N, NE and NW neighbours."""
        cx = [X[:, :-1, :-1], X[:, :-1, 1:], X[:, 1:, 1:], X[:, 1:, :-1]]
        cy = [Y[:, :-1, :-1], Y[:, :-1, 1:], Y[:, 1:, 1:], Y[:, 1:, :-1]]
        sx, sy = (-1, 1, 1, -1), (-1, -1, 1, 1)
        pairs = ((0, 1), (0, 2), (0, 3), (1, 2), (1, 3), (2, 3))
        K = {p: 0.0 for p in pairs}
        q = 1.0 / math.sqrt(3.0)
        for xi, eta in ((-q, -q), (q, -q), (q, q), (-q, q)):
            dxi = [0.25 * a * (1 + b * eta) for a, b in zip(sx, sy)]
            det_ = [0.25 * b * (1 + a * xi) for a, b in zip(sx, sy)]
            xx, xe = sum(d * c for d, c in zip(dxi, cx)), sum(d * c for d, c in zip(det_, cx))
            yx, ye = sum(d * c for d, c in zip(dxi, cy)), sum(d * c for d, c in zip(det_, cy))
            J = xx * ye - xe * yx
            gx = [(ye * a - yx * b) for a, b in zip(dxi, det_)]
            gy = [(xx * b - xe * a) for a, b in zip(dxi, det_)]
            for a, b in pairs:
                K[a, b] = K[a, b] + (gx[a] * gx[b] + gy[a] * gy[b]) / J
            self.valid &= bool((torch.where(self.active, J, 1.0) > 0).all())
        K = {p: torch.where(self.active, m, 0.0) for p, m in K.items()}
        pad = torch.nn.functional.pad
        wE = pad(K[0, 1], (0, 0, 0, 1)) + pad(K[2, 3], (0, 0, 1, 0))             # [v, ny+1, nx]
        wN = pad(K[0, 3], (0, 1)) + pad(K[1, 2], (1, 0))                         # [v, ny, nx+1]
        return wE, wN, K[0, 2], K[1, 3]

    @staticmethod
    def apply(w, p):
        wE, wN, wD, wA = w
        y = torch.zeros_like(p)
        for wt, a, b in ((wE, p[:, :, :-1], p[:, :, 1:]), (wN, p[:, :-1], p[:, 1:]),
                         (wD, p[:, :-1, :-1], p[:, 1:, 1:]), (wA, p[:, :-1, 1:], p[:, 1:, :-1])):
            f = wt * (b - a)
            ya, yb = ((y[:, :, :-1], y[:, :, 1:]) if wt is wE else (y[:, :-1], y[:, 1:]) if wt is wN
                      else (y[:, :-1, :-1], y[:, 1:, 1:]) if wt is wD else (y[:, :-1, 1:], y[:, 1:, :-1]))
            ya += f
            yb -= f
        return y

    def spread(self, f, c):
        """Nodal field of free values f and body values c."""
        return f.reshape(-1).index_put((self.bnode,), c.reshape(-1)[self.where]).reshape(f.shape)

    def sums(self, y):
        return torch.zeros(self.V * self.B, dtype=y.dtype, device=y.device).index_add_(
            0, self.where, y.reshape(-1)[self.bnode]).reshape(self.V, self.B)

    def rows(self, w, field):
        y = self.apply(w, field)
        return torch.where(self.free, y, 0.0), self.sums(y)

    def cg(self, w, rf, rc, most):
        """CG on the free nodes and body values from a zero guess: (field, body values)."""
        dot = lambda a, b, c, d: (a * b).sum((1, 2)) + (c * d).sum(1)  # noqa: E731
        xf, xc = torch.zeros_like(rf), torch.zeros_like(rc)
        pf, pc = rf.clone(), rc.clone()
        g = g0 = dot(rf, rf, rc, rc)
        for it in range(most):
            qf, qc = self.rows(w, self.spread(pf, pc))
            pq = dot(pf, qf, pc, qc)
            al = torch.where(pq > 0, g / pq, 0.0)
            a3, a2 = al[:, None, None], al[:, None]
            xf.addcmul_(a3, pf), xc.addcmul_(a2, pc)
            rf = rf.addcmul(a3, qf, value=-1)
            rc = rc.addcmul(a2, qc, value=-1)
            gn = dot(rf, rf, rc, rc)
            be = torch.where(g > 0, gn / g, 0.0)
            pf = pf.mul_(be[:, None, None]).add_(rf)
            pc = pc.mul_(be[:, None]).add_(rc)
            g = gn
            if it % 64 == 63 and bool((g <= 1e-28 * g0).all()):
                break
        return xf, xc

    def solve(self, w, rf, rc):
        """Two CG solves, the second on the true residual of the first."""
        most = 12 * max(self.nx, self.ny)
        xf, xc = self.cg(w, rf, rc, most)
        yf, yc = self.rows(w, self.spread(xf, xc))
        df, dc = self.cg(w, rf - yf, rc - yc, most)
        return xf + df, xc + dc


def _flat(t):
    return t.reshape(-1)


def exact(case, seed):
    if case["layout"] in ("sweep", "airfoil") or case["kind"] == "study":
        return None                       # hundreds of grids, or polygons
    nodes = case["variants"] * (case["nx"] + 1.0) * (case["nx"] // 2 + 1.0)
    if case["kind"] != "apply" and nodes * case["nx"] > 2.5e10:
        return None                       # minutes of unpreconditioned FP64 CG
    differentiable = case["kind"] in ("grad", "design")
    if differentiable and nodes * case["sweeps"] > 2e8:
        return None                       # the sweeps' graph would not fit the time
    for attempt in range(TRIES):
        e = _Exact(_geometry(case, seed, attempt)[0], differentiable)
        with torch.no_grad():
            w = e.weights(e.X, e.Y)
        if e.valid:
            break
    if case["kind"] == "apply":
        g = torch.Generator(device="cuda").manual_seed(seed % (1 << 62))
        p = torch.randn(int(nodes), dtype=torch.float64, device="cuda", generator=g).reshape(e.free.shape)
        y = e.apply(w, p)
        return {"y": _flat(torch.where(e.free | e.body, y, 0.0)), "body_sums": _flat(e.sums(y)).cpu().numpy()}
    with torch.no_grad():
        lf, lc = e.rows(w, e.g)
        uf, C = e.solve(w, -lf, -lc)
        psi = e.spread(uf + e.g, C)
    body = _flat(C).cpu().numpy()
    lo, hi = 3, 4
    if not differentiable:
        out = {"psi": _flat(psi), "body_psi": body}
        if case["layout"] == "channel":
            q = C[:, hi] - C[:, lo]
            out["copfi"] = torch.stack([q / (e.bodies[:, hi, 1] - e.bodies[:, lo, 1]), q], 1).cpu().numpy()
            out["velocity"] = None
        return out
    # J = (C_hi - C_lo) / (cy_hi - cy_lo); the adjoint lambda solves A lambda = dJ/dC, and
    # dJ = -lambda^T (dK) psi: the graph runs from the weights back to the centres
    gap = e.c[:, hi, 1] - e.c[:, lo, 1]
    J = ((C[:, hi] - C[:, lo]) / gap).detach()
    with torch.no_grad():
        rc = torch.zeros_like(C)
        rc[:, hi], rc[:, lo] = 1.0 / gap.detach(), -1.0 / gap.detach()
        lam = e.spread(*e.solve(w, torch.zeros_like(uf), rc))
    X, Y = e.X.detach().requires_grad_(), e.Y.detach().requires_grad_()
    wE, wN, wD, wA = e.weights(X, Y)
    s = 0.0
    for wt, a, b in ((wE, (..., slice(None, -1)), (..., slice(1, None))),
                     (wN, (slice(None), slice(None, -1)), (slice(None), slice(1, None))),
                     (wD, (slice(None), slice(None, -1), slice(None, -1)), (slice(None), slice(1, None), slice(1, None))),
                     (wA, (slice(None), slice(None, -1), slice(1, None)), (slice(None), slice(1, None), slice(None, -1)))):
        s = s + (wt * (lam[b] - lam[a]) * (psi[b] - psi[a])).sum()
    gX, gY = torch.autograd.grad(s, (X, Y))
    gY = gY - torch.where(e.dirichlet, e.apply(w, lam), 0.0)    # the Dirichlet data is U y
    explicit = ((C[:, hi] - C[:, lo]) / gap).sum()
    (dc,) = torch.autograd.grad((e.X * gX).sum() + (e.Y * gY).sum() + explicit, e.c)
    if case["kind"] == "design":
        return {"J": J[0].cpu(), "dJdc": dc[0].cpu()}
    return {"psi": _flat(psi), "body_psi": body, "dJdX": torch.stack([_flat(gX), _flat(gY)], 1),
            "dJdc": dc.reshape(-1, 2).cpu().numpy(), "J": J.cpu().numpy()}

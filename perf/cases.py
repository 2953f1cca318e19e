"""Performance cases: the calls that a user of this framework makes, over the
range of sizes it is used at.

A case is a dict of plain values:
  path       what one pass does: "apply" (the operator), "solve" (block solves
             with factors in hand), "refactor_solve" (one step of a frequency
             sweep: factor new shifts, solve), "resolvent" (factor new shifts,
             then Algorithm 1), "gradient" (factor, then the gain gradient) or
             "batch" (one run of a batch plan)
  kind       operator: "advdiff" (q = 1), "ns2d" (q = 3), "kz" (q = 4)
  nx, ny     grid; the block of one streamwise column has b = q ny rows
  F, k       shifts and right-hand sides (sketch columns)
  precision  arithmetic of the factors
  adjoint, neumann (the paper's boundary closure), weighted (diagonal W),
  tol        the refinement tolerance

Everything random (base flow, frequencies, right-hand sides, test-matrix
seeds, weights) comes from the seed.
"""
import math
from types import SimpleNamespace

import numpy as np
import torch

import paper_1902_01458_gb300 as rr

DEV = "cuda:0"
Q = {"advdiff": 1, "ns2d": 3, "kz": 4}
KIND = {"advdiff": 1, "ns2d": 3, "kz": 4}
KZ = 2.0 * math.pi
J = 3  # leading gains of the gradient workload
MAX_REFINE = 20
# problems of the batch plan: offsets from the case's nx, ny, k
BATCH_SHAPES = ((0, 0, 0), (0, 0, 1), (1, 0, 0), (0, 1, 2), (1, 1, 0), (0, 0, 0))


def _case(name, path, kind, nx, ny, F, k, precision="fp32", adjoint=False, neumann=False,
          weighted=False, tol=1e-10):
    return {"name": name, "path": path, "kind": kind, "nx": nx, "ny": ny, "F": F, "k": k,
            "precision": precision, "adjoint": adjoint, "neumann": neumann,
            "weighted": weighted, "tol": tol}


def listed():
    return [
        # the scalar advection-diffusion workload's operator applied once: a
        # call that costs its launch and its host path
        _case("apply_small", "apply", "advdiff", 32, 32, 1, 10),
        # residual check of a whole adjoint solve block on the 256x128
        # Navier-Stokes grid with the paper's boundary closure
        _case("apply_adjoint", "apply", "ns2d", 256, 128, 8, 16, adjoint=True, neumann=True),
        # the small Navier-Stokes example end to end in FP64: factor three new
        # frequencies and run Algorithm 1 (setting up a study, smoke tests)
        _case("resolvent_small_fp64", "resolvent", "ns2d", 24, 20, 3, 8, "fp64", tol=1e-12),
        # bi-global operator: solves of a few right-hand sides with weights
        _case("solve_kz_weighted", "solve", "kz", 96, 40, 6, 8, weighted=True, tol=1e-12),
        # adjoint solves at 256x128, eight frequencies of the 16-column sketch
        _case("solve_adjoint_mid", "solve", "ns2d", 256, 128, 8, 16, adjoint=True, tol=1e-12),
        # the headline grid: one solve block of Algorithm 1 at 512x256, k = 32
        _case("solve_large", "solve", "ns2d", 512, 256, 16, 32, tol=1e-12),
        # a step of a frequency sweep on the smallest grid of the batching
        # workload, two frequencies at a time
        _case("sweep_step_small", "refactor_solve", "ns2d", 128, 64, 2, 8, tol=1e-12),
        # a step of the headline frequency sweep: factor and solve at 512x256
        _case("sweep_step_large", "refactor_solve", "ns2d", 512, 256, 6, 32, tol=1e-12),
        # the whole of Algorithm 1 for a batch of frequencies at 256x128
        _case("resolvent_mid", "resolvent", "ns2d", 256, 128, 8, 16, tol=1e-12),
        # a wide sketch on a small grid: QR and small SVD of 64 columns
        _case("resolvent_wide_sketch", "resolvent", "ns2d", 128, 64, 4, 64, tol=1e-12),
        # backward pass of the gain objective: FP64 factors of a chunk of
        # frequencies and the gradient of the three leading gains
        _case("gradient_fp64", "gradient", "ns2d", 128, 64, 4, 16, "fp64"),
        # an uneven batch (grids and k differ) as one graph run
        _case("batch_uneven", "batch", "ns2d", 128, 64, 6, 16, tol=1e-12),
    ]


def _cost(c):
    """Rough seconds of a pass, to keep drawn cases below the largest listed."""
    b = Q[c["kind"]] * c["ny"]
    n = b * c["nx"]
    rate = 6e11 if c["precision"] == "fp64" else 1.5e13
    panel = 16 if b % 8 == 0 and c["precision"] != "fp64" else 8
    factor = c["nx"] * (b / panel * 6e-5 + c["F"] * 8.0 * b ** 3 / rate)
    solve = c["nx"] * (4e-5 + c["F"] * 16.0 * b * b * max(c["k"], 8) / rate)
    dense = c["F"] * n * c["k"] * 30 / 1e11
    return {"apply": dense, "solve": 5 * solve + 3 * dense,
            "refactor_solve": factor + 5 * solve + 3 * dense,
            "resolvent": factor + 15 * solve + 15 * dense + c["F"] * n * c["k"] ** 2 * 60 / 1e12,
            "gradient": factor + 6 * solve + 4 * dense,
            "batch": c["nx"] * 2.5e-3 + 4 * factor}[c["path"]]


def draw(rng):
    def logint(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    while True:
        path = rng.choice(["apply", "solve", "solve", "refactor_solve", "refactor_solve",
                           "resolvent", "gradient", "batch"])
        kind = "ns2d" if path in ("resolvent", "gradient", "batch") else rng.choice(
            ["ns2d", "ns2d", "ns2d", "kz", "advdiff"])
        ny = logint(16, 1000 // Q[kind] if kind != "ns2d" else 256)
        if path == "batch" and ny > 100:  # its plan has grids of up to three times ny
            continue
        if rng.random() < 0.6:
            ny = max(16, ny // 8 * 8)  # most grids are multiples of 8, some are odd
        nx = logint(16, 512)
        F = logint(1, 32) if path != "batch" else rng.randint(3, len(BATCH_SHAPES))
        precision = "fp64" if path == "gradient" else rng.choice(
            ["fp32", "fp32", "fp32", "fp64", "fp32_bf16x6"])
        if path == "resolvent":
            k = rng.choice([4, 8, 12, 16])
            precision = rng.choice(["fp32", "fp64"])
        elif path == "gradient":
            k = rng.choice([8, 16])
        elif path == "batch":
            k, precision = rng.choice([8, 16]), "fp32"
        else:
            k = logint(1, 32) if rng.random() < 0.4 else rng.choice([4, 8, 16, 32])
        c = _case("", path, kind, nx, ny, F, k, precision,
                  adjoint=path in ("apply", "solve", "refactor_solve") and rng.random() < 0.4,
                  neumann=rng.random() < 0.25,
                  weighted=path != "batch" and rng.random() < 0.15,
                  tol=1e-10 if path in ("apply", "gradient") else 1e-12)
        del c["name"]
        b = Q[kind] * ny
        if F * nx * b * b * (16 if precision == "fp64" else 8) > 2.5e10:
            continue
        if F * nx * b * k * 16 > 4e9 or _cost(c) > 0.6 or (path != "apply" and k > nx * b):
            continue
        return c


# ------------------------------------------------------------------ inputs
def _fields(case, seed, nx, ny):
    """A separated shear layer with a recirculation bubble and a smooth seeded
    perturbation of density and velocity, on the interior nodes."""
    rng = np.random.default_rng([int(seed), nx, ny])
    g = _grid(case, nx, ny)
    x = g.x0 + (g.x1 - g.x0) / (nx + 1) * np.arange(1, nx + 1)
    y = g.y0 + (g.y1 - g.y0) / (ny + 1) * np.arange(1, ny + 1)
    X, Y = np.meshgrid(x, y, indexing="ij")
    shear = 0.5 * (1.0 + np.tanh(Y / 0.5))
    bubble = np.exp(-((X - 6.0) / 3.0) ** 2 - ((Y + 0.5) / 0.75) ** 2)
    base = (np.ones_like(X), shear * (1.0 - bubble) - 0.2 * bubble, np.zeros_like(X))
    out = []
    for f in base:
        a, b = rng.uniform(0.3, 1.2, size=2)
        p, q = rng.uniform(0.0, 2.0 * math.pi, size=2)
        out.append(f + 0.02 * np.sin(a * X + p) * np.cos(b * Y + q))
    return out


def _grid(case, nx, ny):
    kind = case["kind"]
    mask = (0, 0, 0, 0)
    if case["neumann"]:
        mask = {"advdiff": (0, 1, 0, 0), "ns2d": (1, 7, 1, 1), "kz": (1, 15, 1, 1)}[kind]
    return SimpleNamespace(kind=KIND[kind], nx=nx, ny=ny, periodic_y=False, x0=0.0, x1=20.0,
                           y0=-5.0, y1=5.0, re=100.0 if kind == "advdiff" else 500.0, mach=0.3,
                           sponge_max=1.0, sponge_frac=0.1, neumann=mask,
                           kz=KZ if kind == "kz" else 0.0)


def _weights(case, seed, n):
    if not case["weighted"]:
        return None
    return np.random.default_rng([int(seed), 7]).uniform(0.5, 2.0, n)


def _shifts(case, seed, F):
    rng = np.random.default_rng([int(seed), 11])
    om = np.exp(rng.uniform(math.log(0.1), math.log(5.0), F))
    return 1j * np.sort(om)


def _seeds(seed, F):
    return [(int(seed) * 1000003 + 1000 + j) & 0x7FFFFFFF for j in range(F)]


def _randn(case, seed, shape, extra=0):
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed) * 31 + extra)
    return torch.randn(*shape, 2, dtype=torch.float64, device=DEV, generator=g)


def _block(case, seed, shape, extra=0):
    return torch.view_as_complex(_randn(case, seed, shape, extra)).contiguous()


def _operator(case, seed, nx, ny):
    rho, u, v = _fields(case, seed, nx, ny)
    w = _weights(case, seed, nx * ny * Q[case["kind"]])
    return rr.Operator(_grid(case, nx, ny), SimpleNamespace(rho=rho, u=u, v=v), weights=w)


def _triplets(case, seed):
    """Orthonormal U, V and descending gains, as Algorithm 1 leaves them."""
    n = case["nx"] * case["ny"] * Q[case["kind"]]
    F, k = case["F"], case["k"]
    U = torch.linalg.qr(_block(case, seed, (F, n, k), 1))[0].contiguous()
    V = torch.linalg.qr(_block(case, seed, (F, n, k), 2))[0].contiguous()
    s = np.sort(np.random.default_rng([int(seed), 13]).uniform(1.0, 50.0, (F, k)))[:, ::-1]
    return U, V, torch.from_numpy(s.copy()).to(DEV)


def _batch_list(case, seed):
    shifts = _shifts(case, seed, len(BATCH_SHAPES))
    seeds = _seeds(seed, len(BATCH_SHAPES))
    return [{"nx": case["nx"] * (1 + a), "ny": case["ny"] * (1 + c), "k": case["k"] >> e,
             "shift": shifts[i], "seed": seeds[i]}
            for i, (a, c, e) in enumerate(BATCH_SHAPES[:case["F"]])]


def prepare(case, seed):
    path, nx, ny, F, k = case["path"], case["nx"], case["ny"], case["F"], case["k"]
    n = nx * ny * Q[case["kind"]]
    st = SimpleNamespace(case=case)
    if path == "batch":
        st.ops = {}
        probs = []
        for p in _batch_list(case, seed):
            key = (p["nx"], p["ny"])
            if key not in st.ops:
                st.ops[key] = _operator(case, seed, *key)
            probs.append({"op": st.ops[key], "shift": p["shift"], "k": p["k"],
                          "seed": p["seed"]})
        st.plan = rr.Batch(probs, precision=case["precision"], refine_tol=case["tol"],
                           max_refine=MAX_REFINE)
        return st
    st.op = _operator(case, seed, nx, ny)
    st.shifts = _shifts(case, seed, F)
    if path == "apply":
        st.x = _block(case, seed, (F, n, k))
        return st
    # a sweep holds factors already (of the step before: other shifts)
    first = st.shifts if path == "solve" else st.shifts * 1.05
    st.fa = st.op.factor(first, case["precision"])
    if path in ("solve", "refactor_solve"):
        st.b = _block(case, seed, (F, n, k))
    elif path == "resolvent":
        st.phi = st.op.phi()
        st.seeds = _seeds(seed, F)
    else:
        st.U, st.V, st.sigma = _triplets(case, seed)
    return st


def run(st):
    c = st.case
    path = c["path"]
    if path == "apply":
        return st.op.apply(st.shifts, st.x, adjoint=c["adjoint"])
    if path == "batch":
        st.plan.run()
        return st.plan.outputs
    if path != "solve":
        st.fa.refactor(st.shifts)
    if path in ("solve", "refactor_solve"):
        x, _ = st.fa.solve(st.b, adjoint=c["adjoint"], refine_tol=c["tol"],
                           max_refine=MAX_REFINE)
        return x
    if path == "resolvent":
        r = st.fa.randomized_resolvent(c["k"], st.seeds, phi=st.phi, refine_tol=c["tol"],
                                       max_refine=MAX_REFINE)
        return {"sigma": r.sigma, "sigma_halko": r.sigma_halko, "U": r.U, "V": r.V}
    grad, _ = st.fa.gain_grad(J, st.U, st.V, st.sigma, refine_tol=c["tol"],
                              max_refine=MAX_REFINE)
    return grad


def work(case):
    """One block inverse per streamwise column (8 b^3 real operations), and
    two products with it per column and right-hand side of a solve; factors
    are read once per direction of a solve, vectors once per call."""
    path = case["path"]
    if path == "batch":
        tot = {"bytes": 0.0, "flops": 0.0}
        for p in _batch_list(case, 0):
            w = work(dict(case, path="resolvent", nx=p["nx"], ny=p["ny"], k=p["k"], F=1))
            tot = {m: tot[m] + w[m] for m in tot}
        return tot
    b = Q[case["kind"]] * case["ny"]
    nx, F, k = case["nx"], case["F"], case["k"]
    n, e = nx * b, 16 if case["precision"] == "fp64" else 8
    nz = {"advdiff": 5, "ns2d": 13, "kz": 16}[case["kind"]]
    vec = 16.0 * F * n * k
    if path == "apply":
        return {"bytes": 2 * vec + 8.0 * n * nz, "flops": 4.0 * F * n * k * nz}
    G = float(e) * F * nx * b * b
    solve = {"bytes": 2 * G + 2 * vec, "flops": 2 * 8.0 * F * nx * b * b * k}
    factor = {"bytes": G, "flops": 8.0 * F * nx * b ** 3}
    if path == "solve":
        return solve
    if path == "refactor_solve":
        return {m: factor[m] + solve[m] for m in solve}
    if path == "resolvent":
        dense = {"bytes": 6 * vec, "flops": 8.0 * F * n * k * k * 6}
        return {m: factor[m] + 3 * solve[m] + dense[m] for m in solve}
    grad = {"bytes": 2 * vec, "flops": 4.0 * F * n * J * nz * 4}
    return {m: factor[m] + 2 * solve[m] * J / k + grad[m] for m in solve}


# ------------------------------------------- the same in 64 bits, in torch
def _roll(a, d, dim):
    """a shifted so that entry i holds a[i + d] (zero beyond the ends)."""
    if d == 0:
        return a
    out = torch.zeros_like(a)
    n = a.shape[dim]
    out.narrow(dim, max(0, -d), n - abs(d)).copy_(a.narrow(dim, max(0, d), n - abs(d)))
    return out


def _diff(n, h, order):
    """Difference matrix of a known field: central, one-sided (first) or
    re-centred (second) at the end nodes."""
    m = np.zeros((n, n))
    for i in range(n):
        if order == 2:
            c = min(max(i, 1), n - 2)
            m[i, c - 1:c + 2] += np.array([1.0, -2.0, 1.0]) / h ** 2
        else:
            lo, hi = max(i - 1, 0), min(i + 1, n - 1)
            m[i, hi] += 1.0 / ((hi - lo) * h)
            m[i, lo] -= 1.0 / ((hi - lo) * h)
    return torch.from_numpy(m).to(DEV)


def _stencil(case, g, rho, u, v):
    """Entries of L per node: [3 (dx), 3 (dy), q (equation), q (variable), nx, ny]."""
    nx, ny, q = g.nx, g.ny, Q[case["kind"]]
    dx, dy = (g.x1 - g.x0) / (nx + 1), (g.y1 - g.y0) / (ny + 1)
    x = g.x0 + dx * torch.arange(1, nx + 1, dtype=torch.float64, device=DEV)[:, None]
    y = g.y0 + dy * torch.arange(1, ny + 1, dtype=torch.float64, device=DEV)[None, :]
    lx, ly = g.sponge_frac * (g.x1 - g.x0), g.sponge_frac * (g.y1 - g.y0)
    xi = torch.maximum(g.x0 + lx - x, x - (g.x1 - lx)).clamp(min=0.0).div(lx).clamp(max=1.0)
    yi = torch.maximum(g.y0 + ly - y, y - (g.y1 - ly)).clamp(min=0.0).div(ly).clamp(max=1.0)
    sg = g.sponge_max * torch.maximum(xi.expand(nx, ny), yi.expand(nx, ny)) ** 2
    cplx = case["kind"] == "kz"
    zero = torch.zeros(nx, ny, dtype=torch.complex128 if cplx else torch.float64, device=DEV)
    ent = {}

    def add(a, c, ox, oy, val):
        key = (ox, oy, a, c)
        ent[key] = ent.get(key, zero) + val

    def d1x(a, c, w):
        add(a, c, 1, 0, w / (2 * dx))
        add(a, c, -1, 0, -w / (2 * dx))

    def d1y(a, c, w):
        add(a, c, 0, 1, w / (2 * dy))
        add(a, c, 0, -1, -w / (2 * dy))

    def d2x(a, c, w):
        for o, f in ((1, 1.0), (-1, 1.0), (0, -2.0)):
            add(a, c, o, 0, f * w / dx ** 2)

    def d2y(a, c, w):
        for o, f in ((1, 1.0), (-1, 1.0), (0, -2.0)):
            add(a, c, 0, o, f * w / dy ** 2)

    def dxy(a, c, w):
        for ox in (1, -1):
            for oy in (1, -1):
                add(a, c, ox, oy, ox * oy * w / (4 * dx * dy))

    one = torch.ones_like(u)
    for a in range(q):
        d1x(a, a, -u)
        d1y(a, a, -v)
        add(a, a, 0, 0, -sg)
    if q == 1:
        d2x(0, 0, one / g.re)
        d2y(0, 0, one / g.re)
    else:
        X1, Y1, X2, Y2 = _diff(nx, dx, 1), _diff(ny, dy, 1), _diff(nx, dx, 2), _diff(ny, dy, 2)
        Dx, Dy = (lambda f: X1 @ f), (lambda f: f @ Y1.T)
        Dxx, Dyy, Dxy = (lambda f: X2 @ f), (lambda f: f @ Y2.T), (lambda f: X1 @ f @ Y1.T)
        c2, mu = 1.0 / g.mach ** 2, 1.0 / (rho * g.re)
        fu = (Dxx(u) + Dyy(u) + (Dxx(u) + Dxy(v)) / 3) / g.re
        fv = (Dxx(v) + Dyy(v) + (Dxy(u) + Dyy(v)) / 3) / g.re
        add(0, 0, 0, 0, -(Dx(u) + Dy(v)))
        d1x(0, 1, -rho)
        add(0, 1, 0, 0, -Dx(rho))
        d1y(0, 2, -rho)
        add(0, 2, 0, 0, -Dy(rho))
        d1x(1, 0, -c2 / rho)
        add(1, 0, 0, 0, (c2 * Dx(rho) - fu) / rho ** 2)
        d2x(1, 1, mu * (4.0 / 3))
        d2y(1, 1, mu)
        add(1, 1, 0, 0, -Dx(u))
        dxy(1, 2, mu / 3)
        add(1, 2, 0, 0, -Dy(u))
        d1y(2, 0, -c2 / rho)
        add(2, 0, 0, 0, (c2 * Dy(rho) - fv) / rho ** 2)
        dxy(2, 1, mu / 3)
        add(2, 1, 0, 0, -Dx(v))
        d2x(2, 2, mu)
        d2y(2, 2, mu * (4.0 / 3))
        add(2, 2, 0, 0, -Dy(v))
        if q == 4:
            ik = 1j * g.kz
            add(0, 3, 0, 0, -ik * rho)
            add(1, 1, 0, 0, -g.kz ** 2 * mu)
            d1x(1, 3, ik * mu / 3)
            add(2, 2, 0, 0, -g.kz ** 2 * mu)
            d1y(2, 3, ik * mu / 3)
            add(3, 0, 0, 0, -ik * c2 / rho)
            d1x(3, 1, ik * mu / 3)
            d1y(3, 2, ik * mu / 3)
            d2x(3, 3, mu)
            d2y(3, 3, mu)
            add(3, 3, 0, 0, -(4.0 / 3) * g.kz ** 2 * mu)
    # ghost nodes: zero, or (a set bit of the side's mask) the adjacent node
    iX = torch.arange(nx, device=DEV)[:, None].expand(nx, ny)
    iY = torch.arange(ny, device=DEV)[None, :].expand(nx, ny)
    out = {}
    for (ox, oy, a, c), val in ent.items():
        gx = (iX + ox < 0) | (iX + ox >= nx)
        gy = (iY + oy < 0) | (iY + oy >= ny)
        fx = (g.neumann[0 if ox < 0 else 1] >> c) & 1
        fy = (g.neumann[2 if oy < 0 else 3] >> c) & 1
        for hx, hy in ((0, 0), (1, 0), (0, 1), (1, 1)):
            if (hx and not ox) or (hy and not oy) or (hx and not fx) or (hy and not fy):
                continue
            sel = (gx if hx else ~gx) & (gy if hy else ~gy)
            key = (0 if hx else ox, 0 if hy else oy, a, c)
            out[key] = out.get(key, zero) + val * sel
    rows = [out.get((ox, oy, a, c), zero) for ox in (-1, 0, 1) for oy in (-1, 0, 1)
            for a in range(q) for c in range(q)]
    return torch.stack(rows).reshape(3, 3, q, q, nx, ny)


class _Exact:
    """s I - L applied and solved in complex128 (block LU over the columns)."""

    def __init__(self, case, seed, nx, ny, fields=None):
        self.g = _grid(case, nx, ny)
        self.q, self.nx, self.ny = Q[case["kind"]], nx, ny
        f = fields or [torch.from_numpy(a).to(DEV) for a in _fields(case, seed, nx, ny)]
        self.rho, self.u, self.v = f
        self.c = _stencil(case, self.g, *f)
        self.blocks, self.lu = {}, {}

    def apply(self, s, x, adjoint=False):
        """x [N, k] -> (s I - L) x or its adjoint."""
        xs = x.reshape(self.nx, self.ny, self.q, -1)
        y = torch.zeros_like(xs)
        for ox in (-1, 0, 1):
            for oy in (-1, 0, 1):
                for a in range(self.q):
                    for c in range(self.q):
                        w = self.c[ox + 1, oy + 1, a, c][:, :, None]
                        if not bool(w.any()):
                            continue
                        if adjoint:
                            y[:, :, c] += _roll(_roll(w.conj() * xs[:, :, a], -ox, 0), -oy, 1)
                        else:
                            y[:, :, a] += w * _roll(_roll(xs[:, :, c], ox, 0), oy, 1)
        s = s.conjugate() if adjoint else s
        return s * x - y.reshape(x.shape)

    def _blk(self, i, ox):
        """Dense block L[column i, column i + ox]."""
        q, ny = self.q, self.ny
        B = torch.zeros(ny, q, ny, q, dtype=torch.complex128, device=DEV)
        iy = torch.arange(ny, device=DEV)
        for oy in (-1, 0, 1):
            m = (iy + oy >= 0) & (iy + oy < ny)
            r = iy[m]
            B[r, :, r + oy, :] += self.c[ox + 1, oy + 1, :, :, i][:, :, m].permute(2, 0, 1)
        return B.reshape(q * ny, q * ny)

    def _col(self, i, ox, adjoint):
        """Block (i, i + ox) of L or of L^H."""
        key = (i + ox, -ox) if adjoint else (i, ox)
        if key not in self.blocks:
            self.blocks[key] = self._blk(*key)
        return self.blocks[key].mH if adjoint else self.blocks[key]

    def _factor(self, s, adjoint):
        key = (s, adjoint)
        if key not in self.lu:
            eye = torch.eye(self.q * self.ny, dtype=torch.complex128, device=DEV)
            sv = s.conjugate() if adjoint else s
            lus, prev, up = [], None, None
            for i in range(self.nx):
                S = sv * eye - self._col(i, 0, adjoint)
                if i:
                    S = S - self._col(i, -1, adjoint) @ torch.linalg.lu_solve(*prev, up)
                prev = torch.linalg.lu_factor(S)
                up = self._col(i, 1, adjoint) if i + 1 < self.nx else None
                lus.append(prev)
            self.lu = {k: v for k, v in self.lu.items() if k[0] == s}  # one shift at a time
            self.lu[key] = lus
        return self.lu[key]

    def _once(self, lus, b, adjoint):
        k = b.shape[1]
        z = b.reshape(self.nx, -1, k).clone()
        for i in range(1, self.nx):
            z[i] += self._col(i, -1, adjoint) @ torch.linalg.lu_solve(*lus[i - 1], z[i - 1])
        for i in range(self.nx - 1, -1, -1):
            if i + 1 < self.nx:
                z[i] += self._col(i, 1, adjoint) @ z[i + 1]
            z[i] = torch.linalg.lu_solve(*lus[i], z[i])
        return z.reshape(b.shape)

    def solve(self, s, b, adjoint=False):
        lus = self._factor(s, adjoint)
        x = self._once(lus, b, adjoint)
        return x + self._once(lus, b - self.apply(s, x, adjoint), adjoint)


def _phi(case, ex):
    h = ((ex.g.x1 - ex.g.x0) / (ex.nx + 1), (ex.g.y1 - ex.g.y0) / (ex.ny + 1))
    X1, Y1 = _diff(ex.nx, h[0], 1), _diff(ex.ny, h[1], 1)
    p = ((X1 @ ex.u) ** 2 + (ex.u @ Y1.T) ** 2 + (X1 @ ex.v) ** 2 + (ex.v @ Y1.T) ** 2).sqrt()
    return p.reshape(-1).repeat_interleave(ex.q)


def _omega(seed, n, k):
    """Philox-4x32-10 (key seed, counter (row, column, 0, 0)), Box-Muller."""
    lo32 = 0xFFFFFFFF

    def mul(m, c):
        hi = (m * (c >> 16) + ((m * (c & 0xFFFF)) >> 16)) >> 16
        return hi & lo32, (m * c) & lo32

    c0 = torch.arange(n, device=DEV)[:, None].expand(n, k).clone()
    c1 = torch.arange(k, device=DEV)[None, :].expand(n, k).clone()
    c2, c3 = torch.zeros_like(c0), torch.zeros_like(c0)
    k0, k1 = seed & lo32, seed >> 32
    for _ in range(10):
        h0, l0 = mul(0xD2511F53, c0)
        h1, l1 = mul(0xCD9E8D57, c2)
        c0, c1, c2, c3 = h1 ^ c1 ^ k0, l1, h0 ^ c3 ^ k1, l0
        k0, k1 = (k0 + 0x9E3779B9) & lo32, (k1 + 0xBB67AE85) & lo32
    u1 = (((c0 >> 5) << 26) + (c1 >> 6) + 1).double() * 2.0 ** -53
    u2 = (((c2 >> 5) << 26) + (c3 >> 6)).double() * 2.0 ** -53
    return torch.sqrt(-2.0 * torch.log(u1)) * torch.cos(2.0 * math.pi * u2)


def _algorithm1(case, seed, ex, s, k, om_seed):
    n = ex.nx * ex.ny * ex.q
    w = _weights(case, seed, n)
    ws = None if w is None else torch.from_numpy(np.sqrt(w)).to(DEV)[:, None]

    def res(b, adj=False):
        if ws is None:
            return ex.solve(s, b, adj)
        return ex.solve(s, b * ws, True) / ws if adj else ws * ex.solve(s, b / ws)

    om = (_phi(case, ex)[:, None] * _omega(om_seed, n, k)).to(torch.complex128)
    q = torch.linalg.qr(res(om))[0]
    v, sh, _ = torch.linalg.svd(res(q, True), full_matrices=False)
    us = res(v)
    sig = torch.linalg.vector_norm(us, dim=0)
    order = torch.argsort(sig, descending=True, stable=True)
    v, u, sig = v[:, order], us[:, order] / sig[order], sig[order]
    e = v.gather(0, v.abs().argmax(dim=0, keepdim=True))
    ph = (e / e.abs()).conj()
    return {"sigma": sig, "sigma_halko": sh, "U": u * ph, "V": v * ph}


def exact(case, seed):
    path, nx, ny, F, k = case["path"], case["nx"], case["ny"], case["F"], case["k"]
    b = Q[case["kind"]] * ny
    n = nx * b

    def seconds(nx, b, F, dirs):  # block LUs and their triangular solves
        return dirs * F * nx * (4e-3 + 15.0 * b ** 3 / 2.5e11)

    shifts = [complex(s) for s in _shifts(case, seed, F)]
    if path == "apply":
        x = _block(case, seed, (F, n, k))
        ex = _Exact(case, seed, nx, ny)
        return torch.stack([ex.apply(s, x[f], case["adjoint"]) for f, s in enumerate(shifts)])
    if path in ("solve", "refactor_solve"):
        if seconds(nx, b, F, 1) > 15:
            return None
        ex = _Exact(case, seed, nx, ny)
        rhs = _block(case, seed, (F, n, k))
        w = _weights(case, seed, n)
        ws = 1.0 if w is None else torch.from_numpy(np.sqrt(w)).to(DEV)[:, None]
        adj = case["adjoint"]
        return torch.stack([ex.solve(s, rhs[f] * ws, True) / ws if adj
                            else ws * ex.solve(s, rhs[f] / ws) for f, s in enumerate(shifts)])
    if path == "resolvent":
        if seconds(nx, b, F, 2) > 15:
            return None
        ex = _Exact(case, seed, nx, ny)
        r = [_algorithm1(case, seed, ex, s, k, o)
             for s, o in zip(shifts, _seeds(seed, F))]
        return {m: torch.stack([t[m] for t in r]) for m in r[0]}
    if path == "batch":
        out = []
        for p in _batch_list(case, seed):
            if seconds(p["nx"], Q[case["kind"]] * p["ny"], 1, 2) > 3:
                out.append({m: None for m in ("sigma", "sigma_halko", "U", "V")})
                continue
            ex = _Exact(case, seed, p["nx"], p["ny"])
            out.append(_algorithm1(case, seed, ex, complex(p["shift"]), p["k"], p["seed"]))
        return out
    if seconds(nx, b, F, 2) > 15:
        return None
    fields = [torch.from_numpy(a).to(DEV).requires_grad_() for a in _fields(case, seed, nx, ny)]
    with torch.no_grad():
        ex = _Exact(case, seed, nx, ny, [f.detach() for f in fields])
        U, V, sg = _triplets(case, seed)
        w = _weights(case, seed, n)
        ws = 1.0 if w is None else torch.from_numpy(np.sqrt(w)).to(DEV)[:, None]
        pairs = []
        for f, s in enumerate(shifts):
            right = ex.solve(s, V[f, :, :J] / ws)
            left = ex.solve(s, U[f, :, :J] * ws, True)
            pairs.append((left, right))
    # d(sum sigma^2) = sum 2 sigma Re(left^H dL right): differentiate the
    # stencil entries contracted with the fixed vectors
    c = _stencil(case, ex.g, *fields)
    total = 0.0
    q = ex.q
    for f, (left, right) in enumerate(pairs):
        ls, rs = left.reshape(nx, ny, q, J), right.reshape(nx, ny, q, J)
        for ox in (-1, 0, 1):
            for oy in (-1, 0, 1):
                sh = _roll(_roll(rs, ox, 0), oy, 1)
                t = torch.einsum("xyaj,xycj,j->acxy", ls.conj(), sh,
                                 2.0 * sg[f, :J].to(torch.complex128)).real
                total = total + (c[ox + 1, oy + 1] * t).sum()
    g = torch.autograd.grad(total, fields, allow_unused=True)
    return torch.stack([torch.zeros(nx, ny, dtype=torch.float64, device=DEV) if a is None else a
                        for a in g])

"""Performance cases of the solver: what its users run, through the public entry points.

A case is one call sequence on one problem.  ``op`` says which:
  solve   a factored matrix and new right-hand sides: Factor.solve (and Factor.refine)
  step    a new matrix and its right-hand sides: Factor.factor, Factor.solve (and Factor.refine)
  graph   the same through Factor.factor_solve_graph (one CUDA graph, replayed)
  host    the same from host arrays to a host array: Factor.factor_solve_host
  batch   many independent problems through BatchGraph

``precision`` 0 is FP64 (eps_ID 1e-8), 1 is mixed (eps_ID 4e-7); a mixed factor is a
preconditioner, so every mixed case refines to the library's 1e-10 residual.  The problem
families are the repository's own (variable-coefficient diffusion, upwind convection-diffusion,
anisotropic convection-diffusion, Helmholtz at ten points per wavelength), generated here on the
GPU.  Grid sides are 16 * 2^k - 1, the sides the library takes.
"""
from __future__ import annotations

import math

import torch

from paper_2408_14193_gb300 import BatchGraph, Factor, NestedDissection

EPS = {0: 1e-8, 1: 4e-7}
SYMMETRIC = {"diffusion": 1, "helmholtz": 1, "convdiff": 0, "aniso": 0}
SIDES = (31, 63, 127, 255, 511, 1023)


def listed():
    return [
        # the smallest call: one more right-hand side for a small factored problem; launches
        # and their latency are all of it
        dict(name="solve_63_fp64", op="solve", kind="diffusion", nx=63, ny=63, nrhs=1, precision=0, refine=False),
        # a small ragged factorization (parameter studies on coarse grids)
        dict(name="step_127x63_fp64", op="step", kind="diffusion", nx=127, ny=63, nrhs=2, precision=0, refine=False),
        # time stepping on a factored mid-size operator, mixed precision, an odd count of
        # right-hand sides
        dict(name="solve_255_mixed", op="solve", kind="diffusion", nx=255, ny=255, nrhs=5, precision=1, refine=True),
        # a non-symmetric operator on a rectangular grid, refined
        dict(name="step_255x127_convdiff_fp64", op="step", kind="convdiff", nx=255, ny=127, nrhs=3, precision=0,
             refine=True),
        # the end-to-end call from page-locked host memory on an ordinary size, more right-hand
        # sides than one chunk of 16
        dict(name="host_511_mixed", op="host", kind="aniso", nx=511, ny=511, nrhs=17, precision=1, refine=True),
        # many small independent problems with one right-hand side each as one graph
        dict(name="batch_24_mixed", op="batch", kind="diffusion", nx=255, ny=255, nrhs=1, precision=1, refine=True,
             count=24),
        # the direct solve of a large factored problem, FP64, a full chunk of right-hand sides
        dict(name="solve_1023_fp64", op="solve", kind="diffusion", nx=1023, ny=1023, nrhs=16, precision=0,
             refine=False),
        # the headline: a new matrix of a million unknowns with 16 right-hand sides, mixed
        dict(name="step_1023_mixed", op="step", kind="diffusion", nx=1023, ny=1023, nrhs=16, precision=1, refine=True),
        # ... the same in the plain FP64 form
        dict(name="step_1023_fp64", op="step", kind="diffusion", nx=1023, ny=1023, nrhs=16, precision=0, refine=False),
        # a sequence of non-symmetric matrices in the same buffers, as one replayed graph
        dict(name="graph_1023_convdiff_mixed", op="graph", kind="convdiff", nx=1023, ny=1023, nrhs=4, precision=1,
             refine=True),
        # high-frequency Helmholtz with point sources: the largest ranks, FP64
        dict(name="step_1023_helmholtz_fp64", op="step", kind="helmholtz", nx=1023, ny=1023, nrhs=8, precision=0,
             refine=True),
    ]


def draw(rng):
    """One more case of the same ranges: sides 31 .. 1023 (mostly not square), 1 .. 20 right-hand
    sides spread over their logarithm, every operation, both precisions, every family."""
    op = rng.choice(["solve", "step", "step", "graph", "host", "batch"])
    nrhs = max(1, min(20, int(round(math.exp(rng.uniform(0.0, math.log(20.5)))))))
    if op == "batch":
        return dict(op=op, kind="diffusion", nx=rng.choice((63, 127, 255)), ny=rng.choice((63, 127, 255)), nrhs=1,
                    precision=1, refine=True, count=rng.randint(3, 24))
    kind = rng.choice(["diffusion", "diffusion", "convdiff", "aniso", "helmholtz"])
    if kind == "helmholtz":
        nx, ny = rng.choice(SIDES[1:5]), rng.choice(SIDES[1:5])
        return dict(op=op, kind=kind, nx=nx, ny=ny, nrhs=min(nrhs, 8), precision=0, refine=True)
    precision = rng.randint(0, 1)
    refine = precision == 1 or op == "graph" or rng.random() < 0.5
    return dict(op=op, kind=kind, nx=rng.choice(SIDES), ny=rng.choice(SIDES), nrhs=nrhs, precision=precision,
                refine=refine)


# ---------------------------------------------------------------- problems
def _field(gen, nx, ny, ell=0.05, var=1.0):
    """A zero-mean Gaussian random field of squared-exponential covariance on the
    (ny + 2) x (nx + 2) node lattice, by circulant embedding."""
    dev = gen.device
    mx, my = (1 << math.ceil(math.log2(2 * (n + 2))) for n in (nx, ny))

    def dist(m, h):
        i = torch.arange(m, device=dev, dtype=torch.float64)
        return torch.minimum(i, m - i) * h

    dx, dy = dist(mx, 1.0 / (nx + 1)), dist(my, 1.0 / (ny + 1))
    cov = var * torch.exp(-(dy[:, None] ** 2 + dx[None, :] ** 2) / (2 * ell**2))
    lam = torch.fft.fft2(cov).real
    lam = torch.where(lam > 1e-10 * lam.max(), lam, torch.zeros_like(lam))
    z = torch.randn((2, my, mx), generator=gen, device=dev, dtype=torch.float64)
    f = torch.fft.fft2(torch.sqrt(lam / (mx * my)) * torch.complex(z[0], z[1]))
    return f.real[: ny + 2, : nx + 2].contiguous()


def _stencil(kind, gen, nx, ny):
    """The five stencil weights (diag, west, east, south, north), each (ny, nx)."""
    hx, hy = 1.0 / (nx + 1), 1.0 / (ny + 1)
    one = torch.ones((ny, nx), device=gen.device, dtype=torch.float64)

    def faces(a1, a2):
        p1, p2 = a1[1:-1, 1:-1], a2[1:-1, 1:-1]
        return (-0.5 * (p1 + a1[1:-1, :-2]) / hx**2, -0.5 * (p1 + a1[1:-1, 2:]) / hx**2,
                -0.5 * (p2 + a2[:-2, 1:-1]) / hy**2, -0.5 * (p2 + a2[2:, 1:-1]) / hy**2)

    if kind == "diffusion":
        a = torch.exp(_field(gen, nx, ny))
        w, e, s, n = faces(a, a)
        return -(w + e + s + n), w, e, s, n
    if kind == "helmholtz":
        k0 = 2 * math.pi * (max(nx, ny) + 1) / 10
        g = _field(gen, nx, ny)[1:-1, 1:-1]
        k2 = k0**2 * (1 + 0.2 * g / g.abs().max())
        w, s = -one / hx**2, -one / hy**2
        return -2 * w - 2 * s - k2, w, w.clone(), s, s.clone()
    if kind == "aniso":
        w, e, s, n = faces(torch.exp(_field(gen, nx, ny)), 10 * torch.exp(_field(gen, nx, ny)))
    else:
        w, e, s, n = -one / hx**2, -one / hx**2, -one / hy**2, -one / hy**2
    theta = 2 * math.pi * float(torch.rand((), generator=gen, device=gen.device, dtype=torch.float64))
    bx, by = 50 * math.cos(theta), 50 * math.sin(theta)
    d = -(w + e + s + n) + abs(bx) / hx + abs(by) / hy      # first-order upwind convection
    w, e = (w - bx / hx, e) if bx > 0 else (w, e + bx / hx)
    s, n = (s - by / hy, n) if by > 0 else (s, n + by / hy)
    return d, w, e, s, n


def _csr(stencil, nx, ny):
    """CSR (int32, int32, float64) in natural order, columns increasing within a row."""
    d, w, e, s, n = stencil
    g = torch.arange(nx * ny, device=d.device).reshape(ny, nx)
    x, y = g % nx, torch.div(g, nx, rounding_mode="floor")
    keep = torch.stack([y > 0, x > 0, x >= 0, x < nx - 1, y < ny - 1], dim=-1)
    cols = torch.stack([g - nx, g - 1, g, g + 1, g + nx], dim=-1)
    vals = torch.stack([s, w, d, e, n], dim=-1)
    rowptr = torch.zeros(nx * ny + 1, dtype=torch.int32, device=d.device)
    rowptr[1:] = torch.cumsum(keep.sum(-1).reshape(-1), 0)
    return rowptr, cols[keep].to(torch.int32).contiguous(), vals[keep].contiguous()


def _rhs(kind, gen, nx, ny, nrhs):
    """(nrhs, N): standard normals, or for Helmholtz Gaussian point sources of width 2h."""
    dev = gen.device
    if kind != "helmholtz":
        return torch.randn((nrhs, nx * ny), generator=gen, device=dev, dtype=torch.float64)
    hx, hy = 1.0 / (nx + 1), 1.0 / (ny + 1)
    c = 0.1 + 0.8 * torch.rand((nrhs, 2), generator=gen, device=dev, dtype=torch.float64)
    xs = (torch.arange(nx, device=dev, dtype=torch.float64) + 1) * hx
    ys = (torch.arange(ny, device=dev, dtype=torch.float64) + 1) * hy
    w = 2 * (2 * max(hx, hy)) ** 2
    ex = torch.exp(-((xs[None, :] - c[:, :1]) ** 2) / w)
    ey = torch.exp(-((ys[None, :] - c[:, 1:]) ** 2) / w)
    return (ey[:, :, None] * ex[:, None, :]).reshape(nrhs, nx * ny).contiguous()


def _problems(case, seed):
    """[(nx, ny, stencil, B)]: one problem, or the batch's (sides cycling through the case's
    largest and the next smaller ones)."""
    gen = torch.Generator(device="cuda")
    out = []
    for i in range(case.get("count", 1)):
        gen.manual_seed(1_000_003 * int(seed) + i)
        nx, ny = case["nx"], case["ny"]
        if "count" in case:
            nx = max(63, ((nx + 1) >> (i % 3)) - 1)
            ny = max(63, ((ny + 1) >> (i % 3)) - 1)
        st = _stencil(case["kind"], gen, nx, ny)
        out.append((nx, ny, st, _rhs(case["kind"], gen, nx, ny, case["nrhs"])))
    return out


# ---------------------------------------------------------------- the calls
def prepare(case, seed):
    p = case["precision"]
    probs = _problems(case, seed)
    state = {"case": dict(case)}
    factors = [Factor(NestedDissection(nx, ny), eps_id=EPS[p], precision=p, symmetric=SYMMETRIC[case["kind"]])
               for nx, ny, _, _ in probs]
    csrs = [_csr(st, nx, ny) for nx, ny, st, _ in probs]
    Bs = [B for _, _, _, B in probs]
    if case["op"] == "batch":
        Xs = [torch.empty_like(B) for B in Bs]
        state.update(graph=BatchGraph(factors, csrs, Bs, Xs, nstreams=16, refine=True), X=Xs)
        return state
    f, csr, B = factors[0], csrs[0], Bs[0]
    state.update(f=f)
    if case["op"] == "host":
        pin = [t.cpu().pin_memory() for t in (*csr, B, torch.empty_like(B))]
        state.update(pin=pin, host=[t.numpy() for t in pin])
        return state
    state.update(csr=csr, B=B, X=torch.empty_like(B))
    if case["op"] == "solve":
        f.factor(*csr)
    return state


def run(state):
    case = state["case"]
    op = case["op"]
    if op == "batch":
        state["graph"].run()
        return state["X"]
    f = state["f"]
    if op == "host":
        rowptr, colind, val, B, X = state["host"]
        return f.factor_solve_host(rowptr, colind, val, B, refine=case["refine"], out=X)[0]
    B, X = state["B"], state["X"]
    if op == "graph":
        f.factor_solve_graph(*state["csr"], B, X)
        return X
    if op == "step":
        f.factor(*state["csr"])
    f.solve(B, X)
    if case["refine"]:
        f.refine(B, X)
    return X


def work(case):
    """Least traffic and arithmetic of one pass.  Per unknown: the matrix (5 entries of 12 bytes
    and a row pointer), each right-hand side read and each solution written; a solve reads the
    factor once (31 band values and about 22 of the levels per unknown).  Arithmetic: the leaf
    eliminations (band LU and 60 band solves, 0.89 MFLOP per 15 x 15 leaf) and about 4.5 kFLOP
    per unknown for the levels (several times that where Helmholtz ranks grow with the side),
    2 FLOP per stored factor value and right-hand side, 10 for a residual."""
    bytes_, flops = 0.0, 0.0
    for i in range(case.get("count", 1)):
        sx, sy = case["nx"] + 1, case["ny"] + 1
        if "count" in case:
            sx, sy = max(64, sx >> (i % 3)), max(64, sy >> (i % 3))
        n, nrhs = float((sx - 1) * (sy - 1)), case["nrhs"]
        bytes_ += n * (64.0 + 16.0 * nrhs)
        flops += n * nrhs * 106.0
        if case["refine"]:
            flops += n * nrhs * 10.0
        if case["op"] == "solve":
            bytes_ += n * 53.0 * (4 if case["precision"] else 8)
        else:
            level = 4.5e3 * (max(1.0, math.sqrt(sx * sy) / 64) if case["kind"] == "helmholtz" else 1.0)
            flops += n / 256.0 * 0.89e6 + n * level
    return {"bytes": bytes_, "flops": flops}


# ---------------------------------------------------------------- the same in 64 bits
def _direct(stencil, nx, ny, B):
    """Block elimination of the five-point matrix line by line (dense inverses of the line
    blocks), then two steps of iterative refinement."""
    d, w, e, s, n = stencil
    Bg = B.reshape(-1, ny, nx)
    if nx > ny:          # lines along the shorter side
        d, w, e, s, n = (t.T.contiguous() for t in (d, s, n, w, e))
        Bg = Bg.transpose(1, 2).contiguous()
    rows, m = d.shape
    inv = []
    for j in range(rows):
        S = torch.diag(d[j]) + torch.diag(w[j, 1:], -1) + torch.diag(e[j, :-1], 1)
        if j:
            S -= s[j][:, None] * inv[-1] * n[j - 1][None, :]
        inv.append(torch.linalg.inv(S))

    def solve(r):        # r: (nrhs, rows, m)
        y = [r[:, 0]]
        for j in range(1, rows):
            y.append(r[:, j] - (y[-1] @ inv[j - 1].T) * s[j])
        x = [y[-1] @ inv[-1].T]
        for j in range(rows - 2, -1, -1):
            x.append((y[j] - n[j] * x[-1]) @ inv[j].T)
        return torch.stack(x[::-1], 1)

    def residual(x):
        r = Bg - d * x
        r[:, :, 1:] -= w[:, 1:] * x[:, :, :-1]
        r[:, :, :-1] -= e[:, :-1] * x[:, :, 1:]
        r[:, 1:] -= s[1:] * x[:, :-1]
        r[:, :-1] -= n[:-1] * x[:, 1:]
        return r

    x = solve(Bg)
    for _ in range(2):
        x = x + solve(residual(x))
    if nx > ny:
        x = x.transpose(1, 2)
    return x.reshape(B.shape).contiguous()


def exact(case, seed):
    xs = [_direct(st, nx, ny, B) for nx, ny, st, B in _problems(case, seed)]
    if case["op"] == "batch":
        return xs
    return xs[0].cpu().numpy() if case["op"] == "host" else xs[0]

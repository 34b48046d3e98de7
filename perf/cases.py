"""Performance cases: the work a user of the library has it do.

Whole solves (FP64 and FP32 basis with FP64 refinement), differentiable
solve steps (forward, adjoint, value gradients), and the layers that the
row-partitioned solver and other callers drive one by one: a block
orthogonalisation, the matrix powers kernel, the Ritz pre-pass alone, and
the ingest of a matrix from host arrays.  Sizes are those of the five
synthetic workloads (workloads/generators.py), of the tests and of the
benchmark, from the 64 x 64 stencil to the 4.19M-row random band, with odd
and ragged ones between.

Inputs are made on the GPU from the seed alone.  Whole solves run to 1e-11
or 1e-12, so that x is fixed by the system and not by where the iteration
happened to stop.
"""
import math

import numpy as np
import torch

import paper_2303_08953_gb300 as sg
from paper_2303_08953_gb300.autograd import sparse_solve

DEV = "cuda:0"

SOLVE = dict(kind="solve", basis="scaled_newton", equilibrate="none")
STEP = dict(kind="step")


def listed():
    return [
        # the smallest system of the benchmark: 35 blocks of 10 columns, every
        # kernel a few microseconds, so launches and host round trips count
        dict(SOLVE, name="solve_stencil2d_64", matrix="stencil2d", nx=64, ny=64, nz=1,
             m=60, s=10, s_min=1, s_max=10, tol=1e-12, precision="fp64"),
        # restarted solve of a 3D convection-diffusion system with the step
        # size estimated: wide blocks, the orthogonalisation dominates
        dict(SOLVE, name="solve_convdiff3d_128", matrix="convdiff3d", nx=128, ny=128, nz=128,
             m=240, s=0, s_min=20, s_max=120, tol=1e-12, precision="fp64"),
        # the same system with the FP32 basis inside FP64 refinement
        dict(SOLVE, name="solve_convdiff3d_128_fp32ir", matrix="convdiff3d", nx=128, ny=128, nz=128,
             m=240, s=0, s_min=20, s_max=120, tol=1e-12, precision="fp32_ir"),
        # the headline workload: unstructured matrix of 4.19M rows and 105M
        # entries, few Krylov columns, so the 120-step Ritz pre-pass dominates
        dict(SOLVE, name="solve_randband_4M", matrix="randband", nx=4194304, ny=1, nz=1,
             m=120, s=0, s_min=1, s_max=120, tol=1e-12, precision="fp64"),
        # an ordinary solve on a ragged grid of odd sides, FP64
        dict(SOLVE, name="solve_convdiff3d_61x47x53", matrix="convdiff3d", nx=61, ny=47, nz=53,
             m=120, s=0, s_min=8, s_max=60, tol=1e-12, precision="fp64"),
        # one training step of a model with a sparse solve inside: new values,
        # forward solve, adjoint solve on the transpose, value gradients
        dict(STEP, name="step_randband_1M_fp32ir", matrix="randband", nx=1000003, ny=1, nz=1,
             m=120, s=0, s_min=1, s_max=60, tol=1e-11, precision="fp32_ir"),
        # the same step on a small 2D grid in FP64
        dict(STEP, name="step_stencil2d_255x257", matrix="stencil2d", nx=255, ny=257, nz=1,
             m=60, s=10, s_min=1, s_max=10, tol=1e-12, precision="fp64"),
        # one block orthogonalised against the basis (second block of the
        # 128^3 system): projection, update, Gram, triangular product
        dict(kind="ortho", name="ortho_fp64_2M_121x120", n=2097152, i=121, s=120,
             precision="fp64"),
        # a narrow block of a short cycle on a small ragged system
        dict(kind="ortho", name="ortho_fp64_65535_41x10", n=65535, i=41, s=10,
             precision="fp64"),
        # the FP32 basis on the 192^3 system (step size 60)
        dict(kind="ortho", name="ortho_fp32_7M_121x60", n=7077888, i=121, s=60,
             precision="fp32"),
        # the matrix powers kernel alone, 192^3 grid
        dict(kind="mpk", name="mpk_convdiff3d_192_s20", matrix="convdiff3d", nx=192, ny=192, nz=192,
             s=20),
        # a matrix handed over from host arrays, then one residual with it
        dict(kind="ingest", name="ingest_randband_262144", matrix="randband", nx=262144, ny=1, nz=1),
    ]


def _log_uniform(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _draw_matrix(rng, scale=1.0):
    matrix = rng.choice(["stencil2d", "convdiff3d", "randband"])
    if matrix == "stencil2d":
        a = _log_uniform(rng, 32, 400)
        return dict(matrix=matrix, nx=a, ny=max(16, int(a * rng.uniform(0.6, 1.6))), nz=1)
    if matrix == "convdiff3d":
        a = _log_uniform(rng, 14, 110)
        return dict(matrix=matrix, nx=a, ny=max(9, int(a * rng.uniform(0.7, 1.15))),
                    nz=max(9, int(a * rng.uniform(0.7, 1.15))))
    return dict(matrix=matrix, nx=_log_uniform(rng, 5000, 3_000_000 * scale), ny=1, nz=1)


def draw(rng):
    kind = rng.choice(["solve", "solve", "solve", "step", "ortho", "ortho", "mpk", "prepass",
                       "ingest"])
    if kind in ("solve", "step"):
        c = dict(SOLVE if kind == "solve" else STEP, **_draw_matrix(rng, 1.0 if kind == "solve" else 0.4))
        c["m"] = rng.randint(48, 240)
        if rng.random() < 0.4:
            c["s"], c["s_min"], c["s_max"] = rng.randint(4, 16), 1, 16
        else:
            c["s"], c["s_min"], c["s_max"] = 0, rng.randint(1, 8), rng.randint(20, min(120, c["m"]))
        c["precision"] = rng.choice(["fp64", "fp32_ir"])
        c["tol"] = 1e-12 if c["precision"] == "fp64" else 1e-11
        return c
    if kind == "ortho":
        n = _log_uniform(rng, 3000, 2_000_000)
        return dict(kind=kind, n=n, i=_log_uniform(rng, 1, 240), s=_log_uniform(rng, 2, 120),
                    precision=rng.choice(["fp64", "fp32"]))
    c = dict(kind=kind, **_draw_matrix(rng, 0.3))
    if kind == "mpk":
        c["s"] = rng.randint(4, 60)
    if kind == "prepass":
        # the FP64 pre-pass of a fixed step size (longer ones amplify rounding
        # through the Krylov basis, and are part of the whole solves)
        c["k"] = rng.randint(3, 6)
    return c


# ------------------------------------------------------------------ inputs
def _gen(seed):
    return torch.Generator(device=DEV).manual_seed(1_000_003 * (int(seed) % 1_000_000_007) + 17)


def _uniform(n, g, lo=-1.0, hi=1.0):
    return torch.rand(n, generator=g, device=DEV, dtype=torch.float64) * (hi - lo) + lo


def _grid(nx, ny, nz, off, diag):
    """CSR (int32, int32, float64) of a constant stencil on a box grid,
    x fastest; off: (dx, dy, dz) -> value in increasing column order."""
    n = nx * ny * nz
    i = torch.arange(n, device=DEV)
    ix, iy, iz = i % nx, (i // nx) % ny, i // (nx * ny)
    cols, ok, vals = [], [], []
    for (dx, dy, dz), v in off:
        cols.append(i + dx + nx * dy + nx * ny * dz)
        ok.append((ix + dx >= 0) & (ix + dx < nx) & (iy + dy >= 0) & (iy + dy < ny)
                  & (iz + dz >= 0) & (iz + dz < nz))
        vals.append(diag if v is None else v)
    ok = torch.stack(ok, 1)
    rowptr = torch.zeros(n + 1, dtype=torch.int64, device=DEV)
    torch.cumsum(ok.sum(1), 0, out=rowptr[1:])
    colind = torch.stack(cols, 1)[ok].to(torch.int32)
    val = torch.tensor(vals, dtype=torch.float64, device=DEV).expand(n, len(vals))[ok]
    return rowptr.to(torch.int32), colind, val.contiguous()


def _randband(n, g, k=24, band=4096, dominance=1.1):
    """n rows with k distinct off-diagonal columns within a band around the
    diagonal, N(0, 1) values, a dominant diagonal; columns sorted."""
    band = min(band, (n - 2) // 3)
    col = torch.empty(n, k + 1, dtype=torch.int32, device=DEV)
    val = torch.empty(n, k + 1, dtype=torch.float64, device=DEV)
    t = torch.arange(k + 1, device=DEV, dtype=torch.int32)
    edge = (torch.arange(k + 1, device=DEV) * (2 * band)) // k
    width = (edge[1:] - edge[:-1]).to(torch.float32)
    for a in range(0, n, 1 << 20):
        b = min(n, a + (1 << 20))
        i = torch.arange(a, b, device=DEV, dtype=torch.int32)[:, None]
        lo = (i - band).clamp(0, n - 1 - 2 * band)
        u = torch.rand(b - a, k, generator=g, device=DEV)
        c = lo + edge[:-1].to(torch.int32) + torch.minimum((u * width).floor(), width - 1).to(torch.int32)
        c = c + (c >= i).to(torch.int32)          # skip the diagonal
        p = (c < i).sum(1, keepdim=True, dtype=torch.int32)
        v = torch.randn(b - a, k, generator=g, device=DEV, dtype=torch.float64)
        before = (t < p)
        left = torch.nn.functional.pad(c, (0, 1))
        right = torch.nn.functional.pad(c, (1, 0))
        col[a:b] = torch.where(before, left, torch.where(t == p, i, right))
        d = dominance * v.abs().sum(1, keepdim=True)
        val[a:b] = torch.where(before, torch.nn.functional.pad(v, (0, 1)),
                               torch.where(t == p, d, torch.nn.functional.pad(v, (1, 0))))
    rowptr = (torch.arange(n + 1, device=DEV) * (k + 1)).to(torch.int32)
    return rowptr, col.reshape(-1), val.reshape(-1)


def _matrix(case, g, vary):
    nx, ny, nz = case["nx"], case["ny"], case["nz"]
    if case["matrix"] == "randband":
        return _randband(nx, g)
    if case["matrix"] == "stencil2d":
        off = [((0, -1, 0), -1.1), ((-1, 0, 0), -1.1), ((0, 0, 0), None), ((1, 0, 0), -0.9),
               ((0, 1, 0), -0.9)]
        rp, ci, v = _grid(nx, ny, nz, off, 4.0)
    else:
        off = [((0, 0, -1), -1.2), ((0, -1, 0), -1.2), ((-1, 0, 0), -1.2), ((0, 0, 0), None),
               ((1, 0, 0), -0.8), ((0, 1, 0), -0.8), ((0, 0, 1), -0.8)]
        rp, ci, v = _grid(nx, ny, nz, off, 6.0)
    if vary:   # a learned matrix: off-diagonal values differ a little from entry to entry
        v = torch.where(v < 0, v * _uniform(v.numel(), g, 0.9, 1.0), v)
    return rp, ci, v


def _rows(rp):
    n = rp.numel() - 1
    return torch.repeat_interleave(torch.arange(n, device=DEV), (rp[1:] - rp[:-1]).long())


def _times(rp, ci, v, x):
    """A x in plain torch."""
    n = rp.numel() - 1
    y = torch.empty(n, dtype=torch.float64, device=DEV)
    step = 1 << 20
    for a in range(0, n, step):
        b = min(n, a + step)
        p, q = int(rp[a]), int(rp[b])
        y[a:b] = torch.segment_reduce(v[p:q] * x[ci[p:q].long()], "sum",
                                      lengths=(rp[a + 1:b + 1] - rp[a:b]).long())
    return y


def _times_t(rp, ci, v, lam):
    """A^T lam in plain torch."""
    out = torch.zeros_like(lam)
    out.index_add_(0, ci.long(), v * lam[_rows(rp)])
    return out


def _solver(rp, ci, v):
    s = sg.Solver(0)
    torch.cuda.current_stream().synchronize()   # the ingest reads on the library's own stream
    s.analyze(rp, ci, v)
    return s


def _blocks(case, g):
    """A basis Q (near-orthonormal columns) and a block X that lies mostly in
    its span, as the matrix powers kernel hands it over; columns of X fall
    off in size."""
    n, i, s = case["n"], case["i"], case["s"]
    dt = torch.float64 if case["precision"] == "fp64" else torch.float32
    ld = (n + 31) // 32 * 32
    Q = torch.zeros(i, ld, dtype=dt, device=DEV)
    X = torch.zeros(s, ld, dtype=dt, device=DEV)
    for k in range(i):
        Q[k, :n] = torch.randn(n, generator=g, device=DEV, dtype=dt) / math.sqrt(n)
    for k in range(s):
        X[k, :n] = torch.randn(n, generator=g, device=DEV, dtype=dt) * (0.97 ** k / math.sqrt(n))
        X[k, :n] += 3.0 * Q[(5 * k + 2) % i, :n]
    # an upper triangular factor of moderate size, as a Cholesky inverse
    Z = torch.triu(0.1 * torch.randn(s, s, generator=g, device=DEV, dtype=torch.float64))
    Z += torch.diag(1.0 + _uniform(s, g, 0.0, 0.5))
    return Q, X, Z.t().contiguous()


def _shifts(case, g):
    """Leja-like real shifts and scales in the range of the spectrum."""
    s = case["s"]
    th = _uniform(s, g, 2.0, 10.0).cpu().numpy()
    return th, np.full(s, 3.0)


def prepare(case, seed):
    g = _gen(seed)
    kind = case["kind"]
    st = {"case": dict(case)}
    if kind == "ortho":
        Q, X, Zt = _blocks(case, g)
        st.update(Q=Q, X=X, Z=Zt, work=torch.empty_like(X), out=torch.zeros_like(X),
                  solver=sg.Solver(0))
        return st
    rp, ci, v = _matrix(case, g, kind == "step")
    n = rp.numel() - 1
    xs = _uniform(n, g)
    if kind == "solve":
        st.update(solver=_solver(rp, ci, v), b=_times(rp, ci, v, xs))
    elif kind == "step":
        lam = _uniform(n, g)
        b = _times(rp, ci, v, xs)
        st.update(solver=_solver(rp, ci, v), target=xs - _times_t(rp, ci, v, lam),
                  values=v.requires_grad_(True), b=b.requires_grad_(True))
    elif kind == "mpk":
        th, gm = _shifts(case, g)
        st.update(solver=_solver(rp, ci, v), q=xs / torch.linalg.vector_norm(xs), theta=th, gamma=gm)
    elif kind == "prepass":
        st.update(solver=_solver(rp, ci, v), q=xs / torch.linalg.vector_norm(xs))
    else:   # ingest: host arrays, as read from a file
        st.update(solver=sg.Solver(0), rowptr=rp.cpu().numpy(), colind=ci.cpu().numpy(),
                  val=v.cpu().numpy(), x=xs, b=_uniform(n, g))
    return st


def _options(case):
    o = dict(m=case["m"], s=case["s"], s_min=case["s_min"], s_max=case["s_max"], tol=case["tol"],
             precision=case["precision"])
    if case["kind"] == "solve":
        o.update(basis=case["basis"], equilibrate=case["equilibrate"])
    return o


def run(state):
    case, solver = state["case"], state["solver"]
    kind = case["kind"]
    if kind == "solve":
        x, _ = solver.solve(state["b"], **_options(case))
        return x
    if kind == "step":
        values, b = state["values"], state["b"]
        x = sparse_solve(values, b, solver, **_options(case))
        loss = 0.5 * (x - state["target"]).square().sum()
        gv, gb = torch.autograd.grad(loss, (values, b))
        return x.detach(), gv, gb
    if kind == "ortho":
        # one pass of the block Gram-Schmidt step on a copy of the block (the
        # caller keeps the powers): W = Q^T X, X -= Q W, G = X^T X, X Z
        Q, X, n = state["Q"], state["work"], case["n"]
        X.copy_(state["X"])
        solver.n = n
        if case["precision"] == "fp64":
            W = solver.block_dot(Q, X)
            solver.block_update(Q, W, X)
            G = solver.block_dot(X, X, sym=True)
            Y = solver.block_update(X, state["Z"], state["out"], alpha=1.0, beta=0.0, upper=True)
        else:
            W = solver.block_dot32(Q, X)
            solver.block_update32(Q, W, X)
            G = solver.block_dot32(X, X, sym=True)
            Y = solver.block_update32(X, state["Z"], state["out"], alpha=1.0, beta=0.0, upper=True)
            W, G = W.float(), G.float()   # their accuracy is FP32's: a caller keeps them so
        return W, X, G, Y
    if kind == "mpk":
        return solver.mpk(state["q"], case["s"], state["theta"], state["gamma"])
    if kind == "prepass":
        H, steps = solver.arnoldi(state["q"], case["k"])
        return H, steps
    solver.analyze(state["rowptr"], state["colind"], state["val"])
    return solver.residual(state["b"], state["x"])


# ------------------------------------------------------------- what it needs
def _size(case):
    nx, ny, nz = case["nx"], case["ny"], case["nz"]
    n = nx * ny * nz
    if case["matrix"] == "randband":
        return n, 25 * n
    d = 5 if case["matrix"] == "stencil2d" else 7
    edge = nx * ny + nx * nz + ny * nz if d == 7 else nx + ny
    return n, d * n - 2 * edge


def _columns(case):
    """Krylov columns that the system takes to its tolerance, about (it is
    set by the spectrum, hardly by the size)."""
    return {"randband": 27, "stencil2d": 420, "convdiff3d": 750}[case["matrix"]] \
        if case["nx"] > 60 or case["matrix"] == "randband" else 300


def _solve_work(case, prepass=True):
    """The method's own work: a k-step Arnoldi pre-pass (the basis read once
    per step), then per column one product with A and two projections on the
    basis so far."""
    n, nnz = _size(case)
    w = 8 if case["precision"] == "fp64" else 4
    idx = 4
    k = min(case["s"] if case["s"] > 0 else case["s_max"], case["m"]) if prepass else 0
    cols = _columns(case)
    cyc, mean = max(1, cols // case["m"]), min(cols, case["m"]) / 2
    a = (w + idx) * nnz + 2 * w * n
    s = case["s"] if case["s"] > 0 else max(case["s_min"], 16)
    by = k * a + w * n * k * (k + 3) / 2 + cols * a + cols / s * w * n * (2 * mean + 6 * s) \
        + cyc * (w * n * min(cols, case["m"]) + (8 + idx) * nnz)
    fl = 2.0 * nnz * (k + cols) + 4.0 * n * k * (k + 1) / 2 + cols * n * (8 * mean + 6.0 * s)
    return by, fl


def work(case):
    kind = case["kind"]
    if kind == "solve":
        by, fl = _solve_work(case)
    elif kind == "step":
        n, nnz = _size(case)
        by, fl = _solve_work(case)
        by2, fl2 = _solve_work(case, prepass=False)
        by, fl = by + by2 + 3 * 12 * nnz + 8 * nnz, fl + fl2 + nnz
    elif kind == "ortho":
        n, i, s = case["n"], case["i"], case["s"]
        w = 8 if case["precision"] == "fp64" else 4
        by = float(w) * n * (i + 3 * s) + 8.0 * (i * s + 2 * s * s)
        fl = n * (4.0 * i * s + 2.0 * s * (s + 1))
    elif kind == "mpk":
        n, nnz = _size(case)
        by, fl = 12.0 * nnz + 8.0 * n * (case["s"] + 1), 2.0 * nnz * case["s"]
    elif kind == "prepass":
        n, nnz = _size(case)
        k = case["k"]
        by, fl = 12.0 * nnz + 8.0 * n, 2.0 * nnz * k + 4.0 * n * k * (k + 1) / 2
    else:
        n, nnz = _size(case)
        by, fl = 12.0 * nnz + 28.0 * n, 2.0 * nnz
    return {"bytes": float(by), "flops": float(fl)}


# ------------------------------------------------------------------- 64 bits
def exact(case, seed):
    g = _gen(seed)
    kind = case["kind"]
    if kind == "ortho":
        Q, X, Zt = _blocks(case, g)
        n, s = case["n"], case["s"]
        W = torch.zeros(s, case["i"], dtype=torch.float64, device=DEV)
        G = torch.zeros(s, s, dtype=torch.float64, device=DEV)
        Xo = torch.zeros_like(X, dtype=torch.float64)
        Y = torch.zeros_like(Xo)
        step = 1 << 18
        for a in range(0, n, step):
            W += X[:, a:a + step].double() @ Q[:, a:a + step].double().t()
        for a in range(0, n, step):
            b = min(n, a + step)
            x = X[:, a:b].double() - W @ Q[:, a:b].double()
            Xo[:, a:b] = x
            G += x @ x.t()
            Y[:, a:b] = Zt @ x
        return W, Xo, G, Y
    rp, ci, v = _matrix(case, g, kind == "step")
    n = rp.numel() - 1
    xs = _uniform(n, g)
    if kind == "solve":
        return xs     # b was formed from it
    if kind == "step":
        lam = _uniform(n, g)
        return xs, -lam[_rows(rp)] * xs[ci.long()], lam
    if kind == "mpk":
        th, gm = _shifts(case, g)
        V = torch.empty(case["s"] + 1, n, dtype=torch.float64, device=DEV)
        V[0] = xs / torch.linalg.vector_norm(xs)
        for j in range(case["s"]):
            V[j + 1] = (_times(rp, ci, v, V[j]) - th[j] * V[j]) / gm[j]
        return V
    if kind == "prepass":
        k = case["k"]
        H = np.zeros((k + 1, k))
        V = [xs / torch.linalg.vector_norm(xs)]
        for j in range(k):
            w = _times(rp, ci, v, V[j])
            for _ in range(2):   # reorthogonalised
                for r in range(j + 1):
                    h = float(V[r] @ w)
                    H[r, j] += h
                    w = w - h * V[r]
            H[j + 1, j] = float(torch.linalg.vector_norm(w))
            V.append(w / H[j + 1, j])
        return H, None
    return _uniform(n, g) - _times(rp, ci, v, xs)

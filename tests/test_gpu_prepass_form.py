"""The FP64 pre-pass on systems whose unknowns have different scales.  Its
fixed-point form holds a vector to the largest entry of a block of rows, so it
may only run where the rows of A are of like size; elsewhere each entry has to
keep FP64's own precision.  H is compared with extended precision (numpy's
long double), relative to the column's largest entry, at 16 times the error
of the same MGS in numpy's FP64 (another summation order) plus 64 u."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA device", allow_module_level=True)

import paper_2303_08953_gb300 as sg  # noqa: E402

U = 2.0 ** -53


@pytest.fixture(scope="module")
def solver():
    s = sg.Solver(0)
    yield s
    s.close()


def _scaled(A, left, right):
    rows = np.repeat(np.arange(A.n), np.diff(A.rowptr))
    return W.CSR(A.n, A.rowptr, A.colind, A.val * left[rows] * right[A.colind])


def _mgs(A, q, k, dt):
    val, V, H = A.val.astype(dt), [q.astype(dt)], np.zeros((k + 1, k), dt)
    for j in range(k):
        w = np.add.reduceat(val * V[j][A.colind], A.rowptr[:-1])
        for i in range(j + 1):
            H[i, j] = np.sum(V[i] * w)
            w = w - H[i, j] * V[i]
        H[j + 1, j] = np.sqrt(np.sum(w * w))
        V.append(w / H[j + 1, j])
    return H


def _error(H, R, k):
    return max(float((np.abs(H[:j + 2, j] - R[:j + 2, j]).max() / np.abs(R[:j + 2, j]).max()))
               for j in range(k))


def _check(A, q, k, H, steps):
    assert steps == k
    R = _mgs(A, q, k, np.longdouble)
    own = _error(_mgs(A, q, k, np.float64), R, k)
    got = _error(H[:k + 1, :k], R, k)
    assert got <= 16 * own + 64 * U, (got, own)


def _arnoldi(solver, q, k):
    return solver.arnoldi(torch.as_tensor(q, dtype=torch.float64, device="cuda:0"), k)


# D B D^-1: neighbouring unknowns 2^e apart, and unknowns of random scales;
# one CTA and several, rows odd in number
@pytest.mark.parametrize("nx,ny,k", [(32, 32, 12), (61, 53, 8), (211, 97, 6)])
@pytest.mark.parametrize("how,e", [("alternating", 30), ("alternating", 40), ("random", 8),
                                   ("random", 33), ("random", 50), ("one unknown", 34)])
def test_unknowns_of_different_scales(solver, nx, ny, k, how, e):
    A = W.stencil2d(nx, ny)
    rng = np.random.default_rng(nx + e)
    if how == "alternating":
        d = 2.0 ** (-e * (np.arange(A.n) % 2))
    elif how == "random":
        d = 2.0 ** rng.integers(0, e + 1, A.n)
    else:
        d = np.ones(A.n)
        d[A.n // 3] = 2.0 ** -e
    q = d * rng.standard_normal(A.n)
    q /= np.linalg.norm(q)
    A = _scaled(A, d, 1.0 / d)
    solver.analyze_csr(A)
    _check(A, q, k, *_arnoldi(solver, q, k))


def test_the_form_follows_the_values(solver):
    """The same pattern and storage with even rows, then graded ones, then
    even ones again: the form (and the captured launches) must follow."""
    A = W.stencil2d(57, 43)
    rng = np.random.default_rng(1)
    d = 2.0 ** rng.integers(0, 41, A.n)
    G = _scaled(A, d, 1.0 / d)
    q = rng.standard_normal(A.n)
    q /= np.linalg.norm(q)
    qd = d * q
    qd /= np.linalg.norm(qd)
    solver.analyze_csr(A)
    first = _arnoldi(solver, q, 7)
    _check(A, q, 7, *first)
    solver.update_values(torch.as_tensor(G.val, device="cuda:0"))
    _check(G, qd, 7, *_arnoldi(solver, qd, 7))
    solver.update_values(torch.as_tensor(A.val, device="cuda:0"))
    again = _arnoldi(solver, q, 7)
    assert np.array_equal(first[0], again[0])


def test_uneven_pattern_with_graded_rows(solver):
    """Rows of uneven length and scale (sorted-window storage)."""
    n, k = 5003, 6
    rng = np.random.default_rng(4)
    ln = rng.integers(4, 14, n)
    ptr = np.zeros(n + 1, np.int32)
    np.cumsum(ln, out=ptr[1:])
    start = np.minimum(np.arange(n), n - ln)
    cols = (np.repeat(start, ln) + np.arange(ptr[-1]) - np.repeat(ptr[:-1], ln)).astype(np.int32)
    d = 2.0 ** rng.integers(0, 36, n)
    A = _scaled(W.CSR(n, ptr, cols, rng.uniform(0.5, 1.0, ptr[-1])), d, 1.0 / d)
    q = d * rng.standard_normal(n)
    q /= np.linalg.norm(q)
    solver.analyze_csr(A)
    _check(A, q, k, *_arnoldi(solver, q, k))


def test_even_rows_whose_product_vanishes(solver):
    """Even rows (the fixed-point form), but w = A v_j is zero over the CTAs
    of the second half while v_j is not, so that w's range has to grow with
    every projection there."""
    n, k = 9001, 6
    half = n // 2
    rows = np.arange(n)
    cols = np.where(rows < half, rows, half - 1).astype(np.int32)
    vals = np.where(rows < half, 1.0 + rows / n, 1.0)
    A = W.CSR(n, np.arange(n + 1, dtype=np.int32), cols, vals)
    q = np.random.default_rng(3).uniform(0.5, 1.0, n)
    q[half - 1] = 0.0
    q /= np.linalg.norm(q)
    solver.analyze_csr(A)
    _check(A, q, k, *_arnoldi(solver, q, k))


# A CTA's rows end inside a warp's batch: 1024-row CTAs hold 512 pairs of
# rows, 4 pairs a thread and batch, so the last batch of the last CTA leaves
# lanes of a warp idle for these row counts (and a whole batch precedes it
# from 4096 rows a CTA on: 152 x 4096 rows and more)
@pytest.mark.parametrize("n", [37, 101, 1024 + 75, 3 * 1024 + 333, 700_001, 1_400_321])
def test_a_batch_that_ends_inside_a_warp(solver, n):
    i = np.arange(n)
    ptr = np.concatenate([[0], np.cumsum(np.where(i + 1 < n, 2, 1))]).astype(np.int32)
    cols = np.empty(ptr[-1], np.int32)
    vals = np.empty(ptr[-1])
    cols[ptr[:-1]] = i
    vals[ptr[:-1]] = 2.0 + (i % 7) / 7.0
    cols[ptr[:-2] + 1] = i[1:]
    vals[ptr[:-2] + 1] = -1.0
    q = np.cos(0.37 * i) + 0.5
    q /= np.linalg.norm(q)
    A = W.CSR(n, ptr, cols, vals)
    solver.analyze_csr(A)
    _check(A, q, 5, *_arnoldi(solver, q, 5))

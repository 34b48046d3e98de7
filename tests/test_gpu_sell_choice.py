"""The storage that an analysed pattern gets: SELL-32 with the rows in order or
sorted within windows of 1024, by the entries each would hold, or CSR.  The
entries with sorted rows come from the lengths' counts, so every kind of
length is here, and a pattern that ends in CSR costs one kernel."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA device", allow_module_level=True)

import paper_2303_08953_gb300 as sg  # noqa: E402


@pytest.fixture(scope="module")
def solver():
    s = sg.Solver(0)
    yield s
    s.close()


def _lengths(kind, n):
    rng = np.random.default_rng(n)
    i = np.arange(n)
    return {
        "even": lambda: np.full(n, 9),
        "uneven": lambda: rng.integers(4, 14, n),
        "a long row in 64": lambda: np.where(i % 64 == 0, 200, 5),
        "two kinds": lambda: np.where(i % 2 == 0, 40, 3),
        "some empty": lambda: np.where(rng.random(n) < 0.5, 0, 17),
        "1022 to 1026": lambda: rng.integers(1022, 1027, n),
        "few very long": lambda: np.where(i % 500 == 7, 1500, 6),
        "many very long": lambda: np.where(i % 16 < 3, 1100 + i % 16, 2),
        "half very long": lambda: np.where(i % 2 == 0, 1023 + (i // 2) % 3 * 400, 8),
    }[kind]()


def _slices(ln):
    p = np.zeros((ln.size + 31) // 32 * 32, np.int64)
    p[:ln.size] = ln
    return 32 * p.reshape(-1, 32).max(1).sum()


def _expected(ln):
    nnz, nsl = int(ln.sum()), (ln.size + 31) // 32
    srt = np.concatenate([np.sort(ln[a:a + 1024])[::-1] for a in range(0, ln.size, 1024)])
    for total in (_slices(ln), _slices(srt)):
        if total <= nnz + nnz // 5 + 32 * nsl:
            return True, int(total)
    return False, nnz


def _matrix(ln):
    n = ln.size
    ptr = np.zeros(n + 1, np.int64)
    np.cumsum(ln, out=ptr[1:])
    start = np.minimum(np.arange(n), n - ln)
    cols = np.repeat(start, ln) + np.arange(ptr[-1]) - np.repeat(ptr[:-1], ln)
    rng = np.random.default_rng(0)
    return W.CSR(n, ptr.astype(np.int32), cols.astype(np.int32), rng.uniform(0.5, 1.0, ptr[-1]))


@pytest.mark.parametrize("n", [2049, 3000, 5120])
@pytest.mark.parametrize("kind", ["even", "uneven", "a long row in 64", "two kinds", "some empty",
                                  "1022 to 1026", "few very long", "many very long",
                                  "half very long"])
def test_storage(solver, kind, n):
    ln = np.minimum(_lengths(kind, n), n)
    A = _matrix(ln)
    solver.analyze_csr(A)
    assert tuple(solver.matrix_info()) == _expected(ln)
    x = np.random.default_rng(1).standard_normal(n)
    b = np.zeros(n)
    r = solver.residual(torch.as_tensor(b, device="cuda:0"), torch.as_tensor(x, device="cuda:0"))
    rows = np.repeat(np.arange(n), ln)
    ref = np.bincount(rows, A.val * x[A.colind], minlength=n)
    mag = np.bincount(rows, np.abs(A.val * x[A.colind]), minlength=n)
    assert np.all(np.abs(-r.cpu().numpy() - ref) <= (ln + 2) * 2.0 ** -53 * mag)


def test_a_pattern_that_ends_in_csr_costs_one_kernel(solver):
    def launches(A):
        before = sg.kernel_launches()
        solver.analyze_csr(A)
        return sg.kernel_launches() - before
    n = 70_000
    checks = launches(W.CSR(n, np.zeros(n + 1, np.int32), np.zeros(0, np.int32), np.zeros(0)))
    ln = _lengths("a long row in 64", n)
    assert launches(_matrix(ln)) == checks + 1
    assert not solver.matrix_info()[0]


def _uneven_diagonal(n, seed):
    """Uneven rows with a dominant diagonal (sorted windows), columns sorted."""
    rng = np.random.default_rng(seed)
    ln = rng.integers(3, 30, n)
    ptr = np.zeros(n + 1, np.int64)
    np.cumsum(ln, out=ptr[1:])
    cols = np.concatenate([np.sort(np.append(i, rng.choice(np.delete(np.arange(max(0, i - 60),
                           min(n, i + 61)), min(i, 60)), l - 1, replace=False)))
                           for i, l in zip(range(n), ln)])
    vals = rng.uniform(-1.0, 1.0, ptr[-1])
    rows = np.repeat(np.arange(n), ln)
    vals[cols == rows] = 1.5 * ln
    return W.CSR(n, ptr.astype(np.int32), cols.astype(np.int32), vals)


def test_sorted_rows_with_column_equilibration(solver):
    """A D_c shares A's row order: the solution to 1e-11 of the residual, for
    columns of sizes up to 2^12 apart (diagonally dominant rows, so x is
    within 1e-9 of the one b was formed from)."""
    A = _uneven_diagonal(4133, 1)
    d = 2.0 ** np.random.default_rng(2).integers(0, 13, A.n)
    A = W.CSR(A.n, A.rowptr, A.colind, A.val * d[A.colind])
    rows = np.repeat(np.arange(A.n), np.diff(A.rowptr))
    x = np.random.default_rng(3).uniform(-1, 1, A.n) / d
    b = np.bincount(rows, A.val * x[A.colind], minlength=A.n)
    solver.analyze_csr(A)
    sell, stored = solver.matrix_info()
    in_order = _slices(np.diff(A.rowptr))
    assert sell and stored < in_order
    got, info = solver.solve(torch.as_tensor(b, device="cuda:0"), m=60, s=6, tol=1e-12,
                             equilibrate="column")
    assert info.converged
    assert np.linalg.norm((got.cpu().numpy() - x) * d) <= 1e-9 * np.linalg.norm(x * d)


def test_sorted_rows_of_a_row_block(solver):
    """A row block in local numbering (more columns than rows, unsorted)."""
    A = _uneven_diagonal(3000, 4)
    lo, hi = 500, 2600
    p, q = A.rowptr[lo], A.rowptr[hi]
    rp = (A.rowptr[lo:hi + 1] - p).astype(np.int32)
    local, halo = sg.halo_plan(rp, A.colind[p:q], lo, hi)
    solver.analyze_rows(rp, local, A.val[p:q], hi - lo + halo.size)
    x = np.random.default_rng(5).standard_normal(A.n)
    xl = np.concatenate([x[lo:hi], x[halo]])
    y = solver.spmv_newton(torch.as_tensor(xl, device="cuda:0"), theta=0.5, gamma=2.0)
    rows = np.repeat(np.arange(hi - lo), np.diff(rp))
    prod = A.val[p:q] * x[A.colind[p:q]]
    ref = (np.bincount(rows, prod, minlength=hi - lo) - 0.5 * x[lo:hi]) / 2.0
    mag = np.bincount(rows, np.abs(prod), minlength=hi - lo) + np.abs(x[lo:hi])
    got = y.cpu().numpy()[:hi - lo]
    assert np.all(np.abs(got - ref) <= 40 * 2.0 ** -53 * mag)
    assert solver.matrix_info()[0]

"""Matrices with rows of uneven length: SELL-32 with the rows sorted inside
windows (products, residual, value updates, pre-pass), and the transpose
built from places and sorted rows (rows up to 32, up to 128 and beyond),
whose values follow update_values on the same pattern."""
import numpy as np
import pytest
import scipy.sparse as sp
import scipy.sparse.linalg as spl

import workloads as W
from oracle import sgmres_oracle as O

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA device", allow_module_level=True)

import paper_2303_08953_gb300 as sg  # noqa: E402


def dev(a):
    return torch.as_tensor(np.ascontiguousarray(a), dtype=torch.float64, device="cuda:0")


@pytest.fixture(scope="module")
def solver():
    s = sg.Solver(0)
    yield s
    s.close()


def _csr(M):
    M = sp.csr_matrix(M)
    M.sort_indices()
    return W.CSR(M.shape[0], M.indptr.astype(np.int32), M.indices.astype(np.int32),
                 M.data.astype(np.float64))


def _uneven(n, seed, mean=25):
    """Poisson row lengths, columns within a band (wide: over all of n)."""
    rng = np.random.default_rng(seed)
    cnt = np.minimum(rng.poisson(mean, n), n - 1)
    rows = np.repeat(np.arange(n), cnt)
    cols = (rows + rng.integers(-min(400, n // 2), min(400, n // 2) + 1, rows.size)) % n
    M = sp.coo_matrix((rng.standard_normal(rows.size), (rows, cols)), shape=(n, n)).tocsr()
    return _csr(M + sp.diags(np.abs(M).sum(1).A1 if hasattr(np.abs(M).sum(1), "A1")
                             else np.asarray(np.abs(M).sum(1)).ravel() + 1.0))


@pytest.mark.parametrize("n", [70, 1023, 1024, 1025, 5003, 70_001])
def test_sorted_windows_products(solver, n):
    A = _uneven(n, n)
    solver.analyze_csr(A)
    sell, stored = solver.matrix_info()
    nsl = (n + 31) // 32
    assert not sell or A.nnz <= stored <= 1.2 * A.nnz + 32 * nsl
    if n >= 1024:
        assert sell          # (in row order the padding is about 40 %)
    rng = np.random.default_rng(1)
    x, z = rng.uniform(-1, 1, n), rng.uniform(-1, 1, n)
    for _ in range(2):
        op = O.as_operator(A)
        y = solver.spmv_newton(dev(x), 0.7, 1.9, dev(z), 0.4).cpu().numpy()
        ref = (op @ x - 0.7 * x + 0.4 * z) / 1.9
        scale = (abs(op) @ np.abs(x) + 0.7 * np.abs(x) + 0.4 * np.abs(z)) / 1.9
        assert np.all(np.abs(y - ref) <= 1e-14 * scale)
        r = solver.residual(dev(z), dev(x)).cpu().numpy()
        assert np.all(np.abs(r - (z - op @ x)) <= 1e-14 * (abs(op) @ np.abs(x) + np.abs(z)))
        new = rng.standard_normal(A.nnz)
        solver.update_values(new)
        A = W.CSR(n, A.rowptr, A.colind, new)


def test_prepass_on_uneven_and_csr_rows(solver):
    """The resident FP64 step with the product in sorted slices and in CSR
    (one row of 900 entries keeps that matrix out of SELL)."""
    for A in (_uneven(5003, 2), _skewed()):
        solver.analyze_csr(A)
        op = O.as_operator(A)
        q = np.random.default_rng(4).uniform(-1, 1, A.n)
        q /= np.linalg.norm(q)
        H, steps = solver.arnoldi(dev(q), 5)
        Ho, so = O.arnoldi_mgs(op, q, 5)
        assert steps == so == 5
        K = [q]
        for _ in range(5):
            v = op @ K[-1]
            K.append(v / np.linalg.norm(v))
        K = np.column_stack(K)
        anorm = abs(op).sum(axis=0).max()
        for j in range(5):
            tol = max(8 * 2.0 ** -53 * np.linalg.cond(K[:, :j + 2]) * anorm, 1e-12 * anorm)
            assert np.all(np.abs(H[:, j] - Ho[:, j]) <= tol)


def _skewed(n=3001, seed=7):
    rng = np.random.default_rng(seed)
    M = sp.random(n, n, density=3.0 / n, random_state=seed, format="lil")
    M.setdiag(4.0)
    M[5, np.sort(rng.choice(n, 900, replace=False))] = 0.01 * rng.standard_normal(900)
    return _csr(M)


def _columns(n, lengths, seed):
    """Diagonally dominant, with column c of lengths[c] entries."""
    rng = np.random.default_rng(seed)
    M = sp.lil_matrix((n, n))
    for c, k in lengths.items():
        M[rng.choice(n, k, replace=False), c] = rng.uniform(-0.5, 0.5, (k, 1))
    M = M.tocsr()
    return _csr(M + sp.diags(np.asarray(abs(M).sum(1)).ravel() + 1.0)
                + sp.diags(rng.uniform(0.1, 0.3, n - 1), 1))


@pytest.mark.parametrize("n,lengths", [
    (1, {}), (33, {0: 31, 5: 30}), (900, {0: 32, 1: 33, 2: 127, 3: 128, 4: 129, 700: 64}),
    (4200, {7: 3000, 8: 500, 4199: 126}), (5000, {})])
@pytest.mark.parametrize("precision", ["fp64", "fp32_ir"])
def test_adjoint_on_the_transpose_and_new_values(solver, n, lengths, precision):
    A = _columns(n, lengths, n) if n > 1 else _csr(sp.csr_matrix([[2.5]]))
    solver.analyze_csr(A)
    rng = np.random.default_rng(11)
    val = A.val
    for step in range(3):
        g = rng.uniform(-1, 1, n)
        M = sp.csr_matrix((val, A.colind, A.rowptr), shape=(n, n))
        lam, info = solver.solve_adjoint(g, m=40, s=4, tol=1e-13, precision=precision)
        ref = spl.spsolve(M.T.tocsc(), g)
        assert info.converged
        # strictly diagonally dominant rows of A: ||A^-1||_inf <= 1, so the
        # error is at most the residual 1e-13 ||g||_2, times sqrt(n) for the
        # norms, plus the direct solve's own rounding
        assert np.linalg.norm(lam - ref) <= 1e-11 * np.sqrt(n) * np.linalg.norm(g)
        val = A.val * rng.uniform(0.9, 1.0, A.nnz)
        rows = np.repeat(np.arange(n), np.diff(A.rowptr))
        val[A.colind == rows] = A.val[A.colind == rows]     # the diagonal stays dominant
        solver.update_values(val if step else dev(val))

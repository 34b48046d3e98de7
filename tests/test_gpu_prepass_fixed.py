"""The resident FP64 pre-pass step (fixed-point MGS, w in shared memory) at
the sizes and values where it can go wrong: single rows and odd row counts,
ends of a CTA's rows and of its batches, CTAs whose rows of w are zero while
the basis is not (w's range grows), extreme scalings (its FP64 form) and
start vectors of a wide dynamic range.  Against the oracle's MGS-Arnoldi with
the tolerance of the entry-by-entry test in test_gpu_parity.py: 8 u
kappa(K_{j+2}) ||A||, at least 1e-12 ||A||_1."""
import numpy as np
import pytest

import workloads as W
from oracle import sgmres_oracle as O

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


def _run(solver, A, q, k):
    solver.analyze_csr(A)
    return solver.arnoldi(torch.as_tensor(q, dtype=torch.float64, device="cuda:0"), k)


def _check(A, q, k, H, steps):
    op = O.as_operator(A)
    Ho, so = O.arnoldi_mgs(op, q, k)
    assert steps == so
    anorm = abs(op).sum(axis=0).max()
    K = [q]
    for _ in range(k):
        v = op @ K[-1]
        K.append(v / np.linalg.norm(v) if np.any(v) else v)
    K = np.column_stack(K)
    for j in range(steps):
        kap = np.linalg.cond(K[:, :j + 2]) if j + 2 <= A.n else 1.0
        tol = max(8 * 2.0 ** -53 * kap * anorm, 1e-12 * anorm)
        assert np.all(np.abs(H[:j + 2, j] - Ho[:j + 2, j]) <= tol), (j, H[:, j], Ho[:, j], tol)


# rows: one, a half pair, the ends of 1024-row CTAs, of 2048- and 4096-row
# batches, several batches past the four that tensor memory keeps (2.6M rows
# on 152 SMs: 17,152 rows a CTA)
@pytest.mark.parametrize("n,k", [(1, 1), (2, 2), (3, 2), (31, 5), (33, 5), (1023, 6), (1025, 6),
                                 (2049, 7), (311_297, 6), (622_593, 5), (1_300_001, 4),
                                 (2_600_003, 4)])
def test_odd_sizes(solver, n, k):
    rng = np.random.default_rng(n)
    i = np.arange(n)
    rows = np.concatenate([i, i[1:], i[:-1]])
    cols = np.concatenate([i, i[:-1], i[1:]])
    vals = np.concatenate([2.0 + rng.uniform(0, 1, n), rng.uniform(-1, 0, n - 1),
                           rng.uniform(-1, 0, n - 1)])
    order = np.lexsort((cols, rows))
    ptr = np.zeros(n + 1, np.int32)
    np.cumsum(np.bincount(rows, minlength=n), out=ptr[1:])
    A = W.CSR(n, ptr, cols[order].astype(np.int32), vals[order])
    q = rng.uniform(-1, 1, n)
    q /= np.linalg.norm(q)
    H, steps = _run(solver, A, q, k)
    _check(A, q, k, H, steps)


@pytest.mark.parametrize("low", [0.0, 1e-30, 2.0 ** -70])
def test_rows_of_w_smaller_than_the_basis(solver, low):
    """Second half of the rows: A's entries are `low`, so w = A v_j is (next
    to) zero there while v_j is not, and every projection adds to it."""
    n, k = 9001, 6
    eig = np.where(np.arange(n) < n // 2, 1.0 + np.arange(n) / n, low)
    A = W.diagonal(eig)
    q = np.random.default_rng(3).uniform(0.5, 1.0, n)
    q /= np.linalg.norm(q)
    H, steps = _run(solver, A, q, k)
    _check(A, q, k, H, steps)


def test_point_source(solver):
    """From one unit entry: most CTAs' rows are zero for several steps."""
    A = W.stencil3d_convdiff(28)
    q = np.zeros(A.n)
    q[A.n // 2 + 400] = 1.0
    H, steps = _run(solver, A, q, 8)
    _check(A, q, 8, H, steps)


def test_wide_dynamic_range(solver):
    A = W.stencil2d(201, 97)
    q = np.exp(12.0 * np.random.default_rng(8).standard_normal(A.n))
    q /= np.linalg.norm(q)
    H, steps = _run(solver, A, q, 6)
    _check(A, q, 6, H, steps)


@pytest.mark.parametrize("e", [300, -300])
def test_power_of_two_scaling_is_exact(solver, e):
    """Every step of the fixed-point form is relative to the data's own
    exponents, so A 2^e gives H 2^e, bit for bit."""
    A = W.stencil3d_convdiff(14)
    q = np.random.default_rng(5).uniform(-1, 1, A.n)
    q /= np.linalg.norm(q)
    H, steps = _run(solver, A, q, 10)
    B = W.CSR(A.n, A.rowptr, A.colind, A.val * 2.0 ** e)
    Hs, steps_s = _run(solver, B, q, 10)
    assert steps == steps_s == 10
    assert np.array_equal(Hs, H * 2.0 ** e)


@pytest.mark.parametrize("e", [600, -600])
def test_norm_outside_the_normal_range(solver, e):
    """||A v_0||^2 overflows or underflows: the FP64 form.  The first
    coefficient is still v_0.A v_0, and the pre-pass ends there."""
    A = W.stencil3d_convdiff(14)
    op = O.as_operator(A)
    q = np.random.default_rng(6).uniform(-1, 1, A.n)
    q /= np.linalg.norm(q)
    B = W.CSR(A.n, A.rowptr, A.colind, A.val * 2.0 ** e)
    H, steps = _run(solver, B, q, 3)
    assert steps == 1
    # q and the products are rounded to 2^-53 each; the sum runs in FP64
    assert abs(H[0, 0] * 2.0 ** -e - q @ (op @ q)) <= 1e-13 * abs(q) @ (abs(op) @ abs(q))


def test_nan_in_the_matrix_reaches_h(solver):
    A = W.stencil2d(40, 40)
    val = A.val.copy()
    val[777] = np.nan
    q = np.full(A.n, 1.0 / 40)
    H, steps = _run(solver, W.CSR(A.n, A.rowptr, A.colind, val), q, 4)
    assert steps == 1 and np.isnan(H[0, 0]) and np.isnan(H[1, 0])

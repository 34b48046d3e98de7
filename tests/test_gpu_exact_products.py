"""FP64 block products from digit slices at the edges of the cut: extreme
digits in every place (level sums at their bounds), values far below their
column's largest, subnormals, zeros of both signs, columns near the ends of
the exponent range, and row counts around the readout and split sizes."""
from fractions import Fraction

import numpy as np
import pytest

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


@pytest.fixture
def tc_always():
    old = sg.set_tc_policy("always")
    yield
    sg.set_tc_policy(old)


def _columns(n, seed):
    """Columns (rows of the result) with hard digit patterns."""
    rng = np.random.default_rng(seed)
    low = np.ldexp(float(0x7F7F7F7F7F7F80 >> 7), 7 - 62)    # digits -128 in every place
    high = np.ldexp(float(0x7F7F7F7F7F7F00 >> 7), 7 - 62)   # digits 127
    c = [np.full(n, low), np.full(n, -low), np.full(n, high),
         np.where(np.arange(n) % 2, low, -high),
         rng.standard_normal(n) * np.exp2(rng.integers(-70, 1, n)),
         rng.standard_normal(n) * 2.0 ** -1000,
         rng.standard_normal(n) * 2.0 ** 480,
         np.where(rng.random(n) < 0.3, -0.0, rng.uniform(-1, 1, n)),
         np.zeros(n),
         rng.integers(-3, 4, n) * 2.0 ** -1074]
    for k in (0, 1, 2, 3):
        c[k][n // 2] = 1.0 - 2.0 ** -53       # sets the exponent: the others lie below
    c[5][::7] = 2.0 ** -1060                  # subnormals in a column of tiny normals
    return np.stack(c)


def _even(A):
    p = np.zeros((A.shape[0], A.shape[1] + A.shape[1] % 2))
    p[:, :A.shape[1]] = A
    return p


def _exponent(col):
    m = np.abs(col).max()
    return int(np.frexp(m)[1]) if m > 0 else -3000


@pytest.mark.parametrize("n", [256, 384, 385, 1000, 2081])
def test_block_dot_hard_digits(solver, tc_always, n):
    """Against the exact rational result: the digits below 2^-62 of a
    column's largest and the level sums past the eighth are left out, at
    most n 2^(eq + ex - 58), subnormals are taken as zero, and each of at
    most n / 128 split sums and their total is rounded once."""
    Q, X = _columns(n, 1), _columns(n, 2)[:, ::-1].copy()
    solver.n = n
    W = solver.block_dot(dev(_even(Q)), dev(_even(X))).cpu().numpy().T
    fq = [[Fraction(v) for v in r] for r in Q]
    fx = [[Fraction(v) for v in r] for r in X]
    for i in range(Q.shape[0]):
        for j in range(X.shape[0]):
            terms = [a * b for a, b in zip(fq[i], fx[j])]
            exact = sum(terms, Fraction(0))
            eq, ex = _exponent(Q[i]), _exponent(X[j])
            size = Fraction(2) ** (eq + ex)
            tol = n * size / 2 ** 58 + sum(abs(t) for t in terms) * (n // 128 + 2) / 2 ** 53
            tol += n * (Fraction(2) ** -1022) * (Fraction(2) ** max(eq, ex)) + Fraction(2) ** -1073
            assert abs(Fraction(W[i, j]) - exact) <= tol, (i, j)


@pytest.mark.parametrize("n", [512, 640, 1001])
@pytest.mark.parametrize("alpha,beta", [(-1.0, 1.0), (-0.7, 1.0), (0.5, 0.0), (1.0, -2.0)])
def test_block_update_hard_digits(solver, tc_always, n, alpha, beta):
    """X = beta X + alpha Q W: besides the digits left out (as above, with
    W' = W 2^(e_k) relative to its own columns' largest) the sum, the
    product with alpha and the addition are rounded once each."""
    Q = _columns(n, 3)
    rng = np.random.default_rng(4)
    i, s = Q.shape[0], 7
    e = np.array([_exponent(q) for q in Q])
    Wm = rng.standard_normal((i, s)) * np.exp2(-np.clip(e, -900, 900))[:, None]
    Wm[:, 3] = 0.0
    X = rng.standard_normal((s, n))
    Xd = dev(_even(X))
    solver.block_update(dev(_even(Q)), dev(np.ascontiguousarray(Wm.T)), Xd, alpha=alpha,
                        beta=beta, n=n)
    got = Xd.cpu().numpy()[:, :n]
    live = e > -2000
    top = (np.abs(Wm) * np.exp2(np.clip(e, -1074, 1023))[:, None])[live].max(0)
    g = np.frexp(top)[1]
    for r in list(range(0, n, 37)) + [n // 2, n - 1]:
        for c in range(s):
            p = Fraction(alpha) * sum((Fraction(Q[k, r]) * Fraction(Wm[k, c]) for k in range(i)),
                                      Fraction(0))
            ref = Fraction(beta) * Fraction(X[c, r]) + p
            drop = i * abs(Fraction(alpha)) * Fraction(2) ** int(g[c]) / 2 ** 58 if top[c] > 0 else 0
            sub = abs(Fraction(alpha)) * sum(abs(Fraction(Wm[k, c])) for k in range(i)) * Fraction(2) ** -1022
            tol = drop + sub + 4 * (abs(p) + abs(ref)) / 2 ** 53
            assert abs(Fraction(got[c, r]) - ref) <= tol, (r, c)


@pytest.mark.parametrize("m,s", [(30, 7), (24, 24), (17, 5)])
@pytest.mark.parametrize("scale", [1.0, 2.0 ** -40, 2.0 ** 40])
def test_solve_with_kept_exponents(tc_always, m, s, scale):
    """Whole restarted solves whose block products all take their column
    exponents from the updates that wrote the columns: the solution of
    A x = scale b (residual to 1e-12; the system's condition number is
    below 1e3) within 1e-9 of the FP64 direct one."""
    import scipy.sparse as sp
    import scipy.sparse.linalg as spl

    import workloads as W
    A = W.config_c1(32)["A"]
    M = sp.csr_matrix((A.val, A.colind, A.rowptr), shape=(A.n, A.n))
    rng = np.random.default_rng(m)
    b = rng.standard_normal(A.n) * scale
    solver = sg.Solver(0)
    try:
        solver.analyze_csr(A)
        x, info = solver.solve(dev(b), m=m, s=s, tol=1e-12)
        assert info.converged and info.restarts >= 1
        ref = spl.spsolve(M.tocsc(), b)
        assert np.linalg.norm(x.cpu().numpy() - ref) <= 1e-9 * np.linalg.norm(ref)
    finally:
        solver.close()

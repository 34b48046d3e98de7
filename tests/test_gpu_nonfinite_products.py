"""FP64 block products with an infinity or a NaN in an operand: it makes the
outputs that it enters non-finite, in the digit-slice form as in the FP64-pipe
form, and leaves every other output's bits as they are with a zero in its
place (the exponents are those of the finite values)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA device", allow_module_level=True)

import paper_2303_08953_gb300 as sg  # noqa: E402

INF, NAN = float("inf"), float("nan")


@pytest.fixture(scope="module")
def solver():
    s = sg.Solver(0)
    yield s
    s.close()


@pytest.fixture(params=["auto", "always", "never"])
def policy(request):
    old = sg.set_tc_policy(request.param)
    yield request.param
    sg.set_tc_policy(old)


def _block(k, n, seed):
    g = torch.Generator(device="cuda:0").manual_seed(seed)
    ld = (n + 31) // 32 * 32
    B = torch.zeros(k, ld, dtype=torch.float64, device="cuda:0")
    B[:, :n] = torch.randn(k, n, generator=g, device="cuda:0", dtype=torch.float64)
    return B * torch.logspace(-20, 20, k, base=2, dtype=torch.float64, device="cuda:0")[:, None]


# (n, i, s): tiles of 128 x 32 outputs with remainders, rows at the ends of
# stages and splits
SHAPES = [(256, 17, 9), (1000, 129, 33), (32768, 41, 10), (40001, 64, 40)]


@pytest.mark.parametrize("n,i,s", SHAPES)
@pytest.mark.parametrize("bad", [NAN, INF, -INF])
def test_dot(solver, policy, n, i, s, bad):
    Q, X = _block(i, n, 1), _block(s, n, 2)
    solver.n = n
    for what, col, row in [("q", 0, 0), ("q", i - 1, n - 1), ("q", i // 2, n // 2), ("x", 0, n - 1),
                           ("x", s - 1, 0), ("x", s // 2, n // 3)]:
        B = Q if what == "q" else X
        old = B[col, row].item()
        B[col, row] = 0.0
        ref = solver.block_dot(Q, X).clone()
        B[col, row] = bad
        W = solver.block_dot(Q, X)
        hit = torch.zeros(s, i, dtype=torch.bool, device="cuda:0")
        if what == "q":
            hit[:, col] = True
        else:
            hit[col, :] = True
        assert not torch.isfinite(W[hit]).any(), (what, col, row)
        assert torch.equal(W[~hit], ref[~hit]), (what, col, row)
        B[col, row] = old


@pytest.mark.parametrize("n,s", [(777, 24), (16384, 60)])
@pytest.mark.parametrize("bad", [NAN, INF])
def test_gram(solver, policy, n, s, bad):
    X = _block(s, n, 3)
    solver.n = n
    X[5, n - 2] = 0.0
    ref = solver.block_dot(X, X, sym=True).clone()
    X[5, n - 2] = bad
    G = solver.block_dot(X, X, sym=True)
    hit = torch.zeros(s, s, dtype=torch.bool, device="cuda:0")
    hit[5, :] = True
    hit[:, 5] = True
    assert not torch.isfinite(G[hit]).any()
    assert torch.equal(G[~hit], ref[~hit])


@pytest.mark.parametrize("n,i,s", SHAPES + [(131, 200, 40), (20000, 1, 70)])
@pytest.mark.parametrize("bad", [NAN, INF, -INF])
def test_update(solver, policy, n, i, s, bad):
    Q, X = _block(i, n, 4), _block(s, n, 5)
    g = torch.Generator(device="cuda:0").manual_seed(6)
    W = torch.randn(s, i, generator=g, device="cuda:0", dtype=torch.float64)
    solver.n = n
    for alpha, beta in ((-1.0, 1.0), (0.3, 0.0)):
        for col, row in ((0, 0), (i - 1, n - 1), (i // 2, n // 2)):
            old = Q[col, row].item()
            Q[col, row] = 0.0
            ref = solver.block_update(Q, W, X.clone(), alpha=alpha, beta=beta)
            Q[col, row] = bad
            Y = solver.block_update(Q, W, X.clone(), alpha=alpha, beta=beta)
            assert not torch.isfinite(Y[:, row]).any(), (col, row)
            Y[:, row] = ref[:, row]
            assert torch.equal(Y[:, :n], ref[:, :n]), (col, row)
            Q[col, row] = old
        old = W[s // 2, i // 2].item()
        ref = solver.block_update(Q, W, X.clone(), alpha=alpha, beta=beta)
        W[s // 2, i // 2] = bad
        Y = solver.block_update(Q, W, X.clone(), alpha=alpha, beta=beta)
        assert not torch.isfinite(Y[s // 2, :n]).any()
        Y[s // 2] = ref[s // 2]
        assert torch.equal(Y[:, :n], ref[:, :n])
        W[s // 2, i // 2] = old


@pytest.mark.parametrize("n,s", [(900, 40), (33000, 96)])
def test_triangular_product(solver, policy, n, s):
    """X Z with Z upper triangular: a NaN in column k of row r reaches the
    columns from k on (those before it are not asked for here: the forms
    multiply it by zeros or leave it out)."""
    X = _block(s, n, 7)
    g = torch.Generator(device="cuda:0").manual_seed(8)
    Z = torch.triu(torch.randn(s, s, generator=g, device="cuda:0", dtype=torch.float64)).t().contiguous()
    solver.n = n
    k, r = s // 2, n - 1
    X[k, r] = 0.0
    ref = solver.block_update(X, Z, torch.zeros_like(X), alpha=1.0, beta=0.0, upper=True)
    X[k, r] = NAN
    Y = solver.block_update(X, Z, torch.zeros_like(X), alpha=1.0, beta=0.0, upper=True)
    assert not torch.isfinite(Y[k:, r]).any()
    Y[:, r] = ref[:, r]
    assert torch.equal(Y[:, :n], ref[:, :n])

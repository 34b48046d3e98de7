"""FP64 block products on few rows: the splits of the rows (down to one
stage of 32), the 32-row update tile, idle columns and inner dimensions that
are no multiple of the stage, on both sides of each line."""
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
    old = sg.set_tc_policy("never")
    s = sg.Solver(0)
    yield s
    s.close()
    sg.set_tc_policy(old)


@pytest.mark.parametrize("n", [31, 33, 127, 4096, 4099, 9729, 19457])
@pytest.mark.parametrize("i,s", [(9, 10), (25, 10), (31, 10), (41, 10), (17, 17), (5, 33), (60, 7)])
def test_products_on_few_rows(solver, n, i, s):
    """Sums of n products, each split and their total rounded in some order:
    at most (n + 8) 2^-53 of the sum of magnitudes; the update likewise with
    i products, alpha and beta."""
    rng = np.random.default_rng(n + 7 * i + s)
    Q, X = rng.standard_normal((i, n)), rng.standard_normal((s, n))
    solver.n = n
    u = 2.0 ** -53
    W = solver.block_dot(dev(Q), dev(X)).cpu().numpy()
    size = np.abs(X).astype(np.longdouble) @ np.abs(Q).T.astype(np.longdouble)
    ref = X.astype(np.longdouble) @ Q.T.astype(np.longdouble)
    assert np.all(np.abs(W - ref) <= (n + 8) * u * size)
    Xd = dev(X)
    G = solver.block_dot(Xd, Xd, sym=True).cpu().numpy()
    gref = X.astype(np.longdouble) @ X.T.astype(np.longdouble)
    assert np.all(np.abs(G - gref) <= (n + 8) * u * (np.abs(X) @ np.abs(X).T))
    assert np.array_equal(G, G.T)
    Wm = rng.standard_normal((s, i))
    for alpha, beta in ((-1.0, 1.0), (0.3, 0.0)):
        Y = dev(X)
        solver.block_update(dev(Q), dev(Wm), Y, alpha=alpha, beta=beta, n=n)
        ref = beta * X.astype(np.longdouble) + alpha * (Wm.astype(np.longdouble) @ Q)
        size = abs(beta) * np.abs(X) + abs(alpha) * (np.abs(Wm) @ np.abs(Q))
        assert np.all(np.abs(Y.cpu().numpy() - ref) <= (i + 8) * u * size)
    Z = np.triu(rng.standard_normal((s, s)))
    T = solver.block_update(Xd, dev(np.ascontiguousarray(Z.T)), torch.zeros_like(Xd), alpha=1.0,
                            beta=0.0, upper=True, n=n).cpu().numpy()
    ref = Z.T.astype(np.longdouble) @ X
    assert np.all(np.abs(T - ref) <= (s + 8) * u * (np.abs(Z.T) @ np.abs(X)))


@pytest.mark.parametrize("n", [33, 4096, 4867, 20_000])
def test_early_launches_keep_their_order(solver, n):
    """A chain of short kernels that overwrite each other's inputs (columns
    at odd 16-byte places, so that CTAs share cache lines) gives the same
    bits every time, and the same as with a synchronisation after each."""
    rng = np.random.default_rng(n)
    i, s, ld = 21, 10, n + n % 2 + 2
    solver.n = n
    Q0, X0 = dev(rng.standard_normal((i, ld))), dev(rng.standard_normal((s, ld)))
    Z = dev(np.ascontiguousarray(np.triu(rng.uniform(0.1, 0.2, (s, s))).T))

    def chain(sync):
        Q, X = Q0.clone(), X0.clone()
        out = []
        for _ in range(6):
            for step in (lambda: out.append(solver.block_dot(Q, X)),
                         lambda: solver.block_update(Q, out[-1] * (0.5 / n), X, n=n),
                         lambda: out.append(solver.block_dot(X, X, sym=True)),
                         lambda: solver.block_update(X, Z, Q[:s], alpha=1.0, beta=0.0, upper=True, n=n)):
                step()
                if sync:
                    torch.cuda.synchronize()
        torch.cuda.synchronize()
        return out + [Q, X]

    ref = chain(True)
    for _ in range(20):
        for a, b in zip(chain(False), ref):
            assert torch.equal(a, b)

"""The eigensolver at the edges of its one-launch orthogonalisation: vectors of
one chunk and of many, chunks of uneven length, subspaces around the groups of
eight and four vectors its reductions use and up to the largest order (128),
and vectors too long for it (separate launches).

H = L x 1 x R (one channel, an identity MPO of dimension 2) with symmetric L and
R: its smallest eigenvalue is the smallest product of an eigenvalue of L and one
of R, known from numpy to 1e-15 of ||H||.  Bounds: the Ritz value of a converged
run carries the rounding of the products and of the recursion, below 1e-13 ||H||
each; the residual of its vector is below the stopping tolerance 1e-12 plus
kmax roundings of 1e-15 ||H||.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import seeded_inputs as si  # noqa: E402


@pytest.fixture(scope="module")
def b():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1501_05504_gb300 import binding
    binding.slib()
    return binding


@pytest.fixture(scope="module")
def ctx(b):
    c = b.dmrg3s_create(0, 2 << 30)
    yield c
    c.close()


def _symmetric(rng, n, gap):
    """Symmetric with spectrum in [0.5, 1] but for the smallest eigenvalue, -gap."""
    q, _ = np.linalg.qr(rng.standard_normal((n, n)))
    s = 0.5 + 0.5 * rng.random(n)
    s[0] = -gap
    a = (q * s) @ q.T
    return 0.5 * (a + a.T)


# (rows, cols, kmax): n = 2 rows cols
CASES = [(1, 1, 4), (1, 3, 8), (5, 7, 40), (11, 12, 33), (16, 8, 128), (64, 64, 128), (61, 83, 9),
         (200, 190, 40), (389, 401, 37), (560, 570, 24)]


@pytest.mark.parametrize("rows,cols,kmax", CASES)
def test_smallest_eigenvalue(b, ctx, rows, cols, kmax):
    rng = si.rng_for(80 + rows)
    Lm = _symmetric(rng, rows, 1.0)
    # R positive definite with a spectrum in [0.75, 1]: few Lanczos steps suffice
    q, _ = np.linalg.qr(rng.standard_normal((cols, cols)))
    Rm = (q * np.linspace(0.75, 1.0, cols)) @ q.T
    Rm = 0.5 * (Rm + Rm.T)
    lam = np.outer(np.linalg.eigvalsh(Lm), np.linalg.eigvalsh(Rm)).min()
    none = np.zeros((1, 0), np.int64)
    bl, br = b.Bond(none, np.array([rows])), b.Bond(none, np.array([cols]))
    W = np.zeros((2, 2, 1, 1))
    W[0, 0] = W[1, 1] = 1.0
    qp = np.zeros((2, 0), np.int64)
    cu = lambda x: torch.from_numpy(np.ascontiguousarray(x)).cuda().reshape(-1)
    L, R = b.Env(none, bl, cu(Lm)), b.Env(none, br, cu(Rm))
    Wm = b.MpoSite(qp, none, none, W)
    x0 = cu(rng.standard_normal(2 * rows * cols))
    M = b.Site(qp, bl, br, x0.clone())
    got, it = b.dmrg3s_eigensolve(ctx, L, Wm, R, M, kmax, 1e-12, "fp64")
    assert 1 <= it <= kmax
    x = M.data.cpu().numpy().reshape(2, rows, cols)
    assert abs(np.linalg.norm(x) - 1.0) < 1e-13
    Hx = Lm @ x @ Rm.T
    assert abs(np.vdot(x, Hx) - got) < 1e-13
    if it < kmax or 2 * rows * cols <= kmax:
        assert abs(got - lam) < 2e-13
        assert np.linalg.norm(Hx - got * x) < 1e-12 + kmax * 1e-15
    # the same start and subspace in numpy, fully reorthogonalised
    V = [x0.cpu().numpy() / np.linalg.norm(x0.cpu().numpy())]
    al, be = [], []
    for k in range(it):
        w = (Lm @ V[k].reshape(2, rows, cols) @ Rm.T).reshape(-1)
        al.append(V[k] @ w)
        B = np.array(V)
        for _ in range(2):
            w = w - B.T @ (B @ w)
        be.append(np.linalg.norm(w))
        if k + 1 < it:
            V.append(w / be[-1])
    T = np.diag(al) + np.diag(be[:-1], 1) + np.diag(be[:-1], -1)
    assert abs(np.linalg.eigvalsh(T)[0] - got) < 1e-12

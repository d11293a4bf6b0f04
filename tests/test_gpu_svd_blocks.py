"""The Jacobi sweeps' block rounds at their edges: column counts around a
block of four (padding columns, a padding block), around the columns a lane
keeps in registers (256), and around the sizes from which a pair of blocks no
longer fits shared memory (512 columns with left vectors, 1024 without).

Bounds as for the other shapes of this SVD: singular values within 1e-13 of the
largest, orthonormal vectors to 1e-12, A = U S V^T to 1e-13 of the largest
singular value.
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
    c = b.dmrg3s_create(0, 1 << 30)
    yield c
    c.close()


def _matrix(rng, m, n, lo):
    qa, _ = np.linalg.qr(rng.standard_normal((m, n)))
    qb, _ = np.linalg.qr(rng.standard_normal((n, n)))
    return (qa * np.logspace(0, lo, n)) @ qb.T


@pytest.mark.parametrize("n,want_u", [(k, True) for k in (1, 3, 4, 5, 8, 9, 12, 13, 255, 256, 257, 512, 513)]
                         + [(257, False), (1024, False), (1025, False)])
def test_block_edges(b, ctx, n, want_u):
    X = _matrix(si.rng_for(50 + n), n + 7, n, -9)
    u, s, vt = (None if t is None else t.cpu().numpy()
                for t in b.dmrg3s_svd(ctx, [torch.from_numpy(X).cuda()], want_u=want_u)[0])
    ref = np.linalg.svd(X, compute_uv=False)
    assert np.all(np.diff(s) <= 0.0)
    assert np.abs(s - ref).max() <= 1e-13 * ref[0]
    assert np.abs(vt @ vt.T - np.eye(n)).max() < 1e-12
    if want_u:
        assert np.abs(u.T @ u - np.eye(n)).max() < 1e-12
        assert np.abs((u * s) @ vt - X).max() <= 1e-13 * ref[0]


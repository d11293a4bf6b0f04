"""Reflectors of columns whose squares leave the FP64 range: after the columns
before it are taken out, a column may be 1e-150 or less while later ones are of
order one.  A norm computed from subnormal squares has few digits, and the
reflection made of it would not be orthogonal on those later columns.

Bounds as for this SVD elsewhere: singular values within 1e-13 of the largest,
orthonormal left vectors to 1e-12, A = U S V^T to 1e-13 of the largest.
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


@pytest.mark.parametrize("m", [40, 1500])          # one CTA, several
@pytest.mark.parametrize("tiny", [1e-140, 1e-150, 1e-158, 1e-161, 1e-165, 1e-310])
def test_tiny_residual_column(b, ctx, m, tiny):
    rng = si.rng_for(811)
    n = 30
    X = np.zeros((m, n))
    X[0, 0] = 10.0
    X[0, 1], X[1:, 1] = 9.0, tiny * rng.standard_normal(m - 1)   # second by norm
    X[:, 2:] = 4.0 * rng.standard_normal((m, n - 2)) / np.sqrt(m)
    (u, s, vt), = b.dmrg3s_svd(ctx, [torch.from_numpy(X).cuda()])
    u, s, vt = u.cpu().numpy(), s.cpu().numpy(), vt.cpu().numpy()
    ref = np.linalg.svd(X, compute_uv=False)
    assert np.abs(s - ref).max() <= 1e-13 * ref[0]
    # (the second column repeats the first: one zero singular value)
    assert np.abs(u.T @ u - np.eye(n)).max() < 1e-12
    assert np.abs((u * s) @ vt - X).max() <= 1e-13 * ref[0]

"""The Householder QR before the Jacobi sweeps, through the SVD that uses it: matrices
of one CTA and of several, more matrices than SMs in one batch, columns split
over warps or not, zero columns, and a matrix whose columns don't fit the shared
memory of the GPU (the library's QR).  Left vectors are Q times the accumulated
rotations, so they test the stored reflectors.

Bounds as for this SVD elsewhere: singular values within 1e-13 of the largest,
orthonormal vectors to 1e-12, A = U S V^T to 1e-13 of the largest singular value.
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


def _check(X, u, s, vt):
    ref = np.linalg.svd(X, compute_uv=False)
    n = X.shape[1]
    assert np.all(np.diff(s) <= 0.0)
    assert np.abs(s - ref).max() <= 1e-13 * ref[0]
    k = int((s > 1e-12 * s[0]).sum())
    assert np.abs(vt[:k] @ vt[:k].T - np.eye(k)).max() < 1e-12
    assert np.abs(u.T @ u - np.eye(n)).max() < 1e-12
    assert np.abs((u * s) @ vt - X).max() <= 1e-13 * ref[0]


def _run(b, ctx, mats):
    out = b.dmrg3s_svd(ctx, [torch.from_numpy(X).cuda() for X in mats])
    for X, res in zip(mats, out):
        _check(X, *(t.cpu().numpy() for t in res))


@pytest.mark.parametrize("m,n", [(1, 1), (2, 1), (3, 2), (17, 16), (33, 33), (129, 40), (700, 3), (300, 299),
                                 (2100, 150), (12000, 2), (13000, 5)])
def test_one_matrix(b, ctx, m, n):
    rng = si.rng_for(90 + m + n)
    X = rng.standard_normal((m, n)) * np.logspace(0, -6, n)
    _run(b, ctx, [X])


def test_many_matrices(b, ctx):
    rng = si.rng_for(91)
    mats = [rng.standard_normal((int(n + rng.integers(0, 30)), int(n))) for n in rng.integers(1, 40, 200)]
    mats += [rng.standard_normal((330, 260)), rng.standard_normal((150, 120))]
    mats[5][:, 0] = 0.0
    mats[7][:] = np.eye(*mats[7].shape)
    _run(b, ctx, mats)

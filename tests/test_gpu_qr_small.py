"""Matrices that one CTA factorises by itself: every reflector is formed by the
CTA's first warps while the others still apply the one before.  Few rows make a
reflector's chain short, and columns of very different direction make its
factors tau differ, so a factor read too late shows in R and Q.

Bounds: A = U S V^T to 1e-13 of the largest singular value and orthonormal vectors
to 1e-12 (as for this SVD elsewhere); the same bits from run to run.
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


@pytest.mark.parametrize("m,n", [(2, 2), (5, 4), (24, 20), (40, 33)])
def test_one_cta_each(b, ctx, m, n):
    rng = si.rng_for(700 + m)
    mats = []
    for k in range(600):
        X = rng.standard_normal((m, n))
        X[:, 1 + k % (n - 1)] = X[:, 0] * (1.0 + 1e-3 * rng.standard_normal(m))   # tau near 1 and near 2
        mats.append(X)
    dev = [torch.from_numpy(X).cuda() for X in mats]
    first = b.dmrg3s_svd(ctx, dev)
    for X, (u, s, vt) in zip(mats, ([t.cpu().numpy() for t in r] for r in first)):
        assert np.abs((u * s) @ vt - X).max() <= 1e-13 * s[0]
        assert np.abs(u.T @ u - np.eye(n)).max() < 1e-12
    for _ in range(3):
        for r0, r1 in zip(first, b.dmrg3s_svd(ctx, dev)):
            assert all(torch.equal(x, y) for x, y in zip(r0, r1))

"""A launch whose stream has fewer SMs than the plan counted on (a green context, a
smaller second device) refuses the cooperative kernels: the eigensolver then
orthogonalises in separate launches and the SVD factorises with cuSOLVER.  Here the
plan is told of more SMs than the GPU has, so that the runtime refuses the launch
before anything runs.

Bounds: eigenvalue and residual as for the eigensolver elsewhere (1e-10 of the
value), singular values 1e-13 of the largest, A = U S V^T to the same.
"""
import ctypes

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import seeded_inputs as si  # noqa: E402
from parity import problem  # noqa: E402


@pytest.fixture(scope="module")
def b():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1501_05504_gb300 import binding
    binding.slib()
    return binding


@pytest.fixture
def many_sms(b):
    lib = b.lib()
    get, put = lib._ZN6dmrg3s9plan_ctasEv, lib._ZN6dmrg3s13set_plan_ctasEi
    get.restype, put.argtypes, put.restype = ctypes.c_int, [ctypes.c_int], None
    ctx = b.dmrg3s_create(0, 1 << 30)
    n = get()
    put(1024)
    yield ctx
    put(n)
    ctx.close()


@pytest.mark.parametrize("prec,tol", [("fp64", 1e-10), ("tf32x3", 1e-5)])
def test_eigensolver(b, many_sms, prec, tol):
    pr = problem("u1", 31, m_left=400, m_right=420)
    L, R = b.env_from_neutral(pr["L"]), b.env_from_neutral(pr["R"])
    W = b.mpo_from_neutral(pr["W"])
    got = []
    for ctx in (many_sms, None):
        if ctx is None:
            ctx = b.dmrg3s_create(0, 1 << 30)      # (sets the GPU's own count again)
        M = b.site_from_neutral(pr["A"])
        got.append((b.dmrg3s_eigensolve(ctx, L, W, R, M, kmax=25, tol=1e-12, prec=prec)[0], M.data.clone()))
    (l0, m0), (l1, m1) = got
    assert abs(l0 - l1) <= tol * abs(l1)
    assert 1.0 - abs(float(m0 @ m1)) <= tol


def test_svd(b, many_sms):
    rng = si.rng_for(33)
    mats = [rng.standard_normal((60, 40)) for _ in range(900)] + [rng.standard_normal((500, 300))]
    out = b.dmrg3s_svd(many_sms, [torch.from_numpy(X).cuda() for X in mats])
    for X, (u, s, vt) in list(zip(mats, out))[-40:]:
        u, s, vt = u.cpu().numpy(), s.cpu().numpy(), vt.cpu().numpy()
        assert np.abs(s - np.linalg.svd(X, compute_uv=False)).max() <= 1e-13 * s[0]
        assert np.abs((u * s) @ vt - X).max() <= 1e-13 * s[0]

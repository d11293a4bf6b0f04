"""The plain FP64 products in every tile size (8, 16, 32, 64): one sector with
dimensions around the tiles' edges, a dense MPO tensor (too many terms for the
sliced form, and below its least work at the small sizes), in the forms N N, N T
and T N of its grouped GEMM.

Tolerance: three stages, each a sum of K <= 1200 products rounded K times at most
in the plain form: relative (Frobenius) 3 sqrt(1200) 2^-53 < 2e-14, and the
reference's own rounding of the same size.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

TOL = 4e-14
W_, D_ = 4, 2


@pytest.fixture(scope="module")
def b():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1501_05504_gb300 import binding
    binding.lib()
    return binding


@pytest.fixture(scope="module")
def ctx(b):
    c = b.dmrg3s_create(0, 1 << 30)
    yield c
    c.close()


@pytest.mark.parametrize("l,r", [(1, 1), (1, 9), (7, 8), (9, 16), (15, 17), (33, 31), (64, 63), (65, 100),
                                 (1, 300), (129, 257), (300, 290)])
def test_tiles(b, ctx, l, r):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(100 * l + r)
    rnd = lambda *s: torch.randn(*s, dtype=torch.float64, device="cuda", generator=gen)
    L, R, M = rnd(W_, l, l), rnd(W_, r, r), rnd(D_, l, r)
    W = rnd(D_, D_, W_, W_)
    none, t, qp = (np.zeros((n, 0), np.int64) for n in (1, W_, D_))
    bl, br = b.Bond(none, np.array([l])), b.Bond(none, np.array([r]))
    Wm = b.MpoSite(qp, t, t, W.cpu().numpy())
    Le, Re, Ms = b.Env(t, bl, L.reshape(-1)), b.Env(t, br, R.reshape(-1)), b.Site(qp, bl, br, M.reshape(-1))
    T2 = torch.einsum("pqbc,bqij->cpij", W, torch.matmul(L[:, None], M[None]))
    U2 = torch.einsum("pqbc,cqij->bpij", W, torch.matmul(M[None], R.transpose(1, 2)[:, None]))
    HA = torch.matmul(T2, R.transpose(1, 2)[:, None]).sum(0)
    out = b.empty_site_like(qp, bl, br)
    b.dmrg3s_apply_heff(ctx, Le, Wm, Re, Ms, out, "fp64")
    E1, E2 = b.empty_env(t, br), b.empty_env(t, bl)
    b.dmrg3s_update_env(ctx, 1, Le, Wm, Ms, E1, "fp64")
    b.dmrg3s_update_env(ctx, -1, Re, Wm, Ms, E2, "fp64")
    b.dmrg3s_sync(ctx)
    for got, ref in ((out.data, HA), (E1.data, torch.matmul(M.transpose(1, 2)[None], T2).sum(1)),
                     (E2.data, torch.matmul(M[None], U2.transpose(2, 3)).sum(1))):
        assert float((got.view(ref.shape) - ref).norm()) <= TOL * float(ref.norm())

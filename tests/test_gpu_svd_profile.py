"""The profiler's count of a Jacobi sweep: 2n flops (a dot product) and 16n bytes for
each of its n (n - 1) / 2 pair tests.  Orthogonal columns are factorised into a
diagonal R, so one sweep tests every pair and rotates none."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import seeded_inputs as si  # noqa: E402

KERNEL_JACOBI = 9


@pytest.mark.parametrize("m,n", [(40, 30), (300, 120)])
def test_pair_tests_without_rotations(m, n):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1501_05504_gb300 import binding as b
    b.slib()
    ctx = b.dmrg3s_create(0, 1 << 28)
    q = np.linalg.qr(si.rng_for(60).standard_normal((m, n)))[0] * np.logspace(0, -3, n)
    b.dmrg3s_profile(ctx, True)
    b.dmrg3s_svd(ctx, [torch.from_numpy(q).cuda()])
    st = b.dmrg3s_profile_read(ctx, KERNEL_JACOBI)
    b.dmrg3s_profile(ctx, False)
    ctx.close()
    assert st["flops"] == 0.5 * n * (n - 1) * 2 * n
    assert st["bytes"] == 0.5 * n * (n - 1) * 16 * n

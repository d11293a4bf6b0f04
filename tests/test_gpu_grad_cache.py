"""The gradient's look-up by arguments stays bounded: a program that varies the MPO
entries makes a new set of arguments with every call.  60 bytes an entry and 150000
calls would be 9 MB; the bound allows 4096 entries, and 3 MB leaves room for the
allocator."""
import os

import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from parity import problem  # noqa: E402


def _resident():
    with open("/proc/self/statm") as f:
        return int(f.read().split()[1]) * os.sysconf("SC_PAGESIZE")


def test_varying_entries():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1501_05504_gb300 import binding as b
    pr = problem("u1", 51, m_left=6, m_right=6)
    ctx = b.dmrg3s_create(0, 1 << 24)
    L, R = b.env_from_neutral(pr["L"]), b.env_from_neutral(pr["R"])
    W, M = b.mpo_from_neutral(pr["W"]), b.site_from_neutral(pr["A"])
    G = torch.zeros(W.W.size, dtype=torch.float64, device="cuda")

    def calls(n, start):
        for k in range(n):
            W.W[0, 0, 0, 0] = start + k
            b.dmrg3s_mpo_grad_site(ctx, L, W, R, M, G)
        torch.cuda.synchronize()
    calls(10000, 1.0)
    before = _resident()
    calls(150000, 1e6)
    assert _resident() - before < 3 << 20
    ctx.close()

"""Componentwise accuracy of the sliced FP64 contractions on graded tensors.

The rows of a site tensor carry the Schmidt weights of the bond that the
contraction sums over, so small and large terms meet in one sum.  An FP64 product
rounds every term at 2^-53 of itself; the tensors here span 14 and 40 decades along
the contracted bond, which a fixed-point form of its rows cannot hold.

* Copies: environments and an MPO that only copy (identity channels, one diagonal
  operator) give h M, whose elements have one rounding in either form.
* Any contraction: |sliced - plain| <= n 2^-53 S elementwise, with S the same
  contraction of the absolute values and n the roundings a term passes in the plain
  form (the additions of its sums: at most K of each stage and the MPO terms) plus
  4 for the two forms' results.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from test_gpu_sliced import CALLS, XXZ_QP, XXZ_T, XXZ_W, Problem, _both, _bonds  # noqa: E402


@pytest.fixture(scope="module")
def b():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1501_05504_gb300 import binding
    binding.lib()
    return binding


def _grade(p, decades):
    """Rows and columns of M by weights of that many decades each, in every sector."""
    for s, i, j, off, r, c in p.M.blocks():
        w = [torch.logspace(0, -decades, int(n), dtype=torch.float64, device="cuda") for n in (r, c)]
        p.M.data[off:off + r * c].view(int(r), int(c)).mul_(w[0][:, None] * w[1][None, :])


def _identity(env, channels):
    """These channels of an environment the identity, the others as they are."""
    for ch, bra, ket, off, r, c in env.blocks():
        if ch in channels:
            env.data[off:off + r * c] = torch.eye(int(r), int(c), dtype=torch.float64, device="cuda").reshape(-1)


DIMS = (200, 257, 130, 33)


@pytest.mark.parametrize("decades", [14, 40])
@pytest.mark.parametrize("call", ("heff", "op", "expand+", "expand-"))
def test_copies_keep_every_digit(b, call, decades):
    W = np.zeros((2, 2, 5, 5))
    W[:, :, 4, 0] = np.diag([0.3, -0.7])
    p = Problem(b, *_bonds(b, DIMS, 1), W=W, seed=21)
    _identity(p.L, (4,))
    _identity(p.R, (0,))
    _grade(p, decades)
    x, y, counts = _both(b, p, call)
    assert counts[0] != counts[1]                  # two forms ran
    assert float(y.abs().max()) > 0.0
    # (the plain form: M exactly, one rounding by h, one by the expansion's factor)
    assert bool(((x - y).abs() <= 2.0 ** -51 * y.abs()).all())


@pytest.mark.parametrize("decades", [0, 14, 40])
@pytest.mark.parametrize("call", CALLS)
def test_componentwise_bound(b, call, decades):
    p = Problem(b, *_bonds(b, DIMS, 2), seed=33)
    _identity(p.L, (4,))
    _identity(p.R, (0,))
    _grade(p, decades)
    x, y, counts = _both(b, p, call)
    assert counts[0] != counts[1]
    q = Problem(b, p.left, p.right, W=np.abs(XXZ_W), seed=33)
    q.L.data, q.R.data, q.M.data = p.L.data.abs(), p.R.data.abs(), p.M.data.abs()
    _, size, _ = _both(b, q, call)
    n = 257 + 4 + 2 * 5 * 257 + 4
    assert bool(((x - y).abs() <= n * 2.0 ** -53 * size).all())


@pytest.mark.parametrize("kind", ("loguniform", "sparse"))
@pytest.mark.parametrize("call", CALLS)
def test_whole_parts_listed(b, call, kind):
    """Elements over 40 decades without an order along any bond, and few that are not
    zero: nearly every element of a part is listed, and formed or found to be zero."""
    p = Problem(b, *_bonds(b, DIMS, 2), seed=34)
    g = torch.Generator(device="cuda").manual_seed(7)
    u = torch.rand(p.M.data.shape, dtype=torch.float64, device="cuda", generator=g)
    p.M.data.mul_(10.0 ** (40 * u - 20) if kind == "loguniform" else (u < 0.02).double())
    x, y, counts = _both(b, p, call)
    assert counts[0] != counts[1]
    q = Problem(b, p.left, p.right, W=np.abs(XXZ_W), seed=34)
    q.L.data, q.R.data, q.M.data = p.L.data.abs(), p.R.data.abs(), p.M.data.abs()
    _, size, _ = _both(b, q, call)
    n = 257 + 4 + 2 * 5 * 257 + 4
    assert bool(((x - y).abs() <= n * 2.0 ** -53 * size).all())


def test_repeating_digits(b):
    """Data that repeat along k: every digit product has the same sign in all terms, so
    the lower levels' sums leave the range that FP32 holds exactly."""
    from fractions import Fraction
    qp, t = np.zeros((1, 0), int), np.zeros((1, 0), int)
    bond = b.Bond(np.zeros((1, 0), int), np.array([300]))
    p = Problem(b, bond, bond, qp, t, np.ones((1, 1, 1, 1)))
    # digits of 255 and of 127 after a first one of 1: the sums of levels 4-7 pass 2^24
    v = sum(Fraction(255, 512 ** (i + 1)) for i in range(5)) + Fraction(1, 2)
    for lead in (Fraction(1), Fraction(1, 512), Fraction(1, 512 ** 3)):
        for x in (p.L, p.M):
            x.data.fill_(float(v * lead))
            x.data[0] = 1.0
        f = b.expanded_bond(p.right, t)
        out = b.empty_site_like(qp, p.left, f)
        ctx = b.dmrg3s_create(0, 1 << 30)
        b.dmrg3s_expand(ctx, 1, p.L, p.W, p.M, 1.0, out, "fp64")
        b.dmrg3s_sync(ctx)
        ctx.close()
        got = out.data.view(300, 300)
        a = Fraction(float(v * lead))
        ref = 300 * a * a                           # rows and columns without the 1
        assert float((got[1:, 1:] - float(ref)).abs().max()) <= 2.0 ** -51 * float(ref)

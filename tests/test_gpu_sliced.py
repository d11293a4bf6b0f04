"""FP64 contractions by exact FP16 slices (csrc/kernels_sliced.cu).

The sliced form runs where its intermediates fit the context workspace; a
context whose workspace holds only the plain form's intermediates runs the
plain FP64 kernels.  Every case runs both forms on the same inputs.

Tolerance: either form rounds an output element after at most three stages; the
plain form's sums of K terms carry at most about sqrt(K) 2^-53 of their
Frobenius scale each, the sliced form 2^-53 per stage.  With K <= 2048 that is
3 (45 + 1) 1.1e-16 < 2e-14 relative (Frobenius).
"""
import itertools

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

TOL = 2e-14

XXZ_QP = np.array([[1], [-1]])
XXZ_T = np.array([[0], [2], [-2], [0], [0]])
# a model MPO: every allowed (operator, channel) pair of the finite-state form,
# with coefficients that are and are not powers of two
XXZ_W = np.zeros((2, 2, 5, 5))
XXZ_W[:, :, 0, 0] = XXZ_W[:, :, 4, 4] = np.eye(2)
XXZ_W[0, 1, 4, 1] = XXZ_W[1, 0, 4, 2] = 1.0
XXZ_W[1, 0, 1, 0], XXZ_W[0, 1, 2, 0] = 0.5, 0.7
XXZ_W[:, :, 4, 3] = np.diag([0.5, -0.5])
XXZ_W[:, :, 3, 0] = np.diag([0.3, -0.3])

# sector dimensions around the tiles' edges (16 columns, 64 k, 128 rows)
EDGES = [(64, 65, 63, 1), (128, 127, 129, 16), (1, 17, 130, 200, 257), (15, 31, 33, 47, 48, 49),
         (80, 95, 97, 113, 2, 3, 255)]


@pytest.fixture(scope="module")
def b():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1501_05504_gb300 import binding
    binding.lib()
    return binding


def _bonds(b, dims, shift):
    n = len(dims)
    left = b.Bond(np.arange(n).reshape(-1, 1) * 2 + 1, np.array(dims))
    rd = tuple(dims[shift % n:]) + tuple(dims[:shift % n])
    right = b.Bond(np.arange(n).reshape(-1, 1) * 2, np.array(rd))
    return left, right


def _random(n, seed):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    return torch.randn(max(n, 1), dtype=torch.float64, device="cuda", generator=gen)


class Problem:
    def __init__(self, b, left, right, qp=XXZ_QP, t=XXZ_T, W=XXZ_W, seed=0):
        self.b, self.qp, self.t = b, qp, t
        self.left, self.right = left, right
        self.W = b.MpoSite(qp, t, t, W)
        self.L, self.R, self.M = b.Env(t, left), b.Env(t, right), b.Site(qp, left, right)
        self.L.data, self.R.data = _random(self.L.size(), seed), _random(self.R.size(), seed + 1)
        self.M.data = _random(self.M.size(), seed + 2)

    def run(self, ctx, call):
        b = self.b
        if call == "heff":
            out = b.empty_site_like(self.qp, self.left, self.right)
            b.dmrg3s_apply_heff(ctx, self.L, self.W, self.R, self.M, out, "fp64")
        elif call == "op":
            out = b.empty_site_like(self.qp, self.left, self.right)
            op = b.HeffOp(ctx, self.L, self.W, self.R, self.M, "fp64")
            op.apply(self.M, out)
            op.close()
        elif call in ("expand+", "expand-"):
            d = 1 if call[-1] == "+" else -1
            f = b.expanded_bond(self.right if d > 0 else self.left, self.t)
            out = b.empty_site_like(self.qp, self.left, f) if d > 0 else b.empty_site_like(self.qp, f, self.right)
            b.dmrg3s_expand(ctx, d, self.L if d > 0 else self.R, self.W, self.M, 0.37, out, "fp64")
        else:
            d = 1 if call[-1] == "+" else -1
            out = b.empty_env(self.t, self.right if d > 0 else self.left)
            b.dmrg3s_update_env(ctx, d, self.L if d > 0 else self.R, self.W, self.M, out, "fp64")
        b.dmrg3s_sync(ctx)
        return out.data.clone()


CALLS = ("heff", "op", "expand+", "expand-", "env+", "env-")


def _plain_bytes(p, call):
    """The workspace of the plain form: T1 and T2 (without T2 for an expansion) in
    FP64, and no sliced operand (each takes 14 bytes an element, padded)."""
    right = call in ("expand-", "env-")
    site, env = p.M.blocks(), (p.R if right else p.L).blocks()
    one, two = 0, {}
    W = p.W.W
    for s, i, j, _, r, c in site:
        for ch, bra, ket, _, er, ec in env:
            if ket != (j if right else i):
                continue
            n = int(r * er if right else er * c)
            one += n
            for so, other in zip(*np.nonzero(W[:, s, :, ch] if right else W[:, s, ch, :])):
                two[(so, other, i if right else bra, bra if right else j)] = n
    return 8 * (one + (0 if call.startswith("expand") else sum(two.values()))) + 256


def _both(b, p, call):
    """The result of the sliced form, that of the plain one, and their launches."""
    big, small = b.dmrg3s_create(0, 1 << 30), b.dmrg3s_create(0, _plain_bytes(p, call))
    counts = []
    out = []
    for ctx in (big, small):
        n0 = b.dmrg3s_launch_count()
        out.append(p.run(ctx, call))
        counts.append(b.dmrg3s_launch_count() - n0)
        ctx.close()
    return out[0], out[1], counts


def _rel(x, y):
    n = y.norm()
    return float((x - y).norm() / (n if n > 0 else 1.0))


@pytest.mark.parametrize("call", CALLS)
@pytest.mark.parametrize("dims,shift", [(d, s) for d, s in zip(EDGES, itertools.cycle((0, 1, 2)))])
def test_sliced_equals_plain_at_tile_edges(b, dims, shift, call):
    p = Problem(b, *_bonds(b, dims, shift), seed=len(dims))
    x, y, counts = _both(b, p, call)
    assert _rel(x, y) < TOL
    if sum(dims) > 250:
        assert counts[0] != counts[1] or not torch.equal(x, y)      # two forms ran


@pytest.mark.parametrize("m", [168, 201, 1800, 2048])
def test_long_contractions_keep_headroom(b, m):
    """One sector, w = 1, constant data of all digit patterns: the sums are exact
    multiples, so the result must be the rounded product (one ulp)."""
    from fractions import Fraction
    qp, t = np.zeros((1, 0), int), np.zeros((1, 0), int)
    bond = b.Bond(np.zeros((1, 0), int), np.array([m]))
    ctx = b.dmrg3s_create(0, 4 << 30)
    for v in (2.0 - 2.0 ** -52, -1.0 / 3.0, 1608428438346605.0):
        p = Problem(b, bond, bond, qp, t, np.ones((1, 1, 1, 1)))
        for x in (p.L, p.R, p.M):
            x.data.fill_(v)
        got = p.run(ctx, "heff")
        t2 = float(Fraction(v) * Fraction(v) * m)
        ref = float(Fraction(t2) * Fraction(v) * m)
        assert float((got - ref).abs().max()) <= 2.0 ** -52 * abs(ref)
    ctx.close()


@pytest.mark.parametrize("call", CALLS)
def test_inf_and_nan_reach_what_the_plain_form_gives(b, call):
    p = Problem(b, *_bonds(b, (128, 127, 129, 16), 1), seed=5)
    p.M.data[3] = float("inf")
    p.M.data[-5] = float("nan")
    p.L.data[1000] = float("-inf")
    p.R.data[7] = float("nan")
    x, y, _ = _both(b, p, call)
    assert torch.equal(torch.isnan(x), torch.isnan(y))
    assert torch.equal(torch.isinf(x), torch.isinf(y))
    f = torch.isfinite(y)
    assert torch.equal(x[torch.isinf(y)], y[torch.isinf(y)])
    assert _rel(x[f], y[f]) < TOL


@pytest.mark.parametrize("scale", [1e-300, 1e-308, 1e290, 1e300, 0.0])
def test_extreme_scales(b, scale):
    """One stage with results in the subnormal range, at zero and beyond the
    largest double.  The plain form rounds every partial sum to the subnormal
    grid: at most 3 x 129 roundings of 2^-1075, below 256 x 2^-1074.  The sliced
    form rounds the whole sum once, so it leaves the finite range only where the
    sum does; there the plain form does too (its partial sums may overflow
    where the whole sum would not)."""
    p = Problem(b, *_bonds(b, (128, 127, 129, 16), 2), seed=9)
    p.M.data.mul_(scale)
    p.L.data.mul_(1e-15 if scale < 1 else 1e10)
    x, y, _ = _both(b, p, "expand+")
    fx, fy = torch.isfinite(x), torch.isfinite(y)
    assert bool((fx | ~fy | (y.abs() > 1e306)).all())
    f = fx & fy
    if bool(f.any()):
        assert bool(((x[f] - y[f]).abs() <= 1e-12 * y[f].abs().max() + 256 * 2.0 ** -1074).all())


def test_graded_rows_and_columns(b):
    """Rows and columns that span 14 decades (Schmidt weights): columnwise errors
    against FP64 stay at the column's own scale."""
    p = Problem(b, *_bonds(b, (200, 210), 0), seed=12)
    for s, i, j, off, r, c in p.M.blocks():
        w = torch.logspace(0, -14, int(c), dtype=torch.float64, device="cuda")
        p.M.data[off:off + r * c].view(int(r), int(c)).mul_(w[None, :])
    x, y, _ = _both(b, p, "expand+")
    f = b.expanded_bond(p.right, p.t)
    tab = b.empty_site_like(p.qp, p.left, f).blocks()
    for s, i, j, off, r, c in tab:
        u, v = x[off:off + r * c].view(int(r), int(c)), y[off:off + r * c].view(int(r), int(c))
        n = v.norm(dim=0)
        assert bool(((u - v).norm(dim=0)[n > 0] <= TOL * n[n > 0]).all())


def test_wait_limit_reports_timeout(b):
    p = Problem(b, *_bonds(b, (128, 127, 129, 16), 1), seed=3)
    ctx = b.dmrg3s_create(0, 1 << 30)
    ref = p.run(ctx, "heff")
    b.dmrg3s_set_wait_limit(ctx, 0.0)
    out = b.empty_site_like(p.qp, p.left, p.right)
    b.dmrg3s_apply_heff(ctx, p.L, p.W, p.R, p.M, out, "fp64")
    with pytest.raises(b.Dmrg3sError) as e:
        b.dmrg3s_sync(ctx)
    assert e.value.status == 8
    b.dmrg3s_set_wait_limit(ctx, 1.0)
    assert torch.equal(p.run(ctx, "heff"), ref)
    ctx.close()


@pytest.mark.parametrize("call", CALLS)
def test_repeated_calls_give_the_same_bits(b, call):
    p = Problem(b, *_bonds(b, (80, 95, 97, 113, 2, 3, 255), 1), seed=4)
    ctx = b.dmrg3s_create(0, 1 << 30)
    ref = p.run(ctx, call)
    for _ in range(10):
        assert torch.equal(p.run(ctx, call), ref)
    ctx.close()

"""Plans found again: a structure's tables are built when a call in a precision first
needs them, and a one-shot call finds its plan by its arguments' contents.  So the
order of the precisions must not matter, an argument changed in place must be
seen, and a call that is refused must not disturb the next one.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from test_gpu_sliced import XXZ_QP, XXZ_T, XXZ_W, Problem, _bonds  # noqa: E402

DIMS = (128, 127, 129, 16)


@pytest.fixture(scope="module")
def b():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1501_05504_gb300 import binding
    binding.slib()
    return binding


def _apply(b, ctx, p, prec, stream=None):
    out = b.empty_site_like(p.qp, p.left, p.right)
    b.dmrg3s_apply_heff(ctx, p.L, p.W, p.R, p.M, out, prec, stream)
    b.dmrg3s_sync(ctx, stream)
    return out.data.clone()


def _fresh(b, p, prec):
    ctx = b.dmrg3s_create(0, 1 << 30)
    x = _apply(b, ctx, p, prec)
    ctx.close()
    return x


@pytest.mark.parametrize("order", [("tf32x3", "fp64", "tf32"), ("fp64", "tf32", "tf32x3"), ("tf32", "tf32x3", "fp64")])
def test_order_of_the_precisions(b, order):
    p = Problem(b, *_bonds(b, DIMS, 1), seed=40)
    ctx = b.dmrg3s_create(0, 1 << 30)
    for prec in order + order:
        assert torch.equal(_apply(b, ctx, p, prec), _fresh(b, p, prec))
        op = b.HeffOp(ctx, p.L, p.W, p.R, p.M, prec)
        out = b.empty_site_like(p.qp, p.left, p.right)
        op.apply(p.M, out)
        b.dmrg3s_sync(ctx)
        assert torch.equal(out.data, _fresh(b, p, prec))
        op.close()
    ctx.close()


def test_arguments_changed_in_place(b):
    W = XXZ_W.copy()
    p = Problem(b, *_bonds(b, DIMS, 1), W=W, seed=41)
    ctx = b.dmrg3s_create(0, 1 << 30)
    first = _apply(b, ctx, p, "fp64")
    p.W.W[1, 0, 1, 0] = 0.25                      # an MPO entry
    second = _apply(b, ctx, p, "fp64")
    assert not torch.equal(first, second)
    assert torch.equal(second, _fresh(b, p, "fp64"))
    q = Problem(b, *_bonds(b, DIMS, 1), W=p.W.W, seed=41)
    q.left.dim[3] = 15                            # a dimension, and what follows from it
    q.L, q.M = b.Env(XXZ_T, q.left), b.Site(XXZ_QP, q.left, q.right)
    q.L.data, q.M.data = p.L.data[:q.L.size()].clone(), p.M.data[:q.M.size()].clone()
    assert torch.equal(_apply(b, ctx, q, "fp64"), _fresh(b, q, "fp64"))
    p.W.W[1, 0, 1, 0] = XXZ_W[1, 0, 1, 0]
    assert torch.equal(_apply(b, ctx, p, "fp64"), first)
    ctx.close()


def test_refused_calls_after_a_good_one(b):
    p = Problem(b, *_bonds(b, DIMS, 1), seed=42)
    ctx = b.dmrg3s_create(0, 1 << 30)
    first = _apply(b, ctx, p, "fp64")
    keep = p.W.W[0, 0, 4, 1]
    for value, status in ((1.0, None), (np.nan, None)):       # breaks the charges; not a number
        p.W.W[0, 0, 4, 1] = value
        with pytest.raises(b.Dmrg3sError):
            _apply(b, ctx, p, "fp64")
    p.W.W[0, 0, 4, 1] = keep
    data, p.R.data = p.R.data, None                           # no data
    with pytest.raises(b.Dmrg3sError):
        _apply(b, ctx, p, "fp64")
    p.R.data = data
    assert torch.equal(_apply(b, ctx, p, "fp64"), first)
    ctx.close()


@pytest.mark.parametrize("prec", ["fp64", "tf32x3"])
def test_on_a_stream_behind_the_callers_kernel(b, prec):
    """The first launch of a call may start early; its reads must wait all the same."""
    p = Problem(b, *_bonds(b, DIMS, 1), seed=43)
    ref = _fresh(b, p, prec)
    ctx = b.dmrg3s_create(0, 1 << 30)
    _apply(b, ctx, p, prec)
    st = torch.cuda.Stream()
    src = p.M.data.clone()
    big = torch.randn(4096, 4096, device="cuda")
    for _ in range(5):
        p.M.data.zero_()
        torch.cuda.synchronize()
        out = b.empty_site_like(p.qp, p.left, p.right)
        with torch.cuda.stream(st):
            for _ in range(4):
                big = big @ big / 64.0                        # keeps the stream busy
            p.M.data.copy_(src)
            b.dmrg3s_apply_heff(ctx, p.L, p.W, p.R, p.M, out, prec, st)
        st.synchronize()
        assert torch.equal(out.data, ref)
    ctx.close()


@pytest.mark.parametrize("prec", ["fp64", "tf32x3"])
def test_captured_call_replays(b, prec):
    """A structure planned before can be captured; the replays see the tensors' contents."""
    p = Problem(b, *_bonds(b, DIMS, 1), seed=44)
    ctx = b.dmrg3s_create(0, 1 << 30)
    first = _apply(b, ctx, p, prec)
    out = b.empty_site_like(p.qp, p.left, p.right)
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        b.dmrg3s_apply_heff(ctx, p.L, p.W, p.R, p.M, out, prec)
    g.replay()
    torch.cuda.synchronize()
    assert torch.equal(out.data, first)
    p.M.data.mul_(-2.0)
    g.replay()
    torch.cuda.synchronize()
    replayed = out.data.clone()
    assert torch.equal(replayed, _apply(b, ctx, p, prec))
    ctx.close()


@pytest.mark.parametrize("call", ("heff", "expand+", "env-"))
def test_first_call_on_a_stream_of_its_own(b, call):
    """The plan's tables are on the device before a stream that does not wait for the
    default stream reads them: first calls on new structures, one after the other."""
    st = torch.cuda.Stream()
    for k in range(12):
        dims = (120 + k, 127, 129 - k, 16)
        p = Problem(b, *_bonds(b, dims, 1), seed=45)
        torch.cuda.synchronize()
        ref_ctx, ctx = b.dmrg3s_create(0, 1 << 29), b.dmrg3s_create(0, 1 << 29)
        p.run(ref_ctx, call)
        ref = p.run(ref_ctx, call)                # (tables long in place)
        with torch.cuda.stream(st):
            got = p.run(ctx, call)
        assert torch.equal(got, ref)
        ctx.close()
        ref_ctx.close()

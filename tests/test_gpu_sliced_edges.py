"""The sliced FP64 form at the edges of its tiles (16 columns, 64 k, 128 rows), beside
sectors large enough that every call takes that form.  Tolerance as in
test_gpu_sliced.py."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from test_gpu_sliced import CALLS, TOL, Problem, _bonds, _both, _rel  # noqa: E402

# (small sectors next to the large ones: they meet in every kind of block)
EDGES = [(15, 31, 33, 256, 240, 47, 48, 49), (64, 65, 63, 257, 250, 1, 2), (16, 17, 300, 230, 32, 80, 79, 81)]


@pytest.fixture(scope="module")
def b():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1501_05504_gb300 import binding
    binding.lib()
    return binding


@pytest.mark.parametrize("call", CALLS)
@pytest.mark.parametrize("dims,shift", [(d, s) for d in EDGES for s in (0, 1)])
def test_every_call_in_both_forms(b, dims, shift, call):
    p = Problem(b, *_bonds(b, dims, shift), seed=len(dims) + shift)
    x, y, counts = _both(b, p, call)
    assert counts[0] != counts[1]                  # two forms ran
    assert _rel(x, y) < TOL

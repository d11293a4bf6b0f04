"""The reciprocal and the square root of csrc/fp64.cuh against CUDA's correctly rounded
ones, over their documented ranges and at the ends of the mantissa.

Bound: one unit in the last place of the rounded value.  What is left out is below
2^-63 (recip: the cube of an FP32 reciprocal's error; sqrt_of: the product of two
2^-43 errors), and the last multiply-add rounds once, half a unit; the rounded value
itself is half a unit from the exact one, so the two are neighbours at most.
"""
import ctypes
import os
import shutil
import subprocess

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SOURCE = r"""
#include <cuda_runtime.h>
#include "fp64.cuh"
__global__ void k(const double* x, double* a, double* b, int n, int root) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  a[i] = root ? dmrg3s::sqrt_of(x[i]) : dmrg3s::recip(x[i]);
  b[i] = root ? __dsqrt_rn(x[i]) : __drcp_rn(x[i]);
}
extern "C" int run(const double* x, double* a, double* b, int n, int root) {
  k<<<(n + 255) / 256, 256>>>(x, a, b, n, root);
  return (int)cudaDeviceSynchronize();
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    d = tmp_path_factory.mktemp("fp64")
    src, out = d / "helpers.cu", d / "helpers.so"
    src.write_text(SOURCE)
    subprocess.run([nvcc, "-O3", "-std=c++17", "-shared", "-Xcompiler", "-fPIC", "-gencode",
                    "arch=compute_103a,code=sm_103a", "-I" + os.path.join(ROOT, "paper_1501_05504_gb300", "csrc"),
                    str(src), "-o", str(out)], check=True)
    lb = ctypes.CDLL(str(out))
    lb.run.argtypes = [ctypes.c_void_p] * 3 + [ctypes.c_int, ctypes.c_int]
    return lb


@pytest.mark.parametrize("root,top", [(0, 1000), (1, 999)])
def test_within_one_unit(lib, root, top):
    rng = np.random.default_rng(70 + root)
    n = 4_000_000
    e = rng.integers(-1000 if not root else -1021, top, n)
    m = rng.uniform(1.0, 2.0, n)
    edge = 1.0 + np.concatenate([np.arange(64), 2 ** 52 - 1 - np.arange(64), 2 ** np.arange(52)]) * 2.0 ** -52
    m[:edge.size] = edge
    m[edge.size:2 * edge.size] = edge
    e[:2 * edge.size] = np.repeat([0, 1], edge.size)
    x = np.ldexp(m, e)
    if not root:
        x *= rng.choice([-1.0, 1.0], n)
    dx = torch.from_numpy(x).cuda()
    a, b = torch.empty_like(dx), torch.empty_like(dx)
    assert lib.run(dx.data_ptr(), a.data_ptr(), b.data_ptr(), n, root) == 0
    ulp = (a.view(torch.int64) - b.view(torch.int64)).abs().max()
    assert int(ulp) <= 1

"""The square roots of the pair kernels (csrc/entry_blocks.cuh) against correctly rounded ones."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

pytestmark = pytest.mark.gpu
SRC = """
#include "entry_blocks.cuh"
__global__ void k(const double* x, int n, double* r, double* a, double* s) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  a[i] = rsqrt3_any(x[i]);
  r[i] = x[i] >= 0x1p-1000 && x[i] <= 0x1p1000 ? rsqrt3(x[i]) : a[i];
  s[i] = sqrt_from(x[i], r[i]);
}
extern "C" int roots(const double* x, int n, double* r, double* a, double* s) {
  k<<<(n + 255) / 256, 256>>>(x, n, r, a, s);
  return cudaDeviceSynchronize();
}
"""


@pytest.fixture(scope="module")
def roots(tmp_path_factory):
    from paper_2607_00790_gb300 import build
    d = tmp_path_factory.mktemp("roots")
    (d / "roots.cu").write_text(SRC)
    so = str(d / "roots.so")
    subprocess.run([build.nvcc(), *build.ARCH, *build.NVCC_FLAGS, "-shared", "-I", build.CSRC,
                    "-I", os.path.join(os.path.dirname(build.HERE), "include"), "-o", so, str(d / "roots.cu")], check=True)
    f = ctypes.CDLL(so).roots
    f.argtypes = [ctypes.c_void_p, ctypes.c_int] + 3 * [ctypes.c_void_p]

    def run(x):
        import torch
        t = torch.as_tensor(x, device="cuda")
        o = [torch.empty_like(t) for _ in range(3)]
        assert f(t.data_ptr(), t.numel(), *[v.data_ptr() for v in o]) == 0
        return [v.cpu().numpy() for v in o]

    return run


def arguments():
    """Every scale that the pair kernels admit (r^2 between 1e-290 and 1e290), squares and their neighbours,
    mantissas all over [1, 4)."""
    rng = np.random.default_rng(0)
    m = rng.integers(1, 2**26, 50000).astype(float)
    sq = m * m
    return np.concatenate([10.0 ** rng.uniform(-290, 290, 200000), 1 + 3 * rng.random(200000), sq, np.nextafter(sq, 0),
                           np.nextafter(sq, np.inf), 2.0 ** np.arange(-960, 961), np.nextafter(2.0 ** np.arange(-960, 961), 0)])


def test_square_root_is_correctly_rounded(roots):
    x = arguments()
    assert np.array_equal(roots(x)[2], np.sqrt(x))


def test_reciprocal_square_root_to_an_ulp(roots):
    """Seed and series leave 2^-60; the step rounds e (relative 2^-53 of a 2^-21 correction), the factor
    and the sum: half an ulp of the result and a little, below one."""
    x = arguments()
    r, a, _ = roots(x)
    one = np.longdouble(1) / np.sqrt(x.astype(np.longdouble))
    ulp = np.spacing(np.asarray(one, dtype=float)).astype(np.longdouble)
    assert np.max(np.abs(r.astype(np.longdouble) - one) / ulp) <= 1
    assert np.array_equal(a, r)


def test_reciprocal_square_root_of_any_argument(roots):
    """Subnormal, huge and infinite ones."""
    x = np.array([5e-324, 1e-310, 2.2e-308, 1e-300, 1e300, 1.7e308, np.inf])
    a = roots(x)[1]
    with np.errstate(divide="ignore"):
        assert np.all(np.abs(a - 1 / np.sqrt(x)) <= 2 * np.spacing(1 / np.sqrt(x)))

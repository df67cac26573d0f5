"""Where the product from residues is taken, and the edges of its tiles, K blocks, accumulation chunks and
pieces at sizes where it is."""
import ctypes

import numpy as np
import pytest

from test_gpu_crt_gemm import check, rand_c

pytestmark = pytest.mark.gpu


def fits(m, n, k):
    from paper_2607_00790_gb300 import binding
    f = ctypes.CDLL(binding.LIB_PATH)["_Z19wsbm_zgemm_crt_fitsiii"]
    f.restype = ctypes.c_bool
    return f(m, n, k)


def test_rule():
    """As measured on 152 SMs: the digit product is the faster one of the first list, the residues of the second."""
    import torch
    if torch.cuda.get_device_properties(0).multi_processor_count != 152:
        pytest.skip("measured on 152 SMs")
    for k in (160, 256, 512, 1000):
        for m, n in ((512, 512), (768, 768), (1024, 1024), (1300, 1300), (512, 2000), (2000, 512), (700, 1500)):
            assert not fits(m, n, k), (m, n, k)
        for m, n in ((1200, 1200), (1600, 1600), (1800, 1800), (512, 3000), (3000, 1000), (1000, 3000), (8192, 8192)):
            assert fits(m, n, k), (m, n, k)
    assert not fits(8192, 8192, 159) and not fits(511, 8192, 256) and not fits(8192, 511, 256)


@pytest.mark.parametrize("m,n,k", [(1153, 1199, 160), (1153, 1200, 161), (1280, 1153, 191), (1281, 1151, 256), (1199, 1201, 257),
                                   (1160, 1180, 513), (1160, 1152, 1024), (1160, 1152, 1025), (1154, 1153, 2100)])
def test_edges(m, n, k):
    assert fits(m, n, k)
    rng = np.random.default_rng(m + n + k)
    A = rand_c(rng, (m, k)) * 10.0 ** rng.uniform(-6, 6, size=(m, 1))
    B = rand_c(rng, (k, n)) * 10.0 ** rng.uniform(-6, 6, size=(1, n))
    A[17] = 0
    B[:, 5] = 0
    C = rand_c(rng, (m, n))
    check(A, B, C, -1.0, 1.0, pad=3)


@pytest.mark.parametrize("alpha,beta", [(1.0, 0.0), (0.5 - 2.0j, -1.25 + 0.75j)])
def test_factors_and_scales(alpha, beta):
    rng = np.random.default_rng(4)
    A = rand_c(rng, (1200, 200)) * 10.0 ** rng.uniform(-130, 130, size=(1200, 1))
    B = rand_c(rng, (200, 1200)) * 10.0 ** rng.uniform(-130, 130, size=(1, 1200))
    check(A, B, rand_c(rng, (1200, 1200)), alpha, beta)
    A = rng.integers(-1000, 1000, size=(1200, 300)) + 1j * rng.integers(-1000, 1000, size=(1200, 300))
    B = rng.integers(-1000, 1000, size=(300, 1200)) + 1j * rng.integers(-1000, 1000, size=(300, 1200))
    from test_gpu_crt_gemm import product
    got = product(A.astype(complex), B.astype(complex), np.zeros((1200, 1200), dtype=complex), 1.0, 0.0)
    assert np.array_equal(got, (A @ B).astype(complex))

"""The product from residues (large zgemm) at the edges of its tiles, K blocks, accumulation chunks and
reconstruction pieces, against numpy's FP64 product at the bound of the digit-plane product; exact on
small integers; in strips when the allocator has no room for the whole work space."""
import ctypes

import numpy as np
import pytest

pytestmark = pytest.mark.gpu
EPS = np.finfo(np.float64).eps


def rand_c(rng, shape):
    return rng.standard_normal(shape) + 1j * rng.standard_normal(shape)


def product(A, B, C, alpha, beta, pad=0):
    """wsbm_zgemm on column-major storage with leading dimensions `pad` above the row counts."""
    import torch
    from paper_2607_00790_gb300 import binding
    m, k = A.shape
    n = B.shape[1]

    def dev(M):
        t = torch.full((M.shape[1], M.shape[0] + pad), complex(7.0, -3.0), dtype=torch.complex128, device="cuda")
        t[:, : M.shape[0]] = torch.as_tensor(M.T.copy(), device="cuda")
        return t

    tA, tB, tC = dev(A), dev(B), dev(C)
    two = lambda z: (ctypes.c_double * 2)(complex(z).real, complex(z).imag)  # noqa: E731
    rc = binding.lib().wsbm_zgemm(m, n, k, two(alpha), tA.data_ptr(), m + pad, tB.data_ptr(), k + pad, two(beta),
                                  tC.data_ptr(), m + pad, None)
    assert rc == 0
    out = tC.cpu().numpy()
    assert np.all(out[:, m:] == complex(7.0, -3.0))  # the padding is untouched
    return out[:, :m].T


def check(A, B, C, alpha, beta, **kw):
    got = product(A, B, C, alpha, beta, **kw)
    ref = alpha * (A @ B) + beta * C
    k = A.shape[1]
    ra = np.maximum(np.abs(A.real), np.abs(A.imag)).max(axis=1)
    cb = np.maximum(np.abs(B.real), np.abs(B.imag)).max(axis=0)
    bound = 8 * EPS * (2 * k * abs(alpha) * ra[:, None] * cb[None, :] + np.abs(ref) + np.abs(beta * C))
    assert np.all(np.abs(got - ref) <= bound), np.max(np.abs(got - ref) / bound)


@pytest.mark.parametrize("m,n,k", [(512, 512, 160), (513, 527, 161), (640, 575, 191), (767, 576, 256), (512, 577, 257),
                                   (600, 700, 513), (530, 520, 1024), (530, 520, 1025), (514, 512, 2100)])
def test_edges(m, n, k):
    rng = np.random.default_rng(m + n + k)
    A = rand_c(rng, (m, k)) * 10.0 ** rng.uniform(-6, 6, size=(m, 1))
    B = rand_c(rng, (k, n)) * 10.0 ** rng.uniform(-6, 6, size=(1, n))
    A[17] = 0
    B[:, 5] = 0
    C = rand_c(rng, (m, n))
    check(A, B, C, -1.0, 1.0, pad=3)


@pytest.mark.parametrize("alpha,beta", [(1.0, 0.0), (1.0, 1.0), (0.5 - 2.0j, -1.25 + 0.75j), (-1.0, 0.0)])
def test_factors(alpha, beta):
    rng = np.random.default_rng(3)
    check(rand_c(rng, (520, 300)), rand_c(rng, (300, 650)), rand_c(rng, (520, 650)), alpha, beta)


def test_extreme_scales():
    """Rows and columns of 10^+-130: results of 10^+-260 and sums of every size between."""
    rng = np.random.default_rng(4)
    A = rand_c(rng, (512, 200)) * 10.0 ** rng.uniform(-130, 130, size=(512, 1))
    B = rand_c(rng, (200, 512)) * 10.0 ** rng.uniform(-130, 130, size=(1, 512))
    check(A, B, np.zeros((512, 512), dtype=complex), 1.0, 0.0)


def test_exact_on_integers():
    rng = np.random.default_rng(5)
    A = rng.integers(-1000, 1000, size=(600, 300)) + 1j * rng.integers(-1000, 1000, size=(600, 300))
    B = rng.integers(-1000, 1000, size=(300, 530)) + 1j * rng.integers(-1000, 1000, size=(300, 530))
    got = product(A.astype(complex), B.astype(complex), np.zeros((600, 530), dtype=complex), 1.0, 0.0)
    assert np.array_equal(got, (A @ B).astype(complex))


def test_strips_when_memory_is_short():
    """An allocator that refuses the work space of one piece: the product runs in strips, with the same
    result bit for bit."""
    import torch
    from paper_2607_00790_gb300 import binding
    rng = np.random.default_rng(6)
    A, B, C = rand_c(rng, (2100, 256)), rand_c(rng, (256, 1900)), rand_c(rng, (2100, 1900))
    whole = product(A, B, C, -1.0, 1.0)
    held, asked = {}, []

    def alloc(nbytes, stream, ctx):
        asked.append(nbytes)
        if nbytes > 28 * (2100 + 2 * 1900) * 256 + (1 << 20):
            return None
        t = torch.empty(int(nbytes), dtype=torch.uint8, device="cuda")
        held[t.data_ptr()] = t
        return t.data_ptr()

    def free(ptr, stream, ctx):
        torch.cuda.synchronize()
        held.pop(ptr, None)

    cb = (binding._ALLOC_FN(alloc), binding._FREE_FN(free))
    assert binding.lib().wsbm_set_allocator(cb[0], cb[1], None) == 0
    try:
        got = product(A, B, C, -1.0, 1.0)
    finally:
        binding.use_torch_allocator(False)
    assert len(asked) == 2 and not held
    assert np.array_equal(got, whole)

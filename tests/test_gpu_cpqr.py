"""The column-pivoted QR of the interpolative decompositions, called batch-wise as the factor calls it."""
import ctypes

import numpy as np
import pytest

pytestmark = pytest.mark.gpu
EPS = np.finfo(np.float64).eps
DESC = np.dtype([("A", "u8"), ("lda", "i8"), ("m", "i4"), ("n", "i4"), ("kt", "i4"), ("pad", "i4"), ("tol", "f8"),
                 ("perm", "u8"), ("state", "u8"), ("norm2", "u8"), ("nref", "u8"), ("tauv", "u8"), ("betav", "u8"),
                 ("rdiag0", "u8")])  # QrDesc (csrc/dense.h)


def cpqr(mats, kt):
    """kt steps (mode 1) on each matrix of one batch: [(reduced matrix, perm, norm2, beta)]."""
    import torch
    from paper_2607_00790_gb300 import binding
    lib = ctypes.CDLL(binding.LIB_PATH)
    run = lib["_Z17wsbm_cpqr_batchedPK6QrDesciiiiP11CUstream_st"]
    run.argtypes = [ctypes.c_void_p] + 4 * [ctypes.c_int] + [ctypes.c_void_p]
    d, keep = np.zeros(len(mats), DESC), []
    for i, M in enumerate(mats):
        m, n = M.shape
        A = torch.as_tensor(np.ascontiguousarray(M.T), device="cuda")
        f64 = torch.zeros(3, n, dtype=torch.float64, device="cuda")
        beta = torch.zeros(n, dtype=torch.complex128, device="cuda")
        i32 = torch.zeros(n + 2, dtype=torch.int32, device="cuda")
        r0 = torch.zeros(1, dtype=torch.float64, device="cuda")
        d[i] = (A.data_ptr(), m, m, n, kt, 0, 0.0, i32.data_ptr() + 8, i32.data_ptr(), f64[0].data_ptr(),
                f64[1].data_ptr(), f64[2].data_ptr(), beta.data_ptr(), r0.data_ptr())
        keep.append((A, i32, f64, beta, r0))
    dd = torch.as_tensor(d.view(np.uint8), device="cuda")
    ms = [M.shape[0] for M in mats]
    small = sum(m <= lib["_Z18wsbm_cpqr_tpc_rowsv"]() for m in ms)
    torch.cuda.synchronize()
    assert run(dd.data_ptr(), len(mats), small, 1, max(ms), None) == 0
    torch.cuda.synchronize()
    assert all(k[1][0].item() == kt for k in keep)
    return [(k[0].cpu().numpy().T, k[1][2:].cpu().numpy(), k[2][0].cpu().numpy(), k[3].cpu().numpy()) for k in keep]


def graded(m, n):
    """One large common direction and parts of 1e-6 0.7^t beside it: the first step cancels 12 digits of
    every squared norm, and the pivots come in the order of t."""
    rng = np.random.default_rng(m)
    e = rng.standard_normal((m, n)) + 1j * rng.standard_normal((m, n))
    e /= np.linalg.norm(e, axis=0)
    A = e[:, :1] + 1e-6 * 0.7 ** np.arange(n) * e
    A[:, 0] = 1.001 * e[:, 0]
    return A


@pytest.mark.parametrize("m", [193, 300, 2100])
def test_norms_after_cancellation(m):
    """Remaining norms that are summed again, from the columns just written by other lanes."""
    n = 41
    A = graded(m, n)
    for kt in (1, 2, 7, 40):
        M, perm, norm2, beta = cpqr([A], kt)[0]
        assert np.array_equal(perm, np.arange(n))
        left = (np.abs(M[kt:, kt:]) ** 2).sum(0)
        # downdated since the last exact sum down to 1e-8 of it: eps / 1e-8 a step, 40 steps
        assert np.all(np.abs(norm2[kt:] - left) <= 40 * EPS / 1e-8 * left)
        R = np.linalg.qr(A, mode="r")
        assert np.all(np.abs(np.abs(beta[:kt]) - np.abs(np.diag(R))[:kt]) <= m * n * EPS)


@pytest.mark.parametrize("m", [150, 193, 300])
@pytest.mark.parametrize("other", [64, 2100, 12288, 12289])
def test_factor_does_not_depend_on_its_batch(m, other):
    """Beside a matrix that another kernel, or another width of the same kernel, takes."""
    A, B = graded(m, 41), graded(other, 6)
    alone, beside = cpqr([A], 6)[0], cpqr([A, B], 6)[0]
    for x, y in zip(alone, beside):
        assert np.array_equal(x, y)


@pytest.mark.parametrize("m", [193, 500, 800, 801])
def test_factor_in_a_large_batch(m):
    """Alone it has a cluster and narrow passes, among 300 a CTA and wide ones."""
    A = graded(m, 41)
    alone, many = cpqr([A], 17)[0], cpqr([A] * 300, 17)
    for got in (many[0], many[299]):
        for x, y in zip(alone, got):
            assert np.array_equal(x, y)

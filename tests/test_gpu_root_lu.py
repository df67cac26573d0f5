"""The large-matrix LU at the edges of its panels (one base panel, ragged last panels, more rows
than one CTA holds) and on columns with ties and zeros, against an elimination in numpy that picks
its pivots by the same rule."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
EPS = np.finfo(np.float64).eps


def key(col):
    """Pivot key: upper 32 bits of max(|Re|, |Im|)."""
    v = np.maximum(np.abs(col.real), np.abs(col.imag))
    return v.view(np.uint64) >> np.uint64(32)


def reference(A):
    A = A.copy()
    piv = np.empty(len(A), dtype=np.int32)
    for j in range(len(A)):
        p = piv[j] = j + int(np.argmax(key(A[j:, j].copy())))  # first row on ties
        A[[j, p]] = A[[p, j]]
        if A[j, j] == 0:
            A[j + 1:, j] = 0
            continue
        A[j + 1:, j] /= A[j, j]
        A[j + 1:, j + 1:] -= np.outer(A[j + 1:, j], A[j, j + 1:])
    return A, piv


def matrix(n, kind):
    rng = np.random.default_rng(n)
    A = rng.standard_normal((n, n)) + 1j * rng.standard_normal((n, n))
    if kind == "ties":  # equal moduli in every column: the first row has to win
        A = np.sign(A.real) + 1j * np.sign(A.imag) + 3.0 * np.tri(n, k=-1).T
    if kind == "zeros":
        A[:, n // 3] = 0
        A[n // 2] = 0
    return A


@pytest.mark.parametrize("kind", ["dense", "ties", "zeros"])
@pytest.mark.parametrize("n", [1, 2, 31, 32, 33, 64, 127, 129, 257, 385])
def test_panel_edges(n, kind):
    import torch
    from paper_2607_00790_gb300 import binding
    A = matrix(n, kind)
    LU, piv = binding.wsbm_lu_dense(torch.as_tensor(A, device="cuda"))
    LU, piv = LU.cpu().numpy(), piv.cpu().numpy()
    assert np.all(piv >= np.arange(n)) and np.all(piv < n)
    if kind == "dense":  # elsewhere rounding decides between equal or vanishing candidates
        assert np.array_equal(piv, reference(A)[1])
    elif kind == "ties":
        assert piv[0] == int(np.argmax(key(A[:, 0].copy())))
    L, U, PA = np.tril(LU, -1) + np.eye(n), np.triu(LU), A.copy()
    for j in range(n):
        PA[[j, piv[j]]] = PA[[piv[j], j]]
    assert np.linalg.norm(PA - L @ U) <= 50 * n * EPS * np.linalg.norm(A) * max(1.0, np.abs(U).max() / (np.abs(A).max() or 1.0))


def test_rows_over_every_cta():
    """5000 rows: 33 rows and more per CTA of the panel kernel; the product of the factors on random vectors."""
    import torch
    from paper_2607_00790_gb300 import binding
    n = 5000
    g = torch.Generator(device="cuda")
    g.manual_seed(1)
    A = torch.randn(n, n, dtype=torch.complex128, device="cuda", generator=g)
    LU, piv = binding.wsbm_lu_dense(A)
    perm = np.arange(n)
    for j, p in enumerate(piv.cpu().numpy()):
        perm[[j, p]] = perm[[p, j]]
    x = torch.randn(n, 4, dtype=torch.complex128, device="cuda", generator=g)
    y = torch.tril(LU, -1) @ (torch.triu(LU) @ x) + torch.triu(LU) @ x
    ref = (A @ x)[torch.as_tensor(perm, device="cuda")]
    growth = float(torch.triu(LU).abs().max() / A.abs().max())
    assert float((y - ref).norm() / ref.norm()) <= 50 * n * EPS * max(1.0, growth)
    assert float(torch.tril(LU, -1).abs().max()) <= 1.4143

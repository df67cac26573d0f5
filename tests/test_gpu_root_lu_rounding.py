"""How often the large-matrix LU rounds an entry at its own size: the diagonal of a second-kind system."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def test_diagonal_of_a_second_kind_system():
    """1/2 on the diagonal and small entries elsewhere: the pivots stay, the products are small, and only the
    subtractions round at the size of the diagonal.  Of its 32-column panel an entry takes the pivots two at a
    time, 8.5 subtractions on average, 1.5 of the updates within 128 columns and (n/128 - 1)/2 of the trailing
    ones: 12 roundings of ulp / sqrt(12) of a value on either side of 1/2 (ulp(1/2) or half of it):
    sqrt(12 / 12 * 5/8) = 0.8 ulp(1/2), with a margin of a quarter.  One subtraction per product has 36."""
    import torch
    from paper_2607_00790_gb300 import binding
    n = 640
    rng = np.random.default_rng(0)
    A = (rng.standard_normal((n, n)) + 1j * rng.standard_normal((n, n))) * (0.25 / np.sqrt(n))
    A[np.arange(n), np.arange(n)] += 0.5
    LU, piv = binding.wsbm_lu_dense(torch.as_tensor(A, device="cuda"))
    LU, PA = LU.cpu().numpy().astype(np.clongdouble), A.copy()
    for j, p in enumerate(piv.cpu().numpy()):
        PA[[j, p]] = PA[[p, j]]
    err = np.array([PA[i, i] - LU[i, i] - LU[i, :i] @ LU[:i, i] for i in range(n)]).astype(complex)
    assert np.sqrt((np.abs(err) ** 2).mean()) <= 1.0 * 2.0**-53

"""wsbm_zgemm whose result takes the place of an operand: the operands are read before it is written."""
import ctypes

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def in_place(m, n, k, over, off=0):
    """C on top of A or B (column `off` on) in one buffer, against the same product with a C of its own."""
    import torch
    from paper_2607_00790_gb300 import binding
    two = lambda r: (ctypes.c_double * 2)(r, 0.0)  # noqa: E731
    run = lambda A, B, C: binding.lib().wsbm_zgemm(m, n, k, two(1.0), A, ld, B, ld, two(0.0), C, ld, None)  # noqa: E731
    ld = max(m, k) + 5
    g = torch.Generator(device="cuda")
    g.manual_seed(m + n + k)
    A, B = (torch.randn(c, ld, dtype=torch.complex128, device="cuda", generator=g) for c in (k, n))
    big = torch.zeros((off + max(k, n) + n), ld, dtype=torch.complex128, device="cuda")
    X = A if over == "A" else B
    big[:X.shape[0]] = X
    ref = torch.zeros(n, ld, dtype=torch.complex128, device="cuda")
    assert run(A.data_ptr(), B.data_ptr(), ref.data_ptr()) == 0
    C = big[off:off + n]
    a, b = (big, B) if over == "A" else (A, big)
    assert run(a.data_ptr(), b.data_ptr(), C.data_ptr()) == 0
    got, want = C[:, :m].cpu().numpy(), ref[:, :m].cpu().numpy()
    # the same integers by either form of the product: 2^-53 of k terms of a row's and a column's largest
    scale = 2 * k * float(A.abs().max() * B.abs().max())
    assert np.abs(got - want).max() <= 8 * np.finfo(np.float64).eps * scale


@pytest.mark.parametrize("over", ["A", "B"])
@pytest.mark.parametrize("m,n,k,off", [(2100, 2000, 256, 0), (1100, 2100, 1100, 0), (1100, 2100, 1100, 7), (1500, 2000, 1030, 1029)])
def test_in_place(m, n, k, off, over):
    in_place(m, n, k, over, off)


def test_strips_in_place():
    """With room for strips only."""
    import torch
    from paper_2607_00790_gb300 import binding
    m, n, k, held, asked = 2100, 1900, 256, {}, []

    def alloc(nbytes, stream, ctx):
        asked.append(nbytes)
        if nbytes > 28 * (m + 2 * n) * k + (1 << 20):
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
        in_place(m, n, k, "B")
    finally:
        binding.use_torch_allocator(False)
    assert len(asked) == 4 and not held

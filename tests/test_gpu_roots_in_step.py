"""Several roots factored in step have the factors that each has alone, also with little memory."""
import ctypes

import numpy as np
import pytest

pytestmark = pytest.mark.gpu
DESC = np.dtype([("A", "u8"), ("lda", "i8"), ("piv", "u8"), ("n", "i4"), ("pad", "i4")])  # LuDesc (csrc/dense.h)


def in_step(mats):
    import torch
    from paper_2607_00790_gb300 import binding
    lib, vp, i32 = ctypes.CDLL(binding.LIB_PATH), ctypes.c_void_p, ctypes.c_int
    run = lib["_Z17wsbm_lu_big_multiPK6LuDesciPvP11CUstream_st"]
    run.argtypes = [vp, i32, vp, vp]
    most = lib["_Z21wsbm_lu_big_multi_maxPK6LuDesci"]
    most.argtypes = [vp, i32]
    size = lib["_Z26wsbm_lu_big_multi_ws_bytesPK6LuDesci"]
    size.argtypes, size.restype = [vp, i32], ctypes.c_size_t
    d, A, P = np.zeros(len(mats), DESC), [], []
    for i, M in enumerate(mats):
        n = len(M)
        A.append(torch.as_tensor(np.ascontiguousarray(M.T), device="cuda"))
        P.append(torch.zeros(n, dtype=torch.int32, device="cuda"))
        d[i] = (A[i].data_ptr(), n, P[i].data_ptr(), n, 0)
    assert most(d.ctypes.data, len(mats)) == len(mats)
    ws = torch.empty(size(d.ctypes.data, len(mats)) + 256, dtype=torch.uint8, device="cuda")
    assert run(d.ctypes.data, len(mats), (ws.data_ptr() + 255) // 256 * 256, None) == 0
    torch.cuda.synchronize()
    return [(a.cpu().numpy().T, p.cpu().numpy()) for a, p in zip(A, P)]


@pytest.mark.parametrize("sizes", [[1], [2, 1], [700, 513, 640, 161, 129, 128, 127, 97, 96, 65, 64, 63, 33, 32, 31, 1], [600, 600, 600],
                                   [2500, 130, 70], [3000, 1], [1100, 1099, 1025, 1024, 1023, 900, 545, 512]])
def test_as_alone(sizes):
    import torch
    from paper_2607_00790_gb300 import binding
    sizes = sorted(sizes, reverse=True)
    rng = np.random.default_rng(len(sizes))
    mats = [rng.standard_normal((n, n)) + 1j * rng.standard_normal((n, n)) for n in sizes]
    for M, (LU, piv) in zip(mats, in_step(mats)):
        LU1, piv1 = binding.wsbm_lu_dense(torch.as_tensor(M, device="cuda"))
        assert np.array_equal(piv, piv1.cpu().numpy()) and np.array_equal(LU, LU1.cpu().numpy())


def test_fewer_in_step_when_memory_is_short():
    """An allocator that has the work space of one root only: the same factors, so the same solutions."""
    import torch
    from paper_2607_00790_gb300 import binding, inputs
    made, params, rhs = [], [], []
    for N in (700, 800, 900, 1000, 1100):
        c = inputs.star(N)
        made.append(binding.make_geom(c))
        params.append(binding.make_params(float(inputs.k0_for_density(c)), 1.5, leaf=64, nproxy=64, id_tol=1e-10))
        rhs.append(torch.randn(2, 2 * N, dtype=torch.complex128, device="cuda").T)

    def solve():
        b = binding.Batch([g for g, _ in made], params)
        b.factor()
        x = [torch.cat(uq).cpu().numpy() for uq in b.solve(rhs)]
        n = sorted((b.solver(i).stats()["root_size"] for i in range(len(made))), reverse=True)
        b.close()
        return x, n

    want, roots = solve()
    assert roots[-1] >= 512
    size = ctypes.CDLL(binding.LIB_PATH)["_Z26wsbm_lu_big_multi_ws_bytesPK6LuDesci"]
    size.argtypes, size.restype = [ctypes.c_void_p, ctypes.c_int], ctypes.c_size_t
    d = np.zeros(len(roots), DESC)
    d["n"] = roots
    need = {k: size(d.ctypes.data, k) for k in (1, 2, 3, 5)}
    held, seen = {}, []

    def alloc(nbytes, stream, ctx):
        if nbytes in (need[2], need[3], need[5]):
            seen.append(nbytes)
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
        got, _ = solve()
    finally:
        binding.use_torch_allocator(False)
    assert seen == [need[5], need[3], need[2]]
    assert all(np.array_equal(a, b) for a, b in zip(got, want))

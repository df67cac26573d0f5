"""A column of a product or a field has the same bits whatever the columns beside it."""
import numpy as np
import pytest

from paper_2607_00790_gb300 import binding, inputs

pytestmark = pytest.mark.gpu


def _t(a):
    import torch
    return torch.as_tensor(np.ascontiguousarray(a), device="cuda")


def problem(N, *shape):
    c = inputs.star(N)
    k0 = float(inputs.k0_for_density(c))
    g, keep = binding.make_geom(c)
    rng = np.random.default_rng(N)
    z = rng.standard_normal(shape) + 1j * rng.standard_normal(shape)
    return g, keep, binding.make_params(k0, 1.5), z, rng


COUNTS = [1, 2, 3, 4, 5, 7, 8, 9, 10, 12]


@pytest.mark.parametrize("trans", [False, True])
@pytest.mark.parametrize("N", [100, 300, 5000, 20000])
def test_matvec_columns(N, trans):
    g, keep, p, x, _ = problem(N, 2 * N, 12)
    full = binding.wsbm_matvec(g, p, _t(x), trans).cpu().numpy()
    for n in COUNTS:
        assert np.array_equal(binding.wsbm_matvec(g, p, _t(x[:, :n]), trans).cpu().numpy(), full[:, :n]), n


def test_matvec_with_little_memory():
    """An allocator that has room for one column at a time: the same bits."""
    import torch
    N = 3000
    g, keep, p, x, _ = problem(N, 2 * N, 9)
    full = binding.wsbm_matvec(g, p, _t(x), False).cpu().numpy()
    held, asked = {}, []

    def alloc(nbytes, stream, ctx):
        asked.append(nbytes)
        if len(asked) < 4:
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
        got = binding.wsbm_matvec(g, p, _t(x), False).cpu().numpy()
    finally:
        binding.use_torch_allocator(False)
    assert asked == [asked[3] * f for f in (8, 4, 2, 1)] and not held
    assert np.array_equal(got, full)


@pytest.mark.parametrize("N,nt", [(300, 70), (5000, 129), (20000, 1000)])
def test_field_columns(N, nt):
    g, keep, p, z, rng = problem(N, 2, N, 12)
    t, s = rng.uniform(0, 2 * np.pi, nt), rng.uniform(0.2, 3.0, nt)
    r = s * (1 + 0.3 * np.cos(5 * t))
    pts = _t(r * np.cos(t)), _t(r * np.sin(t))
    full = binding.field(g, p, _t(z[0]), _t(z[1]), *pts)[0].cpu().numpy()
    for n in COUNTS:
        got = binding.field(g, p, _t(z[0, :, :n]), _t(z[1, :, :n]), *pts)[0].cpu().numpy()
        assert np.array_equal(got, full[:, :n]), n

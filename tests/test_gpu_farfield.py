"""Far field of many right-hand sides, which runs as a tensor-core product: values that its digits cannot
hold, and waits that run out."""
import numpy as np
import pytest

import oracle
from paper_2607_00790_gb300 import binding, inputs

pytestmark = pytest.mark.gpu
N, NRHS, NANG = 300, 200, 13


def _t(a):
    import torch
    return torch.as_tensor(np.ascontiguousarray(a), device="cuda")


@pytest.fixture(scope="module")
def solver():
    c = inputs.star(N)
    ph = oracle.Physics(inputs.k0_for_density(c), n=1.5)
    g, keep = binding.make_geom(c)
    s = binding.Solver(g, binding.make_params(ph.k0, 1.5))
    yield s
    s.close()


def densities():
    rng = np.random.default_rng(0)
    u, q = (rng.standard_normal((N, NRHS)) + 1j * rng.standard_normal((N, NRHS)) for _ in range(2))
    return u, q, rng.uniform(0, 2 * np.pi, NANG)


def test_infinities_and_nans(solver):
    """As the kernel of a few right-hand sides has them, column by column; the others as without them."""
    u, q, ang = densities()
    plain = solver.farfield(_t(u), _t(q), _t(ang)).cpu().numpy()
    u[5, 2] = np.nan
    q[299, 3] = complex(np.inf, 1.0)
    u[0, 7] = complex(1.0, -np.inf)
    q[128, 8] = complex(0.0, np.nan)
    u[17, 19] = 1e308  # times k0 it overflows, times k0 and a weight it does not
    wild = [2, 3, 7, 8, 19]
    got = solver.farfield(_t(u), _t(q), _t(ang)).cpu().numpy()
    one = np.stack([solver.farfield(_t(u[:, [c]]), _t(q[:, [c]]), _t(ang)).cpu().numpy()[:, 0] for c in wild], 1)
    np.testing.assert_array_equal(got[:, wild], one)
    assert not np.isfinite(got[:, wild[:4]]).any() and np.isfinite(got[:, 19]).all()
    tame = [c for c in range(NRHS) if c not in wild]
    assert np.array_equal(got[:, tame], plain[:, tame])


def test_angles_without_a_direction(solver):
    u, q, ang = densities()
    plain = solver.farfield(_t(u), _t(q), _t(ang)).cpu().numpy()
    ang[4], ang[12] = np.nan, np.inf
    got = solver.farfield(_t(u), _t(q), _t(ang)).cpu().numpy()
    rest = [a for a in range(NANG) if a not in (4, 12)]
    assert np.isnan(got[[4, 12]]).all() and np.array_equal(got[rest], plain[rest])


def test_a_wait_that_runs_out_is_reported(solver):
    """By the call whose product it may have cut short, and by no later one."""
    import ctypes

    import torch
    u, q, ang = densities()
    plain = solver.farfield(_t(u), _t(q), _t(ang)).cpu().numpy()
    lib = ctypes.CDLL(binding.LIB_PATH)
    assert lib["_Z19wsbm_tc_expire_waitP11CUstream_st"](None) == 0
    torch.cuda.synchronize()
    with pytest.raises(binding.WsbmError) as e:
        solver.farfield(_t(u), _t(q), _t(ang))
    assert e.value.code == -5  # WSBM_ERR_TIMEOUT
    assert np.array_equal(solver.farfield(_t(u), _t(q), _t(ang)).cpu().numpy(), plain)


def test_rule():
    """The product where it is the cheaper form (measured on 152 SMs), the kernel (one launch) elsewhere."""
    import ctypes

    import torch
    if torch.cuda.get_device_properties(0).multi_processor_count != 152:
        pytest.skip("measured on 152 SMs")
    count = ctypes.CDLL(binding.LIB_PATH)["_Z17wsbm_launch_countv"]
    count.restype = ctypes.c_int64
    for n in (256, 1024, 4096, 16384):
        c = inputs.star(n)
        g, keep = binding.make_geom(c)
        s = binding.Solver(g, binding.make_params(float(inputs.k0_for_density(c)), 1.5))
        for nrhs, nang, product in ((1, 360, False), (8, 360, False), (8, 8, n > 2048), (16, 36, n > 2048), (16, 360, n > 2048),
                                    (64, 8, n > 256), (64, 360, True), (200, 8, True), (9, 7, False)):
            u = torch.ones(nrhs, n, dtype=torch.complex128, device="cuda").T
            a = torch.linspace(0, 6, nang, dtype=torch.float64, device="cuda")
            before = count()
            s.farfield(u, u, a)
            assert (count() - before > 1) == product, (n, nrhs, nang)
        s.close()


@pytest.mark.parametrize("n,nrhs,nang", [(256, 129, 8), (257, 200, 131), (300, 193, 9), (511, 65, 129), (1000, 64, 360)])
def test_product_at_its_edges(n, nrhs, nang):
    c = inputs.star(n)
    ph = oracle.Physics(inputs.k0_for_density(c), n=1.5)
    g, keep = binding.make_geom(c)
    rng = np.random.default_rng(nrhs)
    u, q = (rng.standard_normal((n, nrhs)) + 1j * rng.standard_normal((n, nrhs)) for _ in range(2))
    ang = rng.uniform(0, 2 * np.pi, nang)
    s = binding.Solver(g, binding.make_params(ph.k0, 1.5))
    got = s.farfield(_t(u), _t(q), _t(ang)).cpu().numpy()
    s.close()
    ref = oracle.farfield(c, ph, u, q, ang).reshape(got.shape)
    k0, w = ph.k0, c["w"][:, None]
    terms = (w * (k0 * np.abs(u) + np.abs(q))).sum(0) / np.sqrt(8 * np.pi * k0)
    # an ulp or two of the phase k0 r in each term on both sides, and the rounding of the product:
    # 2^-53 of a row's largest factor times a column's (about 16 times the mean product here)
    tol = np.finfo(np.float64).eps * (16 * k0 * np.hypot(c["x"], c["y"]).max() + 256)
    assert np.all(np.abs(got - ref) <= tol * terms)

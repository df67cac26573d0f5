"""Far field of many right-hand sides, which runs as a tensor-core product: values that its digits cannot
hold, and waits that run out."""
import numpy as np
import pytest

import oracle
from paper_2607_00790_gb300 import binding, inputs

pytestmark = pytest.mark.gpu
N, NRHS, NANG = 300, 20, 13


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

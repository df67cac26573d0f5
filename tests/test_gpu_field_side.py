"""Side of the targets of the field, whatever the size of the curve and its distance from the origin."""
import numpy as np
import pytest

import oracle
from paper_2607_00790_gb300 import binding, inputs

pytestmark = pytest.mark.gpu


def _t(a):
    import torch
    return torch.as_tensor(np.ascontiguousarray(a), device="cuda")


def problem(scale, shift, N=257, nt=300):
    """The star times `scale` at distance `shift`, targets from deep inside to far outside and close to the
    curve, and densities whose field does not depend on `scale`."""
    c = dict(inputs.star(N))
    k0 = float(inputs.k0_for_density(c))
    rng = np.random.default_rng(N)
    t = rng.uniform(0, 2 * np.pi, nt)
    s = np.concatenate([rng.uniform(0.1, 0.9, nt // 3), rng.uniform(1.1, 3.0, nt // 3), 1 + rng.uniform(-0.05, 0.05, nt - 2 * (nt // 3))])
    r = s * (1 + 0.3 * np.cos(5 * t))
    u, q = (rng.standard_normal((N, 2)) + 1j * rng.standard_normal((N, 2)) for _ in range(2))
    for k in ("x", "y"):
        c[k] = c[k] * scale + shift
    c["w"], c["kappa"] = c["w"] * scale, c["kappa"] / scale
    return c, k0 / scale, u, q / scale, r * np.cos(t) * scale + shift, r * np.sin(t) * scale + shift


def side_sums(c, px, py):
    """The Gauss sums in 64 bits: 1 inside, 0 outside, up to the quadrature error."""
    dx, dy = px[:, None] - c["x"], py[:, None] - c["y"]
    r = np.hypot(dx, dy)
    return -(c["w"] / r * (dx / r * c["nx"] + dy / r * c["ny"])).sum(1) / (2 * np.pi)


@pytest.mark.parametrize("scale,shift", [(1.0, 0.0), (1e20, 0.0), (3e18, 0.0), (1e30, 0.0), (1e-16, 0.0), (1e-20, 0.0),
                                         (1e-30, 0.0), (1.0, 1e13), (1e-20, 1e-7), (1e25, -1e35)])
def test_side_at_any_scale(scale, shift):
    c, k0, u, q, px, py = problem(scale, shift)
    g, keep = binding.make_geom(c)
    val, inside = binding.field(g, binding.make_params(k0, 1.5), _t(u), _t(q), _t(px), _t(py))
    sums = side_sums(c, px, py)
    clear = np.abs(sums - 0.5) > 1e-3  # rounding of the sums in 64 bits is far below this
    assert clear.sum() > 250
    assert np.array_equal(inside.cpu().numpy()[clear], sums[clear] > 0.5)
    if shift == 0.0:
        c1, k1, u1, q1, x1, y1 = problem(1.0, 0.0)
        ref, _ = oracle.field(c1, oracle.Physics(k1, n=1.5), u1, q1, x1, y1)
        far = np.arange(200)
        err = np.abs(val.cpu().numpy()[far] - ref[far]) / np.abs(ref[far]).max(axis=0)
        assert err.max() <= 1e-12

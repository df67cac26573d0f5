"""Kernels that are chosen by the form or the size of a call, at the edges of their ranges: index
lists in every order, 1 to 9 right-hand sides, ragged far-field products, and solutions of many
right-hand sides against the same taken one at a time."""
import numpy as np
import pytest

import oracle
from helpers import entry_scale
from paper_2607_00790_gb300 import binding, inputs

pytestmark = pytest.mark.gpu
EPS = np.finfo(np.float64).eps


def _t(a, dt=None):
    import torch
    return torch.as_tensor(np.ascontiguousarray(a), dtype=dt, device="cuda")


def normal(rng, *shape):
    return rng.standard_normal(shape) + 1j * rng.standard_normal(shape)


def star(N, **kw):
    c = inputs.star(N)
    ph = oracle.Physics(inputs.k0_for_density(c), n=1.5)
    g, keep = binding.make_geom(c)
    return c, ph, g, keep, binding.make_params(ph.k0, 1.5, **kw)


def lists(N, form):
    """Index lists of the 2N unknowns: u then q of the same nodes is the paired form."""
    nodes = np.arange(5, 72)
    pairs = np.concatenate([nodes, nodes + N])
    rng = np.random.default_rng(1)
    return {"paired": pairs, "q_first": np.concatenate([nodes + N, nodes]), "odd": pairs[:-1],
            "interleaved": np.stack([nodes, nodes + N], 1).ravel(), "u_only": nodes, "single": nodes[:1] + N,
            "shuffled": rng.permutation(pairs), "repeated": np.concatenate([pairs[:9], pairs[:9], pairs[-3:]]),
            "half_paired": np.concatenate([nodes, nodes[:40] + N, nodes[40:]])}[form]


FORMS = ["paired", "q_first", "odd", "interleaved", "u_only", "single", "shuffled", "repeated", "half_paired"]


@pytest.mark.parametrize("form", FORMS)
def test_entries_of_any_index_list(form):
    N = 97
    c, ph, g, keep, p = star(N)
    for other in ("paired", "shuffled", form):
        for rows, cols in ((lists(N, form), lists(N, other)), (lists(N, other), lists(N, form))):
            got = binding.wsbm_entries_raw(g, p, _t(rows), _t(cols)).cpu().numpy()
            # the tolerance of every entry parity test: 1e-12 of the terms that the entry adds up
            err = np.abs(got - oracle.wsbm_entries(c, ph, rows, cols)) / entry_scale(c, ph, rows, cols)
            assert err.max() <= 1e-12, (other, err.max())


@pytest.mark.parametrize("P", [1, 31, 65])
@pytest.mark.parametrize("form", FORMS)
def test_proxy_block_of_any_index_list(form, P):
    # the circle passes close to nodes outside the box and, with a small radius, close to the box's
    # own: arguments on both sides of the range of the fixed-point functions
    N = 97
    c, ph, g, keep, p = star(N)
    idx = lists(N, form)
    cx, cy, rho = oracle.proxy_circle(c, np.unique(idx % N))
    rho = rho or 0.1  # one node: its circle has no radius, which the call refuses
    for circ in ((cx, cy, rho), (cx, cy, 0.6 * rho)):
        for side, block in ((0, oracle.proxy_row_block), (1, oracle.proxy_col_block)):
            ref = block(c, ph, idx, circ, P)
            got = binding.wsbm_proxy_block(g, p, side, _t(idx), circ, P).cpu().numpy()
            # as the block parity tests: 1e-12 of the largest entry of the proxy point's line
            scale = np.abs(ref).max(axis=1 if side else 0, keepdims=True)
            assert got.shape == ref.shape and np.all(np.abs(got - ref) <= 1e-12 * scale), side


@pytest.mark.parametrize("trans", [False, True])
@pytest.mark.parametrize("nrhs", [1, 2, 3, 4, 5, 7, 8, 9])
def test_matvec_of_several_columns(nrhs, trans):
    N = 131
    c, ph, g, keep, p = star(N)
    idx = np.arange(2 * N)
    A, M = oracle.wsbm_dense(c, ph), entry_scale(c, ph, idx, idx)
    x = normal(np.random.default_rng(nrhs), 2 * N, nrhs)
    y = binding.wsbm_matvec(g, p, _t(x), trans).cpu().numpy()
    if trans:
        A, M = A.T, M.T
    # 1e-12 of each entry's terms, carried through the sum
    assert np.all(np.abs(y - A @ x) <= 1e-12 * (M @ np.abs(x)))


@pytest.mark.parametrize("nrhs", [1, 2, 3, 4, 5, 8, 9])
def test_field_of_several_columns(nrhs):
    N = 257
    c, ph, g, keep, p = star(N)
    rng = np.random.default_rng(nrhs)
    u, q = normal(rng, N, nrhs), normal(rng, N, nrhs)
    tt, ss = rng.uniform(0, 2 * np.pi, 67), rng.uniform(0.2, 3.0, 67)
    rad = ss * (1 + 0.3 * np.cos(5 * tt))
    # two targets one part in 1e7 on either side of a node: the side is decided in FP64
    far = np.abs(ss - 1) > 0.05
    near = 1 + np.array([-1e-7, 1e-7])
    px = np.concatenate([(rad * np.cos(tt))[far], c["x"][10] * near])
    py = np.concatenate([(rad * np.sin(tt))[far], c["y"][10] * near])
    val, inside = binding.field(g, p, _t(u), _t(q), _t(px), _t(py))
    ref, ref_in = oracle.field(c, ph, u, q, px, py)
    n = int(far.sum())
    assert np.array_equal(inside.cpu().numpy(), ref_in)
    err = np.abs(val.cpu().numpy()[:n] - ref[:n]) / np.abs(ref[:n]).max(axis=0)
    assert err.max() <= 1e-12


@pytest.mark.parametrize("N,nrhs,nang", [(255, 8, 8), (256, 8, 8), (257, 7, 33), (257, 8, 7), (257, 9, 131), (300, 64, 129),
                                         (300, 65, 9)])
def test_farfield_sums_and_products(N, nrhs, nang):
    c, ph, g, keep, p = star(N)
    rng = np.random.default_rng(nrhs)
    u, q = normal(rng, N, nrhs), normal(rng, N, nrhs)
    ang = rng.uniform(0, 2 * np.pi, nang)
    s = binding.Solver(g, p)
    got = s.farfield(_t(u), _t(q), _t(ang)).cpu().numpy()
    s.close()
    ref = oracle.farfield(c, ph, u, q, ang).reshape(got.shape)
    k0, w = ph.k0, c["w"][:, None]
    terms = (w * (k0 * np.abs(u) + np.abs(q))).sum(0) / np.sqrt(8 * np.pi * k0)
    # an ulp or two of the phase k0 r in each term on both sides, and the rounding of the product:
    # 2^-53 of a row's largest factor times a column's (about 16 times the mean product here)
    tol = EPS * (16 * k0 * np.hypot(c["x"], c["y"]).max() + 256)
    assert np.all(np.abs(got - ref) <= tol * terms)


@pytest.mark.parametrize("leaf", [64, 128])
def test_many_right_hand_sides_as_one_at_a_time(leaf):
    N = 1000
    c, ph, g, keep, p = star(N, leaf=leaf, nproxy=leaf, id_tol=1e-10)
    s = binding.Solver(g, p)
    s.factor()
    idx = _t(np.arange(2 * N))
    A = binding.wsbm_entries_raw(g, p, idx, idx).cpu().numpy()
    b = normal(np.random.default_rng(leaf), 2 * N, 65)
    for solve, M in ((s.solve, A), (s.solve_transposed, A.T)):
        one = np.concatenate([np.concatenate([t.cpu().numpy() for t in solve(_t(b[:, i:i + 1]))]) for i in range(65)], 1)
        for nrhs in (2, 7, 8, 9, 31, 33, 64, 65):
            x = np.concatenate([t.cpu().numpy() for t in solve(_t(b[:, :nrhs]))])
            d, y = x - one[:, :nrhs], np.abs(one[:, :nrhs])
            # both are backward stable: residuals of n eps of the terms each, with a margin for growth
            assert np.all(np.linalg.norm(M @ d, axis=0) <= 4 * 2 * N * EPS * np.linalg.norm(np.abs(M) @ y, axis=0)), nrhs
    s.close()

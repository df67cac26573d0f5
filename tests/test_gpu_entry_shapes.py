"""Entries by index lists of every shape: few rows by many columns, the reverse, and short lists, whose tiles
are laid out differently."""
import numpy as np
import pytest

import oracle
from helpers import entry_scale
from paper_2607_00790_gb300 import binding, inputs

pytestmark = pytest.mark.gpu
N = 211


def _t(a):
    import torch
    return torch.as_tensor(np.ascontiguousarray(a), device="cuda")


def lists(form, n, seed):
    """n unknowns: scattered, or u and then q of the same nodes (odd n: the last q left out)."""
    rng = np.random.default_rng(seed)
    if form == "scattered":
        return rng.permutation(2 * N)[:n]
    nodes = rng.permutation(N)[: (n + 1) // 2]
    return np.concatenate([nodes, nodes + N])[:n]


@pytest.mark.parametrize("form", ["scattered", "paired"])
@pytest.mark.parametrize("nr,nc", [(1, 1), (1, 400), (2, 399), (3, 64), (7, 401), (8, 65), (9, 130), (62, 63), (62, 126), (63, 400),
                                   (64, 400), (65, 66), (400, 1), (401, 7), (130, 9)])
def test_shapes(nr, nc, form):
    c = inputs.star(N)
    ph = oracle.Physics(inputs.k0_for_density(c), n=1.5)
    g, keep = binding.make_geom(c)
    rows, cols = lists(form, nr, nr), lists(form, nc, nc + 1000)
    got = binding.wsbm_entries_raw(g, binding.make_params(ph.k0, 1.5), _t(rows), _t(cols)).cpu().numpy()
    # the tolerance of every entry parity test: 1e-12 of the terms that the entry adds up
    assert np.max(np.abs(got - oracle.wsbm_entries(c, ph, rows, cols)) / entry_scale(c, ph, rows, cols)) <= 1e-12

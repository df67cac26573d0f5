"""Small dense roots of a batch share their launches."""
import pytest

from paper_2607_00790_gb300 import binding, inputs

pytestmark = pytest.mark.gpu


def factor(N, count):
    c = inputs.star(N)
    k0 = float(inputs.k0_for_density(c))
    made = [binding.make_geom(c) for _ in range(count)]
    b = binding.Batch([g for g, _ in made], [binding.make_params(k0, 1.5, leaf=64, nproxy=64, id_tol=1e-10)] * count)
    b.factor()
    out = b.stats()["launches"], b.solver(0).stats()["root_size"]
    b.close()
    return out


@pytest.mark.parametrize("N", [700, 1024, 1600])
def test_launches_do_not_grow_with_the_roots(N):
    """Equal curves differ in nothing but their number: a root of its own chain would add at least the panel,
    the swap and the update of every 32 columns."""
    one, n = factor(N, 1)
    many, _ = factor(N, 6)
    assert 512 <= n < 2048
    assert many - one < 5 * 3 * (n // 32)

"""mars_autotune times the library's own plan too, so that a tuned solve is no slower than
an untuned one; small instances, whose plan has 128 or 256 threads a CTA."""
import numpy as np
import pytest

from paper_1907_05124_gb300 import instances as I

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    from paper_1907_05124_gb300 import mars
    with mars.Context(0) as c:
        yield c


def _fastest(ctx, inst, R, **kw):
    return min(ctx.solve(inst, R, 0.0, 4.0, seed=3, **kw).descent_seconds for _ in range(20))


@pytest.mark.parametrize("size,R", [(12, 64), (20, 256), (40, 300)])
def test_tuned_is_no_slower_than_untuned(ctx, size, R):
    inst = ctx.add_csr(*I.ea_lattice(size, 2, 1))
    want = ctx.solve(inst, R, 0.0, 4.0, seed=3)
    untuned = _fastest(ctx, inst, R)
    shape, seconds = ctx.autotune(inst, R, 0.0, 4.0, seed=3, repeats=20)
    # two fastest of twenty differ by 2 % here; the best of the other shapes is 15 % off at size 12
    assert seconds <= 1.08 * untuned and _fastest(ctx, inst, R) <= 1.08 * untuned
    got = ctx.solve(inst, R, 0.0, 4.0, seed=3)
    assert got.best_energy == want.best_energy and np.array_equal(got.energies, want.energies)
    ctx.set_shape(inst)
    ctx.set_shape(inst, **shape)  # what a user keeps can be set again
    assert ctx.get_shape(inst) == shape
    ctx.free(inst)

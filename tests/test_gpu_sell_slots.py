"""The number of slots per CTA that a sparse solve takes is about the faster one, also
where replicas take about as many sweeps each (fixed sweeps, a low k_max) and there
are more of them than one wave of one-slot CTAs."""
import pytest

from paper_1907_05124_gb300 import instances as I

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    from paper_1907_05124_gb300 import mars
    with mars.Context(0) as c:
        yield c


@pytest.mark.parametrize("R,kw", [(456, dict(fixed_sweeps=3)), (456, dict(k_max=25)), (512, dict(k_max=100)),
                                  (300, dict(k_max=100)), (320, dict())])
def test_the_faster_slots(ctx, R, kw):
    inst = ctx.add_csr(*I.er_graph(20000, 6, 4))

    def fastest(**shape):
        ctx.set_shape(inst, **shape)
        return min(ctx.solve(inst, R, 0.0, 6.0, seed=3, **kw).descent_seconds for _ in range(4))

    one, two = fastest(sell_rt=1), fastest(sell_rt=2)
    # the wrong one takes 1.1 to 1.4 times as long at these sizes, a rerun within 2 %
    assert fastest() <= 1.08 * min(one, two), (one, two)
    ctx.free(inst)

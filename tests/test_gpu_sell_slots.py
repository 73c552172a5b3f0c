"""The number of slots per CTA that a sparse solve takes is about the faster one, also
where replicas take about as many sweeps each (fixed sweeps, a low k_max) and there
are more of them than one wave of one-slot CTAs; and so is the number of threads where
the couplings are read through the L1."""
import numpy as np
import pytest

from paper_1907_05124_gb300 import instances as I

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    from paper_1907_05124_gb300 import mars
    with mars.Context(0) as c:
        yield c


@pytest.mark.parametrize("n,R,kw", [(20000, 456, dict(fixed_sweeps=3)), (20000, 456, dict(k_max=25)),
                                    (20000, 512, dict(k_max=100)), (20000, 300, dict(k_max=100)),
                                    (20000, 320, dict()), (600, 512, dict(k_max=100)), (2000, 512, dict(k_max=100))])
def test_the_faster_slots(ctx, n, R, kw):
    inst = ctx.add_csr(*I.er_graph(n, 6, 4))

    def fastest(**shape):
        ctx.set_shape(inst, **shape)
        return min(ctx.solve(inst, R, 0.0, 6.0, seed=3, **kw).descent_seconds for _ in range(4))

    one, two = fastest(sell_rt=1), fastest(sell_rt=2)
    # the wrong one takes 1.1 to 1.4 times as long at these sizes, a rerun within 2 %
    assert fastest() <= 1.08 * min(one, two), (one, two)
    ctx.free(inst)


@pytest.mark.parametrize("n,degree,R", [(2000, 12, 64), (2000, 12, 320), (1000, 12, 64), (2000, 20, 64)])
def test_general_couplings_take_the_faster_threads(ctx, n, degree, R):
    g = I.er_graph(n, degree, 4)
    rows = np.repeat(np.arange(n), np.diff(g.row_ptr)).astype(np.int64)
    pair = np.minimum(rows, g.col) * n + np.maximum(rows, g.col)
    edges, of = np.unique(pair, return_inverse=True)
    inst = ctx.add_csr(g.row_ptr, g.col, np.random.default_rng(1).normal(size=len(edges))[of])

    def fastest(**shape):
        ctx.set_shape(inst, **shape)
        return min(ctx.solve(inst, R, 0.0, 2.0 * degree ** 0.5 + 1.0, seed=3).descent_seconds for _ in range(4))

    assert fastest() <= 1.08 * min(fastest(sell_threads=nt) for nt in (256, 512, 1024))
    ctx.free(inst)

"""Every shape of the sliced-ELL kernels (threads, slots, coupling formats,
unrolled and general degrees) returns what the default returns, and the
default what the CSR walk's order gives: whole solves with identical outputs
on odd and even sizes, irregular degrees (odd slice degrees leave half a word
of padding), fields and general weights. The default's fixed-sweep
trajectories are held to the oracle elsewhere."""
import numpy as np
import pytest

from paper_1907_05124_gb300 import instances as I

pytestmark = pytest.mark.gpu

KEYS = ("energies", "spins", "m_final", "replica_sweeps", "replica_levels", "replica_capped")


@pytest.fixture(scope="module")
def ctx():
    from paper_1907_05124_gb300 import mars
    with mars.Context(0) as c:
        yield c


def _instance(name):
    if name == "square":
        return I.ea_lattice(13, 2, 1), None  # degree 4, odd side: three colours
    if name == "cubic":
        return I.ea_lattice(8, 3, 2), None   # degree 6
    if name == "field":
        return I.ea_lattice(12, 2, 3), np.random.default_rng(3).integers(-2, 3, 144).astype(float)
    g = I.er_graph(301, 9, 4)                # degrees 1 to about 20
    if name == "graph":
        return g, None
    w = np.random.default_rng(5).normal(size=g.nnz)
    rows = np.repeat(np.arange(g.n), np.diff(g.row_ptr))
    key = {(min(r, c), max(r, c)): x for r, c, x in zip(rows, g.col, w)}
    return I.Csr(g.row_ptr, g.col, [key[min(r, c), max(r, c)] for r, c in zip(rows, g.col)]), None


@pytest.mark.parametrize("name", ["square", "cubic", "field", "graph", "weights"])
def test_shapes_agree(ctx, monkeypatch, name):
    g, h = _instance(name)
    inst = ctx.add_csr(*g, h=h)
    kw = dict(c_step=0.7, k_max=60, seed=11, outputs=("energies", "spins", "m_final", "sweeps", "levels", "capped"))
    want = ctx.solve(inst, 37, 0.0, 5.0, **kw)
    for rt in ("1", "2", "4"):
        for nt in ("128", "256", "512", "1024"):
            for tab in ("0", "1"):
                monkeypatch.setenv("MARS_SELL_RT", rt)
                monkeypatch.setenv("MARS_SELL_THREADS", nt)
                monkeypatch.setenv("MARS_SELL_SMEM_TABLE", tab)
                got = ctx.solve(inst, 37, 0.0, 5.0, **kw)
                for k in KEYS:
                    assert np.array_equal(getattr(got, k), getattr(want, k)), (rt, nt, tab, k)
    for k in ("MARS_SELL_RT", "MARS_SELL_THREADS", "MARS_SELL_SMEM_TABLE"):
        monkeypatch.delenv(k)
    monkeypatch.setenv("MARS_SELL_HALF_L1", "0")
    monkeypatch.setenv("MARS_SELL_SMEM_TABLE", "0")  # +-1 words (format 1)
    got = ctx.solve(inst, 37, 0.0, 5.0, **kw)
    for k in KEYS:
        assert np.array_equal(getattr(got, k), getattr(want, k)), k
    ctx.free(inst)


def test_last_slot_alone_and_refills(ctx):
    """Slots that run dry at different times: R below, at and above the slots."""
    inst = ctx.add_csr(*I.ea_lattice(10, 2, 6))
    for R in (1, 2, 3, 305, 700):
        a = ctx.solve(inst, R, 0.0, 4.0, seed=2, outputs=("energies", "sweeps"))
        ctx.set_shape(inst, sell_rt=4, sell_threads=512)
        b = ctx.solve(inst, R, 0.0, 4.0, seed=2, outputs=("energies", "sweeps"))
        ctx.set_shape(inst)
        assert np.array_equal(a.energies, b.energies) and np.array_equal(a.replica_sweeps, b.replica_sweeps)
    ctx.free(inst)

"""Repacking the live replicas of the level-synchronous sparse path into full
groups does not change a replica's results: whole solves whose replicas end at
different times, slot widths 2 and 4, a partly filled last group, and a
schedule of few levels (many replicas end at once), with and without it."""
import numpy as np
import pytest

from paper_1907_05124_gb300 import instances as I

pytestmark = pytest.mark.gpu

KEYS = ("energies", "spins", "m_final", "t0", "replica_sweeps", "replica_levels", "replica_capped")


@pytest.fixture(scope="module")
def ctx():
    from paper_1907_05124_gb300 import mars
    with mars.Context(0) as c:
        yield c


@pytest.mark.parametrize("rt,R", [(4, 33), (2, 33), (4, 130)])
@pytest.mark.parametrize("kw", [dict(k_max=50), dict(fixed_sweeps=3), dict(k_max=20, quench=True)])
def test_repacking_keeps_results(ctx, monkeypatch, rt, R, kw):
    inst = ctx.add_csr(*I.ea_lattice(39, 3, 1))  # 59319 spins: beyond shared memory
    ctx.set_shape(inst, sell_rt=rt)
    out = {}
    for on in ("0", "1"):
        monkeypatch.setenv("MARS_WIDE_REPACK", on)
        out[on] = ctx.solve(inst, R, 0.0, 6.0, c_step=0.2, seed=4,
                            outputs=("energies", "spins", "m_final", "t0", "sweeps", "levels", "capped"), **kw)
    for k in KEYS:
        assert np.array_equal(getattr(out["0"], k), getattr(out["1"], k)), k
    if kw == dict(k_max=50):  # with the others replicas end nearly in the order of their slots
        assert out["1"].kernel_launches > out["0"].kernel_launches
    assert len(np.unique(out["1"].replica_sweeps)) > 4
    ctx.free(inst)

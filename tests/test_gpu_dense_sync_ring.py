"""Synchronous dense sweeps whose ring of row buffers is shorter than two rows per
warp, as large n leaves it: 26, 14, 4 and 2 buffers for 16 warps a replica, 10 and 7
for 8, 3 for 4. Every fill of a buffer must be told from the one before it."""
import numpy as np
import pytest

import oracle as O
from paper_1907_05124_gb300 import instances as I

from test_gpu_parity import STRICT_LEVELS, check_trajectory, floored_t0

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    from paper_1907_05124_gb300 import mars
    with mars.Context(0) as c:
        yield c


@pytest.mark.parametrize("n,R", [(2048, 3), (3401, 2), (9000, 2), (13000, 1), (4000, 152), (5000, 153), (5000, 305)])
def test_short_rings_follow_the_oracle(ctx, n, R):
    J = I.sk_gauss(n, n)
    c = 2.5  # levels where an FP32 sweep stays within 1e-5 of FP64
    inst = ctx.add_dense(J)
    m0, t0 = I.replica_inputs(R, n, 0.0, 3.0 * c, n)
    t0 = floored_t0(t0, c, max_levels=STRICT_LEVELS)
    oi = O.Instance.dense(J)
    some = np.unique([0, 1 % R, R // 2, R - 1])
    kw = dict(c_step=c, outputs=("m_final", "sweeps", "levels"))
    g = ctx.solve(inst, R, 0.0, 3.0 * c, fixed_sweeps=1, m0=m0, t0=t0, update="jacobi", **kw)
    o = O.mars_solve(oi, m0[some], t0[some], c_step=c, fixed_sweeps=1, nthreads=8, update=O.UPDATE_JACOBI)
    check_trajectory(g.m_final[some], o["m"], "strict")
    assert np.array_equal(g.replica_sweeps[some], o["sweeps"])
    # without noise (its key is the replica's number, which the oracle's part of them changes)
    g = ctx.solve(inst, R, 0.0, 3.0 * c, m0=m0, t0=t0, method="nmfa", alpha=0.35, **kw)
    o = O.nmfa_solve(oi, m0[some], t0[some], c_step=c, alpha=0.35, nthreads=8)
    check_trajectory(g.m_final[some], o["m"], "strict")
    ctx.free(inst)

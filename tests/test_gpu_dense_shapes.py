"""The dense FP32 kernels' shapes against the oracle's fixed-sweep trajectories
(strict tier): all of J on chip (n = 1 to 232), rings of rows (n = 236 and up),
synchronous sweeps with 16, 8 and 4 warps per replica (R = 3, 161, 319) whose
last CTA is partly filled, n = 60, whose synchronous sweeps keep one warp per
replica, and sizes whose rows start anywhere in a 16-byte piece (n = 1, 2, 3, 61,
67, 233, 250, 1001, 1003)."""
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


@pytest.mark.parametrize("update,n,R", [("gs", 1, 2), ("gs", 2, 3), ("gs", 3, 9), ("gs", 61, 6), ("gs", 233, 3),
                                        ("gs", 250, 7), ("gs", 1003, 2), ("jacobi", 67, 3), ("jacobi", 250, 321),
                                        ("jacobi", 1001, 5), ("gs", 64, 6), ("gs", 232, 5), ("gs", 236, 7),
                                        ("gs", 512, 3),
                                        ("jacobi", 60, 5), ("jacobi", 64, 3), ("jacobi", 132, 161),
                                        ("jacobi", 68, 319), ("jacobi", 1000, 3)])
def test_shapes_follow_the_oracle(ctx, update, n, R):
    J = I.sk_gauss(n, n)
    c = 1.2 if update == "gs" else 2.5  # levels where an FP32 sweep stays within 1e-5 of FP64
    h = np.random.default_rng(n).normal(size=n) if n % 8 else None
    inst = ctx.add_dense(J, h=h)
    m0, t0 = I.replica_inputs(R, n, 0.0, 3.0 * c, n)
    t0 = floored_t0(t0, c, max_levels=STRICT_LEVELS)
    g = ctx.solve(inst, R, 0.0, 3.0 * c, c_step=c, fixed_sweeps=1, m0=m0, t0=t0, update=update,
                  outputs=("m_final", "sweeps", "levels", "energies", "spins"))
    o = O.mars_solve(O.Instance.dense(J, h), m0, t0, c_step=c, fixed_sweeps=1, nthreads=8,
                     update=O.UPDATE_JACOBI if update == "jacobi" else 0)
    check_trajectory(g.m_final, o["m"], "strict")
    assert np.array_equal(g.replica_sweeps, o["sweeps"]) and np.array_equal(g.replica_levels, o["levels"])
    assert np.array_equal(g.energies[:8], O.energies(O.Instance.dense(J, h), g.spins[:8]))
    ctx.free(inst)

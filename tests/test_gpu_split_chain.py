"""The split chain (kernels_dense_chain.cu) returns bit for bit what
chain_body's kernels return: every slot count per CTA, GEMM schedule and
operand type, whole panels and a ragged last one, slot counts that leave
replicas of a CTA idle, with and without a field, under the stopping rule."""
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


@pytest.mark.parametrize("precision", ["bf16", "fp8"])
@pytest.mark.parametrize("n,R", [(128, 1), (300, 33), (640, 200), (513, 520)])
@pytest.mark.parametrize("schedule", ["plain", "overlap", "pair", "plan"])
def test_split_chain_is_chain_body(ctx, monkeypatch, precision, n, R, schedule):
    h = np.random.default_rng(n).integers(-3, 4, n).astype(float) if n % 2 else None
    inst = ctx.add_dense(I.sk_pm1(n, n), h=h)
    if schedule != "plan":
        ctx.set_shape(inst, tc_overlap=int(schedule == "overlap"), tc_pair=int(schedule == "pair"))
    m0, t0 = I.replica_inputs(R, n, 0.0, 1.5 * n ** 0.5, R)
    out = {}
    for rpc in ("0", "8", "16", "32"):
        monkeypatch.setenv("MARS_TC_CHAIN_RPC", rpc)
        out[rpc] = ctx.solve(inst, R, 0.0, 1.5 * n ** 0.5, c_step=0.3 * n ** 0.5, m0=m0, t0=t0, k_max=40,
                             precision=precision,
                             outputs=("energies", "spins", "m_final", "sweeps", "levels", "capped"))
    for rpc in ("8", "16", "32"):
        for k in KEYS:
            assert np.array_equal(getattr(out[rpc], k), getattr(out["0"], k)), (rpc, k)
    ctx.free(inst)

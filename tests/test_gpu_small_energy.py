"""Energies of small dense instances, which take one CTA per vector up to 64 spins and
32768 in all (8192 for integer couplings) and the tiled pass beyond, and those of single-CTA tiled passes (integer
couplings below 256 spins): the oracle's exactly rounded sums, bit for bit."""
import numpy as np
import pytest

import oracle as O

from test_gpu_dense_energy import _couplings

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    from paper_1907_05124_gb300 import mars
    with mars.Context(0) as c:
        yield c


@pytest.mark.parametrize("family", ["pm1", "int8", "f32", "wide", "subnormal"])
@pytest.mark.parametrize("n,count", [(1, 5), (2, 1025), (31, 1057), (31, 1058), (63, 200), (64, 128),
                                     (64, 129), (64, 512), (64, 513), (65, 7), (126, 129), (128, 5), (254, 300), (255, 64)])
def test_small_energies_are_the_oracles(ctx, family, n, count):
    J, h = _couplings(family, n, n + count)
    h = h if n % 2 else None
    rng = np.random.default_rng(count)
    inst = ctx.add_dense(J, h=h, order=rng.permutation(n).astype(np.int32) if n % 3 else None)
    s = np.where(rng.random((count, n)) < 0.5, -1, 1).astype(np.int8)
    e, ei = ctx.energy(inst, s)
    want = O.energies(O.Instance.dense(J, h), s)
    assert np.array_equal(e, want)
    if ctx.info(inst)["integer"]:
        assert np.array_equal(ei, want.astype(np.int64))
    s[-1, -1] = 0
    from paper_1907_05124_gb300 import mars
    with pytest.raises(mars.MarsError):
        ctx.energy(inst, s)
    ctx.free(inst)


@pytest.mark.parametrize("R", [250, 251])
def test_tensor_core_solves_on_both_sides_of_the_pass(ctx, R):
    """Integer couplings, n = 400: the finalize kernel's sums up to 250 replicas, the
    tiled pass (one launch more) beyond."""
    J, _ = _couplings("pm1", 400, 7)
    inst = ctx.add_dense(J)
    r = ctx.solve(inst, R, 0.0, 40.0, c_step=20.0, fixed_sweeps=1, precision="bf16", seed=2,
                  outputs=("energies", "spins"))
    assert np.array_equal(r.energies, O.energies(O.Instance.dense(J), r.spins))
    ctx.free(inst)

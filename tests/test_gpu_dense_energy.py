"""Exact energies of dense instances (kernels_dense_energy.cu) against the
oracle's exactly rounded sums, bit for bit: tile edges of n, vector counts on
both sides of a CTA's 128, integer and FP64 couplings, fields, an explicit
order, and couplings whose digits fill many planes or are subnormal."""
import numpy as np
import pytest

import oracle as O
from paper_1907_05124_gb300 import instances as I

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    from paper_1907_05124_gb300 import mars
    with mars.Context(0) as c:
        yield c


def _couplings(family, n, seed):
    rng = np.random.default_rng(seed)
    if family == "pm1":
        return I.sk_pm1(n, seed), rng.integers(-1000, 1000, n).astype(float)
    if family == "int8":  # every byte value up to +-127
        u = np.triu(rng.integers(-127, 128, (n, n)).astype(float), 1)
        return u + u.T, rng.integers(-(1 << 24), 1 << 24, n).astype(float)
    if family == "f32":
        u = np.triu(rng.normal(size=(n, n)).astype(np.float32), 1).astype(float)
        return u + u.T, rng.normal(size=n)
    if family == "subnormal":
        u = np.triu(rng.integers(-(1 << 22), 1 << 22, (n, n)) * 2.0 ** -1070, 1)
        return u + u.T, rng.integers(-(1 << 22), 1 << 22, n) * 2.0 ** -1070
    u = np.triu(rng.normal(size=(n, n)) * 2.0 ** rng.integers(-60, 60, (n, n)), 1)  # about 180 bits
    return u + u.T, rng.normal(size=n) * 2.0 ** rng.integers(-60, 60, n)


@pytest.mark.parametrize("family", ["pm1", "int8", "f32", "wide", "subnormal"])
@pytest.mark.parametrize("n,count", [(1, 1), (2, 3), (127, 33), (128, 32), (129, 31), (300, 130), (256, 1300)])
@pytest.mark.parametrize("field", [False, True])
def test_dense_energies_are_the_oracles(ctx, family, n, count, field):
    J, h = _couplings(family, n, n + count)
    h = h if field else None
    rng = np.random.default_rng(count)
    order = rng.permutation(n).astype(np.int32) if n % 2 else None
    inst = ctx.add_dense(J, h=h, order=order)
    s = np.where(rng.random((count, n)) < 0.5, -1, 1).astype(np.int8)
    e, ei = ctx.energy(inst, s)
    want = O.energies(O.Instance.dense(J, h), s)
    assert np.array_equal(e, want)
    if ctx.info(inst)["integer"]:
        assert np.array_equal(ei, want.astype(np.int64))
    ctx.free(inst)


@pytest.mark.parametrize("n,count", [(4100, 3), (4225, 17)])
def test_largest_digits_and_long_rows(ctx, n, count):
    """Couplings of 127 and of all-ones significands, aligned spins: the largest
    partial sums there are, over rows longer than one run."""
    rng = np.random.default_rng(n)
    s = np.where(rng.random((count, n)) < 0.5, -1, 1).astype(np.int8)
    s[0], s[1] = 1, -1
    a = np.arange(n)
    par = np.where((a[:, None] + a[None, :]) % 5 == 0, -1.0, 1.0)
    for value, h in ((127.0, None), (1.0 - 2.0 ** -24, None), (1.0 - 2.0 ** -24, np.full(n, 2.0 ** -20))):
        for J in (np.full((n, n), value), value * par):
            np.fill_diagonal(J, 0.0)
            inst = ctx.add_dense(J, h=h)
            e, _ = ctx.energy(inst, s)
            assert np.array_equal(e, O.energies(O.Instance.dense(J, h), s))
            ctx.free(inst)


def test_dense_energy_refuses_other_spin_values(ctx):
    from paper_1907_05124_gb300 import mars
    inst = ctx.add_dense(I.sk_gauss(200, 1))
    s = np.ones((3, 200), np.int8)
    s[2, 199] = 0
    with pytest.raises(mars.MarsError):
        ctx.energy(inst, s)
    ctx.free(inst)

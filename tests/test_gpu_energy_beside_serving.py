"""Blocking energies beside served sparse requests, of the same context and of another.

The serving kernel holds about half of the SMs of every GPC for as long as it has
replicas to take, so a blocking call must not wait for more SMs of one GPC than are
left."""
import time

import numpy as np
import pytest

from paper_1907_05124_gb300 import instances as I

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def mars():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1907_05124_gb300 import build, mars as m
    build.build()
    return m


@pytest.mark.parametrize("same", [True, False])
def test_blocking_calls_end_before_the_served_ones(mars, same):
    with mars.Context(0) as c, mars.Context(0) as other:
        b = c if same else other
        lat = c.add_csr(*I.ea_lattice(64, 2, 1))
        inst = b.add_dense(I.sk_gauss(1500, 2))
        spins = np.where(np.random.default_rng(3).random((512, 1500)) < 0.5, -1, 1).astype(np.int8)
        want = b.energy(inst, spins)[0]
        solved = b.solve(inst, 9, 0.0, 1.0, seed=1, fixed_sweeps=1)
        # a CTA per vector: a sparse and a small dense instance
        others = []
        for x in (b.add_csr(*I.er_graph(700, 6, 4)), b.add_dense(I.sk_gauss(40, 5))):
            s = np.where(np.random.default_rng(6).random((50, 700 if not others else 40)) < 0.5, -1, 1).astype(np.int8)
            others.append((x, s, b.energy(x, s)[0]))
        # replicas for every CTA of the serving kernel, 4000 levels of 200 sweeps each:
        # they hold their SMs for a second or so
        req = c.submit(lat, 300, 1.9, 2.0, c_step=5e-4, fixed_sweeps=200, seed=1)
        time.sleep(0.05)
        for _ in range(3):
            t = time.time()
            assert np.array_equal(b.energy(inst, spins)[0], want)
            assert all(np.array_equal(b.energy(x, s)[0], e) for x, s, e in others)
            got = b.solve(inst, 9, 0.0, 1.0, seed=1, fixed_sweeps=1)
            assert time.time() - t < 0.3, "a blocking call waited for the served replicas"
            assert np.array_equal(got.energies, solved.energies)
        assert c.poll(req) is None
        t = time.time()
        while c.poll(req) is None:
            assert time.time() - t < 120.0
            time.sleep(0.01)

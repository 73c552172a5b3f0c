"""A served request runs at once beside a long one.

The serving kernel's CTAs exit when they find no replica to take. A request
whose last replica goes on for long keeps its launch alive with one CTA; a
request submitted then must not wait for that replica.
"""
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


@pytest.mark.parametrize("longs", [1, 3])
def test_requests_beside_long_replicas(mars, longs):
    with mars.Context(0) as c:
        lat = c.add_csr(*I.ea_lattice(64, 2, 1))
        er = c.add_csr(*I.er_graph(600, 8, 2, "pm1"))
        want = [c.solve(er, 64, 0.0, 4.0, seed=s) for s in range(4)]
        # one replica each, 4000 levels of 200 sweeps: two seconds or so
        slow = []
        for s in range(longs):
            slow.append(c.submit(lat, 1, 1.9, 2.0, c_step=5e-4, fixed_sweeps=200, seed=s))
            time.sleep(0.02)  # the other CTAs find no work and exit
        for s in range(4):
            time.sleep(0.005)
            r = c.submit(er, 64, 0.0, 4.0, seed=s)
            t = time.time()
            while (got := c.poll(r)) is None:
                assert time.time() - t < 60.0
                time.sleep(0.0005)
            assert got.best_energy == want[s].best_energy and got.sweeps == want[s].sweeps
            assert np.array_equal(got.best_spins, want[s].best_spins)
        assert all(c.poll(r) is None for r in slow), "the requests waited for the long replicas"
        t = time.time()
        while any([c.poll(r) is None for r in slow if r in c._req_n]):
            assert time.time() - t < 120.0
            time.sleep(0.01)
        assert c.serve_status() == (0, 0)
        assert c.serve_counters() == (longs + 4, 0)

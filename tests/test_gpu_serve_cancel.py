"""Collecting a cancelled request does not wait for the others: no call of the serving
engine may stand still until the device is idle."""
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


def _timed(f):
    t = time.time()
    r = f()
    return time.time() - t, r


def _collect_cancelled(mars, c, r):
    """The longest call until the cancelled request has been reported."""
    longest = _timed(lambda: c.cancel(r))[0]
    while True:
        t = time.time()
        try:
            assert c.poll(r) is None
        except mars.MarsError as e:
            assert "cancel" in str(e)
            return max(longest, time.time() - t)
        longest = max(longest, time.time() - t)
        time.sleep(0.0005)


def test_cancelled_while_running(mars):
    with mars.Context(0) as c:
        lat = c.add_csr(*I.ea_lattice(64, 2, 1))
        er = c.add_csr(*I.er_graph(600, 8, 2, "pm1"))
        warm = [c.submit(er, 64, 0.0, 4.0) for _ in range(2)]  # leave their result blocks to the next ones
        while any([c.poll(q) is None for q in warm if q in c._req_n]):
            time.sleep(0.001)
        # one replica, 4000 levels of 200 sweeps: two seconds or so
        slow = c.submit(lat, 1, 1.9, 2.0, c_step=5e-4, fixed_sweeps=200, seed=1)
        longest = max(_collect_cancelled(mars, c, c.submit(er, 64, 0.0, 4.0, seed=s)) for s in range(8))
        assert c.poll(slow) is None, "the long request ended first"
        assert longest < 0.2, longest
        while c.poll(slow) is None:
            time.sleep(0.01)


def test_cancelled_when_done(mars):
    """A request that is done has left its stream to the next one."""
    with mars.Context(0) as c:
        g = I.ea_lattice(64, 2, 1)
        w = np.random.default_rng(1).normal(size=g.n)
        rows = np.repeat(np.arange(g.n), np.diff(g.row_ptr))
        # general couplings: on a stream of its own instead of the serving kernel
        lat = c.add_csr(g.row_ptr, g.col, g.val * (1.0 + 0.1 * np.tanh(w[rows] + w[g.col])))
        er = c.add_csr(*I.er_graph(600, 8, 2, "pm1"))
        done = [c.submit(er, 64, 0.0, 4.0, seed=s) for s in range(4)]
        until = time.time() + 20.0
        while c.serve_status()[1] and time.time() < until:
            time.sleep(0.001)
        assert c.serve_status() == (0, 0)
        slow = c.submit(lat, 1, 1.9, 2.0, c_step=5e-4, fixed_sweeps=200, seed=1)
        longest = max(_collect_cancelled(mars, c, r) for r in done)
        assert c.poll(slow) is None, "the long request ended first"
        assert longest < 0.2, longest
        while c.poll(slow) is None:
            time.sleep(0.01)

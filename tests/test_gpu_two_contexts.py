"""Two threads, each with a context of its own, call the library at the same time with
sizes that need different amounts of shared memory. The limit a kernel may take is
the process's, so no call may lower it for another's launch."""
import threading
import time

import numpy as np
import pytest

from paper_1907_05124_gb300 import instances as I

pytestmark = pytest.mark.gpu

N = 160


def _gauss(bits):
    """Couplings that need about `bits` bits, so bits / 7 digit planes."""
    J = np.rint(I.sk_gauss(N, bits) * 2.0 ** 8) * 2.0 ** -8
    J[0, 1] = J[1, 0] = 2.0 ** -(bits - 4)
    return J


def _energies(c, small):
    inst = c.add_dense(_gauss(30 if small else 200))
    sp = np.where(np.random.default_rng(1).random((9, N)) < 0.5, -1, 1).astype(np.int8)
    return lambda: c.energy(inst, sp)[0]


def _dense(c, small):
    inst = c.add_dense(I.sk_gauss(96 if small else 200, 2))
    return lambda: c.solve(inst, 4, 0.0, 2.0, fixed_sweeps=1).energies


def _sparse(c, small):
    inst = c.add_csr(*I.ea_lattice(40 if small else 100, 2, 3))
    return lambda: c.solve(inst, 4, 0.0, 2.0, fixed_sweeps=1).energies


@pytest.mark.parametrize("work", [_energies, _dense, _sparse])
def test_calls_of_two_contexts(work):
    from paper_1907_05124_gb300 import mars
    failed = []
    start = threading.Barrier(2, timeout=60)

    def run(small):
        try:
            with mars.Context(0) as c:
                f = work(c, small)
                want = f()
                start.wait()
                t = time.perf_counter()
                while time.perf_counter() - t < 1.0:
                    assert np.array_equal(f(), want)
        except Exception as e:  # noqa: BLE001 - reported below
            failed.append(e)
            start.abort()

    threads = [threading.Thread(target=run, args=(s,)) for s in (True, False)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not failed, failed

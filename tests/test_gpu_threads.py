"""Contexts of different sizes advanced by several threads at once (the binding
releases the interpreter lock in every call): each chain is the one it is
alone."""
import threading

import numpy as np
import pytest

from paper_1012_5082_gb300 import inputs as I

pytestmark = pytest.mark.gpu

# lattices whose resident forms run the same kernel with little shared memory
# and with more than a launch may have without being allowed it (48 KB)
SMALL, LARGE = ((10, 10, 10), 5), ((80, 80, 40), 20)
SIZES = [LARGE, SMALL, SMALL, LARGE, SMALL, SMALL]


def _context(V, cells, block, seed):
    lat = I.bcc_lattice(*cells)
    types = I.random_types(lat.n, lat.n // 10, seed=seed)
    return V.Context(lat, types, I.eam_tables(), -2.2, 0.01, 900.0, c0=0.1, seed=seed, schedule=V.SCHED_BLOCKS,
                     sched=(block,) * 3 + (2, 2, 2))


def _run(V, k, out):
    try:
        g = _context(V, *SIZES[k], seed=k + 1)
        for _ in range(1500):
            g.steps(64)
        out[k] = (g.types(), g.observables()["flips"])
        g.close()
    except Exception as e:  # reported by the test
        out[k] = e


def test_contexts_of_different_sizes_in_threads():
    from paper_1012_5082_gb300 import vcsgc as V
    alone, together = {}, {}
    for k in range(len(SIZES)):
        _run(V, k, alone)
        assert not isinstance(alone[k], Exception), alone[k]
    threads = [threading.Thread(target=_run, args=(V, k, together)) for k in range(len(SIZES))]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    failed = {(k, SIZES[k]): e for k, e in together.items() if isinstance(e, Exception)}
    assert not failed, failed
    for k in range(len(SIZES)):
        assert together[k][1] == alone[k][1] > 0 and np.array_equal(together[k][0], alone[k][0])

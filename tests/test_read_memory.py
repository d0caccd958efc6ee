"""Host memory that large reads use again: one array a field, bounded over all
simulations, and given back at close()."""
import gc
import weakref

import numpy as np
import pytest

from paper_1410_3464_gb300 import pslbm

MB = 1 << 20


class Library:
    def pslbm_destroy(self, h):
        return 0


@pytest.fixture
def simulation(monkeypatch):
    monkeypatch.setattr(pslbm, "load", Library)

    def make():
        sim = pslbm.Simulation.__new__(pslbm.Simulation)
        sim._reads, sim._spare, sim.h = {}, {}, 1
        return sim
    return make


def owner(a):
    while isinstance(a, np.ndarray):
        a = a.base
    return a


def read(sim, n=MB):
    """An array as read() makes it, and a reference to the memory behind."""
    a = sim._memory("rho1", n).view(np.float64)
    return a, weakref.ref(owner(a).mem)


def test_memory_is_used_again_and_kept_arrays_stay(simulation):
    sim = simulation()
    a, _ = read(sim)
    a[:] = 1.0
    b, rb = read(sim)
    b[:] = 2.0
    del b
    c, rc = read(sim)
    assert rc() is rb() and (a == 1.0).all()
    sim.close()


def test_one_array_a_field_waits(simulation):
    sim = simulation()
    arrays = [read(sim) for _ in range(4)]
    refs = [r for _, r in arrays]
    arrays.clear()
    gc.collect()
    assert sum(r() is not None for r in refs) == 1
    sim.close()


def test_close_gives_all_back_while_an_array_lives(simulation):
    sim = simulation()
    kept, rk = read(sim)
    (a, ra), (b, rb) = read(sim), read(sim)
    del a, b
    sim.close()
    gc.collect()
    assert ra() is None and rb() is None and rk() is not None
    del kept
    gc.collect()
    assert rk() is None


def test_all_simulations_together_are_bounded(simulation, monkeypatch):
    monkeypatch.setattr(pslbm._Spare, "most", pslbm._Spare.held + 5 * MB)
    sims = [simulation() for _ in range(12)]
    refs = []
    for s in sims:
        refs.append(read(s)[1])
    gc.collect()
    assert sum(r() is not None for r in refs) == 5
    for s in sims:
        s.close()
    gc.collect()
    assert not any(r() is not None for r in refs)

"""pslbm_read_fields and Simulation.read: each field goes to a buffer of its own."""
import ctypes
import mmap

import numpy as np
import pytest

from paper_1410_3464_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pslbm():
    from paper_1410_3464_gb300 import build, pslbm as m
    build.build()
    return m


def simulation(pslbm, nx, ny):
    sc = inputs.bubble_grain(nx, ny)
    return pslbm.Simulation(sc["mask"], sc["params"], sc["rho1"], sc["rho2"], sc["conc"], sc["vol"], precision=pslbm.FP64)


@pytest.mark.parametrize("nx,ny", [(128, 64), (512, 128)])
@pytest.mark.parametrize("first", [0, 1])
def test_adjoining_buffers_in_different_allocations(pslbm, nx, ny, first):
    """Two buffers back to back, one of them page-locked: two host ranges, which no
    single copy may span.  64 KiB or 512 KiB each, whole pages."""
    import torch
    rt = torch.cuda.cudart()
    size = 8 * nx * ny
    region = mmap.mmap(-1, 4 * size)
    whole = np.frombuffer(region, np.uint8)
    base = -whole.ctypes.data % 65536
    mem = whole[base:base + 2 * size]
    locked = mem[first * size:(first + 1) * size]
    err = rt.cudaHostRegister(locked.ctypes.data, size, 0)
    assert int(err) == 0
    try:
        with simulation(pslbm, nx, ny) as sim:
            sim.step(3)
            ptrs = (ctypes.c_void_p * 2)(mem.ctypes.data, mem.ctypes.data + size)
            st = pslbm.load().pslbm_read_fields(sim.h, pslbm.F_RHO1 | pslbm.F_RHO2, ptrs)
            assert st == 0, pslbm.load().pslbm_last_error(sim.h)
            ref = sim.read()
            np.testing.assert_array_equal(mem[:size].view(np.float64).reshape(ny, nx), ref["rho1"])
            np.testing.assert_array_equal(mem[size:].view(np.float64).reshape(ny, nx), ref["rho2"])
    finally:
        rt.cudaHostUnregister(locked.ctypes.data)


@pytest.mark.parametrize("fields", [0x01, 0x21, 0x22, 0x3C, 0x5A, 0x60, 0x7F, 0xA8, 0xFF])
def test_every_selection_gives_the_fields_of_a_full_read(pslbm, fields):
    with simulation(pslbm, 128, 64) as sim:
        sim.step(5)
        names = ("rho1", "rho2", "ux", "uy", "conc", "type", "vol", "budget")
        alone = {n: sim.read(1 << i)[n] for i, n in enumerate(names)}
        got = sim.read(fields)
        for i, n in enumerate(names):
            assert (n in got) == bool(fields >> i & 1)
            if n in got:
                np.testing.assert_array_equal(got[n], alone[n], err_msg=n)


def owner(a):
    while isinstance(a, np.ndarray) and a.base is not None:
        a = a.base
    return a


def test_a_kept_array_keeps_no_other(pslbm):
    """Of a small read, the memory behind an array is its own."""
    with simulation(pslbm, 128, 64) as sim:
        r = sim.read()
    for n in ("rho1", "rho2", "ux", "uy", "conc", "type", "vol", "budget"):
        assert owner(r[n]).nbytes == r[n].nbytes, n

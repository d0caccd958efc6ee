"""Node types outside the enumeration: a byte whose low nibble is above OUTLET is a wall.

The scene has such nodes in place of its walls and inside the lattice, next to liquid
and gas; every field must be the same bits as with WALL there.
"""
import numpy as np
import pytest

from paper_1410_3464_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pslbm():
    from paper_1410_3464_gb300 import build, pslbm as m
    build.build()
    return m


def fields(pslbm, sc, mask, precision):
    with pslbm.Simulation(mask, sc["params"], sc["rho1"], sc["rho2"], sc["conc"], sc["vol"], precision=precision) as sim:
        sim.step(20)
        return sim.read()


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("byte", [7, 8, 9, 10, 13, 14, 15, 0x20 | 9])
def test_unknown_types_are_walls(pslbm, byte, precision):
    sc = inputs.bubble_grain(64, 32)
    wall = sc["mask"].copy()
    wall[5:25:4, 3:60:7] = 4
    other = np.where(wall == 4, byte, wall).astype(np.uint8)
    ref, got = fields(pslbm, sc, wall, precision), fields(pslbm, sc, other, precision)
    for name in ref:
        if name != "type":
            np.testing.assert_array_equal(got[name], ref[name], err_msg=name)
    np.testing.assert_array_equal(np.where(got["type"] == byte & 15, 4, got["type"]), ref["type"])

"""Every launch form gives the same bits: one simulation (parameters in the constant
bank), a batch of like members (the first one's parameters) and one of unlike members
(each one's own), one turn of a warp and several, VOP and amendment in one launch and
in two.

The scenes: the beaker (four species, surface reaction, outlet along y), a porous
sample with reservoirs, a periodic scene with ramped inlets along either axis, and
dissolving and overflowing grains.
"""
import numpy as np
import pytest

from paper_1410_3464_gb300 import inputs
from test_gpu_stream import growing, scene

pytestmark = pytest.mark.gpu

PRECISIONS = [0, 1, 2, 3]


@pytest.fixture(scope="module")
def pslbm():
    from paper_1410_3464_gb300 import build, pslbm as m
    build.build()
    return m


def ramped(axis):
    sc = scene(*((60, 23) if axis == "x" else (23, 60)), axis == "y", axis == "x", reservoirs=axis)
    sc["params"].update(inlet_ramp=3, inlet_period_liq=5, inlet_period_gas=4)
    return sc


def overflowing(nx, ny):
    """Grains that dissolve, and precipitate that overflows into neighbours."""
    sc = growing(nx, ny)
    p = sc["params"]
    p.update(G11=0.0, G12=0.0, G21=0.0, idx_F=2, idx_E=-1, k4=0.02, C_F_sat=0.01, Vbar_F=0.2, V_split=2.0, seed=7)
    full = sc["mask"] == 2
    full[:, : nx // 2] = False
    sc["mask"][full] = 3
    sc["vol"][0][full] = 0.0
    sc["vol"][1][full] = np.random.default_rng(2).uniform(1.99, 1.999, full.sum())
    return sc


SCENES = {"beaker": inputs.beaker, "porous": lambda: inputs.porous_discs(nx=100, ny=50, seed=61, rmin=3, rmax=8),
          "ramp x": lambda: ramped("x"), "ramp y": lambda: ramped("y"), "overflow": lambda: overflowing(45, 20)}


def simulation(pslbm, sc, precision):
    return pslbm.Simulation(sc["mask"], sc["params"], sc["rho1"], sc["rho2"], sc["conc"], sc["vol"], precision=precision)


def alone(pslbm, sc, precision, steps, shape=(0, 0)):
    with simulation(pslbm, sc, precision) as sim:
        sim.set_tile_shape(*shape)
        sim.step(steps)
        return sim.read()


def assert_same(got, ref, what):
    for name in ref:
        np.testing.assert_array_equal(got[name], ref[name], err_msg=f"{what} {name}")


@pytest.mark.parametrize("precision", PRECISIONS)
@pytest.mark.parametrize("name", SCENES)
def test_launch_forms_give_the_same_bits(pslbm, name, precision):
    sc = SCENES[name]()
    if precision >= 2 and name.startswith("ramp"):
        sc["params"]["conc_scale"] = (4.0, 16.0, 8.0, 0.0)
    ref = alone(pslbm, sc, precision, 24)
    for shape in ((16, 16), (32, 16)):
        assert_same(alone(pslbm, sc, precision, 24, shape), ref, shape)
    with simulation(pslbm, sc, precision) as sim:
        sim.profile_step(24)
        assert_same(sim.read(), ref, "profiled")
    # the second member has a lattice of its own kind: like parameters, or another interaction
    ns = sc["params"]["n_species"]
    other = inputs.porous_discs(nx=130, ny=70, seed=3) if ns == 3 else inputs.beaker(110, 150)
    for like in (True, False):
        o = dict(other, params=dict(sc["params"], nx=other["params"]["nx"], ny=other["params"]["ny"], k3=0.0))
        if not like:
            o["params"].update(G12=1.1 * sc["params"]["G12"] + 1e-4)
        sims = [simulation(pslbm, s, precision) for s in (sc, o, sc)]
        batch = pslbm.Batch(sims)
        batch.step(24)
        assert_same(sims[0].read(), ref, f"batch, like={like}")
        assert_same(sims[2].read(), ref, f"batch, like={like}, third")
        batch.close()
        for s in sims:
            s.close()

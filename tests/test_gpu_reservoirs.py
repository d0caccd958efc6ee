"""Device bytes of a simulation, by which a server admits, and reservoir nodes anywhere
in the lattice: the bytes stay within the estimate, and the steps agree with the oracle."""
import numpy as np
import pytest

from oracle import lbm
from paper_1410_3464_gb300 import inputs
from test_gpu_stream import scene

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pslbm():
    from paper_1410_3464_gb300 import build, pslbm as m
    build.build()
    return m


@pytest.mark.parametrize("share", [0.0, 0.5, 1.0])
@pytest.mark.parametrize("nx,ny", [(1, 1), (33, 5), (256, 130)])
def test_device_bytes_within_the_estimate(pslbm, nx, ny, share):
    p = inputs.base_params(nx, ny)
    mask = np.where(np.random.default_rng(1).random((ny, nx)) < share, 5, 0).astype(np.uint8)
    rho1, rho2 = np.full((ny, nx), 0.35), np.full((ny, nx), 2e-5)
    for precision in (pslbm.FP64, pslbm.FP32):
        with pslbm.Simulation(mask, p, rho1, rho2, None, None, precision=precision) as sim:
            assert sim.device_bytes() <= pslbm.estimate_device_bytes(p, precision)


@pytest.mark.parametrize("precision,beside", [(0, 65), (1, 49), (2, 49), (3, 49)])
def test_bytes_a_node(pslbm, precision, beside):
    """What a node takes beside its populations: two types, two volumes, potentials
    (their bytes hold the events too), a code, an event code, two lists, a claim and
    two bits: 64.25 bytes in FP64, 48.25 in FP32."""
    sc = inputs.porous_discs(nx=512, ny=256, seed=1)
    n = 512 * 256
    per = 2 * 18 * (4 if precision else 8) + 2 * 5 * 3 * (8, 4, 2, 2)[precision] + beside
    fixed = 64 * 1024
    assert pslbm.estimate_device_bytes(sc["params"], precision) <= n * per + fixed
    with pslbm.Simulation(sc["mask"], sc["params"], sc["rho1"], sc["rho2"], sc["conc"], None, precision=precision) as sim:
        assert sim.device_bytes() <= n * per + fixed


@pytest.mark.parametrize("axis", ["x", "y"])
def test_reservoirs_inside_the_lattice_match_the_oracle(pslbm, axis):
    """A tenth of the nodes feed or drain, next to liquid, gas, grains and each other.
    1e-12 of each field, as for the scenes with reservoirs at the edges; 8 steps."""
    sc = scene(70, 41, 1, 1, reservoirs=axis)
    rng = np.random.default_rng(11)
    sc["mask"][rng.random(sc["mask"].shape) < 0.05] = 5
    sc["mask"][rng.random(sc["mask"].shape) < 0.05] = 6
    fluid = sc["mask"] <= 1
    sc["rho1"], sc["rho2"] = sc["rho1"] * fluid, sc["rho2"] * fluid
    sc["conc"] = sc["conc"] * (sc["mask"] == 0)
    with pslbm.Simulation(sc["mask"], sc["params"], sc["rho1"], sc["rho2"], sc["conc"], None, precision=pslbm.FP64) as sim:
        sim.step(8)
        got = sim.read()
    L = lbm.Lattice(sc["mask"], sc["params"], sc["rho1"], sc["rho2"], sc["conc"], None)
    L.run(8)
    ref = L.fields()
    np.testing.assert_array_equal(got["type"], ref["type"])
    for name, where in (("rho1", ref["type"] <= 1), ("rho2", ref["type"] <= 1), ("conc", ref["type"] == 0)):
        a, b = got[name][..., where], ref[name][..., where]
        assert np.abs(a - b).max() <= 1e-12 * np.abs(b).max(), name
    for name in ("ux", "uy"):
        a, b = got[name][fluid], ref[name][fluid]
        assert np.abs(a - b).max() <= 1e-12 * max(np.abs(b).max(), 0.05), name

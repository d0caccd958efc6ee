"""The list-driven streaming kernels where they can go wrong: lattices at and
around the edges of cells and list tiles, lattices one node wide, both
relaxation forms, reservoirs along either axis, several turns of a warp, lists
that grow, batches of equal and of different parameters, and the read-out.

Against the oracle: 1e-12 relative per field (FP64 on both sides, rounding order
only: 1e-16 an operation, a few hundred operations a node and step, 12 steps;
velocities, which are what is left of sums of populations, against at least 0.05).
Between launch shapes: the same bits, since a node's arithmetic does not depend on
which warp does it.
"""
import numpy as np
import pytest

from oracle import lbm
from paper_1410_3464_gb300 import inputs

pytestmark = pytest.mark.gpu

TOL = 1e-12


@pytest.fixture(scope="module")
def pslbm():
    from paper_1410_3464_gb300 import build, pslbm as m
    build.build()
    return m


def rel(a, b, where, least=0.0):
    a, b = a[..., where], b[..., where]
    den = max(np.abs(b).max(), least) if b.size else 0.0
    return float(np.abs(a - b).max() / den) if den else (float(np.abs(a).max()) if a.size else 0.0)


def scene(nx, ny, px, py, tau=(1.0, 1.0), reservoirs=None, seed=3):
    rng = np.random.default_rng(seed)
    p = inputs.base_params(nx, ny)
    p.update(periodic_x=px, periodic_y=py, rho_ref=(0.3, 1e-3), n_species=3, idx_A=0, idx_B=1, idx_E=2, tau=tau,
             J0=(1 / 3, 0.2, 0.5, 0), tau_g=(0.8, 1.1, 1.0, 1), k1=0.01, k2=0.02, k3=0.02, gas_yield=0.5, inv_M_C=1.0,
             w_adh=(-0.02, 0.01), body_force=(1e-6, -2e-6))
    mask = np.where(rng.random((ny, nx)) < 0.12, 2, 0).astype(np.uint8)
    mask[rng.random((ny, nx)) < 0.1] = 1
    if reservoirs == "x":
        mask[:, 0], mask[:, -1] = 5, 6
    elif reservoirs == "y":
        mask[0], mask[-1] = 5, 6
    if reservoirs:
        a = 0 if reservoirs == "x" else 1
        p.update(inlet_axis=a, outlet_axis=a, rho_in_liq=(0.31, 2e-5), rho_in_gas=(0.02, 2e-3), rho_out=(0.3, 2e-5),
                 rho_out_gas=(0.01, 2e-3), conc_in=(1.0, 0.1, 0.2, 0.0), inlet_period_liq=4, inlet_period_gas=3)
    rl, rg = inputs.COEX_ORIGINAL_07
    rho1 = np.where(mask == 0, rl * (1 + 0.01 * rng.standard_normal((ny, nx))), np.where(mask == 1, rg, 0.0))
    rho2 = np.where(mask == 1, 0.002, 2e-5) * (mask <= 1)
    conc = np.stack([np.where(mask == 0, c, 0.0) for c in (1.0, 0.2, 0.3)])
    return dict(mask=mask, rho1=rho1, rho2=rho2, conc=conc, vol=None, params=p)


def state(pslbm, sc, steps, precision, shape=(0, 0)):
    with pslbm.Simulation(sc["mask"], sc["params"], sc["rho1"], sc["rho2"], sc["conc"], sc["vol"],
                          precision=precision) as sim:
        sim.set_tile_shape(*shape)
        sim.step(steps)
        return sim.read()


@pytest.mark.parametrize("tau", [(1.0, 1.0), (0.9, 1.2)])
@pytest.mark.parametrize("nx,ny,px,py,reservoirs", [
    (1, 33, 1, 1, None), (33, 1, 1, 1, None), (31, 8, 1, 0, None), (32, 9, 0, 1, None), (33, 17, 0, 0, None),
    (40, 13, 0, 1, "x"), (13, 40, 1, 0, "y")])
def test_fp64_matches_oracle(pslbm, nx, ny, px, py, reservoirs, tau):
    sc = scene(nx, ny, px, py, tau, reservoirs)
    got = state(pslbm, sc, 12, pslbm.FP64)
    L = lbm.Lattice(sc["mask"], sc["params"], sc["rho1"], sc["rho2"], sc["conc"], None)
    L.run(12)
    ref = L.fields()
    np.testing.assert_array_equal(got["type"], ref["type"])
    for name in ("rho1", "rho2", "ux", "uy"):
        e = rel(got[name], ref[name], ref["type"] <= 1, 0.05 if name[0] == "u" else 0.0)
        assert e <= TOL, f"{name}: {e:.3e}"
    for name, where in (("conc", ref["type"] == 0), ("vol_d", ref["type"] == 2)):
        e = rel(got[name], ref[name], where)
        assert e <= TOL, f"{name}: {e:.3e}"


def growing(nx, ny):
    """Scattered grains that dissolve within a few steps, not all in the same one."""
    sc = scene(nx, ny, 1, 1, seed=nx)
    sc["params"]["k2"] = 0.1
    sc["params"]["Vbar_D"] = 1.0
    vol = np.zeros((2, ny, nx))
    solid = sc["mask"] == 2
    vol[0][solid] = np.random.default_rng(1).uniform(0.005, 0.4, solid.sum())
    sc["vol"] = vol
    return sc


@pytest.mark.parametrize("precision", [0, 1, 2])
@pytest.mark.parametrize("nx,ny", [(45, 20), (420, 260)])
def test_turns_and_growing_lists_give_the_same_bits(pslbm, nx, ny, precision):
    """The default plan (one turn on the small lattice, several on the large one)
    against the pinned ones, with nodes that dissolve and join the lists."""
    sc = growing(nx, ny)
    ref = state(pslbm, sc, 30, precision)
    assert (ref["type"] == 2).sum() < (sc["mask"] == 2).sum() - 8, "hardly a node dissolved"
    for shape in ((16, 16), (32, 16)):
        got = state(pslbm, sc, 30, precision, shape)
        for name in ref:
            np.testing.assert_array_equal(got[name], ref[name], err_msg=f"{shape} {name}")


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("same", [True, False])
def test_batch_of_equal_and_of_different_parameters(pslbm, same, precision):
    """Members with one set of parameters share those of the first; others read
    their own.  Either way as alone."""
    scs = [growing(45, 20), growing(130, 70), scene(40, 13, 0, 1, reservoirs="x")]
    for k, sc in enumerate(scs):
        sc["params"].update(k1=0.01 * (k + 1), seed=k + 1)
        if not same:
            sc["params"].update(G12=sc["params"]["G12"] * (1 + 0.1 * k), tau=(1.0 + 0.1 * k, 1.0))
    sims = [pslbm.Simulation(s["mask"], s["params"], s["rho1"], s["rho2"], s["conc"], s["vol"], precision=precision)
            for s in scs]
    batch = pslbm.Batch(sims)
    batch.step(20)
    batch.sync()
    for k, sim in enumerate(sims):
        got, ref = sim.read(), state(pslbm, scs[k], 20, precision)
        for name in ref:
            np.testing.assert_array_equal(got[name], ref[name], err_msg=f"member {k} {name}")
    batch.close()
    for sim in sims:
        sim.close()


@pytest.mark.parametrize("nx,ny", [(45, 21), (200, 101)])
def test_reads_are_independent_arrays(pslbm, nx, ny):
    """Arrays that are kept stay as they are when later reads reuse the memory of
    those that were not, and one field alone equals the same field among all."""
    sc = scene(nx, ny, 1, 1)
    with pslbm.Simulation(sc["mask"], sc["params"], sc["rho1"], sc["rho2"], sc["conc"], precision=pslbm.FP32) as sim:
        kept, want = [], []
        for _ in range(5):
            sim.step(1)
            r = sim.read()
            one = {n: sim.read(1 << i)[n] for i, n in enumerate(("rho1", "rho2", "ux", "uy", "conc", "type", "vol", "budget"))}
            for n, a in one.items():
                np.testing.assert_array_equal(a, r[n], err_msg=n)
            kept.append(r["rho1"])
            want.append(r["rho1"].copy())
    for a, b in zip(kept, want):
        np.testing.assert_array_equal(a, b)
    assert not np.array_equal(want[0], want[1])


@pytest.mark.parametrize("precision", [0, 1, 3])
@pytest.mark.parametrize("nx,ny", [(45, 20), (45, 60)])
def test_one_launch_for_vop_and_amendment(pslbm, nx, ny, precision):
    """step() takes VOP and amendment in one launch while every list of reactive
    minerals was at most 256 long (45x20 has 101, 45x60 326);
    profile_step() always takes two.  Dissolution, overflow and list growth on the way."""
    sc = growing(nx, ny)
    p = sc["params"]
    p.update(G11=0.0, G12=0.0, G21=0.0, idx_F=2, idx_E=-1, k4=0.02, Vbar_F=0.2, V_split=2.0, seed=7)
    full = sc["mask"] == 2
    full[:, : nx // 2] = False
    sc["mask"][full] = 3
    sc["vol"][0][full] = 0.0
    sc["vol"][1][full] = np.random.default_rng(2).uniform(1.99, 1.999, full.sum())
    ref = state(pslbm, sc, 30, precision)
    assert (ref["type"] == 3).sum() > full.sum(), "no overflow"
    assert (ref["type"] == 2).sum() < (sc["mask"] == 2).sum(), "no node dissolved"
    with pslbm.Simulation(sc["mask"], p, sc["rho1"], sc["rho2"], sc["conc"], sc["vol"], precision=precision) as sim:
        sim.profile_step(30)
        got = sim.read()
    for name in ref:
        np.testing.assert_array_equal(got[name], ref[name], err_msg=name)

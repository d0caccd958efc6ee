"""The lists of fluid nodes and of minerals over long runs: made again every thousand
steps or so, which leaves no trace in the results and keeps a step as fast as that of
a fresh simulation of the same state."""
import time

import numpy as np
import pytest

from paper_1410_3464_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pslbm():
    from paper_1410_3464_gb300 import build, pslbm as m
    build.build()
    return m


def bank(nx, ny, rows, Vbar):
    """Liquid over a bank of D(s) whose nodes dissolve one after the other; the top row
    supplies the dissolving species."""
    p = inputs.base_params(nx, ny)
    p.update(periodic_x=1, periodic_y=0, n_species=2, idx_A=-1, idx_B=0, idx_E=-1, idx_F=1, G11=0.0, G12=0.0, G21=0.0,
             J0=(0.2, 0.3, 0, 0), tau_g=(1.0, 0.9, 1, 1), k2=0.2, Vbar_D=Vbar, V_split=2.0, body_force=(1e-7, 0.0), inlet_axis=1,
             outlet_axis=1, conc_in=(1.0, 0, 0, 0), rho_in_liq=(0.35813, 2e-5), rho_in_gas=(0.35813, 2e-5))
    mask = np.zeros((ny, nx), np.uint8)
    mask[-rows:], mask[0] = 2, 5
    liquid, solid = mask == 0, mask == 2
    vol = np.zeros((2, ny, nx))
    vol[0][solid] = np.random.default_rng(1).uniform(0.02, 0.2, solid.sum())
    return dict(mask=mask, params=p, rho1=0.35813 * liquid, rho2=2e-5 * liquid, conc=np.stack([1.0 * liquid, 0.0 * liquid]), vol=vol)


def simulation(pslbm, sc, precision):
    return pslbm.Simulation(sc["mask"], sc["params"], sc["rho1"], sc["rho2"], sc["conc"], sc["vol"], precision=precision)


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("rows", [20, 40])
def test_new_lists_leave_no_trace(pslbm, rows, precision):
    """step() makes the lists again, profile_step() does not; nodes dissolve all along."""
    sc = bank(70, 60, rows, 0.05)
    sc["mask"][rng_holes(rows)] = 2
    with simulation(pslbm, sc, precision) as a, simulation(pslbm, sc, precision) as b:
        left = [(sc["mask"] == 2).sum()]
        for n in (700, 900, 1100, 1):
            a.step(n)
            b.profile_step(n)
            got, ref = a.read(), b.read()
            for name in ref:
                np.testing.assert_array_equal(got[name], ref[name], err_msg=f"{n} {name}")
            left.append((ref["type"] == 2).sum())
        assert (np.diff(left[:4]) < -5).all(), left
        # as members of a batch, which takes the age of the lists over
        batch = pslbm.Batch([a])
        batch.step(1200)
        batch.sync()
        batch.close()
        b.profile_step(1200)
        got, ref = a.read(), b.read()
        for name in ref:
            np.testing.assert_array_equal(got[name], ref[name], err_msg=name)


def rng_holes(rows):
    """Some grains in the liquid."""
    m = np.zeros((60, 70), bool)
    m[5:60 - rows - 5:6, 3::9] = True
    return m


def us(sim, n=256):
    best = 1e9
    for _ in range(5):
        sim.sync()
        t = time.perf_counter()
        sim.step(n)
        sim.sync()
        best = min(best, (time.perf_counter() - t) / n * 1e6)
    return best


def test_a_long_run_stays_as_fast_as_a_fresh_one(pslbm):
    """Some thousand minerals have dissolved by then; a step, best of five, takes no
    longer than 1.2 times that of a simulation made from the state reached."""
    sc = bank(100, 160, 130, 0.3)
    with simulation(pslbm, sc, pslbm.FP32) as sim:
        for _ in range(12):
            sim.step(1500)
            sim.sync()
        r = sim.read()
        assert (r["type"] == 2).sum() < (sc["mask"] == 2).sum() - 3000, (r["type"] == 2).sum()
        old = us(sim)
    now = dict(sc, mask=r["type"], rho1=r["rho1"], rho2=r["rho2"], conc=r["conc"], vol=r["vol"])
    with simulation(pslbm, now, pslbm.FP32) as sim:
        fresh = us(sim)
    assert old <= 1.2 * fresh, (old, fresh)


@pytest.mark.parametrize("members", [0, 2])
def test_plans_follow_the_lists(pslbm, members):
    """Nodes that dissolve fast: the list of minerals passes the length up to which VOP
    and amendment are one launch and, made again, falls below it; the lists outgrow the
    work laid out for them.  Each sync lets the host see their lengths.  One simulation,
    and a batch, against steps that keep list and plan."""
    sc = bank(200, 120, 80, 3.0)
    with simulation(pslbm, sc, pslbm.FP32) as b:
        sims = [simulation(pslbm, sc, pslbm.FP32) for _ in range(max(1, members))]
        run = pslbm.Batch(sims) if members else sims[0]
        gone = [0]
        for n in (150, 150, 400, 400, 300, 200):
            run.step(n)
            run.sync()
            b.profile_step(n)
            ref = b.read()
            for s in sims:
                got = s.read()
                for name in ref:
                    np.testing.assert_array_equal(got[name], ref[name], err_msg=f"{n} {name}")
            gone.append(int((sc["mask"] == 2).sum() - (ref["type"] == 2).sum()))
        assert gone[2] > 300 and gone[-1] > 2300, gone
        if members:
            run.close()
        for s in sims:
            s.close()

"""FP64 arithmetic of the potentials and velocities, operation by operation.

A state at rest gives velocities that follow from the densities by a few dozen
operations (Eqs. 11-13, 19 and the body force).  Here they are done on the host with
correctly rounded operations (addition, product, quotient, square root, fused
multiply-add) in the order of the device code; the device has to give the same bits:
its quotient, reciprocal and square root are the correctly rounded ones.
"""
import ctypes
import math

import numpy as np
import pytest

from paper_1410_3464_gb300 import inputs

pytestmark = pytest.mark.gpu

_libm = ctypes.CDLL("libm.so.6")
_libm.fma.restype = ctypes.c_double
_libm.fma.argtypes = [ctypes.c_double] * 3
fma = np.vectorize(lambda a, b, c: _libm.fma(a, b, c), otypes=[np.float64])


@pytest.fixture(scope="module")
def pslbm():
    from paper_1410_3464_gb300 import build, pslbm as m
    build.build()
    return m


def psi(rho, p):
    eta = (p["eos_b"] / 4.0) * rho
    om = 1.0 - eta
    poly = fma(eta, fma(eta, om, 1.0), 1.0)
    num = (rho * (p["eos_R"] * p["eos_T"])) * poly
    pr = fma(-(p["eos_a"] * rho), rho, num / ((om * om) * om))
    arg = (6.0 / p["G11"]) * (pr - rho * (1.0 / 3.0))
    assert (arg >= 0).all()
    return np.sqrt(arg)


@pytest.mark.parametrize("top", [1.0, 1e-3])
@pytest.mark.parametrize("G11", [True, False])
def test_velocities_at_rest_are_correctly_rounded(pslbm, G11, top):
    """Densities over the liquid (top 1) and the gas (top 1e-3) range; with the EOS
    forces, and with the body force alone (the reciprocal of the density)."""
    nx, ny = 48, 40
    rng = np.random.default_rng(5)
    p = inputs.base_params(nx, ny)
    p.update(periodic_x=1, periodic_y=1, n_species=0, idx_A=-1, idx_B=-1, idx_E=-1, idx_F=-1, G12=0.0, G21=0.0,
             w_adh=(0.0, 0.0), body_force=(1.3e-5, -7.1e-6))
    if not G11:
        p["G11"] = 0.0
    rho1 = top * inputs.COEX_ORIGINAL_07[0] * rng.uniform(0.9, 1.1, (ny, nx))
    rho2 = rng.uniform(1e-5, 2e-3, (ny, nx))
    with pslbm.Simulation(np.zeros((ny, nx), np.uint8), p, rho1, rho2, None, None, precision=pslbm.FP64) as sim:
        got = sim.read()
    r1, r2 = got["rho1"], got["rho2"]
    F1 = [np.zeros_like(r1), np.zeros_like(r1)]
    if G11:
        s0 = psi(r1, p)
        v = [s0] + [np.roll(s0, (-ey, -ex), (0, 1)) for ex, ey in ((1, 0), (0, 1), (-1, 0), (0, -1), (1, 1), (-1, 1), (-1, -1), (1, -1))]
        d57, d86 = v[5] - v[7], v[8] - v[6]
        S = (fma(1.0 / 9.0, v[1] - v[3], (1.0 / 36.0) * (d57 + d86)), fma(1.0 / 9.0, v[2] - v[4], (1.0 / 36.0) * (d57 - d86)))
        F1 = [-((p["G11"] * s0) * s) for s in S]
    for i, name in ((0, "ux"), (1, "uy")):
        g = p["body_force"][i]
        f1, f2 = fma(r1, g, F1[i]), r2 * g
        u = (0.5 * (f1 + f2)) * (1.0 / (r1 + r2))
        np.testing.assert_array_equal(got[name], u, err_msg=name)
    assert math.isfinite(float(got["ux"].sum()))


W9 = (4.0 / 9.0,) + (1.0 / 9.0,) * 4 + (1.0 / 36.0,) * 4
E9 = ((0, 0), (1, 0), (0, 1), (-1, 0), (0, -1), (1, 1), (-1, 1), (-1, -1), (1, -1))


def feq9(rho, ux, uy):
    """Eq. 8, opposite directions together (the even part, then plus and minus the odd one)."""
    uu = 1.5 * fma(ux, ux, uy * uy)
    f = [None] * 9
    f[0] = W9[0] * fma(rho, -uu, rho)
    for p, m, e in ((1, 3, ux), (2, 4, uy), (5, 7, ux + uy), (6, 8, uy - ux)):
        sym = W9[p] * fma(rho, fma(4.5, e * e, -uu), rho)
        asym = ((1.0 / 3.0 if p < 5 else 1.0 / 12.0) * rho) * e
        f[p], f[m] = sym + asym, sym - asym
    return f


def streamed_sum(f, e):
    f = [np.roll(v, (e[a][1], e[a][0]), (0, 1)) for a, v in enumerate(f)]
    s = f[0]
    for v in f[1:]:
        s = s + v
    return s


def reacting(nx, ny, tau_g, seed=8):
    """Liquid at rest with a body force and one species that turns into gas."""
    rng = np.random.default_rng(seed)
    p = inputs.base_params(nx, ny)
    p.update(periodic_x=1, periodic_y=1, n_species=1, idx_A=0, idx_B=-1, idx_E=-1, idx_F=-1, G11=0.0, G12=0.0, G21=0.0,
             w_adh=(0.0, 0.0), body_force=(3e-4, -2e-4), J0=(0.3, 0, 0, 0), tau_g=(tau_g, 1, 1, 1), k1=2e-3, gas_yield=0.4)
    rho1 = rng.uniform(7.0, 8.5, (ny, nx))
    rho2 = rng.uniform(1e-5, 2e-3, (ny, nx))
    return p, rho1, rho2, rng.uniform(0.2, 1.5, (1, ny, nx))


@pytest.mark.parametrize("tau_g", [0.8])
def test_one_fluid_step_is_correctly_rounded(pslbm, tau_g):
    p, rho1, rho2, conc = reacting(44, 36, tau_g)
    with pslbm.Simulation(np.zeros(rho1.shape, np.uint8), p, rho1, rho2, conc, None, precision=pslbm.FP64) as sim:
        r0 = sim.read()
        sim.step(1)
        got = sim.read()
    y1 = p["gas_yield"] * (p["k1"] * r0["conc"][0])
    for name, S in (("rho1", -y1), ("rho2", y1)):
        rho = r0[name]
        ux, uy = ((rho * g) * (1.0 / rho) for g in p["body_force"])
        f = [fma(w, S, v) for w, v in zip(W9, feq9(rho, ux, uy))]
        np.testing.assert_array_equal(got[name], streamed_sum(f, E9), err_msg=name)


@pytest.mark.parametrize("tau_g", [0.8, 1.0, 3.3])
def test_one_solute_step_is_correctly_rounded(pslbm, tau_g):
    p, rho1, rho2, conc = reacting(44, 36, tau_g, seed=9)
    with pslbm.Simulation(np.zeros(rho1.shape, np.uint8), p, rho1, rho2, conc, None, precision=pslbm.FP64) as sim:
        r0 = sim.read()
        sim.step(1)
        got = sim.read()
    r1, r2, C = r0["rho1"], r0["rho2"], r0["conc"][0]
    J0 = p["J0"][0]
    J = [J0] + [(1.0 - J0) / 4.0] * 4
    h = 0.5 * (1.0 / (r1 + r2))
    ux, uy = (h * (r1 * g + r2 * g) for g in p["body_force"])      # no momentum yet
    sa, ax, ay = J[1] * C, (0.5 * C) * ux, (0.5 * C) * uy
    ge = [J0 * C, sa + ax, sa + ay, sa - ax, sa - ay]
    S = -(p["k1"] * C)
    go = [fma(J[a], S, fma(ge[a] - J[a] * conc[0], 1.0 / tau_g, J[a] * conc[0])) for a in range(5)]
    np.testing.assert_array_equal(got["conc"][0], streamed_sum(go, E9))


def test_potentials_of_eq_15(pslbm):
    """phi_1 = 1 - exp(-x), x = rho_2 / rho_20, is a series below 1/16; phi_2 = a0 -
    exp(-z), z = rho_1 / rho_10, is a0 where the exponential is below half an ulp of it.
    Sources (rho_2 > 0) stand alone in fours, so that the velocity of the node east of
    one is G21 phi_2 (own) phi_1 (source) / 9 / (2 rho_1).  Bounds: phi_1 to an ulp, phi_2
    to an ulp of a0 + exp(-z) and the rounding of z, and six roundings more."""
    n = 64
    p = inputs.base_params(n, n)
    p.update(periodic_x=1, periodic_y=1, n_species=0, idx_A=-1, idx_B=-1, idx_E=-1, idx_F=-1, G11=0.0, G12=0.0, G21=1.0,
             w_adh=(0.0, 0.0), body_force=(0.0, 0.0))
    m = n // 4
    k = m * m
    cut = math.log(2.0 ** 55 / p["a0"])
    x = np.concatenate([np.geomspace(1e-12, 0.06, k // 2), 0.0625 * (1 + np.linspace(-1e-3, 1e-3, k // 4)),
                        np.nextafter(0.0625, [0, 1]), np.geomspace(0.063, 30.0, k - k // 2 - k // 4 - 2)])
    z = np.concatenate([np.geomspace(1e-3, 30.0, k // 2), cut * (1 + np.linspace(-0.02, 0.02, k // 4)),
                        np.linspace(cut + 1, 300.0, k - k // 2 - k // 4)])
    z = np.random.default_rng(3).permutation(z)
    rho1, rho2 = np.full((n, n), 0.1), np.zeros((n, n))
    rho2[::4, 1::4] = (x * p["rho20"]).reshape(m, m)
    rho1[::4, 2::4] = (z * p["rho10"]).reshape(m, m)
    with pslbm.Simulation(np.zeros((n, n), np.uint8), p, rho1, rho2, None, None, precision=pslbm.FP64) as sim:
        got = sim.read()
    L = np.longdouble
    r1, r2 = got["rho1"][::4, 2::4].astype(L), got["rho2"][::4, 1::4].astype(L)
    ex = np.exp(-r1 / L(p["rho10"]))
    phi1, phi2 = -np.expm1(-r2 / L(p["rho20"])), L(p["a0"]) - ex
    want = phi2 * phi1 / 9 / (2 * r1)
    eps = 2.0 ** -53
    bound = eps * phi1 / 9 / (2 * r1) * (12 * np.abs(phi2) + 2 * p["a0"] + 2 * ex * (1 + 2 * r1 / L(p["rho10"])))
    err = np.abs(got["ux"][::4, 2::4].astype(L) - want)
    worst = np.unravel_index((err / bound).argmax(), err.shape)
    assert (err <= bound).all(), (float((err / bound).max()), float(r2[worst] / p["rho20"]), float(r1[worst] / p["rho10"]))

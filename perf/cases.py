"""The work a user of this library has it do, as cases with a fixed set of
inputs, so that two builds can be timed and compared on the same calls.

A case is a dict of plain values; `prepare` builds what a program holds before
the call (the simulation handle, the batch, or the queued scenes), `run` is one
pass through the public Python binding, `exact` the same numbers from a plain
FP64 torch restatement of the method.

Kinds of pass:
  steps   an existing simulation advances `steps` time steps and its whole
          state is read back (the loop of every long run);
  batch   an existing batch of geometries advances `steps` steps and every
          member's state is read back;
  server  a list of requests is submitted to a new server, advanced until all
          are done, and their fields fetched (creation, batching, budgets and
          read-out included).
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_1410_3464_gb300 import inputs, pslbm

PRECISIONS = {"fp64": pslbm.FP64, "fp32": pslbm.FP32, "fp16": pslbm.FP32_SOLUTE_F16, "bf16": pslbm.FP32_SOLUTE_BF16}
FIELDS = (pslbm.F_RHO1 | pslbm.F_RHO2 | pslbm.F_UX | pslbm.F_UY | pslbm.F_CONC | pslbm.F_TYPE | pslbm.F_VOL)
NAMES = ("rho1", "rho2", "ux", "uy", "conc", "type", "vol")
SPECIES = {"plain": 2, "beaker": 4, "droplet": 0, "fracture": 1, "porous": 3}
FLUID = {"plain": 0.92, "beaker": 0.93, "droplet": 0.99, "fracture": 0.34, "porous": 0.6}


def listed():
    return [
        # one step of the plain 128x64 scene and its fields: a coupling or
        # debugging loop that looks at every step (all latency)
        dict(name="plain_128x64_fp64_1", kind="steps", scene="plain", nx=128, ny=64, precision="fp64", steps=1),
        # the plain scene as the parity runs use it, in long strides
        dict(name="plain_128x64_fp64", kind="steps", scene="plain", nx=128, ny=64, precision="fp64", steps=200),
        # the paper's beaker (four transported species, all four reactions)
        dict(name="beaker_100x160_fp32", kind="steps", scene="beaker", nx=100, ny=160, precision="fp32", steps=200),
        # the contact-angle study: no species, an odd periodic lattice
        dict(name="droplet_201x201_fp64", kind="steps", scene="droplet", nx=201, ny=201, precision="fp64", steps=200),
        # the fracture study: one species, single phase, dissolving walls
        dict(name="fracture_102x90_fp64", kind="steps", scene="fracture", nx=102, ny=90, precision="fp64", steps=200),
        # a porous sample of odd size (rows that no vector load divides)
        dict(name="porous_333x217_fp32", kind="steps", scene="porous", nx=333, ny=217, precision="fp32", steps=200),
        # the benchmark's single lattice in the three storage precisions
        dict(name="porous_1024x512_fp32", kind="steps", scene="porous", nx=1024, ny=512, precision="fp32", steps=200),
        dict(name="porous_1024x512_fp16", kind="steps", scene="porous", nx=1024, ny=512, precision="fp16", steps=200),
        dict(name="porous_1024x512_fp64", kind="steps", scene="porous", nx=1024, ny=512, precision="fp64", steps=100),
        # the large lattice
        dict(name="porous_4096x2048_fp32", kind="steps", scene="porous", nx=4096, ny=2048, precision="fp32", steps=300),
        # geometries of the benchmark's request trace stepped as one batch
        dict(name="batch_24_fp32", kind="batch", members=24, max_side=1024, trace=4, precision="fp32", steps=200),
        # a short queue of requests served from submission to fetched fields
        dict(name="server_8_fp32", kind="server", members=8, max_side=512, max_budget=800, trace=5, precision="fp32"),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["steps"] * 6 + ["batch", "server"])
    if kind == "batch":
        return dict(kind=kind, members=rng.randint(4, 24), max_side=rng.choice([256, 512, 768]), trace=rng.randint(1, 999),
                    precision=rng.choice(["fp32", "fp32", "fp16", "fp64"]), steps=_log_int(rng, 20, 100))
    if kind == "server":
        return dict(kind=kind, members=rng.randint(2, 8), max_side=rng.choice([192, 320, 512]),
                    trace=rng.randint(1, 999), max_budget=_log_int(rng, 200, 800), precision=rng.choice(["fp32", "bf16"]))
    scene = rng.choice(["plain", "beaker", "droplet", "fracture", "porous", "porous", "porous"])
    precision = rng.choice(["fp64", "fp32", "fp32", "fp16", "bf16"])
    if scene in ("droplet",) and precision in ("fp16", "bf16"):
        precision = "fp32"                       # 16-bit storage needs species
    if scene == "beaker":
        nx, ny = rng.randint(64, 160), rng.randint(130, 220)
    elif scene == "droplet":
        nx = rng.randint(121, 301)
        ny = rng.randint(nx // 2 + 30, nx + 40)
    elif scene == "fracture":
        nx, ny = rng.randint(60, 300), rng.randint(60, 160)
    elif scene == "plain":
        nx, ny = _log_int(rng, 80, 400), _log_int(rng, 48, 200)
    else:
        nx, ny = _log_int(rng, 128, 2048), _log_int(rng, 128, 1024)
    # the number of steps shrinks as the lattice grows, and in FP64
    most = 2.0e8 / (nx * ny) / (8.0 if precision == "fp64" else 1.0)
    return dict(kind=kind, scene=scene, nx=nx, ny=ny, precision=precision, steps=max(1, min(_log_int(rng, 1, 400), int(most))))


# ------------------------------------------------------------------- inputs

def _scene(case, seed):
    """The scene of a case from a seed: geometry, densities, concentrations,
    volumes and parameters (host arrays, what pslbm_create takes)."""
    rng = np.random.default_rng(seed)
    nx, ny, name = case["nx"], case["ny"], case["scene"]
    if name == "plain":
        r = 0.19 * ny
        sc = inputs.bubble_grain(nx, ny, grain=(0.5 * nx + rng.uniform(-4, 4), 0.5 * ny + rng.uniform(-2, 2), r),
                                 bubble=(0.19 * nx + rng.uniform(-2, 2), 0.5 * ny + rng.uniform(-2, 2), 0.8 * r))
    elif name == "beaker":
        r = 0.15 * nx
        sc = inputs.beaker(nx, ny, grain=(0.5 * nx + rng.uniform(-3, 3), 0.31 * ny + rng.uniform(-3, 3), r),
                           level=int(0.625 * ny) + int(rng.integers(-3, 4)))
    elif name == "droplet":
        sc = inputs.droplet(nx, ny, radius=0.25 * nx + rng.uniform(-3, 3), w=-0.1 * rng.uniform())
    elif name == "fracture":
        sc = inputs.fracture(L=nx - 2, H=ny, h0=ny // 3, conc_in=0.5 + 0.5 * rng.uniform())
    else:
        # few and small bubbles, half the default driving gradient and a slow R1
        # (whose gas accumulates): the scene stays in the EOS domain for tens of
        # thousands of steps, whatever the seed
        gseed = int(rng.integers(1, 1 << 20))
        rmax = max(4.0, min(24.0, min(nx, ny) / 6.0))
        sc = inputs.porous_discs(nx, ny, seed=gseed, rmin=min(8.0, rmax / 2), rmax=rmax, k1=1e-6, bubbles=max(1, nx * ny // 6667),
                                 bubble_r=(3.0, 6.0), overpressure=1.0 + 0.005 * min(1.0, nx / 1024.0))
    mask, p = sc["mask"], sc["params"]
    ns = p["n_species"]
    if name == "porous":
        # solutes as a run restarted after about a thousand steps holds them
        top = np.array([0.02, 0.003, 0.004]).reshape(3, 1, 1)
        smooth = 0.5 + 0.5 * np.sin(np.arange(nx) * (2 * np.pi * 3 / nx) + rng.uniform(0, 6.28, (3, 1, 1)))
        noise = rng.random((3, ny, nx), dtype=np.float32)
        sc["conc"] = np.where(mask == inputs.LIQUID, top * smooth * (0.9 + 0.1 * noise), 0.0)
    elif name == "plain":
        # product already dissolving the grain, whose rim is partly consumed:
        # nodes of it turn liquid as the run goes on
        sc["conc"][1][mask == inputs.LIQUID] = 0.2 + 0.2 * rng.uniform()
        vd = np.where(mask == inputs.SOLID_D, rng.uniform(0.01, 1.0, mask.shape), 0.0)
        sc["vol"] = np.stack([vd, np.zeros_like(vd)])
    elif name == "fracture":
        sc["conc"][0][mask == inputs.LIQUID] = rng.uniform(0.2, 0.6)
    elif name == "beaker":
        sc["conc"][1][mask == inputs.LIQUID] = 0.01 * rng.uniform(0.5, 1.0)
    assert ns == SPECIES[name]
    return sc


def _trace(case):
    """Sizes, porosities, rates and budgets of the benchmark's request generator
    for the case's trace number."""
    return inputs.request_stream(case["members"], seed=case["trace"], size_range=(128, case["max_side"]),
                                 budget_range=(200, max(201, case.get("max_budget", 800))), stop_fraction=0.0)


def _requests(case, seed):
    """The requests of a trace with geometries and bubbles from the seed, at the
    gentle flow of the porous scene above."""
    out = []
    for r in _trace(case):
        _, k3, k2, k4 = r["rates"]
        rmax = max(4.0, min(24.0, min(r["nx"], r["ny"]) / 6.0))
        sc = inputs.porous_discs(r["nx"], r["ny"], seed=r["seed"] + seed, porosity=r["porosity"], rmin=min(8.0, rmax / 2),
                                 rmax=rmax, k1=1e-6, k3=k3, k2=min(k2, 1e-2), k4=min(k4, 1e-2), bubble_r=(3.0, 6.0),
                                 bubbles=max(1, r["nx"] * r["ny"] // 6667), overpressure=1.0 + 0.005 * min(1.0, r["nx"] / 1024.0))
        out.append((sc, r["step_budget"]))
    return out


def _simulation(sc, precision):
    return pslbm.Simulation(sc["mask"], sc["params"], sc["rho1"], sc["rho2"], sc["conc"], sc["vol"], precision=PRECISIONS[precision])


def prepare(case, seed):
    if case["kind"] == "steps":
        return dict(kind="steps", sim=_simulation(_scene(case, seed), case["precision"]), steps=case["steps"])
    if case["kind"] == "batch":
        sims = [_simulation(sc, case["precision"]) for sc, _ in _requests(case, seed)]
        return dict(kind="batch", batch=pslbm.Batch(sims), sims=sims, steps=case["steps"])
    return dict(kind="server", requests=_requests(case, seed), precision=PRECISIONS[case["precision"]])


def run(state):
    if state["kind"] == "steps":
        sim = state["sim"]
        sim.step(state["steps"])
        got = sim.read(FIELDS)
        return {k: got[k] for k in NAMES if got[k].size}
    if state["kind"] == "batch":
        state["batch"].step(state["steps"])
        state["batch"].sync()
        got = [s.read(FIELDS) for s in state["sims"]]
        return {k: np.concatenate([g[k].ravel() for g in got]) for k in NAMES}
    srv = pslbm.Server(precision=state["precision"], chunk_steps=100)
    ids = [srv.submit(sc["mask"], sc["params"], sc["rho1"], sc["rho2"], sc["conc"], sc["vol"], step_budget=budget, keep_fields=True)
           for sc, budget in state["requests"]]
    while sum(srv.advance()[:2]):
        pass
    got = [srv.fetch(i) for i in ids]
    srv.close()
    return got


def work(case):
    """Per time step: every population, solute population and node type read
    once and written once at the nodes that hold them; then the state read out.
    Operations per fluid node and step as counted for the FP64 kernel with three
    species (675), less 65 for each species a scene does not have."""
    if case["kind"] == "steps":
        ns, fluid, lattices = SPECIES[case["scene"]], FLUID[case["scene"]], [(case["nx"] * case["ny"], case["steps"])]
    else:
        ns, fluid = 3, 0.6
        lattices = [(r["nx"] * r["ny"], case.get("steps", r["step_budget"])) for r in _trace(case)]
    sf = 8 if case["precision"] == "fp64" else 4
    sg = {"fp64": 8, "fp32": 4}.get(case["precision"], 2)
    step_bytes = fluid * (36 * sf + 10 * ns * sg) + 2
    read = 8 * (6 + ns) + 1
    return {"bytes": sum(n * (steps * step_bytes + read) for n, steps in lattices),
            "flops": sum(n * steps for n, steps in lattices) * fluid * (480 + 65 * ns)}


# ------------------------------------------------- the same numbers in 64 bits

LIQUID, GAS, SOLID_D, SOLID_F, WALL, INLET, OUTLET = range(7)
EX = (0, 1, 0, -1, 0, 1, -1, -1, 1)
EY = (0, 0, 1, 0, -1, 1, 1, -1, -1)
OPP = (0, 3, 4, 1, 2, 7, 8, 5, 6)
W9 = (4 / 9,) + (1 / 9,) * 4 + (1 / 36,) * 4


class _Exact:
    """The time step in FP64 torch, whole arrays, from the method's equations
    (forces with mirror-image walls, lagged half-maximum marking, halfway
    bounce-back, reactive links, volume of pixel).  Overflowing nodes are not
    modelled: `spilled` records that one occurred."""

    def __init__(self, sc):
        self.dev = torch.device("cuda" if torch.cuda.is_available() else "cpu")
        p = self.p = sc["params"]
        t = lambda a: torch.as_tensor(np.ascontiguousarray(a), device=self.dev)  # noqa: E731
        self.px, self.py, self.ns = bool(p["periodic_x"]), bool(p["periodic_y"]), p["n_species"]
        self.type = t(sc["mask"])
        self.type0 = self.type.clone()
        fluid = self.type <= GAS
        z = torch.zeros((), dtype=torch.float64, device=self.dev)
        r1, r2 = (torch.where(fluid, t(sc[k]).double(), z) for k in ("rho1", "rho2"))
        self.f = [[w * r for w in W9] for r in (r1, r2)]
        self.theta = 0.5 * torch.where(fluid, r1, z).max()
        c = [torch.where(self.type == LIQUID, t(sc["conc"][k]).double(), z) for k in range(self.ns)] if self.ns else []
        self.g = [[self.j(k, a) * c[k] for a in range(5)] for k in range(self.ns)]
        self.V = [(self.type == SOLID_D).double(), (self.type == SOLID_F).double()] if sc["vol"] is None else [t(v).double() for v in sc["vol"]]
        self.spilled = torch.zeros((), dtype=torch.bool, device=self.dev)
        self.step_no = 0
        self.res_any = bool(((self.type == INLET) | (self.type == OUTLET)).any())
        self.zero = torch.zeros_like(r1)

    def j(self, k, a):
        J0 = self.p["J0"][k]
        return J0 if a == 0 else (1.0 - J0) / 4.0

    def nb(self, a, dx, dy, fill):
        out = torch.roll(a, (-dy, -dx), (0, 1)) if dx or dy else a
        if dx and not self.px:
            out[:, -1 if dx > 0 else 0] = fill
        if dy and not self.py:
            out[-1 if dy > 0 else 0, :] = fill
        return out

    def moments(self):
        m = []
        for f in self.f:
            m.append((sum(f[1:], f[0]), f[1] - f[3] + f[5] - f[6] + f[8] - f[7], f[2] - f[4] + f[5] - f[8] + f[6] - f[7]))
        return m

    def reservoirs(self, fluid, m):
        """Densities and velocities of the reservoir nodes."""
        p, typ = self.p, self.type
        if not self.res_any:
            return self.zero, self.zero, self.zero, self.zero
        inlet, outlet = typ == INLET, typ == OUTLET
        idx, idy = (1, 0) if p["inlet_axis"] == 0 else (0, 1)
        odx, ody = (-1, 0) if p["outlet_axis"] == 0 else (0, -1)
        up = self.nb(fluid & (m[0][0] > self.theta), odx, ody, False)
        rho = torch.where(fluid, m[0][0] + m[1][0], 1.0)
        out = []
        for s in range(2):
            ro = torch.where(up, self.zero + p["rho_out"][s], p["rho_out_gas"][s])
            out.append(torch.where(inlet, p["rho_in_liq"][s], torch.where(outlet, ro, 0.0)))
        for i in (1, 2):
            u = torch.where(fluid, (m[0][i] + m[1][i]) / rho, self.zero)
            out.append(torch.where(inlet, self.nb(u, idx, idy, 0.0), torch.where(outlet, self.nb(u, odx, ody, 0.0), self.zero)))
        return out

    def forces(self, fluid, m, r1res, r2res):
        p = self.p
        live = fluid | (self.type == INLET) | (self.type == OUTLET)
        r1, r2 = torch.where(fluid, m[0][0], r1res), torch.where(fluid, m[1][0], r2res)
        eta = p["eos_b"] * r1 / 4.0
        pr = r1 * p["eos_R"] * p["eos_T"] * (1 + eta + eta**2 - eta**3) / (1 - eta) ** 3 - p["eos_a"] * r1**2
        psi = torch.sqrt(torch.where(live, 6.0 / p["G11"] * (pr - r1 / 3.0), self.zero).clamp(min=0.0))
        phi1 = torch.where(live, -torch.expm1(-r2 / p["rho20"]), self.zero)
        phi2 = torch.where(live, p["a0"] - torch.exp(-r1 / p["rho10"]), self.zero)
        lv = [live] + [self.nb(live, EX[a], EY[a], False) for a in range(1, 9)]

        def wsum(v):
            n = [v] + [self.nb(v, EX[a], EY[a], 0.0) for a in range(1, 9)]
            q = [v]
            for a in range(1, 9):
                if a < 5:
                    image = v
                else:
                    h, w = (1 if EX[a] > 0 else 3), (2 if EY[a] > 0 else 4)
                    image = torch.where(lv[h] & ~lv[w], n[h], torch.where(lv[w] & ~lv[h], n[w], v))
                q.append(torch.where(lv[a], n[a], image))
            return ((q[1] - q[3]) / 9 + (q[5] - q[7] + q[8] - q[6]) / 36, (q[2] - q[4]) / 9 + (q[5] - q[7] - q[8] + q[6]) / 36)

        sp, s2, s1 = wsum(psi), wsum(phi2), wsum(phi1)
        s = [0.0] + [(~lv[a]).double() for a in range(1, 9)]
        ss = ((s[1] - s[3]) / 9 + (s[5] - s[7] + s[8] - s[6]) / 36, (s[2] - s[4]) / 9 + (s[5] - s[7] - s[8] + s[6]) / 36)
        F1 = [-p["G11"] * psi * sp[i] - p["G12"] * phi1 * s2[i] - p["w_adh"][0] * psi * ss[i] + m[0][0] * p["body_force"][i] for i in (0, 1)]
        F2 = [-p["G21"] * phi2 * s1[i] - p["w_adh"][1] * m[1][0] * ss[i] + m[1][0] * p["body_force"][i] for i in (0, 1)]
        return F1, F2

    def velocities(self, fluid, m, F1, F2):
        t1, t2 = self.p["tau"]
        r1, r2 = torch.where(fluid, m[0][0], 1.0), torch.where(fluid, m[1][0], 1.0)
        den = r1 / t1 + r2 / t2
        u1, u2, ur = [], [], []
        for i in (0, 1):
            j1, j2 = m[0][i + 1], m[1][i + 1]
            up = (j1 / t1 + j2 / t2) / den
            u1.append(up + torch.where(r1 == 0, self.zero, t1 * F1[i] / r1))
            u2.append(up + torch.where(r2 == 0, self.zero, t2 * F2[i] / r2))
            ur.append((j1 + j2 + 0.5 * (F1[i] + F2[i])) / (r1 + r2))
        return u1, u2, ur

    @staticmethod
    def feq(a, rho, u):
        eu = EX[a] * u[0] + EY[a] * u[1]
        return W9[a] * rho * (1 + 3 * eu + 4.5 * eu * eu - 1.5 * (u[0] * u[0] + u[1] * u[1]))

    def step(self):
        p, typ, ns, nb, zero = self.p, self.type, self.ns, self.nb, self.zero
        fluid = typ <= GAS
        res = (typ == INLET) | (typ == OUTLET)
        m = self.moments()
        rho1, rho2 = m[0][0], m[1][0]
        r1res, r2res, uxr, uyr = self.reservoirs(fluid, m)
        liq, old = fluid & (rho1 > self.theta), typ == LIQUID
        res_liq = res & (r1res > self.theta)
        C = [sum(g[1:], g[0]) for g in self.g]
        C0, g = C, self.g
        if ns:     # solutes of nodes whose marking changed
            gone, new, stay = old & ~liq, fluid & ~old & liq, old & liq
            nrec = sum(nb(liq, EX[b], EY[b], False).double() for b in range(1, 5))
            share = torch.where(gone & (nrec > 0), 1.0 / nrec.clamp(min=1.0), zero)
            nsrc = sum(nb(stay, EX[b], EY[b], False).double() for b in range(1, 5)).clamp(min=1.0)
            g = []
            for k in range(ns):
                cs, cm = C[k] * share, torch.where(stay, C[k], zero)
                dC = sum(nb(cs, EX[b], EY[b], 0.0) for b in range(1, 5))
                base = sum(nb(cm, EX[b], EY[b], 0.0) for b in range(1, 5)) / nsrc
                g.append([torch.where(new, self.j(k, a) * (base + dC), torch.where(stay, self.g[k][a] + self.j(k, a) * dC, self.g[k][a])) for a in range(5)])
            C = [sum(x[1:], x[0]) for x in g]
        F1, F2 = self.forces(fluid, m, r1res, r2res)
        u1, u2, ur = self.velocities(fluid, m, F1, F2)
        # homogeneous reactions
        S, R1 = [zero] * ns, zero
        iA, iB, iE, iF = p["idx_A"], p["idx_B"], p["idx_E"], p["idx_F"]
        if ns:
            CB, CE = (C[i] if i >= 0 else zero for i in (iB, iE))
            CA = C[iA] if iA >= 0 else (p["c_total_per_rho1"] * rho1 - sum(C)).clamp(min=0.0) if iA == -2 else zero
            near = torch.zeros_like(fluid)
            for b in range(1, 5):
                near = near | (nb(typ, EX[b], EY[b], WALL) == SOLID_D)
            k1 = torch.where(near, zero + p["k1"] * (p["r1_surface_factor"] or 1.0), p["k1"])
            R1 = torch.where(liq, k1 * (CA - p["inv_Keq"] * CB * torch.sqrt((rho2 * p["inv_M_C"]).clamp(min=0.0))), zero)
            R3 = torch.where(liq, p["k3"] * CB * CE, zero)
            for i, r in ((iA, -R1), (iB, R1 - R3), (iE, -R3), (iF, R3)):
                if i >= 0:
                    S[i] = S[i] + r
        # fluid collision and streaming
        src = [nb(typ, -EX[a], -EY[a], WALL) for a in range(9)]
        fnew = []
        for s, (rho, u, sgn, rr) in enumerate(((rho1, u1, -1.0, r1res), (rho2, u2, 1.0, r2res))):
            star = [self.f[s][a] - (self.f[s][a] - self.feq(a, rho, u)) / p["tau"][s] + W9[a] * sgn * p["gas_yield"] * R1 for a in range(9)]
            out = []
            for a in range(9):
                v = torch.where(src[a] <= GAS, nb(star[a], -EX[a], -EY[a], 0.0), star[OPP[a]])
                if self.res_any:
                    v = torch.where(src[a] >= INLET, nb(self.feq(a, rr, (uxr, uyr)), -EX[a], -EY[a], 0.0), v)
                out.append(torch.where(fluid, v, self.f[s][a]))
            fnew.append(out)
        # solute collision and streaming, reactive links
        gnew, qB, qF = [], [zero] * 5, [zero] * 5
        odx, ody = (-1, 0) if p["outlet_axis"] == 0 else (0, -1)
        star = [[g[k][a] - (g[k][a] - C[k] * (self.j(k, a) + 0.5 * (EX[a] * ur[0] + EY[a] * ur[1]))) / p["tau_g"][k] + self.j(k, a) * S[k]
                 for a in range(5)] for k in range(ns)]
        sliq = [nb(liq, -EX[a], -EY[a], False) for a in range(5)]
        for k in range(ns):
            cres = torch.where(typ == INLET, p["conc_in"][k], torch.where(typ == OUTLET, nb(torch.where(liq, C0[k], zero), odx, ody, 0.0), zero))
            out = [torch.where(liq, star[k][0], zero)]
            for a in range(1, 5):
                v = torch.where(sliq[a], nb(star[k][a], -EX[a], -EY[a], 0.0), star[k][OPP[a]])
                if self.res_any:
                    ge = cres * (self.j(k, a) + 0.5 * (EX[a] * uxr + EY[a] * uyr))
                    v = torch.where(nb(res_liq, -EX[a], -EY[a], False), nb(ge, -EX[a], -EY[a], 0.0), v)
                out.append(torch.where(liq, v, zero))
            gnew.append(out)
        for a in range(1, 5):
            d = OPP[a]
            onD = liq & (src[a] == SOLID_D)
            onM = onD | (liq & (src[a] == SOLID_F))
            if iB >= 0 and p["k2"] != 0.0:
                kap = p["k2"] / (2 * self.j(iB, 1))
                qB[d] = torch.where(onD, star[iB][d] * (2 * kap / (1 + kap)), zero)
                gnew[iB][a] = gnew[iB][a] - qB[d]
                if iE >= 0:
                    gnew[iE][a] = gnew[iE][a] + qB[d]
            if iF >= 0 and p["k4"] != 0.0:
                kap = p["k4"] / (2 * self.j(iF, 1))
                qF[d] = torch.where(onM, star[iF][d] * (2 * kap / (1 + kap)) - p["k4"] * p["C_F_sat"] / (1 + kap), zero)
                gnew[iF][a] = gnew[iF][a] - qF[d]
        # volume of pixel and dissolving nodes
        mineral = (typ == SOLID_D) | (typ == SOLID_F)
        touch = torch.zeros_like(fluid)
        sB, sF = zero, zero
        for b in range(1, 5):
            touch = touch | nb(liq, EX[b], EY[b], False)
            sB = sB + nb(qB[OPP[b]], EX[b], EY[b], 0.0)
            sF = sF + nb(qF[OPP[b]], EX[b], EY[b], 0.0)
        act = mineral & touch
        VD = torch.where(act & (typ == SOLID_D), (self.V[0] - p["Vbar_D"] * sB).clamp(min=0.0), self.V[0])
        VF = torch.where(act, self.V[1] + p["Vbar_F"] * sF, self.V[1])
        diss = act & (VD + VF <= 0)
        self.spilled |= (act & (VD + VF >= p["V_split"])).any()
        t8 = lambda v: torch.full_like(typ, v)  # noqa: E731
        newtyp = torch.where(fluid, torch.where(liq, t8(LIQUID), t8(GAS)), typ)
        newtyp = torch.where(act, torch.where(VD > 0, t8(SOLID_D), t8(SOLID_F)), newtyp)
        newtyp = torch.where(diss, t8(LIQUID), newtyp)
        self.V = [torch.where(diss, zero, VD), torch.where(diss, zero, VF)]
        nf = sum(nb(fluid, EX[b], EY[b], False).double() for b in range(1, 5))
        nl = sum(nb(liq, EX[b], EY[b], False).double() for b in range(1, 5))
        for s in range(2):
            rn = torch.where(fluid, sum(fnew[s][1:], fnew[s][0]), zero)
            fill = torch.where(nf > 0, sum(nb(rn, EX[b], EY[b], 0.0) for b in range(1, 5)) / nf.clamp(min=1.0), p["rho_ref"][s])
            fnew[s] = [torch.where(diss, W9[a] * fill, fnew[s][a]) for a in range(9)]
        for k in range(ns):
            cn = torch.where(liq, sum(gnew[k][1:], gnew[k][0]), zero)
            fill = sum(nb(cn, EX[b], EY[b], 0.0) for b in range(1, 5)) / nl.clamp(min=1.0)
            gnew[k] = [torch.where(diss, self.j(k, a) * fill, gnew[k][a]) for a in range(5)]
        self.theta = 0.5 * torch.where(fluid, rho1, -math.inf).max()
        self.f, self.g, self.type = fnew, gnew, newtyp
        self.step_no += 1

    def fields(self):
        fluid, m = self.type <= GAS, self.moments()
        r1res, r2res, _, _ = self.reservoirs(fluid, m)
        F1, F2 = self.forces(fluid, m, r1res, r2res)
        _, _, ur = self.velocities(fluid, m, F1, F2)
        host = lambda v: torch.where(fluid, v, self.zero).cpu().numpy()  # noqa: E731
        out = dict(rho1=host(m[0][0]), rho2=host(m[1][0]), ux=host(ur[0]), uy=host(ur[1]))
        if self.ns:
            out["conc"] = torch.stack([torch.where(self.type == LIQUID, sum(g[1:], g[0]), self.zero) for g in self.g]).cpu().numpy()
        return dict(out, type=None, vol=torch.stack(self.V).cpu().numpy())


def exact(case, seed):
    if case["kind"] != "steps":
        return None        # many lattices one after another: too long
    e = _Exact(_scene(case, seed))
    for _ in range(case["steps"]):
        e.step()
    return None if bool(e.spilled) else e.fields()

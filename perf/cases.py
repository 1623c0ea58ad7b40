"""The workloads this framework's speed is measured on.

A case is one pass of a program that uses the library the way its README and
its benchmark do: advance a ring-polymer system (or a batch of them, or a
server's jobs) by some MD steps, take the App. A estimators, and read the
state back.  The trajectory goes on from pass to pass unless the case resumes
from its checkpoint.

Sizes come from the repository's own tests and benchmark: 64 oscillators x 8
beads, the 64-molecule x 32-bead box, 512 molecules x 64 beads, the oscillator
sweep, the 256-replica mix, the serving trace; the rest are odd sizes and
keyword combinations of the same ranges (1..128 beads, BAOAB / OBABO, normal
modes / Cartesian beads, NVE / PILE_L, fixcom, fictitious masses, barostats,
FP64 / split precision).

State read from a split-precision engine is kept in single precision, as
trajectory frames are (bead deviations, internal-mode velocities and forces
are FP32 there); FP64 state stays in double precision.
"""
from __future__ import annotations

import math
import random
import time

import numpy as np
import torch

from paper_2602_13553_gb300 import binding, inputs

KB = 8.617333262e-5              # eV / K
PLANCK = 4.135667403e-3          # eV ps
MVV2E = 1.0364269e-4             # eV per amu A^2 / ps^2
HBAR = PLANCK / (2.0 * math.pi)
OMEGA_HO = 0.1 / HBAR            # hbar omega = 0.1 eV
# the water-like liquid's own pressure near 1 g/cm^3 and 300 K (eV/A^3): a
# barostat set to it keeps the box near its starting size over a long run
PEXT = 7.5e-3


# ---------------------------------------------------------------------------
# the cases
# ---------------------------------------------------------------------------
def handle_case(**kw):
    c = dict(engine="handle", potential="water", size=64, beads=32, precision="fp64", integrator="baoab",
             thermostat=True, method="nmpimd", fixcom=False, fmmode="physical", barostat="none",
             deuterium=False, T=300.0, dt_fs=0.5, steps=100, samples=1, resume=False)
    unknown = set(kw) - set(c) - {"name"}
    if unknown:
        raise TypeError("unknown case fields %s" % sorted(unknown))
    c.update(kw)
    return c


def listed():
    return [
        # An outer driver that advances one step at a time and reads the
        # estimators and the state after each (coupling to other programs,
        # debugging): the smallest calls, launches and latency.
        handle_case(name="osc64x8-fp64-each-step", potential="oscillator", size=64, beads=8, dt_fs=0.25, steps=1),
        # The benchmark system, sampled every 100 steps: NVT water box, FP64.
        handle_case(name="water64x32-fp64-nvt"),
        # Constant pressure, the setting of the method's own example input:
        # OBABO with the anisotropic barostat.
        handle_case(name="water125x16-fp64-npt", size=125, beads=16, integrator="obabo", barostat="aniso",
                    dt_fs=0.25, steps=50),
        # Cartesian beads ("method pimd") with the paper's default fixcom yes;
        # a bead count that is no power of two.
        handle_case(name="water100x12-fp64-cartesian", size=100, beads=12, method="pimd", fixcom=True,
                    dt_fs=0.25, steps=50),
        # Odd everything: heavy water, 17 beads, OBABO, fixcom, fictitious
        # masses of fmmode normal.
        handle_case(name="water91x17-fp64-obabo-fixcom", size=91, beads=17, integrator="obabo", fixcom=True,
                    fmmode="normal", deuterium=True, T=260.0, steps=50),
        # A converged low-temperature box in FP64: 1536 atoms x 64 beads.
        handle_case(name="water512x64-fp64-nvt", size=512, beads=64, T=150.0, steps=20),
        # Throughput of the FP64 integrator on a large ideal system (the
        # oscillator sweep at 32 beads).
        handle_case(name="osc65536x32-fp64", potential="oscillator", size=65536, beads=32, dt_fs=0.25, steps=20),
        # The same in split precision, the production setting.
        handle_case(name="osc65536x32-split", potential="oscillator", size=65536, beads=32, precision="split",
                    dt_fs=0.25, steps=100),
        # The large box in split precision, resumed from its checkpoint.
        handle_case(name="water512x64-split-resume", size=512, beads=64, precision="split", steps=20, resume=True),
        # A bead count between the powers of two in split precision.
        handle_case(name="water216x20-split-nvt", size=216, beads=20, precision="split", T=200.0, steps=20),
        # The batched mix: 256 uneven replicas in one engine, sampled.
        dict(name="batch256-mix", engine="batch", replicas=256, beads="8,16,32,64", min_mol=32, max_mol=512,
             steps=20, frames=False),
        # The job server: a burst of uneven jobs, submitted, polled and
        # fetched with their final states.
        dict(name="server24-burst", engine="server", replicas=24, beads="4,8,16,32,64,128", min_mol=32,
             max_mol=512, steps=30, frames=True),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng: random.Random):
    kind = rng.choice(["osc-fp64", "osc-split", "water-fp64", "water-fp64", "water-npt", "water-cart",
                       "water-split", "water-split", "batch", "server"])
    P = rng.choice([rng.choice([4, 8, 16, 32, 64, 128]), rng.randint(2, 100)])
    T = round(rng.uniform(100.0, 400.0), 1)
    integ = rng.choice(["baoab", "baoab", "obabo"])
    if kind in ("osc-fp64", "osc-split"):
        total = _log_int(rng, 512, 1 << 21)          # bead-atoms
        N = max(1, total // P)
        steps = rng.choice([1, 10, 20]) if total > (1 << 18) else rng.choice([1, 20, 100])
        return handle_case(potential="oscillator", size=N, beads=P, precision=kind[4:], integrator=integ,
                           thermostat=rng.random() < 0.8, T=T, dt_fs=0.25, steps=steps)
    nmol = min(_log_int(rng, 24, 512), max(24, 32768 // P))
    steps = rng.choice([1, 10, 20, 40])
    if kind == "water-npt":
        return handle_case(size=max(100, min(nmol, 256)), beads=min(P, 48), integrator=integ,
                           barostat=rng.choice(["iso", "aniso"]), T=300.0, dt_fs=0.25, steps=steps)
    if kind == "water-cart":
        return handle_case(size=nmol, beads=P, method="pimd", integrator=integ, fixcom=rng.random() < 0.5, T=T,
                           dt_fs=0.25, steps=steps)
    if kind == "water-fp64":
        return handle_case(size=nmol, beads=P, integrator=integ, fixcom=rng.random() < 0.3,
                           fmmode=rng.choice(["physical", "physical", "normal"]),
                           deuterium=rng.random() < 0.5, T=T, steps=steps, resume=rng.random() < 0.3)
    if kind == "water-split":
        return handle_case(size=nmol, beads=P, precision="split", integrator=integ,
                           deuterium=rng.random() < 0.5, T=T, steps=min(steps, 20), resume=rng.random() < 0.3)
    lo = rng.randint(24, 64)
    beads = rng.choice(["8,16,32,64", "4,8,16,32,64,128", "%d,%d" % (P, rng.randint(2, 40)), "6,12,24,48"])
    return dict(engine=kind, replicas=_log_int(rng, 2, 96 if kind == "batch" else 16), beads=beads, min_mol=lo,
                max_mol=rng.randint(lo + 8, 400), steps=rng.choice([10, 20, 30]),
                frames=kind == "server" or rng.random() < 0.5)


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------
def _sub_seed(seed, what):
    return int(np.random.SeedSequence([int(seed) & 0x7FFFFFFF, what]).generate_state(1, np.uint32)[0]) & 0x3FFFFFFF


def _water(nmol, P, seed, T, dt_fs, deuterium):
    """One water-like system: box at 1 g/cm^3, cutoff 6 A or 0.48 L."""
    L = inputs.box_length(nmol)
    x0, mass = inputs.water_lattice_box(nmol, L, P, seed, jitter=0.02, deuterium=deuterium)
    return dict(x0=x0, mass=mass, T=T, dt=dt_fs * 1e-3, ff=inputs.water_ff_for_box(L), box=(L, L, L),
                seed=seed + 1)


def _handle_system(case, seed):
    s = _sub_seed(seed, 1)
    if case["potential"] == "oscillator":
        x0, mass = inputs.harmonic(case["size"], case["beads"], seed=s, std=0.1)
        return dict(x0=x0, mass=mass, T=case["T"], dt=case["dt_fs"] * 1e-3, ff=(OMEGA_HO,), box=(0.0, 0.0, 0.0),
                    seed=s + 1)
    return _water(case["size"], case["beads"], s, case["T"], case["dt_fs"], case["deuterium"])


def _handle_params(case):
    return dict(integrator=binding.OBABO if case["integrator"] == "obabo" else binding.BAOAB,
                thermostat=binding.THERMO_PILE_L if case["thermostat"] else binding.THERMO_NONE,
                method=binding.METHOD_PIMD if case["method"] == "pimd" else binding.METHOD_NMPIMD,
                precision=binding.PREC_SPLIT if case["precision"] == "split" else binding.PREC_FP64,
                fixcom=1 if case["fixcom"] else 0,
                fmmode=binding.FMMODE_NORMAL if case["fmmode"] == "normal" else binding.FMMODE_PHYSICAL,
                barostat={"none": 0, "iso": binding.BARO_BZP_ISO, "aniso": binding.BARO_BZP_ANISO}[case["barostat"]],
                pext=PEXT if case["barostat"] != "none" else 0.0, taup=1.0)


def _replica_systems(case, seed):
    """Uneven water-like replicas: molecules log-uniform, bead counts of the
    case's list in turn, T in [100, 400] K, H or D."""
    g = np.random.default_rng(_sub_seed(seed, 2))
    # sizes are part of the case, not of the seed: the work stays the same
    gs = np.random.default_rng(case["replicas"] * 1000003 + case["min_mol"] * 1009 + case["max_mol"])
    beads = [int(b) for b in case["beads"].split(",")]
    out = []
    for r in range(case["replicas"]):
        nmol = int(round(math.exp(gs.uniform(math.log(case["min_mol"]), math.log(case["max_mol"])))))
        P = beads[r % len(beads)]
        out.append(_water(min(nmol, max(case["min_mol"], 32768 // P)), P, int(g.integers(1, 1 << 30)),
                          float(g.uniform(100.0, 400.0)), 0.5, bool(g.random() < 0.5)))
    return out


def _pinned(shape):
    t = torch.empty(shape, dtype=torch.float64, pin_memory=torch.cuda.is_available())
    return t, t.numpy()


def prepare(case, seed):
    st = {"case": case}
    if case["engine"] == "handle":
        s = _handle_system(case, seed)
        prm = _handle_params(case)
        st["sim"] = sim = binding.Simulation(
            s["x0"], s["mass"], T=s["T"], dt=s["dt"], ff=s["ff"], box=s["box"], seed=s["seed"],
            potential=binding.POT_HARMONIC if case["potential"] == "oscillator" else binding.POT_WATERLIKE, **prm)
        st["x_t"], st["x"] = _pinned(s["x0"].shape)
        st["v_t"], st["v"] = _pinned(s["x0"].shape)
        if case["precision"] == "split":
            st["x32"] = torch.empty(s["x0"].shape, dtype=torch.float32)
            st["v32"] = torch.empty(s["x0"].shape, dtype=torch.float32)
        if case["resume"]:
            st["cx_t"], st["cx"] = _pinned(s["x0"].shape)
            st["cv_t"], st["cv"] = _pinned(s["x0"].shape)
            _, _, st["cstep"] = sim.get_state(st["cx"], st["cv"])
        return st
    systems = _replica_systems(case, seed)
    st["systems"] = systems
    n = sum(s["x0"].size for s in systems)
    if case["frames"]:
        st["x"] = np.empty(n, dtype=np.float32)
        st["v"] = np.empty(n, dtype=np.float32)
    if case["engine"] == "batch":
        st["batch"] = b = binding.Batch(len(systems))
        st["slots"] = [b.add(s["x0"], s["mass"], T=s["T"], dt=s["dt"], nsteps=10 ** 12, ff=s["ff"], box=s["box"],
                             seed=s["seed"]) for s in systems]
        return st
    st["server"] = binding.Server(64 << 30, max_replicas=64, chunk_steps=case["steps"], keep_state=True)
    return st


# ---------------------------------------------------------------------------
# one pass
# ---------------------------------------------------------------------------
ENERGIES = ("H", "K_PR", "K_VR", "K_CV")
PRESSURES = ("P_PR", "P_MD", "P_CV")


def _thermo(rows, dtype, periodic):
    """The estimators of several samples (or replicas), one array per kind."""
    out = {k: np.concatenate([r[k] for r in rows]).astype(dtype, copy=False) for k in ("K_mode", "S_mode", "U_bead")}
    out["energies"] = np.array([[r[k] for k in ENERGIES] for r in rows], dtype=dtype)
    out["T_ring"] = np.array([r["T_ring"] for r in rows], dtype=dtype)
    if periodic:
        out["pressures"] = np.array([[r[k] for k in PRESSURES] for r in rows], dtype=dtype)
    return out


def run(state):
    case = state["case"]
    if case["engine"] == "handle":
        sim = state["sim"]
        if case["resume"]:
            sim.set_state(state["cx"], state["cv"], state["cstep"])
        rows = []
        for _ in range(case["samples"]):
            sim.step(case["steps"])
            rows.append(sim.estimators())
        _, _, step = sim.get_state(state["x"], state["v"])
        split = case["precision"] == "split"
        out = _thermo(rows, np.float32 if split else np.float64, case["potential"] == "water")
        if split:
            out["x"] = state["x32"].copy_(state["x_t"])
            out["v"] = state["v32"].copy_(state["v_t"])
        else:
            out["x"], out["v"] = state["x_t"], state["v_t"]
        if case["barostat"] != "none":
            out["box"] = rows[-1]["box"]
            out["vW"] = np.append(rows[-1]["vWa"], rows[-1]["vW"])
            out["enthalpy"] = np.array([r["enthalpy"] for r in rows])
        out["step"] = step
        return out
    if case["engine"] == "batch":
        b = state["batch"]
        b.run(case["steps"])
        est = b.estimators()
        rows = [est[s] for s in state["slots"]]
        fetch = (b.get_state(s) for s in state["slots"])
    else:
        srv = state["server"]
        jobs = [srv.submit(s["x0"], s["mass"], T=s["T"], dt=s["dt"], nsteps=case["steps"], ff=s["ff"],
                           box=s["box"], seed=s["seed"]) for s in state["systems"]]
        done = {}
        while len(done) < len(jobs):
            for j in jobs:
                if j not in done:
                    r = srv.poll(j)
                    if r is not None:
                        done[j] = r
            if len(done) < len(jobs):
                time.sleep(5e-4)
        rows = [done[j] for j in jobs]
        fetch = (srv.get_state(j) for j in jobs)
    out = _thermo(rows, np.float32, True)
    if case["frames"]:
        at = 0
        for x, v, _ in fetch:
            state["x"][at:at + x.size] = x.reshape(-1)
            state["v"][at:at + x.size] = v.reshape(-1)
            at += x.size
        out["x"], out["v"] = state["x"], state["v"]
    out["step"] = np.array([r["step"] for r in rows], dtype=np.int64)
    return out


# ---------------------------------------------------------------------------
# work of one pass
# ---------------------------------------------------------------------------
def _system_work(N, P, water, steps, split, cart):
    """Bytes: the state (x, v) comes in and goes out once a pass (FP64 words:
    the library's host layout), and again every step where it cannot stay on
    the chip (over 100 MB of x, v, F).  Flops per step: three folded
    transforms, the kick, two rotations and the O update; about 200 per
    bead-atom of water forces (30 per O-O pair inside the cutoff, 120 per
    molecule and bead), 6 of a harmonic well."""
    n = N * P
    word = 4 if split else 8
    step_flops = (30.0 if cart else 9.0 * P + 78.0) + (200.0 if water else 6.0)
    state = 9.0 * word * n
    moved = 96.0 * n + (steps * 21.0 * word * n if state > 100e6 else 0.0)
    return moved, steps * step_flops * n


def work(case):
    if case["engine"] == "handle":
        water = case["potential"] == "water"
        N = case["size"] * (3 if water else 1)
        b, f = _system_work(N, case["beads"], water, case["steps"] * case["samples"],
                            case["precision"] == "split", case["method"] == "pimd")
        return {"bytes": b, "flops": f}
    b = f = 0.0
    beads = [int(p) for p in case["beads"].split(",")]
    gs = np.random.default_rng(case["replicas"] * 1000003 + case["min_mol"] * 1009 + case["max_mol"])
    for r in range(case["replicas"]):
        nmol = int(round(math.exp(gs.uniform(math.log(case["min_mol"]), math.log(case["max_mol"])))))
        P = beads[r % len(beads)]
        bb, ff = _system_work(3 * min(nmol, max(case["min_mol"], 32768 // P)), P, True, case["steps"], True, False)
        b += bb
        f += ff
    return {"bytes": b, "flops": f}


# ---------------------------------------------------------------------------
# the same in plain 64-bit torch
# ---------------------------------------------------------------------------
_M32 = 0xFFFFFFFF


def _philox(c0, c1, c2, c3, k0, k1):
    """Philox-4x32-10 on int64 tensors that hold 32-bit words."""
    for r in range(10):
        if r:
            k0 = (k0 + 0x9E3779B9) & _M32
            k1 = (k1 + 0xBB67AE85) & _M32
        a = c0 * 0xD2511F53          # wraps modulo 2^64: both halves stay right
        b = c2 * 0xCD9E8D57
        c0, c1, c2, c3 = ((b >> 32) & _M32) ^ c1 ^ k0, b & _M32, ((a >> 32) & _M32) ^ c3 ^ k1, a & _M32
    return c0, c1, c2, c3


class _Exact:
    """Independent systems of one bead count, side by side, in FP64: x and v
    are [P][n][3] over the atoms of all of them."""

    def __init__(self, systems, case, water, split):
        dev = "cuda" if torch.cuda.is_available() else "cpu"
        f8 = dict(dtype=torch.float64, device=dev)
        self.P = P = systems[0]["x0"].shape[0]
        self.R = R = len(systems)
        self.case, self.water, self.split, self.f8, self.dev = case, water, split, f8, dev
        self.sizes = [s["x0"].shape[1] for s in systems]
        self.x = torch.cat([torch.as_tensor(s["x0"], **f8) for s in systems], dim=1)
        self.mm = torch.cat([torch.as_tensor(s["mass"], **f8) for s in systems]) * MVV2E
        self.rep = torch.repeat_interleave(torch.arange(R, device=dev), torch.tensor(self.sizes, device=dev))
        self.atom = torch.cat([torch.arange(n, device=dev) for n in self.sizes])
        self.T = torch.tensor([s["T"] for s in systems], **f8)
        self.dt = systems[0]["dt"]
        self.box = torch.tensor([s["box"] for s in systems], **f8)
        self.ff = torch.tensor([list(s["ff"]) + [0.0] * (8 - len(s["ff"])) for s in systems], **f8)
        seeds = torch.tensor([s["seed"] for s in systems], dtype=torch.int64, device=dev)[self.rep]
        self.key = (seeds & _M32, (seeds >> 32) & _M32)
        cart = case.get("method") == "pimd"
        self.cart, self.obabo = cart, case.get("integrator") == "obabo"
        self.thermo = case.get("thermostat", True)
        # mode tables per system (Eq. 2, App. B, App. D)
        k = torch.arange(P, **f8)
        j = torch.arange(P, **f8)
        ang = 2.0 * math.pi * torch.remainder(k[:, None] * j[None, :], P) / P
        M = math.sqrt(2.0 / P) * torch.where(2 * k[:, None] < P, torch.cos(ang), torch.sin(ang))
        M[0] = 1.0 / math.sqrt(P)
        if P % 2 == 0:
            M[P // 2] = (1.0 - 2.0 * torch.remainder(j, 2)) / math.sqrt(P)
        self.M = M
        self.lam = 4.0 * torch.sin(math.pi * k / P) ** 2
        self.wn = P * KB * self.T / HBAR
        self.mu = torch.ones(P, **f8)
        if case.get("fmmode") == "normal" and not cart:
            self.mu[1:] = self.lam[1:]
        om = self.wn[None, :] * torch.sqrt(self.lam / self.mu)[:, None]            # [P][R]
        self.tA = self.dt if self.obabo else 0.5 * self.dt
        tO = 0.5 * self.dt if self.obabo else self.dt
        safe = torch.where(om > 0, om, torch.ones_like(om))
        self.cA = torch.cos(om * self.tA)
        self.sA = torch.where(om > 0, torch.sin(om * self.tA) / safe, torch.full_like(om, self.tA))
        self.wA = om * torch.sin(om * self.tA)
        if cart:
            gam = (2.0 * self.wn)[None, :].expand(P, R)
        else:
            gam = 2.0 * om.clone()
            gam[0] = 1.0
        self.c1 = torch.exp(-tO * gam)
        self.c2 = torch.sqrt(1.0 - self.c1 ** 2)
        self.step_no = 0
        self.sig = (P * KB * self.T[self.rep] / self.mm).sqrt()[None, :] / self.mu.sqrt()[:, None]   # [P][n]
        self.v = self.sig[:, :, None] * self.noise(2, 0, full=True)
        # barostat
        self.baro = case.get("barostat", "none")
        self.vW = torch.zeros(3, **f8)
        if self.baro != "none":
            self.Wb = (3.0 if self.baro == "iso" else 1.0) * P * self.sizes[0] * KB * float(self.T[0])   # taup = 1
        if water:
            self._pairs()
        self.forces()

    def noise(self, stream, step, full=False, atom=None, mode=None):
        """N(0, 1) deviates [P][n][3]: Box-Muller on the Philox words, 32-bit
        uniforms (24-bit ones on the split-precision path)."""
        k = torch.arange(self.P, device=self.dev)[:, None] if mode is None else torch.tensor([[mode]], device=self.dev)
        a = self.atom[None, :] if atom is None else torch.tensor([[atom]], device=self.dev)
        k0, k1 = (self.key[0][None, :], self.key[1][None, :]) if atom is None else (self.key[0][:1], self.key[1][:1])
        z = torch.zeros_like(a + k)
        w = _philox(z + a, z + (k | (stream << 16)), z + (step & _M32), z + (step >> 32), k0, k1)
        if self.split and not full:
            u = [((t >> 8).double() + 0.5) * 2.0 ** -24 for t in w]
        else:
            u = [(t.double() + 0.5) * 2.0 ** -32 for t in w]
        r0, r1 = torch.sqrt(-2.0 * torch.log(u[0])), torch.sqrt(-2.0 * torch.log(u[2]))
        return torch.stack([r0 * torch.cos(2 * math.pi * u[1]), r0 * torch.sin(2 * math.pi * u[1]),
                            r1 * torch.cos(2 * math.pi * u[3])], dim=-1)

    def _pairs(self):
        """O-O pairs whose centroids start within the cutoff + 4 A: no bead
        pair of another pair comes inside the cutoff over the short runs here."""
        ii, jj, at = [], [], 0
        c = self.x[:, 0::3].mean(dim=0)
        for r, n in enumerate(self.sizes):
            m = n // 3
            cr = c[at:at + m]
            d = cr[:, None, :] - cr[None, :, :]
            d = d - self.box[r] * torch.round(d / self.box[r])
            near = (d * d).sum(-1) < (self.ff[r, 6] + 4.0) ** 2
            i, j = torch.nonzero(torch.triu(near, 1), as_tuple=True)
            ii.append(i + at)
            jj.append(j + at)
            at += m
        self.pi, self.pj = torch.cat(ii), torch.cat(jj)
        self.mrep = self.rep[0::3]

    def forces(self):
        P, R = self.P, self.R
        x = self.x
        self.U = torch.zeros(P, R, **self.f8)
        self.vir = torch.zeros(P, R, 3, **self.f8)
        if not self.water:
            ks = self.mm * self.ff[self.rep, 0] ** 2
            self.F = -ks[None, :, None] * x
            u = (0.5 * ks[None, :, None] * x * x).sum(-1)
            self.U.index_add_(1, self.rep, u)
            self.vir.index_add_(1, self.rep, x * self.F)
            return
        F = torch.zeros_like(x)
        box = self.box[self.mrep]
        ff = self.ff[self.mrep]
        O = x[:, 0::3]
        d = []
        for h in (1, 2):
            e = x[:, h::3] - O
            d.append(e - box * torch.round(e / box))
        r = [e.norm(dim=-1) for e in d]
        fh = []
        u = torch.zeros_like(r[0])
        for e, rr in zip(d, r):
            dr = rr - ff[:, 1]
            u = u + 0.5 * ff[:, 0] * dr * dr
            fh.append(-(ff[:, 0] * dr / rr)[..., None] * e)
        cth = (d[0] * d[1]).sum(-1) / (r[0] * r[1])
        th = torch.acos(cth.clamp(-1.0, 1.0))
        dth = th - ff[:, 3]
        u = u + 0.5 * ff[:, 2] * dth * dth
        pref = ff[:, 2] * dth / torch.sqrt(1.0 - cth * cth)
        for h in (0, 1):
            g = 1 - h
            fh[h] = fh[h] + pref[..., None] * (d[g] / (r[0] * r[1])[..., None] - (cth / r[h] ** 2)[..., None] * d[h])
        self.U.index_add_(1, self.mrep, u)
        self.vir.index_add_(1, self.mrep, d[0] * fh[0] + d[1] * fh[1])
        F[:, 1::3] = fh[0]
        F[:, 2::3] = fh[1]
        FO = -(fh[0] + fh[1])
        pr = self.mrep[self.pi]
        pb, pf = self.box[pr], self.ff[pr]
        lo, per = 0, max(1, (1 << 26) // max(1, P))
        while lo < len(self.pi):      # pairs in slices, to bound the memory
            s = slice(lo, lo + per)
            e = O[:, self.pj[s]] - O[:, self.pi[s]]
            e = e - pb[s] * torch.round(e / pb[s])
            r2 = (e * e).sum(-1)
            inside = r2 < pf[s, 6] ** 2
            s6 = (pf[s, 5] ** 2 / r2) ** 3
            zero = torch.zeros_like(r2)
            self.U.index_add_(1, pr[s], torch.where(inside, 4.0 * pf[s, 4] * (s6 * s6 - s6), zero))
            fp = torch.where(inside, 24.0 * pf[s, 4] * (2.0 * s6 * s6 - s6) / r2, zero)[..., None] * e
            FO.index_add_(1, self.pj[s], fp)
            FO.index_add_(1, self.pi[s], -fp)
            self.vir.index_add_(1, pr[s], e * fp)
            lo += per
        F[:, 0::3] = FO
        self.F = F

    def _nm(self, a):
        return torch.tensordot(self.M, a, dims=([1], [0]))

    def _kick(self, t):
        if self.cart:
            ring = 2.0 * self.x - torch.roll(self.x, 1, 0) - torch.roll(self.x, -1, 0)
            f = self.F - (self.mm * self.wn[self.rep] ** 2)[None, :, None] * ring
            self.v = self.v + t * f / self.mm[None, :, None]
        else:
            self.v = self.v + t * self._nm(self.F) / (self.mm[None, :] * self.mu[:, None])[..., None]

    def _drift(self, q):
        """A of length tA on every mode (the centroid by hand under a barostat)."""
        if self.cart:
            self.x = self.x + self.tA * self.v
            return q
        c, s, w = (t[:, self.rep][..., None] for t in (self.cA, self.sA, self.wA))
        qn, vn = c * q + s * self.v, c * self.v - w * q
        if self.baro != "none":
            a = self.tA * self.vW
            ea, ema = torch.exp(a), torch.exp(-a)
            sh = torch.where(a.abs() < 1e-8, self.tA * (1.0 + a * a / 6.0),
                             (ea - ema) / (2.0 * torch.where(self.vW == 0, torch.ones_like(a), self.vW)))
            qn[0] = ea * q[0] + sh * self.v[0]
            vn[0] = ema * self.v[0]
            self.box = self.box * ea
        self.v = vn
        return qn

    def _bath(self, stream):
        if not self.thermo:
            return
        self.v = (self.c1[:, self.rep][..., None] * self.v +
                  (self.c2[:, self.rep] * self.sig)[..., None] * self.noise(stream, self.step_no))
        if self.baro != "none":
            tO = 0.5 * self.dt if self.obabo else self.dt
            c1 = math.exp(-tO)                       # tau = 1 ps
            e = self.noise(3, self.step_no, atom=0xFFFFFFFF, mode=stream)[0, 0]
            sg = math.sqrt((1.0 - c1 * c1) * self.P * KB * float(self.T[0]) / self.Wb)
            self.vW = c1 * self.vW + sg * (e if self.baro == "aniso" else e[0])

    def _baro_kick(self, t):
        if self.baro == "none":
            return
        mm = self.mm[:, None]
        f0, v0 = self._nm(self.F)[0], self.v[0]
        rcf = ((self.x - self.x.mean(dim=0)) * self.F).sum((0, 1))
        mv2, fv, f2m = (mm * v0 * v0).sum(0), (f0 * v0).sum(0), (f0 * f0 / mm).sum(0)
        vir = self.vir.sum((0, 1))
        V = self.box[0].prod()
        nkT = self.P * KB * self.T[0]
        if self.baro == "iso":
            self.vW = self.vW + (3.0 * t / self.Wb * ((mv2 - rcf + vir).sum() / 3.0 - self.P * V * PEXT + nkT) +
                                 t * t / self.Wb * fv.sum() + t ** 3 / (3.0 * self.Wb) * f2m.sum())
        else:
            self.vW = self.vW + (t / self.Wb * (mv2 - rcf + vir - self.P * V * PEXT + nkT) + t * t / self.Wb * fv +
                                 t ** 3 / (3.0 * self.Wb) * f2m)

    def run(self, n):
        h = 0.5 * self.dt
        for _ in range(n):
            if self.obabo:
                self._bath(0)
                self._baro_kick(h)
                self._kick(h)
                q = None if self.cart else self._nm(self.x)
                q = self._drift(q)
            else:
                self._baro_kick(h)
                self._kick(h)
                q = None if self.cart else self._nm(self.x)
                q = self._drift(q)
                self._bath(0)
                q = self._drift(q)
            if not self.cart:
                self.x = torch.tensordot(self.M.t(), q, dims=([1], [0]))
            self.forces()
            self._baro_kick(h)
            self._kick(h)
            if self.obabo:
                self._bath(1)
            if self.case.get("fixcom"):
                rows = self.v if self.cart else self.v[:1]
                m = self.mm[None, :, None]
                rows -= (m * rows).sum(1, keepdim=True) / m.sum()
            self.step_no += 1

    def estimators(self):
        """The estimators of every system, as the library's dictionaries."""
        P, R = self.P, self.R

        def per(a):        # sum over atoms and components -> [P][R]
            return torch.zeros(P, R, **self.f8).index_add_(1, self.rep, a.sum(-1))

        m = self.mm[None, :, None]
        K = per(0.5 * m * self.mu[:, None, None] * self.v ** 2)
        wn2 = (self.wn[self.rep] ** 2)[None, :, None]
        dn = self.x - torch.roll(self.x, -1, 0)
        spring = per(m * wn2 * dn * dn).sum(0)
        if self.cart:
            dp = self.x - torch.roll(self.x, 1, 0)
            S = per(0.25 * m * wn2 * (dn * dn + dp * dp))
            v0 = self.v.sum(0) / math.sqrt(P)
        else:
            S = per(0.5 * m * wn2 * self.lam[:, None, None] * self._nm(self.x) ** 2)
            v0 = self.v[0]
        mv0 = torch.zeros(R, **self.f8).index_add_(0, self.rep, (self.mm[:, None] * v0 * v0).sum(-1))
        rF = per(self.x * self.F).sum(0)
        rcF = per((self.x - self.x.mean(0)) * self.F).sum(0)
        vir = self.vir.sum((0, 2))
        V = self.box.prod(1)
        kT = KB * self.T
        n = torch.tensor([float(s) for s in self.sizes], **self.f8)
        H = (K + S + self.U).sum(0)
        cols = dict(H=H, K_PR=1.5 * P * n * kT - 0.5 * spring / P, K_VR=-rF / (2.0 * P),
                    K_CV=1.5 * n * kT - rcF / (2.0 * P), T_ring=2.0 * K.sum(0) / (3.0 * n * P * KB))
        if self.water:
            cols.update(P_PR=(3.0 * P * n * kT - spring / P + vir / P) / (3.0 * V),
                        P_MD=(2.0 * K.sum(0) + vir) / (3.0 * V), P_CV=(mv0 - rcF + vir) / (3.0 * P * V))
        rows = []
        for r in range(R):
            e = {k: float(c[r]) for k, c in cols.items()}
            e.update(K_mode=K[:, r].cpu().numpy(), S_mode=S[:, r].cpu().numpy(), U_bead=self.U[:, r].cpu().numpy())
            if self.baro != "none":
                box = self.box[0].cpu().numpy()
                vw = self.vW.cpu().numpy()
                iso = self.baro == "iso"
                e["box"] = box
                e["vWa"] = np.zeros(3) if iso else vw
                e["vW"] = float(vw[0]) if iso else 0.0
                KW = 0.5 * self.Wb * (vw[0] ** 2 if iso else (vw ** 2).sum())
                e["enthalpy"] = (e["H"] + KW + P * PEXT * float(V[r]) - P * float(kT[r]) * np.log(box).sum())
            rows.append(e)
        return rows


def exact(case, seed):
    if case["engine"] == "handle":
        water = case["potential"] == "water"
        sim = _Exact([_handle_system(case, seed)], case, water, case["precision"] == "split")
        rows = []
        for _ in range(case["samples"]):
            sim.run(case["steps"])
            rows.append(sim.estimators()[0])
        out = _thermo(rows, np.float64, water)
        out["x"], out["v"] = sim.x.cpu(), sim.v.cpu()
        if case["barostat"] != "none":
            out["box"] = rows[-1]["box"]
            out["vW"] = np.append(rows[-1]["vWa"], rows[-1]["vW"])
            out["enthalpy"] = np.array([r["enthalpy"] for r in rows])
        out["step"] = None
        return out
    systems = _replica_systems(case, seed)
    rows = [None] * len(systems)
    xs, vs = [None] * len(systems), [None] * len(systems)
    for P in sorted({s["x0"].shape[0] for s in systems}):
        at = [r for r, s in enumerate(systems) if s["x0"].shape[0] == P]
        sim = _Exact([systems[r] for r in at], {}, True, True)
        sim.run(case["steps"])
        est = sim.estimators()
        x, v = torch.split(sim.x, sim.sizes, dim=1), torch.split(sim.v, sim.sizes, dim=1)
        for q, r in enumerate(at):
            rows[r] = est[q]
            if case["frames"]:
                xs[r], vs[r] = x[q].cpu().reshape(-1), v[q].cpu().reshape(-1)
    out = _thermo(rows, np.float64, True)
    if case["frames"]:
        out["x"], out["v"] = torch.cat(xs), torch.cat(vs)
    out["step"] = None
    return out

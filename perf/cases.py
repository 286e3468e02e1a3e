"""Performance cases of the quasi-static wake library: what its users have it do.

Kinds of case (every one through the public entry points of paper_1411_3246_gb300.wake):
  march    one xi-march of one or several simulations with the frozen driver of Eq. 12: a wake
           for given bunches, or a scan of the plasma temperature
  steps    a beam carried through the plasma: load the bunches, wake_step(steps), read the beam
  sweep    many simulations of uneven size, temperature and witness delay stepped by one handle
  push     test particles pushed through a frozen wake the caller holds, then deposited
  adjoint  the witness's observables and their gradient

The fields go to caller-owned grids in the form's own type (wake_bind_fields), one array of
psi, E_z, E_r and B_theta per simulation; the beam comes back as wake_get_beam gives it.  The
mixed forms' beam is handed on in single precision, the precision of their momenta and fields.
A nonlinear wake in single precision has nodes where one plasma electron that recrosses the
axis a slice earlier or later moves E_z, so two runs of the same code differ there; a program
that carries a beam through it reads the beam, and the marches that return fields are those of
weak drivers (every regime in FP64).
"""
import math
from types import SimpleNamespace

import numpy as np
import torch

from paper_1411_3246_gb300 import wake

PRECISION = {"fp64": wake.WAKE_FP64, "mixed": wake.WAKE_MIXED}

# Physics of the repository's workloads (lengths in 1/k_p, densities in n_p, momenta in m c).
PHYSICS = {
    # one weak bi-Gaussian driver in a cold plasma
    "linear": dict(rmax=6.0, ximax=10.0, n_d=0.1, sigma_r=0.5, sigma_zd=1.0, xi_d=4.0),
    # the same driver with a witness behind it (the sweep and the differentiation)
    "sweep": dict(rmax=6.0, ximax=10.0, n_d=0.1, sigma_r=0.5, sigma_zd=1.0, xi_d=4.0, eps_n=1e-2, q_ratio=0.3,
                  delay=4.5),
    # a stronger driver and witness, still short of blowout (designs and scans)
    "scan": dict(rmax=6.0, ximax=10.0, n_d=0.3, sigma_r=0.5, sigma_zd=1.0, xi_d=4.0, q_ratio=0.3, delay=4.5),
    # nonlinear blowout, two bunches
    "blowout": dict(rmax=8.0, ximax=12.0, n_d=8.0, sigma_r=0.2, sigma_zd=0.6, xi_d=2.4, eps_n=1e-2, q_ratio=0.3,
                    delay=4.5),
    # the large configuration's box with the blowout bunches
    "large": dict(rmax=10.0, ximax=16.0, n_d=8.0, sigma_r=0.2, sigma_zd=0.6, xi_d=2.4, eps_n=1e-2, q_ratio=0.3,
                  delay=4.5),
    # the two-bunch FACET parameters of Table I
    "table1": dict(rmax=6.0, ximax=16.0, n_d=3.56, n_w=2.85, sigma_r=0.42, sigma_zd=1.44, sigma_zw=0.81, xi_d=5.76,
                   xi_w=11.24, gamma_b=23.0e3 / 0.511, eps_n=0.0),
    # the single bunch of the OSIRIS comparison
    "osiris": dict(rmax=10.0, ximax=25.0, n_d=3.6, sigma_r=0.19, sigma_zd=1.72, xi_d=6.88, gamma_b=30.0e3 / 0.511,
                   eps_n=0.0),
}


def listed():
    return [
        # the check-grade run: plain FP64, linear regime, one march (the smallest configuration)
        dict(name="march_linear_fp64", kind="march", physics="linear", precision="fp64", nr=128, nxi=256, ppc=4,
             u_th=0.0, sims=1),
        # the same march in the mixed form: the shortest call a design loop makes
        dict(name="march_linear_mixed", kind="march", physics="linear", precision="mixed", nr=128, nxi=256, ppc=4,
             u_th=0.0, sims=1),
        # temperature scan (to 0.5 eV) behind two bunches with 32 rings per cell, every temperature
        # one simulation of a handle
        dict(name="march_scan_mixed", kind="march", physics="scan", precision="mixed", nr=96, nxi=1024, ppc=32,
             u_th=0.001, sims=8),
        # one wake with as many rings and slices as the blowout workload
        dict(name="march_full_mixed", kind="march", physics="linear", precision="mixed", nr=256, nxi=2048, ppc=16,
             u_th=0.0, sims=1),
        # the headline run: 200 beam steps of the blowout with 2^20 beam particles
        dict(name="steps_blowout_mixed", kind="steps", physics="blowout", precision="mixed", nr=512, nxi=2048, ppc=8,
             u_th=0.01, n_beam=1 << 20, steps=200, slab=False),
        # the OSIRIS comparison carried 1.4 m: a dense beam on a small cold grid, many steps
        dict(name="steps_osiris_mixed", kind="steps", physics="osiris", precision="mixed", nr=200, nxi=500, ppc=9,
             u_th=0.0, n_beam=2_500_000, steps=763, slab=False),
        # slab geometry on a ragged grid
        dict(name="steps_slab_mixed", kind="steps", physics="blowout", precision="mixed", nr=301, nxi=777, ppc=6,
             u_th=0.01, n_beam=200_001, steps=40, slab=True),
        # the FP64 form of the pipelined steps, as the mixed form is checked against
        dict(name="steps_blowout_fp64", kind="steps", physics="blowout", precision="fp64", nr=128, nxi=512, ppc=8,
             u_th=0.01, n_beam=1 << 17, steps=24, slab=False),
        # the large configuration's radial grid and plasma (rings in global memory), few slices
        dict(name="steps_large_mixed", kind="steps", physics="large", precision="mixed", nr=2048, nxi=96, ppc=32,
             u_th=0.02, n_beam=1 << 20, steps=8, slab=False),
        # a sweep of uneven simulations
        dict(name="sweep_mixed", kind="sweep", physics="sweep", precision="mixed", sims=32, nr_max=1024, nxi_max=2048,
             n_beam=1 << 16, steps=10),
        # test particles through a frozen wake (the beam kernels on their own)
        dict(name="push_frozen_mixed", kind="push", physics="osiris", precision="mixed", nr=200, nxi=500,
             n_beam=1 << 22, steps=8),
        # gradients of the witness's energy gain and spread
        dict(name="adjoint_fp64", kind="adjoint", physics="sweep", precision="fp64", nr=128, nxi=256, ppc=4,
             u_th=0.005, n_beam=1 << 16, steps=16, bins=64),
    ]


def draw(rng):
    def log(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(["march", "march", "steps", "steps", "steps", "sweep", "push", "adjoint"])
    fp64 = kind in ("march", "steps") and rng.random() < 0.3
    if kind == "march":
        physics = rng.choice(["linear", "scan", "blowout"] if fp64 else ["linear", "scan"])
        fine = physics == "scan" and not fp64  # single precision with many rings per cell
        return dict(kind=kind, physics=physics, precision="fp64" if fp64 else "mixed",
                    nr=log(48, 160) if fp64 else log(40, 100) if fine else log(64, 280), nxi=log(256, 400) if fp64 else log(256, 2000),
                    ppc=2 * rng.randint(8, 16) if fine else rng.randint(3, 6) if physics == "linear" else 2 * rng.randint(2, 4),
                    u_th=dict(linear=0.0, scan=rng.uniform(0.0002, 0.001), blowout=0.01)[physics],
                    sims=rng.choice([1, 1, 3, 7]))
    if kind == "steps":
        physics = rng.choice(["blowout", "blowout", "table1", "osiris", "large"])
        warm = physics != "osiris"
        return dict(kind=kind, physics=physics, precision="fp64" if fp64 else "mixed",
                    nr=log(48, 130) if fp64 else log(96, 420), nxi=log(300, 500) if fp64 else log(400, 1500),
                    ppc=2 * rng.randint(2, 4) if warm else rng.randint(5, 9),
                    u_th=rng.uniform(0.005, 0.02) if warm else 0.0,
                    n_beam=log(1 << 14, 1 << 17) if fp64 else log(1 << 15, 1 << 20),
                    steps=log(4, 24) if fp64 else log(4, 170), slab=physics == "blowout" and rng.random() < 0.3)
    if kind == "sweep":
        return dict(kind=kind, physics="sweep", precision="mixed", sims=log(4, 32), nr_max=rng.choice([256, 512, 1024]),
                    nxi_max=rng.choice([1024, 2048]), n_beam=log(1 << 14, 1 << 16), steps=rng.randint(2, 10))
    if kind == "push":
        return dict(kind=kind, physics=rng.choice(["osiris", "blowout"]),
                    precision=rng.choice(["mixed", "mixed", "fp64"]), nr=log(60, 500), nxi=log(200, 1000),
                    n_beam=log(1 << 12, 1 << 22), steps=rng.randint(1, 8))
    return dict(kind=kind, physics="sweep", precision="fp64", nr=log(40, 140), nxi=log(64, 280),
                ppc=rng.choice([2, 4, 6]), u_th=rng.uniform(0.002, 0.01), n_beam=log(1 << 12, 1 << 16),
                steps=rng.randint(2, 16), bins=rng.choice([0, 17, 64]))


# ---------------------------------------------------------------------------------------
# parameters and inputs
# ---------------------------------------------------------------------------------------

def _config(physics, **more):
    """Parameters of one simulation with the attribute names wake.params_of reads."""
    p = dict(u_th=0.0, n_w=0.0, sigma_zw=1.0, xi_w=0.0, gamma_b=4.0e4, eps_n=0.0, ds=5.0, n_beam=0, n_drive=0,
             geometry=0, ppc=4)
    p.update(PHYSICS[physics])
    p.update(more)
    q, delay = p.pop("q_ratio", None), p.pop("delay", None)
    if q is not None:  # Eq. 12's witness: sigma_zw and its charge from the drive's
        p["sigma_zw"] = 0.5625 * p["sigma_zd"]
        p["xi_w"] = p["xi_d"] + delay
        p["n_w"] = q * p["n_d"] * p["sigma_zd"] / p["sigma_zw"]
    c = SimpleNamespace(**p)
    if c.n_beam:  # macroparticles split between the bunches by charge
        qd, qw = c.n_d * c.sigma_zd, c.n_w * c.sigma_zw
        c.n_drive = c.n_beam - int(round(c.n_beam * qw / (qd + qw)))
    return c


def _sweep_sizes(case):
    """(nr, nxi, n_beam) of a sweep's simulations: powers of two log-uniform, the beams log-uniform
    from a quarter of the case's up to it."""
    rng = np.random.default_rng(case["sims"])
    return [(2 ** int(rng.integers(7, int(math.log2(case["nr_max"])) + 1)),
             2 ** int(rng.integers(9, int(math.log2(case["nxi_max"])) + 1)),
             int(case["n_beam"] * 4.0 ** rng.uniform(-1, 0))) for _ in range(case["sims"])]


def _configs(case, seed):
    """The case's simulations: the physics of its kind, the numbers a study varies from the seed."""
    kind, phys = case["kind"], case["physics"]
    rng = np.random.default_rng(seed)
    # no two designs use the same driver: its density within 2%, its place within 0.05
    vary = dict(n_d=PHYSICS[phys]["n_d"] * rng.uniform(0.98, 1.02), xi_d=PHYSICS[phys]["xi_d"] + rng.uniform(-0.05, 0.05))
    if kind == "sweep":  # sizes by the case, largest anywhere; temperature and delay by the seed
        return [_config(phys, nr=nr, nxi=nxi, n_beam=nb, u_th=float(rng.uniform(0.0005, 0.003)),
                        delay=float(rng.uniform(3.5, 5.5))) for nr, nxi, nb in _sweep_sizes(case)]
    size = dict(nr=case["nr"], nxi=case["nxi"], ppc=case.get("ppc", 4), geometry=1 if case.get("slab") else 0, **vary)
    if kind == "march":  # a scan takes its temperatures up to the case's, evenly
        n = case["sims"]
        return [_config(phys, u_th=case["u_th"] * (i + 1) / n, **size) for i in range(n)]
    return [_config(phys, u_th=case.get("u_th", 0.0), n_beam=case["n_beam"], **size)]


def _plasma_normals(c, gen):
    """(rings, 3) standard normals in mirrored pairs; None for a cold plasma."""
    if c.u_th == 0.0:
        return None
    half = torch.randn(c.nr * c.ppc // 2, 3, dtype=torch.float64, device="cuda", generator=gen)
    return torch.stack((half, -half), dim=1).reshape(-1, 3).contiguous()


def _inputs(case, seed):
    cfgs = _configs(case, seed)
    gen = torch.Generator(device="cuda").manual_seed(seed)
    plasma = [_plasma_normals(c, gen) for c in cfgs]
    beam = [torch.randn(5, c.n_beam, dtype=torch.float64, device="cuda", generator=gen) if c.n_beam else None
            for c in cfgs]
    return cfgs, plasma, beam


def _frozen_wake(c, dtype):
    """A smooth wake on the grid, as another program would hand it over: E_z a plasma
    oscillation behind the driver, E_r and B_theta focusing."""
    r = torch.linspace(0.0, c.rmax, c.nr + 1, dtype=torch.float64, device="cuda")[None, :]
    xi = torch.linspace(0.0, c.ximax, c.nxi + 1, dtype=torch.float64, device="cuda")[:, None]
    shape = torch.exp(-0.5 * (r / 1.5) ** 2)
    ez = 0.6 * torch.sin(xi) * shape
    bth = -0.05 * r * torch.cos(0.3 * xi) * shape
    er = bth + 0.25 * r * (1.0 + 0.3 * torch.cos(xi)) * shape
    return [t.to(dtype).contiguous() for t in (ez, er, bth)]


def _bunches(c, nm):
    """The 6 x n state of Eq. 12's bunches from standard normals, as a caller's own beam."""
    drive = torch.arange(c.n_beam, device="cuda") < c.n_drive
    xi = torch.where(drive, c.xi_d + c.sigma_zd * nm[4], c.xi_w + c.sigma_zw * nm[4])
    su = 1e-2 / c.sigma_r
    return torch.stack((c.sigma_r * nm[0], c.sigma_r * nm[1], xi, su * nm[2], su * nm[3],
                        torch.full_like(xi, c.gamma_b))).contiguous()


class _State:
    """A program's handle and the arrays it keeps with it; closed when dropped."""

    def __init__(self, case):
        self.case, self.handle = case, None

    def __del__(self):
        if self.handle is not None:
            self.handle.close()


def prepare(case, seed):
    s = _State(case)
    cfgs, s.plasma, s.normals = _inputs(case, seed)
    c = cfgs[0]
    if case["kind"] == "adjoint":
        s.theta = [c.n_w, c.xi_w - c.xi_d, c.sigma_zd, c.u_th]
        s.profile = [1.0] * case["bins"]
        s.handle = wake.Adjoint(c, case["steps"], case["bins"], s.plasma[0], s.normals[0])
        return s
    s.handle = sims = wake.Simulations(cfgs, PRECISION[case["precision"]], torch.cuda.Stream())
    dtype = torch.float64 if case["precision"] == "fp64" else torch.float32
    s.fields = []  # per simulation psi, E_z, E_r, B_theta
    torch.cuda.synchronize()
    for i, c in enumerate(cfgs):
        s.fields.append(torch.empty(4, c.nxi + 1, c.nr + 1, dtype=dtype, device="cuda"))
        wake.wake_bind_fields(sims.h, i, *s.fields[i])
        wake.wake_load_plasma(sims.h, i, s.plasma[i])
    if case["kind"] == "push":
        s.bunches = _bunches(c, s.normals[0])
        torch.cuda.synchronize()
        wake.wake_set_beam(sims.h, 0, s.bunches)
        wake.wake_beam_deposit(sims.h)
        wake.wake_plasma_march(sims.h)
        torch.cuda.synchronize()
        for k, v in zip((1, 2, 3), _frozen_wake(c, dtype)):
            s.fields[0][k].copy_(v)
    return s


def run(s):
    case, sims = s.case, s.handle
    if case["kind"] == "adjoint":
        obs = sims.forward(s.theta, s.profile)
        grad = sims.backward([1.0, 1.0])
        return {"obs": np.array(obs), "grad": np.array(grad)}
    if case["kind"] == "march":
        wake.wake_plasma_march(sims.h)
        sims._order()
        return {"fields": s.fields}
    if case["kind"] == "push":
        wake.wake_set_beam(sims.h, 0, s.bunches)
        wake.wake_beam_push_steps(sims.h, case["steps"])
        wake.wake_beam_deposit(sims.h)
        xyz, lost = sims.beam(0)
        return {"beam": _handed_on(case, xyz), "lost": lost, "nb": _handed_on(case, sims.nb(0))}
    for i in range(len(sims.cfgs)):
        wake.wake_load_beam(sims.h, i, s.normals[i])
    wake.wake_step(sims.h, case["steps"])
    if case["kind"] == "sweep":
        return {"beam": [_handed_on(case, sims.beam(i)[0]) for i in range(len(sims.cfgs))]}
    xyz, lost = sims.beam(0)
    out = {"beam": _handed_on(case, xyz), "lost": lost}
    if case["precision"] == "fp64":
        out["fields"] = s.fields
    return out


def _handed_on(case, t):
    return t if case["precision"] == "fp64" else t.to(torch.float32)


# ---------------------------------------------------------------------------------------
# the work that cannot be left out
# ---------------------------------------------------------------------------------------

# Operations of one plasma push (both RK2 stages), of one node and field stage, and of one beam push
PUSH_FLOP, NODE_FLOP, BEAM_FLOP = 250.0, 62.0, 140.0


def work(case):
    kind, word = case["kind"], 8 if case["precision"] == "fp64" else 4
    particle = 4 * word + 16 + word + 1  # x, y, u_x, u_y; xi and u_z; weight; flag
    if kind == "push":
        grid, beam, steps = (case["nr"] + 1) * (case["nxi"] + 1), case["n_beam"], case["steps"]
        return {"bytes": beam * (48 + steps * 2 * particle + 49) + grid * (3 * word * steps + 2 * word),
                "flops": steps * beam * BEAM_FLOP}
    ppc, steps, total = case.get("ppc", 4), case.get("steps", 1), {"bytes": 0.0, "flops": 0.0}
    sizes = _sweep_sizes(case) if kind == "sweep" else [(case["nr"], case["nxi"], case.get("n_beam", 0))] * case.get("sims", 1)
    for nr, nxi, beam in sizes:
        grid = (nr + 1) * (nxi + 1)
        march = (nxi + 1) * (nr * ppc * PUSH_FLOP + 2 * (nr + 1) * NODE_FLOP)
        total["bytes"] += grid * word * 4 + nr * ppc * 40
        if kind == "march":
            total["bytes"] += grid * word
            total["flops"] += march
        else:
            total["bytes"] += beam * (40 + 49) + steps * beam * 2 * particle
            total["flops"] += steps * (march + beam * BEAM_FLOP)
    if kind == "adjoint":  # forward, and a reverse of at least twice its operations
        total = {k: 3 * v for k, v in total.items()}
    return total


# ---------------------------------------------------------------------------------------
# the same in 64 bits, plainly (numpy): the readings of the library's header, nothing of its code
# ---------------------------------------------------------------------------------------

def _cell(s, n):
    c = np.clip(np.floor(s).astype(np.int64), 0, n - 1)
    return c, s - c


class _Plain:
    """The quasi-static march, the beam deposit and the Boris push of one simulation."""

    def __init__(self, c):
        self.c, self.slab = c, c.geometry == 1
        self.dr, self.dxi, n = c.rmax / c.nr, c.ximax / c.nxi, c.nr
        m = np.arange(n + 1)
        r = m * self.dr
        with np.errstate(divide="ignore"):
            if self.slab:
                self.V = np.full(n + 1, self.dr)
                self.V[[0, n]] *= 0.5
                self.alpha, self.metric, self.curv = np.full(n + 1, 0.5), np.ones(n + 1), np.zeros(n + 1)
            else:
                self.V = r * self.dr
                self.V[0], self.V[n] = self.dr ** 2 / 6, self.dr * (r[n] / 2 - self.dr / 6)
                self.alpha = 0.5 - 1 / (6.0 * np.maximum(m, 1))
                self.metric = np.where(m > 0, 1 / np.maximum(r, 1e-300), 0.0)
                self.curv = self.metric
        self.alpha[n] = 1.0
        self.metric = np.where(m > 0, self.metric, 0.0)
        i, d2 = m[1:], 1 / self.dr ** 2  # rows of the B system: nodes 1 .. nr
        if self.slab:
            self.a, self.cc, self.b = np.full(n, d2), np.full(n, d2), np.full(n, -2 * d2)
            self.a[-1] = 2 * d2
        else:
            self.a, self.cc = (i - 1) / (i - 0.5) * d2, (i + 1) / (i + 0.5) * d2
            self.b = -i * (1 / (i + 0.5) + 1 / (i - 0.5)) * d2
            self.a[-1], self.b[-1] = 2 * (n - 1) / (n - 0.5) * d2, -2 * n / (n - 0.5) * d2
        self.a[0], self.cc[-1] = 0.0, 0.0

    def rings(self, nm):
        c = self.c
        k, m = np.divmod(np.arange(c.nr * c.ppc), c.ppc)
        u = np.zeros((3, k.size)) if nm is None else c.u_th * nm.T
        where = (m + 0.5) / c.ppc if nm is None else (m // 2 + 0.5) / (c.ppc // 2)
        r, g = (k + where) * self.dr, np.sqrt(1 + (u ** 2).sum(0))
        self.l, self.G0 = (u[1] if self.slab else r * u[1]), g - u[2]
        self.w = (1.0 if self.slab else r) * self.dr / c.ppc * self.G0 / g
        self.r0, self.ur0 = r, u[0]

    def hats(self, cell, f, v):
        n1 = self.c.nr + 1
        return np.bincount(cell, v * (1 - f), n1) + np.bincount(cell + 1, v * f, n1)

    def inward(self, d):
        out = np.zeros_like(d)
        out[:-1] = -np.cumsum((0.5 * self.dr * (d[:-1] + d[1:]))[::-1])[::-1]
        return out

    def solve_b(self, chi, d):
        a, b, c = self.a, self.b - chi, self.cc  # cyclic reduction of every row at once
        k, n = 1, a.size
        while k < n:
            pad = np.zeros(k)
            up = lambda v, fill=pad: np.concatenate((fill, v[:-k]))  # noqa: E731
            down = lambda v, fill=pad: np.concatenate((v[k:], fill))  # noqa: E731
            k1, k2 = a / up(b, pad + 1), c / down(b, pad + 1)
            a, b, c, d = (-up(a) * k1, b - k1 * up(c) - k2 * down(a), -down(c) * k2, d - k1 * up(d) - k2 * down(d))
            k *= 2
        return np.concatenate(([0.0], d / b))

    def stage(self, r, ur, ut, nb):
        cell, f = _cell(r / self.dr, self.c.nr)
        at = lambda v: (1 - f) * v[cell] + f * v[cell + 1]  # noqa: E731
        delta = self.hats(cell, f, self.w) - self.rho0
        below = np.concatenate(([0.0], np.cumsum(delta)[:-1]))
        dpsi = (below + self.alpha * delta) * self.metric
        psi = self.inward(dpsi)
        G, dp, w, n = self.G0 + at(psi), at(dpsi), self.w, self.c.nr
        up2 = ur ** 2 + ut ** 2
        gam = (1 + up2 + G ** 2) / (2 * G)
        a, F = ur / G, gam / G * dp
        cent = 0.0 if self.slab else np.where(r > 0, ut ** 2 / (G * np.maximum(r, 1e-300)), 0.0)
        jz = self.hats(cell, f, -w * (gam - G) / G) / self.V - nb
        chi, T = self.hats(cell, f, w / G) / self.V, self.hats(cell, f, w * a ** 2) / self.V
        P, U = self.hats(cell, f, w * (a ** 2 * dp - F - cent) / G) / self.V, self.hats(cell, f, w * a / G) / self.V
        K = np.bincount(cell, w * a, n + 1)
        dez = np.zeros(n + 1)
        dez[1:] = -((1 - self.alpha[1:]) * K[:-1] + self.alpha[1:] * K[1:]) / self.dr * self.metric[1:]
        ez = self.inward(dez)
        Q, d = P + ez * U, np.empty(n)
        d[:-1] = ((jz[2:] - jz[:-2]) + (T[2:] - T[:-2])) / (2 * self.dr) + Q[1:-1] + T[1:-1] * self.curv[1:-1]
        d[-1] = Q[n] + (T[n] - T[n - 1]) / self.dr + T[n] * self.curv[n] - (jz[n - 1] + jz[n]) / self.dr
        bth = self.solve_b(chi[1:], d)
        return psi, dpsi, ez, bth, G, F - at(bth)

    def march(self, nb):
        c, h = self.c, self.dxi
        r, ur = self.r0.copy(), self.ur0.copy()
        cell, f = _cell(r / self.dr, c.nr)
        self.rho0 = self.hats(cell, f, self.w)
        out = {k: np.zeros((c.nxi + 1, c.nr + 1)) for k in ("psi", "ez", "er", "bth")}

        def move(x, y, ux, uy):  # back to (r, u_r, u_theta), specular at the wall
            rr = np.hypot(x, y)
            safe = np.where(rr > 0, rr, 1.0)
            un = np.where(rr > 0, (x * ux + y * uy) / safe, np.hypot(ux, uy))
            ut = np.where(rr > 0, (x * uy - y * ux) / safe, 0.0)
            return np.where(rr > c.rmax, 2 * c.rmax - rr, rr), np.where(rr > c.rmax, -un, un), ut

        for k in range(c.nxi + 1):
            ut = self.l if self.slab else np.where(r > 0, self.l / np.where(r > 0, r, 1.0), 0.0)
            psi, dpsi, ez, bth, G1, F1 = self.stage(r, ur, ut, nb[k])
            out["psi"][k], out["ez"][k], out["bth"][k] = psi, ez, bth
            out["er"][k, 1:] = (bth - dpsi)[1:]
            if k == c.nxi:
                return out
            uy = np.zeros_like(r) if self.slab else ut
            xh, yh, uxh = r + 0.5 * h * ur / G1, 0.5 * h * uy / G1, ur + 0.5 * h * F1
            rm, urm, utm = move(xh, yh, uxh, uy)
            G2, F2 = self.stage(rm, urm, self.l if self.slab else utm, 0.5 * (nb[k] + nb[k + 1]))[4:]
            rh = np.hypot(xh, yh)
            ex, ey = np.where(rh > 0, xh / np.where(rh > 0, rh, 1), 1.0), np.where(rh > 0, yh / np.where(rh > 0, rh, 1), 0.0)
            r, ur, _ = move(r + h * uxh / G2, h * uy / G2, ur + h * F2 * ex, uy + h * F2 * ey)

    def driver(self):
        c = self.c
        r, xi = np.arange(c.nr + 1) * self.dr, np.arange(c.nxi + 1) * self.dxi
        lon = c.n_d * np.exp(-0.5 * ((xi - c.xi_d) / c.sigma_zd) ** 2)
        if c.n_w:
            lon = lon + c.n_w * np.exp(-0.5 * ((xi - c.xi_w) / c.sigma_zw) ** 2)
        return lon[:, None] * np.exp(-0.5 * (r / c.sigma_r) ** 2)[None, :]

    def load(self, state):
        """A beam of 6 x n with the bunches' macroparticle weights."""
        c, s2pi = self.c, math.sqrt(2 * math.pi)
        self.beam = state.copy()
        if self.slab:
            self.beam[[1, 4]] = 0.0
        tr = 0.5 * s2pi * c.sigma_r if self.slab else c.sigma_r ** 2
        drive = np.arange(c.n_beam) < c.n_drive
        self.wb = np.where(drive, c.n_d * s2pi * tr * c.sigma_zd / max(1, c.n_drive),
                           c.n_w * s2pi * tr * c.sigma_zw / max(1, c.n_beam - c.n_drive))
        self.lost = np.zeros(c.n_beam, dtype=bool)
        self.lost |= ~self.inside()

    def inside(self):
        x, y, xi = self.beam[:3]
        return (xi >= 0) & (xi < self.c.ximax) & (np.hypot(x, y) < self.c.rmax)

    def corners(self, live):
        c, n1 = self.c, self.c.nr + 1
        x, y, xi = self.beam[:3, live]
        cr, f = _cell(np.hypot(x, y) / self.dr, c.nr)
        k, g = _cell(xi / self.dxi, c.nxi)
        i = k * n1 + cr
        return ((i, (1 - f) * (1 - g)), (i + 1, f * (1 - g)), (i + n1, (1 - f) * g), (i + n1 + 1, f * g))

    def deposit(self):
        c, live = self.c, ~self.lost
        shape, nb = (c.nxi + 1, c.nr + 1), 0.0
        for i, v in self.corners(live):
            nb = nb + np.bincount(i, self.wb[live] * v, shape[0] * shape[1])
        vx = np.full(c.nxi + 1, self.dxi)
        vx[[0, -1]] *= 0.5
        return nb.reshape(shape) / (vx[:, None] * self.V[None, :])

    def push(self, ez, er, bth):
        live, h = ~self.lost, -0.5 * self.c.ds
        x, y, xi, ux, uy, uz = self.beam[:, live]
        at = [sum(v * g.reshape(-1)[i] for i, v in self.corners(live)) for g in (ez, er, bth)]
        r = np.hypot(x, y)
        cs, sn = np.where(r > 0, x / np.where(r > 0, r, 1), 0.0), np.where(r > 0, y / np.where(r > 0, r, 1), 0.0)
        Ex, Ey, Bx, By = at[1] * cs, at[1] * sn, -at[2] * sn, at[2] * cs
        mx, my, mz = ux + h * Ex, uy + h * Ey, uz + h * at[0]
        gm = np.sqrt(1 + mx ** 2 + my ** 2 + mz ** 2)
        tx, ty = h * Bx / gm, h * By / gm
        px, py, pz = mx - mz * ty, my + mz * tx, mz + (mx * ty - my * tx)
        s = 2 / (1 + tx ** 2 + ty ** 2)
        ux, uy = mx - pz * s * ty + h * Ex, my + pz * s * tx + h * Ey
        uz = uz + (2 * h * at[0] + (px * s * ty - py * s * tx))
        up2 = ux ** 2 + uy ** 2
        gam = np.sqrt(1 + up2 + uz ** 2)
        dt = self.c.ds
        self.beam[:, live] = (x + dt * ux / gam, y + dt * uy / gam, xi + dt * (1 + up2) / (gam * (gam + uz)), ux, uy, uz)
        self.lost |= ~self.inside()


def _eq12(c, nm):
    """The 6 x n state of the bunches of Eq. 12 from their standard normals."""
    drive, su = np.arange(c.n_beam) < c.n_drive, c.eps_n / c.sigma_r
    xi = np.where(drive, c.xi_d + c.sigma_zd * nm[4], c.xi_w + c.sigma_zw * nm[4])
    return np.stack((c.sigma_r * nm[0], c.sigma_r * nm[1], xi, su * nm[2], su * nm[3], np.full(c.n_beam, c.gamma_b)))


def _stack(f):
    return np.stack([f[k] for k in ("psi", "ez", "er", "bth")])


def _seconds(case):
    """A guess at what _Plain takes on one core."""
    if case["kind"] == "sweep":
        return math.inf
    rings = case["nr"] * case.get("ppc", 4)
    march = (case["nxi"] + 1) * (1.2e-3 + 4e-7 * rings)
    push = 1.5e-6 * case.get("n_beam", 0)
    if case["kind"] == "march":
        return march * case["sims"]
    return case["steps"] * (push + (0.0 if case["kind"] == "push" else march))


def exact(case, seed):
    if _seconds(case) > 20:
        return None
    cfgs, plasma, normals = _inputs(case, seed)
    host = [None if t is None else t.cpu().numpy() for t in plasma]
    if case["kind"] == "march":
        out = []
        for c, nm in zip(cfgs, host):
            p = _Plain(c)
            p.rings(nm)
            out.append(p.march(p.driver()))
        return {"fields": [_stack(f) for f in out]}
    c, p = cfgs[0], _Plain(cfgs[0])
    if case["kind"] == "push":
        p.load(_bunches(c, normals[0]).cpu().numpy())
        dtype = torch.float64 if case["precision"] == "fp64" else torch.float32
        f = [t.double().cpu().numpy() for t in _frozen_wake(c, dtype)]
        for _ in range(case["steps"]):
            p.push(*f)
        return {"beam": p.beam, "lost": p.lost.astype(np.uint8), "nb": p.deposit()}
    p.load(_eq12(c, normals[0].cpu().numpy()))
    p.rings(host[0])
    fields = None
    for _ in range(case["steps"]):
        fields = p.march(p.deposit())
        p.push(fields["ez"], fields["er"], fields["bth"])
    if case["kind"] == "adjoint":  # the observables; their gradient has no plain counterpart
        live = ~p.lost & (np.arange(c.n_beam) >= c.n_drive)
        gain = np.sqrt(1 + (p.beam[3:, live] ** 2).sum(0)) - c.gamma_b
        return {"obs": np.array([gain.mean(), gain.std()]), "grad": None}
    out = {"beam": p.beam, "lost": p.lost.astype(np.uint8)}
    if case["precision"] == "fp64":
        out["fields"] = [_stack(fields)]
    return out

"""The work a user has this library do, as measurable cases: whole sweeps of single simulations
and batches, and plane-wave moves alone, each through the public Python entry points.

A case is a dict of plain values:
  kind       "sim" (one Simulation), "batch" (one Batch) or "planewave" (moves alone on a Simulation)
  system     "chain", "chains", "suspension", "paper_chains" or "ensemble"
  precision  "fp64" or "mixed"
  sweeps     sweeps (or plane-wave moves) per pass
and the sizes and options of the system. One pass advances the simulation(s) and reads the
unwrapped positions into a device buffer, as a sampling program does; the simulation goes on from
where the last pass left it.
"""
import functools
import math

import numpy as np
import torch

from paper_1611_09160_gb300 import inputs, validate, wmcd

SPHERES, CHAINS, CHAIN_LEN = 4_000_000, 1000, 1024       # the large suspension at scale 1


def listed():
    return [
        # the smallest call: one short chain, every move in the serial phase, plain binary64
        dict(name="chain32_fp64", kind="sim", system="chain", n=32, box=64.0, precision="fp64", sweeps=10),
        # a lone chain of odd length with the default schedule; the infinite system's plane waves
        dict(name="chain1001_infinite", kind="sim", system="chain", n=1001, phi=1e-3, precision="mixed", sweeps=2,
             planewaves="infinite"),
        # many short FENE chains in the paper's reduced units (relaxation and diffusivity runs)
        dict(name="fene_chains_20k", kind="sim", system="paper_chains", chains=2000, chain_len=10, gap=25.0,
             precision="mixed", sweeps=2),
        # dilute polymer solution, in both precisions
        dict(name="dilute16k_mixed", kind="sim", system="chains", chains=256, chain_len=64, phi=1e-3,
             precision="mixed", sweeps=1),
        dict(name="dilute16k_fp64", kind="sim", system="chains", chains=256, chain_len=64, phi=1e-3,
             precision="fp64", sweeps=1),
        # semi-dilute solutions: the acceptance-spectrum run with the full periodic mode set, and
        # the million-bead one
        dict(name="semidilute65k_full", kind="sim", system="chains", chains=1024, chain_len=64, phi=0.05,
             precision="mixed", sweeps=1, planewaves="full"),
        dict(name="semidilute1M", kind="sim", system="chains", chains=4096, chain_len=256, phi=0.05,
             precision="mixed", sweeps=1, colour_K=3),
        # the large dilute suspension of spheres and chains, and its 1/64 subsample
        dict(name="suspension5M", kind="sim", system="suspension", spheres=SPHERES, chains=CHAINS,
             chain_len=CHAIN_LEN, phi=1e-3, precision="mixed", sweeps=1, max_fine=768, n_cap=128, level2=1),
        dict(name="suspension79k", kind="sim", system="suspension", spheres=62_500, chains=16, chain_len=CHAIN_LEN,
             phi=1e-3, precision="mixed", sweeps=1),
        # an ensemble of uneven single chains advanced as one batch, a serving step at a time; the
        # few short requests left at the end of a stream
        dict(name="ensemble1024", kind="batch", system="ensemble", sims=1024, hi=2048,
             precision="mixed", sweeps=16),
        dict(name="ensemble_tail24", kind="batch", system="ensemble", sims=24, hi=256,
             precision="mixed", sweeps=8),
        # plane-wave moves alone: every bead moves, the streaming part of a sweep
        dict(name="planewave628k", kind="planewave", system="suspension", spheres=SPHERES // 8, chains=CHAINS // 8,
             chain_len=CHAIN_LEN, phi=1e-3, precision="mixed", sweeps=2),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case of the same ranges: sizes over their logarithm, odd ones among them."""
    what = rng.choice(["chain", "chains", "semi", "paper_chains", "suspension", "batch", "planewave"])
    precision = rng.choice(["mixed", "mixed", "fp64"])
    if what == "chain":
        return dict(kind="sim", system="chain", n=_log(rng, 16, 2048), phi=1e-3, precision=precision,
                    sweeps=rng.randint(1, 10), planewaves=rng.choice(["sphere", "full", "infinite"]))
    if what == "chains":
        return dict(kind="sim", system="chains", chains=_log(rng, 16, 1024), chain_len=_log(rng, 8, 128),
                    phi=round(math.exp(rng.uniform(math.log(1e-3), math.log(1e-2))), 5), precision=precision, sweeps=1)
    if what == "semi":
        return dict(kind="sim", system="chains", chains=_log(rng, 256, 2048), chain_len=_log(rng, 32, 128),
                    phi=round(rng.uniform(0.02, 0.05), 4), precision="mixed", sweeps=1,
                    planewaves=rng.choice(["sphere", "full"]), colour_K=rng.choice([2, 3]))
    if what == "paper_chains":
        return dict(kind="sim", system="paper_chains", chains=_log(rng, 200, 4000), chain_len=_log(rng, 4, 32),
                    gap=25.0, precision=precision, sweeps=rng.randint(1, 2))
    if what == "suspension":
        s = math.exp(rng.uniform(math.log(1 / 256), math.log(1 / 4)))
        return dict(kind="sim", system="suspension", spheres=int(SPHERES * s), chains=max(1, int(CHAINS * s)),
                    chain_len=CHAIN_LEN, phi=1e-3, precision="mixed", sweeps=1, max_fine=768, n_cap=128,
                    level2=rng.choice([0, 1]))
    if what == "batch":
        return dict(kind="batch", system="ensemble", sims=_log(rng, 4, 512), hi=_log(rng, 64, 2048),
                    precision=precision, sweeps=rng.randint(1, 16))
    s = math.exp(rng.uniform(math.log(1 / 256), math.log(1 / 8)))
    return dict(kind="planewave", system="suspension", spheres=int(SPHERES * s), chains=max(1, int(CHAINS * s)),
                chain_len=CHAIN_LEN, phi=1e-3, precision=precision, sweeps=rng.randint(1, 8))


# ---- inputs ---------------------------------------------------------------------------

def _generate(case, seed):
    if case["system"] == "chain":
        box = case.get("box") or inputs.box_for_volume_fraction(case["n"], case["phi"])
        return inputs.single_chain(case["n"], box, seed=seed)
    if case["system"] == "chains":
        return inputs.dilute_chains(case["chains"], case["chain_len"], case["phi"], seed=seed)
    if case["system"] == "paper_chains":
        box = case["gap"] * case["chains"] ** (1.0 / 3.0)
        bond = validate.BOND_START_BAR
        return inputs.make_system([case["chain_len"]] * case["chains"], 0, box, seed, bond=bond,
                                  min_dist=0.999 * min(validate.SIGMA_BAR, bond))
    return inputs.suspension(case["spheres"], case["chains"], case["chain_len"], case["phi"], seed=seed)


@functools.lru_cache(maxsize=2)
def _base(items):
    return _generate(dict(items), 1)


@functools.lru_cache(maxsize=1)
def _pool():
    """Single chains at volume fraction 1e-3, lengths log-uniform in [16, 2048]."""
    return inputs.ensemble(1024, 16, 2048, 1e-3, seed=1)


def _seen_anew(base, rng):
    """A configuration from another origin and with other axes: as new an input, at no cost."""
    L = base.box_L
    pos = np.mod(base.pos[:, rng.permutation(3)] + rng.uniform(0.0, L, 3), L)
    return inputs.System(np.minimum(pos, np.nextafter(L, 0.0)), base.chain_len, L)


def _system(case, seed):
    """The case's starting configuration; a large one is generated once and seen anew for each seed."""
    beads = case.get("spheres", 0) + case.get("chains", 0) * case.get("chain_len", 0)
    if beads < 200_000:
        return _generate(case, seed)
    keys = ("system", "spheres", "chains", "chain_len", "phi", "gap")
    return _seen_anew(_base(tuple((k, case[k]) for k in keys if k in case)), np.random.default_rng(seed))


def _systems(case, seed):
    """The batch's members: chains of the pool with at most `hi` beads, the same ones for a case, each
    seen anew for each seed."""
    fit = [s for s in _pool() if s.n_beads <= case["hi"]]
    some = np.random.default_rng(case["sims"]).permutation(max(len(fit), case["sims"]))[:case["sims"]] % len(fit)
    rng = np.random.default_rng(seed)
    return [_seen_anew(fit[k], rng) for k in some]


def _params(case, system, seed, **extra):
    modes = {"sphere": (wmcd.PLANEWAVE_PERIODIC, 8), "full": (wmcd.PLANEWAVE_PERIODIC_FULL, 15),
             "infinite": (wmcd.PLANEWAVE_INFINITE, 8)}
    mode, lcut = modes[case.get("planewaves", "sphere")]
    for k in ("colour_K", "max_fine", "n_cap", "level2"):
        if k in case:
            extra[k] = case[k]
    if case["system"] == "paper_chains":
        extra.update(validate.paper_unit_params("good"))
    precision = wmcd.MIXED if case["precision"] == "mixed" else wmcd.FP64
    return wmcd.default_params(system.n_beads, system.box_L, seed=seed, precision=precision, planewave_mode=mode,
                               lcut=lcut, **extra)


def prepare(case, seed):
    if case["kind"] == "batch":
        systems = _systems(case, seed)
        # chains short enough for the shared-memory serial phase run all their moves there
        params = [_params(case, s, seed, sim_id=k, serial_only=True) for k, s in enumerate(systems)]
        batch = wmcd.Batch(len(systems), sum(wmcd.batch_need(p) for p in params) + (1 << 20))
        slots = [batch.admit(p, s.pos, s.chain_len) for p, s in zip(params, systems)]
        ends = np.cumsum([0] + [s.n_beads for s in systems])
        out = torch.empty((int(ends[-1]), 3), dtype=torch.float64, device="cuda")
        parts = [out[a:b] for a, b in zip(ends[:-1], ends[1:])]
        return dict(batch=batch, sims=[batch.sim(k) for k in slots], parts=parts, out=out, sweeps=case["sweeps"])
    system = _system(case, seed)
    sim = wmcd.Simulation(_params(case, system, seed), system.pos, system.chain_len)
    out = torch.empty((system.n_beads, 3), dtype=torch.float64, device="cuda")
    return dict(sim=sim, out=out, sweeps=case["sweeps"], planewave=case["kind"] == "planewave")


def run(state):
    if "batch" in state:
        state["batch"].step(state["sweeps"])
        for sim, part in zip(state["sims"], state["parts"]):
            sim.positions(unwrapped=True, out=part)
        return state["out"]
    if state["planewave"]:
        state["sim"].planewave(state["sweeps"])
    else:
        state["sim"].sweep(state["sweeps"])
    state["sim"].positions(unwrapped=True, out=state["out"])
    return state["out"]


# ---- what a pass cannot do without ------------------------------------------------------

def _lengths(case):
    if case["kind"] == "batch":
        return case["sims"] * (case["hi"] - 16) / math.log(case["hi"] / 16)       # expected beads of the members
    if case["system"] == "chain":
        return case["n"]
    return case.get("spheres", 0) + case["chains"] * case["chain_len"]


def work(case):
    """Positions read and written once, and read out once. Operations: about 60 per bead of a
    move's support (offset, displacement, new position) and about 40 per bead for the energies of
    its bonds and nearest partners; a sweep attempts about one wavelet move per bead with a
    support of a bead or more, and a plane wave moves every bead."""
    n = _lengths(case)
    return {"bytes": n * 24.0 * 3.0, "flops": 100.0 * n * case["sweeps"]}


# ---- the same results in plain numpy, 64 bits --------------------------------------------
#
# The method itself (Dyer & Ball, arXiv:1611.09160) one move after another: scales from
# P_lambda (Eq. 32), centres and polarisations by rejection, displacements (Eqs. 21, 23, 29),
# energies (Eqs. 1, 2), the Metropolis test (Eq. 20), plane waves (Sec. VI), on the counter-based
# Philox stream a simulation's seed names. Only for systems whose moves all run in sequence and
# for plane waves alone: the sequential sweep of a larger, coloured system takes minutes here.

COUNT, SLOT, VB, VP, ACC, PWCOUNT, PWMODE, PWDIR, PWACC, DPWMODE, DPWDIR, DPWACC = range(1, 13)
U32 = np.uint64(0xFFFFFFFF)


def _draw(seed, sim_id, kind, layer, sweep, index, attempt=0):
    """Philox4x32-10 words for arrays of indices: counter (index, sweep, kind | layer | attempt, 0)."""
    index = np.atleast_1d(np.asarray(index, dtype=np.uint64))
    c = [index, np.full_like(index, sweep), np.full_like(index, (kind << 24) | (layer << 16) | attempt),
         np.zeros_like(index)]
    k0, k1 = seed & 0xFFFFFFFF, ((seed >> 32) ^ sim_id) & 0xFFFFFFFF
    for _ in range(10):
        a, b = c[0] * np.uint64(0xD2511F53), c[2] * np.uint64(0xCD9E8D57)
        c = [(b >> np.uint64(32)) ^ c[1] ^ np.uint64(k0), b & U32, (a >> np.uint64(32)) ^ c[3] ^ np.uint64(k1), a & U32]
        k0, k1 = (k0 + 0x9E3779B9) & 0xFFFFFFFF, (k1 + 0xBB67AE85) & 0xFFFFFFFF
    return c


def _u53(hi, lo):
    return (((hi >> np.uint64(5)) << np.uint64(26)) | (lo >> np.uint64(6))).astype(np.float64) * 2.0 ** -53


def _ball(seed, sim_id, kind, layer, sweep, count, nonzero):
    """A point of the unit ball per index: the first of up to 64 attempts that lies in it."""
    out = np.zeros((count, 3))
    if nonzero:
        out[:, 2] = 1.0
    left = np.arange(count)
    for a in range(64):
        if left.size == 0:
            break
        w = _draw(seed, sim_id, kind, layer, sweep, left, a)
        p = np.stack([x.astype(np.float64) * 2.0 ** -31 - 1.0 for x in w[:3]], axis=1)
        q = (p * p).sum(axis=1)
        ok = (q <= 1.0) & ((q > 0.0) | (not nonzero))
        out[left[ok]] = p[ok]
        left = left[~ok]
    return out


def _phi(k):
    """Transform of the tapered wavelet (Eq. 25), by its power series near k = 0."""
    small = k < 1.5
    s, f = np.zeros_like(k), 24.0
    ks = np.where(small, k, 0.0)
    for p in range(3, 24):
        f1, f2 = f * (2 * p - 1), f * (2 * p - 1) * (2 * p)
        s += (-1.0) ** (p - 1) * (5.0 / f1 - 1.0 / f - 8.0 / f2) * ks ** (2 * p - 6)
        f = f2
    kl = np.where(small, 2.0, k)
    big = (5.0 * kl * np.sin(kl) - (kl * kl - 8.0) * np.cos(kl) - 8.0) / kl ** 6
    return 4.0 * math.pi * np.where(small, s, big)


def _panel(a, b):
    x, w = np.polynomial.legendre.leggauss(10)
    q = 0.5 * (a + b)[:, None] + 0.5 * (b - a)[:, None] * x
    return (w * q ** 3 * _phi(q) ** 2).sum(axis=1) * 0.5 * (b - a)


@functools.lru_cache(maxsize=1)
def _weights():
    """G(Q) = Int_Q^inf q^3 phi^2 (Eqs. 49, 51) on a grid, the smooth tail beyond it exactly."""
    h, n = math.pi / 20.0, 40_000
    edge = np.arange(n + 1) * h
    K = edge[-1]
    tail = 16.0 * math.pi ** 2 * (0.125 * K ** -4 + 0.75 * K ** -6 + 12.0 * K ** -8)
    return edge, tail + np.concatenate([np.cumsum(_panel(edge[:-1], edge[1:])[::-1])[::-1], [0.0]])


def _modes(L, lmax, lcut=8):
    """Modes |l| <= lcut, their cumulative probabilities and the sum of their weights."""
    r = np.arange(-lcut, lcut + 1)
    m = np.stack(np.meshgrid(r, r, r, indexing="ij"), axis=-1).reshape(-1, 3)
    m = m[(m * m).sum(axis=1) <= lcut * lcut]
    Q = 2.0 * math.pi * np.sqrt((m * m).sum(axis=1)) / L * lmax
    edge, acc = _weights()
    top = np.minimum((Q / edge[1]).astype(int) + 1, len(edge) - 1)
    g = acc[top] + _panel(Q, edge[top])
    return m, np.cumsum(g) / g.sum(), g.sum()


class _Exact:
    """One simulation in plain numpy: harmonic bonds, WCA, periodic plane waves."""

    def __init__(self, p, pos, chain_len):
        self.p, self.L, self.seed, self.sid = p, p["box_L"], int(p["seed"]), int(p["sim_id"])
        self.x, self.N = pos.copy(), len(pos)
        self.img = np.zeros((self.N, 3))
        self.bond = np.ones(self.N, dtype=bool)          # bead i bonded to i + 1
        self.bond[np.cumsum(chain_len) - 1] = False
        lmin, lmax = p["lambda_min"], p["lambda_max"]
        self.modes, self.cdf, Z = _modes(self.L, lmax, p["lcut"])
        rl, M6 = lmax / lmin, 8.0 * math.pi ** 3 / 5.0
        R = (self.L / lmax) ** 3 * M6 / Z / (6.0 * math.pi ** 2)
        self.pF = 1.0 / (1.0 + R * (rl ** 3 - 1.0))
        nL = 1
        while lmin * 2.0 ** nL < lmax:
            nL += 1
        edges = [lmin * 2.0 ** l for l in range(nL)] + [lmax]
        self.bands = list(zip(edges[:-1], edges[1:]))
        self.carry, self.sweep, self.call, self.carry_k = [0.0] * nL, 0, 0, None

    def mi(self, d):
        return d - self.L * np.round(d / self.L)

    def place(self, m, new):
        """New positions of beads m wrapped into the box, with their image counts."""
        up, down = new >= self.L, new < 0.0
        self.x[m] = np.where(up, new - self.L, np.where(down, new + self.L, new))
        self.img[m] += up.astype(float) - down

    def wca(self, r2):
        p = self.p
        rc2 = (1.122462048309373 * p["wca_sigma"]) ** 2
        s6 = (p["wca_sigma"] ** 2 / np.where(r2 < rc2, r2, 1.0)) ** 3
        return np.where(r2 < rc2, 4.0 * p["wca_eps"] * (s6 * s6 - s6) + p["wca_eps"], 0.0)

    def spring(self, r2):
        return 0.5 * self.p["bond_k"] * (np.sqrt(r2) - self.p["bond_r0"]) ** 2

    def count(self, kind, layer, x):
        w = _draw(self.seed, self.sid, kind, layer, self.sweep, 0)
        return int(x) + int(_u53(w[0], w[1])[0] < x - int(x))

    def threshold(self, w):
        return -self.p["kT"] * np.log(1.0 - _u53(w[0], w[1]))

    def change(self, m, new):
        """Energy change when beads m move to `new` (every other bead stays)."""
        y = self.x.copy()
        y[m] = new
        member = np.zeros(self.N, dtype=bool)
        member[m] = True
        rank = np.arange(self.N)
        count = ~member[None, :] | (rank[None, :] > m[:, None])       # each pair once
        near = count & ((self.mi(self.x[m][:, None] - self.x[None]) ** 2).sum(axis=2) < (3.0 + self.p["lambda_max"]) ** 2)
        a, b = np.nonzero(near)
        a = m[a]
        d = self.wca((self.mi(y[a] - y[b]) ** 2).sum(axis=1)) - self.wca((self.mi(self.x[a] - self.x[b]) ** 2).sum(axis=1))
        lo = np.unique(np.concatenate([m, m - 1]))
        lo = lo[lo >= 0]
        lo = lo[self.bond[lo]]
        s = self.spring((self.mi(y[lo] - y[lo + 1]) ** 2).sum(axis=1)) - \
            self.spring((self.mi(self.x[lo] - self.x[lo + 1]) ** 2).sum(axis=1))
        return d.sum() + s.sum()

    def layer(self, l):
        lo, hi = self.bands[l]
        p, args = self.p, (l, self.sweep)
        mass = (lo ** -3 - hi ** -3) / (self.bands[0][0] ** -3 - self.bands[-1][1] ** -3)
        M = self.count(COUNT, l, self.N * (1.0 - self.pF) * mass)
        if M == 0:
            return
        w = _draw(self.seed, self.sid, SLOT, *args, np.arange(M))
        lam_own = (lo ** -3 - _u53(w[0], w[1]) * (lo ** -3 - hi ** -3)) ** (-1.0 / 3.0)
        n64 = np.uint64(self.N)
        bead = ((w[2] * n64 + ((w[3] * n64) >> np.uint64(32))) >> np.uint64(32)).astype(int)
        V = _ball(self.seed, self.sid, VB, *args, M, False)
        P = _ball(self.seed, self.sid, VP, *args, M, True)
        P /= np.sqrt((P * P).sum(axis=1))[:, None]
        thr = self.threshold(_draw(self.seed, self.sid, ACC, *args, np.arange(M)))
        for j in range(M):
            lam = self.carry[l] or lam_own[j]
            d = self.mi(self.x - (self.x[bead[j]] + lam * V[j]))
            d2 = (d * d).sum(axis=1)
            m = np.nonzero(d2 < lam * lam)[0]
            ok = True
            if m.size:
                s = p["A0"] * lam / math.sqrt(m.size) * (1.0 - np.sqrt(d2[m]) / lam) / lam
                new = self.x[m] + s[:, None] * np.cross(P[j], d[m])
                ok = self.change(m, new) <= thr[j]
                if ok:
                    self.place(m, new)
            self.carry[l] = 0.0 if ok else lam

    def plane_wave(self, index, ctr, kinds):
        p, N, L = self.p, self.N, self.L
        w1 = _draw(self.seed, self.sid, kinds[0], 0, ctr, index)
        w2 = _draw(self.seed, self.sid, kinds[1], 0, ctr, index)
        phi, psi = _u53(w1[2], w1[3])[0], _u53(w2[0], w2[1])[0]
        if self.carry_k is not None:
            perm = [(0, 1, 2), (0, 2, 1), (1, 0, 2), (1, 2, 0), (2, 0, 1), (2, 1, 0)][(int(w2[2][0]) * 6) >> 32]
            lv = np.array([self.carry_k[a] for a in perm])
            lv = np.where([(int(w2[3][0]) >> a) & 1 for a in range(3)], -lv, lv)
        else:
            lv = self.modes[np.searchsorted(self.cdf, _u53(w1[0], w1[1])[0], side="right")]
        self.carry_k = None
        if not lv.any():
            return
        l = math.sqrt(float((lv * lv).sum()))
        AF = 2.0 * p["A0"] / (2.0 * math.pi * l / L * math.sqrt(5.0 * N))
        u1 = np.array([1.0, 0.0, 0.0])
        if lv[0] or lv[1]:
            u1 = np.array([lv[1], -lv[0], 0.0]) / math.hypot(lv[0], lv[1])
        e = math.cos(2.0 * math.pi * psi) * u1 + math.sin(2.0 * math.pi * psi) * np.cross(lv / l, u1)
        new = self.x + (AF * np.cos(2.0 * math.pi * (self.x @ lv / L + phi)))[:, None] * e
        a, b = _pairs(self.x, L, 1.122462048309373 * p["wca_sigma"] + 2.0 * AF)
        d = self.wca((self.mi(new[a] - new[b]) ** 2).sum(axis=1)) - self.wca((self.mi(self.x[a] - self.x[b]) ** 2).sum(axis=1))
        lo = np.nonzero(self.bond)[0]
        s = self.spring((self.mi(new[lo] - new[lo + 1]) ** 2).sum(axis=1)) - \
            self.spring((self.mi(self.x[lo] - self.x[lo + 1]) ** 2).sum(axis=1))
        if d.sum() + s.sum() <= self.threshold(_draw(self.seed, self.sid, kinds[2], 0, ctr, index))[0]:
            self.place(slice(None), new)
        else:
            self.carry_k = lv

    def sweep_once(self):
        for l in range(len(self.bands)):
            self.layer(l)
        for k in range(self.count(PWCOUNT, 0, self.N * self.pF)):
            self.plane_wave(k, self.sweep, (PWMODE, PWDIR, PWACC))
        self.sweep += 1

    def positions(self):
        return self.x + self.img * self.L


def _pairs(x, L, r):
    """Pairs of beads within r of each other (minimum image), each once, by sorted cells."""
    g = max(1, int(L / r))
    if g < 3:
        a, b = np.triu_indices(len(x), 1)
    else:
        c = np.minimum((x * (g / L)).astype(np.int64), g - 1)
        key = c[:, 0] + g * (c[:, 1] + g * c[:, 2])
        order = np.argsort(key, kind="stable")
        sk, pa, pb = key[order], [], []
        for ox, oy, oz in [(i, j, k) for i in (-1, 0, 1) for j in (-1, 0, 1) for k in (-1, 0, 1)]:
            t = (c + np.array([ox, oy, oz])) % g
            tk = t[:, 0] + g * (t[:, 1] + g * t[:, 2])
            first, last = np.searchsorted(sk, tk, "left"), np.searchsorted(sk, tk, "right")
            for s in range(int((last - first).max())):
                i = np.nonzero(first + s < last)[0]
                j = order[first[i] + s]
                pa.append(i[i < j])
                pb.append(j[i < j])
        a, b = np.concatenate(pa), np.concatenate(pb)
    d = x[a] - x[b]
    d -= L * np.round(d / L)
    near = (d * d).sum(axis=1) < r * r
    return a[near], b[near]


def exact(case, seed):
    if case.get("planewaves", "sphere") != "sphere" or case["system"] == "paper_chains":
        return None
    if case["kind"] == "planewave" and _lengths(case) * case["sweeps"] < 1_600_000:
        system = _system(case, seed)
        e = _Exact(_params(case, system, seed), system.pos, system.chain_len)
        for k in range(case["sweeps"]):
            e.plane_wave(k, 0, (DPWMODE, DPWDIR, DPWACC))
        return torch.from_numpy(e.positions())
    if case["kind"] == "batch" and case["hi"] <= 256 and case["sims"] * case["sweeps"] <= 200:
        systems = _systems(case, seed)
        params = [_params(case, s, seed, sim_id=k, serial_only=True) for k, s in enumerate(systems)]
    elif case["kind"] == "sim" and case["system"] == "chain" and case["n"] <= 64:
        systems = [_system(case, seed)]
        params = [_params(case, systems[0], seed)]
        if any(params[0]["grid_layer"]):
            return None
    else:
        return None
    out = []
    for p, s in zip(params, systems):
        e = _Exact(p, s.pos, s.chain_len)
        for _ in range(case["sweeps"]):
            e.sweep_once()
        out.append(e.positions())
    return torch.from_numpy(np.concatenate(out))

"""What is measured: the calls a sampling program makes, over the sizes it makes them with.

A state is a `synth` bilayer on the GPU with the handle (`mdas.System`) that a
program keeps; a pass is one public call (or the upload, run, download triple
of a checkpointed round).  MD passes are 10 or 20 steps, as a sampler or the
serving loop advances a job between its other work; each pass continues where
the last one ended, as a sampling run does.  Returned per system: the velocities, the displacement of
every bead since `prepare` (position units of L / 2^32, minimum image) and the
lipid types.

`exact` is an independent FP64 evaluation in torch: Lennard-Jones with
potential shift and reaction field inside rc, harmonic bonds, cosine angles,
leapfrog with velocity rescaling, exchange and mutation trials, alchemical
moves and the box motion, with the counter-based random numbers (Philox
4x32-10) the calls document.
"""
import itertools
import math

import numpy as np
import torch

from paper_2005_08348_gb300 import mdas, synth

STEPS = 20                       # MD steps per pass (10 for the large bilayers)
BOX_COUPLING = dict(p_ref=1.0, tau_p=1e4, compressibility=3e-4, nstpcouple=10)


def listed():
    return [
        # MC-MD on the smallest bilayer (128 lipids): bound by latency, every launch and barrier counts
        dict(name="mcmd_128", kind="md", lipids=128, types=2, steps=STEPS, swap_every=5),
        # the headline workload: 1152 lipids, a trial after every MD step
        dict(name="mcmd_1152", kind="md", lipids=1152, types=3, steps=STEPS, swap_every=1),
        # plain MD of the large bilayer between its moves, default step shape
        dict(name="md_4608", kind="md", lipids=4608, types=3, steps=10, swap_every=0),
        # the largest served patch, with the step shape documented for such systems
        dict(name="mcmd_16384", kind="md", lipids=16384, types=3, steps=10, swap_every=5, lanes=2),
        # double precision, as the trajectories checked against the oracle
        dict(name="mcmd_128_fp64", kind="md", lipids=128, types=2, steps=STEPS, swap_every=10, precision="fp64"),
        # constant pressure: a box update every 10 steps
        dict(name="npt_1152", kind="md", lipids=1152, types=3, steps=20, swap_every=1, pressure=True),
        # an MDAS move: 16 lipids along 10 lambda steps of 5 MD steps
        dict(name="mdas_4608", kind="mdas", lipids=4608, types=3, pairs=8, lambdas=10, md=5, soft=0.0),
        # replicas of different sizes advanced together, then their trials
        dict(name="replicas_16", kind="replicas", count=16, least=128, most=2048, steps=STEPS, trials=STEPS, lanes=2),
        # a served exchange job on a patch of ordinary size
        dict(name="swaps_1424", kind="swaps", lipids=1424, types=3, trials=256),
        # semi-grand mutations on the large bilayer
        dict(name="mutations_4608", kind="mutations", lipids=4608, types=3, trials=256),
        # forces and energies of one state, as an analysis or another integrator asks for them
        dict(name="forces_1152", kind="forces", lipids=1152, types=3, precision="fp32"),
        # a checkpointed round: upload the packed state, run, download it
        dict(name="round_1152", kind="round", lipids=1152, types=3, steps=STEPS, swap_every=1),
    ]


def _spread(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case: lipid counts log-uniform over 128 - 16384 (even, most grids ragged)."""
    kind = rng.choice(["md", "md", "md", "md", "mdas", "replicas", "swaps", "mutations", "forces", "round"])
    types = rng.choice([2, 3])
    if kind == "md":
        how = rng.choice(["fp32", "fp32", "fp32", "fp64", "pressure"])
        most = {"fp32": 15500, "fp64": 600, "pressure": 4608}[how]
        c = dict(kind=kind, lipids=_spread(rng, 128, most), types=types, steps=rng.randint(5, STEPS),
                 swap_every=rng.choice([0, 1, 2, 3, 5, 10]), lanes=rng.choice([2, 4]))
        if how == "fp64":
            c["precision"] = "fp64"
        if how == "pressure":
            c["pressure"] = True
        if c["lipids"] > 3000:
            c["steps"] = min(c["steps"], 10)
        if rng.random() < 0.3:
            c["skin"] = round(rng.uniform(0.2, 0.5), 3)
    elif kind == "mdas":
        c = dict(kind=kind, lipids=_spread(rng, 128, 4608), types=types, pairs=rng.randint(1, 8),
                 lambdas=rng.randint(2, 10), md=rng.randint(1, 4), soft=rng.choice([0.0, 0.0, 0.05]))
    elif kind == "replicas":
        c = dict(kind=kind, count=rng.randint(2, 16), least=128, most=_spread(rng, 256, 2000), steps=rng.randint(5, STEPS),
                 trials=rng.randint(0, STEPS), lanes=rng.choice([2, 4]))
    elif kind in ("swaps", "mutations"):
        c = dict(kind=kind, lipids=_spread(rng, 128, 4608), types=types, trials=_spread(rng, 1, 512))
    elif kind == "forces":
        precision = rng.choice(["fp32", "fp32", "fp64"])
        c = dict(kind=kind, lipids=_spread(rng, 128, 8192 if precision == "fp32" else 1152), types=types, precision=precision)
    else:
        c = dict(kind=kind, lipids=_spread(rng, 128, 2048), types=types, steps=rng.randint(5, STEPS), swap_every=rng.choice([0, 1, 5]))
    if "lipids" in c:
        c["lipids"] -= c["lipids"] % 2
    return c


def _bilayer(lipids, types, seed, system_id=0):
    """The named workloads at their sizes, a patch on a near-square grid at any other."""
    fracs = [0.5, 0.5] if types == 2 else [0.4, 0.4, 0.2]
    grid = {128: (8, 1700), 1152: (24, 20000), 4608: (48, 85000)}.get(lipids)
    if grid:
        return synth.membrane(grid[0], n_lipid_types=types, fracs=fracs, n_water=grid[1], seed=seed, system_id=system_id)
    return synth.patch(lipids, types, seed=seed, system_id=system_id)


def _membranes(case, seed):
    seed = int(seed) % (1 << 30) + 1
    if case["kind"] != "replicas":
        return [_bilayer(case["lipids"], case["types"], seed)]
    # the spread of sizes belongs to the case, the bilayers to the seed
    sizes = np.linspace(case["least"], case["most"], case["count"]).astype(int) // 2 * 2
    return [_bilayer(int(n), 2 + k % 2, seed * 64 + k, system_id=k) for k, n in enumerate(sizes)]


_STREAM = []


def _stream():
    if not _STREAM:
        _STREAM.append(torch.cuda.Stream())
    return _STREAM[0]


def prepare(case, seed):
    with torch.cuda.stream(_stream()):
        ms = _membranes(case, seed)
        systems = [mdas.System(m, precision=case.get("precision", "fp32"), stream=_stream().cuda_stream,
                               list_skin=case.get("skin", 0.3 if case["kind"] == "replicas" else 0.0),
                               pcouple=BOX_COUPLING if case.get("pressure") else None) for m in ms]
        state = dict(case=case, systems=systems, views=[], start=[])
        for s in systems:
            if case.get("lanes", 4) != 4:
                s.set_list_lanes(case["lanes"])
            if case.get("soft"):
                s.set_soft_core(case["soft"])
            view = s.device_views()
            state["views"].append(view)
            state["start"].append(view["pos"][:, :3].clone())
        if case["kind"] == "round":
            n, nl = ms[0].n_beads, ms[0].n_lipids
            state["host"] = (torch.empty((n, 4), dtype=torch.int32).pin_memory(),
                             torch.empty((n, 4), dtype=torch.float32).pin_memory(),
                             torch.empty(nl, dtype=torch.int32).pin_memory())
            systems[0].get_state_packed(*state["host"])
            state["from"] = state["host"][0][:, :3].clone()
        if case["kind"] == "mutations":
            state["mu"] = np.array([0.0, 0.5, -0.3])[: case["types"]]
    return state


def run(state):
    case, systems = state["case"], state["systems"]
    s, kind = systems[0], case["kind"]
    with torch.cuda.stream(_stream()):
        if kind == "md":
            s.md_steps(case["steps"], swap_every=case["swap_every"])
            out = _moved(state, 0)
            if case.get("pressure"):
                box, speed, pressure = s.box()
                out.update(box=box, box_velocity=speed.astype(np.float32), pressure=pressure.astype(np.float32))
            return out
        if kind == "mdas":
            r = s.alchemical_move(case["pairs"], case["lambdas"], case["md"])
            return dict(w=r["w"], u=r["u"], accepted=r["accepted"], pairs=r["pairs"], **_moved(state, 0))
        if kind == "replicas":
            mdas.batch_run(systems, case["steps"], case["trials"])
            return [_moved(state, k) for k in range(len(systems))]
        if kind in ("swaps", "mutations"):
            if kind == "swaps":
                stats, rec = s.swap_trials(case["trials"])
            else:
                stats, rec = s.mutation_trials(case["trials"], mu=state["mu"])
            out = {k: np.ascontiguousarray(rec[k]) for k in ("a", "b", "null", "accepted", "dE", "u")}
            return dict(out, count=stats["accepted"], types=state["views"][0]["ltype"])
        if kind == "forces":
            F = s.forces()
            e = s.energy()
            return dict(e, forces=F if case["precision"] == "fp64" else F.astype(np.float32))
        s.set_state_packed(*state["host"])
        s.md_steps(case["steps"], swap_every=case["swap_every"])
        pos, vel, types = s.get_state_packed(*state["host"])
        return dict(moved=(pos[:, :3] - state["from"]).float(), vel=vel, types=types)


def _moved(state, k):
    v = state["views"][k]
    real = v["vel"].dtype
    return dict(moved=(v["pos"][:, :3] - state["start"][k]).to(real), vel=v["vel"], types=v["ltype"])


def _sizes(case):
    """Beads and lipids of each system, from its recipe (no arrays made)."""
    def beads(lipids):
        grid = {128: (8, 1700), 1152: (24, 20000), 4608: (48, 85000)}.get(lipids)
        if grid:
            return 12 * lipids + grid[1]
        nx = math.ceil(math.sqrt(lipids // 2))
        ny = math.ceil((lipids // 2) / nx)
        return 12 * lipids + int(8.3 * 0.64 * nx * ny * 5.0)
    if case["kind"] == "replicas":
        counts = [int(x) // 2 * 2 for x in np.linspace(case["least"], case["most"], case["count"])]
    else:
        counts = [case["lipids"]]
    return [(beads(n), n) for n in counts]


def work(case):
    """Bytes: each bead's position and velocity in and out once, the lipid types;
    flops: 30 per pair inside the cutoff (about 21 pairs per bead) and evaluation,
    about 40 per pair of a bead whose type a trial changes."""
    wide = 2 if case.get("precision") == "fp64" else 1
    kind, total = case["kind"], dict(bytes=0.0, flops=0.0)
    for n, nl in _sizes(case):
        state = n * (16 + 16 * wide) + 4 * nl
        if kind in ("md", "round"):
            steps, every = case["steps"], case["swap_every"]
            trials = steps // every if every else 0
            total["bytes"] += 2 * state
            total["flops"] += steps * n * 21 * 30 + trials * 10 * 42 * 40
        elif kind == "mdas":
            total["bytes"] += 2 * state
            total["flops"] += case["lambdas"] * (case["md"] * n * 21 * 30 + 2 * case["pairs"] * 5 * 42 * 40)
        elif kind == "replicas":
            total["bytes"] += 2 * state
            total["flops"] += case["steps"] * n * 21 * 30 + case["trials"] * 10 * 42 * 40
        elif kind in ("swaps", "mutations"):
            beads = 10 if kind == "swaps" else 5
            total["bytes"] += case["trials"] * (beads * 43 * 16 + 48)
            total["flops"] += case["trials"] * beads * 42 * 40
        else:
            total["bytes"] += state + 24 * n
            total["flops"] += n * 21 * (30 + 40)
    return total


# ------------------------------------------------------- FP64 evaluation
KB, COULOMB, BAR = 0.0083144626, 138.935458, 16.6053906717
TWO32 = 4294967296.0
M32 = 0xFFFFFFFF


def _philox(c, key):
    """Philox 4x32-10 of one counter (four words) and key (two words)."""
    c, k = list(c), list(key)
    for _ in range(10):
        p0, p1 = 0xD2511F53 * c[0], 0xCD9E8D57 * c[2]
        c = [(p1 >> 32) ^ c[1] ^ k[0], p1 & M32, (p0 >> 32) ^ c[3] ^ k[1], p0 & M32]
        k = [(k[0] + 0x9E3779B9) & M32, (k[1] + 0xBB67AE85) & M32]
    return c


def _unit(a, b):
    return (((a >> 5) << 26 | (b >> 6)) + 1.0) / 9007199254740992.0


class Reference:
    """One system in FP64 on the GPU (fixed-point positions, as the state holds them)."""

    def __init__(self, m, pressure=False, soft=0.0):
        d = torch.device("cuda")
        self.m, self.n, self.nl = m, m.n_beads, m.n_lipids
        self.x = torch.as_tensor(m.pos_u.astype(np.int64), device=d)
        self.v = torch.as_tensor(m.vel, dtype=torch.float64, device=d)
        self.start = self.x.clone()
        self.types = m.lipid_type.astype(np.int64).copy()
        self.box = np.array(m.box, np.float64)
        self.lbt = m.lipid_bead_type.astype(np.int64)
        self.bpl = self.lbt.shape[1]
        eps = torch.as_tensor(m.eps, device=d)
        s6 = torch.as_tensor(m.sigma, device=d) ** 6
        q = torch.as_tensor(m.charge, device=d)
        self.c12, self.c6 = 4 * eps * s6 * s6, 4 * eps * s6
        self.qq = COULOMB * q[:, None] * q[None, :] / m.eps_r
        self.krf, self.crf = 0.5 / m.rc ** 3, 1.5 / m.rc
        self.shift = self.c12 / m.rc ** 12 - self.c6 / m.rc ** 6
        self.key = ((m.seed & M32) ^ m.system_id, m.seed >> 32)
        self.kT = KB * m.temperature
        self.step = self.trial = self.move = self.at_step = 0
        self.built = None
        self.soft = soft
        self.pressure, self.boxv, self.pres = pressure, np.zeros(3), np.zeros(3)
        self.group = torch.zeros(self.n, dtype=torch.int64, device=d)
        self.group[self.nl * self.bpl:] = 1

    def beads(self, types):
        """Bead types under the given lipid types."""
        t = torch.full((self.n,), int(self.m.water_bead_type), dtype=torch.int64)
        t[: self.nl * self.bpl] = torch.as_tensor(self.lbt[types].reshape(-1))
        return t.cuda()

    def sep(self, a, b):
        """Minimum-image separation of fixed-point positions, nm."""
        d = (a - b) & M32
        d = d - ((d >> 31) << 32)
        return d.double() * torch.as_tensor(self.box / TWO32, device=d.device)

    def near(self):
        """Pairs (i, j, d, r2) inside rc, bonded pairs left out; the candidates
        (inside rc + 0.3 nm or a third of the shortest edge) last 3 calls."""
        if self.built is None or self.age >= 3:
            self.built, self.age = self.candidates(), 0
        self.age += 1
        i, j = self.built
        d = self.sep(self.x[i], self.x[j])
        r2 = (d * d).sum(1)
        keep = (r2 < self.m.rc ** 2) & (r2 > 0)
        return i[keep], j[keep], d[keep], r2[keep]

    def candidates(self):
        rl = min(self.m.rc + 0.3, float(self.box.min()) / 3)
        dims = [max(3, int(L // rl)) for L in self.box]
        c = (self.x * torch.as_tensor(dims, device="cuda")) >> 32
        cell = (c[:, 2] * dims[1] + c[:, 1]) * dims[0] + c[:, 0]
        ncell = dims[0] * dims[1] * dims[2]
        count = torch.bincount(cell, minlength=ncell)
        order = torch.argsort(cell, stable=True)
        first = torch.cumsum(count, 0) - count
        cap = int(count.max())
        slot = torch.arange(self.n, device="cuda") - first[cell[order]]
        table = torch.full((ncell, cap), -1, dtype=torch.int64, device="cuda")
        table[cell[order], slot] = order
        g = torch.arange(ncell, device="cuda")
        gx, gy, gz = g % dims[0], (g // dims[0]) % dims[1], g // (dims[0] * dims[1])
        lip = torch.arange(self.n, device="cuda") // self.bpl
        lip[self.nl * self.bpl:] = -1
        bonded = torch.zeros((self.bpl, self.bpl), dtype=torch.bool, device="cuda")
        for a, b in self.m.bonds:
            bonded[a, b] = bonded[b, a] = True
        half = [o for o in itertools.product((-1, 0, 1), repeat=3) if o > (0, 0, 0)] + [(0, 0, 0)]
        I, J = [], []
        for o in half:
            other = ((gz + o[0]) % dims[2] * dims[1] + (gy + o[1]) % dims[1]) * dims[0] + (gx + o[2]) % dims[0]
            for part in torch.split(g, max(1, 40_000_000 // (cap * cap))):
                a, b = table[part][:, :, None].expand(-1, cap, cap), table[other[part]][:, None, :].expand(-1, cap, cap)
                ok = (a >= 0) & (b >= 0)
                if o == (0, 0, 0):
                    ok = ok & (a < b)
                a, b = a[ok], b[ok]
                d = self.sep(self.x[a], self.x[b])
                ok = (d * d).sum(1) < rl * rl
                a, b = a[ok], b[ok]
                ok = ~((lip[a] == lip[b]) & (lip[a] >= 0) & bonded[a % self.bpl, b % self.bpl])
                I.append(a[ok])
                J.append(b[ok])
        return torch.cat(I), torch.cat(J)

    def forces(self, lam=None, other=None):
        """Forces, and the per-axis virial sum over pairs, bonds and angles."""
        m, t = self.m, self.beads(self.types)
        i, j, d, r2 = self.near()
        r = r2.sqrt()

        def lj(x, s2):
            s6 = 1 / (s2 * s2 * s2)
            return (12 * self.c12.flatten()[x] * s6 - 6 * self.c6.flatten()[x]) * s6 / s2

        nt = self.c12.shape[0]
        a = t[i] * nt + t[j]
        qq, f = self.qq.flatten()[a], None
        if other is None:
            f = lj(a, r2)
        else:
            u = self.beads(other)
            b = u[i] * nt + u[j]
            delta = torch.where((t[i] != u[i]) | (t[j] != u[j]), self.soft, 0.0)
            f = (1 - lam) * lj(a, r2 + delta * lam) + lam * lj(b, r2 + delta * (1 - lam))
            qq = (1 - lam) * qq + lam * self.qq.flatten()[b]
        f = f + qq * (1 / (r * r2) - 2 * self.krf)
        F = torch.zeros((self.n, 3), dtype=torch.float64, device="cuda")
        p = f[:, None] * d
        F.index_add_(0, i, p)
        F.index_add_(0, j, -p)
        vir = (p * d).sum(0)
        nb = self.nl * self.bpl
        X, B = self.x[:nb].view(self.nl, self.bpl, 3), torch.zeros((self.nl, self.bpl, 3), dtype=torch.float64, device="cuda")
        for a, b in m.bonds:
            d = self.sep(X[:, a], X[:, b])
            r = d.norm(dim=1, keepdim=True)
            p = -m.kb * (r - m.b0) / r * d
            B[:, a] += p
            B[:, b] -= p
            vir = vir + (p * d).sum(0)
        cos0 = math.cos(math.radians(m.theta0_deg))
        for a, b, c in m.angles:
            A, C = self.sep(X[:, a], X[:, b]), self.sep(X[:, c], X[:, b])
            la, lc = A.norm(dim=1, keepdim=True), C.norm(dim=1, keepdim=True)
            cs = (A * C).sum(1, keepdim=True) / (la * lc)
            pre = -m.ktheta * (cs - cos0)
            fa, fc = pre * (C / (la * lc) - cs * A / la ** 2), pre * (A / (la * lc) - cs * C / lc ** 2)
            B[:, a] += fa
            B[:, c] += fc
            B[:, b] -= fa + fc
            vir = vir + (A * fa + C * fc).sum(0)
        F[:nb] += B.view(nb, 3)
        return F, vir

    def energy(self):
        m, t = self.m, self.beads(self.types)
        i, j, d, r2 = self.near()
        x = t[i] * self.c12.shape[0] + t[j]
        s6 = 1 / r2 ** 3
        lj = ((self.c12.flatten()[x] * s6 - self.c6.flatten()[x]) * s6 - self.shift.flatten()[x]).sum()
        rf = (self.qq.flatten()[x] * (r2 ** -0.5 + self.krf * r2 - self.crf)).sum()
        X = self.x[: self.nl * self.bpl].view(self.nl, self.bpl, 3)
        bond = sum((0.5 * m.kb * (self.sep(X[:, a], X[:, b]).norm(dim=1) - m.b0) ** 2).sum() for a, b in m.bonds)
        cos0, angle = math.cos(math.radians(m.theta0_deg)), 0.0
        for a, b, c in m.angles:
            A, C = self.sep(X[:, a], X[:, b]), self.sep(X[:, c], X[:, b])
            angle = angle + (0.5 * m.ktheta * ((A * C).sum(1) / (A.norm(dim=1) * C.norm(dim=1)) - cos0) ** 2).sum()
        out = dict(lj=float(lj), rf=float(rf), bond=float(bond), angle=float(angle),
                   kinetic=float(0.5 * m.mass * (self.v ** 2).sum()))
        out["potential"] = out["lj"] + out["rf"] + out["bond"] + out["angle"]
        out["total"] = out["potential"] + out["kinetic"]
        return out

    def delta(self, near, ids, new):
        """Energy change when beads `ids` take the types `new`."""
        i, j, d, r2 = near
        t = self.bead_now
        u = t.clone()
        flag = torch.zeros(self.n, dtype=torch.bool, device="cuda")
        ids = torch.as_tensor(ids, device="cuda")
        u[ids] = torch.as_tensor(new, device="cuda")
        flag[ids] = True
        sel = flag[i] | flag[j]
        i, j, r2 = i[sel], j[sel], r2[sel]
        nt = self.c12.shape[0]
        a, b = t[i] * nt + t[j], u[i] * nt + u[j]
        s6 = 1 / r2 ** 3

        def of(tab):
            return tab.flatten()[b] - tab.flatten()[a]

        return float(((of(self.c12) * s6 - of(self.c6)) * s6 - of(self.shift)
                      + of(self.qq) * (r2 ** -0.5 + self.krf * r2 - self.crf)).sum())

    def alpha(self, group, tag, counter):
        m = self.m
        nf = 3 * (self.nl * self.bpl if group == 0 else self.n - self.nl * self.bpl)
        K = float(0.5 * m.mass * (self.v[self.group == group] ** 2).sum())
        if nf < 3 or K <= 0:
            return 1.0

        def normal(call):
            w = _philox((group, counter, tag, call), self.key)
            return math.sqrt(-2 * math.log(_unit(w[0], w[1]))) * math.cos(2 * math.pi * _unit(w[2], w[3]))

        shape = 0.5 * (nf - 1)
        d = shape - 1 / 3
        gamma = shape
        for t in range(32):
            x = normal(1 + 2 * t)
            v = (1 + x / math.sqrt(9 * d)) ** 3
            w = _philox((group, counter, tag, 2 + 2 * t), self.key)
            if v > 0 and math.log(_unit(w[0], w[1])) < 0.5 * x * x + d - d * v + d * math.log(v):
                gamma = d * v
                break
        c, kt = math.exp(-m.dt / m.tau_t), 0.5 * nf * self.kT
        a = math.sqrt(c * K) + normal(0) * math.sqrt((1 - c) * kt / nf)
        return math.sqrt((a * a + (1 - c) * kt / nf * 2 * gamma) / K)

    def md_step(self, lam=None, other=None):
        m, at = self.m, lam is not None
        counter = self.at_step if at else self.step
        al = [self.alpha(g, 5 if at else 1, counter) for g in (0, 1)]
        F, vir = self.forces(lam, other)
        scale = torch.tensor(al, dtype=torch.float64, device="cuda")[self.group][:, None]
        if self.pressure and not at:
            scale = scale - torch.as_tensor(m.dt * self.boxv / self.box, device="cuda")
        self.v = scale * self.v + F * (m.dt / m.mass)
        self.x = (self.x + (self.v * torch.as_tensor(m.dt * TWO32 / self.box, device="cuda")).round().long()) & M32
        if at:
            self.at_step += 1
            return
        self.step += 1
        nst = BOX_COUPLING["nstpcouple"]
        if self.pressure and self.step % nst == 0:
            V, L = float(np.prod(self.box)), self.box
            K = (0.5 * m.mass * (self.v ** 2).sum(0)).cpu().numpy()
            self.pres = (2 * K + vir.cpu().numpy()) / V * BAR
            lat = 0.5 * (self.pres[0] + self.pres[1])
            winv = 4 * math.pi ** 2 * BOX_COUPLING["compressibility"] / (3 * BOX_COUPLING["tau_p"] ** 2) / L.max()
            dtp = nst * m.dt
            self.boxv = self.boxv + dtp * V * winv * (np.array([lat, lat, self.pres[2]]) - BOX_COUPLING["p_ref"]) / L
            self.box = L + dtp * self.boxv

    def changed(self, pairs):
        """Bead ids and new bead types when the listed (lipid, new type) pairs are applied."""
        ids, new = [], []
        for l, t in pairs:
            for k in range(self.bpl):
                if self.lbt[self.types[l]][k] != self.lbt[t][k]:
                    ids.append(l * self.bpl + k)
                    new.append(int(self.lbt[t][k]))
        return ids, new

    def swap(self, near):
        w = _philox((0, self.trial, 2, 0), self.key)
        self.trial += 1
        a, b, u = (w[0] * self.nl) >> 32, (w[1] * self.nl) >> 32, _unit(w[2], w[3])
        ta, tb = int(self.types[a]), int(self.types[b])
        if a == b or ta == tb:
            return dict(dE=0.0, u=u)
        ids, new = self.changed([(a, tb), (b, ta)])
        dE = self.delta(near, ids, new)
        if dE + self.kT * math.log(u) <= 0:
            self.types[a], self.types[b] = tb, ta
            self.bead_now = self.beads(self.types)
        return dict(dE=dE, u=u)

    def mutate(self, near, mu):
        w = _philox((0, self.trial, 6, 0), self.key)
        self.trial += 1
        nt = self.lbt.shape[0]
        a, u = (w[0] * self.nl) >> 32, _unit(w[2], w[3])
        old = int(self.types[a])
        new = (old + 1 + ((w[1] * (nt - 1)) >> 32)) % nt
        ids, beads = self.changed([(a, new)])
        dE = self.delta(near, ids, beads)
        if dE - (mu[new] - mu[old]) + self.kT * math.log(u) <= 0:
            self.types[a] = new
            self.bead_now = self.beads(self.types)
        return dict(dE=dE, u=u)

    def trials(self, count, kind=None, mu=None):
        near, self.bead_now = self.near(), self.beads(self.types)
        recs = [self.swap(near) if kind is None else self.mutate(near, mu) for _ in range(count)]
        return {k: np.array([r[k] for r in recs]) for k in ("dE", "u")}

    def md(self, steps, every):
        for s in range(steps):
            self.md_step()
            if every and (s + 1) % every == 0:
                self.trials(1)

    def alchemical(self, pairs, lambdas, md):
        chosen, used = [], set()
        for j in range(64 * pairs + 64):
            if len(chosen) == pairs:
                break
            w = _philox((j, self.move, 3, 0), self.key)
            a, b = (w[0] * self.nl) >> 32, (w[1] * self.nl) >> 32
            if a != b and self.types[a] != self.types[b] and not {a, b} & used:
                chosen.append((a, b))
                used |= {a, b}
        other = self.types.copy()
        for a, b in chosen:
            other[a], other[b] = self.types[b], self.types[a]
        x0, v0, w = self.x, self.v, 0.0
        ids, new = self.changed([(l, int(other[l])) for p in chosen for l in p])
        for k in range(lambdas):
            for _ in range(md):
                self.md_step(k / lambdas, other)
            w += self.work(k / lambdas, (k + 1) / lambdas, ids, new)
        r = _philox((0, self.move, 4, 0), self.key)
        u = _unit(r[2], r[3])
        if w + self.kT * math.log(u) <= 0:
            self.types = other
        else:
            self.x, self.v = x0, v0
        return w, u

    def work(self, l0, l1, ids, new):
        near, self.bead_now = self.near(), self.beads(self.types)
        if not self.soft:
            return (l1 - l0) * self.delta(near, ids, new)
        i, j, d, r2 = near
        t, u = self.bead_now, self.bead_now.clone()
        u[torch.as_tensor(ids, device="cuda")] = torch.as_tensor(new, device="cuda")
        sel = (t[i] != u[i]) | (t[j] != u[j])
        i, j, r2 = i[sel], j[sel], r2[sel]
        nt = self.c12.shape[0]

        def lj(x, s2):
            s6 = 1 / s2 ** 3
            return (self.c12.flatten()[x] * s6 - self.c6.flatten()[x]) * s6

        def at(lam):
            e = 0.0
            for x, wt in ((t[i] * nt + t[j], 1 - lam), (u[i] * nt + u[j], lam)):
                extra, rc2 = self.soft * (1 - wt), torch.tensor(self.m.rc ** 2, dtype=torch.float64, device="cuda")
                e = e + wt * (lj(x, r2 + extra) - lj(x, rc2 + extra)
                              + self.qq.flatten()[x] * (r2 ** -0.5 + self.krf * r2 - self.crf))
            return e.sum()

        return float(at(l1) - at(l0))

    def moved(self):
        d = (self.x - self.start) & M32
        vel = torch.zeros((self.n, 4), dtype=torch.float64, device="cuda")
        vel[:, :3] = self.v
        return dict(moved=(d - ((d >> 31) << 32)).double(), vel=vel, types=None)


def exact(case, seed):
    refs = [Reference(m, bool(case.get("pressure")), case.get("soft", 0.0)) for m in _membranes(case, seed)]
    r, kind = refs[0], case["kind"]
    if kind in ("md", "round"):
        r.md(case["steps"], case["swap_every"])
        out = r.moved()
        if case.get("pressure"):
            out.update(box=r.box, box_velocity=r.boxv, pressure=r.pres)
        return out
    if kind == "mdas":
        w, u = r.alchemical(case["pairs"], case["lambdas"], case["md"])
        return dict(w=w, u=u, accepted=None, pairs=None, **r.moved())
    if kind == "replicas":
        for x in refs:
            x.md(case["steps"], 0)
            x.trials(case["trials"])
        return [x.moved() for x in refs]
    if kind in ("swaps", "mutations"):
        rec = r.trials(case["trials"], None if kind == "swaps" else kind, [0.0, 0.5, -0.3])
        return dict(a=None, b=None, null=None, accepted=None, dE=rec["dE"], u=rec["u"], count=None, types=None)
    return dict(r.energy(), pairs=None, forces=r.forces()[0])

"""The molecular-dynamics work that a user of this library has it do, as cases that
can be timed: listed() and draw() give them, prepare() builds what a program holds
before the call, run() is one pass through the public entry points, work() counts
what a pass cannot do without and exact() computes the same outputs in 64 bits.

A pass is one round of a program's run loop: advance the resident system by some
steps, read the thermodynamic state (the log line) and read a frame (unwrapped
positions and full-step velocities, or the forces).  The next pass goes on from
there.  The mixed-precision path computes its pair forces in FP32 and its frames
and log lines are kept in 32 bits, as trajectory files hold them; the FP64 path's
stay in 64 bits.
"""
import math

import numpy as np
import torch

from paper_1308_5587_gb300 import gbmd, workloads as wl

# per potential: the constant pair table of its single-type fluid
PAIRS = {"lj": wl.lj_single, "mie": wl.mie_single, "wca": wl.wca_single,
         "yukawa": wl.yukawa_single, "gauss": wl.gauss_single}
# FP32 / FP64 operations of one pair inside the cut-off, transcendentals as one
FLOPS = {"lj": 27, "wca": 27, "mie": 31, "yukawa": 29, "gauss": 24}

LJ = {"kind": "run", "pot": "lj", "binary": False, "rho": 0.84, "T": 1.2, "rcut": 2.5,
      "buff": 0.4, "prec": "mixed", "nvt": False, "nlist": "cell", "sort": 100,
      "read": "frame"}


def listed():
    def case(name, n, steps, **kw):
        return dict(LJ, name=name, n=n, steps=steps, **kw)
    return [
        # the smallest call: a driver outside (biasing, a learned correction) that
        # advances a small replica by single steps and reads the forces each time
        case("lj_500_one_step", 500, 1, read="forces", sort=0),
        # the plain FP64 workload of the benchmark at its small size
        case("lj_4k_fp64", 4000, 50, prec="fp64", sort=0),
        # the benchmark's fluid, mixed and plain FP64
        case("lj_64k_mixed", 64000, 50),
        case("lj_64k_fp64", 64000, 20, prec="fp64"),
        # the paper's own benchmark shape: dilute, r_cut 3, NVT, full FP64
        case("paper_64k_nvt_fp64", 64000, 20, prec="fp64", rho=0.382, rcut=3.0, nvt=True),
        # NVT in mixed precision at a ragged size with another potential
        case("yukawa_20011_nvt_mixed", 20011, 50, pot="yukawa", nvt=True),
        # a potential with transcendental functions on the 64k geometry
        case("mie_64k_mixed", 64000, 50, pot="mie"),
        # the upper end of the served requests' sizes, ragged
        case("lj_199999_mixed", 199999, 30, rho=0.8, sort=0),
        # size-disperse colloids on the tree neighbour list
        case("colloid_tree_r10", 100000, 40, kind="colloid", pot="wca", ratio=10.0,
             nlist="tree"),
        # many replicas stepped together, then each one's log line and frame
        case("batch_48_replicas", 20000, 64, kind="batch", replicas=48),
        # a configuration scan: new positions in, per-particle energies, virials and
        # forces out (import, sort, list build and readouts; no step)
        case("ka_20011_single_point", 20011, 0, kind="point", binary=True, rho=1.2, T=1.0,
             buff=0.3),
        # the headline workload: Kob-Andersen, a million particles
        case("ka_1m_mixed", 1000000, 20, binary=True, rho=1.2, T=1.0, buff=0.3,
             read="forces"),
    ]


def log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    c = dict(LJ)
    what = rng.choice(["run"] * 8 + ["one_step", "batch", "point", "colloid"])
    if what == "colloid":
        c.update(kind="colloid", pot="wca", nlist="tree", n=log_int(rng, 20000, 200000),
                 steps=rng.randint(10, 40), ratio=round(rng.uniform(5.0, 10.0), 2),
                 sort=rng.choice([0, 100]))
        return c
    if what == "batch":
        c.update(kind="batch", n=log_int(rng, 2000, 20000), replicas=rng.randint(5, 40),
                 steps=rng.randint(16, 64))
        return c
    c["rho"] = round(rng.uniform(0.7, 0.9), 3)
    c["T"] = round(rng.uniform(0.8, 1.5), 3)
    c["sort"] = rng.choice([0, 100])
    if rng.random() < 0.3:
        c.update(binary=True, rho=1.2, T=1.0, buff=0.3)
    elif rng.random() < 0.4:
        c["pot"] = rng.choice(["mie", "wca", "yukawa", "gauss"])
        c["rho"] = 0.84
    if what == "one_step":
        c.update(n=log_int(rng, 256, 20000), steps=1, read="forces")
    elif what == "point":
        c.update(kind="point", n=log_int(rng, 500, 200000), steps=0)
    elif rng.random() < 0.3:   # FP64
        c.update(prec="fp64", n=log_int(rng, 500, 64000), steps=rng.randint(8, 24))
    else:
        c.update(n=log_int(rng, 256, 400000), steps=rng.randint(16, 50))
    if c["kind"] == "run" and c["steps"] > 1:
        c["nvt"] = rng.random() < 0.25
        c["read"] = rng.choice(["frame", "frame", "forces"])
    return c


def pair_table(case):
    if case["binary"]:
        return wl.kob_andersen()
    if case["pot"] == "lj":
        return wl.lj_single(rcut=case["rcut"])
    return PAIRS[case["pot"]]()


def fluid(case, n, rho, T, seed):
    return wl.lj_fluid(n, rho, T, seed, pairs=pair_table(case), binary=case["binary"],
                       r_buff=case["buff"])


def inputs(case, seed):
    """The systems of a case, as the workload generator draws them."""
    seed = wl.BASE_SEED + 1009 * int(seed)
    if case["kind"] == "colloid":
        return [wl.colloid_mixture(case["n"], ratio=case["ratio"], seed=seed)]
    if case["kind"] == "batch":
        # the ensemble's sizes, densities and temperatures are the case's own
        params = wl.replica_params(case["replicas"], wl.BASE_SEED, 500, case["n"])
        return [fluid(case, n, rho, T, seed + k) for k, (n, rho, T, _) in enumerate(params)]
    return [fluid(case, case["n"], case["rho"], case["T"], seed)]


def system(case, w):
    kw = {"nlist": case["nlist"]}
    if case["nvt"]:
        kw.update(integrator="nvt", kT=case["T"], tau=1.0)
    return gbmd.System.from_workload(w, precision=case["prec"], sort_period=case["sort"],
                                     stream=torch.cuda.current_stream().cuda_stream, **kw)


def pinned(n, columns, dtype=torch.float64):
    return torch.empty((n, columns), dtype=dtype, pin_memory=True)


def prepare(case, seed):
    ws = inputs(case, seed)
    n = sum(w.n for w in ws)
    s = {"case": case, "n": [w.n for w in ws], "keep": torch.float64 if case["prec"] == "fp64"
         else torch.float32, "box": [torch.from_numpy(w.box) for w in ws]}
    if case["kind"] == "point":
        # the scan starts from some other configuration of the same system
        other = inputs(case, int(seed) + 1)[0]
        s["systems"] = [system(case, wl.Workload(other.pos, other.vel, ws[0].types, ws[0].box,
                                                 ws[0].pairs, ws[0].r_buff, ws[0].dt))]
        s["new_pos"], s["new_vel"] = pinned(n, 3), pinned(n, 3)
        s["new_pos"].copy_(torch.from_numpy(ws[0].pos))
        s["new_vel"].copy_(torch.from_numpy(ws[0].vel))
        s["forces"] = pinned(n, 3)
        return s
    s["systems"] = [system(case, w) for w in ws]
    if case["kind"] == "batch":
        s["batch"] = gbmd.Batch(case["prec"], stream=torch.cuda.current_stream().cuda_stream)
        for x in s["systems"]:
            s["batch"].add(x)
    if case["read"] == "forces":
        s["forces"] = pinned(n, 3)
    else:
        s["pos"], s["vel"], s["image"] = pinned(n, 3), pinned(n, 3), pinned(n, 3, torch.int32)
    return s


def log_line(t):
    return [t["pe"], t["ke"], t["temperature"], t["pressure"], *t["virial"], t["xi"], t["eta"]]


def run(s):
    case = s["case"]
    if case["kind"] == "point":
        x = s["systems"][0]
        x.set_state(s["new_pos"].numpy(), s["new_vel"].numpy())
        u, w = x.per_particle()
        x.forces(s["forces"].numpy())
        return {"u": torch.from_numpy(u).to(s["keep"]), "w": torch.from_numpy(w).to(s["keep"]),
                "forces": s["forces"].to(s["keep"])}
    (s["batch"] if case["kind"] == "batch" else s["systems"][0]).step(case["steps"])
    lines, at, out = [], 0, {}
    for x, n, box in zip(s["systems"], s["n"], s["box"]):
        if case["steps"] > 1:
            lines.append(log_line(x.thermo()))
        if case["read"] == "forces":
            x.forces(s["forces"][at:at + n].numpy())
        else:
            pos, vel, image = (s[k][at:at + n] for k in ("pos", "vel", "image"))
            gbmd.gbmd_get_state(x.handle, n, pos.numpy(), vel.numpy(), image.numpy())
            pos += image * box   # unwrapped
        at += n
    if lines:
        out["log"] = torch.tensor(lines, dtype=torch.float64).to(s["keep"])
    for k in ("forces",) if case["read"] == "forces" else ("pos", "vel"):
        out[k] = s[k].to(s["keep"])
    return out


def neighbours_inside(case):
    """(particles, sum over particles of the neighbours within r_cut) from the densities."""
    if case["kind"] == "batch":   # N log-uniform in [500, n], rho around 0.8
        n = case["replicas"] * (case["n"] - 500) / math.log(case["n"] / 500.0)
        return n, n * 0.8 * 4.0 / 3.0 * math.pi * 2.5 ** 3
    if case["kind"] == "colloid":   # small ones among themselves, large shells over small
        ratio, n = case["ratio"], case["n"]
        large = n / ratio ** 3
        rho = 0.2 / (math.pi / 6.0)
        cut = 2.0 ** (1.0 / 6.0)
        shell = (cut * 0.5 * (1 + ratio)) ** 3 - (0.5 * (1 + ratio)) ** 3
        return n + large, 4.0 / 3.0 * math.pi * rho * (n * (cut ** 3 - 1) + 2 * large * shell)
    t = pair_table(case)
    rc = 2.0 ** (1.0 / 6.0) * t.sigma if case["pot"] == "wca" else t.rcut
    x = np.array([0.8, 0.2]) if case["binary"] else np.ones(1)
    return case["n"], case["n"] * case["rho"] * 4.0 / 3.0 * math.pi * float(x @ rc ** 3 @ x)


def work(case):
    """Per step: positions and velocities read and written once, every pair inside the
    cut-off evaluated once.  Per read: what the program takes."""
    n, inside = neighbours_inside(case)
    pairs = 0.5 * inside * FLOPS[case["pot"]]
    if case["kind"] == "point":
        return {"bytes": n * (48 + 24 + 56), "flops": 2 * pairs}
    read = 24 if case["read"] == "forces" else 60
    return {"bytes": n * (96 * case["steps"] + read), "flops": pairs * (case["steps"] + 1)}


# ---- the same outputs in 64 bits, plain torch ------------------------------------

def half_pairs(x, box, types, rl):
    """Index pairs (i, j), each once, with minimum-image r < rl[type i, type j]."""
    n, dev = x.shape[0], x.device
    nc = [int(b // float(rl.max())) for b in box.tolist()]
    if min(nc) < 3:
        nc = [1, 1, 1]
    u = torch.remainder(x / box + 0.5, 1.0)
    m = torch.tensor(nc, device=dev)
    c = torch.minimum((u * m).long(), m - 1)
    cell = (c[:, 2] * nc[1] + c[:, 1]) * nc[0] + c[:, 0]
    order = torch.argsort(cell)
    count = torch.bincount(cell, minlength=nc[0] * nc[1] * nc[2])
    start = torch.cumsum(count, 0) - count
    most = int(count.max())
    rl2 = (rl * rl).reshape(-1)
    nt = rl.shape[0]
    steps = [(0, 0, 0)]
    if nc[0] > 1:
        steps += [(dx, dy, dz) for dz in (-1, 0, 1) for dy in (-1, 0, 1) for dx in (-1, 0, 1)
                  if (dz, dy, dx) > (0, 0, 0)]
    rows = max(1, 30_000_000 // most)
    found = []
    for a in range(0, n, rows):
        i = torch.arange(a, min(n, a + rows), device=dev)
        ci = c[i]
        for d in steps:
            q = (ci + torch.tensor(d, device=dev)) % m
            nb = (q[:, 2] * nc[1] + q[:, 1]) * nc[0] + q[:, 0]
            k = torch.arange(int(count[nb].max()), device=dev)
            at = start[nb][:, None] + k
            ok = k < count[nb][:, None]
            j = order[at.clamp(max=n - 1)]
            if d == (0, 0, 0):
                ok &= j > i[:, None]
            r2 = torch.zeros(j.shape, dtype=torch.float64, device=dev)
            for e in range(3):
                z = x[i, e][:, None] - x[:, e][j]
                z -= box[e] * torch.round(z / box[e])
                r2 += z * z
            ok &= r2 < rl2[types[i][:, None] * nt + types[j]]
            at = ok.nonzero()
            found.append((i[at[:, 0]], j[at[:, 0], at[:, 1]]))
    return torch.cat([f[0] for f in found]), torch.cat([f[1] for f in found])


def pair_terms(pot, t, p, r2):
    """f (force = f d) and the shifted energy of pairs of table entry p at r^2."""
    def of(table):
        return torch.as_tensor(np.asarray(table, np.float64).reshape(-1), device=r2.device)[p]
    eps = of(t.eps)
    rc2 = (2.0 ** (1.0 / 3.0)) * of(t.sigma) ** 2 if pot == "wca" else of(t.rcut) ** 2

    def lj(q):
        s6 = (of(t.sigma) ** 2 / q) ** 3
        return 24 * eps * (2 * s6 * s6 - s6) / q, 4 * eps * (s6 * s6 - s6)

    def mie(q):
        a, b = of(t.mie_n), of(t.mie_m)
        c = a / (a - b) * (a / b) ** (b / (a - b)) * eps
        s = of(t.sigma) ** 2 / q
        x, y = s ** (a / 2), s ** (b / 2)
        return c * (a * x - b * y) / q, c * (x - y)

    def yukawa(q):
        r, k = q.sqrt(), of(t.kappa)
        v = eps * torch.exp(-k * r) / r
        return v * (1 + k * r) / q, v

    def gauss(q):
        s2 = of(t.sigma) ** 2
        v = eps * torch.exp(-q / (2 * s2))
        return v / s2, v

    form = {"lj": lj, "wca": lj, "mie": mie, "yukawa": yukawa, "gauss": gauss}[pot]
    f, v = form(r2)
    inside = r2 < rc2
    zero = torch.zeros_like(f)
    return torch.where(inside, f, zero), torch.where(inside, v - form(rc2)[1], zero)


class Exact:
    """One system in FP64: a list with its own skin, rebuilt when a particle has moved
    more than half of it."""

    def __init__(self, case, w, skin=0.5):
        self.t, self.pot, self.w, self.skin = w.pairs, w.pairs.potential, w, skin
        dev = torch.device("cuda")
        self.x = torch.as_tensor(w.pos, device=dev).clone()
        self.v = torch.as_tensor(w.vel, device=dev).clone()
        self.box = torch.as_tensor(w.box, device=dev)
        self.types = torch.as_tensor(w.types, device=dev).long()
        rc = 2.0 ** (1.0 / 6.0) * w.pairs.sigma if self.pot == "wca" else w.pairs.rcut
        self.rc = torch.as_tensor(np.asarray(rc, np.float64), device=dev)
        self.kT = case["T"] if case["nvt"] else 0.0
        self.xi = self.eta = 0.0
        self.built = None

    def pairs(self):
        if self.built is None or 2 * float((self.x - self.built).norm(dim=1).max()) > self.skin:
            self.i, self.j = half_pairs(self.x, self.box, self.types, self.rc + self.skin)
            self.p = self.types[self.i] * self.rc.shape[0] + self.types[self.j]
            self.built = self.x.clone()
        d = self.x[self.i] - self.x[self.j]
        d -= self.box * torch.round(d / self.box)
        return d, *pair_terms(self.pot, self.t, self.p, (d * d).sum(1))

    def forces(self):
        d, f, _ = self.pairs()
        fd = f[:, None] * d
        return torch.zeros_like(self.x).index_add_(0, self.i, fd).index_add_(0, self.j, -fd)

    def per_particle(self):
        d, f, v = self.pairs()
        a, b = [0, 0, 0, 1, 1, 2], [0, 1, 2, 1, 2, 2]
        e = 0.5 * torch.cat([v[:, None], f[:, None] * d[:, a] * d[:, b]], 1)
        e = torch.zeros((len(self.x), 7), dtype=e.dtype, device=e.device).index_add_(
            0, self.i, e).index_add_(0, self.j, e)
        return e[:, 0], e[:, 1:]

    def kinetic(self):
        return 0.5 * self.w.mass * float((self.v * self.v).sum())

    def drive(self):
        """d xi / dt of the thermostat (tau 1)."""
        return 2.0 * self.kinetic() / ((3 * len(self.x) - 3) * self.kT) - 1.0

    def step(self, steps):
        dt, h = self.w.dt, 0.5 * self.w.dt
        F = self.forces()
        for _ in range(steps):
            if self.kT:
                self.xi += h * self.drive()
                self.eta += h * self.xi
                self.v *= math.exp(-h * self.xi)
            self.v += h / self.w.mass * F
            self.x += dt * self.v
            F = self.forces()
            self.v += h / self.w.mass * F
            if self.kT:
                self.v *= math.exp(-h * self.xi)
                self.eta += h * self.xi
                self.xi += h * self.drive()
        self.F = F

    def line(self):
        u, w = self.per_particle()
        n, ke = len(self.x), self.kinetic()
        T = 2.0 * ke / (3 * n - 3)
        w = w.sum(0)
        p = (n * T + float(w[0] + w[3] + w[5]) / 3.0) / float(self.box.prod())
        return [float(u.sum()), ke, T, p, *w.tolist(), self.xi, self.eta]


def exact(case, seed):
    systems = [Exact(case, w) for w in inputs(case, seed)]
    if case["kind"] == "point":
        u, w = systems[0].per_particle()
        return {"u": u, "w": w, "forces": systems[0].forces()}
    for e in systems:
        e.step(case["steps"])
    out = {}
    if case["steps"] > 1:
        out["log"] = torch.tensor([e.line() for e in systems], dtype=torch.float64)
    if case["read"] == "forces":
        out["forces"] = torch.cat([e.F for e in systems])
    else:
        out["pos"] = torch.cat([e.x for e in systems])
        out["vel"] = torch.cat([e.v for e in systems])
    return out

"""The workloads whose speed counts, as a program that uses this package runs them.

Each case is a dict of plain values.  `kind` says which entry point it goes
through:

* ``md``      RBE.step / RBEBatch.step: a block of MD steps in place, replayed
              from a CUDA graph (the package's main use);
* ``host``    RBE.step_host: one MD step on the caller's pinned host arrays
              (an MD engine that keeps its state on the host);
* ``forces``  RBE.forces: one mixed-precision force evaluation (an engine with
              an integrator of its own), or RBE.forces_f64;
* ``energy``  RBEEnergy forward and backward (a differentiable energy);
* ``observables``  RBE.observables: the full-Ewald energy and pressure.

Systems are the electrolytes and the water-like point charges of the package's
workloads and benchmark: monovalent ions at density 0.064 (alpha 0.3, r_c 5),
a 2:1 electrolyte at density 0.05 (alpha 0.2, r_c 6), the paper's
charge-correlation electrolyte at density 0.3 (alpha 0.55, r_c 4, sigma 0.2,
Andersen thermostat) and rigid three-site molecules at 0.0334 per unit volume
(alpha 0.1, r_c 10, no Lennard-Jones).

`exact` restates the method in 64-bit torch: Philox draws, the structure
factors and the Fourier force of the batch, the real-space and Lennard-Jones
pairs, the thermostats, and the full Ewald sum of the observables.
"""
import math

import numpy as np
import torch

DEV = "cuda"
WCA = 2.0 ** (1.0 / 6.0)

# density, charges, alpha, r_c, LJ (eps, sigma, cutoff), time step, closest approach
SYSTEMS = {
    "1:1": dict(density=0.064, qp=1.0, qn=-1.0, alpha=0.3, r_c=5.0, lj=(1.0, 1.0, WCA), dt=1e-3,
                near=0.9),
    "2:1": dict(density=0.05, qp=2.0, qn=-1.0, alpha=0.2, r_c=6.0, lj=(1.0, 1.0, WCA), dt=1e-3,
                near=0.9),
    "dh": dict(density=0.3, qp=1.0, qn=-1.0, alpha=0.55, r_c=4.0, lj=(1.0, 0.2, 4.0), dt=2e-3,
               near=0.25),
    "water": dict(density=3 * 0.0334, alpha=0.1, r_c=10.0, lj=(0.0, 1.0, WCA), dt=1e-3),
}
ANDERSEN_NU, NH_TAU = 3.0, 0.5


def listed():
    return [
        # the paper's charge-correlation run: 300 ions, batch 10, Andersen, 1e5 steps and more
        dict(name="md_dh300", kind="md", system="dh", n=300, P=10, thermostat="andersen", steps=50),
        # a small electrolyte, the size most method studies use
        dict(name="md_1000", kind="md", system="1:1", n=1000, P=100, thermostat="langevin",
             steps=20),
        # the asymmetric electrolyte of the benchmark, tuned, with each step's force recorded
        dict(name="md_2to1_8001", kind="md", system="2:1", n=8001, P=200, thermostat="langevin",
             steps=10, autotune=True, force=True),
        # an odd middle size and batch, the deterministic thermostat, library defaults
        dict(name="md_nh_50021", kind="md", system="1:1", n=50021, P=137,
             thermostat="nose_hoover", steps=5, force=True),
        # the benchmark's large electrolyte, tuned as a production run is
        dict(name="md_1048576", kind="md", system="1:1", n=1 << 20, P=500, thermostat="langevin",
             steps=2, autotune=True),
        # 64 independent systems of different size in one handle (parameter scans, replicas)
        dict(name="md_replicas", kind="md", system="1:1", n=1000, n_hi=65536, replicas=64, P=100,
             thermostat="langevin", steps=2),
        # an engine with its state in pinned host memory, one step per call
        dict(name="host_262144", kind="host", system="1:1", n=1 << 18, P=500,
             thermostat="langevin", steps=1),
        # an engine with its own integrator: forces only
        dict(name="forces_100003", kind="forces", system="1:1", n=100003, P=200, bits=32),
        # training against charges and positions: energy, forces and potentials of a frozen batch
        dict(name="energy_water_30000", kind="energy", system="water", n=30000, P=100),
        # FP64 dynamics of a small system (reference trajectories)
        dict(name="md64_1000", kind="md", system="1:1", n=1000, P=100, thermostat="langevin",
             steps=5, bits=64),
        # FP64 forces, energy and potentials (validation of a mixed run)
        dict(name="forces64_8001", kind="forces", system="2:1", n=8001, P=200, bits=64),
        # the observables a run samples now and then
        dict(name="observables_8001", kind="observables", system="2:1", n=8001, P=200),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["md", "md", "md", "md", "replicas", "host", "forces", "energy", "md64",
                       "forces64", "observables"])
    if kind == "md":
        system = rng.choice(["1:1", "1:1", "2:1", "dh"])
        n = _log(rng, 250, 2000) if system == "dh" else _log(rng, 400, 1 << 20)
        c = dict(kind="md", system=system, n=n,
                 P=_log(rng, 8, 500),
                 thermostat=rng.choice(["langevin", "andersen", "nose_hoover"]),
                 steps=50 if n < 700 else 20 if n < 4000 else 10 if n < 20000 else
                 5 if n < 200000 else 2)
        if rng.random() < 0.5:
            c["force"] = True
        return c
    if kind == "replicas":
        return dict(kind="md", system="1:1", n=rng.randint(600, 1500), n_hi=_log(rng, 4000, 50000),
                    replicas=rng.randint(3, 48), P=_log(rng, 50, 150),
                    thermostat=rng.choice(["langevin", "nose_hoover"]), steps=2)
    if kind == "host":
        return dict(kind="host", system="1:1", n=_log(rng, 1000, 1 << 18), P=_log(rng, 50, 500),
                    thermostat="langevin", steps=1)
    if kind == "forces":
        return dict(kind="forces", system=rng.choice(["1:1", "2:1"]), n=_log(rng, 500, 600000),
                    P=_log(rng, 10, 500), bits=32)
    if kind == "energy":
        return dict(kind="energy", system=rng.choice(["water", "1:1"]),
                    n=3 * _log(rng, 1000, 12000), P=_log(rng, 50, 200))
    if kind == "md64":
        return dict(kind="md", system="1:1", n=_log(rng, 400, 4000), P=_log(rng, 20, 200),
                    thermostat=rng.choice(["langevin", "andersen"]), steps=5, bits=64)
    if kind == "forces64":
        return dict(kind="forces", system=rng.choice(["1:1", "2:1"]), n=_log(rng, 500, 20000),
                    P=_log(rng, 20, 300), bits=64)
    return dict(kind="observables", system=rng.choice(["1:1", "2:1"]), n=_log(rng, 500, 8001),
                P=100)


# ------------------------------------------------------------------ inputs
def _sizes(case):
    """Particles of each system of the case."""
    if not case.get("replicas"):
        return [case["n"]]
    r = np.random.default_rng([case["n"], case["n_hi"], case["replicas"]])
    ns = np.exp(r.uniform(math.log(case["n"]), math.log(case["n_hi"]), size=case["replicas"]))
    return [int(v) for v in ns]


def _systems(case, seed):
    """Parameters of each system: what params_from reads."""
    d = SYSTEMS[case["system"]]
    out = []
    for s, n in enumerate(_sizes(case)):
        L = (n / d["density"]) ** (1.0 / 3.0)
        eps, sigma, lj_cut = d["lj"]
        out.append(dict(n=n, box=L, alpha=d["alpha"], r_c=min(d["r_c"], L / 2), P=case["P"],
                        seed=int(seed) % (1 << 31), stream=s, coulomb_prefactor=1.0, lj_eps=eps,
                        lj_sigma=sigma, lj_rcut=min(lj_cut, d["r_c"], L / 2), gamma=1.0, kT=1.0,
                        dt=d["dt"], mass=1.0,
                        thermostat={"langevin": 0, "andersen": 1,
                                    "nose_hoover": 2}[case.get("thermostat", "langevin")],
                        andersen_nu=ANDERSEN_NU, nh_tau=NH_TAU))
    return out


def _place(n, L, near, g):
    """n points at least about `near` apart: distinct random sites of a fine
    lattice, each jittered (dense enough in sites that the occupancy
    fluctuates as in a fluid)."""
    side = max(int(math.ceil(n ** (1.0 / 3.0))), int(L / (1.35 * near)))
    a = L / side
    sites = torch.randperm(side ** 3, generator=g, device=DEV)[:n]
    idx = torch.stack([sites % side, (sites // side) % side, sites // (side * side)], 1).double()
    jit = (torch.rand((n, 3), generator=g, device=DEV, dtype=torch.float64) - 0.5) * max(
        0.0, a - near)
    return (idx + 0.5) * a + jit


def _water(n_mol, L, g):
    """Rigid three-site molecules, O-H 1.0, 109.47 degrees, random orientations,
    centres on a jittered lattice at least 2.5 apart."""
    side = int(math.ceil(n_mol ** (1.0 / 3.0) - 1e-9))
    a = L / side
    sites = torch.randperm(side ** 3, generator=g, device=DEV)[:n_mol]
    idx = torch.stack([sites % side, (sites // side) % side, sites // (side * side)], 1).double()
    jit = (torch.rand((n_mol, 3), generator=g, device=DEV, dtype=torch.float64) - 0.5) * max(
        0.0, a - 2.5)
    u = torch.randn((2, n_mol, 3), generator=g, device=DEV, dtype=torch.float64)
    e1 = u[0] / u[0].norm(dim=1, keepdim=True)
    e2 = u[1] - (u[1] * e1).sum(1, keepdim=True) * e1
    e2 = e2 / e2.norm(dim=1, keepdim=True)
    h = math.radians(109.47) / 2
    c = (idx + 0.5) * a + jit
    H = math.cos(h) * e1
    return torch.stack([c, c + H + math.sin(h) * e2, c + H - math.sin(h) * e2], 1).reshape(-1, 3)


def _inputs(case, seed):
    """(pos_q, vel) float32 [n, 4] of all systems, concatenated."""
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed))
    d = SYSTEMS[case["system"]]
    pos, vel = [], []
    for p in _systems(case, seed):
        n, L = p["n"], p["box"]
        if case["system"] == "water":
            r = _water(n // 3, L, g)
            q = torch.tensor([-0.8476, 0.4238, 0.4238], device=DEV,
                             dtype=torch.float64).repeat(n // 3)
        else:
            r = _place(n, L, d["near"], g)
            npos = n // 2 if d["qp"] == -d["qn"] else n // 3
            q = torch.full((n,), d["qn"], device=DEV, dtype=torch.float64)
            q[torch.randperm(n, generator=g, device=DEV)[:npos]] = d["qp"]
        r = torch.remainder(r, L).float()
        r = torch.where(r >= np.float32(L), torch.zeros_like(r), r)
        v = torch.zeros((n, 4), device=DEV)
        v[:, :3] = torch.randn((n, 3), generator=g, device=DEV) * math.sqrt(p["kT"] / p["mass"])
        pos.append(torch.cat([r, q.float()[:, None]], 1))
        vel.append(v)
    return torch.cat(pos).contiguous(), torch.cat(vel).contiguous()


class _Params:
    def __init__(self, d):
        self.__dict__.update(d)


def prepare(case, seed):
    import paper_2010_01559_gb300 as rbe
    pos, vel = _inputs(case, seed)
    systems = _systems(case, seed)
    if case.get("replicas"):
        h = rbe.RBEBatch([rbe.params_from(_Params(p), n_max=p["n"]) for p in systems],
                         [p["n"] for p in systems])
    else:
        h = rbe.RBE(rbe.params_from(_Params(systems[0]), n_max=systems[0]["n"]))
    s = dict(case=case, h=h, step=0)
    kind = case["kind"]
    if kind == "host":
        s["pos"], s["vel"] = pos.cpu().pin_memory(), vel.cpu().pin_memory()
        h.set_graph(True)
        return s
    if kind == "energy":
        s["pos"] = pos[:, :3].contiguous().requires_grad_()
        s["q"] = pos[:, 3].contiguous().requires_grad_()
        s["apply"] = rbe.RBEEnergy.apply
        return s
    if case.get("bits") == 64:
        pos, vel = pos.double(), vel.double()
    s["pos"], s["vel"] = pos, vel
    if kind == "md":
        s["step_dev"] = torch.zeros(1, dtype=torch.int64, device=DEV)
        s["F"] = torch.zeros_like(pos) if case.get("force") else None
        if case.get("autotune"):
            h.autotune(pos)
        h.set_graph(True)
    return s


def run(s):
    case, h, kind = s["case"], s["h"], s["case"]["kind"]
    if kind == "md":
        h.step(s["pos"], s["vel"], case["steps"], s["step_dev"], F_out=s["F"])
        return {"pos": s["pos"], "vel": s["vel"], "F": s["F"]}
    step = s["step"]
    s["step"] = step + case.get("steps", 1)
    if kind == "host":
        h.step_host(s["pos"], s["vel"], case["steps"], step)
        return {"pos": s["pos"], "vel": s["vel"]}
    if kind == "energy":
        e = s["apply"](s["pos"], s["q"], h, step)
        gpos, gq = torch.autograd.grad(e, (s["pos"], s["q"]))
        return {"E": e.detach(), "gpos": gpos, "gq": gq}
    if kind == "observables":
        return h.observables(s["pos"], s["vel"])
    if case["bits"] == 64:
        F, E, phi = h.forces_f64(s["pos"], step, energy=True, phi=True)
        return {"F": F, "E": E, "phi": phi}
    F, _, _ = h.forces(s["pos"], step, energy=False)
    return {"F": F}


def work(case):
    """Each input read once, each output written once; floating-point
    operations of the Fourier sums (a sine or a cosine counts one: 12 per
    particle and wave vector for the structure factors, 13 for the force) and
    of the pairs within the cutoff (about 40 each)."""
    d = SYSTEMS[case["system"]]
    wide = 8 if case.get("bits") == 64 else 4
    steps = case.get("steps", 1)
    nbytes = flops = 0.0
    for n in _sizes(case):
        L = (n / d["density"]) ** (1.0 / 3.0)
        rc = min(d["r_c"], L / 2)
        pairs = n * 4.0 / 3.0 * math.pi * rc ** 3 * d["density"]
        if case["kind"] == "observables":
            m = math.ceil(math.sqrt(d["alpha"] * L * L * 64 * math.log(2)) / math.pi)
            flops += 12.0 * n * ((2 * m + 1) ** 3 - 1) / 2 + 40 * pairs
            nbytes += 32 * n
            continue
        flops += steps * (25.0 * n * case["P"] + 40 * pairs)
        if case["kind"] in ("md", "host"):
            # positions and velocities in and out, the last step's force where it is asked for
            nbytes += wide * n * (16 + (4 if case.get("force") else 0))
        elif case["kind"] == "energy":
            nbytes += wide * n * 8
        else:
            nbytes += wide * n * (9 if case["bits"] == 64 else 8)
    return {"bytes": nbytes, "flops": flops}


# ------------------------------------------------------- 64-bit restatement
def _philox(c0, c1, c2, c3, seed):
    """Philox4x32-10 on uint64 arrays holding 32-bit words."""
    m32 = np.uint64(0xFFFFFFFF)
    k0, k1 = np.uint64(seed & 0xFFFFFFFF), np.uint64(seed >> 32)
    c0, c1, c2, c3 = np.broadcast_arrays(*[np.asarray(c, dtype=np.uint64) for c in (c0, c1, c2, c3)])
    for r in range(10):
        if r:
            k0 = (k0 + np.uint64(0x9E3779B9)) & m32
            k1 = (k1 + np.uint64(0xBB67AE85)) & m32
        p0, p1 = c0 * np.uint64(0xD2511F53), c2 * np.uint64(0xCD9E8D57)
        c0, c1, c2, c3 = ((p1 >> np.uint64(32)) ^ c1 ^ k0, p1 & m32,
                          (p0 >> np.uint64(32)) ^ c3 ^ k1, p0 & m32)
    return c0, c1, c2, c3


def _axis_table(alpha, L):
    M = int(math.ceil(math.sqrt(alpha * L * L * (64.0 * math.log(2.0))) / math.pi))
    w = np.exp(-(math.pi ** 2 / (alpha * L * L)) * np.arange(-M, M + 1, dtype=np.float64) ** 2)
    cum = np.cumsum(w)
    T = np.minimum(np.floor(cum / cum[-1] * 4294967296.0), 4294967295.0).astype(np.uint64)
    T[-1] = np.uint64(1 << 32)
    return M, T, float(cum[-1])


def _batch(p, step):
    """The P wave vectors (integers) of a step and S."""
    M, T, H = _axis_table(p["alpha"], p["box"])
    m = np.zeros((p["P"], 3))
    todo, att = np.arange(p["P"]), 0
    while len(todo):
        w = _philox(todo, att, step & 0xFFFFFFFF, (p["stream"] << 8) | 1, p["seed"])
        got = np.stack([np.searchsorted(T, x, side="right") - M for x in w[:3]], 1)
        m[todo] = got
        todo, att = todo[(got == 0).all(1)], att + 1
    return torch.from_numpy(m).to(DEV), H ** 3 - 1.0


def _fourier(p, r, q, step):
    """(force, dE/dq, energy) of the Fourier part with self and background terms."""
    L, V, a = p["box"], p["box"] ** 3, p["alpha"]
    m, S = _batch(p, step)
    k = m * (2 * math.pi / L)
    k2 = (k * k).sum(1)
    coef = p["coulomb_prefactor"] * (S / p["P"]) * 4 * math.pi / (V * k2)
    chunk = max(1, (1 << 24) // p["P"])
    frac = r / L
    turn = 2 * math.pi

    def phases(x):
        t = x @ m.T
        return (t - torch.round(t)) * turn

    re, im = torch.zeros_like(k2), torch.zeros_like(k2)
    for b in range(0, len(q), chunk):
        th = phases(frac[b:b + chunk])
        re += q[b:b + chunk] @ torch.cos(th)
        im += q[b:b + chunk] @ torch.sin(th)
    F, phi = torch.empty_like(r), torch.empty_like(q)
    for b in range(0, len(q), chunk):
        th = phases(frac[b:b + chunk])
        c, s = torch.cos(th), torch.sin(th)
        F[b:b + chunk] = -q[b:b + chunk, None] * ((c * (coef * im) - s * (coef * re)) @ k)
        phi[b:b + chunk] = (c * (coef * re) + s * (coef * im)).sum(1)
    Q, Q2 = q.sum(), (q * q).sum()
    self_c = p["coulomb_prefactor"] * math.sqrt(a / math.pi)
    bg = p["coulomb_prefactor"] * math.pi / (V * a)
    E = (0.5 * coef * (re * re + im * im)).sum() - self_c * Q2 - 0.5 * bg * Q * Q
    return F, phi - 2 * self_c * q - bg * Q, E


def _pairs(r, L, rc):
    """Batches (i, j, displacement) of the directed pairs within rc."""
    n = len(r)
    r = torch.remainder(r, L)
    ncd = int(L / rc)
    if n <= 4096 or ncd < 3:
        step = max(1, (1 << 24) // n)
        for b in range(0, n, step):
            d = r[None] - r[b:b + step, None]
            d -= L * torch.round(d / L)
            ok = (d * d).sum(2) < rc * rc
            ok[torch.arange(len(d), device=DEV), torch.arange(b, b + len(d), device=DEV)] = False
            i, j = ok.nonzero(as_tuple=True)
            yield i + b, j, d[i, j]
        return
    c = torch.clamp((r * (ncd / L)).long(), 0, ncd - 1)
    cell = (c[:, 2] * ncd + c[:, 1]) * ncd + c[:, 0]
    order = torch.argsort(cell)
    cnt = torch.bincount(cell, minlength=ncd ** 3)
    cap = int(cnt.max())
    start = torch.cumsum(cnt, 0) - cnt
    table = torch.full((ncd ** 3, cap), -1, dtype=torch.long, device=DEV)
    sc = cell[order]
    table[sc, torch.arange(n, device=DEV) - start[sc]] = order
    ids = torch.arange(ncd ** 3, device=DEV)
    cx, cy, cz = ids % ncd, (ids // ncd) % ncd, ids // (ncd * ncd)
    step = max(1, (1 << 23) // (cap * cap))
    for o in range(27):
        dx, dy, dz = o % 3 - 1, (o // 3) % 3 - 1, o // 9 - 1
        nb = (((cz + dz) % ncd) * ncd + (cy + dy) % ncd) * ncd + (cx + dx) % ncd
        for b in range(0, ncd ** 3, step):
            i, j = table[b:b + step, :, None], table[nb[b:b + step], None, :]
            ok = ((i >= 0) & (j >= 0) & (i != j)).nonzero(as_tuple=True)
            i, j = table[b:b + step][ok[0], ok[1]], table[nb[b:b + step]][ok[0], ok[2]]
            d = r[j] - r[i]
            d -= L * torch.round(d / L)
            near = (d * d).sum(1) < rc * rc
            yield i[near], j[near], d[near]


def _real(p, r, q):
    """Real-space Coulomb and Lennard-Jones: force, dE/dq, energies and virials."""
    a, lB, eps = p["alpha"], p["coulomb_prefactor"], p["lj_eps"]
    F, phi = torch.zeros_like(r), torch.zeros_like(q)
    sums = torch.zeros(4, dtype=torch.float64, device=DEV)
    sr6c = (p["lj_sigma"] / p["lj_rcut"]) ** 6
    shift = -4 * eps * (sr6c * sr6c - sr6c)
    for i, j, d in _pairs(r, p["box"], p["r_c"]):
        r2 = (d * d).sum(1)
        x = torch.sqrt(r2)
        er = torch.erfc(math.sqrt(a) * x) / x
        ga = 2 * math.sqrt(a / math.pi) * torch.exp(-a * r2)
        qq = lB * q[i] * q[j]
        f = -qq * (er + ga) / r2
        lj = (r2 < p["lj_rcut"] ** 2) if eps else None
        sums[0] += 0.5 * (qq * er).sum()
        sums[2] += 0.5 * (qq * (er + ga)).sum()
        if eps:
            s6 = torch.where(lj, (p["lj_sigma"] ** 2 / r2) ** 3, torch.zeros_like(r2))
            mag = 24 * eps * (2 * s6 * s6 - s6) / r2
            f = f - mag
            sums[1] += 0.5 * (4 * eps * (s6 * s6 - s6) + shift * lj).sum()
            sums[3] += 0.5 * (mag * r2).sum()
        F.index_add_(0, i, f[:, None] * d)
        phi.index_add_(0, i, lB * q[j] * er)
    return F, phi, sums


def _normals(p, step, n, bits):
    """The thermostat's normals of a step and the Andersen collisions."""
    andersen = p["thermostat"] == 1
    i = np.arange(n)
    tag = (p["stream"] << 8) | (7 if andersen else 2)
    c = _philox(i, 0, step, tag, p["seed"])
    w = _philox(i, 1, step, tag, p["seed"]) if andersen else c
    thr = np.floor(p["andersen_nu"] * p["dt"] * 4294967296.0)
    hit = torch.from_numpy(c[0].astype(np.float64) < thr).to(DEV) if andersen else None
    if bits == 64:
        u = [x.astype(np.float64) for x in w]
        u1, u2, u3, u4 = ((u[0] + 1) / 2 ** 32, u[1] / 2 ** 32, (u[2] + 1) / 2 ** 32,
                          u[3] / 2 ** 32)
    else:
        u = [(x >> np.uint64(8)).astype(np.float64) for x in w]
        u1, u2, u3, u4 = ((u[0] + 1) / 2 ** 24, u[1] / 2 ** 24, (u[2] + 1) / 2 ** 24,
                          u[3] / 2 ** 24)
    a, b = np.sqrt(-2 * np.log(u1)), np.sqrt(-2 * np.log(u3))
    xi = np.stack([a * np.cos(2 * np.pi * u2), a * np.sin(2 * np.pi * u2),
                   b * np.cos(2 * np.pi * u4)], 1)
    return torch.from_numpy(xi).to(DEV), hit


def _dynamics(p, r, v, q, steps, bits):
    """`steps` MD steps from step 0: positions, velocities, the last step's force."""
    L, dt, m = p["box"], p["dt"], p["mass"]
    xi_nh, k2, F = 0.0, None, None
    for step in range(steps):
        F = _fourier(p, r, q, step)[0] + _real(p, r, q)[0]
        if p["thermostat"] == 2:
            if k2 is not None:
                xi_nh += dt / (3.0 * len(q) * p["nh_tau"] ** 2) * (k2 - 3.0 * len(q))
            hx = 0.5 * xi_nh * dt
            v = (v * (1 - hx) + (dt / m) * F) / (1 + hx)
            k2 = float((v * v).sum()) * m / p["kT"]
            r = r + dt * v
        else:
            xi, hit = _normals(p, step, len(q), bits)
            v = v + (dt / m) * F
            if p["thermostat"] == 0:
                c1 = math.exp(-p["gamma"] * dt / m)
                v = c1 * v + math.sqrt((1 - c1 * c1) * p["kT"] / m) * xi
            r = r + dt * v
            if hit is not None:
                v = torch.where(hit[:, None], math.sqrt(p["kT"] / m) * xi, v)
        r = r - L * torch.floor(r / L)
    return r, v, F


def _observables(p, r, q, v):
    """The full Ewald sum over the cube |m| <= M, kinetic energy, pressure."""
    L, V, a, lB = p["box"], p["box"] ** 3, p["alpha"], p["coulomb_prefactor"]
    M = _axis_table(a, L)[0]
    m = torch.arange(-M, M + 1, dtype=torch.float64, device=DEV)
    axes = []
    for x in range(3):
        t = m[:, None] * (r[:, x] / L)[None]
        t = (t - torch.round(t)) * (2 * math.pi)
        axes.append(torch.complex(torch.cos(t), torch.sin(t)))
    axes[0] = axes[0] * q
    ef, wf = 0.0, 0.0
    zt = axes[2].T.contiguous()
    for x in range(M + 1):                      # half space: m_x > 0, or 0 with half the weight
        rho = (axes[0][M + x] * axes[1]) @ zt
        k2 = (2 * math.pi / L) ** 2 * (x * x + m[:, None] ** 2 + m[None] ** 2)
        if x == 0:
            k2[M, M] = 1.0
        e = 2 * (2 * math.pi * lB / V) * torch.exp(-k2 / (4 * a)) / k2 * (rho.real ** 2
                                                                        + rho.imag ** 2)
        if x == 0:
            e[M, M] = 0.0
            e = 0.5 * e
        ef += float(e.sum())
        wf += float((e * (1 - k2 / (2 * a))).sum())
    s = [float(x) for x in _real(p, r, q)[2]]
    Q, Q2 = float(q.sum()), float((q * q).sum())
    bg = -lB * math.pi * Q * Q / (2 * V * a)
    Ef = ef - lB * math.sqrt(a / math.pi) * Q2 + bg
    ke = 0.5 * p["mass"] * float((v * v).sum())
    W = wf + s[2] + s[3] + 3 * bg
    return dict(E_total=Ef + s[0] + s[1], E_fourier=Ef, E_real=s[0], E_lj=s[1], E_kin=ke,
                W_fourier=wf, W_real=s[2], W_lj=s[3], W_bg=3 * bg,
                pressure=(2 * ke + W) / (3 * V), T_kin=2 * ke / (3 * len(q)))


def exact(case, seed):
    pos, vel = _inputs(case, seed)
    if case["kind"] == "host":
        pos, vel = pos.to(DEV), vel.to(DEV)
    pos, vel = pos.double(), vel.double()
    kind, bits, b = case["kind"], case.get("bits", 32), 0
    got = []
    for p in _systems(case, seed):
        x, v0 = pos[b:b + p["n"]], vel[b:b + p["n"], :3]
        r, q = x[:, :3], x[:, 3]
        b += p["n"]
        if kind in ("md", "host"):
            r, v, F = _dynamics(p, r, v0, q, case["steps"], bits)
            zero = torch.zeros_like(q)[:, None]
            got.append((torch.cat([r, q[:, None]], 1), torch.cat([v, zero], 1),
                        torch.cat([F, zero], 1)))
        elif kind == "observables":
            return [_observables(p, r, q, v0)]
        else:
            F, phi, E = _fourier(p, r, q, 0)
            Fr, pr, sums = _real(p, r, q)
            F, phi = F + Fr, phi + pr
            if kind == "energy":
                return {"E": E + sums[0] + sums[1], "gpos": -F, "gq": phi}
            F4 = torch.cat([F, torch.zeros_like(q)[:, None]], 1)
            if bits == 64:
                return {"F": F4, "E": torch.stack([E + sums[0] + sums[1], E, sums[0],
                                                   sums[1]])[None], "phi": phi}
            return {"F": F4}
    pos, vel, F = (torch.cat(t) for t in zip(*got))
    out = {"pos": pos, "vel": vel}
    if kind == "md":
        out["F"] = F if case.get("force") else None
    return out

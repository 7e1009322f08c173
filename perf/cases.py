"""The work a user has this library do, as cases that can be timed and checked.

A case is one pass through the public entry points of ``paper_1907_10514_gb300`` on a
handle that the user's program keeps: evolve a simulation and read its state back,
advance a batch, evaluate forces into the caller's device memory, minimise, build the
normal-mode Hessian, or evolve with records.  Sizes, traps and clouds are those of the
library's own workloads (64 Ca+ in a cube, a few hundred ions with laser cooling, the
4096-ion two-species cloud, the 32768-ion crystal, 512 uneven ensembles) and sizes between
and around them, most of them odd.

``exact`` evaluates the same passes in plain float64 torch, with nothing of the library.
"""
import math

import numpy as np
import torch

import paper_1907_10514_gb300 as it

# CODATA 2018, as the library's header states its units (amu, e)
E, KB, EPS0, AMU = 1.602176634e-19, 1.380649e-23, 8.8541878128e-12, 1.66053906660e-27
KE2 = E * E / (4.0 * math.pi * EPS0)
CA, NH3 = (39.96, 1.0), (17.03, 1.0)
OMEGA = 2.0 * math.pi * 3.85e6
DT = 2.0 * math.pi / OMEGA / 20.0


def listed():
    return [
        # a small cloud (the 64-ion workload): ten RF periods between two looks at the state; latency only
        {"name": "evolve_n64", "kind": "evolve", "cloud": "cube", "n": 64, "steps": 200, "mixed": False, "laser": False, "fp64": False},
        # sympathetic cooling: two species with a bath each, one of them laser-cooled
        {"name": "evolve_n321_laser", "kind": "evolve", "cloud": "gauss", "n": 321, "steps": 200, "mixed": True, "laser": True, "fp64": False},
        # an ordinary single simulation of the size that the serving stream sends most of
        {"name": "evolve_n1500", "kind": "evolve", "cloud": "gauss", "n": 1500, "steps": 100, "mixed": False, "laser": False, "fp64": False},
        # the headline workload: 3072 Ca+ and 1024 NH3+ in a 100 um cloud
        {"name": "evolve_n4096_mix", "kind": "evolve", "cloud": "mix", "n": 4096, "steps": 100, "mixed": True, "laser": False, "fp64": False},
        # a crystal between the headline's size and the largest
        {"name": "evolve_n9001_crystal", "kind": "evolve", "cloud": "crystal", "n": 9001, "steps": 15, "mixed": False, "laser": False, "fp64": False},
        # the crystal workload, a few steps of it
        {"name": "evolve_n32768_crystal", "kind": "evolve", "cloud": "crystal", "n": 32768, "steps": 15, "mixed": False, "laser": False, "fp64": False},
        # the plain FP64 form, for runs whose trajectories have to be reproduced to the last digits
        {"name": "evolve_n2500_fp64", "kind": "evolve", "cloud": "gauss", "n": 2500, "steps": 10, "mixed": True, "laser": False, "fp64": True},
        # 512 uneven ensembles advanced together
        {"name": "batched_512", "kind": "batched", "count": 512, "steps": 100},
        # forces for a host program that owns its device memory and integrates by itself
        {"name": "forces_n5000", "kind": "forces", "n": 5000, "mixed": True},
        # relaxation of a new cloud in the pseudopotential
        {"name": "minimize_n200", "kind": "minimize", "n": 200, "iters": 200, "mixed": True},
        # normal modes of a crystal
        {"name": "hessian_n300", "kind": "hessian", "n": 300, "mixed": True},
        # dump and timeAvg: positions, velocities and the secular velocity once per RF period
        {"name": "record_n1000", "kind": "record", "cloud": "mix", "n": 1000, "records": 6, "every": 20, "mixed": True},
    ]


def _size(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["small", "small", "large", "fp64", "batched", "forces", "minimize", "hessian", "record"])
    mixed = rng.random() < 0.5
    if kind == "small":  # every single simulation below the crystals
        n = _size(rng, 16, 7000)
        return {"kind": "evolve", "cloud": rng.choice(["gauss", "gauss", "cube" if n <= 512 else "mix"]), "n": n, "steps": 200 if n < 100 else 100, "mixed": mixed,
                "laser": rng.random() < 0.3, "fp64": False}
    if kind == "large":
        return {"kind": "evolve", "cloud": "crystal", "n": _size(rng, 7001, 32768), "steps": 15, "mixed": False, "laser": False, "fp64": False}
    if kind == "fp64":
        return {"kind": "evolve", "cloud": "gauss", "n": _size(rng, 32, 4096), "steps": 10, "mixed": mixed, "laser": rng.random() < 0.3, "fp64": True}
    if kind == "batched":
        return {"kind": "batched", "count": _size(rng, 24, 500), "steps": 100}
    if kind == "forces":
        return {"kind": "forces", "n": _size(rng, 64, 8192), "mixed": mixed}
    if kind == "minimize":
        return {"kind": "minimize", "n": _size(rng, 20, 2000), "iters": 200, "mixed": mixed}
    if kind == "hessian":
        return {"kind": "hessian", "n": _size(rng, 24, 800), "mixed": mixed}
    return {"kind": "record", "cloud": "mix", "n": _size(rng, 50, 4000), "records": rng.randint(2, 6), "every": rng.choice([20, 25, 40]), "mixed": mixed}


# ------------------------------------------------------------------ inputs

def _spaced(fill, group, rng, dmin=1e-6):
    """Positions (m, 3) from fill(rng, indices); of two ions of one group closer than
    dmin the later one is drawn again until no such pair is left."""
    m = len(group)
    pts = fill(rng, np.arange(m))
    order_off = [(a, b, c) for a in (-1, 0, 1) for b in (-1, 0, 1) for c in (-1, 0, 1) if (a, b, c) >= (0, 0, 0)]
    for _ in range(1000):
        cell = np.floor(pts / dmin).astype(np.int64)
        cell -= cell.min(axis=0) - 1
        dim = cell.max(axis=0) + 2
        key = ((group.astype(np.int64) * dim[0] + cell[:, 0]) * dim[1] + cell[:, 1]) * dim[2] + cell[:, 2]
        order = np.argsort(key, kind="stable")
        sk = key[order]
        bad = []
        for a, b, c in order_off:
            want = key + (a * dim[1] + b) * dim[2] + c
            lo, hi = np.searchsorted(sk, want, "left"), np.searchsorted(sk, want, "right")
            k = 0
            while True:
                i = np.nonzero(lo + k < hi)[0]
                if not len(i):
                    break
                j = order[lo[i] + k]
                near = (i != j) & (((pts[i] - pts[j]) ** 2).sum(axis=1) < dmin * dmin)
                bad.append(np.maximum(i[near], j[near]))
                k += 1
        bad = np.unique(np.concatenate(bad)) if bad else np.zeros(0, np.int64)
        if not len(bad):
            return pts
        pts[bad] = fill(rng, bad)
    raise RuntimeError("no room for the ions")


def _cloud(case, n, rng):
    kind = case.get("cloud", "gauss")
    if kind == "cube":  # 50 um cube at 64 ions, the same density at other sizes
        side = 50e-6 * (n / 64.0) ** (1.0 / 3.0)
        fill = lambda r, i: r.uniform(-side / 2, side / 2, (len(i), 3))  # noqa: E731
    elif kind == "crystal":  # uniform prolate spheroid, 400 x 400 x 1200 um at 32768 ions
        f = (n / 32768.0) ** (1.0 / 3.0)

        def fill(r, i):
            d = r.normal(size=(len(i), 3))
            d /= np.linalg.norm(d, axis=1, keepdims=True)
            return d * r.uniform(size=(len(i), 1)) ** (1.0 / 3.0) * np.array([400e-6 * f, 400e-6 * f, 1.2e-3 * f])
    else:  # Gaussian: 100 um at 4096 ions ("mix"), else 30 um and, above 2048 ions, that density
        sigma = 100e-6 * (n / 4096.0) ** (1.0 / 3.0) if kind == "mix" else 30e-6 * max(1.0, (n / 2048.0) ** (1.0 / 3.0))
        fill = lambda r, i: r.normal(0.0, sigma, (len(i), 3))  # noqa: E731
    return np.ascontiguousarray(_spaced(fill, np.zeros(n, np.int64), rng).T)


def _single(case, seed):
    """Species, labels, positions, velocities, trap and cooling of a one-simulation case."""
    n = case["n"]
    rng = np.random.default_rng([seed, n, 5])
    species = [CA, NH3] if case["mixed"] else [CA]
    sp = np.zeros(n, np.uint8)
    if case["mixed"]:
        sp[n - n // (4 if case.get("cloud") == "mix" else 5):] = 1
    x = _cloud(case, n, rng)
    v = np.zeros((3, n))
    if case.get("cloud") == "mix":  # 10 mK
        v = rng.normal(size=(3, n)) * np.sqrt(KB * 10e-3 / np.array([species[s][0] * AMU for s in sp]))[None, :]
    crystal = case.get("cloud") == "crystal"
    trap = {"Omega": OMEGA, "a": -0.001 if case.get("cloud") == "mix" else 0.0, "q": 0.2 if crystal else 0.3,
            "omega_z": 2.0 * math.pi * (0.05e6 if crystal else 0.2e6), "gamma": 2e5 if crystal else 1e5, "T_bath": 1e-3, "dt": DT,
            "seed": int(rng.integers(1 << 40)), "flags": it.IONTRAP_PSEUDO if case["kind"] in ("minimize", "hessian") else 0}
    cooling = None
    if case.get("laser"):  # species 0 laser-cooled along an oblique beam, without a bath; the other in a bath
        cooling = [(0.0, 0.0, (8e4, 5e4, 3e4)), (1e5, 2e-3, (0.0, 0.0, 0.0))][: len(species)]
    return species, sp, x, v, trap, cooling


def _batch(case, seed):
    """Sizes, traps and positions of uneven single-species ensembles, N log-uniform in [16, 2048]."""
    sizes = np.round(np.exp(np.random.default_rng(case["count"]).uniform(math.log(16), math.log(2048), case["count"]))).astype(int)
    rng = np.random.default_rng([seed, case["count"], 6])
    group = np.repeat(np.arange(len(sizes)), sizes)
    pts = _spaced(lambda r, i: r.normal(0.0, 30e-6, (len(i), 3)), group, rng)
    out, at = [], 0
    for n in sizes:
        trap = {"Omega": OMEGA, "a": rng.uniform(-0.005, 0.0), "q": rng.uniform(0.2, 0.4), "omega_z": 2.0 * math.pi * rng.uniform(0.1e6, 0.25e6),
                "gamma": 1e5, "T_bath": 1e-3, "dt": DT, "seed": int(rng.integers(1 << 40)), "flags": 0}
        out.append(([CA], np.zeros(n, np.uint8), np.ascontiguousarray(pts[at:at + n].T), np.zeros((3, n)), trap, None))
        at += n
    return out


def _simulation(inputs, fp64=False, stream=None):
    species, sp, x, v, trap, cooling = inputs
    p = it.make_params(precision=it.IONTRAP_PREC_FP64 if fp64 else it.IONTRAP_PREC_FP32, **trap)
    sim = it.Simulation(species, sp, x, v, p, stream=stream)
    if cooling is not None:
        sim.set_params(p, cooling)
    return sim


def prepare(case, seed):
    kind = case["kind"]
    if kind == "batched":
        stream = torch.cuda.Stream()
        sims = [_simulation(i, stream=stream) for i in _batch(case, seed)]
        return {"case": case, "stream": stream, "sims": sims, "steps": [case["steps"]] * len(sims)}
    inputs = _single(case, seed)
    state = {"case": case}
    if kind == "forces":
        state["species"] = inputs[0]
        state["sp"], state["x"] = torch.from_numpy(inputs[1]).cuda(), torch.from_numpy(inputs[2]).cuda()
        return state
    state["sim"] = _simulation(inputs, case.get("fp64", False))
    if kind == "minimize":
        state["x"], state["zero"] = inputs[2], np.zeros((3, case["n"]))
    if kind == "record":
        state["out"] = torch.empty((case["records"], 3, 3, case["n"]), dtype=torch.float64, device="cuda")
    return state


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "evolve":
        x, v, step, _ = state["sim"].step(case["steps"]).state()
        return {"x": x, "v": v, "step": step}
    if kind == "batched":
        it.iontrap_step_many([s.handle for s in state["sims"]], state["steps"])
        got = [s.state() for s in state["sims"]]
        return {"x": np.concatenate([g[0] for g in got], axis=1), "v": np.concatenate([g[1] for g in got], axis=1)}
    if kind == "forces":
        acc = torch.empty_like(state["x"])
        it.iontrap_forces_noalloc(state["species"], state["sp"].data_ptr(), state["x"].data_ptr(), case["n"], acc.data_ptr())
        return acc
    sim = state["sim"]
    if kind == "minimize":  # the next cloud of a series, relaxed on the handle that is there
        sim.restore(state["x"], state["zero"], state["zero"], 0)
        iters, fnorm = sim.minimize(case["iters"], 5e-7, 0.0, 5e-8)
        return {"iters": iters, "fnorm": fnorm, "x": sim.state()[0]}
    if kind == "hessian":
        return sim.hessian()
    sim.step_record(case["records"] * case["every"], case["every"], it.IONTRAP_REC_X | it.IONTRAP_REC_V | it.IONTRAP_REC_VAVG, 20, state["out"].data_ptr())
    return {"x": state["out"][:, 0], "v": state["out"][:, 1], "v_avg": state["out"][:, 2]}


def work(case):
    kind = case["kind"]
    n = case.get("n", 0)
    # an unordered pair of ions: the difference, r^2, r^-3 and both ions' sums; the Verlet
    # step of an ion: two kicks, a drift, trap, drag and noise
    pairs = lambda m: 23.0 * m * (m - 1) / 2.0 + 60.0 * m  # noqa: E731
    if kind == "evolve":
        return {"bytes": 121.0 * n, "flops": case["steps"] * pairs(n)}
    if kind == "batched":
        # N log-uniform in [16, 2048]: means of n and n^2
        L = math.log(2048 / 16)
        m1, m2 = (2048 - 16) / L, (2048 ** 2 - 16 ** 2) / (2 * L)
        return {"bytes": 121.0 * case["count"] * m1, "flops": case["count"] * case["steps"] * (11.5 * m2 + 48.5 * m1)}
    if kind == "forces":
        return {"bytes": 49.0 * n, "flops": pairs(n)}
    if kind == "minimize":
        return {"bytes": 121.0 * n, "flops": (case["iters"] + 1) * pairs(n)}
    if kind == "hessian":
        return {"bytes": 72.0 * n * n + 25.0 * n, "flops": 20.0 * n * (n - 1)}
    return {"bytes": 121.0 * n + 72.0 * n * case["records"], "flops": case["records"] * case["every"] * pairs(n)}


# ------------------------------------------------------------------ the same in float64

def _dev():
    return torch.device("cuda" if torch.cuda.is_available() else "cpu")


def _coulomb(x, w):
    """sum_j w_j (x_i - x_j) / r^3 for x (g, 3, n), w (g, n) with zeros for padding."""
    g, _, n = x.shape
    out = torch.empty_like(x)
    step = max(1, (1 << 25) // (g * n))
    j = torch.arange(n, device=x.device)
    for i0 in range(0, n, step):
        i1 = min(n, i0 + step)
        d = [x[:, c, i0:i1, None] - x[:, c, None, :] for c in range(3)]
        r2 = d[0] * d[0] + d[1] * d[1] + d[2] * d[2]
        r2.masked_fill_((j[i0:i1, None] == j[None, :])[None] | (w == 0)[:, None, :], math.inf)
        s = w[:, None, :] / (r2 * r2.sqrt())
        for c in range(3):
            out[:, c, i0:i1] = (s * d[c]).sum(dim=2)
    return out


def _mulhilo(a, b):
    """High and low 64 bits of the unsigned product of int64 tensors a and the constant b."""
    m32 = 0xFFFFFFFF
    b1, b0 = (b >> 32) & m32, b & m32
    a1, a0 = (a >> 32) & m32, a & m32
    t = a0 * b0
    u = a1 * b0 + ((t >> 32) & m32)  # below 2^64: the sum wraps in int64 as it would unsigned
    v = a0 * b1 + (u & m32)
    hi = a1 * b1 + ((u >> 32) & m32) + ((v >> 32) & m32)
    bs = b - (1 << 64) if b >= (1 << 63) else b
    return hi, a * bs


def _normals(seed, counter, ids):
    """Three standard normals (Philox-4x64-10, key (seed, 0), counter (counter, id, 0, 0); Box-Muller)
    for int64 tensors seed, counter and ids of one shape."""
    sgn = lambda k: k - (1 << 64) if k >= (1 << 63) else k  # noqa: E731
    c = [counter.clone(), ids.clone(), torch.zeros_like(ids), torch.zeros_like(ids)]
    k0, k1 = seed.clone(), torch.zeros_like(seed)
    for _ in range(10):
        h0, l0 = _mulhilo(c[0], 0xD2E7470EE14C6C93)
        h1, l1 = _mulhilo(c[2], 0xCA5A826395121157)
        c = [h1 ^ c[1] ^ k0, l1, h0 ^ c[3] ^ k1, l0]
        k0, k1 = k0 + sgn(0x9E3779B97F4A7C15), k1 + sgn(0xBB67AE8584CAA73B)
    u = [(((q >> 41) & ((1 << 23) - 1)).double() + 0.5) * 2.0 ** -23 for q in c]
    r1, r2 = torch.sqrt(-2.0 * torch.log(u[0])), torch.sqrt(-2.0 * torch.log(u[2]))
    return torch.stack([r1 * torch.cos(2 * math.pi * u[1]), r1 * torch.sin(2 * math.pi * u[1]), r2 * torch.cos(2 * math.pi * u[3])], dim=1)


class _Systems:
    """Systems of unequal sizes padded to one: (g, 3, n) states advanced in float64."""

    def __init__(self, systems):
        dev = _dev()
        self.sizes = [len(s[1]) for s in systems]
        g, n = len(systems), max(self.sizes)
        a = {k: np.zeros((g, n)) for k in ("w", "M", "rho", "gamma", "sigma", "lrate")}
        a["M"][:] = 1.0
        x, v, kdir = np.zeros((g, 3, n)), np.zeros((g, 3, n)), np.zeros((g, 3, n))
        trap = {k: np.zeros((g, 1)) for k in ("a", "q", "wz")}
        seeds = np.zeros((g, n), np.int64)
        for e, (species, sp, x0, v0, t, cooling) in enumerate(systems):
            m = len(sp)
            x[e, :, :m], v[e, :, :m] = x0, v0
            mass, z = np.array([s[0] for s in species])[sp], np.array([s[1] for s in species])[sp]
            a["M"][e, :m], a["w"][e, :m] = mass * AMU, z
            a["rho"][e, :m] = (z / mass) / (species[0][1] / species[0][0])
            cool = cooling or [(t["gamma"], t["T_bath"], (0.0, 0.0, 0.0))] * len(species)
            for s, (gam, T, L) in enumerate(cool):
                on = np.nonzero(sp == s)[0]
                a["gamma"][e, on] = gam
                a["sigma"][e, on] = np.sqrt(2.0 * gam * KB * T / (a["M"][e, on] * t["dt"]))
                ln = math.sqrt(sum(q * q for q in L))
                a["lrate"][e, on] = ln
                for c in range(3):
                    kdir[e, c, on] = L[c] / ln if ln else 0.0
            trap["a"][e], trap["q"][e], trap["wz"][e] = t["a"], t["q"], t["omega_z"]
            seeds[e] = t["seed"]
        to = lambda q: torch.from_numpy(q).to(dev)  # noqa: E731
        self.__dict__.update({k: to(q) for k, q in a.items()}, x=to(x), v=to(v), kdir=to(kdir), seeds=to(seeds), **{k: to(q) for k, q in trap.items()})
        self.ids = torch.arange(n, device=dev).expand(g, n)
        self.ke = KE2 * self.w / self.M
        self.step = 0

    def acceleration(self, x, v, step):
        c = math.cos(OMEGA * (step * DT))
        q4, wz2 = OMEGA * OMEGA / 4.0 * self.rho, self.rho * self.wz * self.wz
        k = torch.stack([q4 * (self.a - 2.0 * self.q * c) - 0.5 * wz2, q4 * (self.a + 2.0 * self.q * c) - 0.5 * wz2, wz2], dim=1)
        xi = _normals(self.seeds, torch.full_like(self.ids, step), self.ids)
        lp = self.lrate * (self.kdir * v).sum(dim=1)
        return (self.ke[:, None] * _coulomb(x, self.w) - k * x - self.gamma[:, None] * v + self.sigma[:, None] * xi - lp[:, None] * self.kdir)

    def start(self):
        self.acc = self.acceleration(self.x, self.v, 0)
        return self

    def advance(self, steps):
        for _ in range(steps):
            vh = self.v + 0.5 * DT * self.acc
            self.x = self.x + DT * vh
            self.step += 1
            self.acc = self.acceleration(self.x, vh, self.step)
            self.v = vh + 0.5 * DT * self.acc


def _springs(trap, rho):
    wz2 = rho * trap["omega_z"] ** 2
    kr = OMEGA ** 2 / 4.0 * (rho * trap["a"] - 2.0 * wz2 / OMEGA ** 2 + 0.5 * (rho * trap["q"]) ** 2)
    return np.stack([kr, kr, wz2])


def exact(case, seed):
    kind = case["kind"]
    dev = _dev()
    if kind == "batched":
        systems = _batch(case, seed)
        order = sorted(range(len(systems)), key=lambda e: len(systems[e][1]))
        got = [None] * len(systems)
        for k in range(0, len(order), 16):
            some = order[k:k + 16]
            S = _Systems([systems[e] for e in some]).start()
            S.advance(case["steps"])
            x, v = S.x.cpu().numpy(), S.v.cpu().numpy()
            for r, e in enumerate(some):
                m = S.sizes[r]
                got[e] = (x[r, :, :m], v[r, :, :m])
        return {"x": np.concatenate([q[0] for q in got], axis=1), "v": np.concatenate([q[1] for q in got], axis=1)}
    inputs = _single(case, seed)
    species, sp, x0, v0, trap, _ = inputs
    mass, z = np.array([s[0] for s in species])[sp], np.array([s[1] for s in species])[sp]
    M, rho = mass * AMU, (z / mass) / (species[0][1] / species[0][0])
    to = lambda q: torch.from_numpy(np.ascontiguousarray(q)).to(dev)  # noqa: E731
    if kind == "evolve":
        S = _Systems([inputs]).start()
        S.advance(case["steps"])
        return {"x": S.x[0].cpu().numpy(), "v": S.v[0].cpu().numpy(), "step": None}
    if kind == "forces":
        return to(KE2 * z / M) * _coulomb(to(x0)[None], to(z)[None])[0]
    if kind == "hessian":
        x, n = to(x0), case["n"]
        d = x[:, :, None] - x[:, None, :]
        r2 = (d * d).sum(dim=0)
        r2.fill_diagonal_(math.inf)
        r3, r5 = r2 ** 1.5, r2 ** 2.5
        kq = KE2 * to(z)[:, None] * to(z)[None, :]
        H = torch.zeros((n, 3, n, 3), dtype=torch.float64, device=dev)
        k = _springs(trap, rho)
        for a in range(3):
            for b in range(3):
                h = kq * ((1.0 if a == b else 0.0) / r3 - 3.0 * d[a] * d[b] / r5)
                h.diagonal().copy_(-h.sum(dim=1) + (to(M * k[a]) if a == b else 0.0))
                H[:, a, :, b] = h
        w = to(M ** -0.5).repeat_interleave(3)
        return (H.reshape(3 * n, 3 * n) * w[:, None] * w[None, :]).cpu().numpy()
    if kind == "minimize":
        x, v, k, m, zz = to(x0), to(np.zeros_like(x0)), to(_springs(trap, rho)), to(M), to(z)
        dt, dmax = 5e-8, 5e-7

        def force(x):
            a = KE2 * zz / m * _coulomb(x[None], zz[None])[0] - k * x
            return a, m * a
        for _ in range(case["iters"]):
            a, F = force(x)
            vF, FF = (v * F).sum(), (F * F).sum()
            v = torch.where(vF > 0, vF / FF, torch.zeros_like(vF)) * F + dt * a
            d = dt * v
            s = torch.clamp(dmax / (d * d).sum(dim=0).sqrt().max(), max=1.0)
            x, v = x + s * d, s * v
        F = force(x)[1]
        return {"iters": None, "fnorm": float((F * F).sum().sqrt()), "x": x.cpu().numpy()}
    S = _Systems([inputs]).start()
    out = torch.empty((case["records"], 3, 3, case["n"]), dtype=torch.float64, device=dev)
    for r in range(case["records"]):
        S.advance(case["every"] - 20)
        mean = torch.zeros_like(S.v)
        for _ in range(20):
            S.advance(1)
            mean += S.v / 20.0
        out[r, 0], out[r, 1], out[r, 2] = S.x[0], S.v[0], mean[0]
    return {"x": out[:, 0], "v": out[:, 1], "v_avg": out[:, 2]}

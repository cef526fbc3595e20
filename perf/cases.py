"""The work that a user of this library has it do, as measurable cases.

Every case starts from a Lennard-Jones liquid at density 0.8442 (a short melt
of the FCC lattice made here, in plain torch, from the seed), and goes through
the package's public calls.  Results of the mixed-precision path, whose pair
forces are single precision, are kept in single precision (frames and logs as
trajectory files hold them); FP64 results stay in double precision.

The free-running calls (`run_free`, `advance_async`) are not among the cases:
how many steps a replica makes there is decided at run time, so two runs of
the same inputs differ.  They run the same kernel as the others.
"""
from __future__ import annotations

import math

import numpy as np
import torch

RHO = 0.8442
RC = 2.5
DT = 0.005
TAU = 0.5
SIZES = (256, 500, 864, 1372, 2048, 2916, 4000)  # atoms of FCC boxes whose half side exceeds the list radius


def listed():
    return [
        # one attempt over a ladder gathered from several contexts (the sharded ladder's
        # decision on every rank): the smallest call, all latency
        {"name": "decide 64", "kind": "decide", "replicas": 64, "lam": False, "distance": 1},
        # the same for a long ladder of parameter sets (T, lam), non-nearest pairs
        {"name": "decide 1000 lam", "kind": "decide", "replicas": 1000, "lam": True, "distance": 2},
        # forces of one configuration on device tensors: a small box with an odd atom count,
        # and a box of the largest size the batched path is used for
        {"name": "forces 987 mixed", "kind": "forces", "atoms": 987, "precision": "mixed", "alloc": True},
        {"name": "forces 4000 fp64", "kind": "forces", "atoms": 4000, "precision": "fp64", "alloc": True},
        # the same from inside another framework's memory pool
        {"name": "forces 2048 noalloc", "kind": "forces", "atoms": 2048, "precision": "fp64", "alloc": False},
        # the plain method in FP64: 8 replicas of 256 atoms, an attempt every 100 steps, the
        # frame and the energies read at the attempt
        {"name": "fp64 8x256", "kind": "cycle", "atoms": 256, "replicas": 8, "steps": 100,
         "skin": 0.5, "t_min": 0.8, "t_max": 1.6, "precision": "fp64", "frame": True},
        # the short-stride ladder: 64 replicas of 864 atoms, an attempt every 10 steps
        {"name": "cycle 64x864", "kind": "cycle", "atoms": 864, "replicas": 64, "steps": 10,
         "skin": 0.3, "t_min": 0.7, "t_max": 2.0, "precision": "mixed", "frame": False},
        # an odd ladder of the default skin, whose frame is written after the attempt
        {"name": "frame 37x1372", "kind": "cycle", "atoms": 1372, "replicas": 37, "steps": 7,
         "skin": 0.5, "t_min": 0.7, "t_max": 2.0, "precision": "mixed", "frame": True},
        # the logged run with asynchronous budgets: every replica its own number of steps
        # between attempts, the record of every attempt read back
        {"name": "record 48x500", "kind": "record", "atoms": 500, "replicas": 48, "cycles": 2,
         "lo": 2, "hi": 18, "skin": 0.4, "t_min": 0.7, "t_max": 2.0, "precision": "mixed"},
        # five ensembles of uneven sizes advanced together, budgets 5..50
        {"name": "uneven group", "kind": "group", "scale": 16, "lo": 5, "hi": 50, "skin": 0.4,
         "t_min": 0.7, "t_max": 2.5, "precision": "mixed"},
        # large replicas, an attempt every 5 steps
        {"name": "cycle 256x4000", "kind": "cycle", "atoms": 4000, "replicas": 256, "steps": 5,
         "skin": 0.5, "t_min": 0.75, "t_max": 1.8, "precision": "mixed", "frame": False},
        # the long ladder with an attempt after every step, cycles replayed as one graph
        {"name": "run 1024x2048", "kind": "run", "atoms": 2048, "replicas": 1024, "cycles": 4,
         "skin": 0.5, "t_min": 0.7, "t_max": 3.0, "precision": "mixed"},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["decide", "forces", "cycle", "cycle", "cycle", "record", "group", "run"])
    if kind == "decide":
        return {"kind": kind, "replicas": _log_int(rng, 2, 4096), "lam": rng.random() < 0.5,
                "distance": rng.choice([1, 1, 2, 3])}
    if kind == "forces":
        # mixed boxes up to 4000 atoms, FP64 ones the same; below 256 no cells fit
        return {"kind": kind, "atoms": _log_int(rng, 256, 4000),
                "precision": rng.choice(["mixed", "fp64"]), "alloc": True} if rng.random() < 0.7 else \
            {"kind": kind, "atoms": _log_int(rng, 256, 4000), "precision": "fp64", "alloc": False}
    skin = rng.choice([0.3, 0.4, 0.5])
    hot = round(rng.uniform(1.4, 2.6), 2)
    if kind == "group":
        return {"kind": kind, "scale": _log_int(rng, 2, 16), "lo": 5, "hi": rng.randint(6, 30),
                "skin": skin, "t_min": 0.7, "t_max": hot, "precision": "mixed"}
    atoms = rng.choice(SIZES)
    if kind == "run":
        return {"kind": kind, "atoms": atoms, "replicas": _log_int(rng, 2, min(1024, 2097152 // atoms)),
                "cycles": rng.randint(1, 4), "skin": skin, "t_min": 0.7, "t_max": hot,
                "precision": "mixed"}
    if kind == "record":
        return {"kind": kind, "atoms": atoms, "replicas": _log_int(rng, 2, min(200, 200000 // atoms)),
                "cycles": rng.randint(1, 2), "lo": rng.randint(0, 4), "hi": rng.randint(5, 18),
                "skin": skin, "t_min": 0.7, "t_max": hot, "precision": "mixed"}
    if rng.random() < 0.3:
        return {"kind": kind, "atoms": rng.choice(SIZES[:4]), "replicas": _log_int(rng, 1, 24),
                "steps": rng.randint(1, 40), "skin": skin, "t_min": 0.7, "t_max": hot,
                "precision": "fp64", "frame": True}
    return {"kind": kind, "atoms": atoms, "replicas": _log_int(rng, 1, min(300, 400000 // atoms)),
            "steps": rng.randint(1, 12), "skin": skin, "t_min": 0.7, "t_max": hot,
            "precision": "mixed", "frame": rng.random() < 0.3}


# ------------------------------------------------------------------ inputs
def _side(n_box):
    return (n_box / RHO) ** (1.0 / 3.0)


def _box_atoms(n):
    """The smallest 4 k^3 >= n."""
    k = 1
    while 4 * k ** 3 < n:
        k += 1
    return 4 * k ** 3


def _melt(n_box, temps, gen):
    """Liquid configurations (len(temps), n_box, 3) in [0, L), FP64, one per temperature:
    velocity Verlet from the FCC lattice in FP32, all pairs, 0.6 time units at T = 3 and
    then 0.6 at the target temperature by velocity scaling."""
    L = _side(n_box)
    k = round((n_box / 4) ** (1 / 3))
    cell = torch.arange(k ** 3)
    base = torch.stack([cell // (k * k), (cell // k) % k, cell % k], 1)[:, None, :].double()
    basis = torch.tensor([[0, 0, 0], [.5, .5, 0], [0, .5, .5], [.5, 0, .5]]).double()
    x = ((base + basis + 0.25) * (L / k)).reshape(1, n_box, 3).cuda().float()
    S = len(temps)
    x = x.repeat(S, 1, 1).permute(2, 0, 1).contiguous()  # (3, S, N)
    target = torch.tensor(temps, dtype=torch.float32, device="cuda")[None, :, None]
    v = torch.randn(3, S, n_box, generator=gen, device="cuda") * math.sqrt(3.0)

    def force(x):
        d = [c[:, :, None] - c[:, None, :] for c in x]
        for c in d:
            c -= L * torch.round(c / L)
        r2 = d[0] * d[0]
        r2.addcmul_(d[1], d[1]).addcmul_(d[2], d[2])
        near = (r2 < RC * RC) & (r2 > 0)
        s = 1.0 / torch.where(near, r2.clamp_(min=0.5), torch.inf)
        s3 = s * s * s
        fs = (48.0 * s3 - 24.0) * s3 * s
        return torch.stack([(fs * c).sum(2) for c in d])

    f = force(x)
    for step in range(240):
        if step % 8 == 0:
            want = target if step >= 120 else torch.full_like(target, 3.0)
            v = v - v.mean(2, keepdim=True)
            t = (v * v).sum((0, 2), keepdim=True) / (3 * n_box - 3)
            v = v * torch.sqrt(want / t)
        v = v + (0.5 * DT) * f
        x = x + DT * v
        f = force(x)
        v = v + (0.5 * DT) * f
    return torch.remainder(x.permute(1, 2, 0).double(), L)


def _ladder(t_min, t_max, R):
    return t_min * (t_max / t_min) ** (np.arange(R) / max(1, R - 1))


def _ensemble(n, temps, gen):
    """Positions and velocities (R, n, 3), FP64 CUDA tensors: every replica a melted
    configuration of about its temperature, turned, reflected and shifted at random, with
    Maxwell-Boltzmann velocities of zero total momentum."""
    R, L = len(temps), _side(n)
    S = min(R, 3)
    at = np.unique(np.linspace(0, R - 1, S).round().astype(int))
    liquid = _melt(n, [float(temps[a]) for a in at], gen)
    pick = torch.tensor(np.abs(np.log(temps)[:, None] - np.log(temps[at])[None, :]).argmin(1)).cuda()
    axes = torch.rand(R, 3, generator=gen, device="cuda").argsort(1)
    sign = torch.where(torch.rand(R, 1, 3, generator=gen, device="cuda") < 0.5, -1.0, 1.0).double()
    shift = torch.rand(R, 1, 3, generator=gen, device="cuda", dtype=torch.float64) * L
    x = liquid[pick].gather(2, axes[:, None, :].expand(R, n, 3)) * sign + shift
    x = torch.remainder(x, L)
    v = torch.randn(R, n, 3, generator=gen, device="cuda", dtype=torch.float64)
    v -= v.mean(1, keepdim=True)
    v *= torch.sqrt(torch.tensor(temps).cuda())[:, None, None]
    return x, v


def _inputs(case, seed):
    """Everything a case starts from, by the seed alone."""
    gen = torch.Generator(device="cuda").manual_seed(int(seed))
    rng = np.random.default_rng(int(seed))
    kind = case["kind"]
    if kind == "decide":
        R = case["replicas"]
        lam = np.exp(rng.uniform(-0.2, 0.2, R)) if case["lam"] else None
        return {"T": rng.permutation(_ladder(0.7, 3.0, R)), "lam": lam,
                "U": rng.normal(-5000.0, 50.0, R), "attempt": int(rng.integers(0, 1000))}
    if kind == "forces":
        n = case["atoms"]
        n_box = _box_atoms(n)
        x = _melt(n_box, [1.0], gen)[0]
        keep = torch.rand(n_box, generator=gen, device="cuda").argsort()[:n].sort().values
        return {"x": x[keep].contiguous(), "L": _side(n_box)}
    if kind == "group":
        shapes = [(256, 1), (500, 2), (864, 3), (2048, 4), (4000, 6)]
        ens = []
        for n, w in shapes:
            temps = _ladder(case["t_min"], case["t_max"], w * case["scale"])
            ens.append((n, temps) + _ensemble(n, temps, gen))
        R = sum(len(e[1]) for e in ens)
        return {"ens": ens, "budgets": rng.integers(case["lo"], case["hi"] + 1, (1, R), dtype=np.int32)}
    n, R = case["atoms"], case["replicas"]
    temps = _ladder(case["t_min"], case["t_max"], R)
    got = {"ens": [(n, temps) + _ensemble(n, temps, gen)]}
    if kind == "record":
        got["budgets"] = rng.integers(case["lo"], case["hi"] + 1, (case["cycles"], R), dtype=np.int32)
    else:
        steps = case["steps"] if kind == "cycle" else 1
        got["budgets"] = np.full((case.get("cycles", 1), R), steps, np.int32)
    return got


# ------------------------------------------------------------------ the calls
def prepare(case, seed):
    import paper_0812_1633_gb300 as re
    inp = _inputs(case, seed)
    st = {"re": re, "case": case, "seed": int(seed)}
    if case["kind"] == "decide":
        cu = lambda a: None if a is None else torch.tensor(a, device="cuda")
        st.update(T=cu(inp["T"]), lam=cu(inp["lam"]), U=cu(inp["U"]), attempt=inp["attempt"])
        return st
    if case["kind"] == "forces":
        st.update(inp)
        return st
    nx = case["steps"] if case["kind"] == "cycle" else 1
    members = []
    for k, (n, temps, x, v) in enumerate(inp["ens"]):
        ctx = re.Context(n, _side(n), RC, temps, st["seed"] + k, dt=DT, tau=TAU, skin=case["skin"],
                         nx=nx, precision=case["precision"])
        ctx.set_state(x.reshape(-1, 3).cpu().numpy(), v.reshape(-1, 3).cpu().numpy())
        members.append(ctx)
    st["budgets"] = inp["budgets"]
    if case["kind"] == "group":
        st["ctx"] = re.Context.group(members)
        for m in members:
            m.close()
    else:
        st["ctx"] = members[0]
    st["ctx"].sync()
    return st


def _kept(a, case):
    """FP64 results as they are; the mixed path's in single precision."""
    return a.astype(np.float32) if case["precision"] == "mixed" else a


def run(state):
    re, case, kind = state["re"], state["case"], state["case"]["kind"]
    if kind == "decide":
        if state["lam"] is None and case["distance"] == 1:
            T, partner, acc, vs = re.exchange_device(state["T"], state["U"], state["seed"],
                                                     state["attempt"])
            return {"T": T, "partner": partner, "accepted": acc, "vscale": vs}
        T, lam, partner, acc, vs, us = re.exchange_device_h(
            state["T"], state["lam"], state["U"], state["seed"], state["attempt"],
            distance=case["distance"])
        return {"T": T, "lam": lam, "partner": partner, "accepted": acc, "vscale": vs, "uscale": us}
    if kind == "forces":
        if case["alloc"]:
            f, U = re.lj_forces_device(state["x"], state["L"], RC, precision=case["precision"])
        else:
            f, U = re.lj_forces_device_noalloc(state["x"], state["L"], RC)
        return {"f": f.float(), "U": U.float()} if case["precision"] == "mixed" else {"f": f, "U": U}
    ctx = state["ctx"]
    if kind == "record":
        rec = ctx.run_record(case["cycles"], state["budgets"])
        return {k: _kept(a, case) if a.dtype == np.float64 else a for k, a in rec.items()}
    out = {}
    if kind == "run":
        ctx.run(case["cycles"])
    else:
        if kind == "group":
            ctx.advance(state["budgets"][0])
        else:
            ctx.advance()
        out["partner"], out["accepted"] = ctx.exchange(outputs=True)
    out["U"], out["K"], out["H"] = (_kept(a, case) for a in ctx.energies())
    out["T"] = ctx.temps()
    if case.get("frame"):
        out["x"], out["v"] = (_kept(a, case) for a in ctx.get_state())
    return out


# 37 flop per pair inside the cutoff (34 for the pair, 3 for the reaction), 27.3 such
# pairs per atom of this liquid; state of an atom in and out: 3 positions and velocities
PAIRS = 27.3
FLOP_PER_PAIR = 37.0
STATE_BYTES = 48.0


def work(case):
    kind = case["kind"]
    if kind == "decide":
        R = case["replicas"]
        return {"bytes": R * ((24 if case["lam"] else 16) + 21 + (16 if case["lam"] else 0)),
                "flops": 40.0 * R}
    if kind == "forces":
        n = case["atoms"]
        return {"bytes": 48.0 * n, "flops": n * PAIRS * FLOP_PER_PAIR}
    if kind == "group":
        atoms = case["scale"] * (256 + 2 * 500 + 3 * 864 + 4 * 2048 + 6 * 4000)
        steps, passes, reps = 0.5 * (case["lo"] + case["hi"]), 1, 16 * case["scale"]
    else:
        reps = case["replicas"]
        atoms = case["atoms"] * reps
        steps, passes = case.get("steps", 1), 1
        if kind == "record":
            steps, passes = 0.5 * (case["lo"] + case["hi"]), case["cycles"]
        elif kind == "run":
            steps, passes = 1, case["cycles"]
    # the cycles of a pass depend on one another only through the state: read and written once
    return {"bytes": 2 * STATE_BYTES * atoms + (STATE_BYTES * atoms if case.get("frame") else 0) + 37.0 * reps * passes,
            "flops": atoms * steps * passes * PAIRS * FLOP_PER_PAIR}


# ------------------------------------------------------------------ the same in 64 bits
M64 = (1 << 64) - 1


def _mulhi(a, b):
    """High 64 bits of a * b, a a Python int, b a uint64 array."""
    lo32 = np.uint64(0xFFFFFFFF)
    s = np.uint64(32)
    a0, a1 = np.uint64(a & 0xFFFFFFFF), np.uint64(a >> 32)
    b0, b1 = b & lo32, b >> s
    mid = a1 * b0 + (a0 * b0 >> s)
    mid2 = a0 * b1 + (mid & lo32)
    return a1 * b1 + (mid >> s) + (mid2 >> s)


def _uniforms(seed, stream, index, tag, sub):
    """Philox4x64-10 (Salmon et al., SC'11), key (seed, stream), counter (index, tag, sub,
    0): four uniforms (word >> 11) 2^-53 per entry of the array `stream`."""
    stream = np.asarray(stream, np.uint64)
    full = lambda c: np.broadcast_to(np.asarray(c, np.uint64), stream.shape).copy()
    x0, x1, x2, x3 = full(index), full(tag), full(sub), full(0)
    k0, k1 = seed & M64, stream.copy()
    with np.errstate(over="ignore"):
        for r in range(10):
            if r:
                k0 = (k0 + 0x9E3779B97F4A7C15) & M64
                k1 = k1 + np.uint64(0xBB67AE8584CAA73B)
            h0, l0 = _mulhi(0xD2E7470EE14C6C93, x0), np.uint64(0xD2E7470EE14C6C93) * x0
            h1, l1 = _mulhi(0xCA5A826395121157, x2), np.uint64(0xCA5A826395121157) * x2
            x0, x1, x2, x3 = h1 ^ x1 ^ np.uint64(k0), l1, h0 ^ x3 ^ k1, l0
    return [(w >> np.uint64(11)).astype(np.float64) * 2.0 ** -53 for w in (x0, x1, x2, x3)]


def _noise(seed, R, step, nf):
    """R1 ~ N(0, 1) and S ~ chi^2 with nf - 1 degrees of every replica at this step."""
    streams = np.arange(R)
    u = _uniforms(seed, streams, step, 2, 0)
    r1 = np.sqrt(-2 * np.log(1 - u[0])) * np.cos(2 * np.pi * u[1])
    d = 0.5 * (nf - 1) - 1.0 / 3.0
    c = 1.0 / math.sqrt(9 * d)
    s, open_ = np.zeros(R), np.ones(R, bool)
    for t in range(256):
        if not open_.any():
            break
        u = _uniforms(seed, streams, step, 3, t)
        x = np.sqrt(-2 * np.log(1 - u[0])) * np.cos(2 * np.pi * u[1])
        w = 1 + c * x
        v = np.where(w > 0, w, 1.0) ** 3
        ok = (w > 0) & ((u[2] < 1 - 0.0331 * x ** 4) |
                        (np.log(np.maximum(u[2], 1e-300)) < 0.5 * x * x + d * (1 - v + np.log(v))))
        s = np.where(open_ & ok, 2 * d * v, s)
        open_ &= ~ok
    return r1, s


def _attempt(T, lam, U, seed, attempt, distance):
    """One exchange attempt: partner, accepted, T, lam after it."""
    R = len(T)
    order = np.argsort(T / lam, kind="stable")
    u = _uniforms(seed, np.arange(R), attempt, 4, 0)[0]
    partner, acc = np.full(R, -1, np.int32), np.zeros(R, np.uint8)
    Tn, ln = T.copy(), lam.copy()
    o = (attempt & 1) * distance
    for q in range(o, R - distance):
        if (q - o) % (2 * distance) >= distance:
            continue
        a, b = int(order[q]), int(order[q + distance])
        partner[a], partner[b] = b, a
        d = (lam[a] / T[a] - lam[b] / T[b]) * (U[a] / lam[a] - U[b] / lam[b])
        if d >= 0 or u[min(a, b)] < math.exp(d):
            acc[a] = acc[b] = 1
            Tn[a], Tn[b], ln[a], ln[b] = T[b], T[a], lam[b], lam[a]
    return partner, acc, Tn, ln


class _Exact:
    """One ensemble in FP64: all pairs within rc + 0.9 listed at times, forces from the list."""

    def __init__(self, n, temps, x, v, seed, L):
        self.n, self.R, self.L, self.seed = n, len(x), L, seed
        self.T, self.x, self.v = np.array(temps), x.clone(), v.clone()
        self.step, self.attempt = np.zeros(self.R, np.int64), 0
        self.econs, self.ref = np.zeros(self.R), None
        self.vscale = np.ones(self.R)
        self.f, self.U = self.forces()
        self.K = 0.5 * (self.v ** 2).sum((1, 2)).cpu().numpy()

    def image(self, d):
        return d - self.L * torch.round(d / self.L)

    def forces(self):
        if self.ref is None or float(self.image(self.x - self.ref).norm(dim=2).max()) > 0.44:
            self.ref, self.pairs = self.x.clone(), []
            some = max(1, 60_000_000 // (self.n * self.n))
            for r in range(0, self.R, some):
                y = self.x[r:r + some]
                r2 = sum(self.image(y[:, :, None, k] - y[:, None, :, k]) ** 2 for k in range(3))
                near = r2 < (RC + 0.9) ** 2
                near.diagonal(dim1=1, dim2=2).zero_()
                m = int(near.sum(2).max())
                rank, idx = near.to(torch.int8).topk(m, dim=2)
                self.pairs.append((r, r + len(y), idx, rank.bool()))
        f, U = torch.zeros_like(self.x), []
        uc = 4 * (RC ** -12 - RC ** -6)
        for lo, hi, idx, real in self.pairs:
            y = self.x[lo:hi]
            at = idx.reshape(len(y), -1)
            d = [self.image(y[:, :, None, k] - y[:, :, k].gather(1, at).reshape(idx.shape))
                 for k in range(3)]
            r2 = d[0] ** 2 + d[1] ** 2 + d[2] ** 2
            near = real & (r2 < RC * RC)
            s3 = torch.where(near, r2, torch.inf) ** -3
            fs = torch.where(near, (48 * s3 * s3 - 24 * s3) / r2, 0.0)
            for k in range(3):
                f[lo:hi, :, k] = (fs * d[k]).sum(2)
            e = torch.where(near, 4 * (s3 * s3 - s3) - uc, 0.0)
            U.append(0.5 * e.sum((1, 2)))
        return f, torch.cat(U).cpu().numpy()

    def advance(self, budgets):
        nf = 3 * self.n - 3
        c, omc = math.exp(-DT / TAU), -math.expm1(-DT / TAU)
        cu = lambda a: torch.tensor(a, device="cuda")[:, None, None]
        self.v *= cu(self.vscale)
        self.vscale = np.ones(self.R)
        for k in range(int(max(budgets))):
            on = np.asarray(budgets) > k
            g = cu(on.astype(np.float64))
            vh = self.v + 0.5 * DT * self.f
            self.x = self.x + g * DT * vh
            f, U = self.forces()
            vn = vh + 0.5 * DT * f
            K = 0.5 * (vn ** 2).sum((1, 2)).cpu().numpy()
            noise = {}
            r1, s = np.zeros(self.R), np.zeros(self.R)
            for at in np.unique(self.step[on]):
                noise = _noise(self.seed, self.R, at, nf)
                w = on & (self.step == at)
                r1[w], s[w] = noise[0][w], noise[1][w]
            kbar = 0.5 * nf * self.T
            kp = c * K + omc * kbar * (r1 * r1 + s) / nf + 2 * r1 * np.sqrt(c * omc * kbar * K / nf)
            alpha = np.sqrt(kp / K)
            alpha = np.where(r1 + np.sqrt(c * nf * K / (omc * kbar)) < 0, -alpha, alpha)
            self.v = torch.where(g > 0, vn * cu(alpha), self.v)
            self.f = torch.where(g > 0, f, self.f)
            self.econs = np.where(on, self.econs + K - kp, self.econs)
            self.U, self.K = np.where(on, U, self.U), np.where(on, kp, self.K)
            self.step = self.step + on

    def exchange(self):
        one = np.ones(self.R)
        partner, acc, Tn, _ = _attempt(self.T, one, self.U, self.seed, self.attempt, 1)
        self.vscale = np.sqrt(Tn / self.T)
        K = self.K * Tn / self.T
        self.econs, self.K, self.T = self.econs + self.K - K, K, Tn
        self.attempt += 1
        return {"partner": partner, "accepted": acc, "T": self.T, "U": self.U, "K": self.K,
                "H": self.U + self.K + self.econs}

    def frame(self):
        v = self.v * torch.tensor(self.vscale, device="cuda")[:, None, None]
        return (torch.remainder(self.x, self.L).reshape(-1, 3).cpu().numpy(),
                v.reshape(-1, 3).cpu().numpy())


def exact(case, seed):
    inp = _inputs(case, seed)
    kind = case["kind"]
    if kind == "decide":
        T = inp["T"]
        lam = np.ones(len(T)) if inp["lam"] is None else inp["lam"]
        partner, acc, Tn, ln = _attempt(T, lam, inp["U"], int(seed), inp["attempt"], case["distance"])
        out = {"T": Tn, "partner": partner, "accepted": acc, "vscale": np.sqrt(Tn / T)}
        if case["lam"] or case["distance"] != 1:
            out.update(lam=ln, uscale=ln / lam)
        return out
    if kind == "forces":
        x, L = inp["x"][None], inp["L"]
        e = _Exact(x.shape[1], [1.0], x, torch.zeros_like(x), 0, L)
        return {"f": e.f[0], "U": e.U}
    ens = [_Exact(n, temps, x, v, int(seed) + k, _side(n))
           for k, (n, temps, x, v) in enumerate(inp["ens"])]
    del inp["ens"]
    rows = []
    for row in inp["budgets"]:
        at, parts = 0, []
        for e in ens:
            e.advance(row[at:at + e.R])
            at += e.R
            parts.append(e.exchange())
        rows.append({k: np.concatenate([p[k] for p in parts]) for k in parts[0]})
    if kind == "record":
        return {k: np.stack([r[k] for r in rows]) for k in rows[0]}
    out = dict(rows[-1])
    if kind == "run":
        del out["partner"], out["accepted"]
    if case.get("frame"):
        out["x"], out["v"] = ens[0].frame()
    return out

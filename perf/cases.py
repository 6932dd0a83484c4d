"""Timed cases of the library: what a user's program has it do, through its public entry points.

Every case is one call (or one captured step) that such a program makes many
times: lattices of one replica and of batches, at every domain side, with
records, scores and the colour orders in use; rings and small partitioned
lattices as ensembles of trajectories.  Inputs are synthetic and follow from
the seed: per-trajectory seeds, and for batches the sides, temperatures and
fields.  `exact` computes the same trajectories with plain tensor arithmetic.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_1403_4674_gb300 as kmc
from paper_1403_4674_gb300 import autograd, autotune

SCHEDULE = {"palindrome": kmc.KMC_SCHEDULE_PALINDROME, "random": kmc.KMC_SCHEDULE_RANDOM_PERM}
LAW = {"metropolis": kmc.KMC_RATE_METROPOLIS, "barker": kmc.KMC_RATE_BARKER}
CLOCK = {"exponential": kmc.KMC_TIME_EXPONENTIAL, "expected": kmc.KMC_TIME_EXPECTED}


def _lattice(name, L, n, Ld, k, T, sched, **more):
    """n replicas of an L x L lattice in one context; k = 0: the replicas take k in {1, 4, 16} and three temperatures."""
    c = {"name": name, "family": "lattice", "L": L, "n": n, "Ld": Ld, "k": k, "T": T, "h": 0.0, "sched": sched,
         "obs_every": 10, "per_pass": False, "up": False, "law": "metropolis", "clock": "exponential",
         "schedule": "palindrome", "plan": "default"}
    c.update(more)
    return c


def listed():
    return [
        # the smallest call: one sweep of a small lattice and its record, as a program that watches a trajectory makes it
        _lattice("lattice64_one_sweep", 64, 1, 16, 1, 2.5, 1, obs_every=1),
        # a small lattice for a thousand sweeps: a single trajectory for a correlation time
        _lattice("lattice64_k1", 64, 1, 16, 1, 2.5, 1000),
        # one ordinary lattice near the critical point, from the ordered start
        _lattice("lattice1024_k4", 1024, 1, 32, 4, 2.269, 200, up=True),
        # a parameter scan in one launch: three temperatures, two starts, three visit lengths
        _lattice("lattice1024x18_scan", 1024, 18, 32, 0, 0.0, 100, plan="round_robin"),
        # the largest lattice: 67 million sites, with a field
        _lattice("lattice8192_k8", 8192, 1, 64, 8, 2.269, 50, h=0.01),
        # an uneven batch of replicas (sides 32 to 512, own temperatures and fields) as a captured step
        {"name": "batch512_graph", "family": "batch", "n": 512, "L_lo": 32, "L_hi": 512, "Ld": 8, "k": 16, "sched": 60,
         "obs_every": 10},
        # likelihood-ratio gradients of the mean energy: forward and backward through autograd
        {"name": "gradient256x256", "family": "grad", "L": 256, "n": 256, "Ld": 32, "k": 8, "T": 2.4, "h": 0.02,
         "sched": 100, "observable": "e"},
        # the random colour order with the other rate law and clock, a record after every pass
        _lattice("lattice256x16_random_order", 256, 16, 16, 8, 2.6, 40, law="barker", clock="expected",
                 schedule="random", per_pass=True, obs_every=4),
        # the ring experiment: 48000 trajectories of 8 spins, 800 steps, sums over the ensemble after every process
        {"name": "ring8_ensemble", "family": "ring", "N": 8, "n": 48000, "Ld": 2, "k": 5, "sweeps": 40, "beta": 0.5,
         "schedule": "random", "records": False},
        # long rings with a record per trajectory
        {"name": "ring64_records", "family": "ring", "N": 64, "n": 6000, "Ld": 8, "k": 10, "sweeps": 10, "beta": 0.5,
         "schedule": "palindrome", "records": True},
        # the 100 x 100 stripes of the paper's second experiment
        {"name": "stripes100", "family": "part", "L": 100, "n": 50, "blocks": False, "ND": 4, "k": 5, "sweeps": 800,
         "T": 2.4, "schedule": "random", "obs_every": 0},
        # its 12 x 12 blocks with one step per visit
        {"name": "blocks12_k1", "family": "part", "L": 12, "n": 500, "blocks": True, "ND": 4, "k": 1, "sweeps": 4000,
         "T": 2.4, "schedule": "random", "obs_every": 400},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    family = rng.choice(["lattice", "lattice", "lattice", "batch", "grad", "ring", "part", "part"])
    if family == "lattice":
        Ld = rng.choice([8, 16, 16, 32, 32, 64])
        L = 2 * Ld * max(1, _log_int(rng, 64, 1536) // (2 * Ld))
        n = max(1, min(64, int((1 << 23) / (L * L)), _log_int(rng, 1, 64)))
        k = rng.choice([1, 2, 3, 4, 7, 8, 16, 24, 33])
        sites = n * (L // Ld) ** 2 * k
        sched = max(1, min(_log_int(rng, 1, 1000), 4_000_000 // sites, 4000 // k))
        random_order = rng.random() < 0.25
        c = _lattice("", L, n, Ld, k, round(rng.uniform(1.5, 3.5), 3), sched, h=round(rng.uniform(-0.1, 0.1), 3),
                     obs_every=rng.choice([0, 1, 3, 10]), per_pass=rng.random() < 0.2, up=rng.random() < 0.4,
                     law=rng.choice(["metropolis", "metropolis", "barker"]),
                     clock=rng.choice(["exponential", "exponential", "expected"]),
                     schedule="random" if random_order else "palindrome",
                     plan=rng.choice(["default", "default", "round_robin"]) if Ld > 8 and not random_order else "default")
        del c["name"]
        return c
    if family == "batch":
        Ld = rng.choice([8, 8, 16])
        lo = 2 * Ld * rng.randint(1, 3)
        return {"family": "batch", "n": _log_int(rng, 16, 384), "L_lo": lo, "L_hi": lo * rng.randint(2, 6), "Ld": Ld,
                "k": rng.choice([4, 8, 16, 32]), "sched": rng.randint(10, 40), "obs_every": rng.choice([5, 10])}
    if family == "grad":
        Ld = rng.choice([16, 32])
        L = 2 * Ld * rng.randint(1, 4)
        return {"family": "grad", "L": L, "n": max(8, min(128, int((1 << 22) / (L * L)))), "Ld": Ld,
                "k": rng.choice([2, 4, 8, 12]), "T": round(rng.uniform(2.0, 3.0), 3), "h": round(rng.uniform(0.0, 0.05), 3),
                "sched": rng.randint(10, 60), "observable": rng.choice(["e", "m", "em"])}
    if family == "ring":
        Ld = rng.choice([1, 2, 4, 8])
        N = Ld * 2 * rng.randint(1, 32 // Ld)
        k = rng.choice([1, 2, 5, 10])
        return {"family": "ring", "N": N, "n": _log_int(rng, 500, 48000), "Ld": Ld, "k": k,
                "sweeps": max(1, 600 // (k * (N // Ld))), "beta": round(rng.uniform(0.2, 0.9), 3),
                "schedule": rng.choice(["random", "palindrome"]), "records": rng.random() < 0.3}
    blocks = rng.random() < 0.5
    ND = rng.choice([4, 16]) if blocks else rng.choice([2, 4, 6])
    side = (math.isqrt(ND) if blocks else ND)
    L = side * rng.randint(max(2, 12 // side), 128 // side)
    k = rng.choice([1, 2, 5, 10, 20, 40])
    return {"family": "part", "L": L, "n": _log_int(rng, 20, 600), "blocks": blocks, "ND": ND, "k": k,
            "sweeps": max(1, rng.randint(1500, 8000) // (k * ND)), "T": round(rng.uniform(1.8, 3.2), 3),
            "schedule": rng.choice(["random", "random", "palindrome"]), "obs_every": rng.choice([0, 0, 4, 40])}


def _inputs(case, seed):
    """Per replica or trajectory: side, steps per visit, start (1: all up), beta, h, seed."""
    rng = np.random.default_rng(seed)
    n, f = case["n"], case["family"]
    one = {"k": case["k"], "up": 0, "h": case.get("h", 0.0)}
    if f == "batch":
        grid = 2 * case["Ld"]
        # the batch's sides are part of the case: the seed sets what its replicas simulate
        L = np.exp(np.random.default_rng(n).uniform(np.log(case["L_lo"]), np.log(case["L_hi"]), n))
        reps = [dict(one, L=max(grid, int(grid * round(x / grid))), beta=float(1 / t), h=float(h))
                for x, t, h in zip(L, rng.uniform(1.5, 3.5, n), rng.uniform(-0.1, 0.1, n))]
    elif f == "ring":
        # as the experiment has it: all down but one pair of neighbours, the pair's place in turn
        N = case["N"]
        reps = [dict(one, L=N, beta=case["beta"], word=(1 << (i % N)) | (1 << ((i + 1) % N))) for i in range(n)]
    elif f == "lattice" and case["k"] == 0:
        grid = [(k, up, T) for k in (1, 4, 16) for up in (0, 1) for T in (1.5, 2.269, 3.0)]
        reps = [{"L": case["L"], "k": k, "up": up, "beta": 1 / T, "h": 0.0} for k, up, T in (grid[i % 18] for i in range(n))]
    else:
        reps = [dict(one, L=case["L"], beta=1 / case["T"], up=1 if case.get("up") or f == "part" else 0) for _ in range(n)]
    for r, s in zip(reps, rng.integers(1, 2**63 - 1, size=n, dtype=np.int64)):
        r["seed"] = int(s)
    return reps


def prepare(case, seed):
    reps = _inputs(case, seed)
    f, n = case["family"], case["n"]

    def col(key):
        return [r[key] for r in reps]
    if f == "lattice":
        mixed = case["k"] == 0
        lat = kmc.Lattice(col("L"), case["Ld"], reps[0]["k"], col("seed"), init=reps[0]["up"])
        if mixed:
            lat.set_replica_params(k=col("k"), init=col("up"))
        if case["plan"] == "round_robin":
            lat.set_launch(kmc.KMC_LAUNCH_THREADS, 2, 4)
        lat.set_rates(col("beta"), col("h"), law=LAW[case["law"]])
        if case["per_pass"]:
            lat.set_observation(kmc.KMC_OBS_PASS)
        return {"case": case, "lat": lat, "init": kmc.KMC_INIT_PER_REPLICA if mixed else reps[0]["up"]}
    if f == "batch":
        choice = autotune.GroupChoice(list(range(n)), case["Ld"], case["k"], (kmc.KMC_LAUNCH_AUTO, 0, 16), 0.0)
        batch = autotune.Batch(col("L"), col("beta"), col("h"), col("seed"), [choice])
        return {"case": case, "batch": batch, "graph": batch.capture(case["sched"], case["obs_every"])}
    if f == "grad":
        lat = kmc.Lattice(col("L"), case["Ld"], case["k"], col("seed"))
        lat.enable_grad(True)
        beta = torch.tensor(reps[0]["beta"], dtype=torch.float64, device="cuda", requires_grad=True)
        h = torch.tensor(reps[0]["h"], dtype=torch.float64, device="cuda", requires_grad=True)
        return {"case": case, "lat": lat, "beta": beta, "h": h}
    if f == "ring":
        ring = kmc.Ring(case["N"], case["Ld"], case["k"], col("seed"), col("word"))
        ring.set_rates(col("beta"))
        return {"case": case, "ring": ring}
    part = kmc.Partitioned(case["L"], kmc.KMC_PART_BLOCKS if case["blocks"] else kmc.KMC_PART_STRIPES, case["ND"],
                           case["k"], col("seed"))
    part.set_rates(col("beta"))
    return {"case": case, "part": part}


def run(state):
    case = state["case"]
    f = case["family"]
    if f == "lattice":
        lat = state["lat"]
        lat.reset(state["init"])
        obs = lat.run(case["sched"], schedule=SCHEDULE[case["schedule"]], time_mode=CLOCK[case["clock"]],
                      obs_every=case["obs_every"])
        return {"spins": lat.spins, "records": obs}
    if f == "batch":
        state["graph"].replay()
        return {"spins": state["batch"].lattices[0].spins, "records": state["batch"].outs[0]}
    if f == "grad":
        beta, h = state["beta"], state["h"]
        beta.grad = h.grad = None
        value = autograd.expectation(state["lat"], beta, h, case["sched"], observable=case["observable"])
        value.backward()
        return {"spins": state["lat"].spins, "value": value.detach(), "beta_grad": beta.grad, "h_grad": h.grad}
    if f == "ring":
        obs, _, ens = state["ring"].run(case["sweeps"], schedule=SCHEDULE[case["schedule"]], obs_every=_ring_every(case),
                                        records=case["records"], ensemble=not case["records"])
        return {"records": obs, "ensemble": ens}
    # the next ensemble of trajectories from the all-up start (the context's schedule count goes on, so they are new ones)
    part = state["part"]
    part.spins.fill_(1)
    obs = part.run(case["sweeps"], schedule=SCHEDULE[case["schedule"]], obs_every=case["obs_every"])
    return {"spins": part.spins, "records": obs}


def _ring_every(case):
    """Sums after every process; records per trajectory after every sweep."""
    passes = kmc.ring_passes(SCHEDULE[case["schedule"]], case["N"] // case["Ld"])
    return passes if case["records"] else 1


def _steps(case, reps):
    """Uniformised steps of one pass, sites and records of a pass."""
    f = case["family"]
    if f in ("lattice", "batch", "grad"):
        visits = 1 if case.get("schedule") == "random" else 2
        steps = sum(visits * (r["L"] // case["Ld"]) ** 2 * r["k"] for r in reps) * case["sched"]
        sites = sum(r["L"] ** 2 for r in reps)
        units = case["sched"] * ((4 if visits == 1 else 8) if case.get("per_pass") else 1)
        every = case["sched"] if f == "grad" else case["obs_every"]
        return steps, sites, units // every * len(reps) if every else 0
    ND = case["N"] // case["Ld"] if f == "ring" else case["ND"]
    visits = ND * (1 if case["schedule"] == "random" else 2)
    steps = len(reps) * visits * case["k"] * case["sweeps"]
    if f == "ring":
        passes = case["sweeps"] * kmc.ring_passes(SCHEDULE[case["schedule"]], ND)
        return steps, 0, passes // _ring_every(case) * (len(reps) if case["records"] else 1)
    passes = case["sweeps"] * kmc.part_passes(0 if case["blocks"] else 1, SCHEDULE[case["schedule"]], ND)
    return steps, len(reps) * case["L"] ** 2, passes // case["obs_every"] * len(reps) if case["obs_every"] else 0


def work(case):
    """Bytes: the spins and records written, and the spins read where the call starts from the caller's.  Operations:
    a hundred integer ones per uniformised step (a Philox block, the target's comparison, the clock's product)."""
    reps = _inputs(case, 1)
    steps, sites, recs = _steps(case, reps)
    width = (4 + case["N"]) if case["family"] == "ring" and not case["records"] else 4
    reads = sites if case["family"] == "part" else 24 * len(reps)
    return {"bytes": sites + reads + 8 * width * recs, "flops": 100 * steps}


# ---------------------------------------------------------------------------
# The same trajectories in plain tensor arithmetic
# ---------------------------------------------------------------------------
_M32 = 0xFFFFFFFF


def _philox(c, key):
    """Philox4x32-10 of int64 tensors that hold 32-bit words."""
    c, (k0, k1) = list(c), key
    for _ in range(10):
        p0, p1 = c[0] * 0xD2511F53, c[2] * 0xCD9E8D57
        c = [((p1 >> 32) & _M32) ^ c[1] ^ k0, p1 & _M32, ((p0 >> 32) & _M32) ^ c[3] ^ k1, p0 & _M32]
        k0, k1 = (k0 + 0x9E3779B9) & _M32, (k1 + 0xBB67AE85) & _M32
    return c


def _scaled(w0, w1, M):
    """floor((w1 2^32 + w0) M / 2^64) for M <= 2^63."""
    m0, m1 = M & _M32, M >> 32
    hi, lo = (lambda p: (p >> 32) & _M32), (lambda p: p & _M32)
    p00, p01, p10 = w0 * m0, w0 * m1, w1 * m0
    return w1 * m1 + hi(p01) + hi(p10) + ((hi(p00) + lo(p01) + lo(p10)) >> 32)


class _Chain:
    """Replicas as one flat vector of spins (0 or 1), each cut into domains of n_d sites in row-major order."""

    def __init__(self, shapes, dom_w, dom_h, reps, law, dev):
        # shapes: (width, height) of each replica; a height of 1 is a ring
        self.dev, self.reps = dev, reps
        # sites, neighbours and domains of one replica of each shape, moved to where the replica begins
        one = {}
        for w, h in set(shapes):
            at = torch.arange(w * h, device=dev).view(h, w)
            sides = [at.roll(1, 1), at.roll(-1, 1)] + ([at.roll(1, 0), at.roll(-1, 0)] if h > 1 else [])
            dom = at.view(h // dom_h, dom_h, w // dom_w, dom_w).permute(0, 2, 1, 3).reshape(-1, dom_h * dom_w)
            one[w, h] = (torch.stack(sides, -1).view(w * h, -1).to(torch.int32), dom.to(torch.int32))
        sites = torch.tensor([w * h for w, h in shapes], device=dev)
        count = torch.tensor([len(one[x][1]) for x in shapes], device=dev)
        begin = sites.cumsum(0) - sites
        self.off, self.first_dom, self.total = begin.tolist(), (count.cumsum(0) - count).tolist(), int(sites.sum())
        if len(one) == 1:
            (nbr, dom), = one.values()
            move = begin.to(torch.int32).view(-1, 1, 1)
            self.nbr, self.doms = (nbr + move).view(-1, nbr.shape[1]), (dom + move).view(-1, dom.shape[1])
        else:
            self.nbr = torch.cat([one[x][0] + o for x, o in zip(shapes, self.off)])
            self.doms = torch.cat([one[x][1] + o for x, o in zip(shapes, self.off)])
        self.size = sites.double()
        number = torch.arange(len(shapes), device=dev)
        self.rep, self.site_rep = torch.repeat_interleave(number, count), torch.repeat_interleave(number, sites)
        self.local = torch.arange(len(self.doms), device=dev) - torch.tensor(self.first_dom, device=dev)[self.rep]
        self.nd, nn = self.doms.shape[1], self.nbr.shape[1]
        self.P = 63 - (self.nd - 1).bit_length()
        self.ncls, self.nn = 2 * (nn + 1), nn
        A, a, gb, gh = [], [], [], []
        for r in reps:
            for up in (0, 1):
                for q in range(nn + 1):
                    s = 1.0 if up else -1.0
                    dE = 2.0 * s * ((2 * q - nn) + r["h"])
                    x = (1.0 if dE <= 0 else math.exp(-r["beta"] * dE)) if law == "metropolis" else 1.0 / (1.0 + math.exp(r["beta"] * dE))
                    slope = (0.0 if dE <= 0 else 1.0) if law == "metropolis" else 1.0 - x
                    a.append(x)
                    A.append(int(np.rint(math.ldexp(x, self.P))))
                    gb.append(-dE * slope)
                    gh.append(-r["beta"] * 2.0 * s * slope)

        def table(v, t):
            return torch.tensor(v, dtype=t, device=dev).view(len(reps), self.ncls)
        self.A, self.a = table(A, torch.int64), table(a, torch.float64)
        self.gb, self.gh = table(gb, torch.float64), table(gh, torch.float64)
        self.k = torch.tensor([r["k"] for r in reps], device=dev)
        seed = [r["seed"] for r in reps]
        self.key = (torch.tensor([s & _M32 for s in seed], device=dev), torch.tensor([s >> 32 for s in seed], device=dev))
        self.h = torch.tensor([r["h"] for r in reps], dtype=torch.float64, device=dev)
        self.S = torch.zeros(self.total, dtype=torch.uint8, device=dev)
        self.clock = torch.zeros(2, len(reps), dtype=torch.float64, device=dev)  # sum of -ln v and what its rounding lost
        self.steps = torch.zeros(len(reps), dtype=torch.float64, device=dev)
        self.score = torch.zeros(len(self.doms), 2, dtype=torch.float64, device=dev)

    def draws(self, doms, phase):
        """Targets, ln of the clock variates [visits, steps]; doms and phase broadcast to one visit each."""
        rep = self.rep[doms].unsqueeze(-1)
        j = torch.arange(int(self.k.max()), device=self.dev)
        ph = phase.unsqueeze(-1).expand(rep.shape)
        shape = torch.broadcast_shapes(rep.shape, j.shape)
        c = [x.expand(shape) for x in (j, self.local[doms].unsqueeze(-1), ph & _M32, (ph >> 32) & 0xFFFFFF)]
        w = _philox(c, (self.key[0][rep], self.key[1][rep]))
        V = ((((w[3] << 32) | w[2]) >> 11) & ((1 << 53) - 1)) + 1
        return _scaled(w[0], w[1], self.nd << self.P), V.double().mul_(2.0**-53).log_()

    def visit(self, doms, tgt, lnv, scores):
        """One process in each of the domains (none next to another)."""
        rep, sites = self.rep[doms], self.doms[doms].long()
        A, k = self.A[rep], self.k[rep]
        near = self.nbr[sites]
        done = torch.arange(tgt.shape[-1], device=self.dev) < k.unsqueeze(1)
        t = -(lnv * done).sum(1)
        y = torch.zeros_like(self.clock[0]).index_add_(0, rep, t) - self.clock[1]
        z = self.clock[0] + y
        self.clock[1], self.clock[0] = (z - self.clock[0]) - y, z
        self.steps.index_add_(0, rep, k.double())
        for j in range(tgt.shape[-1]):
            s = self.S[sites]
            cls = s * (self.nn + 1) + sum(self.S[near[..., q].long()] for q in range(self.nn))
            n = torch.stack([(cls == c).sum(1) for c in range(self.ncls)], 1)
            W = n * A
            C = W.cumsum(1)
            t = tgt[:, j]
            real = (t < C[:, -1]) & done[:, j]
            c = (t.unsqueeze(1) >= C).sum(1).clamp_(max=self.ncls - 1).unsqueeze(1)
            jj = (t - (C - W).gather(1, c)[:, 0]) // A.gather(1, c)[:, 0]
            rank = (cls == c).cumsum(1, dtype=torch.int32)
            at = (rank <= jj.unsqueeze(1)).sum(1).clamp_(max=self.nd - 1)
            site = sites.gather(1, at.unsqueeze(1))[:, 0]
            if scores:
                free = torch.ldexp(((1 << 62) - C[:, -1] + (1 << 62)).double(), torch.tensor(float(-self.P), device=self.dev))
                for i, g in enumerate((self.gb[rep], self.gh[rep])):
                    null = -(n * self.a[rep] * g).sum(1) / free
                    self.score[doms, i] += torch.where(done[:, j], torch.where(real, g.gather(1, c)[:, 0], null), 0.0)
            self.S[site] ^= real.to(torch.uint8)

    def record(self, expected):
        """{e, m, e m, T} of every replica."""
        s = self.S.long() * 2 - 1
        pairs = s * sum(s[self.nbr[:, q].long()] for q in range(self.nn))
        sums = torch.zeros(2, len(self.reps), dtype=torch.int64, device=self.dev)
        bonds = sums[0].index_add_(0, self.site_rep, pairs) // 2
        mag = sums[1].index_add_(0, self.site_rep, s)
        e = (-bonds.double() - self.h * mag.double()) / self.size
        m = mag.double() / self.size
        t = (self.steps if expected else self.clock[0]) / self.size
        return torch.stack([e, m, e * m, t], 1), bonds, mag


def _colours(chain, shapes, dom_w, dom_h, blocks):
    """Domains of each colour over all replicas."""
    lists, one = None, {}
    for r, (w, h) in enumerate(shapes):
        if (w, h) not in one:
            Dx = w // dom_w
            d = torch.arange(Dx * (h // dom_h), device=chain.dev)
            col = (d % Dx % 2) + 2 * (d // Dx % 2) if blocks else d % 2
            one[w, h] = [d[col == q] for q in range(1 if len(d) == 1 else 4 if blocks else 2)]
        lists = lists or [[] for _ in one[w, h]]
        for q, d in enumerate(one[w, h]):
            lists[q].append(d + chain.first_dom[r])
    return [torch.cat(x) for x in lists]


def _orders(chain, n0, count, ND):
    """Random domain orders of schedules n0 .. n0 + count - 1 of every trajectory: [count, trajectories, ND]."""
    n = torch.arange(n0, n0 + count, device=chain.dev).view(-1, 1, 1)
    i = torch.arange(1, max(ND, 2), device=chain.dev).view(1, 1, -1)
    B = len(chain.reps)
    shape = (count, B, i.shape[-1])
    w = _philox([x.expand(shape) for x in (i, i * 0, n, n * 0 + (2 << 24))], (chain.key[0].view(1, -1, 1), chain.key[1].view(1, -1, 1)))
    order = torch.arange(ND, device=chain.dev).repeat(count, B, 1)
    for q in range(ND - 1, 0, -1):
        # floor(x (q + 1) / 2^64)
        lo, hi = w[0][..., q - 1] * (q + 1), w[1][..., q - 1] * (q + 1)
        to = ((hi + (lo >> 32)) >> 32).unsqueeze(-1)
        a, b = order[..., q:q + 1].clone(), order.gather(-1, to)
        order.scatter_(-1, to, a)
        order[..., q:q + 1] = b
    return order


def exact(case, seed):
    dev = torch.device("cuda")
    f, reps = case["family"], _inputs(case, seed)
    ring = f == "ring"
    if ring:
        shapes, dom_w, dom_h, blocks, slots = [(case["N"], 1)] * len(reps), case["Ld"], 1, False, 64
    elif f == "part":
        L, side = case["L"], math.isqrt(case["ND"]) if case["blocks"] else case["ND"]
        shapes, dom_w, dom_h, blocks, slots = [(L, L)] * len(reps), L // side, (L // side if case["blocks"] else L), case["blocks"], 64
    else:
        shapes, dom_w, dom_h, blocks, slots = [(r["L"], r["L"]) for r in reps], case["Ld"], case["Ld"], True, 8
    law = case.get("law", "barker" if f in ("ring", "part") else "metropolis")
    if f == "lattice" and case["k"] == 0:
        # replicas of one visit length at a time, put back in their order
        out = []
        for k in (1, 4, 16):
            mine = [r for r in reps if r["k"] == k]
            out.append(_exact_lattice(case, mine, shapes[:len(mine)], law, dev))
        return {"spins": torch.cat([o["spins"] for o in out]), "records": torch.cat([o["records"] for o in out], 1)}
    if f in ("lattice", "batch", "grad"):
        return _exact_lattice(case, reps, shapes, law, dev)
    chain = _Chain(shapes, dom_w, dom_h, reps, law, dev)
    B, ND = len(reps), len(chain.doms) // len(reps)
    if ring:
        words = torch.tensor([r["word"] - (1 << 64 if r["word"] >> 63 else 0) for r in reps], device=dev)
        chain.S = ((words.unsqueeze(1) >> torch.arange(case["N"], device=dev)) & 1).to(torch.uint8).reshape(-1)
    else:
        chain.S.fill_(1)
    perm = case["schedule"] == "random"
    lists = None
    if not perm:
        lists = _colours(chain, shapes, dom_w, dom_h, blocks)
        lists = lists + lists[::-1]
    passes = ND if perm else len(lists)
    every = _ring_every(case) if ring else case["obs_every"]
    first = torch.tensor(chain.first_dom, device=dev)
    records, ens, done = [], [], 0
    chunk = max(1, min(case["sweeps"], 2_000_000 // (B * ND * case["k"])))
    for n0 in range(0, case["sweeps"], chunk):
        count = min(chunk, case["sweeps"] - n0)
        if perm:
            order = _orders(chain, n0, count, ND) + first.view(1, -1, 1)
            doms = order.permute(0, 2, 1)
        else:
            doms = torch.stack(lists).unsqueeze(0).expand(count, -1, -1)
        phase = (torch.arange(n0, n0 + count, device=dev) * slots).view(-1, 1, 1) + torch.arange(passes, device=dev).view(1, -1, 1)
        tgt, lnv = chain.draws(doms, phase.expand(doms.shape))
        for i in range(count):
            for p in range(passes):
                chain.visit(doms[i, p], tgt[i, p], lnv[i, p], False)
                done += 1
                if every and done % every == 0:
                    rec, bonds, mag = chain.record(False)
                    records.append(rec)
                    if ring and not case["records"]:
                        up = chain.S.view(B, -1).long().sum(0)
                        ens.append(torch.cat([torch.stack([bonds.sum(), mag.sum(), (bonds * mag).sum(), (mag * mag).sum()]), up]))
    rec = torch.stack(records) if records else None
    if ring:
        return {"records": rec if case["records"] else None, "ensemble": None if case["records"] else torch.stack(ens)}
    return {"spins": (chain.S.to(torch.int8) * 2 - 1).view(B, case["L"], case["L"]), "records": rec}


def _exact_lattice(case, reps, shapes, law, dev):
    Ld = case["Ld"]
    chain = _Chain(shapes, Ld, Ld, reps, law, dev)
    for r, rep in enumerate(reps):
        n = shapes[r][0] ** 2
        if rep["up"]:
            chain.S[chain.off[r]:chain.off[r] + n] = 1
        else:
            b = torch.arange(n // 128, device=dev)
            w = torch.stack(_philox([b & _M32, b >> 32, b * 0, b * 0 + (1 << 24)], (rep["seed"] & _M32, rep["seed"] >> 32)), 1)
            chain.S[chain.off[r]:chain.off[r] + n] = ((w.unsqueeze(2) >> torch.arange(32, device=dev)) & 1).to(torch.uint8).reshape(-1)
    grad, random_order = case["family"] == "grad", case.get("schedule") == "random"
    per_pass, expected = case.get("per_pass", False), case.get("clock") == "expected"
    every = case["sched"] if grad else case["obs_every"]
    lists = torch.stack(_colours(chain, shapes, Ld, Ld, True))
    records, done = [], 0
    first = torch.tensor(chain.first_dom, device=dev)
    for n in range(case["sched"]):
        if random_order:
            # each replica its own order of the four colours: the digits of floor(x 24 / 2^64) in factorial base
            z = torch.zeros(len(reps), dtype=torch.int64, device=dev)
            w = _philox([z, z, z + n, z + (2 << 24)], chain.key)
            idx = ((w[1] * 24 + ((w[0] * 24) >> 32)) >> 32).tolist()
            doms = []
            per = [[] for _ in range(4)]
            for r, x in enumerate(idx):
                pool = [0, 1, 2, 3]
                for p, fac in enumerate((6, 2, 1, 1)):
                    q = pool.pop(x // fac)
                    x %= fac
                    mine = len(lists[q]) // len(reps)
                    per[p].append(lists[q][r * mine:(r + 1) * mine])
            doms = torch.stack([torch.cat(x) for x in per])
        else:
            doms = torch.cat([lists, lists.flip(0)])
        phase = (n * 8 + torch.arange(len(doms), device=dev)).view(-1, 1)
        tgt, lnv = chain.draws(doms, phase.expand(doms.shape))
        for p in range(len(doms)):
            chain.visit(doms[p], tgt[p], lnv[p], grad)
            done += 1
            unit = done if per_pass else done // len(doms) if done % len(doms) == 0 else 0
            if every and unit and unit % every == 0:
                records.append(chain.record(expected)[0])
    spins = chain.S.to(torch.int8) * 2 - 1
    rec = torch.stack(records) if records else None
    if not grad:
        return {"spins": spins, "records": rec}
    score = torch.zeros(len(reps), 2, dtype=torch.float64, device=dev).index_add_(0, chain.rep, chain.score)
    e, m, em = rec[-1, :, 0], rec[-1, :, 1], rec[-1, :, 2]
    v, dh = {"e": (e, -m), "m": (m, m * 0), "em": (em, -m * m)}[case["observable"]]
    g = ((v - v.mean()).unsqueeze(1) * score).sum(0) / (len(reps) - 1)
    return {"spins": spins, "value": v.mean(), "beta_grad": g[0], "h_grad": g[1] + dh.mean()}

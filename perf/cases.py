"""The work that users of this package have it do, as timed cases.

Every case is one call, or a short chain of calls, of the package's public
interface (the REWL, Batch and Server classes, and rewl_run_static of the C
ABI): a density-of-states run in each of its stages (the first rounds at
ln f = 1, the long late stage at a small ln f, the 1/t stage), small and large
lattices, one instance, a few dozen and thousands, jobs served to convergence,
fixed-weight production, a whole short run with its set-up, and the run that
allocates nothing.  Sizes are those of workloads.CONFIGS and of the package's
batched and serving workloads, or lie in their ranges.

A pass advances its run by a fixed number of rounds, as a user's program does
between two reads of the results, and reads the walkers' ln g, histograms,
energies and configurations back to the host.
"""
import ctypes as C

import numpy as np
import torch

from paper_1312_3004_gb300 import REWL, Batch, Server, _lib, workloads


# ---- the cases --------------------------------------------------------------
def _instance(name, kind, rounds, config, **more):
    p = workloads.CONFIGS[config]
    case = dict(name=name, kind=kind, q=p["q"], L=p["L"], h=p["h"], m=p["m"], K=p["exchange_interval"],
                lnf_final=p["lnf_final"], bits=p["spin_bits"], rounds=rounds)
    case.update(more)
    return case


def listed():
    return [
        # the smallest run: 2D Ising, 8 walkers; nothing but each walker's own chain
        # of steps (ln f_final lower than the test configuration's, so that a long
        # series of passes does not reach the end of the run)
        _instance("ising_L8", "run", 8, "ising_L8", lnf_final=1e-12),
        # the 10-state model on a small lattice: 32 walkers, converged runs in the tests
        _instance("potts10_L20", "run", 8, "potts10_L20"),
        # the benchmark's workload from its start: 1024 walkers, ln f = 1
        _instance("potts10_L80", "run", 64, "potts10_L80", join=True),
        # the same at a late ln f: where nearly all of the time of a converged run goes
        _instance("potts10_L80_late", "late", 64, "potts10_L80", join=True),
        # the paper's own size: 2151 walkers on lattices of 45 KB (configurations are
        # left on the device: the energies say what they hold)
        _instance("potts10_L300", "run", 16, "potts10_L300", spins=False),
        # the 1/t schedule's last stage (ln f = bins / steps, another value each round)
        _instance("potts10_L80_1t", "1/t", 16, "potts10_L80"),
        # 2048 uneven instances together: throughput (the batched workload)
        dict(name="batched2048", kind="batch", n=2048, K=10_000, rounds=24),
        # a few dozen instances: a parameter study, too few walkers to fill the GPU one each to a thread
        dict(name="batched64", kind="batch", n=64, K=10_000, rounds=16),
        # short jobs arriving together, served until every one has converged
        dict(name="serve24", kind="serve", n=24, L_lo=6, L_hi=8, K=2000, lnf_final=0.05),
        # sampling with fixed weights after a run: H(E, O) in 64 classes
        _instance("production_L80", "production", 16, "potts10_L80", classes=64),
        # a whole short run: create, run, read, destroy (seeded start and window entry included)
        _instance("whole_L40", "whole", 1, "potts10_L40_w291"),
        # the run that allocates nothing, set-up included: a short latency-bound call
        _instance("static_L8", "static", 4, "ising_L8", K=1000),
    ]


def _log(rng, lo, hi):
    return int(round(lo * (hi / lo) ** rng.random()))


def draw(rng):
    kind = rng.choice(["run", "run", "late", "late", "1/t", "batch", "batch", "serve", "production", "whole", "static"])
    if kind == "batch":
        n = _log(rng, 8, 1500)
        return dict(kind=kind, n=n, K=rng.choice([5000, 10_000]), rounds=rng.randint(4, 12))
    if kind == "serve":
        return dict(kind=kind, n=rng.randint(2, 16), L_lo=6, L_hi=8, K=rng.choice([1000, 2000]), lnf_final=0.1)
    L = _log(rng, 6, 16 if kind == "static" else 48 if kind == "whole" else 112)
    h = _log(rng, 2, 8 if kind == "static" else 64)
    while 2 * L * L / (1.0 + 0.25 * (h - 1)) < 24:  # windows of at least two dozen bins
        h -= 1
    m = rng.randint(1, 4) if kind == "static" else rng.randint(1, 16)
    q = rng.choice([2, 3, 4, 5, 8, 10, 10, 16, 20])
    K = rng.choice([1000, 2500]) if kind == "static" else rng.choice([2000, 5000, 10_000])
    case = dict(kind=kind, q=q, L=L, h=h, m=m, K=K, lnf_final=1e-12, bits=rng.choice([0, 0, 8]),
                rounds=1 if kind == "whole" else rng.randint(2, 16))
    if kind == "production":
        case["classes"] = rng.choice([1, 16, 64])
    return case


# ---- inputs -------------------------------------------------------------------
def _job_seed(seed, i=0):
    return (0x9E3779B97F4A7C15 * (2 * int(seed) + 1) + 0xD1B54A32D192ED03 * i) % (1 << 63)


def _args(case, seed):
    return (case["q"], case["L"], case["h"], 0.75, case["m"], case["lnf_final"], 0.8, case["K"], _job_seed(seed))


def _batch_jobs(case, seed):
    jobs = workloads.batched_instances(case["n"])  # (the same sizes for every seed)
    for i, j in enumerate(jobs):
        j["seed"] = _job_seed(seed, i)
        j["exchange_interval"] = case["K"]
        j["lnf_final"] = 1e-8  # (a series of passes does not reach the end of the smallest ones)
    return jobs


def _served_jobs(case, seed):
    rng = np.random.default_rng(case["n"])  # (the same sizes for every seed)
    return [dict(q=int(rng.integers(2, 11)), L=int(rng.integers(case["L_lo"], case["L_hi"] + 1)),
                 h=int(rng.integers(2, 5)), overlap=0.75, m=int(rng.integers(2, 5)), lnf_final=case["lnf_final"],
                 flatness=0.8, exchange_interval=case["K"], seed=_job_seed(seed, i)) for i in range(case["n"])]


def _refine(r, last):
    """ln g as a run has it late on: rounds at ln f = 1, then at smaller and
    smaller ln f, each long enough for a walker to cross its window."""
    per = min(24, max(4, -(-20 * r.B // int(r.K))))
    for lnf, n in ((1.0, 4 * per), (2.0**-2, per), (2.0**-4, per), (2.0**-6, per), (2.0**-8, per), (2.0**-11, per)):
        r.set("lnf", np.full(r.h, lnf))
        r.run(n)
    if last is not None:
        r.set("lnf", np.full(r.h, last))


def _handle(case, seed):
    r = REWL(*_args(case, seed), spin_bits=case["bits"])
    r.K = case["K"]
    return r


def prepare(case, seed):
    kind = case["kind"]
    if kind == "batch":
        b = Batch(_batch_jobs(case, seed))
        return case, b, [b.instance(i) for i in range(len(b))]
    if kind == "serve":
        jobs = _served_jobs(case, seed)
        return case, Server(64 << 20, max_jobs=len(jobs)), jobs
    if kind == "whole":
        return case, _args(case, seed)
    if kind == "static":
        q, L, h, o, m, lf, fl, K, sd = _args(case, seed)
        W = -(-2 * L * L * 4 // (h + 3))  # ceil(2 N / (1 + (h - 1) / 4))
        lng = torch.zeros((h, W + 1), dtype=torch.float64, device="cuda")
        mask = torch.zeros((h, W + 1), dtype=torch.uint8, device="cuda")
        return case, _lib.Params(q, L, h, o, m, lf, fl, K, sd), lng, mask
    r = _handle(case, seed)
    if kind == "late":
        _refine(r, 2.0**-20)
    elif kind == "1/t":
        r.set_option(_lib.OPT_SCHEDULE, 1)
        _refine(r, None)
        r.set("phase", np.ones(r.h))  # the windows follow ln f = bins / steps from here on
    elif kind == "production":
        _refine(r, None)
        n = case["L"] ** 2
        r.production_start(min(case["classes"], n - -(-n // case["q"]) + 1))
    return case, r


# ---- one pass -----------------------------------------------------------------
def _read(r, case):
    out = {f: r.get(f) for f in ("lng", "hist", "mask", "energy", "lnf")}
    if case.get("spins", True):
        out["spins"] = r.get("spins")
    if case.get("join"):
        out["joined"] = r.lng(partial=True)
    return out


def run(state):
    case, kind = state[0], state[0]["kind"]
    if kind == "batch":
        _, b, views = state
        b.run(case["rounds"])
        return {"lng": np.concatenate([v.get("lng").ravel() for v in views]),
                "energy": np.concatenate([v.get("energy") for v in views])}
    if kind == "serve":
        _, srv, jobs = state
        ids = [srv.submit(**j) for j in jobs]
        while srv.step(8) != (0, 0):
            pass
        out = np.concatenate([srv.result(i) for i in ids])
        for i in ids:
            srv.release(i)
        return out
    if kind == "whole":
        r = REWL(*state[1], spin_bits=case["bits"])
        r.run(case["rounds"])
        out = _read(r, case)
        r.close()
        return out
    if kind == "static":
        _, params, lng, mask = state
        conv = C.c_int(0)
        _lib.check(_lib.load().rewl_run_static(
            C.byref(params), case["bits"], case["rounds"], C.c_void_p(lng.data_ptr()), C.c_void_p(mask.data_ptr()),
            lng.numel(), C.byref(conv), C.c_void_p(torch.cuda.current_stream().cuda_stream)))
        return {"lng": lng, "mask": mask}
    r = state[1]
    if kind == "production":
        r.production_run(case["rounds"])
        return {"heo": r.heo(), "energy": r.get("energy"), "spins": r.get("spins")}
    r.run(case["rounds"])
    return _read(r, case)


# ---- what a pass cannot do without ----------------------------------------------
def _sizes(q, L, h, m, bits):
    N = L * L
    B = -(-2 * N * 4 // (h + 3)) + 1
    G = h * m
    lat = N * (bits or (4 if q <= 16 else 8)) // 8
    return G, G * (lat + 12 * B + 24)  # walkers; their lattices, ln g (f64) and histograms (u32)


def work(case):
    """bytes: each walker's state read once and written once a pass, and the
    results.  flops: 118 operations a proposal (24 integer multiplies, 68
    logic, add and compare operations, 11 memory operations and 15 of the
    acceptance test: the counts of the benchmark's roofline)."""
    kind = case["kind"]
    if kind in ("batch", "serve"):
        jobs = _batch_jobs(case, 0) if kind == "batch" else _served_jobs(case, 0)
        steps = case["K"] * case["rounds"] if kind == "batch" else 400_000
        walkers = state = 0
        for j in jobs:
            g, s = _sizes(j["q"], j["L"], j["h"], j["m"], 0)
            walkers, state = walkers + g, state + s
    else:
        walkers, state = _sizes(case["q"], case["L"], case["h"], case["m"], case["bits"])
        steps = case["K"] * case["rounds"]
    return {"bytes": 2.0 * state, "flops": 118.0 * walkers * steps}


# ---- the same run in numpy, every walker at once --------------------------------
def _philox(c0, c1, c2, c3, key):
    c = [np.asarray(x, dtype=np.uint64) for x in np.broadcast_arrays(c0, c1, c2, c3)]
    k0, k1, low = key & 0xFFFFFFFF, key >> 32, np.uint64(0xFFFFFFFF)
    for _ in range(10):
        a, b = c[0] * np.uint64(0xD2511F53), c[2] * np.uint64(0xCD9E8D57)
        c = [(b >> np.uint64(32)) ^ c[1] ^ np.uint64(k0), b & low, (a >> np.uint64(32)) ^ c[3] ^ np.uint64(k1), a & low]
        k0, k1 = (k0 + 0x9E3779B9) & 0xFFFFFFFF, (k1 + 0xBB67AE85) & 0xFFFFFFFF
    return c


def _below(word, n):
    return ((word * np.uint64(n)) >> np.uint64(32)).astype(np.int64)


def _unit(a, b):
    return ((a >> np.uint64(5)) * np.uint64(1 << 26) + (b >> np.uint64(6))).astype(np.float64) * 2.0**-53


class _Plain:
    """The method on arrays: spins (G, N), ln g and H (G, B)."""

    def __init__(self, q, L, h, overlap, m, lnf_final, flatness, K, seed):
        self.q, self.L, self.h, self.m, self.K = q, L, h, m, K
        self.key, self.flat, self.lnf_final = seed, flatness, lnf_final
        N, G = L * L, h * m
        R = 2 * N
        self.W = min(R, int(np.ceil(R / (1.0 + (h - 1) * (1.0 - overlap)))))
        lo = np.array([-R + ((2 * i * (R - self.W) + h - 1) // (2 * (h - 1)) if h > 1 else 0) for i in range(h)])
        self.win = np.repeat(np.arange(h), m)
        self.lo, self.w_lo, self.g = lo[self.win], lo, np.arange(G)
        s = np.arange(N)
        x, y = s % L, s // L
        self.nb = np.stack([y * L + (x + 1) % L, y * L + (x - 1) % L, (y + 1) % L * L + x, (y - 1) % L * L + x], 1)
        words = np.stack(_philox((np.arange(-(-N // 4)))[None, :], 0, self.g[:, None], 1, seed), 2).reshape(G, -1)
        self.s = _below(words[:, :N], q)
        self.E = -(sum((self.s == self.s[:, self.nb[:, k]]).sum(1) for k in (0, 2)))
        high = self.E > self.lo + self.W
        c = _below(_philox(0, 0, self.g, 2, seed)[0], q)
        self.s[high] = c[high, None]
        self.E[high] = -R
        n = 1
        todo = np.nonzero(self.E < self.lo)[0]
        while todo.size:  # up from below the window, never down, never past its top
            r = _philox(n, 0, todo, 2, seed)
            site = _below(r[0], N)
            cur, new, dE = self._proposal(todo, site, _below(r[1], q - 1))
            ok = (dE >= 0) & (self.E[todo] + dE <= self.lo[todo] + self.W)
            self.s[todo[ok], site[ok]] = new[ok]
            self.E[todo[ok]] += dE[ok]
            todo = todo[self.E[todo] < self.lo[todo]]
            n += 1
        B = self.W + 1
        self.lng, self.H = np.zeros((G, B)), np.zeros((G, B), dtype=np.int64)
        self.mask, self.lnf, self.done = np.zeros((h, B), dtype=bool), np.ones(h), np.zeros(h, dtype=bool)
        self.t = np.zeros(G, dtype=np.uint64)
        self.round = 0

    def _proposal(self, who, site, v):
        cur = self.s[who, site]
        new = v + (v >= cur)
        near = self.s[who[:, None], self.nb[site]]
        return cur, new, (near == cur[:, None]).sum(1) - (near == new[:, None]).sum(1)

    def sweep(self):
        who = np.nonzero(~self.done[self.win])[0]
        E, lo, lnf = self.E[who] - self.lo[who], self.lo[who], self.lnf[self.win[who]]
        s, W, row, wrow = self.s.reshape(-1), self.W, who * (self.L * self.L), who * (self.W + 1)
        lng, H = self.lng.reshape(-1), self.H.reshape(-1)
        for k0 in range(0, self.K, 500):  # the random numbers of 500 steps at a time
            n = min(500, self.K - k0)
            t = self.t[who] + np.arange(k0, k0 + n, dtype=np.uint64)[:, None]
            r = _philox(t & np.uint64(0xFFFFFFFF), t >> np.uint64(32), who, 0, self.key)
            sites, vs, us = _below(r[0], self.L * self.L), _below(r[1], self.q - 1), _unit(r[2], r[3])
            places, nears = row + sites, row[:, None] + self.nb[sites]
            for i in range(n):
                place, v = places[i], vs[i]
                cur, near = s[place], s[nears[i]]
                new = v + (v >= cur)
                En = E + ((near == cur[:, None]) * 1 - (near == new[:, None])).sum(1)
                inside = (En >= 0) & (En <= W)
                d = lng[wrow + E] - lng[wrow + np.where(inside, En, E)]
                acc = inside & (us[i] < np.exp(np.minimum(d, 0.0)))  # (u < 1 = exp(0))
                s[place] = np.where(acc, new, cur)
                E = np.where(acc, En, E)
                lng[wrow + E] += lnf
                H[wrow + E] += 1
        self.E[who] = E + lo
        self.t[who] += np.uint64(self.K)

    def barrier(self):
        m = self.m
        for w in range(self.h):
            if self.done[w]:
                continue
            rows = slice(w * m, w * m + m)
            self.mask[w] |= (self.H[rows] > 0).any(0)
            H = self.H[rows][:, self.mask[w]]
            if not (H.min(1) >= self.flat * (H.sum(1) / H.shape[1])).all():
                continue
            part = [self.lng[w * m + k].copy() for k in range(m)]
            stride = 1
            while stride < m:
                for k in range(0, m - stride, 2 * stride):
                    part[k] = part[k] + part[k + stride]
                stride *= 2
            self.lng[rows], self.H[rows] = part[0] / m, 0
            self.lnf[w] *= 0.5
            self.done[w] = self.lnf[w] < self.lnf_final
        for a in range(self.round % 2, self.h - 1, 2):
            if self.done[a] or self.done[a + 1]:
                continue
            pi = list(range(m))
            for i in range(m - 1, 0, -1):
                n = m - 1 - i
                j = int(_below(_philox(self.round, n >> 2, a, 3, self.key)[n & 3], i + 1))
                pi[i], pi[j] = pi[j], pi[i]
            la, lb = self.w_lo[a], self.w_lo[a + 1]
            for k in range(m):
                i, j = a * m + k, (a + 1) * m + pi[k]
                Ei, Ej = self.E[i], self.E[j]
                if not (lb <= Ei <= lb + self.W and la <= Ej <= la + self.W):
                    continue
                d = (self.lng[i, Ei - la] - self.lng[i, Ej - la]) + (self.lng[j, Ej - lb] - self.lng[j, Ei - lb])
                r = _philox(self.round, k, a, 4, self.key)
                if d >= 0 or _unit(r[0], r[1]) < np.exp(d):
                    self.s[[i, j]], self.E[[i, j]] = self.s[[j, i]], self.E[[j, i]]
        self.round += 1


def exact(case, seed):
    if case["kind"] not in ("run", "whole", "static"):
        return None  # these go on from a run that numpy would take minutes for
    walkers = case["h"] * case["m"]
    steps = case["K"] * case["rounds"] + (8 * case["L"] ** 2 if case["L"] > 8 else 0)
    if case["L"] > 64 or steps * (60.0 + 0.4 * walkers) > 12e6 or case.get("join"):  # about microseconds
        return None
    p = _Plain(*_args(case, seed))
    for _ in range(case["rounds"]):
        p.sweep()
        p.barrier()
    if case["kind"] == "static":
        return {"lng": p.lng[::p.m], "mask": p.mask.astype(np.uint8)}
    out = {"lng": p.lng, "hist": p.H, "mask": p.mask.astype(np.uint8), "energy": p.E, "lnf": p.lnf}
    if case.get("spins", True):
        out["spins"] = p.s.astype(np.uint8)
    return out

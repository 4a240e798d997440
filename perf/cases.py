"""The calls a user of this framework makes, as measurable cases.

A case is one pass through the public entry points of
`paper_1811_04384_gb300`: a Lattice that goes on from where it stands
(`sweep_record`), a sequence of uploaded configurations (`run_states`), a
Batch of replicas, the paper's own layout and chain, or a set of jobs given
to the server.  `listed()` has the named cases, `draw(rng)` one more of the
same ranges, `prepare` makes what a program holds before the call, `run` is
the call, `work` what it cannot do without, and `exact` the same results from
a plain torch restatement of the conventions in include/ising.h.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_1811_04384_gb300 as ising
from paper_1811_04384_gb300 import serving

T_C = 2.269                         # the temperature of the plain and large configurations
BATCH_SIDES = (32, 64, 128, 256, 512, 1024, 2048)        # the batched configuration's lattices
JOB_SIDES = (64, 128, 256, 512, 1024)                     # served jobs of one pass


def listed():
    return [
        # an interactive call: a few sweeps of a small lattice, a record after each (latency and launches)
        {"name": "short_call_64", "kind": "lattice", "L": 64, "T": T_C, "sweeps": 10, "every": 1, "rng": 10},
        # the plain configuration: one small lattice, a long recorded series
        {"name": "plain_64", "kind": "lattice", "L": 64, "T": T_C, "sweeps": 1000, "every": 1, "rng": 10},
        # one mid-size lattice, a record every 10 sweeps
        {"name": "mid_296", "kind": "lattice", "L": 296, "T": T_C, "sweeps": 1000, "every": 10, "rng": 10},
        # the larger of the paper's test lattices (Table 2), a record every 10 sweeps
        {"name": "paper_2016", "kind": "lattice", "L": 2016, "T": T_C, "sweeps": 300, "every": 10, "rng": 10},
        # the smaller one in the paper's own word layout
        {"name": "paper_layout_1008", "kind": "interleaved", "L": 1008, "T": T_C, "sweeps": 500, "every": 10,
         "rng": 10},
        # the paper's own chain: random memory words, its 72 processes, a record after each iteration
        {"name": "random_words_1008", "kind": "random_words", "L": 1008, "T": T_C, "strips": 72, "iterations": 5},
        # a large lattice of no special side (ragged last word and row group)
        {"name": "launches_5002", "kind": "lattice", "L": 5002, "T": T_C, "sweeps": 30, "every": 10, "rng": 10},
        # the large configuration's step: 10 sweeps and a record
        {"name": "large_16384", "kind": "lattice", "L": 16384, "T": T_C, "sweeps": 10, "every": 10, "rng": 10},
        # configurations kept on the host, uploaded one after another and swept
        {"name": "states_4096", "kind": "states", "L": 4096, "T": T_C, "states": 4, "sweeps": 10, "every": 10},
        # the energy-versus-temperature scan: one batch, T = 1.0 .. 3.5, every sweep recorded
        {"name": "scan_1024", "kind": "scan", "L": 1024, "replicas": 26, "T_low": 1.0, "T_high": 3.5, "sweeps": 100,
         "every": 1},
        # replicas of uneven sides, each at its own temperature
        {"name": "batch_uneven", "kind": "batch", "replicas": 256, "sides": 7, "sweeps": 50, "every": 1},
        # jobs of several users, served together
        {"name": "serving", "kind": "serving", "jobs": 48, "sides": 5, "sweeps_low": 100, "sweeps_high": 500},
    ]


def _log_int(rng, low, high):
    return int(round(math.exp(rng.uniform(math.log(low), math.log(high)))))


def _even(rng, low, high):
    return min(high, max(low, 2 * (_log_int(rng, low, high) // 2)))


def draw(rng):
    kind = rng.choice(["small", "mid", "mid", "interleaved", "random_words", "large", "large", "states", "scan",
                       "batch", "serving"])
    T = round(rng.uniform(1.5, 3.5), 3)
    rounds = 7 if rng.random() < 0.2 else 10           # the opt-in 7-round draws
    if kind == "small":
        return {"kind": "lattice", "L": _even(rng, 16, 128), "T": T, "sweeps": _log_int(rng, 10, 1000),
                "every": rng.choice([1, 1, 3, 10]), "rng": rounds}
    if kind == "mid":
        L = _even(rng, 130, 3000)
        most = min(1000, int(1.2e9 / (L * L)))
        return {"kind": "lattice", "L": L, "T": T, "sweeps": _log_int(rng, 20, most), "every": rng.choice([1, 5, 10]),
                "rng": rounds}
    if kind == "large":
        L = _even(rng, 3002, 16384)
        return {"kind": "lattice", "L": L, "T": T, "sweeps": _log_int(rng, 5, min(60, int(3.2e9 / (L * L)) + 5)),
                "every": rng.choice([1, 5, 10]), "rng": rounds}
    if kind == "interleaved":
        L = 84 * _log_int(rng, 2, 36)
        return {"kind": "interleaved", "L": L, "T": T, "sweeps": _log_int(rng, 20, min(1000, int(1e9 / (L * L)))),
                "every": rng.choice([1, 5, 10]), "rng": rounds}
    if kind == "random_words":
        L = 84 * _log_int(rng, 3, 24)
        strips = rng.choice([s for s in (21, 28, 36, 42, 63, 72, 84, 126, 144, 252) if L % s == 0 and L // s >= 2])
        return {"kind": "random_words", "L": L, "T": T, "strips": strips, "iterations": rng.randint(1, 4)}
    if kind == "states":
        return {"kind": "states", "L": _even(rng, 900, 8192), "T": T, "states": rng.randint(2, 5),
                "sweeps": rng.choice([5, 10, 20]), "every": 5}
    if kind == "scan":
        return {"kind": "scan", "L": _even(rng, 128, 1400), "replicas": rng.randint(8, 30),
                "T_low": round(rng.uniform(1.0, 1.8), 2), "T_high": round(rng.uniform(2.8, 3.6), 2),
                "sweeps": _log_int(rng, 20, 120), "every": rng.choice([1, 1, 10])}
    if kind == "batch":
        return {"kind": "batch", "replicas": _log_int(rng, 16, 256), "sides": rng.randint(3, 7),
                "sweeps": _log_int(rng, 20, 50), "every": rng.choice([1, 1, 5])}
    return {"kind": "serving", "jobs": _log_int(rng, 4, 48), "sides": rng.randint(2, 5), "sweeps_low": 50,
            "sweeps_high": rng.choice([200, 500])}


# ---- what a user's program holds before the call ---------------------------

def _replicas(case):
    """Sides and temperatures of a Batch (the replicas' places in their ranges do not depend on the seed)."""
    if case["kind"] == "scan":
        n = case["replicas"]
        return [case["L"]] * n, [case["T_low"] + (case["T_high"] - case["T_low"]) * k / (n - 1) for k in range(n)]
    r = np.random.default_rng(11)
    sides = BATCH_SIDES[:case["sides"]]
    L = [int(v) for v in r.choice(sides, size=case["replicas"])]
    return L, [float(v) for v in r.uniform(1.5, 3.5, size=case["replicas"])]


def _jobs(case):
    r = np.random.default_rng(13)
    n = case["jobs"]
    L = r.choice(JOB_SIDES[:case["sides"]], size=n)
    T = r.uniform(1.5, 3.5, size=n)
    s = np.exp(r.uniform(math.log(case["sweeps_low"]), math.log(case["sweeps_high"]), size=n))
    return [(int(a), 1.0 / float(b), int(c)) for a, b, c in zip(L, T, s)]


def _seeds(seed, n):
    return [int(v) for v in np.random.default_rng(seed).integers(1, 2**63, size=n, dtype=np.uint64)]


def _host_states(case, seed):
    L = case["L"]
    g = torch.Generator().manual_seed(seed)
    return [(torch.randint(0, 2, (L, L), dtype=torch.int8, generator=g) * 2 - 1) for _ in range(case["states"])]


def prepare(case, seed):
    kind = case["kind"]
    if kind in ("lattice", "states"):
        # the lattice lives in torch's device memory, so its words are at hand as a tensor
        L = case["L"]
        buffer = torch.zeros(ising.bytes_required(L), dtype=torch.uint8, device="cuda")
        torch.cuda.synchronize()
        lat = ising.Lattice(L, _seeds(seed, 1)[0], buffer=buffer)
        if kind == "lattice":
            lat.init_hot()
            lat.set_rng(ising.ISING_RNG_PHILOX4X32_7 if case["rng"] == 7 else ising.ISING_RNG_PHILOX4X32_10)
        lat.set_beta(1.0 / case["T"])
        _, pitch, _ = lat.layout()
        words = []
        for c in (0, 1):
            at = lat.device_words(c) - buffer.data_ptr()
            words.append(buffer[at:at + 8 * L * pitch].view(torch.int64).reshape(L, pitch))
        state = {"case": case, "lat": lat, "words": words}
        if kind == "states":
            state["pinned"] = [s.pin_memory() for s in _host_states(case, seed)]
            state["arrays"] = [s.numpy() for s in state["pinned"]]
        return state
    if kind in ("interleaved", "random_words"):
        lat = ising.Lattice(case["L"], _seeds(seed, 1)[0], layout=ising.ISING_LAYOUT_COLUMN_INTERLEAVED)
        lat.init_hot()
        lat.set_beta(1.0 / case["T"])
        if kind == "random_words":
            lat.set_chain(ising.ISING_CHAIN_RANDOM_WORDS, case["strips"])
        else:
            lat.set_rng(ising.ISING_RNG_PHILOX4X32_7 if case["rng"] == 7 else ising.ISING_RNG_PHILOX4X32_10)
        pinned = torch.empty((case["L"], case["L"]), dtype=torch.int8).pin_memory()
        return {"case": case, "lat": lat, "pinned": pinned, "spins": pinned.numpy()}
    if kind in ("scan", "batch"):
        L, T = _replicas(case)
        return {"case": case,
                "batch": ising.Batch(L, [1.0 / t for t in T], _seeds(seed, len(L)), np.ones(len(L), dtype=np.uint8))}
    jobs = _jobs(case)
    return {"case": case, "server": serving.Server(512 << 20), "jobs": jobs, "seeds": _seeds(seed, len(jobs))}


# ---- the call --------------------------------------------------------------

def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "lattice":
        E, M = state["lat"].sweep_record(case["sweeps"], case["every"])
        return {"E": E, "M": M, "words": state["words"]}
    if kind == "states":
        E, M = state["lat"].run_states(state["arrays"], case["sweeps"], case["every"])
        return {"E": E, "M": M, "words": state["words"]}
    if kind in ("interleaved", "random_words"):
        lat = state["lat"]
        if kind == "interleaved":
            E, M = lat.sweep_record(case["sweeps"], case["every"])
        else:
            E, M = lat.sweep_record(case["iterations"], 1)
        return {"E": E, "M": M, "spins": lat.get_spins(state["spins"])}
    if kind in ("scan", "batch"):
        E, M = state["batch"].sweep(case["sweeps"], every=case["every"])
        return {"E": np.stack(E), "M": np.stack(M)}
    server = state["server"]
    requests = [serving.Request(L, beta, seed, sweeps) for (L, beta, sweeps), seed in zip(state["jobs"], state["seeds"])]
    for r in requests:
        server.submit(r)
    for r in requests:
        server.wait(r.id)
        server.release(r.id)
    return {"E": np.concatenate([r.E for r in requests]), "M": np.concatenate([r.M for r in requests])}


# ---- what a pass cannot do without -----------------------------------------

# Integer operations of one proposed spin flip: a quarter of a Philox4x32 call
# (per round two 32x32->64 products and four XORs), two threshold compares and
# the word logic of its 1/21 word; the random-word chain draws 24 words (six
# calls) for the 21 spins of a word and proposes each spin 10 times a sweep.
def _ops_per_update(rounds):
    return rounds * 6 / 4 + 2 + 1


def work(case):
    kind = case["kind"]
    if kind in ("lattice", "interleaved", "random_words", "states"):
        L = case["L"]
        packed = L * L * 8 / 21
        if kind == "random_words":
            n = case["iterations"]
            return {"bytes": 2 * packed + 16 * n + L * L, "flops": 10.0 * n * L * L * (10 * 6 * 6 / 21 + 3)}
        if kind == "states":
            n = case["states"]
            return {"bytes": n * L * L + packed + 16 * n, "flops": float(n) * case["sweeps"] * L * L * _ops_per_update(10)}
        spins = L * L if kind == "interleaved" else 0
        return {"bytes": 2 * packed + 16 * (case["sweeps"] // case["every"]) + spins,
                "flops": float(case["sweeps"]) * L * L * _ops_per_update(case["rng"])}
    if kind in ("scan", "batch"):
        sites = sum(L * L for L in _replicas(case)[0])
        return {"bytes": 2 * sites * 8 / 21 + 16.0 * case["replicas"] * (case["sweeps"] // case["every"]),
                "flops": float(case["sweeps"]) * sites * _ops_per_update(10)}
    jobs = _jobs(case)
    return {"bytes": sum(L * L * 8 / 21 + 16.0 * s for L, _, s in jobs),
            "flops": sum(float(s) * L * L for L, _, s in jobs) * _ops_per_update(10)}


# ---- the same results in plain torch ----------------------------------------

_M32 = 0xFFFFFFFF


def _philox(x0, x1, x2, x3, k0, k1, rounds):
    """Philox4x32 (Salmon et al., SC'11) on int64 tensors that hold 32-bit values."""
    def wide(x, m):                 # 32 x 32 -> (hi, lo) through 64-bit wrap-around products
        p = x * m
        return (p >> 32) & _M32, p & _M32
    for _ in range(rounds):
        h0, l0 = wide(x0, 0xD2511F53)
        h1, l1 = wide(x2, 0xCD9E8D57)
        x0, x1, x2, x3 = h1 ^ x1 ^ k0, l1, h0 ^ x3 ^ k1, l0
        k0, k1 = (k0 + 0x9E3779B9) & _M32, (k1 + 0xBB67AE85) & _M32
    return x0, x1, x2, x3


class _Chain:
    """R lattices of side L with their own seeds and temperatures; colour c of row i holds columns 2m + ((i + c) & 1)."""

    def __init__(self, L, seeds, betas):
        self.L, self.R, self.t = L, len(seeds), 0
        dev = torch.device("cuda" if torch.cuda.is_available() else "cpu")
        col = lambda v: torch.tensor(v, dtype=torch.int64, device=dev).reshape(-1, 1, 1)  # noqa: E731
        self.k0, self.k1 = col([s & _M32 for s in seeds]), col([s >> 32 for s in seeds])
        thr = [[min(2**32, math.floor(math.exp(-(8.0 - 4.0 * a) * b) * 4294967296.0)) for b in betas] for a in (0, 1)]
        self.thr = [col(v) for v in thr]
        self.g = torch.arange((L + 3) // 4, device=dev).reshape(1, -1, 1)
        self.m = torch.arange(L // 2, device=dev).reshape(1, 1, -1)
        self.even = (torch.arange(L, device=dev) & 1 == 0).reshape(1, -1, 1)
        self.A = [(self.draws(0, c, 10) < 2**31).to(torch.int8) for c in (0, 1)]

    def draws(self, t, c, rounds):
        # a chunk of row groups at a time: the 64-bit temporaries of a large lattice would not fit otherwise
        parts, step = [], max(1, (1 << 25) // (self.R * (self.L // 2)))
        for g0 in range(0, self.g.shape[1], step):
            g = self.g[:, g0:g0 + step]
            x = torch.stack(torch.broadcast_tensors(*_philox(
                g, self.m, torch.full_like(g, t & _M32), torch.full_like(g, (t >> 32) << 1 | c), self.k0, self.k1,
                rounds)), 2)                                     # (R, groups, 4, L/2)
            parts.append(x.reshape(self.R, -1, self.L // 2))
        return torch.cat(parts, 1)[:, :self.L]

    def neighbours(self, c):
        o = self.A[1 - c]
        left = self.even if c == 0 else ~self.even
        side = torch.where(left, o.roll(1, 2), o.roll(-1, 2))
        return o.roll(1, 1), o.roll(-1, 1), o, side

    def sweep(self, rounds):
        self.t += 1
        for c in (0, 1):
            s = self.A[c]
            a = sum((n ^ s) for n in self.neighbours(c))
            r = self.draws(self.t, c, rounds)
            flip = (a >= 2) | ((a == 1) & (r < self.thr[1])) | ((a == 0) & (r < self.thr[0]))
            self.A[c] = s ^ flip.to(torch.int8)

    def record(self):
        N = self.L * self.L
        anti = sum((n ^ self.A[1]).sum((1, 2), dtype=torch.int64) for n in self.neighbours(1))
        up = sum(a.sum((1, 2), dtype=torch.int64) for a in self.A)
        return (2 * anti - 2 * N).cpu().numpy(), (2 * up - N).cpu().numpy()

    def spins(self):
        s = torch.empty((self.R, self.L, self.L // 2, 2), dtype=torch.int8, device=self.A[0].device)
        for c in (0, 1):
            first = self.even if c == 0 else ~self.even
            s[..., 0] = torch.where(first, self.A[c], s[..., 0])
            s[..., 1] = torch.where(first, s[..., 1], self.A[c])
        return (2 * s - 1).reshape(self.R, self.L, self.L)

    def set_spins(self, s):
        s = (s.to(self.A[0].device) > 0).to(torch.int8).reshape(1, self.L, self.L // 2, 2)
        for c in (0, 1):
            self.A[c] = torch.where(self.even if c == 0 else ~self.even, s[..., 0], s[..., 1])

    def words(self):
        W = (self.L // 2 + 20) // 21
        out = []
        for a in self.A:
            f = torch.nn.functional.pad(a[0].to(torch.int64), (0, 21 * W - self.L // 2)).reshape(self.L, W, 21)
            w = sum(f[:, :, k] << (3 * k) for k in range(21))
            out.append(torch.nn.functional.pad(w, (0, (W + 1) // 2 * 2 - W)))
        return out

    def series(self, sweeps, every, rounds=10):
        rec = []
        for k in range(1, sweeps + 1):
            self.sweep(rounds)
            if k % every == 0:
                rec.append(self.record())
        E, M = (np.array([r[q] for r in rec], dtype=np.int64).reshape(-1, self.R).T for q in (0, 1))
        return np.ascontiguousarray(E), np.ascontiguousarray(M)


def exact(case, seed):
    """The pass after prepare(case, seed); None for the sequential random-word chain, the served jobs and passes
    whose restatement would take long (few large or many small steps on one device)."""
    kind = case["kind"]
    if kind in ("random_words", "serving"):
        return None
    if kind in ("lattice", "interleaved"):
        L = case["L"]
        if case["sweeps"] * L * L > 2e10:
            return None
        c = _Chain(L, _seeds(seed, 1), [1.0 / case["T"]])
        E, M = c.series(case["sweeps"], case["every"], case["rng"])
        if kind == "interleaved":
            return {"E": E[0], "M": M[0], "spins": c.spins()[0]}
        return {"E": E[0], "M": M[0], "words": c.words()}
    if kind == "states":
        L = case["L"]
        c = _Chain(L, _seeds(seed, 1), [1.0 / case["T"]])
        E, M = [], []
        for s in _host_states(case, seed):
            c.set_spins(s)
            e, m = c.series(case["sweeps"], case["every"])
            E.append(e[0])
            M.append(m[0])
        return {"E": np.stack(E), "M": np.stack(M), "words": c.words()}
    sides, T = _replicas(case)
    seeds = _seeds(seed, len(sides))
    n = case["sweeps"] // case["every"]
    E, M = np.zeros((len(sides), n), dtype=np.int64), np.zeros((len(sides), n), dtype=np.int64)
    for L in sorted(set(sides)):
        at = [k for k, v in enumerate(sides) if v == L]
        c = _Chain(L, [seeds[k] for k in at], [1.0 / T[k] for k in at])
        E[at], M[at] = c.series(case["sweeps"], case["every"])
    return {"E": E, "M": M}

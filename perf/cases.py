"""Performance cases: the work that a user of the framework has it do, through its public entry points.

A case is a dict of plain values.  Its "kind" says which calls one pass makes:
  run       a realization advances (sweeps with exchange steps, measured), then the user reads its
            observables and takes a checkpoint (spins, permutation, counters)
  adapt     a realization is created and its temperature set adapted from trial runs
  serve     a batch of independent realizations of mixed sizes goes through the server
  exchange  one exchange step on the caller's own device buffers
exact() recomputes a pass in plain torch: integers as such, real numbers in 64 bits.
"""
import math

import numpy as np
import torch

import paper_1508_06268_gb300 as rf
from paper_1508_06268_gb300 import inputs

FIELDS = {"bimodal": rf.FIELD_BIMODAL, "gaussian": rf.FIELD_GAUSSIAN, "explicit": rf.FIELD_EXPLICIT}
LAYOUTS = {"bit": rf.LAYOUT_BITPACK, "int8": rf.LAYOUT_INT8}


def _run(L, R, field, sweeps, every, *, layout="bit", h=1.0, t_min=1.0, xi=False, mh=0, tile=0, calls="run"):
    return {"kind": "run", "L": L, "R": R, "layout": layout, "field": field, "h": h, "t_min": t_min, "sweeps": sweeps,
            "every": every, "xi": xi, "mh": mh, "tile": tile, "calls": calls}


def listed():
    return [
        # the smallest realization of the benchmark (L = 8, R = 16): a short run, all latency
        dict(_run(8, 16, "gaussian", 200, 10, t_min=1.5), name="l8_r16_gaussian"),
        # the bimodal configuration of the benchmark (L = 16, R = 32, exchange every 5)
        dict(_run(16, 32, "bimodal", 500, 5, h=1.5), name="l16_r32_bimodal"),
        # production sweeps of the adapted set of the benchmark's L = 32 configuration
        dict(_run(32, 70, "gaussian", 1000, 10), name="l32_r70_gaussian"),
        # the headline workload: L = 64, R = 128
        dict(_run(64, 128, "gaussian", 1000, 10), name="l64_r128_gaussian"),
        # the same lattices stored as bytes
        dict(_run(64, 128, "gaussian", 300, 10, layout="int8"), name="l64_r128_int8"),
        # correlation length at large L: few replicas, the structure factor at every measuring step
        dict(_run(64, 12, "bimodal", 200, 10, h=1.5, xi=True), name="l64_r12_bimodal_xi"),
        # a size between the powers of two (byte layout, rows of whole Philox blocks)
        dict(_run(24, 40, "gaussian", 100, 5, layout="int8"), name="l24_r40_int8"),
        # an odd size with the user's own field: rows that are no whole blocks, driven call by call
        dict(_run(10, 24, "explicit", 40, 4, layout="int8", calls="steps"), name="l10_r24_int8_steps"),
        # multi-hit sweeps of the double checkerboard
        dict(_run(32, 40, "bimodal", 40, 2, mh=4, tile=8), name="l32_r40_multihit"),
        # the adaptive temperature set of the L = 32 configuration, from the start
        {"kind": "adapt", "L": 32, "R": 64, "field": "gaussian", "h": 1.0, "t_min": 1.0, "trials": 3, "sweeps": 2000,
         "every": 10, "inserts": 2, "name": "l32_adapt_r64_r70"},
        # disorder average: mixed sizes, R matched to L, through the batched server
        {"kind": "serve", "n": 24, "sweeps": 200, "every": 10, "xi": False, "field": "gaussian", "h": 1.0,
         "name": "serve_24_mixed"},
        # the exchange step of a caller who owns all device memory
        {"kind": "exchange", "L": 32, "R": 70, "field": "explicit", "h": 1.0, "name": "exchange_l32_r70"},
    ]


def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choices(("run", "odd", "multihit", "adapt", "serve", "exchange"), (10, 4, 2, 1, 1, 2))[0]
    field = rng.choice(("gaussian", "bimodal", "explicit"))
    h = rng.choice((0.5, 1.0, 1.5, 2.0))
    if kind in ("run", "odd"):
        if kind == "run":
            L = rng.choice((8, 16, 32, 64))
            layout = rng.choice(("bit", "bit", "int8"))
        else:
            L = rng.choice((4, 6, 10, 12, 14, 18, 20, 22, 24, 26, 28, 30, 36, 40, 48, 50, 56))
            layout = "int8"
        R = _log_int(rng, 2, 200 if L > 32 else 400)
        every = _log_int(rng, 1, 20)
        work = math.exp(rng.uniform(math.log(2e5), math.log(1.5e10 if kind == "run" else 1e9)))
        steps = max(1, min(100, int(work / (L ** 3 * R * every))))
        return _run(L, R, field, steps * every, every, layout=layout, h=h, t_min=rng.choice((0.5, 1.0, 1.5)),
                    xi=rng.random() < 0.25, calls=rng.choice(("run", "run", "steps")))
    if kind == "multihit":
        L, tile = rng.choice(((16, 8), (32, 8), (32, 16), (64, 8), (64, 16), (64, 32)))
        R, mh, every = _log_int(rng, 2, 140), _log_int(rng, 1, 20), _log_int(rng, 1, 5)
        steps = max(1, min(40, int(5e9 / (L ** 3 * R * mh * every))))
        return _run(L, R, field, steps * every, every, h=h, mh=mh, tile=tile)
    if kind == "adapt":
        L = rng.choice((8, 16, 32, 64))
        return {"kind": "adapt", "L": L, "R": _log_int(rng, 4, 100), "field": field, "h": h, "t_min": 1.0,
                "trials": rng.randint(1, 4), "sweeps": 10 * rng.randint(3, 30), "every": rng.choice((5, 10)),
                "inserts": rng.randint(1, 3)}
    if kind == "serve":
        return {"kind": "serve", "n": rng.randint(4, 23), "sweeps": 10 * rng.randint(5, 19), "every": rng.choice((5, 10)),
                "xi": rng.random() < 0.3, "field": rng.choice(("gaussian", "bimodal")), "h": h}
    return {"kind": "exchange", "L": rng.choice((8, 16, 32, 64)), "R": _log_int(rng, 2, 300), "field": field, "h": h}


# ---- inputs ---------------------------------------------------------------------------------------

def _temps(case):
    return inputs.geometric_temps(case["t_min"], 5.0, case["R"])


def _field(case, seed):
    """The user's own field (explicit kinds), else None: the library draws it from the seed."""
    return inputs.gaussian_field(case["L"], seed % (1 << 30) + 7) if case["field"] == "explicit" else None


def _seeds(seed):
    return {"seed": (seed * 2654435761 + 42) % (1 << 32), "field_seed": (seed * 40503 + 1) % (1 << 32),
            "realization": seed % 1009}


def _requests(case, seed):
    """The realizations of a served batch: L cycles over 8, 16, 32, 64 with R = 16, 32, 64, 128."""
    out = []
    for i in range(case["n"]):
        L, R = ((8, 16), (16, 32), (32, 64), (64, 128))[i % 4]
        out.append({"L": L, "R": R, "t_min": 1.0, "field": case["field"], "h": case["h"], "xi": case["xi"], "mh": 0,
                    "tile": 0, "sweeps": case["sweeps"], "every": case["every"],
                    "seeds": dict(_seeds(seed), realization=i)})
    return out


def _exchange_inputs(case, seed):
    """Random spins of uneven magnetisation in the bit layout, the caller's field and an identity assignment."""
    L, R = case["L"], case["R"]
    gen = torch.Generator(device="cuda").manual_seed(seed)
    dev = {"device": "cuda"}
    up = torch.rand(R, 2, L ** 3 // 64, 32, generator=gen, **dev) < torch.linspace(0.9, 0.5, R, **dev)[:, None, None, None]
    bits = (up.long() << torch.arange(32, **dev)).sum(-1)
    if case["field"] == "bimodal":
        field = inputs.bimodal_field(L, seed % (1 << 30))
    else:
        field = inputs.gaussian_field(L, seed % (1 << 30))
    beta = torch.from_numpy(1.0 / inputs.geometric_temps(1.0, 5.0, R)).cuda()
    return bits, torch.from_numpy(field).cuda(), beta


def prepare(case, seed):
    kind = case["kind"]
    if kind == "serve":
        return {"case": case, "server": rf.Server(mem_budget_bytes=1 << 30, max_slots=64, measure_xi=case["xi"]),
                "requests": _requests(case, seed)}
    if kind == "exchange":
        L, R = case["L"], case["R"]
        bits, field, beta = _exchange_inputs(case, seed)
        i32, i64, f64 = torch.int32, torch.int64, torch.float64
        b = {"spins": torch.where(bits >= 1 << 31, bits - (1 << 32), bits).to(i32), "field": field, "beta": beta,
             "t2r": torch.arange(R, dtype=i32, device="cuda"), "r2t": torch.arange(R, dtype=i32, device="cuda"),
             "att": torch.zeros(R - 1, dtype=i64, device="cuda"), "acc": torch.zeros(R - 1, dtype=i64, device="cuda"),
             "obs": torch.zeros(R, 5, dtype=f64, device="cuda"), "n_meas": torch.zeros(1, dtype=i64, device="cuda"),
             "E": torch.zeros(R, dtype=f64, device="cuda"), "M": torch.zeros(R, dtype=i64, device="cuda")}
        s = _seeds(seed)
        eb = rf.ExchangeBuffers(L=L, R=R, J=1.0, h=case["h"], field_kind=FIELDS[case["field"]], seed=s["seed"],
                                realization=s["realization"], stage=0, **{k: t.data_ptr() for k, t in b.items()})
        return {"case": case, "buffers": b, "args": eb, "j": 0}
    if kind == "adapt":
        return {"case": case, "temps": _temps(case), "field": _field(case, seed), "seeds": _seeds(seed)}
    real = rf.Realization(case["L"], _temps(case), h=case["h"], field_kind=FIELDS[case["field"]], field=_field(case, seed),
                          layout=LAYOUTS[case["layout"]], **_seeds(seed))
    if case["xi"]:
        real.set_measure_xi()
    if case["mh"]:
        real.set_multihit(case["mh"], case["tile"])
    return {"case": case, "real": real}


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "serve":
        srv = state["server"]
        tickets = [srv.submit(q["L"], inputs.geometric_temps(1.0, 5.0, q["R"]), q["sweeps"], q["every"],
                              q["sweeps"] // q["every"] // 2, h=q["h"], field_kind=FIELDS[q["field"]], **q["seeds"])
                   for q in state["requests"]]
        got = [srv.wait(t) for t in tickets]
        return {k: np.concatenate([g[k] for g in got]) for k in ("T", "e", "e2", "absm", "m2", "m4", "F", "att", "acc")}
    if kind == "exchange":
        rf.exchange_noalloc(state["args"], state["j"], 0)
        state["j"] += 1
        b = state["buffers"]
        return {k: b[k] for k in ("t2r", "r2t", "att", "acc", "obs", "n_meas", "E", "M")}
    if kind == "adapt":
        with rf.Realization(case["L"], state["temps"], R_capacity=case["R"] + case["trials"] * case["inserts"], h=case["h"],
                            field_kind=FIELDS[case["field"]], field=state["field"], **state["seeds"]) as real:
            temps, rates = real.adapt_temps(case["trials"], case["sweeps"], case["every"], case["inserts"], return_rates=True)
        return {"temps": temps, "rates": rates}
    real = state["real"]
    steps = case["sweeps"] // case["every"]
    if case["calls"] == "steps":
        for _ in range(steps):
            real.sweep(case["every"])
            real.exchange(steps // 2)
    else:
        real.run(case["sweeps"], case["every"], steps // 2)
    return {"obs": real.observables(), "state": {k: v for k, v in real.get_state().items() if v is not None}}


def work(case):
    kind = case["kind"]
    if kind == "serve":
        parts = [work(dict(q, kind="run")) for q in _requests(case, 0)]
        return {k: sum(p[k] for p in parts) for k in ("bytes", "flops")}
    L, R = case["L"], case["R"]
    N = L ** 3
    field = N / 8 if case["field"] == "bimodal" else 4 * N
    if kind == "exchange":
        return {"bytes": N / 8 * R + 4 * N + 100 * R, "flops": 8.0 * N * R}
    # an attempt: a quarter of a Philox4x32-10 block (5 products, 5 xors), 6 neighbours, the field, exp, test
    sweeps = case["sweeps"] * (case["trials"] if kind == "adapt" else max(1, case.get("mh", 0)))
    flops = 20.0 * N * R * sweeps + 8.0 * N * R * (case["sweeps"] // case["every"])
    return {"bytes": field + N / 8 * R + (0 if kind == "adapt" else N * R) + 100.0 * R, "flops": flops}


# ---- the same in plain torch ------------------------------------------------------------------------

_M32 = 0xFFFFFFFF
_INIT, _METRO, _EXCH, _FIELD = 1, 2, 3, 4


def _philox(k0, k1, c):
    """Philox4x32-10 on four int64 tensors (or ints) holding 32-bit words."""
    c0, c1, c2, c3 = c
    for _ in range(10):
        p0, p1 = 0xD2511F53 * c0, 0xCD9E8D57 * c2
        c0, c1, c2, c3 = ((p1 >> 32) & _M32) ^ c1 ^ k0, p1 & _M32, ((p0 >> 32) & _M32) ^ c3 ^ k1, p0 & _M32
        k0, k1 = (k0 + 0x9E3779B9) & _M32, (k1 + 0xBB67AE85) & _M32
    return c0, c1, c2, c3


def _tag(tag, stage, colour):
    return (tag << 28) | (stage << 1) | colour


class _Plain:
    """One realization, straight from the definitions: Metropolis checkerboard sweeps and exchange steps."""

    def __init__(self, L, T, h, field, seeds, xi=False, mh=0, tile=0):
        self.L, self.N, self.h, self.xi, self.mh, self.tile = L, L ** 3, h, xi, mh, tile
        self.key = (seeds["seed"], seeds["realization"])
        dev = {"device": "cuda"}
        N = self.N
        i = torch.arange(N, **dev)
        if isinstance(field, str):
            k = (seeds["field_seed"], seeds["realization"])
            if field == "bimodal":
                w = torch.stack(self._words(k, i[: N // 4], 0, 0, _tag(_FIELD, 0, 0)), -1).reshape(-1)
                raw = torch.where(w >> 31 == 1, -1.0, 1.0).double()
            else:
                w = torch.stack(self._words(k, i[: N // 2], 1, 0, _tag(_FIELD, 0, 0)), -1).reshape(N, 2).double()
                u = (w + 0.5) / 2.0 ** 32
                raw = (torch.sqrt(-2.0 * torch.log(u[:, 0])) * torch.cos(2.0 * math.pi * u[:, 1])).float().double()
        else:
            raw = torch.from_numpy(np.asarray(field, dtype=np.float64)).cuda()
        self.raw = raw
        self.hh = (np.float32(h).item() * raw).float().double()  # the library's input is hh_i in 32 bits
        x, y, z = i % L, i // L % L, i // (L * L)
        self.xyz = (x, y, z)
        self.sites, self.nbrs, self.tiles = [], [], []
        for c in (0, 1):
            q = torch.arange(N // 2, **dev)
            qy, qz = q // (L // 2) % L, q // (L // 2) // L
            qx = 2 * (q % (L // 2)) + ((c + qy + qz) & 1)
            at = lambda a, b, d: a % L + L * (b % L + L * (d % L))  # noqa: E731
            self.sites.append(at(qx, qy, qz))
            self.nbrs.append([at(qx + 1, qy, qz), at(qx - 1, qy, qz), at(qx, qy + 1, qz), at(qx, qy - 1, qz),
                              at(qx, qy, qz + 1), at(qx, qy, qz - 1)])
            self.tiles.append((qx // tile + qy // tile + qz // tile) & 1 if mh else None)
        self.start(T, 0)

    @staticmethod
    def _words(key, c0, c1, c2, c3):
        return _philox(key[0], key[1], (c0, c1, c2, c3))

    def start(self, T, stage):
        self.T, self.R, self.stage, self.sweep, self.j = np.asarray(T, dtype=np.float64), len(T), stage, 0, 0
        R, N = self.R, self.N
        self.r = torch.arange(R, device="cuda")[:, None]
        w = torch.stack(self._words(self.key, torch.arange(N // 4, device="cuda")[None], self.r, 0, _tag(_INIT, stage, 0)), -1)
        self.s = torch.where(w.reshape(R, N) >> 31 == 1, -1, 1).to(torch.int8)
        self.t2r = np.arange(R)
        self.att, self.acc = np.zeros(R - 1, np.uint64), np.zeros(R - 1, np.uint64)
        self.sums, self.F, self.n_meas = np.zeros((R, 5)), np.zeros(R), 0

    def _half(self, c, counter, coarse=None):
        words = self._words(self.key, torch.arange(self.N // 8, device="cuda")[None], self.r, counter, _tag(_METRO, self.stage, c))
        u = torch.stack(words, -1).reshape(self.R, self.N // 2).double() / 2.0 ** 32
        n = sum(self.s[:, k] for k in self.nbrs[c])
        s = self.s[:, self.sites[c]]
        dE = 2.0 * s * (n.double() + self.hh[self.sites[c]])
        beta = np.empty(self.R)
        beta[self.t2r] = 1.0 / self.T
        ok = (dE <= 0) | (u < torch.exp(-torch.from_numpy(beta).cuda()[:, None] * dE))
        if coarse is not None:
            ok &= self.tiles[c] == coarse
        self.s[:, self.sites[c]] = torch.where(ok, -s, s)

    def one_sweep(self):
        counter = self.sweep & _M32
        if self.mh:
            for coarse in (0, 1):
                for hit in range(self.mh):
                    for c in (0, 1):
                        self._half(c, (counter * self.mh + hit) & _M32, coarse)
        else:
            for c in (0, 1):
                self._half(c, counter)
        self.sweep += 1

    def energies(self):
        s = self.s.view(self.R, self.L, self.L, self.L)
        B = sum((s * torch.roll(s, -1, d)).sum((1, 2, 3), dtype=torch.int64) for d in (1, 2, 3))
        E = -B.double() - (self.s.double() * self.hh).sum(1)
        return E.cpu().numpy(), self.s.sum(1, dtype=torch.int64).cpu().numpy()

    def exchange(self, measure_from):
        E, M = self.energies()
        beta = 1.0 / self.T
        for k in range(self.j % 2, self.R - 1, 2):
            a, b = self.t2r[k], self.t2r[k + 1]
            delta = (beta[k] - beta[k + 1]) * (E[a] - E[b])
            u = self._words(self.key, k, 0, self.j & _M32, _tag(_EXCH, self.stage, 0))[0] / 2.0 ** 32
            self.att[k] += 1
            if delta >= 0 or u < math.exp(delta):
                self.acc[k] += 1
                self.t2r[k], self.t2r[k + 1] = b, a
        if self.j >= measure_from:
            e, m = E[self.t2r] / self.N, M[self.t2r] / self.N
            self.sums += np.stack([e, e * e, np.abs(m), m * m, m ** 4], 1)
            self.n_meas += 1
            if self.xi:
                self.F += self._structure()[self.t2r]
        self.j += 1
        return E, M

    def _structure(self):
        s = self.s.view(self.R, self.L, self.L, self.L).double()
        t = torch.arange(self.L, device="cuda").double() * (2.0 * math.pi / self.L)
        F = sum((m @ torch.cos(t)) ** 2 + (m @ torch.sin(t)) ** 2 for m in (s.sum((1, 2)), s.sum((1, 3)), s.sum((2, 3))))
        return (F / (3.0 * self.N)).cpu().numpy()

    def run(self, sweeps, every, measure_from):
        for _ in range(sweeps):
            self.one_sweep()
            if self.sweep % every == 0:
                self.exchange(measure_from)

    def observables(self):
        out = {k: self.sums[:, i].copy() for i, k in enumerate(("e", "e2", "absm", "m2", "m4"))}
        out.update(T=self.T, F=self.F, att=self.att, acc=self.acc, n_meas=self.n_meas, sums=self.sums)
        return out


def _follows(field, attempts, half_sweeps):
    """Whether a trajectory can be followed in 64 bits in the time there is.  Bimodal decisions are exact; with a
    float field a 32-bit decision differs from the 64-bit one about once in 10^7, after which the paths part."""
    return attempts <= (3e9 if field == "bimodal" else 2e6) and half_sweeps <= 8000


def exact(case, seed):
    kind = case["kind"]
    if kind == "exchange":
        return _exact_exchange(case, seed)
    if kind == "serve":
        reqs = _requests(case, seed)
        if not _follows(case["field"], sum(q["L"] ** 3 * q["R"] * q["sweeps"] for q in reqs), 2 * case["sweeps"] * case["n"]):
            return None
        got = []
        for q in reqs:
            p = _Plain(q["L"], inputs.geometric_temps(1.0, 5.0, q["R"]), q["h"], q["field"], q["seeds"], q["xi"])
            p.run(q["sweeps"], q["every"], q["sweeps"] // q["every"] // 2)
            got.append(p.observables())
        return {k: np.concatenate([g[k] for g in got]) for k in ("T", "e", "e2", "absm", "m2", "m4", "F", "att", "acc")}
    N, mh = case["L"] ** 3, case.get("mh", 0)
    total = case["sweeps"] * (case["trials"] if kind == "adapt" else 1)
    if not _follows(case["field"], N * case["R"] * total * max(1, mh), total * (4 * mh if mh else 2)):
        return None
    own = _field(case, seed)
    p = _Plain(case["L"], _temps(case), case["h"], case["field"] if own is None else own, _seeds(seed), case.get("xi", False),
               mh, case.get("tile", 0))
    if kind == "adapt":
        T = p.T
        rates = np.zeros((case["trials"], case["R"] + case["trials"] * case["inserts"]))
        for t in range(1, case["trials"] + 1):
            p.start(T, t)
            p.run(case["sweeps"], case["every"], 1 << 62)
            rate = np.where(p.att > 0, p.acc / np.maximum(p.att, 1), 0.0)
            rates[t - 1, : len(rate)] = rate
            low = np.argsort(rate, kind="stable")[: case["inserts"]]
            T = np.sort(np.concatenate([T, 0.5 * (T[low] + T[low + 1])]))
        return {"temps": T, "rates": rates}
    steps = case["sweeps"] // case["every"]
    p.run(case["sweeps"], case["every"], steps // 2)
    return {"obs": p.observables(), "state": {"spins": p.s.cpu().numpy(), "t2r": p.t2r.astype(np.int32),
                                              "sweep": p.sweep, "xstep": p.j}}


def _exact_exchange(case, seed):
    L, R = case["L"], case["R"]
    bits, field, _ = _exchange_inputs(case, seed)
    p = _Plain(L, inputs.geometric_temps(1.0, 5.0, R), case["h"], field.cpu().numpy(), _seeds(seed))
    up = (bits[..., None] >> torch.arange(32, device="cuda")) & 1  # [R][2][words][bit]
    k = torch.arange(32, device="cuda")
    flat = up[..., 8 * (k & 3) + (k >> 2)].reshape(R, 2, -1)  # site q of a colour: word q >> 5, position q & 31
    for c in (0, 1):
        p.s[:, p.sites[c]] = (2 * flat[:, c] - 1).to(torch.int8)
    E, M = p.exchange(0)
    r2t = np.empty(R, np.int32)
    r2t[p.t2r] = np.arange(R)
    return {"t2r": p.t2r.astype(np.int32), "r2t": r2t, "att": p.att.astype(np.int64), "acc": p.acc.astype(np.int64),
            "obs": p.sums, "n_meas": np.array([p.n_meas]), "E": E, "M": M}

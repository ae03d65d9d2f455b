"""Performance cases: the work users of this library have it do.

A case is one call (or one short, fixed sequence of calls) through the public
Python binding, over the sizes that the repository's workloads use
(paper_1003_1898_gb300/workloads.py: the small configuration of 256 streams,
the roofline bulk fill, the luxury sweep, the jump fills, the batched requests
and the serving clients) and ragged sizes between them.  Kinds:

  fill   every stream of one handle draws n_per outputs (u32, f32 or f64)
  jump   one long sequence filled in parallel by jump-ahead
  batch  many fill requests of uneven lengths in one graph launch, each
         re-seeding its own handle first
  tick   one tick of a serving loop: the fills of several resident clients in
         one batcher launch, then four Ising half-sweeps of the clients that
         run a lattice
  fused  one sweep (both colours) of an Ising lattice whose draws are consumed
         where they are made

Launch tiles are the library's defaults.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_1003_1898_gb300 as P
from paper_1003_1898_gb300 import workloads as W

SHIFT = {"ggl": 7, "xor128": 8, "ranecu": 7, "ranmar": 0, "ranlux": 0, "mt19937": 8}
HALF_SWEEPS = 4                      # half-sweeps a running lattice advances per tick
MAX_NUMBERS = 2**30                  # draws of the largest fill or jump


def listed():
    return [
        # The smallest call: a few hundred walkers ask for one short row each.
        {"name": "fill_ggl_u32_256x16", "kind": "fill", "gen": "ggl", "lux": 0, "dtype": "u32",
         "streams": 256, "per": 16},
        # The small configuration: a modest simulation's floats, few streams, longer rows.
        {"name": "fill_xor128_f32_256x4096", "kind": "fill", "gen": "xor128", "lux": 0, "dtype": "f32",
         "streams": 256, "per": 4096},
        # A serving client of high-luxury RANLUX drawing about a million numbers.
        {"name": "fill_ranlux223_f32_4096x248", "kind": "fill", "gen": "ranlux", "lux": 223, "dtype": "f32",
         "streams": 4096, "per": 248},
        # Ragged sizes: odd rows, streams that fill no block, the third generator family.
        {"name": "fill_ranmar_u32_10007x1001", "kind": "fill", "gen": "ranmar", "lux": 0, "dtype": "u32",
         "streams": 10007, "per": 1001},
        # The roofline bulk fill of a combined generator.
        {"name": "fill_ranecu_f32_131072x8192", "kind": "fill", "gen": "ranecu", "lux": 0, "dtype": "f32",
         "streams": 131072, "per": 8192},
        # The roofline bulk fill of the Mersenne twister.
        {"name": "fill_mt19937_u32_8192x131072", "kind": "fill", "gen": "mt19937", "lux": 0, "dtype": "u32",
         "streams": 8192, "per": 131072},
        # The luxury sweep's highest standard level.
        {"name": "fill_ranlux389_f32_65536x4096", "kind": "fill", "gen": "ranlux", "lux": 389, "dtype": "f32",
         "streams": 65536, "per": 4096},
        # Doubles for a double-precision integration.
        {"name": "fill_xor128_f64_65536x2048", "kind": "fill", "gen": "xor128", "lux": 0, "dtype": "f64",
         "streams": 65536, "per": 2048},
        # One serial Mersenne-twister sequence, as a serial program would draw it, in parallel.
        {"name": "jump_mt19937_u32_2e28", "kind": "jump", "gen": "mt19937", "dtype": "u32",
         "n": 2**28, "chunks": 8192},
        # A tenth of the batched workload: 2,000 mixed requests of 10^2 to 10^7 numbers.
        {"name": "batch_2000", "kind": "batch", "requests": 2000, "max_len": 10**7},
        # A busy tick of the serving loop: 48 resident clients, half of them RANLUX p = 223.
        {"name": "tick_48", "kind": "tick", "clients": 48},
        # A sweep of the largest serving lattice without a draw buffer.
        {"name": "fused_ranmar_4096", "kind": "fused", "gen": "ranmar", "lux": 0, "L": 4096,
         "streams": 65536},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["fill"] * 6 + ["jump", "batch", "tick", "fused"])
    if kind == "fill":
        gen = rng.choice(W.GENS)
        lux = rng.choice(W.LUXURY_LEVELS) if gen == "ranlux" else 0
        streams = _log_int(rng, 256, 8192 if gen == "mt19937" else 131072)
        per = _log_int(rng, 16, 131072 if gen == "mt19937" else 8192)
        if rng.random() < 0.6:          # rows that start on 16-byte boundaries, and rows that do not
            per = 4 * -(-per // 4)
        dtype = rng.choice(["u32", "f32", "f32", "u32", "f64"])
        if dtype == "f64":
            per = max(8, per // 2)
        return {"kind": kind, "gen": gen, "lux": lux, "dtype": dtype, "streams": streams, "per": per}
    if kind == "jump":
        gen = rng.choice(["ggl", "ranecu", "xor128", "mt19937"])
        n = _log_int(rng, 10**5, 2**28 if gen == "mt19937" else MAX_NUMBERS)
        return {"kind": kind, "gen": gen, "dtype": rng.choice(["u32", "f32"]), "n": n,
                "chunks": _log_int(rng, 64, 8192 if gen == "mt19937" else 65536)}
    if kind == "batch":
        return {"kind": kind, "requests": _log_int(rng, 100, 2000),
                "max_len": _log_int(rng, 10**5, 10**7)}
    if kind == "tick":
        return {"kind": kind, "clients": rng.randrange(4, 49)}
    gen = rng.choice(W.GENS)
    return {"kind": kind, "gen": gen, "lux": 223 if gen == "ranlux" else 0, "L": rng.choice([256, 1024, 4096]),
            "streams": rng.choice([512, 1024, 4096]) if gen == "mt19937" else rng.choice([4096, 16384, 32768])}


# ------------------------------------------------------------------ states

def _base_seed(seed):
    return (W.SEED_BASE + (int(seed) << 33)) & (2**64 - 1)


def _jump_x0(gen, seed):
    s = (int(seed) * 2654435761 + 12345) & 0xFFFFFFFF
    if gen == "ggl":
        return 1 + s % (2**31 - 2)
    if gen == "ranecu":
        return (1 + s % 2147483562) | ((1 + (s * 69069 + 1) % 2147483398) << 32)
    return s


def _round4(n):
    return 4 * -(-n // 4)


def _batch_requests(case, seed):
    reqs = W.batched_requests(case["requests"], max_len=case["max_len"])   # lengths and generators: the case's
    for r in reqs:                                                         # stream seeds: the seed's
        r["seed"] = (r["seed"] + (int(seed) << 48)) & (2**64 - 1)
    return reqs


def _tick_plan(case, seed):
    """Clients of a tick and what each asks for: the serving workload's clients,
    lattices and fill lengths in its proportions (a fill takes the whole block
    of its streams' next draws)."""
    rng = np.random.default_rng(0x71C0 + case["clients"])    # the shape of the tick: same for every seed
    specs = W.serving_clients(case["clients"], seed=(int(seed) << 40) + 0x5E5E)
    plan = []
    for c, (gen, lux, s) in enumerate(specs):
        # every other pair of clients runs a lattice, so both halves hold RANLUX and other clients
        ising = (c // 2) % 2 == 1
        ln = int(10.0 ** rng.uniform(3, 6))
        per = _round4(-(-ln // W.SERVE_STREAMS))
        plan.append({"gen": gen, "lux": lux, "seed": s, "ising": ising, "per": per, "n": per * W.SERVE_STREAMS,
                     "f32": bool(rng.integers(0, 2)), "L": W.SERVE_ISING_L[int(rng.integers(0, 3))]})
    # clients' generators are drawn from the seed; the tick's cost should not be
    others = [g for g in W.GENS if g != "ranlux"]
    for c, p in enumerate(plan):
        p["gen"], p["lux"] = ("ranlux", 223) if c % 2 == 0 else (others[(c // 2) % len(others)], 0)
    return plan


class _Batch:
    """A planned batch and the handles it fills, released together."""

    def __init__(self, reqs):
        self.handles = [P.prng_create(r["gen"], r["seed"], r["n_streams"], r["luxury"]) for r in reqs]
        size = {True: 0, False: 0}
        at = []
        for r in reqs:
            at.append(size[r["f32"]])
            size[r["f32"]] += _round4(r["n"])
        self.out = {True: torch.zeros(max(4, size[True]), dtype=torch.float32, device="cuda"),
                    False: torch.zeros(max(4, size[False]), dtype=torch.int32, device="cuda")}
        self.batch = P.prng_batch_create([
            {"st": h, "d_out": self.out[r["f32"]].data_ptr() + 4 * a, "n_per_stream": r["n_per"],
             "n_valid": r["n"], "seed": r["seed"], "f32": r["f32"], "reseed": True}
            for h, r, a in zip(self.handles, reqs, at)])

    def __del__(self):
        torch.cuda.synchronize()
        P.prng_batch_destroy(self.batch)
        for h in self.handles:
            P.prng_destroy(h)


class _Tick:
    """Resident clients with their launch rows, as the serving loop keeps them."""

    def __init__(self, plan):
        n = W.SERVE_STREAMS
        t4, t8 = P.prng_ising_thresholds(0.4406868)
        self.gens = [P.Generator(p["gen"], p["seed"], n, p["lux"]) for p in plan]
        size = {"f32": 0, "u32": 0, "spins": 0, "draws": 0}
        place = []
        for p in plan:
            if p["ising"]:
                place.append((size["spins"], size["draws"]))
                size["spins"] += p["L"] * p["L"]
                size["draws"] += HALF_SWEEPS * (p["L"] * p["L"] // 2)
            else:
                k = "f32" if p["f32"] else "u32"
                place.append((size[k],))
                size[k] += p["n"]
        self.out = {"f32": torch.zeros(max(4, size["f32"]), dtype=torch.float32, device="cuda"),
                    "u32": torch.zeros(max(4, size["u32"]), dtype=torch.int32, device="cuda"),
                    "spins": torch.ones(max(16, size["spins"]), dtype=torch.int8, device="cuda")}
        self.draws = torch.empty(max(4, size["draws"]), dtype=torch.int32, device="cuda")
        self.fills = np.zeros(len(plan), P.FILL_REQ_DTYPE)
        steps = [[] for _ in range(HALF_SWEEPS)]
        for i, (p, g, at) in enumerate(zip(plan, self.gens, place)):
            if p["ising"]:
                per = p["L"] * p["L"] // (2 * n)
                sp, dp = self.out["spins"].data_ptr() + at[0], self.draws.data_ptr() + 4 * at[1]
                self.fills[i] = (g.handle.value, dp, HALF_SWEEPS * per, 0, 0, 0, 0)
                for t in range(HALF_SWEEPS):
                    steps[t].append((sp, dp + 4 * t * per, p["L"], t & 1, P.prng_float_shift(p["gen"]),
                                     t4, t8, per, HALF_SWEEPS * per))
            else:
                d = self.out["f32" if p["f32"] else "u32"].data_ptr() + 4 * at[0]
                self.fills[i] = (g.handle.value, d, p["per"], 0, 0, int(p["f32"]), 0)
        self.steps = [np.array(s, P.ISING_REQ_DTYPE) for s in steps if s]
        self.batcher = P.prng_batcher_create(len(plan), len(plan) * (n // 2) + 1024)

    def __del__(self):
        torch.cuda.synchronize()
        P.prng_batcher_destroy(self.batcher)


def prepare(case, seed):
    kind = case["kind"]
    if kind == "fill":
        dt = {"u32": torch.int32, "f32": torch.float32, "f64": torch.float64}[case["dtype"]]
        return {"kind": kind, "gen": P.Generator(case["gen"], _base_seed(seed), case["streams"], case["lux"]),
                "out": torch.empty((case["streams"], case["per"]), dtype=dt, device="cuda"),
                "per": case["per"], "dtype": case["dtype"]}
    if kind == "jump":
        dt = torch.float32 if case["dtype"] == "f32" else torch.int32
        return {"kind": kind, "call": P.prng_fill_jump_f32 if case["dtype"] == "f32" else P.prng_fill_jump_u32,
                "gen": case["gen"], "x0": _jump_x0(case["gen"], seed), "n": case["n"], "chunks": case["chunks"],
                "out": torch.empty(case["n"], dtype=dt, device="cuda")}
    if kind == "batch":
        return {"kind": kind, "work": _Batch(_batch_requests(case, seed))}
    if kind == "tick":
        return {"kind": kind, "work": _Tick(_tick_plan(case, seed))}
    t4, t8 = P.prng_ising_thresholds(0.4406868)
    L = case["L"]
    return {"kind": kind, "gen": P.Generator(case["gen"], _base_seed(seed), case["streams"], case["lux"]),
            "spins": torch.ones((L, L), dtype=torch.int8, device="cuda"), "L": L, "t4": t4, "t8": t8}


def run(state):
    kind = state["kind"]
    if kind == "fill":
        return state["gen"].fill(state["per"], state["dtype"], out=state["out"])
    if kind == "jump":
        state["call"](state["gen"], state["x0"], state["n"], state["chunks"], state["out"])
        return state["out"]
    if kind == "batch":
        w = state["work"]
        P.prng_batch_launch(w.batch)
        return {"u32": w.out[False], "f32": w.out[True]}
    if kind == "tick":
        w = state["work"]
        P.prng_batcher_launch(w.batcher, w.fills)
        for rows in w.steps:
            P.prng_ising_half_sweep(rows)
        return w.out
    for colour in (0, 1):
        P.prng_ising_fused(state["gen"].handle, state["spins"], state["L"], colour, state["t4"], state["t8"])
    return state["spins"]


def _state_bytes(gen, streams):
    return 4 * streams * P.STATE_WORDS[P.GEN_IDS[gen]]


def work(case):
    """Outputs written once; resident stream states read and written once."""
    kind = case["kind"]
    if kind == "fill":
        out = case["streams"] * case["per"] * (8 if case["dtype"] == "f64" else 4)
        b = out + 2 * _state_bytes(case["gen"], case["streams"])
    elif kind == "jump":
        b = 4 * case["n"]
    elif kind == "batch":   # the states are seeded in the pass, then written back
        b = sum(4 * r["n"] + _state_bytes(r["gen"], r["n_streams"]) for r in _batch_requests(case, 0))
    elif kind == "tick":    # lattices read and written per half-sweep
        b = 0
        for p in _tick_plan(case, 0):
            b += 2 * _state_bytes(p["gen"], W.SERVE_STREAMS)
            b += HALF_SWEEPS * 2 * p["L"] ** 2 if p["ising"] else 4 * p["n"]
    else:
        b = 2 * (2 * case["L"] ** 2 + 2 * _state_bytes(case["gen"], case["streams"]))
    return {"bytes": b, "flops": 0}


# ------------------------------------------------------------------ expected values
#
# The generators' recurrences (Sections 3.2 to 3.7 and Appendix A of the
# paper) step by step over all streams at once, in 64-bit integers.

_U64 = np.uint64


def _splitmix64(x):
    with np.errstate(over="ignore"):
        z = x + _U64(0x9E3779B97F4A7C15)
        z = (z ^ (z >> _U64(30))) * _U64(0xBF58476D1CE4E5B9)
        z = (z ^ (z >> _U64(27))) * _U64(0x94D049BB133111EB)
    return z ^ (z >> _U64(31))


def _stream_seeds(case, seed):
    with np.errstate(over="ignore"):
        s = _splitmix64(_U64(_base_seed(seed)) + np.arange(case["streams"], dtype=_U64))
    return s, (s & _U64(0xFFFFFFFF)).astype(np.int64), (s >> _U64(32)).astype(np.int64)


def _dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def _ggl(case, seed):
    s, _, _ = _stream_seeds(case, seed)
    x = _dev((_U64(1) + s % _U64(2**31 - 2)).astype(np.int64))
    while True:
        x = x * 16807 % (2**31 - 1)
        yield x


def _xor128(case, seed):
    s, lo, hi = _stream_seeds(case, seed)
    t = _splitmix64(s)
    x, y = _dev(lo), _dev(hi)
    z, w = _dev((t & _U64(0xFFFFFFFF)).astype(np.int64)), _dev((t >> _U64(32)).astype(np.int64))
    while True:
        u = x ^ ((x << 11) & 0xFFFFFFFF)
        x, y, z, w = y, z, w, w ^ (w >> 19) ^ u ^ (u >> 8)
        yield w


def _ranecu(case, seed):
    _, lo, hi = _stream_seeds(case, seed)
    m1, m2 = 2147483563, 2147483399
    a, b = _dev(1 + lo % (m1 - 1)), _dev(1 + hi % (m2 - 1))
    while True:
        a, b = a * 40014 % m1, b * 40692 % m2
        z = a - b
        yield torch.where(z < 1, z + (m1 - 1), z)


def _ranmar(case, seed):
    _, lo, hi = _stream_seeds(case, seed)
    ij, kl = _dev(lo % 31329), _dev(hi % 30082)
    i, j, k, m = (ij // 177) % 177 + 2, ij % 177 + 2, (kl // 169) % 178 + 1, kl % 169
    u = [None] * 98
    for e in range(1, 98):
        acc = torch.zeros_like(i)
        for _ in range(24):
            t = i * j % 179 * k % 179
            i, j, k = j, k, t
            m = (53 * m + 1) % 169
            acc = 2 * acc + (m * t % 64 >= 32)
        u[e] = acc
    c, p, q = 362436, 97, 33
    while True:
        v = (u[p] - u[q]) & 0xFFFFFF
        u[p] = v
        p, q = p - 1 or 97, q - 1 or 97
        c = c - 7654321
        c += 16777213 if c < 0 else 0
        yield (v - c) & 0xFFFFFF


def _ranlux(case, seed):
    s, _, _ = _stream_seeds(case, seed)
    v = (s % _U64(2147483563)).astype(np.int64)
    v[v == 0] = 19780503
    x, ring = _dev(v), []
    for _ in range(24):
        x = x * 40014 % 2147483563
        ring.append((x & 0xFFFFFF).to(torch.int32))
    c = (ring[23] == 0).to(torch.int32)
    at, n = 0, 0
    while True:
        t = ring[(at + 14) % 24] - ring[at] - c
        c = (t >> 31) & 1
        ring[at] = t & 0xFFFFFF
        if n % case["lux"] < 24:
            yield ring[at].to(torch.int64)
        at, n = (at + 1) % 24, n + 1


def _mt19937(case, seed):
    _, lo, _ = _stream_seeds(case, seed)
    v = _dev(lo)
    mt = torch.empty((624, case["streams"]), dtype=torch.int64, device="cuda")
    for k in range(624):
        mt[k] = v
        v = (1812433253 * (v ^ (v >> 30)) + k + 1) & 0xFFFFFFFF

    def mix(a, b, far):
        y = (a & 0x80000000) | (b & 0x7FFFFFFF)
        return far ^ (y >> 1) ^ (y & 1) * 0x9908B0DF

    while True:
        for a, b in ((0, 227), (227, 454), (454, 623)):
            far = mt[a + 397:b + 397] if a == 0 else mt[a - 227:b - 227]
            mt[a:b] = mix(mt[a:b], mt[a + 1:b + 1], far)
        mt[623] = mix(mt[623], mt[0], mt[396])
        y = mt ^ (mt >> 11)
        y = y ^ (y << 7) & 0x9D2C5680
        y = y ^ (y << 15) & 0xEFC60000
        y = y ^ (y >> 18)
        for k in range(624):
            yield y[k]


_STEP = {"ggl": _ggl, "xor128": _xor128, "ranecu": _ranecu, "ranmar": _ranmar, "ranlux": _ranlux,
         "mt19937": _mt19937}


def exact(case, seed):
    """Float fills: the exact scaling of the integers.  The rest are whole numbers."""
    if case["kind"] != "fill" or case["dtype"] == "u32":
        return None
    gen, n, per = case["gen"], case["streams"], case["per"]
    out = torch.empty((per, n), dtype=torch.float64, device="cuda")
    seq = _STEP[gen](case, seed)
    if case["dtype"] == "f32":
        for k in range(per):
            out[k] = (next(seq) >> SHIFT[gen]).double() * 2.0**-24
    else:
        for k in range(per):
            a, b = next(seq), next(seq)
            if gen in ("ranmar", "ranlux"):
                out[k] = (a * 2**24 + b).double() * 2.0**-48
            else:
                drop = 4 if gen in ("ggl", "ranecu") else 5
                out[k] = ((a >> drop) * 2**26 + (b >> (drop + 1))).double() * 2.0**-53
    return out.t()

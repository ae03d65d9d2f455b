"""Continuous-batching serving loop over device-resident client streams.

Each client owns a handle (one generator, n_streams streams) whose state
stays on the device between requests.  A request is either a fill of n
numbers (the first n of the client's next stream-major block, n_per =
ceil(n / n_streams) draws per stream) or an Ising run: `sweeps` checkerboard
Metropolis sweeps of an L x L lattice (cold start), every half-sweep
consuming the client's next L*L/2 draws (L*L/(2 n_streams) per stream).

The loop works in ticks.  A tick admits arrived requests in arrival order
while their client is free and the state-plus-output memory stays under the
cap, advances every running Ising request by up to `half_sweeps_per_tick`
half-sweeps, and enqueues one batched fill (prng_batcher_launch: the new
fills plus, per running Ising request, one fill holding the draws of all its
half-sweeps of the tick, each half-sweep's block a column range of the
stream rows) and then one batched half-sweep launch (prng_ising_half_sweep)
per half-sweep step on the server's stream.  Up to `max_inflight` ticks
are on the GPU while the host forms the next, so requests that arrive while
others run join the next tick.  A client's requests are served in order and
only its own requests touch its streams, so every result is the same as the
client would get alone.  Latency = completion (the end event of the tick
that finishes the request, on the device clock) - arrival.
"""
from __future__ import annotations

import collections
import dataclasses
import time

from . import (FILL_REQ_DTYPE, GEN_IDS, ISING_REQ_DTYPE, prng_batcher_create,
               prng_batcher_destroy, prng_batcher_launch, prng_create, prng_destroy, prng_info,
               prng_float_shift, prng_ising_half_sweep, prng_ising_thresholds)

ISING_BETA = 0.4406868


@dataclasses.dataclass
class Request:
    rid: int
    client: int
    kind: str                  # "fill" or "ising"
    arrival: float = 0.0       # seconds after the start of the run
    n: int = 0                 # fill: numbers wanted
    f32: bool = False          # fill: float output
    L: int = 0                 # ising: lattice side
    sweeps: int = 16           # ising: full sweeps
    # filled in by the server
    out: object = None         # fill output (CUDA tensor), kept when the server keeps results
    spins: object = None       # ising lattice (CUDA int8 tensor)
    draws: object = None
    half_done: int = 0
    done: float = None         # completion time, seconds after the start
    numbers: int = 0           # draws this request consumed


class Client:
    def __init__(self, cid: int, gen, luxury: int, seed: int, n_streams: int):
        self.cid = cid
        self.gen = GEN_IDS[gen] if isinstance(gen, str) else int(gen)
        self.luxury = luxury
        self.n_streams = n_streams
        self.handle = prng_create(self.gen, seed, n_streams, luxury)
        self.state_bytes = prng_info(self.handle)["state_bytes"]
        self.shift = prng_float_shift(self.gen)   # 24-bit acceptance value = draw >> shift
        self.busy = None           # running Ising request

    def close(self):
        if self.handle is not None:
            prng_destroy(self.handle)
            self.handle = None


class Server:
    def __init__(self, client_specs, n_streams: int = 1024, mem_cap: float = 40e9,
                 max_inflight: int = 2, beta: float = ISING_BETA, keep_results: bool = False,
                 max_active: int = 0, half_sweeps_per_tick: int = 4, scan_limit: int = 1024):
        """max_active > 0 caps the requests in progress (1 = a plain FIFO queue,
        one request at a time, the baseline continuous batching is measured
        against).  half_sweeps_per_tick: Ising half-sweeps a running request
        advances per tick (one fill holds all their draws, read as column
        blocks of the stream rows).  The host work of a tick -- gathering
        the launch rows, planning the batcher's work items, launching --
        is what bounds the loop at saturation, so more half-sweeps per tick
        raise throughput; with clients of 4,096 streams they lowered the
        latency at moderate load too (4 against 1: p50/p99 1.8/9.2 against
        3.0/13.6 ms at 2,000 requests/s).  mem_cap counts
        states, lattices, draws and outputs; the library's own scratch (four
        launches' descriptors and work items, and RANLUX segment starts from a
        pool that keeps 1 GiB at most) lies outside it.  scan_limit: pending requests
        examined for admission per tick (in arrival order); the rest wait,
        so the host work of a tick stays bounded when the queue is long."""
        import torch
        self.torch = torch
        self.clients = [Client(i, g, lux, seed, n_streams)
                        for i, (g, lux, seed) in enumerate(client_specs)]
        self.n_streams = n_streams
        self.mem_cap = mem_cap
        self.mem_state = sum(c.state_bytes for c in self.clients)
        self.mem_used = self.mem_state
        self.max_inflight = max_inflight
        self.max_active = max_active
        self.hpt = max(1, int(half_sweeps_per_tick))
        self.scan_limit = max(1, int(scan_limit))
        self.keep = keep_results
        self.t4, self.t8 = prng_ising_thresholds(beta)
        self.stream = torch.cuda.Stream()
        # every client contributes at most one fill per tick; items per
        # request are at most n_streams / 2 (MT19937 takes 2 streams per item)
        self.batcher = prng_batcher_create(len(self.clients),
                                           len(self.clients) * max(1, n_streams // 2) + 1024)

    def close(self):
        if self.batcher is not None:
            self.stream.synchronize()
            prng_batcher_destroy(self.batcher)
            self.batcher = None
        for c in self.clients:
            c.close()

    # ------------------------------------------------------------------ sizes
    def fill_shape(self, n):
        """Draws per stream and block size of a fill of n numbers: ceil(n /
        n_streams) rounded up to a multiple of 4 (16-byte row starts, so the
        kernels keep their vector stores); the first n are the output."""
        per = 4 * -(-(-(-n // self.n_streams)) // 4)
        return per, self.n_streams * per

    def request_bytes(self, r: Request) -> int:
        """Device bytes a request holds while it runs (counted against the cap)."""
        if r.kind == "fill":
            return 4 * self.fill_shape(r.n)[1]
        return r.L * r.L + self.hpt * 2 * r.L * r.L   # int8 lattice + draws of hpt half-sweeps

    # ------------------------------------------------------------------ run
    def run(self, requests, realtime: bool = True):
        """Serve `requests` (sorted by arrival).  With realtime the loop
        releases each request at its arrival time; otherwise all are
        available at once.  Returns the requests with their completion
        times.

        Each request's launch rows (its fill descriptor, and for an Ising
        run its half-sweep descriptors of either colour) are written once,
        at admission, into numpy tables laid out as the library's structs;
        a tick gathers the rows of the running requests with array
        indexing, so its host cost does not grow with Python work per
        request."""
        import numpy as np
        torch = self.torch
        reqs = sorted(requests, key=lambda r: (r.arrival, r.rid))
        for r in reqs:
            if r.kind == "ising":
                if r.L % 2 or (r.L * r.L) % (2 * self.n_streams):
                    raise ValueError("L*L/2 must be a multiple of the client's stream count")
            elif r.n <= 0:
                raise ValueError("fill requests need n > 0")
        n_req = len(reqs)
        # host time of the ticks' launch sections (gather + batcher + half-sweeps)
        self.stats = {"ticks": 0, "launch_s": 0.0, "batcher_s": 0.0, "gpu_s": 0.0}
        tick_events = []                       # (start, end) of each tick's GPU work
        fill_tab = np.zeros(n_req, FILL_REQ_DTYPE)           # row of request i
        ising_tab = np.zeros((n_req, 2), ISING_REQ_DTYPE)    # its half-sweeps, colour 0 / 1
        per_tab = np.zeros(n_req, np.int64)                  # Ising draws per stream and half-sweep
        half_done = np.zeros(n_req, np.int64)
        half_total = np.zeros(n_req, np.int64)
        pending = collections.deque()
        inflight = collections.deque()         # (end event, [requests finishing])
        nxt = 0
        t_start = torch.cuda.Event(enable_timing=True)
        with torch.cuda.stream(self.stream):
            t_start.record(self.stream)
        wall0 = time.perf_counter()
        running = np.zeros(0, np.int64)        # Ising requests in progress (indices into reqs)
        left = n_req
        hpt = self.hpt
        sid = self.stream.cuda_stream

        def retire(block: bool):
            nonlocal left
            while inflight and (block or inflight[0][0].query()):
                ev, finishing = inflight.popleft()
                ev.synchronize()
                t = t_start.elapsed_time(ev) / 1e3
                for r in finishing:
                    r.done = t
                    left -= 1
                    self.mem_used -= self.request_bytes(r)
                    if not self.keep:
                        r.out = r.spins = None
                    r.draws = None
                block = False

        while left > 0:
            now = time.perf_counter() - wall0
            while nxt < n_req and (not realtime or reqs[nxt].arrival <= now):
                pending.append(nxt)
                nxt += 1
            retire(False)
            if len(inflight) >= self.max_inflight:
                retire(True)
                continue
            new_fills, new_ising, finishing = [], [], []
            taken = set()                      # clients admitted this tick (one request each)
            keep = collections.deque()
            active = len(running) + sum(len(f) for _, f in inflight)
            scanned = 0
            while pending:                      # admission in arrival order
                if scanned == self.scan_limit or (self.max_active and active >= self.max_active):
                    break                       # the rest keep their places in the queue
                scanned += 1
                i = pending.popleft()
                r = reqs[i]
                c = self.clients[r.client]
                need = self.request_bytes(r)
                active += 1
                if r.client in taken or c.busy is not None or self.mem_used + need > self.mem_cap:
                    keep.append(i)
                    taken.add(r.client)         # a client's later requests wait behind this one
                    continue
                taken.add(r.client)
                self.mem_used += need
                with torch.cuda.stream(self.stream):
                    if r.kind == "fill":
                        per, total = self.fill_shape(r.n)
                        r.out = torch.empty(total, dtype=torch.float32 if r.f32 else torch.int32,
                                            device="cuda")
                        fill_tab[i] = (c.handle.value, r.out.data_ptr(), per, r.n, 0, int(r.f32), 0)
                        r.numbers = r.n
                        new_fills.append(i)
                        finishing.append(r)
                    else:
                        per = r.L * r.L // (2 * self.n_streams)
                        r.spins = torch.ones((r.L, r.L), dtype=torch.int8, device="cuda")
                        r.draws = torch.empty(hpt * (r.L * r.L // 2), dtype=torch.int32,
                                              device="cuda")
                        sp, dp = r.spins.data_ptr(), r.draws.data_ptr()
                        fill_tab[i] = (c.handle.value, dp, per, 0, 0, 0, 0)
                        for colour in (0, 1):
                            ising_tab[i, colour] = (sp, dp, r.L, colour, c.shift, self.t4,
                                                    self.t8, per, 0)
                        per_tab[i] = per
                        half_total[i] = 2 * r.sweeps
                        half_done[i] = 0
                        r.numbers = r.sweeps * r.L * r.L
                        c.busy = r
                        new_ising.append(i)
            keep.extend(pending)
            pending = keep
            if new_ising:
                running = np.concatenate([running, np.asarray(new_ising, np.int64)])
            if not new_fills and not len(running):   # nothing to launch now
                future = realtime and nxt < n_req
                if inflight and not future:
                    retire(True)                # only completions can free slots or memory
                elif future:
                    wait = reqs[nxt].arrival - (time.perf_counter() - wall0)
                    if wait > 0:
                        time.sleep(min(wait, 5e-5 if inflight else 1e-3))
                elif not inflight and pending:
                    raise RuntimeError("a request does not fit the memory cap")
                continue
            # One fill per running Ising request holding its next h half-sweeps'
            # draws (row pitch h * per), then half-sweep t of every lattice reads
            # column block t of its rows.
            t_tick = time.perf_counter()
            R = running
            h = np.minimum(hpt, half_total[R] - half_done[R])
            fills = fill_tab[R]
            fills["n_per_stream"] = h * per_tab[R]
            steps = []
            for t in range(hpt):
                m = h > t
                if not m.any():
                    break
                Rt = R[m]
                st = ising_tab[Rt, (half_done[Rt] + t) & 1]
                if hpt > 1:
                    st["d_draws"] += (4 * t * per_tab[Rt]).astype(np.uint64)
                    st["pitch"] = np.where(h[m] > 1, h[m] * per_tab[Rt], 0)
                steps.append(st)
            half_done[R] += h
            done_mask = half_done[R] == half_total[R]
            if new_fills:
                fills = np.concatenate([fill_tab[np.asarray(new_fills, np.int64)], fills])
            t_plan = time.perf_counter()
            ev0 = torch.cuda.Event(enable_timing=True)
            ev0.record(self.stream)
            prng_batcher_launch(self.batcher, fills, sid)
            self.stats["batcher_s"] += time.perf_counter() - t_plan
            for st in steps:                   # half-sweep t of every running lattice
                prng_ising_half_sweep(st, sid)
            ev = torch.cuda.Event(enable_timing=True)
            ev.record(self.stream)
            for i in R[done_mask]:
                r = reqs[int(i)]
                r.half_done = int(half_done[i])
                self.clients[r.client].busy = None
                finishing.append(r)
            inflight.append((ev, finishing))
            self.stats["ticks"] += 1
            self.stats["launch_s"] += time.perf_counter() - t_tick
            tick_events.append((ev0, ev))
            running = R[~done_mask]
        self.stream.synchronize()
        self.stats["gpu_s"] = sum(a.elapsed_time(b) for a, b in tick_events) / 1e3
        return reqs


def latency_stats(reqs):
    lat = sorted(r.done - r.arrival for r in reqs)
    pct = lambda q: lat[min(len(lat) - 1, int(q * len(lat)))]
    span = max(r.done for r in reqs) - min(r.arrival for r in reqs)
    numbers = sum(r.numbers for r in reqs)
    return {"requests": len(reqs), "p50_ms": 1e3 * pct(0.50), "p99_ms": 1e3 * pct(0.99),
            "max_ms": 1e3 * lat[-1], "numbers": numbers,
            "numbers_per_s": numbers / span if span > 0 else None, "span_s": span}

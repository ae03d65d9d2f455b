"""The tensor-core RANLUX fills (tile 128 x 24: streams whole, or long ones cut
into segments) against the oracle: heads, tails and copy-outs of every length class, every output mode, aligned and unaligned
rows, and the states at which its modular arithmetic could go wrong."""
import numpy as np
import pytest

import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_1003_1898_gb300 as P  # noqa: E402

LEVELS = (97, 223, 389, 120, 240, 408)


@pytest.fixture(scope="module", autouse=True)
def _built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1003_1898_gb300 import build
    build.build()
    P.lib()


@pytest.fixture(autouse=True, params=[1, 2], ids=["whole", "segments"])
def _tile(request):
    saved = {p: P.prng_get_tile("ranlux", p) for p in LEVELS}
    for p in LEVELS:
        P.prng_set_tile("ranlux", p, 128, 24, request.param)
    yield
    for p, t in saved.items():
        P.prng_set_tile("ranlux", p, *t)


def _steps(V, c, n):
    """n subtract-with-borrow steps on 24 words, oldest first (Appendix A)."""
    V, out = list(V), []
    for _ in range(n):
        t = V[14] - V[0] - c
        c = 1 if t < 0 else 0
        V = V[1:] + [t % 2**24]
        out.append(V[-1])
    return V, c, out


@pytest.mark.parametrize("lux", LEVELS)
@pytest.mark.parametrize("ns", [1, 129, 301])
def test_positions(lux, ns):
    # fills that end inside the open block, heads of 1..23, tails of 1..23,
    # whole blocks, aligned and unaligned row pitches and start positions
    pieces = [8, 4, 2, 10, 100, 4, 76, 1, 3, 48, 252, 24, 5, 96, 1000, 12, 7, 1024, 20, 32, 23, 25, 56, 60]
    ref = oracle.fill("ranlux", 91, ns, sum(pieces), luxury=lux)
    h = P.prng_create("ranlux", 91, ns, lux)
    try:
        col = 0
        for i, k in enumerate(pieces):
            f32 = i % 3 == 2
            out = torch.full((ns * k + 4,), -7, dtype=torch.int32, device="cuda")
            (P.prng_fill_f32 if f32 else P.prng_fill_u32)(h, out, k)
            got = out.cpu().numpy()
            want = ref[:, col:col + k]
            if f32:
                want = oracle.to_f32("ranlux", want).view(np.uint32)
            np.testing.assert_array_equal(got[:ns * k].view(np.uint32).reshape(ns, k), want,
                                          err_msg=f"piece {i} ({k} draws)")
            assert np.all(got[ns * k:] == -7), f"piece {i} wrote past its rows"
            col += k
    finally:
        P.prng_destroy(h)


@pytest.mark.parametrize("lux", [97, 223, 408])
def test_doubles_and_misaligned_output(lux):
    ns = 131
    for pieces, off in (([8, 50, 2, 300], 0), ([6, 50, 123], 1)):
        ref = oracle.fill_f64("ranlux", 92, ns, sum(pieces), luxury=lux)
        h = P.prng_create("ranlux", 92, ns, lux)
        col = 0
        for k in pieces:
            out = torch.zeros(ns * k + off, dtype=torch.float64, device="cuda")
            P.prng_fill_f64(h, out.data_ptr() + 8 * off, k)
            np.testing.assert_array_equal(out.cpu().numpy()[off:].reshape(ns, k), ref[:, col:col + k])
            col += k
        P.prng_destroy(h)


def test_fused_half_sweeps():
    t4, t8 = P.prng_ising_thresholds(oracle.ISING_BETA)
    for L, ns in ((130, 65), (256, 256), (96, 4608)):
        h = P.prng_create("ranlux", 93, ns, 223)
        spins = torch.ones((L, L), dtype=torch.int8, device="cuda")
        for _ in range(3):
            for colour in (0, 1):
                P.prng_ising_fused(h, spins, L, colour, t4, t8)
        want, _ = oracle.ising_run("ranlux", 93, ns, L, 3, luxury=223)
        np.testing.assert_array_equal(spins.cpu().numpy(), want)
        P.prng_destroy(h)


@pytest.mark.parametrize("lux", [97, 389])
def test_extreme_states(lux):
    # Blobs a user may restore: all zero, all ones, single bits, long runs of
    # ones and zeros -- where a value meets the modulus or a carry runs through.
    rng = np.random.default_rng(5)
    top = 2**24 - 1
    states = [([0] * 24, 0), ([top] * 24, 1), ([0] * 24, 1), ([top] * 24, 0), ([0] * 23 + [1], 0),
              ([1] + [0] * 23, 0), ([0] * 14 + [1] + [0] * 9, 0), ([1] + [0] * 13 + [1] + [0] * 9, 0)]
    for _ in range(120):
        V = [int(rng.choice([0, top, 1, int(rng.integers(0, 2**24))], p=[.35, .35, .1, .2])) for _ in range(24)]
        states.append((V, int(rng.integers(0, 2))))
    ns = len(states)
    h = P.prng_create("ranlux", 1, ns, lux)
    try:
        hdr = np.frombuffer(P.prng_get_state(h), dtype=np.uint32)[:8].copy()
        hdr[6] = 24                                  # at the end of a block
        body = np.array([V + [c] for V, c in states], dtype=np.uint32)
        P.prng_set_state(h, hdr.tobytes() + body.tobytes())
        got = []
        for k in (24, 29, 72):
            out = torch.empty((ns, k), dtype=torch.int32, device="cuda")
            P.prng_fill_u32(h, out, k)
            got.append(out.cpu().numpy())
        got = np.concatenate(got, axis=1)
        for i, (V, c) in enumerate(states):
            want = []
            while len(want) < 125:
                V, c, _ = _steps(V, c, lux - 24)
                V, c, o = _steps(V, c, 24)
                want += o
            np.testing.assert_array_equal(got[i], want[:125], err_msg=str(states[i]))
    finally:
        P.prng_destroy(h)


def test_bulk_equals_borrow_chain():
    # 128 Mi words against the staged borrow-chain tile, and the state after it
    ns, per = 65536, 2048
    outs, blobs = [], []
    for tile in ((128, 24, 1), (128, 48, 1)):
        P.prng_set_tile("ranlux", 389, *tile)
        h = P.prng_create("ranlux", 7, ns, 389)
        out = torch.empty((ns, per), dtype=torch.int32, device="cuda")
        P.prng_fill_u32(h, out, per)
        outs.append(out)
        blobs.append(P.prng_get_state(h))
        P.prng_destroy(h)
    assert torch.equal(outs[0], outs[1])
    assert blobs[0] == blobs[1]


@pytest.mark.parametrize("lux", [97, 223, 408])
def test_batches_of_segments(lux):
    # Requests of several shapes in one launch, streams long enough to be cut,
    # a limit inside a row, unaligned rows, continued over three launches.
    specs = [(70, 24 * 100 + 7, 0), (1, 4100, 0), (129, 2400, 129 * 2400 - 3000), (33, 2404, 2404 * 32 + 17),
             (5, 30, 0), (40, 20, 0)]
    for batcher in (False, True):
        hs, outs, reqs, refs = [], [], [], []
        for i, (ns, per, valid) in enumerate(specs):
            hs.append(P.prng_create("ranlux", 500 + i, ns, lux))
            outs.append(torch.full((ns * per,), -7, dtype=torch.int32, device="cuda"))
            reqs.append({"st": hs[-1], "d_out": outs[-1], "n_per_stream": per, "n_valid": valid, "f32": i % 2 == 1})
            refs.append(oracle.fill("ranlux", 500 + i, ns, 3 * per, luxury=lux))
        b = P.prng_batcher_create(len(specs), 4096) if batcher else P.prng_batch_create(reqs)
        for k in range(3):
            for o in outs:
                o.fill_(-7)
            P.prng_batcher_launch(b, reqs) if batcher else P.prng_batch_launch(b)
            for i, ((ns, per, valid), o, ref) in enumerate(zip(specs, outs, refs)):
                want = ref[:, k * per:(k + 1) * per].reshape(-1)[:valid or None]
                if i % 2 == 1:
                    want = oracle.to_f32("ranlux", want).view(np.uint32)
                got = o.cpu().numpy()
                np.testing.assert_array_equal(got[:want.size].view(np.uint32), want, err_msg=f"{specs[i]} launch {k}")
                assert np.all(got[want.size:] == -7), f"{specs[i]} wrote past n_valid"
        torch.cuda.synchronize()
        (P.prng_batcher_destroy if batcher else P.prng_batch_destroy)(b)
        for h in hs:
            P.prng_destroy(h)


@pytest.mark.parametrize("per", [20, 24 * 8, 24 * 24 + 5, 24 * 40])
def test_batch_on_either_side_of_the_line(per):
    # Short requests stay on the borrow chain, long ones take the products.
    ns = 33
    ref = oracle.fill("ranlux", 91, ns, 3 * per, luxury=223)
    h = P.prng_create("ranlux", 91, ns, 223)
    out = torch.empty(ns * per, dtype=torch.int32, device="cuda")
    reqs = [{"st": h, "d_out": out, "n_per_stream": per, "n_valid": 0, "f32": False}]
    batch, batcher = P.prng_batch_create(reqs), P.prng_batcher_create(1, 64)
    for k in range(3):
        P.prng_batch_launch(batch) if k != 1 else P.prng_batcher_launch(batcher, reqs)
        got = out.cpu().numpy().view(np.uint32).reshape(ns, per)
        np.testing.assert_array_equal(got, ref[:, k * per:(k + 1) * per])
    torch.cuda.synchronize()
    P.prng_batch_destroy(batch)
    P.prng_batcher_destroy(batcher)
    P.prng_destroy(h)

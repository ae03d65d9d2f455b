"""Staged tiles that are not copied out plainly: short rows, ends of rows, unaligned
rows and outputs, few streams, in every staged tile and output type; and batcher
launches whose lengths differ in any byte."""
import numpy as np
import pytest

import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_1003_1898_gb300 as P  # noqa: E402


@pytest.fixture(scope="module", autouse=True)
def _built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1003_1898_gb300 import build
    build.build()
    P.lib()


@pytest.mark.parametrize("tile", [(128, 32, 1), (128, 32, 2), (128, 64, 1), (256, 32, 1)])
@pytest.mark.parametrize("gen", ["xor128", "ggl"])
@pytest.mark.parametrize("ns", [1, 33, 130, 300])
def test_odd_tiles(gen, tile, ns):
    saved = P.prng_get_tile(gen)
    P.prng_set_tile(gen, 0, *tile)
    pieces = [(1, "u32", 0), (5, "f64", 0), (31, "f32", 1), (33, "u32", 0), (17, "f64", 1), (63, "f32", 0), (65, "u32", 3),
              (61, "f64", 0), (100, "f32", 0), (36, "f64", 0), (129, "u32", 1)]
    total = sum(n * (2 if dt == "f64" else 1) for n, dt, _ in pieces)
    ref = oracle.fill(gen, 31, ns, total)
    h = P.prng_create(gen, 31, ns)
    try:
        at = 0
        for n, dt, off in pieces:
            td, f = {"u32": (torch.int32, P.prng_fill_u32), "f32": (torch.float32, P.prng_fill_f32),
                     "f64": (torch.float64, P.prng_fill_f64)}[dt]
            room = torch.full((ns * n + off + 8,), -7, dtype=td, device="cuda")
            f(h, room[off:], n)
            got = room.cpu().numpy()
            draws = n * (2 if dt == "f64" else 1)
            want = ref[:, at:at + draws]
            if dt == "f64":
                a, b = want[:, 0::2].astype(np.uint64), want[:, 1::2].astype(np.uint64)
                drop = 4 if gen == "ggl" else 5
                want = ((a >> np.uint64(drop)) * np.uint64(2**26) + (b >> np.uint64(drop + 1))) * 2.0**-53
            elif dt == "f32":
                want = oracle.to_f32(gen, want)
            else:
                want = want.view(np.int32)
            np.testing.assert_array_equal(got[off:off + ns * n].reshape(ns, n), want, err_msg=f"{n} {dt}")
            assert np.all(got[:off] == -7) and np.all(got[off + ns * n:] == -7), f"{n} {dt} wrote past its rows"
            at += draws
    finally:
        P.prng_destroy(h)
        P.prng_set_tile(gen, 0, *saved)


def test_batcher_orders_lengths_that_differ_in_any_byte():
    rng = np.random.default_rng(9)
    lens = [int(x) for x in np.concatenate([rng.integers(1, 300, 30), rng.integers(250, 70000, 20), [65536, 65537, 131072, 255, 256]])]
    hs = [P.prng_create("ggl", 900 + i, 2) for i in range(len(lens))]
    outs = [torch.full((2 * n,), -7, dtype=torch.int32, device="cuda") for n in lens]
    b = P.prng_batcher_create(len(lens), 4096)
    P.prng_batcher_launch(b, [{"st": h, "d_out": o, "n_per_stream": n} for h, o, n in zip(hs, outs, lens)])
    torch.cuda.synchronize()
    for i, (n, o) in enumerate(zip(lens, outs)):
        np.testing.assert_array_equal(o.cpu().numpy().view(np.uint32).reshape(2, n), oracle.fill("ggl", 900 + i, 2, n))
    P.prng_batcher_destroy(b)
    for h in hs:
        P.prng_destroy(h)

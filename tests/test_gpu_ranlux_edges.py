"""RANLUX fills at the edges of their division into segments and tiles."""
import ctypes

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


@pytest.mark.parametrize("ns,per", [(256, 984), (4096, 984), (33, 24 * 8 * 5 + 24), (1, 24 * 8 * 17 + 12)])
def test_fresh_rows_one_block_past_whole_segments(ns, per):
    # An open block of a whole 24 draws leaves one block fewer to cut.
    ref = oracle.fill("ranlux", 5, ns, 2 * per, luxury=223)
    h = P.prng_create("ranlux", 5, ns, 223)
    try:
        for k in range(2):
            out = torch.empty((ns, per), dtype=torch.int32, device="cuda")
            P.prng_fill_u32(h, out, per)
            np.testing.assert_array_equal(out.cpu().numpy().view(np.uint32), ref[:, k * per:(k + 1) * per])
    finally:
        P.prng_destroy(h)


@pytest.mark.parametrize("pitch,has_map", [(1024, True), (2**31 - 32, True), (2**31, False), (2**31 + 32, False),
                                           (2**32 - 4, False)])
def test_rows_past_the_tile_engine_have_no_map(pitch, has_map):
    # The engine's column coordinate would turn negative and its tiles be dropped;
    # such rows are stored by the warps.  Only the map is asked for: nothing is filled.
    f = P.lib()._ZN4prng11lux_out_mapEPvmmP14CUtensorMap_st
    f.restype = ctypes.c_bool
    f.argtypes = [ctypes.c_void_p, ctypes.c_uint64, ctypes.c_uint64, ctypes.c_void_p]
    out = torch.empty(1024, dtype=torch.int32, device="cuda")
    room = ctypes.create_string_buffer(128 + 64)
    at = (ctypes.addressof(room) + 63) // 64 * 64
    assert f(out.data_ptr(), pitch, 1, at) == has_map


@pytest.mark.parametrize("lux", [223, 389])
def test_batcher_outputs_that_move_between_launches(lux):
    # Every launch rewrites a slot's tensor maps at the same addresses: other
    # outputs, pitches and limits each time, over more launches than slots, with
    # nothing between them.
    ns, n = 96, 11
    hs = [P.prng_create("ranlux", 700 + i, ns, lux) for i in range(2)]
    b = P.prng_batcher_create(2, 4096)
    rng = np.random.default_rng(lux)
    drawn, launched = [0, 0], []
    for k in range(n):
        reqs = []
        for i, h in enumerate(hs):
            per = 4 * int(rng.integers(100, 700))
            valid = int(rng.integers(1, ns * per)) if k % 3 == 1 else 0
            out = torch.full((ns * per + 64,), -7, dtype=torch.int32, device="cuda")
            reqs.append({"st": h, "d_out": out, "n_per_stream": per, "n_valid": valid})
            launched.append((i, drawn[i], per, valid, out))
            drawn[i] += per
        P.prng_batcher_launch(b, reqs)
    torch.cuda.synchronize()
    refs = [oracle.fill("ranlux", 700 + i, ns, drawn[i], luxury=lux) for i in range(2)]
    for i, at, per, valid, out in launched:
        got = out.cpu().numpy()
        want = refs[i][:, at:at + per].reshape(-1)[:valid or None]
        np.testing.assert_array_equal(got[:want.size].view(np.uint32), want)
        assert np.all(got[want.size:] == -7)
    P.prng_batcher_destroy(b)
    for h in hs:
        P.prng_destroy(h)


def test_a_given_up_wait_reaches_every_later_call():
    # The word that a kernel sets when it gives up (here the test sets it): every
    # call that would draw from a RANLUX handle of the device, or read its state,
    # reports it before it launches anything.
    h = P.prng_create("ranlux", 3, 64, 223)
    g = P.prng_create("ggl", 3, 64)
    out = torch.empty((64, 64), dtype=torch.int32, device="cuda")
    spins = torch.ones((16, 16), dtype=torch.int8, device="cuda")
    req = [{"st": h, "d_out": out, "n_per_stream": 24}]
    batch, batcher = P.prng_batch_create(req), P.prng_batcher_create(1, 64)
    f = P.lib()._ZN4prng15lux_failed_wordEi
    f.restype = ctypes.POINTER(ctypes.c_uint32)
    word = f(torch.cuda.current_device())
    blob = P.prng_get_state(h)
    calls = [lambda: P.prng_fill_u32(h, out, 24), lambda: P.prng_fill_f64(h, out, 24), lambda: P.prng_skip(h, 24),
             lambda: P.prng_ising_fused(h, spins, 16, 0, 1, 1), lambda: P.prng_batch_launch(batch),
             lambda: P.prng_batcher_launch(batcher, req), lambda: P.prng_batch_fill_noalloc(req),
             lambda: P.prng_get_state(h)]
    word[0] = 1
    try:
        for i, call in enumerate(calls):
            with pytest.raises(P.PrngError) as e:
                call()
            assert e.value.code == -6, i
        P.prng_fill_u32(g, out, 24)             # other generators do not use it
    finally:
        word[0] = 0
    assert P.prng_get_state(h) == blob
    for call in calls:
        call()
    torch.cuda.synchronize()
    P.prng_batch_destroy(batch)
    P.prng_batcher_destroy(batcher)
    P.prng_destroy(h)
    P.prng_destroy(g)

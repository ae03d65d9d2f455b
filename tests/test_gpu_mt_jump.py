"""MT19937 jump fills at the edges of their cuts: one chunk, a few, more than a
power of two of them, short last chunks, a start inside the sequence."""
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


@pytest.fixture(scope="module")
def sequence():
    return oracle.serial_fill("mt19937", 20100, 6000000)


@pytest.mark.parametrize("first", [0, 1, 623, 777777])
@pytest.mark.parametrize("n", [1, 623, 624, 1249, 131072, 262145, 400001, 1048577, 3300000, 5200000])
def test_cuts(sequence, n, first):
    for f32 in (False, True):
        out = torch.full((n + 4,), -7, dtype=torch.float32 if f32 else torch.int32, device="cuda")
        call = P.prng_fill_jump_at_f32 if f32 else P.prng_fill_jump_at_u32
        call("mt19937", 20100, first, n, 64, out)
        got = out.cpu().numpy()
        want = sequence[first:first + n]
        want = oracle.to_f32("mt19937", want).view(np.uint32) if f32 else want
        np.testing.assert_array_equal(got[:n].view(np.uint32), want)
        assert np.all(got[n:] == -7)


@pytest.mark.parametrize("ns,per", [(1, 5000), (1024, 512), (300, 1249), (7, 623)])
def test_cta_per_stream_continues(ns, per):
    # fills that start and end inside a table, aligned or not
    pieces = [per, 1, 624, 100, per + 3]
    ref = oracle.fill("mt19937", 84, ns, sum(pieces))
    saved = P.prng_get_tile("mt19937")
    P.prng_set_tile("mt19937", 0, 256, 227, 1)
    h = P.prng_create("mt19937", 84, ns, 0)
    try:
        col = 0
        for i, k in enumerate(pieces):
            out = torch.full((ns * k + 4,), -7, dtype=torch.int32, device="cuda")
            (P.prng_fill_f32 if i % 2 else P.prng_fill_u32)(h, out, k)
            got = out.cpu().numpy()
            want = ref[:, col:col + k]
            want = oracle.to_f32("mt19937", want).view(np.uint32) if i % 2 else want
            np.testing.assert_array_equal(got[:ns * k].view(np.uint32).reshape(ns, k), want)
            assert np.all(got[ns * k:] == -7)
            col += k
    finally:
        P.prng_destroy(h)
        P.prng_set_tile("mt19937", 0, *saved)

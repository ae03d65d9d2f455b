"""Requests whose n_valid leaves whole streams unwanted: the first n_valid
elements are the oracle's, nothing after them is written, and every stream of
the handle still advances."""
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


@pytest.mark.parametrize("gen,lux", [(g, 223 if g == "ranlux" else 0) for g in P.GEN_NAMES])
@pytest.mark.parametrize("per,valid", [(16, 16 * 5), (16, 16 * 5 + 3), (700, 700 * 2 + 4), (13, 13 * 9 + 1)])
def test_n_valid_cuts_whole_streams(gen, lux, per, valid):
    ns = 41
    h = P.prng_create(gen, 321, ns, lux)
    out = torch.full((ns * per,), -7, dtype=torch.int32, device="cuda")   # room for every stream's row
    b = P.prng_batcher_create(1, 1024)
    try:
        P.prng_batcher_launch(b, [{"st": h, "d_out": out, "n_per_stream": per, "n_valid": valid}])
        nxt = torch.empty(ns * per, dtype=torch.int32, device="cuda")
        P.prng_fill_u32(h, nxt, per)
        torch.cuda.synchronize()
        ref = oracle.fill(gen, 321, ns, 2 * per, luxury=lux)
        got = out.cpu().numpy()
        np.testing.assert_array_equal(got[:valid].view(np.uint32), ref[:, :per].reshape(-1)[:valid])
        assert np.all(got[valid:] == -7), "write past n_valid"
        np.testing.assert_array_equal(nxt.cpu().numpy().view(np.uint32).reshape(ns, per), ref[:, per:])
    finally:
        P.prng_batcher_destroy(b)
        P.prng_destroy(h)

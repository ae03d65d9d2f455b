"""RANLUX skips choose their kernel by shape, as fills do: on the borrow chain and on
the tensor cores, from every place of the open block."""
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


@pytest.mark.parametrize("lux", [24, 48, 97, 223, 389, 408])
@pytest.mark.parametrize("ns", [1, 129])
def test_skips_by_shape(lux, ns):
    pieces = [(5, 7), (1, 24 * 20), (24 * 3, 4), (24 * 300 + 11, 24 * 40), (23, 24 * 130 + 1)]   # draws, then a skip
    total = sum(a + b for a, b in pieces) + 30
    ref = oracle.fill("ranlux", 64, ns, total, luxury=lux)
    h = P.prng_create("ranlux", 64, ns, lux)
    try:
        at = 0
        for n, skip in pieces + [(30, 0)]:
            out = torch.empty((ns, n), dtype=torch.int32, device="cuda")
            P.prng_fill_u32(h, out, n)
            np.testing.assert_array_equal(out.cpu().numpy().view(np.uint32), ref[:, at:at + n], err_msg=f"at {at}")
            P.prng_skip(h, skip)
            at += n + skip
    finally:
        P.prng_destroy(h)

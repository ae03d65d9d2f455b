"""Fills captured into a CUDA graph: few long streams, which would otherwise be
cut into segments with scratch, replayed twice continue the streams twice."""
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


@pytest.mark.parametrize("gen,lux,per", [("xor128", 0, 4096), ("ranlux", 389, 2400), ("ranecu", 0, 1000)])
def test_captured_fill_replays(gen, lux, per):
    # per is a whole number of luxury blocks, so every replay starts where its
    # recorded position says
    ns = 33
    h = P.prng_create(gen, 17, ns, lux)
    try:
        if gen == "ranlux":
            P.prng_skip(h, 24)
        out = torch.empty((ns, per), dtype=torch.int32, device="cuda")
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g):
            P.prng_fill_u32(h, out, per)
        ref = oracle.fill(gen, 17, ns, 24 + 2 * per, luxury=lux)
        ref = ref[:, 24:] if gen == "ranlux" else ref
        for k in range(2):
            g.replay()
            np.testing.assert_array_equal(out.cpu().numpy().view(np.uint32), ref[:, k * per:(k + 1) * per])
    finally:
        P.prng_destroy(h)

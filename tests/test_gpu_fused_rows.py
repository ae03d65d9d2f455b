"""Fused half-sweeps whose rows are a few sites, or end inside a tile: the chunks
of four sites, the single sites and the lattices that have no chunks."""
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


@pytest.mark.parametrize("L,ns", [(64, 2048), (64, 1024), (64, 512), (64, 256), (64, 32), (96, 4608), (96, 1536), (96, 512),
                                  (96, 384), (96, 128), (30, 450), (30, 150), (30, 90), (30, 25), (100, 1000), (48, 8)])
@pytest.mark.parametrize("offset", [0, 1])
def test_xor128_rows_shorter_than_a_tile(L, ns, offset):
    t4, t8 = P.prng_ising_thresholds(oracle.ISING_BETA)
    h = P.prng_create("xor128", 45, ns, 0)
    room = torch.ones(L * L + offset, dtype=torch.int8, device="cuda")      # offset 1: no 8-byte chunks
    spins = room[offset:]
    try:
        for _ in range(3):
            for colour in (0, 1):
                P.prng_ising_fused(h, spins, L, colour, t4, t8)
        want, _ = oracle.ising_run("xor128", 45, ns, L, 3)
        np.testing.assert_array_equal(spins.cpu().numpy().reshape(L, L), want)
    finally:
        P.prng_destroy(h)

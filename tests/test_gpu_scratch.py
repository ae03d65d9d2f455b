"""The scratch that the library keeps between calls is bounded."""
import pytest

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


def test_large_scratch_goes_back():
    # A jump fill in 2^27 chunks of one draw takes 2 GiB of chunk starts.
    n = 2**27
    out = torch.empty(n, dtype=torch.int32, device="cuda")
    P.prng_fill_jump_u32("xor128", 7, 2**20, 64, out)
    torch.cuda.synchronize()
    before = torch.cuda.mem_get_info()[0]
    P.prng_fill_jump_u32("xor128", 7, n, n, out)
    torch.cuda.synchronize()
    torch.cuda.synchronize()
    assert before - torch.cuda.mem_get_info()[0] <= 2**30 + 2**28

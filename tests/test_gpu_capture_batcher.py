"""A batcher launch captured into a CUDA graph takes no scratch, as captured fills."""
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


def test_captured_batcher_launch_allocates_nothing():
    # RANLUX streams long enough to be cut: the captured launch holds no allocation
    # node (a graph with one can be instantiated once only), and two instances of it
    # continue the streams in turn.
    ns, per = 33, 2400
    ref = oracle.fill("ranlux", 18, ns, 24 + 2 * per, luxury=389)
    h = P.prng_create("ranlux", 18, ns, 389)
    P.prng_skip(h, 24)
    out = torch.full((ns, per), -7, dtype=torch.int32, device="cuda")
    b = P.prng_batcher_create(1, 4096)
    s = torch.cuda.Stream()
    torch.cuda.synchronize()
    cu = ctypes.CDLL("libcuda.so.1")
    stream, graph, n = ctypes.c_void_p(s.cuda_stream), ctypes.c_void_p(), ctypes.c_size_t()
    assert cu.cuStreamBeginCapture_v2(stream, 2) == 0
    try:
        P.prng_batcher_launch(b, [{"st": h, "d_out": out, "n_per_stream": per}], stream=s)
    finally:
        assert cu.cuStreamEndCapture(stream, ctypes.byref(graph)) == 0
    assert cu.cuGraphGetNodes(graph, None, ctypes.byref(n)) == 0
    nodes = (ctypes.c_void_p * n.value)()
    assert cu.cuGraphGetNodes(graph, nodes, ctypes.byref(n)) == 0
    kinds = []
    for node in nodes:
        k = ctypes.c_int()
        assert cu.cuGraphNodeGetType(ctypes.c_void_p(node), ctypes.byref(k)) == 0
        kinds.append(k.value)
    assert 10 not in kinds and 11 not in kinds, kinds          # memory allocation and release
    execs = []
    for _ in range(2):
        e = ctypes.c_void_p()
        assert cu.cuGraphInstantiateWithFlags(ctypes.byref(e), graph, ctypes.c_ulonglong(0)) == 0
        execs.append(e)
    for k, e in enumerate(execs):
        assert cu.cuGraphLaunch(e, stream) == 0
        s.synchronize()
        np.testing.assert_array_equal(out.cpu().numpy().view(np.uint32), ref[:, 24 + k * per:24 + (k + 1) * per])
    for e in execs:
        cu.cuGraphExecDestroy(e)
    cu.cuGraphDestroy(graph)
    P.prng_batcher_destroy(b)
    P.prng_destroy(h)

"""XOR128 fills that are cut into segments (few streams, long rows): ragged last
segments, every output mode, unaligned rows, and the states they leave."""
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


CHILD = '''
import sys; sys.path.insert(0, {root!r})
import numpy as np, torch, oracle
import paper_1003_1898_gb300 as P
# a process of its own: no other test has chosen XOR128's tile here
for ns in (1, 65, 300):
    pieces = [1024, 899, 8192, 4100, 2051, 1, 3000, 1600]
    ref = oracle.fill("xor128", 81, ns, sum(pieces))
    h = P.prng_create("xor128", 81, ns, 0)
    col = 0
    for i, k in enumerate(pieces):
        f32 = i % 2 == 1
        out = torch.full((ns * k + 4,), -7, dtype=torch.float32 if f32 else torch.int32, device="cuda")
        (P.prng_fill_f32 if f32 else P.prng_fill_u32)(h, out, k)
        got = out.cpu().numpy()
        want = ref[:, col:col + k]
        want = oracle.to_f32("xor128", want) if f32 else want
        np.testing.assert_array_equal(got[:ns * k].view(np.uint32).reshape(ns, k), want.view(np.uint32))
        assert np.all(got[ns * k:] == -7)
        col += k
    P.prng_destroy(h)
    ref = oracle.fill_f64("xor128", 82, ns, 1500 + 333)
    h = P.prng_create("xor128", 82, ns, 0)
    for a, b in ((0, 1500), (1500, 1833)):
        out = torch.empty((ns, b - a), dtype=torch.float64, device="cuda")
        P.prng_fill_f64(h, out, b - a)
        np.testing.assert_array_equal(out.cpu().numpy(), ref[:, a:b])
    P.prng_destroy(h)
t4, t8 = P.prng_ising_thresholds(oracle.ISING_BETA)
for L, ns in ((256, 32), (130, 5), (96, 9)):
    h = P.prng_create("xor128", 83, ns, 0)
    spins = torch.ones((L, L), dtype=torch.int8, device="cuda")
    for _ in range(2):
        for colour in (0, 1):
            P.prng_ising_fused(h, spins, L, colour, t4, t8)
    want, _ = oracle.ising_run("xor128", 83, ns, L, 2)
    np.testing.assert_array_equal(spins.cpu().numpy(), want)
    P.prng_destroy(h)
print("segments ok")
'''


def test_segments():
    import os
    import subprocess
    import sys
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    r = subprocess.run([sys.executable, "-c", CHILD.format(root=root)], capture_output=True, text=True, timeout=300,
                       cwd=root)
    assert r.returncode == 0 and "segments ok" in r.stdout, r.stdout[-2000:] + r.stderr[-4000:]


WIDE = '''
import sys; sys.path.insert(0, {root!r})
import numpy as np, torch, oracle
import paper_1003_1898_gb300 as P
# enough draws for the wide segments: streams x draws, then a short call from the states left
for ns, n, kind in ((2048, 65000, "u32"), (32767, 4099, "f32"), (33001, 5000, "f32"), (40000, 6001, "u32"),
                    (65537, 4500, "u32"), (32768, 4096, "f64"), (98304, 3072, "f64"), (100351, 2100, "f64")):
    h = P.prng_create("xor128", 84, ns, 0)
    f64 = kind == "f64"
    ty = dict(u32=torch.int32, f32=torch.float32, f64=torch.float64)[kind]
    fill = dict(u32=P.prng_fill_u32, f32=P.prng_fill_f32, f64=P.prng_fill_f64)[kind]
    per = n // 2 if f64 else n
    out = torch.full((ns * per + 8,), -7, dtype=ty, device="cuda")
    fill(h, out, per)
    tail = torch.empty((ns, 8), dtype=torch.int32, device="cuda")
    P.prng_fill_u32(h, tail, 8)
    assert torch.all(out[ns * per:] == -7)
    got = out[:ns * per].view(ns, per)
    for r0 in (0, ns // 2 - 65, ns - 130):
        ref = oracle.fill("xor128", 84 + r0, 130, n + 8)
        if f64:
            want = oracle.fill_f64("xor128", 84 + r0, 130, per)
        else:
            want = oracle.to_f32("xor128", ref[:, :n]) if kind == "f32" else ref[:, :n].view(np.int32)
        np.testing.assert_array_equal(got[r0:r0 + 130].cpu().numpy(), want)
        np.testing.assert_array_equal(tail[r0:r0 + 130].cpu().numpy().view(np.uint32), ref[:, n:])
    P.prng_destroy(h)
print("wide ok")
'''


def test_wide_segments():
    import os
    import subprocess
    import sys
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    r = subprocess.run([sys.executable, "-c", WIDE.format(root=root)], capture_output=True, text=True, timeout=300,
                       cwd=root)
    assert r.returncode == 0 and "wide ok" in r.stdout, r.stdout[-2000:] + r.stderr[-4000:]

"""MT19937 plain fills whose tile the library chooses by shape: both sides of each line."""
import os
import subprocess
import sys

import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

CHILD = """
import sys; sys.path.insert(0, sys.argv[1])
import numpy as np, torch, oracle
import paper_1003_1898_gb300 as P
# a process of its own: no other test has chosen MT19937's tile here
ns, n, f32 = int(sys.argv[2]), int(sys.argv[3]), sys.argv[4] == "f32"
h = P.prng_create("mt19937", 91, ns, 0)
out = torch.full((ns * n + 4,), -7, dtype=torch.float32 if f32 else torch.int32, device="cuda")
(P.prng_fill_f32 if f32 else P.prng_fill_u32)(h, out, n)
tail = torch.empty((ns, 5), dtype=torch.int32, device="cuda")
P.prng_fill_u32(h, tail, 5)
assert torch.all(out[ns * n:] == -7)
got = out[:ns * n].view(ns, n)
for r0 in (0, ns // 2, ns - 9):
    ref = oracle.fill("mt19937", 91 + r0, 9, n + 5)
    want = oracle.to_f32("mt19937", ref[:, :n]) if f32 else ref[:, :n].view(np.int32)
    np.testing.assert_array_equal(got[r0:r0 + 9].cpu().numpy(), want)
    np.testing.assert_array_equal(tail[r0:r0 + 9].cpu().numpy().view(np.uint32), ref[:, n:])
print("shape ok")
"""


@pytest.fixture(scope="module", autouse=True)
def _built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1003_1898_gb300 import build
    build.build()


@pytest.mark.parametrize("ns,n,kind", [(912, 30001, "u32"), (913, 30001, "f32"), (2433, 10000, "u32"),
                                       (2729, 10007, "f32"), (2432, 10000, "u32"), (8513, 10000, "u32")])
def test_shape(ns, n, kind):
    r = subprocess.run([sys.executable, "-c", CHILD, ROOT, str(ns), str(n), kind], capture_output=True, text=True,
                       timeout=300, cwd=ROOT)
    assert r.returncode == 0 and "shape ok" in r.stdout, r.stdout[-2000:] + r.stderr[-4000:]

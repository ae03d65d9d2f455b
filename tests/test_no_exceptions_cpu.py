"""Host memory that runs out inside a C entry point is an error code, not an
exception through the C boundary."""
import os
import shutil
import subprocess
import sys

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

# operator new that fails from the k-th call on, in front of the library's.
FAILING_NEW = r"""
#include <cstdlib>
#include <new>
static long left = -1;
extern "C" void fail_after(long k) { left = k; }
void* operator new(std::size_t n) {
  if (left == 0) throw std::bad_alloc();
  if (left > 0) left--;
  void* p = std::malloc(n ? n : 1);
  if (!p) throw std::bad_alloc();
  return p;
}
void operator delete(void* p) noexcept { std::free(p); }
void operator delete(void* p, std::size_t) noexcept { std::free(p); }
"""

CHILD = r"""
import ctypes, sys
new = ctypes.CDLL(sys.argv[1], mode=ctypes.RTLD_GLOBAL)
L = ctypes.CDLL(sys.argv[2])
new.fail_after.argtypes = [ctypes.c_long]

class State(ctypes.Structure):      # a handle as far as planning reads it: GGL or RANLUX, 100 streams
    _fields_ = [("gen", ctypes.c_int), ("p", ctypes.c_int), ("n", ctypes.c_uint64), ("state", ctypes.c_void_p),
                ("pos", ctypes.c_uint32), ("device", ctypes.c_int)]

class Req(ctypes.Structure):
    _fields_ = [("st", ctypes.c_void_p), ("d_out", ctypes.c_void_p), ("n_per", ctypes.c_uint64),
                ("n_valid", ctypes.c_uint64), ("seed", ctypes.c_uint64), ("f32", ctypes.c_int32),
                ("reseed", ctypes.c_int32)]

seen = set()
for k in range(40):
    h = ctypes.c_void_p()
    new.fail_after(k)
    rc = L.prng_create(ctypes.byref(h), 4, ctypes.c_uint64(1), 10, 389)
    new.fail_after(-1)
    assert rc in (-5, -6), rc                                # no memory, or no device
    if k == 0:
        assert rc == -5
for k in range(60):
    sts = (State * 2)(State(0, 0, 100, None, 0, 0), State(4, 223, 100, None, 0, 0))
    reqs = (Req * 2)(*[Req(ctypes.addressof(s), 16, 5000, 0, 0, 0, 1) for s in sts])
    b = ctypes.c_void_p()
    new.fail_after(k)
    rc = L.prng_batch_create(ctypes.byref(b), reqs, 2)
    new.fail_after(-1)
    assert rc in (-5, -6) and not b.value, rc
print("ok")
"""


def test_allocation_failures_are_error_codes(tmp_path):
    from paper_1003_1898_gb300 import build
    lib = build.build()
    src, so = tmp_path / "new.cpp", tmp_path / "new.so"
    src.write_text(FAILING_NEW)
    cxx = shutil.which("g++") or shutil.which("c++")
    subprocess.run([cxx, "-O1", "-std=c++17", "-shared", "-fPIC", str(src), "-o", str(so)], check=True)
    env = dict(os.environ, CUDA_VISIBLE_DEVICES="")          # no device, wherever it runs
    r = subprocess.run([sys.executable, "-c", CHILD, str(so), lib], capture_output=True, text=True, env=env)
    assert r.returncode == 0 and r.stdout.strip() == "ok", r.stderr

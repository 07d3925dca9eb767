"""Host allocations and threads that fail while work lists are built come back as HS_ERR_NOMEM (or are
done without): every allocation of a call is made to fail once, in a child process, by an
operator new in front of the library's. No GPU needed: hs_sweep_lists runs the same list
builder, on enough windows that it starts threads."""

import os
import shutil
import subprocess
import sys
import textwrap

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

NEW = r"""
#include <atomic>
#include <cstdlib>
#include <new>
static std::atomic<long> left{-1};
extern "C" void fail_after(long n) { left = n; }
extern "C" long remaining() { return left; }
void* operator new(std::size_t n) {
    if (left >= 0 && left-- == 0) throw std::bad_alloc();
    void* p = std::malloc(n ? n : 1);
    if (!p) throw std::bad_alloc();
    return p;
}
void operator delete(void* p) noexcept { std::free(p); }
void operator delete(void* p, std::size_t) noexcept { std::free(p); }
"""

CHILD = r"""
import ctypes as C, sys
import numpy as np
from paper_1806_04596_gb300 import hypersara as hs
new = C.CDLL(sys.argv[1], mode=C.RTLD_GLOBAL)
new.remaining.restype = C.c_long
new.fail_after.argtypes = [C.c_long]
lib = hs.load()
K, L, M = 64, 4, 20000
rng = np.random.default_rng(1)
off = np.arange(L + 1, dtype=np.int64) * M
k0x = rng.integers(0, K - 8, L * M).astype(np.int32)
k0y = rng.integers(0, K, L * M).astype(np.int32)
ni, ne = C.c_int64(), C.c_int64()
def call():
    return lib.hs_sweep_lists(K, K, L, off.ctypes.data, k0x.ctypes.data, k0y.ctypes.data, 0, 0, None, C.byref(ni),
                              None, C.byref(ne))
assert call() == hs.HS_OK
want = (ni.value, ne.value)
n, failed = 0, 0
while True:
    new.fail_after(n)
    st = call()
    unused = new.remaining() >= 0
    new.fail_after(-1)
    assert st in (hs.HS_OK, hs.HS_ERR_NOMEM), (n, st)
    failed += st == hs.HS_ERR_NOMEM
    if st == hs.HS_OK:
        assert (ni.value, ne.value) == want, n
    if unused:
        break
    n += 1 if n < 40 else 1 + n // 16
assert failed > 10
assert call() == hs.HS_OK and (ni.value, ne.value) == want
print("ok", n, failed)
"""


def test_every_host_allocation_may_fail(tmp_path):
    gxx = shutil.which("g++")
    if gxx is None:
        pytest.skip("no g++")
    import __graft_entry__ as ge
    ge.build()
    src, lib = tmp_path / "new.cpp", tmp_path / "libnew.so"
    src.write_text(NEW)
    subprocess.run([gxx, "-O1", "-shared", "-fPIC", "-o", str(lib), str(src)], check=True)
    env = dict(os.environ, LD_PRELOAD=str(lib), PYTHONPATH=ROOT)
    r = subprocess.run([sys.executable, "-c", textwrap.dedent(CHILD), str(lib)], capture_output=True, text=True,
                       env=env, cwd=ROOT, timeout=600)
    assert r.returncode == 0, (r.returncode, r.stdout[-500:], r.stderr[-1500:])

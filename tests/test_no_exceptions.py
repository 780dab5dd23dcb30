"""No C++ exception leaves the C ABI: creating a handle without memory returns a status (the caller may be C)."""
import os
import subprocess
import sys

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

# operator new that throws on the n-th call from now (0: never)
PRELOAD = r"""
#include <cstdlib>
#include <new>
static long left = 0;
extern "C" void fail_new(long n) { left = n; }
void *operator new(size_t n) {
    if (left > 0 && --left == 0) throw std::bad_alloc();
    if (void *p = malloc(n ? n : 1)) return p;
    throw std::bad_alloc();
}
"""

CHILD = """
import ctypes as C, sys
from paper_2509_16434_b200 import binding as ppo
lib = ppo.lib()
fail = C.CDLL(sys.argv[1]).fail_new
d = ppo.model_desc(120, 160, (16, 32, 64, 128), (3, 3, 3, 3), (512, 512, 256), norm=True, embed=32, n_lstm=2, lstm_h=1024)
b = ppo.buffer_desc(4, 2, 16, 24)
seen = set()
for n in range(1, 12):
    h = C.c_void_p()
    fail(n)
    s = lib.ppo_model_create(C.byref(d), C.byref(h))
    fail(0)
    assert (s == 0) == bool(h.value), (n, s)
    seen.add(s)
    if h.value:
        assert lib.ppo_model_num_tensors(h) == 33
        lib.ppo_model_destroy(h)
assert seen == {0, 1}, seen
print("ok")
"""


def test_creating_a_model_without_memory_returns_a_status(tmp_path):
    src, so = tmp_path / "fail_new.cpp", tmp_path / "libfail_new.so"
    src.write_text(PRELOAD)
    subprocess.run(["g++", "-shared", "-fPIC", "-w", "-o", str(so), str(src)], check=True)
    run = subprocess.run([sys.executable, "-c", CHILD, str(so)], cwd=ROOT, capture_output=True, text=True, timeout=300,
                         env=dict(os.environ, LD_PRELOAD=str(so)))
    assert run.returncode == 0 and run.stdout.strip() == "ok", run.stdout + run.stderr[-2000:]

"""No C++ exception crosses the C boundary: host allocations that fail at any
point of a call end in GENCD_ENOMEM.  Run on the CPU, in a process whose
operator new fails on demand, with the serving dry run (the same loader and
stepper as the server's)."""

import os
import re
import subprocess
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

FAILING_NEW = """
#include <atomic>
#include <cstdlib>
#include <new>
static std::atomic<long> left{-1};
extern "C" void arm(long n) { left = n; }
void* operator new(std::size_t n) {
  long v = left.load();
  while (v > 0 && !left.compare_exchange_weak(v, v - 1)) {
  }
  if (v == 0) throw std::bad_alloc();
  void* p = std::malloc(n ? n : 1);
  if (!p) throw std::bad_alloc();
  return p;
}
void* operator new(std::size_t n, const std::nothrow_t&) noexcept {
  try {
    return operator new(n);
  } catch (...) {
    return nullptr;
  }
}
void operator delete(void* p) noexcept { std::free(p); }
void operator delete(void* p, std::size_t) noexcept { std::free(p); }
"""

CALLER = """
import ctypes as C
import sys
from paper_1206_6409_gb300 import binding as gb
new = C.CDLL(sys.argv[1])
new.arm.argtypes = [C.c_long]
def call():
    try:
        gb.gencd_serve_dry_run([(1000, 1000, 5000)] * 8, [0.0] * 8, [0.0] * 8, budget_bytes=1e12, workers=3)
        return 0
    except gb.GencdError as e:
        return e.code
call()
codes = []
for n in range(12):
    new.arm(n)
    c = call()
    new.arm(-1)
    codes.append(c)
print(codes, call())
"""


def test_failing_allocations_return_an_error(tmp_path):
    from paper_1206_6409_gb300 import build

    build.build()
    src, lib = tmp_path / "new.cpp", tmp_path / "libnew.so"
    src.write_text(FAILING_NEW)
    subprocess.run(["g++", "-O1", "-shared", "-fPIC", "-std=c++17", str(src), "-o", str(lib)], check=True)
    r = subprocess.run([sys.executable, "-c", CALLER, str(lib)], cwd=ROOT, capture_output=True, text=True, timeout=120,
                       env=dict(os.environ, LD_PRELOAD=str(lib)))
    assert r.returncode == 0, r.stderr[-2000:]
    codes, after = eval("(" + r.stdout.strip().replace("] ", "], ") + ")")
    assert codes[0] == -2 and set(codes) <= {0, -2}, codes
    assert after == 0


@pytest.mark.parametrize("source", ["api.cu", "batch.cu", "noalloc.cu", "serve.cu", "color_balanced.cu"])
def test_every_entry_point_catches(source):
    with open(os.path.join(ROOT, "paper_1206_6409_gb300", "csrc", source)) as fh:
        text = fh.read()
    entries = list(re.finditer(r"^(?:extern \"C\" )?int (gencd_\w+)\([^;{}]*\) (try )?\{\n(.*?)^\}\n(GENCD_CATCH)?", text,
                               re.M | re.S))
    assert entries
    for m in entries:
        assert (m.group(2) and m.group(4)) or "catch (" in m.group(3), m.group(1)

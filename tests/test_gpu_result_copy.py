"""Large results to the host when the process cannot start the threads that
back the buffer's pages: the call copies all the same."""
import os
import shutil
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

# every operator new of the armed thread fails
SHIM = r"""
#include <cstdlib>
#include <new>
static thread_local int armed = 0;
extern "C" void arm(int v) { armed = v; }
void *operator new(std::size_t n) {
  void *p = armed ? nullptr : std::malloc(n ? n : 1);
  if (!p) throw std::bad_alloc();
  return p;
}
void operator delete(void *p) noexcept { std::free(p); }
void operator delete(void *p, std::size_t) noexcept { std::free(p); }
"""

CHILD = r"""
import ctypes
import numpy as np
from paper_1708_01608_gb300 import lbm
L = lbm.Lattice("D3Q19", 128, 128, 96, storage="f32")
L.seed_bubbles([[64.0, 64.0, 48.0, 20.0]], 2.0, 0.15, 2.0, 1e-3, 1)
a = L.read("rho")  # 12.6 MB; the library's own buffers exist after it
arm = ctypes.CDLL(None).arm
arm(1)
b = L.read("rho")
arm(0)
assert (a == b).all()
L.close()
print("ok")
"""


def test_read_without_memory_for_threads(tmp_path):
    gxx = shutil.which("g++")
    if gxx is None:
        pytest.skip("no g++")
    src, so = tmp_path / "shim.cpp", tmp_path / "shim.so"
    src.write_text(SHIM)
    subprocess.run([gxx, "-O1", "-shared", "-fPIC", str(src), "-o", str(so)], check=True)
    r = subprocess.run([sys.executable, "-c", CHILD], cwd=ROOT, capture_output=True, text=True,
                       timeout=300, env=dict(os.environ, LD_PRELOAD=str(so)))
    assert r.returncode == 0 and r.stdout.strip().endswith("ok"), r.stderr[-2000:]

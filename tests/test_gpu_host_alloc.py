"""Steps, explicit driving modes and the density PDF allocate nothing on the host: an
allocation that failed there would throw across the C ABI, in steps with work of the
device under way.  A preloaded operator new counts the calling thread's allocations."""
import os
import shutil
import subprocess
import sys

import pytest

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytestmark = pytest.mark.skip(reason="no CUDA device")

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

COUNT = r'''
#include <cstdlib>
#include <new>
static thread_local long on = 0, n = 0;
extern "C" void count_start() { n = 0; on = 1; }
extern "C" long count_end() { on = 0; return n; }
static void* take(size_t s) { n += on; return std::malloc(s ? s : 1); }
static void* need(size_t s) { void* p = take(s); if (!p) throw std::bad_alloc(); return p; }
void* operator new(size_t s) { return need(s); }
void* operator new[](size_t s) { return need(s); }
void* operator new(size_t s, const std::nothrow_t&) noexcept { return take(s); }
void* operator new[](size_t s, const std::nothrow_t&) noexcept { return take(s); }
void operator delete(void* p) noexcept { std::free(p); }
void operator delete[](void* p) noexcept { std::free(p); }
void operator delete(void* p, size_t) noexcept { std::free(p); }
void operator delete[](void* p, size_t) noexcept { std::free(p); }
'''

CHILD = r'''
import ctypes as C, sys
import numpy as np
from paper_2401_06841_gb300 import AdiabaticSolver, Solver, inputs as I
P = C.CDLL(sys.argv[1])
P.count_end.restype = C.c_long
def counted(call):
    P.count_start()
    rc = call()
    n = P.count_end()
    assert rc == 0, rc
    return n
t, d = C.c_double(), C.c_double()
s = Solver(4, 2, precision="f32")
s.set_state(I.random_state(4, 2, seed=3, v_rms=0.3))
s.set_forcing(mach=2.0, seed=3)
s.step(2)  # kernels loaded
h = np.zeros(37)
kv, am = np.array([[1, 0, 0], [-1, 2, 0]], dtype=np.int32), np.ones((2, 3, 2))
a = AdiabaticSolver(4, 2, precision="f32")
a.set_state(I.random_energy_state(4, 2, seed=3, v_rms=0.3, p_mean=5.0, gamma=1.4))
a.set_forcing(mach=2.0, seed=3)
a.step(2)
s.density_pdf(-1.0, 1.0, 37)
print("step", counted(lambda: s.L.dg_step(s.h, 4, 0.0, C.byref(t), C.byref(d))))
print("adi_step", counted(lambda: s.L.dg_adi_step(a.h, 4, 0.0, C.byref(t), C.byref(d))))
print("density_pdf", counted(lambda: s.L.dg_density_pdf(s.h, C.c_double(-1.0), C.c_double(1.0), 37, h.ctypes.data)))
print("forcing_from_modes", counted(lambda: s.L.dg_forcing_from_modes(s.h, 2, kv.ctypes.data, am.ctypes.data)))
'''


@pytest.mark.gpu
def test_no_host_allocation_in_steps_modes_and_pdf(tmp_path):
    cxx = shutil.which("g++") or shutil.which("c++")
    if not cxx:
        pytest.skip("no C++ compiler")
    (tmp_path / "count.cpp").write_text(COUNT)
    so = str(tmp_path / "count.so")
    subprocess.run([cxx, "-std=c++17", "-O1", "-shared", "-fPIC", str(tmp_path / "count.cpp"), "-o", so], check=True)
    env = dict(os.environ, LD_PRELOAD=so, PYTHONPATH=ROOT + os.pathsep + os.environ.get("PYTHONPATH", ""))
    r = subprocess.run([sys.executable, "-c", CHILD, so], cwd=ROOT, env=env, capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stderr
    got = dict(x.split() for x in r.stdout.split("\n") if x)
    assert got == {"step": "0", "adi_step": "0", "density_pdf": "0", "forcing_from_modes": "0"}

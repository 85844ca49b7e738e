"""Scratch from the library's memory pool after cudaDeviceReset: the pool of the context that the reset ended is not used
again; spectra, FW-H sums, contexts and their release work as before it.  In a process of its own (a reset ends the
device's context for everything in the process)."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

CHILD = r"""
import ctypes as C, sys
import numpy as np
sys.path.insert(0, ".")
from paper_2501_05709_gb300 import fr as F
from paper_2501_05709_gb300 import workloads as W
L = F.lib()
rt = C.CDLL([l.split()[-1] for l in open("/proc/self/maps") if "libcudart" in l][0])
def dev(a):
    p = C.c_void_p()
    assert rt.cudaMalloc(C.byref(p), C.c_size_t(a.nbytes)) == 0
    assert rt.cudaMemcpy(p, C.c_void_p(a.ctypes.data), C.c_size_t(a.nbytes), 1) == 0
    return p
def host(p, shape):
    a = np.empty(shape)
    assert rt.cudaMemcpy(C.c_void_p(a.ctypes.data), p, C.c_size_t(a.nbytes), 2) == 0
    return a
rng = np.random.default_rng(0)
x = rng.standard_normal((3, 400))
y, n, dS = W.sphere_surface(1.0, 6, 2 * np.pi / 9)
hist = np.concatenate([np.full((80, len(y), 1), 1.2), np.zeros((80, len(y), 3)), 1e5 + rng.standard_normal((80, len(y), 1))], -1)
obs, M = np.array([[9.0, 1.0, 0.0]]), np.zeros(3)
def calls():
    xd, psd, nf = dev(x), dev(np.zeros((3, 101))), C.c_int()
    assert L.fwh_psd(xd, 3, 400, 400, C.c_double(0.1), 3, psd, 101, C.byref(nf), None) == 0, L.fr_last_error()
    p, nt, t0 = dev(np.zeros((1, 200))), np.zeros(1, np.int32), np.zeros(1)
    d = [dev(np.ascontiguousarray(a)) for a in (hist, y, n, dS)]
    f = C.c_double
    assert L.fwh_integrate(d[0], 80, len(y), d[1], d[2], d[3], f(1e-3), f(0), C.c_void_p(obs.ctypes.data), 1,
                           C.c_void_p(M.ctypes.data), f(340), f(1.2), f(1e5), f(0), 1, p, 200, C.c_void_p(nt.ctypes.data),
                           C.c_void_p(t0.ctypes.data), None) == 0, L.fr_last_error()
    return host(psd, (3, 101)), host(p, (1, 200))[0, :nt[0]]
mesh = W.box_mesh(2, [3, 3], 0.0, 1.0, q=1)
a = calls()
for again in range(2):
    assert rt.cudaDeviceReset() == 0
    b = calls()
    F.fr_mesh_load(mesh, F.options(order=1)).close()
    c = calls()
    assert all(np.array_equal(u, v) and np.array_equal(u, w) and np.any(u) for u, v, w in zip(a, b, c))
print("same after the reset")
"""


def test_scratch_after_a_device_reset():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2501_05709_gb300 import build as B
    B.build()
    r = subprocess.run([sys.executable, "-c", CHILD], cwd=ROOT, capture_output=True, text=True, timeout=120)
    assert r.returncode == 0 and "same after the reset" in r.stdout, r.stdout + r.stderr

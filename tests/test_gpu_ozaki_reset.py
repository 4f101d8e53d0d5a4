"""The product after a reset of the device: its workspace pool ends with the context
that made it. The reset is cudaDeviceReset in a process of its own, between calls, with
nothing in flight; it ends that process's context only."""
import os
import subprocess
import sys

import pytest

from parity_util import have_gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

pytestmark = [pytest.mark.gpu, pytest.mark.skipif(not have_gpu(), reason="needs a GPU")]

CHILD = r"""
import ctypes, numpy as np, paper_2409_11765_gb300 as eng
eng.lib()
rt = ctypes.CDLL("libcudart.so.13")  # the one that the library has loaded

def ok(r):
    assert r == 0, r

rng = np.random.default_rng(5)
for trial in range(3):
    A, B = rng.standard_normal((200, 130)), rng.standard_normal((130, 170))
    C = np.empty((200, 170), order="F")
    dev = []
    for x in (A, B, C):
        p = ctypes.c_void_p()
        ok(rt.cudaMalloc(ctypes.byref(p), ctypes.c_size_t(x.nbytes)))
        f = np.asfortranarray(x)
        ok(rt.cudaMemcpy(p, f.ctypes.data_as(ctypes.c_void_p), ctypes.c_size_t(x.nbytes), 1))
        dev.append(p)
    for again in range(2):
        eng.cmaes_ozaki_dgemm(200, 170, 130, 1.0, dev[0].value, 200, dev[1].value, 130, 0.0, dev[2].value, 200, None)
    ok(rt.cudaMemcpy(C.ctypes.data_as(ctypes.c_void_p), dev[2], ctypes.c_size_t(C.nbytes), 2))
    assert np.abs(C - A @ B).max() < 1e-12 * 130
    for p in dev:
        ok(rt.cudaFree(p))
    ok(rt.cudaDeviceReset())
print("done")
"""


def test_product_after_device_resets():
    env = dict(os.environ)
    env["LD_LIBRARY_PATH"] = "/usr/local/cuda/lib64:" + env.get("LD_LIBRARY_PATH", "")
    r = subprocess.run([sys.executable, "-c", CHILD], cwd=ROOT, env=env, capture_output=True, text=True, timeout=300)
    assert r.stdout.split() == ["done"], (r.returncode, r.stdout, r.stderr)

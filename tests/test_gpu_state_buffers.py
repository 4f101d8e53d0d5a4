"""The pinned buffers that states pass through outlive their handles: handles alive
together have one each, and none is used again after the context that made it."""
import os
import subprocess
import sys

import numpy as np
import pytest

import paper_2409_11765_gb300 as eng
from paper_2409_11765_gb300 import workloads as W
from parity_util import SEED, have_gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

pytestmark = [pytest.mark.gpu, pytest.mark.skipif(not have_gpu(), reason="needs a GPU")]


def handle(n, state):
    h = eng.cmaes_create_batch([n], [12], [np.zeros(n)], [1.0], SEED, eng.cmaes_default_options())
    eng.cmaes_set_state(h, 0, dict(n=n, lam=12, sigma=0.5, **state))
    return h


def test_handles_alive_together_and_after_one_another():
    ns = [5, 40, 40, 200, 300]
    states = [{k: v for k, v in W.random_state(n, SEED, 80 + i).items() if k != "sigma"} for i, n in enumerate(ns)]
    for _ in range(3):
        hs = [handle(n, st) for n, st in zip(ns, states)]
        for order in (range(5), reversed(range(5))):
            for i in order:
                got = eng.cmaes_get_state(hs[i], 0, ns[i])
                for key in ("m", "ps", "pc", "C", "B", "D"):
                    assert np.array_equal(got[key], states[i][key]), (ns[i], key)
        for h in hs:
            eng.cmaes_destroy(h)


CHILD = r"""
import ctypes, numpy as np, paper_2409_11765_gb300 as eng
eng.lib()
rt = ctypes.CDLL("libcudart.so.13")  # the one that the library has loaded
for trial in range(3):
    for n in (10, 100):
        h = eng.cmaes_create_batch([n], [12], [np.full(n, 0.25 * trial)], [1.0], 7, eng.cmaes_default_options(precision=trial))
        eng.cmaes_set_problem(h, 0, eng.OBJ_SPHERE, xstar=np.ones(n))
        assert np.array_equal(eng.cmaes_get_state(h, 0, n)["m"], np.full(n, 0.25 * trial))
        eng.cmaes_step_batch(h, 2)
        assert np.isfinite(eng.cmaes_get_state(h, 0, n)["C"]).all()
        eng.cmaes_destroy(h)
    assert rt.cudaDeviceReset() == 0  # nothing in flight; ends this process's context only
print("done")
"""


def test_handles_after_device_resets():
    env = dict(os.environ)
    env["LD_LIBRARY_PATH"] = "/usr/local/cuda/lib64:" + env.get("LD_LIBRARY_PATH", "")
    r = subprocess.run([sys.executable, "-c", CHILD], cwd=ROOT, env=env, capture_output=True, text=True, timeout=300)
    assert r.stdout.split() == ["done"], (r.returncode, r.stdout, r.stderr)

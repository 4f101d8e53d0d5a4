"""Failing allocations inside cmaes_create, on the CPU: a stand-in for the CUDA runtime
calls it makes (preloaded before libcudart) refuses one of them."""
import os
import subprocess
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

SHIM = r"""
#include <stdlib.h>
#include <string.h>
static int left(const char* what) { /* calls of this kind before the refused one */
  static int count[2];
  const char* v = getenv(what);
  return v ? atoi(v) - count[strcmp(what, "REFUSE_MALLOC") == 0]++ : -1;
}
int cudaMalloc(void** p, size_t n) { if (left("REFUSE_MALLOC") == 0) return 2; *p = malloc(16); return 0; }
int cudaHostAlloc(void** p, size_t n, unsigned f) { if (left("REFUSE_HOST") == 0) return 2; *p = malloc(n); return 0; }
int cudaFree(void* p) { free(p); return 0; }
int cudaFreeHost(void* p) { free(p); return 0; }
int cudaGetDevice(int* d) { *d = 0; return 0; }
int cudaDeviceGetAttribute(int* v, int a, int d) { *v = 152; return 0; }
int cudaFuncGetAttributes(void* a, const void* f) { memset(a, 0, 64); return 0; }
int cudaFuncSetAttribute(const void* f, int a, int v) { return 0; }
int cudaOccupancyMaxActiveBlocksPerMultiprocessor(int* b, const void* f, int t, size_t n) { *b = 1; return 0; }
int cudaStreamCreateWithFlags(void** s, unsigned f) { *s = (void*)8; return 0; }
int cudaStreamDestroy(void* s) { return 0; }
int cudaStreamSynchronize(void* s) { return 0; }
int cudaMemsetAsync(void* p, int v, size_t n, void* s) { return 0; }
int cudaMemcpyAsync(void* d, const void* s, size_t n, int k, void* st) { return 0; }
int cudaGetLastError(void) { return 0; }
const char* cudaGetErrorString(int e) { return "refused"; }
"""

CHILD = r"""
import numpy as np, paper_2409_11765_gb300 as eng
try:
    eng.cmaes_create(10, 10, np.zeros(10), 1.0, 1)
except eng.CmaesError as e:
    print("status", e.status)
"""


@pytest.mark.parametrize("refused", [{"REFUSE_MALLOC": "0"}, {"REFUSE_HOST": "0"}, {"REFUSE_MALLOC": "1"},
                                     {"REFUSE_MALLOC": "2"}], ids=["arena", "state buffer", "status word", "searches"])
def test_refused_allocation_is_out_of_memory(tmp_path, refused):
    import __graft_entry__
    __graft_entry__.build()
    (tmp_path / "shim.c").write_text(SHIM)
    shim = str(tmp_path / "shim.so")
    subprocess.run(["gcc", "-shared", "-fPIC", "-w", "-o", shim, str(tmp_path / "shim.c")], check=True)
    r = subprocess.run([sys.executable, "-c", CHILD], cwd=ROOT, env=dict(os.environ, LD_PRELOAD=shim, **refused),
                       capture_output=True, text=True, timeout=300)
    assert r.stdout.split() == ["status", "2"], (r.stdout, r.stderr)

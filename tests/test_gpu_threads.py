"""Handles of different sizes on different threads: a kernel's dynamic shared-memory
limit belongs to the process, so no launch may depend on a limit that another
handle's launch can lower."""
import threading

import numpy as np
import pytest

import paper_2409_11765_gb300 as eng
from parity_util import SEED, have_gpu

pytestmark = [pytest.mark.gpu, pytest.mark.skipif(not have_gpu(), reason="needs a GPU")]


def one_generation(n, method):
    opt = eng.cmaes_default_options(eig_every=1, eig_method=method, stop_mask=0)
    h = eng.cmaes_create_batch([n], [8], [np.zeros(n)], [1.0], SEED, opt)
    try:
        eng.cmaes_set_problem(h, 0, eng.OBJ_SPHERE, xstar=np.ones(n))
        eng.cmaes_step_batch(h, 1)
        eng.cmaes_sync(h)
    finally:
        eng.cmaes_destroy(h)


@pytest.mark.parametrize("big,small,method", [(160, 40, eng.EIG_AUTO), (160, 70, eng.EIG_AUTO),
                                              (300, 170, eng.EIG_JACOBI)])
def test_sizes_beside_each_other(big, small, method):
    errors = []
    gate = threading.Barrier(2)

    def work(n):
        try:
            for _ in range(300 if big <= 160 else 20):
                gate.wait(30)
                one_generation(n, method)
        except Exception as e:  # noqa: BLE001
            errors.append((n, repr(e)))
            gate.abort()

    threads = [threading.Thread(target=work, args=(n,)) for n in (big, small)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not [e for e in errors if "BrokenBarrier" not in e[1]]

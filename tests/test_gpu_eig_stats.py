"""cmaes_eig_stats counts the sweeps that ran: FP32 ones on every Jacobi route, none on
the tridiagonal route."""
import numpy as np
import pytest

import paper_2409_11765_gb300 as eng
from paper_2409_11765_gb300 import workloads as W
from parity_util import SEED, have_gpu

pytestmark = [pytest.mark.gpu, pytest.mark.skipif(not have_gpu(), reason="needs a GPU")]


@pytest.mark.parametrize("precision", [eng.FP64, eng.MIXED_TF32], ids=["fp64", "tf32"])
@pytest.mark.parametrize("n,method", [(5, eng.EIG_AUTO), (32, eng.EIG_AUTO), (33, eng.EIG_AUTO), (160, eng.EIG_AUTO),
                                      (200, eng.EIG_JACOBI), (200, eng.EIG_AUTO), (40, eng.EIG_TRIDIAGONAL)])
def test_sweeps_are_counted(n, method, precision):
    d = W.random_state(n, SEED, 7)
    opt = eng.cmaes_default_options(eig_every=1, eig_method=method, stop_mask=0, precision=precision)
    h = eng.cmaes_create_batch([n], [12], [np.zeros(n)], [1.0], SEED, opt)
    try:
        eng.cmaes_set_problem(h, 0, eng.OBJ_SPHERE, xstar=np.ones(n))
        turn = W.haar_orthogonal(n, W.rng_for(SEED, 51, n))  # far from the eigenvectors
        eng.cmaes_set_state(h, 0, dict(n=n, lam=12, sigma=0.1, m=np.zeros(n), ps=d["ps"], pc=d["pc"], C=d["C"], B=turn,
                                       D=np.ones(n), gen=3))
        eng.cmaes_step_batch(h, 2)
        st = eng.cmaes_eig_stats(h, 0)
    finally:
        eng.cmaes_destroy(h)
    assert st["decompositions"] == 2
    jacobi = method == eng.EIG_JACOBI or (method == eng.EIG_AUTO and n <= 160)
    assert (st["sweeps32"] >= 4) if jacobi else (st["sweeps32"] == 0)

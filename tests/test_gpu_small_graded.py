"""Searches with n <= 32 whose covariance matrix is graded along the axes (a learned
scaling of separable coordinates) keep the relative accuracy of every eigenvalue, as a
Jacobi method with a relative test on each pair does (Demmel & Veselic 1992)."""
import numpy as np
import pytest

import paper_2409_11765_gb300 as eng
from paper_2409_11765_gb300 import workloads as W
from parity_util import SEED, have_gpu

pytestmark = [pytest.mark.gpu, pytest.mark.skipif(not have_gpu(), reason="needs a GPU")]


def eigenvalues(C):
    """Cyclic Jacobi in extended precision, ascending."""
    A = C.astype(np.longdouble)
    n = len(A)
    for _ in range(40):
        turned = False
        for p in range(n):
            for q in range(p + 1, n):
                if abs(A[p, q]) <= np.longdouble(1e-18) * np.sqrt(A[p, p] * A[q, q]):
                    continue
                turned = True
                th = (A[q, q] - A[p, p]) / (2 * A[p, q])
                t = (1 if th >= 0 else -1) / (abs(th) + np.sqrt(th * th + 1))
                c = 1 / np.sqrt(t * t + 1)
                s, apq = t * c, A[p, q]
                app, aqq = A[p, p] - t * apq, A[q, q] + t * apq
                x, y = A[:, p].copy(), A[:, q].copy()
                A[:, p], A[:, q] = c * x - s * y, s * x + c * y
                A[p, :], A[q, :] = A[:, p], A[:, q]
                A[p, p], A[q, q], A[p, q], A[q, p] = app, aqq, 0, 0
        if not turned:
            return np.sort(np.diag(A))
    raise AssertionError("no convergence")


def generation(n, C, scale, precision):
    """C of a search (its B = I and D = scale) updated and decomposed."""
    opt = eng.cmaes_default_options(eig_every=1, stop_mask=0, precision=precision)
    h = eng.cmaes_create_batch([n], [4], [np.zeros(n)], [1.0], SEED, opt)
    try:
        eng.cmaes_set_problem(h, 0, eng.OBJ_SPHERE, xstar=np.ones(n))
        eng.cmaes_set_state(h, 0, dict(n=n, lam=4, sigma=0.1, m=np.zeros(n), ps=np.zeros(n), pc=np.zeros(n), C=C,
                                       B=np.eye(n), D=scale, gen=3))
        eng.cmaes_step_batch(h, 1)
        return eng.cmaes_get_state(h, 0, n)
    finally:
        eng.cmaes_destroy(h)


@pytest.mark.parametrize("precision", [eng.FP64, eng.MIXED_TF32], ids=["fp64", "tf32"])
@pytest.mark.parametrize("n", [3, 10, 17, 32])
@pytest.mark.parametrize("cond", [1e4, 1e12])
def test_small_eigenvalues(n, cond, precision):
    """A graded matrix with a close pair at its small end, which the FP32 sweeps and the
    first-order corrections leave to the last sweeps."""
    rng = W.rng_for(SEED, 71, n)
    K = np.triu(rng.standard_normal((n, n)) * 0.1 / np.sqrt(n), 1)
    t = np.arange(n) / (n - 2.0)
    t[n - 1] = t[n - 2]
    K[: n - 2, n - 2:] *= 1e-9
    K[n - 2, n - 1] = 7e-7
    scale = np.sqrt(cond) ** -t
    want = (np.eye(n) + K + K.T) * scale[:, None] * scale[None, :]
    # the state whose update is that matrix: the update's terms come from B and D alone
    # (definite states: the guard of an indefinite one would shift the diagonal)
    once, twice = (generation(n, np.diag(k * scale ** 2), scale, precision)["C"] for k in (1.0, 2.0))
    added, keep = 2.0 * once - twice, twice[0, 0] - once[0, 0]
    g = generation(n, (want - added) / keep, scale, precision)
    assert abs(g["C"][n - 2, n - 1]) < 1e-6 * g["C"][n - 1, n - 1]
    want = eigenvalues(0.5 * (g["C"] + g["C"].T))
    # the rotation threshold, 1e-14 a pair, and the rounding of the products that form
    # B^T C B relative to its scaled entries
    tol = n * 1e-14 + 4 * n * n * 2.0 ** -53
    assert np.abs(g["D"] ** 2 / want - 1).max() <= tol
    assert np.abs(g["B"].T @ g["B"] - np.eye(n)).max() <= 1e-13 * n

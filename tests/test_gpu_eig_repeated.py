"""Repeated eigenvalues on the Jacobi routes (n <= 160): groups of them far from their old
basis, and C = I plus the low-rank updates of a descent's first generations."""
import numpy as np
import pytest

import paper_2409_11765_gb300 as eng
from paper_2409_11765_gb300 import workloads as W
from parity_util import SEED, have_gpu

pytestmark = [pytest.mark.gpu, pytest.mark.skipif(not have_gpu(), reason="needs a GPU")]


def check(g, n, precision):
    """B orthonormal to 1e-13 n. B D^2 B^T = C and the eigenvalues to 1e-12 of ||C||, or to the
    entries that the last sweeps leave in X^T C X, n^2 of them below n eps64 max a_ii (4 n eps64
    on mixed handles): the bound that holds where no gap in the spectrum keeps them smaller."""
    B, D, C = g["B"], g["D"], g["C"]
    left = n * n * 2.0 ** -53 * (1 if precision == eng.FP64 else 4)
    tol = max(1e-12, left)
    scale = np.linalg.norm(C)
    assert np.all(np.diff(D) >= 0)
    assert np.abs(B.T @ B - np.eye(n)).max() <= 1e-13 * n
    assert np.linalg.norm((B * D ** 2) @ B.T - C) <= tol * scale
    ev = np.linalg.eigvalsh(C / scale)
    assert np.abs(D ** 2 / scale - ev).max() <= 1e-12 * ev.max() + left * ev.max()


def run(n, lam, gens, precision, state=None):
    opt = eng.cmaes_default_options(eig_every=1, stop_mask=0, precision=precision)
    h = eng.cmaes_create_batch([n], [lam], [np.zeros(n)], [1.0], SEED, opt)
    try:
        eng.cmaes_set_problem(h, 0, eng.OBJ_SPHERE, xstar=np.ones(n))
        if state is not None:
            eng.cmaes_set_state(h, 0, dict(n=n, lam=lam, sigma=0.1, m=np.zeros(n), ps=np.zeros(n), pc=np.zeros(n), gen=3,
                                           **state))
        eng.cmaes_step_batch(h, gens)
        return eng.cmaes_get_state(h, 0, n)
    finally:
        eng.cmaes_destroy(h)


@pytest.mark.parametrize("precision", [eng.FP64, eng.MIXED_TF32], ids=["fp64", "tf32"])
@pytest.mark.parametrize("kind", ["one", "four"])
@pytest.mark.parametrize("n", [10, 32, 33, 40, 64, 100, 131, 150, 160])
def test_groups(n, kind, precision):
    rng = W.rng_for(SEED, 19, n)
    B = W.haar_orthogonal(n, rng)
    d2 = np.ones(n) if kind == "one" else np.repeat([1.0, 2.0, 3.0, 10.0], (n + 3) // 4)[:n]
    C = (B * d2) @ B.T
    turn = np.linalg.qr(np.eye(n) + 0.05 / np.sqrt(n) * rng.standard_normal((n, n)))[0]
    check(run(n, 4, 1, precision, dict(C=0.5 * (C + C.T), B=B @ turn, D=np.sqrt(d2))), n, precision)


@pytest.mark.parametrize("precision", [eng.FP64, eng.MIXED_TF32], ids=["fp64", "tf32"])
@pytest.mark.parametrize("gens", [1, 2, 3, 6, 12])
@pytest.mark.parametrize("n", [10, 32, 33, 40, 100, 131, 160])
def test_first_generations(n, gens, precision):
    for lam in (6, 12, 30, 2 * n):
        check(run(n, lam, gens, precision), n, precision)

"""The fused products of the refined Jacobi eigendecomposition (32 < n <= 160) at the
sizes where they can go wrong: around the steps of 32 k, columns that do and do not
divide over the cluster, each number of columns per thread, odd n, spectra at the ends
of the number range and repeated eigenvalues, several sizes in one batch, and a size
above the fused range beside them."""
import numpy as np
import pytest

import paper_2409_11765_gb300 as eng
from paper_2409_11765_gb300 import workloads as W
from parity_util import SEED, have_gpu
from test_gpu_trd_reduce import check, spectrum

pytestmark = [pytest.mark.gpu, pytest.mark.skipif(not have_gpu(), reason="needs a GPU")]


def decompose(ns, kind, precision=eng.FP64, poison=None):
    """C after one update is decomposed, warm-started from the basis of a nearby C."""
    opt = eng.cmaes_default_options(eig_every=1, eig_method=eng.EIG_JACOBI, stop_mask=0, precision=precision)
    h = eng.cmaes_create_batch(ns, [4] * len(ns), [np.zeros(n) for n in ns], [1.0] * len(ns), SEED, opt)
    try:
        for i, n in enumerate(ns):
            rng = W.rng_for(SEED, 19, n)
            B = W.haar_orthogonal(n, rng)
            d2 = spectrum(kind, n)
            C = np.eye(n) if kind == "identity" else (B * d2) @ B.T
            C = 0.5 * (C + C.T)
            if poison is not None:
                C[n // 2, 3] = C[3, n // 2] = poison
            turn = np.linalg.qr(np.eye(n) + 0.05 / np.sqrt(n) * rng.standard_normal((n, n)))[0]
            eng.cmaes_set_problem(h, i, eng.OBJ_SPHERE, xstar=np.ones(n))
            eng.cmaes_set_state(h, i, dict(n=n, lam=4, sigma=0.1, m=np.zeros(n), ps=np.zeros(n), pc=np.zeros(n),
                                           C=C, B=B @ turn, D=np.sqrt(d2), gen=3))
        eng.cmaes_step_batch(h, 1)
        eng.cmaes_sync(h)
        return [eng.cmaes_get_state(h, i, n) for i, n in enumerate(ns)]
    finally:
        eng.cmaes_destroy(h)


@pytest.mark.parametrize("precision", [eng.FP64, eng.MIXED_TF32], ids=["fp64", "tf32"])
@pytest.mark.parametrize("n", [33, 40, 41, 63, 64, 65, 95, 97, 100, 127, 128, 129, 145, 159, 160])
def test_sizes(n, precision):
    check(decompose([n], "spread", precision)[0], n)


@pytest.mark.parametrize("kind", ["wide", "rank-one", "tiny", "huge"])
@pytest.mark.parametrize("n", [40, 131])
def test_ranges(n, kind):
    check(decompose([n], kind)[0], n)


@pytest.mark.parametrize("n", [40, 131])
def test_repeated_eigenvalues(n):
    """Exactly equal eigenvalues: differences of zero in both halves of a correction."""
    g = decompose([n], "identity")[0]
    assert np.isfinite(g["B"]).all() and np.all(np.diff(g["D"]) >= 0)


def test_batch():
    ns = [160, 33, 100, 10, 200] * 8
    got = decompose(ns, "spread")
    for n, g in list(zip(ns, got))[:5]:
        check(g, n)
    for n, g in zip(ns[5:], got[5:]):
        assert np.all(np.diff(g["D"]) >= 0) and np.abs(g["B"].T @ g["B"] - np.eye(n)).max() <= 1e-13 * n


def test_not_a_number_stays_one():
    g = decompose([64], "spread", poison=np.nan)[0]
    assert not np.isfinite(g["D"]).all()

"""The fixed-point Householder reduction at the sizes where it can go wrong: CTA
counts that do and do not divide n, one row more or less than a warp, a work
unit or a CTA's threads, columns in shared memory and in HBM, groups of one CTA,
and the spectra at the ends of its number range."""
import numpy as np
import pytest

import paper_2409_11765_gb300 as eng
from paper_2409_11765_gb300 import workloads as W
from parity_util import SEED, have_gpu

pytestmark = [pytest.mark.gpu, pytest.mark.skipif(not have_gpu(), reason="needs a GPU")]


def spectrum(kind, n):
    t = np.arange(n) / max(1, n - 1)
    return {"spread": 10.0 ** t, "wide": 10.0 ** (12.0 * t - 12.0), "rank-one": np.r_[1.0 + 1e-3 * t[1:], 1e4],
            "tiny": 1e-120 * (1.0 + t), "huge": 1e120 * (1.0 + t), "identity": np.ones(n)}[kind]


def decompose(ns, kind):
    """Decomposes C after one update (c_1, c_mu small: its spectrum is the state's)."""
    opt = eng.cmaes_default_options(eig_every=1, eig_method=eng.EIG_TRIDIAGONAL, stop_mask=0)
    h = eng.cmaes_create_batch(ns, [4] * len(ns), [np.zeros(n) for n in ns], [1.0] * len(ns), SEED, opt)
    try:
        for i, n in enumerate(ns):
            rng = W.rng_for(SEED, 9, n)
            B = W.haar_orthogonal(n, rng)
            d2 = spectrum(kind, n)
            C = np.eye(n) if kind == "identity" else (B * d2) @ B.T
            C = 0.5 * (C + C.T)
            eng.cmaes_set_problem(h, i, eng.OBJ_SPHERE, xstar=np.ones(n))
            eng.cmaes_set_state(h, i, dict(n=n, lam=4, sigma=0.1, m=np.zeros(n), ps=np.zeros(n), pc=np.zeros(n),
                                           C=C, B=B, D=np.sqrt(d2), gen=3))
        eng.cmaes_step_batch(h, 1)
        eng.cmaes_sync(h)
        return [eng.cmaes_get_state(h, i, n) for i, n in enumerate(ns)]
    finally:
        eng.cmaes_destroy(h)


def check(g, n):
    """The contract of the decomposition: B orthonormal to 1e-13 n, B D^2 B^T = C to
    1e-12 ||C||, ascending eigenvalues (the bounds of the parity tests)."""
    B, D, C = g["B"], g["D"], g["C"]
    scale = np.linalg.norm(C)
    assert np.all(np.diff(D) >= 0)
    assert np.abs(B.T @ B - np.eye(n)).max() <= 1e-13 * n
    assert np.linalg.norm((B * D ** 2) @ B.T - C) <= 1e-12 * scale
    ev = np.linalg.eigvalsh(C / scale)
    assert np.abs(D ** 2 / scale - ev).max() <= 1e-12 * ev.max()


@pytest.mark.parametrize("n", [33, 34, 63, 64, 65, 127, 129, 255, 257, 513, 608, 609, 1025])
def test_sizes(n):
    check(decompose([n], "spread")[0], n)


@pytest.mark.parametrize("kind", ["wide", "rank-one", "tiny", "huge", "identity"])
@pytest.mark.parametrize("n", [40, 200])
def test_ranges(n, kind):
    check(decompose([n], kind)[0], n)


@pytest.mark.parametrize("ns", [[1800], [1500, 700, 33], [900] * 6, [100] * 40, [64, 1100] + [200] * 30 + [35] * 200],
                         ids=["hbm", "shared", "six", "forty", "many"])
def test_groups(ns):
    """Shares of the GPU: one search that no longer fits in shared memory, uneven
    ones with their columns in it, and batches whose searches get one CTA."""
    got = decompose(ns, "spread")
    seen = {}
    for n, g in zip(ns, got):
        if n not in seen:  # (the numpy checks of one search of each size)
            check(g, n)
            seen[n] = g
        assert np.isfinite(g["B"]).all() and np.all(np.diff(g["D"]) >= 0)

"""The integer products behind the FP64 GEMM tile, through the allocation-free
evaluation: ragged tiles and K steps, points of very different scale side by side,
zeros, and infinite and NaN coordinates beside finite points."""
import numpy as np
import pytest

import paper_2409_11765_gb300 as eng
from paper_2409_11765_gb300 import workloads as W
from parity_util import SEED, have_gpu

pytestmark = [pytest.mark.gpu, pytest.mark.skipif(not have_gpu(), reason="needs a GPU")]


def evaluate(X, Q, lamdiag, xstar):
    import torch
    n, lam = X.shape
    dev = [torch.from_numpy(np.ascontiguousarray(a)).cuda() for a in (X.T, Q.T, lamdiag, xstar)]
    f = torch.zeros(lam, dtype=torch.float64, device="cuda")
    eng.cmaes_evaluate_noalloc(eng.OBJ_ELLIPSOID, n, lam, dev[0].data_ptr(), n, dev[1].data_ptr(), n,
                               dev[2].data_ptr(), dev[3].data_ptr(), f.data_ptr(), None)
    torch.cuda.synchronize()
    return f.cpu().numpy()


def check(X, Q, lamdiag, xstar):
    """f = sum lambda u^2 with u = Q r: each u is off by at most the entries'
    rounding and the steps' (2^-57 of the largest |q| and |r|, n times, a factor
    of four for the step sums), f by twice that times lambda |u| and n roundings."""
    n = X.shape[0]
    f = evaluate(X, Q, lamdiag, xstar)
    r = (X - xstar[:, None]).astype(np.longdouble)
    with np.errstate(all="ignore"):
        u = Q.astype(np.longdouble) @ r
        want = (lamdiag[:, None] * u * u).sum(0)
        du = 4 * n * 2.0 ** -57 * np.abs(Q).max(1)[:, None] * np.abs(r).max(0)[None, :]
        tol = (lamdiag[:, None] * (2 * np.abs(u) * du + du * du)).sum(0) + (n + 4) * 2.0 ** -53 * np.abs(want)
    fine = np.isfinite(r).all(0)
    assert (np.abs(f[fine] - want[fine]) <= tol[fine]).all()
    assert not np.isfinite(f[~fine]).any()


@pytest.mark.parametrize("n,lam", [(1, 1), (2, 3), (31, 33), (32, 64), (33, 65), (63, 1), (64, 129), (65, 200), (130, 70)])
def test_shapes(n, lam):
    rng = W.rng_for(SEED, 12, n)
    check(rng.standard_normal((n, lam)), W.haar_orthogonal(n, rng), W.ellipsoid_diag(n, 1e6), rng.standard_normal(n))


@pytest.mark.parametrize("n", [40, 100])
def test_scales_and_specials(n):
    rng = W.rng_for(SEED, 13, n)
    lam = 150
    X = rng.standard_normal((n, lam)) * 10.0 ** rng.integers(-70, 70, lam)[None, :]
    X[:, 5] = 0.0
    X[3::7, 9] *= 1e-200
    X[n // 2, 20] = np.nan
    X[1, 64] = np.inf
    X[n - 1, 65] = -np.inf
    check(X, W.haar_orthogonal(n, rng), np.ones(n), np.zeros(n))

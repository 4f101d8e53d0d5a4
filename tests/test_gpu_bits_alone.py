"""A search gives the same bits alone and inside any batch: on the tridiagonal route
whatever the number of eigenvalues of the whole handle, which decides how the
eigenvalues' bisection is spread over lanes."""
import numpy as np
import pytest

import paper_2409_11765_gb300 as eng
from paper_2409_11765_gb300 import workloads as W
from parity_util import SEED, have_gpu
from test_gpu_trd_reduce import spectrum

pytestmark = [pytest.mark.gpu, pytest.mark.skipif(not have_gpu(), reason="needs a GPU")]


def first_search(ns, precision, kind):
    """The first of the searches after one generation and decomposition."""
    opt = eng.cmaes_default_options(eig_every=1, eig_method=eng.EIG_TRIDIAGONAL, stop_mask=0, precision=precision)
    h = eng.cmaes_create_batch(ns, [12] * len(ns), [np.zeros(n) for n in ns], [1.0] * len(ns), SEED, opt)
    try:
        for i, n in enumerate(ns):
            eng.cmaes_set_problem(h, i, eng.OBJ_SPHERE, xstar=np.ones(n))
        n = ns[0]
        B = W.haar_orthogonal(n, W.rng_for(SEED, 31, n))
        d2 = spectrum(kind, n)
        C = (B * d2) @ B.T
        eng.cmaes_set_state(h, 0, dict(n=n, lam=12, sigma=0.1, m=np.zeros(n), ps=np.zeros(n), pc=np.zeros(n),
                                       C=0.5 * (C + C.T), B=B, D=np.sqrt(d2), gen=3))
        eng.cmaes_step_batch(h, 1)
        return eng.cmaes_get_state(h, 0, n)
    finally:
        eng.cmaes_destroy(h)


@pytest.mark.parametrize("precision", [eng.FP64, eng.MIXED_TF32], ids=["fp64", "tf32"])
@pytest.mark.parametrize("n,kind", [(33, "spread"), (200, "spread"), (257, "wide"), (300, "rank-one")])
def test_tridiagonal_route(n, kind, precision):
    alone = first_search([n], precision, kind)
    # 16, 8, 4 lanes and 1 per eigenvalue; the reduction's columns in shared memory and in HBM,
    # CTAs of 512 and of 256 threads, one launch and several
    for neighbours in ([400], [400] * 4, [400] * 11, [400] * 36, [64] * 140, [64] * 320, [600] * 100):
        batch = first_search([n] + neighbours, precision, kind)
        for key in ("m", "ps", "pc", "C", "B", "D"):
            assert np.array_equal(alone[key], batch[key]), (len(neighbours), key)
        assert alone["sigma"] == batch["sigma"]


SMALL = [(1, 2), (1, 700), (2, 6), (2, 1000), (3, 7), (5, 8), (10, 10), (10, 204), (16, 128), (17, 100), (20, 12),
         (31, 14), (31, 66), (32, 14), (32, 64)]


def small_search(n, lam, kind, gens, neighbour=False, profiling=False, tell=False, **over):
    """State and last generation of an FP64 search with n <= 32 after `gens` generations."""
    opt = eng.cmaes_default_options(**over)
    ns, lams = [n] + [40] * neighbour, [lam] + [12] * neighbour
    prob = W.make_problem(kind, n, SEED, 61)
    d = W.random_state(n, SEED, 7)
    h = eng.cmaes_create_batch(ns, lams, [np.zeros(k) for k in ns], [0.7] * len(ns), SEED, opt)
    try:
        eng.cmaes_set_problem(h, 0, kind, prob.Q, prob.lamdiag, prob.xstar)
        if neighbour:
            eng.cmaes_set_problem(h, 1, eng.OBJ_SPHERE, xstar=np.ones(40))
        eng.cmaes_set_state(h, 0, dict(n=n, lam=lam, sigma=0.3, m=d["m"], ps=d["ps"], pc=d["pc"], C=d["C"], B=d["B"],
                                       D=d["D"], gen=5))
        eng.cmaes_set_profiling(h, profiling)
        if tell:
            for _ in range(gens):
                if eng.cmaes_query(h, 0)["done"]:
                    break
                eng.cmaes_tell(h, 0, evaluate(kind, prob, eng.cmaes_ask(h, 0, n)))
        else:
            eng.cmaes_step_batch(h, gens)
        return eng.cmaes_get_state(h, 0, n), eng.cmaes_get_generation(h, 0, n)
    finally:
        eng.cmaes_destroy(h)


def evaluate(kind, prob, X):
    """f of the columns of X by the allocation-free evaluation."""
    import torch
    n, lam = X.shape
    dev = [torch.from_numpy(np.ascontiguousarray(a)).cuda() if a is not None else None
           for a in (X.T, None if prob.Q is None else prob.Q.T, prob.lamdiag, prob.xstar)]
    f = torch.zeros(lam, dtype=torch.float64, device="cuda")
    ptr = [0 if a is None else a.data_ptr() for a in dev]
    eng.cmaes_evaluate_noalloc(kind, n, lam, ptr[0], n, ptr[1], n, ptr[2], ptr[3], f.data_ptr(), None)
    torch.cuda.synchronize()
    return f.cpu().numpy()


def same(a, b):
    for key in ("m", "ps", "pc", "C", "B", "D", "best_x", "hist"):
        assert np.array_equal(a[0][key], b[0][key], equal_nan=True), key
    for key in ("sigma", "best_f", "gen", "restart", "lam", "done", "flags"):
        assert a[0][key] == b[0][key], key
    for x, y in zip(a[1], b[1]):
        assert np.array_equal(x, y)


@pytest.mark.parametrize("kind", [W.ELLIPSOID, W.RASTRIGIN, W.SPHERE])
@pytest.mark.parametrize("n,lam", SMALL)
def test_small_searches(n, lam, kind):
    """Whole generations in one launch against the phase kernels, which run beside a larger
    search, under profiling, and between ask and tell."""
    alone = small_search(n, lam, kind, 12)
    same(alone, small_search(n, lam, kind, 12, neighbour=True))
    same(alone, small_search(n, lam, kind, 12, profiling=True))
    same(alone, small_search(n, lam, kind, 12, tell=True))


@pytest.mark.parametrize("n,lam", [(3, 7), (10, 10), (24, 20)])
def test_small_searches_through_restarts(n, lam):
    over = dict(max_restarts=2, max_iter=17, f_target=-1.0)
    alone = small_search(n, lam, W.RASTRIGIN, 60, **over)
    assert alone[0]["restart"] > 0
    same(alone, small_search(n, lam, W.RASTRIGIN, 60, neighbour=True, **over))
    same(alone, small_search(n, lam, W.RASTRIGIN, 60, profiling=True, **over))


def test_many_small_searches():
    """Beside so many that the kernel's denser form runs."""
    n, lam = 10, 10
    prob = W.make_problem(W.RASTRIGIN, n, SEED, 61)
    got = []
    for count in (1, 700):
        opt = eng.cmaes_default_options(max_restarts=1, max_iter=9)
        h = eng.cmaes_create_batch([n] * count, [lam] * count, [np.ones(n)] * count, [0.7] * count, SEED, opt)
        try:
            for i in range(count):
                eng.cmaes_set_problem(h, i, W.RASTRIGIN, prob.Q, prob.lamdiag, prob.xstar)
            eng.cmaes_step_batch(h, 15)
            got.append((eng.cmaes_get_state(h, 0, n), eng.cmaes_get_generation(h, 0, n)))
        finally:
            eng.cmaes_destroy(h)
    same(*got)


@pytest.mark.parametrize("precision", [eng.FP64, eng.MIXED_TF32], ids=["fp64", "tf32"])
@pytest.mark.parametrize("n,count", [(33, 100), (40, 12), (40, 200), (41, 60), (80, 100), (81, 20), (160, 30)])
def test_jacobi_route(n, count, precision):
    """With clusters of 16 CTAs alone, and of 8, 4 and 2 in a batch."""
    d = W.random_state(n, SEED, 7, cond=30.0)
    got = []
    for searches in (1, count):
        opt = eng.cmaes_default_options(eig_every=1, stop_mask=0, precision=precision)
        h = eng.cmaes_create_batch([n] * searches, [12] * searches, [np.zeros(n)] * searches, [1.0] * searches, SEED, opt)
        try:
            for i in range(searches):
                eng.cmaes_set_problem(h, i, eng.OBJ_SPHERE, xstar=np.ones(n))
            eng.cmaes_set_state(h, 0, dict(n=n, lam=12, sigma=0.3, m=d["m"], ps=d["ps"], pc=d["pc"], C=d["C"],
                                           B=d["B"], D=d["D"], gen=5))
            eng.cmaes_step_batch(h, 3)
            got.append((eng.cmaes_get_state(h, 0, n), eng.cmaes_get_generation(h, 0, n)))
        finally:
            eng.cmaes_destroy(h)
    same(*got)


@pytest.mark.parametrize("n,lam", [(40, 30), (100, 64), (161, 70)])
def test_fp64_products(n, lam):
    """The products of a few tiles and of more than the GPU has SMs."""
    d = W.random_state(n, SEED, 7, cond=30.0)
    prob = W.make_problem(W.RASTRIGIN, n, SEED, 61)
    got = []
    for searches in (1, 160):
        opt = eng.cmaes_default_options(eig_every=1, stop_mask=0)
        h = eng.cmaes_create_batch([n] * searches, [lam] * searches, [np.zeros(n)] * searches, [1.0] * searches, SEED, opt)
        try:
            for i in range(searches):
                eng.cmaes_set_problem(h, i, W.RASTRIGIN, prob.Q, prob.lamdiag, prob.xstar)
            eng.cmaes_set_state(h, 0, dict(n=n, lam=lam, sigma=0.3, m=d["m"], ps=d["ps"], pc=d["pc"], C=d["C"],
                                           B=d["B"], D=d["D"], gen=5))
            eng.cmaes_step_batch(h, 3)
            got.append((eng.cmaes_get_state(h, 0, n), eng.cmaes_get_generation(h, 0, n)))
        finally:
            eng.cmaes_destroy(h)
    same(*got)

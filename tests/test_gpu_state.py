"""States written and read back through one launch: around the 32 x 32 tiles, on both
sides of the largest size whose matrices go through the buffer, with fields left out,
with a history longer than its ring, and the B diag(D) that sampling uses."""
import numpy as np
import pytest

import paper_2409_11765_gb300 as eng
from paper_2409_11765_gb300 import workloads as W
from parity_util import SEED, have_gpu

pytestmark = [pytest.mark.gpu, pytest.mark.skipif(not have_gpu(), reason="needs a GPU")]
FIELDS = ("m", "ps", "pc", "D", "best_x", "C", "B")


def state(n, seed, lam=12):
    rng = W.rng_for(SEED, 21, seed)
    A = rng.standard_normal((n, n))
    return dict(n=n, lam=lam, sigma=0.25, best_f=3.5, gen=7, restart=1, m=rng.standard_normal(n),
                ps=rng.standard_normal(n), pc=rng.standard_normal(n), D=1.0 + rng.random(n),
                best_x=rng.standard_normal(n), C=A @ A.T, B=np.linalg.qr(A)[0])


def handle(ns, precision=eng.FP64):
    h = eng.cmaes_create_batch(ns, [12] * len(ns), [np.zeros(n) for n in ns], [1.0] * len(ns), SEED,
                               eng.cmaes_default_options(precision=precision, stop_mask=0))
    for i, n in enumerate(ns):
        eng.cmaes_set_problem(h, i, eng.OBJ_SPHERE, xstar=np.ones(n))
    return h


@pytest.mark.parametrize("precision", [eng.FP64, eng.MIXED_TF32, eng.MIXED_BF16])
def test_round_trip(precision):
    ns = [2, 31, 32, 33, 64, 100, 255, 256, 257, 300]
    h = handle(ns, precision)
    try:
        want = [state(n, i) for i, n in enumerate(ns)]
        for i, d in enumerate(want):
            eng.cmaes_set_state(h, i, d)
        for i, n in enumerate(ns):
            g = eng.cmaes_get_state(h, i, n)
            for k in FIELDS:
                assert np.array_equal(g[k], want[i][k]), (n, k)
            assert (g["sigma"], g["best_f"], g["gen"], g["restart"], g["lam"]) == (0.25, 3.5, 7, 1, 12)
            # a part of the state: the rest keeps its values
            eng.cmaes_set_state(h, i, dict(n=n, lam=12, sigma=0.5, ps=np.ones(n)))
            g = eng.cmaes_get_state(h, i, n)
            assert np.array_equal(g["ps"], np.ones(n)) and g["sigma"] == 0.5
            for k in FIELDS:
                assert k == "ps" or np.array_equal(g[k], want[i][k]), (n, k)
    finally:
        eng.cmaes_destroy(h)


@pytest.mark.parametrize("precision", [eng.FP64, eng.MIXED_TF32])
@pytest.mark.parametrize("n", [33, 256, 257])
def test_parts_equal_the_whole(n, precision):
    """Restored at once or field by field (D and B each without the other), the next
    generation draws the same points."""
    d = state(n, 3)
    out = []
    for parts in ([FIELDS], [("D",), ("B",), ("m", "ps", "pc", "best_x", "C")], [("B",), ("D", "C", "m"), ("ps", "pc", "best_x")]):
        h = handle([n], precision)
        try:
            for p in parts:
                eng.cmaes_set_state(h, 0, {k: v for k, v in d.items() if k in p or k not in FIELDS})
            eng.cmaes_step_batch(h, 1)
            eng.cmaes_sync(h)
            out.append(eng.cmaes_get_state(h, 0, n))
        finally:
            eng.cmaes_destroy(h)
    for g in out[1:]:
        for k in FIELDS:
            assert np.array_equal(g[k], out[0][k]), k


def test_history():
    n, lam = 40, 12
    h = handle([n])
    try:
        length = 10 + int(np.ceil(30.0 * n / lam))
        hist = np.arange(length + 25, dtype=float)
        eng.cmaes_set_state(h, 0, dict(state(n, 5), hist=hist))
        assert np.array_equal(eng.cmaes_get_state(h, 0, n)["hist"], hist[25:])
        eng.cmaes_step_batch(h, 3)
        eng.cmaes_sync(h)
        assert np.array_equal(eng.cmaes_get_state(h, 0, n)["hist"][:-3], hist[28:])
    finally:
        eng.cmaes_destroy(h)

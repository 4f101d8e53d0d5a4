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
    for neighbours in ([400], [400] * 3, [400] * 8, [400] * 18):  # below and above 700, 2500 and 7000 eigenvalues
        batch = first_search([n] + neighbours, precision, kind)
        for key in ("m", "ps", "pc", "C", "B", "D"):
            assert np.array_equal(alone[key], batch[key]), (len(neighbours), key)
        assert alone["sigma"] == batch["sigma"]

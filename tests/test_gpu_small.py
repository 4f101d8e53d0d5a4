"""Small searches, whose generations run in one CTA each: a teacher-forced
generation against the oracle at the ends of the range (one coordinate, odd
sizes, n = 32, the largest population panel and the first one beyond it), and the
same bits whether the generations come in one call or one by one."""
import numpy as np
import pytest

import paper_2409_11765_gb300 as eng
from paper_2409_11765_gb300 import workloads as W
from parity_util import SEED, check_generation, have_gpu, teacher_forced

pytestmark = [pytest.mark.gpu, pytest.mark.skipif(not have_gpu(), reason="needs a GPU")]

SHAPES = [(1, 2), (1, 2048), (1, 2049), (2, 5), (3, 682), (3, 683), (5, 7), (31, 14), (31, 66), (31, 67), (32, 64),
          (32, 2)]


@pytest.mark.parametrize("n,lam", SHAPES)
def test_teacher_forced_generation(n, lam):
    gpu, ora = teacher_forced([n], [lam], [1 + (n + lam) % 3], [W.random_state(n, SEED, 300 + n)], eig_every=1)
    check_generation(gpu, ora)


def test_one_call_or_many():
    shapes = [s for s in SHAPES if s[0] * s[1] <= 2048]

    def run(calls):
        opt = eng.cmaes_default_options(max_restarts=3)
        h = eng.cmaes_create_batch([n for n, _ in shapes], [lam for _, lam in shapes],
                                   [W.start_point(n, -4, 4, SEED, 70 + i) for i, (n, _) in enumerate(shapes)],
                                   [1.0] * len(shapes), SEED, opt)
        try:
            for i, (n, _) in enumerate(shapes):
                p = W.make_problem(1 + i % 3, n, SEED, 70 + i, cond=1e3)
                eng.cmaes_set_problem(h, i, p.kind, p.Q, p.lamdiag, p.xstar)
            for _ in range(calls):
                eng.cmaes_step_batch(h, 12 // calls)
            eng.cmaes_sync(h)
            return [(eng.cmaes_get_state(h, i, n), eng.cmaes_get_generation(h, i, n))
                    for i, (n, _) in enumerate(shapes)]
        finally:
            eng.cmaes_destroy(h)

    for (a, la), (b, lb) in zip(run(1), run(12)):
        for k in ("m", "ps", "pc", "C", "B", "D", "hist", "best_x"):
            assert np.array_equal(a[k], b[k], equal_nan=True), k
        assert all(np.array_equal(p, q) for p, q in zip(la, lb))
        assert (a["gen"], a["restart"], a["flags"], a["sigma"]) == (b["gen"], b["restart"], b["flags"], b["sigma"])

"""The reduction of a batch with more large searches than the GPU has CTAs to spare:
several launches, largest searches first, each search in exactly one of them."""
import numpy as np
import pytest

from parity_util import have_gpu
from test_gpu_trd_reduce import check, decompose

pytestmark = [pytest.mark.gpu, pytest.mark.skipif(not have_gpu(), reason="needs a GPU")]


@pytest.mark.parametrize("ns", [[520] * 90 + [170] * 10, [170] * 5 + [600, 33, 520] * 27], ids=["sorted", "mixed"])
def test_several_launches(ns):
    got = decompose(ns, "spread")
    seen = {}
    for n, g in zip(ns, got):
        if n not in seen:
            check(g, n)
            seen[n] = g
        # searches of one size share their matrix, not their paths: eigenvalues agree to
        # the update's size, orthogonality holds in each
        assert np.all(np.diff(g["D"]) >= 0)
        assert np.abs(g["B"].T @ g["B"] - np.eye(n)).max() <= 1e-13 * n

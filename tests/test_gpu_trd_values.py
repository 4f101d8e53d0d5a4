"""Eigenvalues and eigenvectors of T at the sizes where the counts and solves can
go wrong: row counts around their unrolled groups (4, 8 and 16 rows), each number
of lanes per eigenvalue, blocks of a split T, clustered and graded spectra."""
import numpy as np
import pytest

from parity_util import have_gpu
from test_gpu_trd_reduce import check, decompose

pytestmark = [pytest.mark.gpu, pytest.mark.skipif(not have_gpu(), reason="needs a GPU")]


# one search each: 16 lanes up to 700 eigenvalues, 8 up to 2500
@pytest.mark.parametrize("n", [35, 36, 37, 41, 48, 49, 50, 81, 699, 701])
def test_row_groups(n):
    check(decompose([n], "spread")[0], n)


# 4 lanes (2500 < eigenvalues <= 7000), 1 lane above
@pytest.mark.parametrize("ns", [[400] * 7, [170] * 45], ids=["four-lanes", "one-lane"])
def test_lanes(ns):
    for g in decompose(ns, "spread")[:3]:
        check(g, ns[0])


@pytest.mark.parametrize("kind", ["identity", "rank-one", "wide"])
@pytest.mark.parametrize("n", [100, 300, 720])
def test_split_and_clustered(n, kind):
    g = decompose([n], kind)[0]
    check(g, n)
    if kind == "identity":  # C is a multiple of I plus a rank-three update
        assert np.ptp(g["D"][: n - 4]) <= 1e-12 * g["D"][-1]

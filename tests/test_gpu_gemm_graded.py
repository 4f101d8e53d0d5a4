"""The FP64 GEMM tile on operands where large entries do not meet large ones: a sum's
error is bounded by sum |a b|, as that of FP64 multiply-adds is, and not only by the
largest entries of a row and a column."""
import numpy as np
import pytest

import paper_2409_11765_gb300 as eng
from paper_2409_11765_gb300 import workloads as W
from parity_util import SEED, have_gpu
from test_gpu_gemm_tile import evaluate

pytestmark = [pytest.mark.gpu, pytest.mark.skipif(not have_gpu(), reason="needs a GPU")]


def check(X, Q, lamdiag):
    """f = sum lambda u^2, u = Q x, x* = 0. A step of K terms on integers rounds the entries at
    2^-58 of the scales and leaves their low limbs' product out, 3 K 2^-58 of the scales'
    product, of which sum |q x| is at least 2^-4 (or the step is in FP64: K 2^-53 sum |q x|):
    1.5 n 2^-53 sum |q x| for all steps, their own sums 0.1 n 2^-53 more. f is off by twice that
    times lambda |u| and n + 4 roundings of its own."""
    n = X.shape[0]
    f = evaluate(X, Q, lamdiag, np.zeros(n))
    q, x = Q.astype(np.longdouble), X.astype(np.longdouble)
    u = q @ x
    du = 2 * n * np.longdouble(2.0) ** -53 * (np.abs(q) @ np.abs(x))
    want = (lamdiag[:, None] * u * u).sum(0)
    tol = (lamdiag[:, None] * (2 * np.abs(u) * du + du * du)).sum(0) + (n + 4) * np.longdouble(2.0) ** -53 * want
    assert (np.abs(f - want) <= tol).all(), float((np.abs(f - want) / tol).max())


@pytest.mark.parametrize("n", [2, 10, 33, 64, 100])
@pytest.mark.parametrize("cond", [1e6, 1e12, 1e30])
def test_axis_aligned(n, cond):
    """Q = I on points whose coordinates have the scales of a converged search: u = x exactly."""
    lam = W.ellipsoid_diag(n, cond)
    X = W.rng_for(SEED, 41, n).standard_normal((n, 70)) / np.sqrt(lam)[:, None]
    check(X, np.eye(n), lam)


@pytest.mark.parametrize("n", [33, 100])
def test_graded_rows_against_graded_columns(n):
    """Rows that fall by 2^-60 towards one end, columns that fall towards the other."""
    rng = W.rng_for(SEED, 42, n)
    fall = 2.0 ** np.linspace(0, -60, n)
    check(rng.standard_normal((n, 66)) * fall[::-1, None], rng.standard_normal((n, n)) * fall[None, :], np.ones(n))


def test_small_entries_only_meet_large_ones():
    Q = np.array([[1.0, 2.0 ** -60], [2.0 ** -60, 1.0]])
    X = np.array([[2.0 ** -60, 0.0, 3.0], [1.0, 5e-324, 2.0 ** -1030]])
    u = np.array([[2.0 ** -59, 0.0, 3.0], [1.0, 0.0, 3.0 * 2.0 ** -60]])
    assert np.array_equal(evaluate(X, Q, np.array([1.0, 0.0]), np.zeros(2)), u[0] ** 2)
    assert np.array_equal(evaluate(X, Q, np.array([0.0, 1.0]), np.zeros(2)), u[1] ** 2)
    # subnormal entries count
    tiny = np.array([[2.0 ** -1060, 2.0 ** -1030], [2.0 ** -1070, 0.0]])
    got = evaluate(tiny * 2.0 ** 0, np.eye(2), np.full(2, 2.0 ** 1000), np.zeros(2))
    assert np.array_equal(got, (np.full((2, 1), 2.0 ** 1000) * tiny * tiny).sum(0))


def test_neighbours_in_a_tile_do_not_show():
    """A point's value is the same beside NaN, infinite and graded points as alone."""
    n = 40
    rng = W.rng_for(SEED, 43, n)
    Q = W.haar_orthogonal(n, rng)
    X = rng.standard_normal((n, 64))
    lam = W.ellipsoid_diag(n, 1e6)
    want = evaluate(X, Q, lam, np.zeros(n))
    Y = X.copy()
    Y[3, 7], Y[5, 9] = np.nan, np.inf
    Y[:, 11] *= 2.0 ** -np.arange(n)
    got = evaluate(Y, Q, lam, np.zeros(n))
    same = [k for k in range(64) if k not in (7, 9, 11)]
    assert np.array_equal(got[same], want[same])

"""In-HBM panel kernels of the factorizations at the edges of their blocks.

Cholesky: orders around the 16-column sub-blocks and the 64-order block, a pivot that fails at
every kind of place, and pivots outside the range of the corrected root.  LU: panel heights
around the rows of a warp, a cluster's shares and the cluster's limit; permuted triangular
matrices with exact factors; ties, zero columns and NaN.
"""
import numpy as np
import pytest

from gpu_util import np64, pinned

pytestmark = pytest.mark.gpu


def _potrf(ooc, uplo, A):
    n = A.shape[0]
    a = pinned(n, n)
    a.numpy()[:] = A
    rc, info = ooc.ooc_dpotrf(uplo, n, a, n, 32 << 20, None, None)
    assert rc == 0, ooc.ooc_last_error()
    return np64(a), info


@pytest.mark.parametrize("uplo", "LU")
@pytest.mark.parametrize("n", [1, 2, 15, 16, 17, 31, 33, 63, 64, 65, 100])
def test_cholesky_of_integer_factors_is_exact(ooc, uplo, n):
    rng = np.random.default_rng(n)
    L = np.tril(rng.integers(-3, 4, (n, n)).astype(float), -1) + np.diag(rng.integers(1, 8, n).astype(float))
    got, info = _potrf(ooc, uplo, L @ L.T)
    assert info == 0
    assert np.array_equal(np.tril(got) if uplo == "L" else np.triu(got).T, L)


@pytest.mark.parametrize("n,bad", [(1, 0), (64, 0), (64, 1), (64, 15), (64, 16), (64, 63), (100, 70), (40, 39)])
@pytest.mark.parametrize("value", [0.0, -1.0, float("nan")])
def test_cholesky_first_failing_pivot(ooc, n, bad, value):
    d = np.full(n, 4.0)
    d[bad] = value
    assert _potrf(ooc, "L", np.diag(d))[1] == bad + 1


def test_cholesky_pivots_at_the_ends_of_the_range(ooc):
    d = 4.0 ** np.arange(-500, 500, 16)[:63]
    got, info = _potrf(ooc, "L", np.diag(d))
    assert info == 0 and np.array_equal(np.diag(got), np.sqrt(d))


def _getrf(ooc, A, budget=64 << 20):
    n = A.shape[0]
    a, piv = pinned(n, n), np.zeros(n, dtype=np.int64)
    a.numpy()[:] = A
    rc, info = ooc.ooc_dgetrf(n, a, n, piv, budget, None, None)
    assert rc == 0, ooc.ooc_last_error()
    return np64(a), piv, info


def _permute(A, piv):
    A = A.copy()
    for k, p in enumerate(piv):
        A[[k, p]] = A[[p, k]]
    return A


@pytest.mark.parametrize("n", [1, 2, 31, 32, 33, 63, 64, 65, 127, 129, 300, 513, 700])
def test_lu_of_dyadic_factors_is_exact(ooc, n):
    rng = np.random.default_rng(n)
    # |l| <= 1/2 and one entry of each column of a permuted P L U is its unique pivot
    L = np.tril(rng.integers(-2, 3, (n, n)) / 4.0, -1) * (np.abs(np.subtract.outer(range(n), range(n))) < 6) + np.eye(n)
    U = np.triu(rng.integers(-1, 2, (n, n)).astype(float), 1) * (np.abs(np.subtract.outer(range(n), range(n))) < 6) \
        + np.diag(np.where(rng.random(n) < 0.5, -4.0, 4.0))
    A = np.empty((n, n))
    order = rng.permutation(n)
    A[order] = L @ U
    got, piv, info = _getrf(ooc, A)
    assert info == 0 and np.array_equal(_permute(A, piv), L @ U)
    assert np.array_equal(np.tril(got, -1) + np.eye(n), L) and np.array_equal(np.triu(got), U)


def test_lu_ties_zero_columns_and_nan(ooc):
    n = 100
    A = np.ones((n, n))                       # ties: the first row; then every column is zero
    got, piv, info = _getrf(ooc, A)
    assert info == 2 and np.array_equal(piv, np.arange(n))
    assert np.array_equal(got, np.vstack([np.ones(n), np.hstack([np.ones((n - 1, 1)), np.zeros((n - 1, n - 1))])]))
    A = np.diag(np.arange(1.0, n + 1))
    A[40, 40] = np.nan                        # a NaN is never chosen while a number remains
    assert _getrf(ooc, A)[1][40] == 41

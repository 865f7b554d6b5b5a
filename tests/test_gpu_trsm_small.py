"""Substitution kernel of the triangular solves: its counts of lanes per vector, orders below its
block of 64, and divisors outside the range of its corrected quotient.

A triangular solve by substitution has the componentwise residual |alpha B - op(A) X| <=
2 (n + 4) 2^-53 |op(A)| |X| + 2^-53 |alpha B| in any order of its sums (n products, their
additions and one quotient per element); the check evaluates the residual in long double.
"""
import numpy as np
import pytest

from gpu_util import np64, pinned

pytestmark = pytest.mark.gpu


def _solve(ooc, side, uplo, A, B):
    n = A.shape[0]
    a, b = pinned(n, n), pinned(*B.shape)
    a.numpy()[:], b.numpy()[:] = A, B
    rc = ooc.ooc_dtrsm(side, uplo, "N", "N", *B.shape, 1.0, a, n, b, B.shape[1], 64 << 20, None, None)
    assert rc == 0, ooc.ooc_last_error()
    return np64(b)


def _residual_ok(side, T, X, B, n):
    L = np.longdouble
    R = (L(B) - L(T) @ L(X)) if side == "L" else (L(B) - L(X) @ L(T))
    S = np.abs(T) @ np.abs(X) if side == "L" else np.abs(X) @ np.abs(T)
    return (np.abs(R) <= 2 * (n + 4) * 2.0 ** -53 * S + 2.0 ** -53 * np.abs(B)).all()


@pytest.mark.parametrize("n", [1, 2, 33, 63, 64])
@pytest.mark.parametrize("nv", [1, 5, 640, 1300, 2500, 5000, 10000])   # 32 ... 2 lanes per vector
def test_lanes_per_vector(ooc, n, nv):
    rng = np.random.default_rng(n * 100 + nv)
    for side, uplo in (("L", "L"), ("R", "L"), ("L", "U")):
        T = np.tril(rng.standard_normal((n, n))) + 3 * np.eye(n)
        T = T if uplo == "L" else T.T.copy()
        A = np.where(T != 0, T, np.nan)   # the other triangle is not read
        B = rng.standard_normal((n, nv) if side == "L" else (nv, n))
        assert _residual_ok(side, T, _solve(ooc, side, uplo, A, B), B, n)


def test_divisors_at_the_ends_of_the_range(ooc):
    n, nv = 64, 40
    rng = np.random.default_rng(7)
    d = 2.0 ** np.linspace(-1040, 1000, n)          # subnormal to nearly the largest
    T = np.diag(d)
    X = rng.standard_normal((n, nv))
    B = np.where(np.arange(n)[:, None] % 5 == 0, 0.0, d[:, None] * X)
    got = _solve(ooc, "L", "L", T, B)
    with np.errstate(all="ignore"):
        assert np.array_equal(got, B / d[:, None])  # quotients rounded as by division, zeros exact


def test_zero_divisor_gives_what_division_gives(ooc):
    T = np.diag([2.0, 0.0, 4.0])
    B = np.array([[1.0, 2.0], [3.0, 0.0], [5.0, 6.0]])
    got = _solve(ooc, "L", "L", T, B)
    assert np.isinf(got[1, 0]) and np.isnan(got[1, 1]) and np.array_equal(got[0], [0.5, 1.0])

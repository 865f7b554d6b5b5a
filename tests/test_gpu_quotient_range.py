"""Corrected quotients of the solves and factorizations against division, dividends from subnormal
to large over divisors that leave the quotient well inside the range."""
import numpy as np
import pytest

from gpu_util import np64, pinned

pytestmark = pytest.mark.gpu


def _pairs(n, nv):
    """Dividends m 2^a, a from the smallest subnormals up, and divisors m 2^b, one per row."""
    rng = np.random.default_rng(11)
    b = np.linspace(-940, -100, n).round()
    d = np.ldexp(rng.uniform(1, 2, n), b.astype(int))
    a = rng.integers(-1070, -930, (n, nv))
    a[:, ::4] = rng.integers(-930, 900, (n, (nv + 3) // 4)).clip(None, 1000 + b[:, None].astype(int))
    s = np.ldexp(rng.uniform(1, 2, (n, nv)), a) * rng.choice([-1.0, 1.0], (n, nv))
    return s, d


@pytest.mark.parametrize("nv", [300, 5000])
def test_solve_with_tiny_right_hand_sides(ooc, nv):
    n = 64
    s, d = _pairs(n, nv)
    a, b = pinned(n, n), pinned(n, nv)
    a.numpy()[:], b.numpy()[:] = np.diag(d), s
    rc = ooc.ooc_dtrsm("L", "L", "N", "N", n, nv, 1.0, a, n, b, nv, 64 << 20, None, None)
    assert rc == 0, ooc.ooc_last_error()
    assert np.array_equal(np64(b), s / d[:, None])


def test_lu_multipliers_of_tiny_columns(ooc):
    """Rows below an arrow's diagonal: multiplier s / pivot, all else zero."""
    n = 200
    rng = np.random.default_rng(12)
    A = np.zeros((n, n))
    piv0 = np.ldexp(1.37, -950)
    A[0, 0] = piv0
    A[1:, 0] = np.ldexp(rng.uniform(1, 2, n - 1), rng.integers(-1070, -952, n - 1))
    A[np.arange(1, n), np.arange(1, n)] = 1.0
    a, piv = pinned(n, n), np.zeros(n, dtype=np.int64)
    a.numpy()[:] = A
    rc, info = ooc.ooc_dgetrf(n, a, n, piv, 64 << 20, None, None)
    assert rc == 0 and info == 0, ooc.ooc_last_error()
    assert np.array_equal(piv, np.arange(n))
    got = np64(a)
    assert np.array_equal(got[1:, 0], A[1:, 0] / piv0)
    assert np.array_equal(got[:, 1:], A[:, 1:]) and got[0, 0] == piv0

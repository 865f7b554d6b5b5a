"""LU panels taller than the small orders reach: rows walked twice by a cluster's CTAs (above 4096
rows), a cluster at its limit (16 CTAs of 736 rows) and the cooperative kernel above it, which
keeps its rows in shared memory.

Entries N(0,1).  The factors satisfy |P A - L U| <= 2 (n + 4) 2^-53 |L| |U| componentwise whatever
the order of their sums (n products, their additions and one quotient), checked on sampled rows,
and partial pivoting leaves no multiplier above one.
"""
import numpy as np
import pytest

import synth
from gpu_util import pinned_from

pytestmark = pytest.mark.gpu


# 4500: 282 rows a CTA.  12032: four 64-column sub-panels by the cooperative kernel, then 11,776
# rows, the most a cluster takes
@pytest.mark.parametrize("n", [4500, 12032])
def test_factors_of_a_random_matrix(ooc, n):
    a = pinned_from(99, 0, n, n, synth.NORMAL)
    F, A = a.numpy(), a.numpy().copy()
    piv = np.zeros(n, dtype=np.int64)
    rc, info = ooc.ooc_dgetrf(n, a, n, piv, 128 << 20, None, None)
    assert rc == 0, ooc.ooc_last_error()
    assert info == 0
    order = np.arange(n)
    for k, p in enumerate(piv):
        assert k <= p < n
        order[[k, p]] = order[[p, k]]
    rows = np.unique(np.concatenate([[0, 1, 63, 64, 255, 256, 257, n - 1],
                                     np.random.default_rng(n).integers(0, n, 24)]))
    L = F[rows]
    L[np.arange(n)[None, :] > rows[:, None]] = 0.0
    L[np.arange(len(rows)), rows] = 1.0
    for i in range(0, n, 1024):                       # multipliers, a strip at a time
        assert np.abs(np.tril(F[i:i + 1024], i - 1)).max() <= 1.0
    U = np.triu(F)
    got, size = L @ U, np.abs(L) @ np.abs(U)
    assert (np.abs(A[order[rows]] - got) <= 2 * (n + 4) * 2.0 ** -53 * size).all()

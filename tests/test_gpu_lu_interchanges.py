"""LU row interchanges outside the panel, by the device in host memory and by the host.

Permuted products of dyadic factors (unique pivots, exact arithmetic) over several panels and
padded leading dimensions: factors and pivots bit for bit, padding untouched, on both paths.
"""
import numpy as np
import pytest

from gpu_util import np64, pinned

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("by_host", [0, 1])
@pytest.mark.parametrize("n,ld,budget", [(65, 65, 1 << 20), (300, 300, 1 << 20), (1100, 1107, 4 << 20),
                                         (1500, 1500, 64 << 20)])
def test_interchanges_over_panels(ooc, monkeypatch, by_host, n, ld, budget):
    monkeypatch.setenv("OOC_LU_HOST_ROWS", str(by_host))
    rng = np.random.default_rng(n)
    near = np.abs(np.subtract.outer(range(n), range(n))) < 6
    L = np.tril(rng.integers(-2, 3, (n, n)) / 4.0, -1) * near + np.eye(n)
    U = np.triu(rng.integers(-1, 2, (n, n)).astype(float), 1) * near \
        + np.diag(np.where(rng.random(n) < 0.5, -4.0, 4.0))
    LU = L @ U
    a, piv = pinned(n, ld), np.zeros(n, dtype=np.int64)
    a.numpy()[:] = np.nan
    a.numpy()[rng.permutation(n), :n] = LU
    A = np64(a)[:, :n].copy()
    rc, info = ooc.ooc_dgetrf(n, a, ld, piv, budget, None, None)
    assert rc == 0, ooc.ooc_last_error()
    got = np64(a)
    for k, p in enumerate(piv):
        A[[k, p]] = A[[p, k]]
    assert info == 0 and np.array_equal(A, LU)
    assert np.array_equal(np.tril(got[:, :n], -1) + np.eye(n), L) and np.array_equal(np.triu(got[:, :n]), U)
    assert np.isnan(got[:, n:]).all()

"""In-HBM panel updates of Ozaki calls on both sides of the size that sends them to the FP64 tile kernel.

Integer triangles and solutions: each update is exact in either form (entries far inside 53 bits, and
the 9 digits hold 54), so the solution must come back bit for bit.
"""
import numpy as np
import pytest

from gpu_util import np64, pinned

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("side", "LR")
@pytest.mark.parametrize("n,nv", [(128, 1), (128, 4882), (128, 4883), (192, 2441), (192, 2442), (256, 1600)])
def test_trsm_with_small_and_large_updates(ooc, side, n, nv):
    rng = np.random.default_rng(n + nv)
    T = np.tril(rng.integers(-2, 3, (n, n)) * (rng.random((n, n)) < 0.2), -1).astype(float) + np.eye(n)
    X = rng.integers(-9, 10, (n, nv) if side == "L" else (nv, n)).astype(float)
    a, b = pinned(n, n), pinned(*X.shape)
    a.numpy()[:] = T
    b.numpy()[:] = T @ X if side == "L" else X @ T
    rc = ooc.ooc_dtrsm(side, "L", "N", "N", *X.shape, 1.0, a, n, b, X.shape[1], 256 << 20,
                       ooc.make_opts(form=2), None)
    assert rc == 0, ooc.ooc_last_error()
    assert np.array_equal(np64(b), X)

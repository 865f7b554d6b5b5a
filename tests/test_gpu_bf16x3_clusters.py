"""BF16x3 tile kernel: K lengths at its drains and launches whose tiles are shared by clusters.

Every element must lie inside the form's componentwise bound (tests/bounds.py) whatever the
number of CTAs that share a tile, and integer products, exact in every order, must be exact.
"""
import numpy as np
import pytest
import torch

import bounds
import oracle
import synth
from gpu_util import np64, pinned_from

pytestmark = pytest.mark.gpu


def _run(ooc, M, N, K, kind=synth.UNIFORM, param=0.0, alpha=1.0, beta=0.0, **kw):
    A, B, C = (pinned_from(95, s, r, c, kind, param, dtype=torch.float32)
               for s, r, c in ((0, M, K), (1, K, N), (2, M, N)))
    c0 = np64(C)
    rc = ooc.ooc_sgemm("N", "N", M, N, K, alpha, A, K, B, N, beta, C, N, 1 << 30, ooc.make_opts(**kw), None)
    assert rc == 0, ooc.ooc_last_error()
    return np64(A), np64(B), c0, np64(C)


# one K block, the leading accumulator's chunk (512) and the small ones' (2048), just beyond each;
# 4 tiles: clusters of 8 share them once K is long enough, some CTAs with no K block of their own
@pytest.mark.parametrize("K", [1, 64, 65, 512, 513, 1100, 2048, 2100, 5000])
def test_k_lengths(ooc, K):
    A, B, c0, got = _run(ooc, 130, 140, K, alpha=-2.5, beta=0.5)
    ref = oracle.gemm("N", "N", -2.5, A, B, 0.5, c0)
    assert bounds.worst_ratio(got, ref, bounds.bf16x3_bound(A, B, -2.5, 0.5, c0)) <= 1.0


@pytest.mark.parametrize("mb,nb", [(128, 128), (384, 512), (640, 768), (2048, 1536)])   # 1, 12, 30, 192 tiles
@pytest.mark.parametrize("K", [700, 3000])
def test_tiles_shared_by_clusters(ooc, mb, nb, K):
    A, B, _, got = _run(ooc, 2048, 1536, K, mb=mb, nb=nb)
    ref = oracle.gemm("N", "N", 1.0, A, B, 0.0, np.zeros_like(got))
    assert bounds.worst_ratio(got, ref, bounds.bf16x3_bound(A, B, 1.0, 0.0, None)) <= 1.0
    A, B, _, got = _run(ooc, 2048, 1536, K, kind=synth.INTEGER, param=16, mb=mb, nb=nb)
    assert np.array_equal(got, A @ B)

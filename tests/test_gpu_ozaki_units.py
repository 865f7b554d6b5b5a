"""Ozaki tile kernel: the cuts of a tile's work and the K lengths where its order changes.

Every element must lie inside the form's componentwise bound (tests/bounds.py, stated for
digits of 6 bits; the kernel's 8-bit digits carry at least as many).  Its sums are 64-bit
integers, so a block's result may not depend on how many CTAs share a tile: blockings whose
launches have one tile (eight CTAs each) and many tiles (one CTA each) give the same bits.
"""
import numpy as np
import pytest

import bounds
import oracle
import synth
from gpu_util import np64, pinned, pinned_from

pytestmark = pytest.mark.gpu


def _run(ooc, M, N, K, S, kind=synth.LOGSPREAD, param=0.0, alpha=1.0, beta=0.0, ta="N", tb="N", **kw):
    sa, sb = ((M, K) if ta == "N" else (K, M)), ((K, N) if tb == "N" else (N, K))
    A, B = pinned_from(91, 0, *sa, kind, param), pinned_from(91, 1, *sb, kind, param)
    C = pinned_from(91, 2, M, N, kind, param)
    c0 = np64(C)
    rc = ooc.ooc_dgemm(ta, tb, M, N, K, alpha, A, sa[1], B, sb[1], beta, C, N, 1 << 30,
                       ooc.make_opts(form=ooc.OOC_FORM_OZAKI, slices=S, **kw), None)
    assert rc == 0, ooc.ooc_last_error()
    return np64(A), np64(B), c0, np64(C)


# K blocks of 64: one, the longest K whose diagonals share accumulators (128, 256, 512), just
# beyond each, the exact-sum limit (1024) and beyond, an odd tail
@pytest.mark.parametrize("K", [1, 64, 65, 128, 129, 256, 257, 512, 513, 1024, 1025, 2100])
@pytest.mark.parametrize("S", [8, 9])
def test_k_lengths(ooc, K, S):
    A, B, c0, got = _run(ooc, 130, 140, K, S, alpha=-2.5, beta=0.5)
    ref = oracle.gemm("N", "N", -2.5, A, B, 0.5, c0)
    assert bounds.worst_ratio(got, ref, bounds.ozaki_bound(A, B, -2.5, 0.5, c0, S)) <= 1.0


@pytest.mark.parametrize("S", [2, 3, 4, 5, 6, 7, 10])
def test_slice_counts(ooc, S):
    A, B, c0, got = _run(ooc, 150, 70, 300, S, ta="T", tb="T")
    ref = oracle.gemm("T", "T", 1.0, A, B, 0.0, c0)
    assert bounds.worst_ratio(got, ref, bounds.ozaki_bound(A.T, B.T, 1.0, 0.0, None, S)) <= 1.0


@pytest.mark.parametrize("K", [70, 700, 3000])
def test_result_does_not_depend_on_the_cut(ooc, K):
    many = _run(ooc, 2048, 1536, K, 8, mb=2048, nb=1536)[3]   # 192 tiles: persistent CTAs
    for mb, nb in ((128, 128), (384, 512), (640, 768)):       # 1, 12 and 30 tiles: clusters of 8, 8 and 4
        assert np.array_equal(_run(ooc, 2048, 1536, K, 8, mb=mb, nb=nb)[3], many)


def test_extreme_values(ooc):
    """Digits at their limits (every element the same largest value: sums of 1024 products reach
    2^24), powers of two at both ends of the exponent range, and rows of zeros."""
    M, N, K = 128, 128, 1024
    A, B, C = pinned(M, K), pinned(K, N), pinned(M, N)
    A.fill_(1.0 - 2.0 ** -53)
    B.fill_(-(1.0 - 2.0 ** -53))
    A.numpy()[5] = 2.0 ** 500
    A.numpy()[6] = 2.0 ** -500
    A.numpy()[7] = 0.0
    B.numpy()[:, 9] = 2.0 ** -400
    B.numpy()[:, 10] = 0.0
    rc = ooc.ooc_dgemm("N", "N", M, N, K, 1.0, A, K, B, N, 0.0, C, N, 1 << 30,
                       ooc.make_opts(form=ooc.OOC_FORM_OZAKI), None)
    assert rc == 0, ooc.ooc_last_error()
    ref = oracle.gemm("N", "N", 1.0, np64(A), np64(B), 0.0, np64(C))
    bd = bounds.ozaki_bound(np64(A), np64(B), 1.0, 0.0, None, 8)
    assert bounds.worst_ratio(np64(C), ref, bd) <= 1.0
    assert (np64(C)[7] == 0).all() and (np64(C)[:, 10] == 0).all()

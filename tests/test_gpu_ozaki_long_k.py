"""Ozaki form with 9 and 10 slices over a long K: sums finer than the kernel's usual 64-bit unit.

From K 4097 and 65 on seven and eight planes of 8-bit digits sum their finest diagonals in a unit
2^16 times finer, six planes from K 262,145 on (csrc/ozaki_gemm.cu, the wide kernel).  The rms
error over a block of dot products, in units of 2^(e_i + f_j) (operands scaled below 1), is made of
    the dropped products      sqrt((P - 1) K) 5461 2^(2 - 8 (P + 2)): P - 1 of them per k on the first
                              diagonal left out, digits spread evenly over +-128 (mean square 5461);
                              a digit count P and weight 2^2 for the two scales 2^(e + 1), 2^(f + 1)
    the rounded operands      0.29 2^(1 - 8 P) (|x| + |y|), Euclidean norms
    FP64 roundings of C       at most six of 2^-53 rms |C|
and may be twice that.  The reference sums in long double (K 2^-64 of it and less).
"""
import numpy as np
import pytest

import bounds
import oracle
import synth
from gpu_util import np64, pinned_from

pytestmark = pytest.mark.gpu


def _run(ooc, M, N, K, S, kind, param=0.0, alpha=1.0, beta=0.0, budget=1 << 30, **kw):
    A, B = pinned_from(97, 0, M, K, kind, param), pinned_from(97, 1, K, N, kind, param)
    C = pinned_from(97, 2, M, N, synth.NORMAL)
    c0, st = np64(C), ooc.ooc_stats()
    rc = ooc.ooc_dgemm("N", "N", M, N, K, alpha, A, K, B, N, beta, C, N, budget,
                       ooc.make_opts(form=ooc.OOC_FORM_OZAKI, slices=S, **kw), st)
    assert rc == 0, ooc.ooc_last_error()
    return np64(A), np64(B), c0, np64(C), st


@pytest.mark.parametrize("kind,param", [(synth.NORMAL, 0.0), (synth.LOGSPREAD, 4.0)])
@pytest.mark.parametrize("S,K", [(9, 16384), (9, 65536), (10, 16384), (10, 65536)])
def test_slices_keep_their_accuracy(ooc, S, K, kind, param):
    A, B, _, got, st = _run(ooc, 24, 16, K, S, kind, param, kb=K)
    assert st.steps == 1
    x = A / np.exp2(bounds._exps(np.abs(A).max(axis=1)))[:, None]
    y = B / np.exp2(bounds._exps(np.abs(B).max(axis=0)))[None, :]
    scale = np.exp2(bounds._exps(np.abs(A).max(axis=1)))[:, None] * np.exp2(bounds._exps(np.abs(B).max(axis=0)))
    ref = A.astype(np.longdouble) @ B.astype(np.longdouble)
    rms = lambda v: float(np.sqrt(np.mean(np.square(v))))  # noqa: E731
    P = -(-3 * S // 4)
    dropped = np.sqrt((P - 1) * K) * 5461 * 2.0 ** (2 - 8 * (P + 2))
    operands = 0.29 * 2.0 ** (1 - 8 * P) * np.hypot(rms(np.linalg.norm(x, axis=1)), rms(np.linalg.norm(y, axis=0)))
    rounding = 6 * 2.0 ** -53 * rms((ref / scale).astype(np.float64))
    assert rms(((got - ref) / scale).astype(np.float64)) <= 2 * (dropped + operands + rounding)


# the last K of one unit and the first of two (64 for eight planes, 4096 for seven), a drain's
# K blocks, long and ragged K
@pytest.mark.parametrize("S,K", [(10, 64), (10, 65), (10, 257), (10, 1000), (10, 5000), (9, 4096), (9, 4097),
                                 (9, 8200), (9, 70000)])
def test_bounds(ooc, S, K):
    A, B, c0, got, st = _run(ooc, 130, 140, K, S, synth.LOGSPREAD, 4.0, alpha=-2.5, beta=0.5, kb=K)
    ref = oracle.gemm("N", "N", -2.5, A, B, 0.5, c0)
    assert bounds.worst_ratio(got, ref, bounds.ozaki_bound(A, B, -2.5, 0.5, c0, S)) <= 1.0


@pytest.mark.parametrize("S", [9, 10])
def test_result_does_not_depend_on_the_cut(ooc, S):
    many = _run(ooc, 2048, 1536, 5000, S, synth.LOGSPREAD, 4.0, mb=2048, nb=1536, budget=4 << 30)[3]
    for mb, nb in ((128, 128), (384, 512), (640, 768)):       # 1, 12 and 30 tiles: clusters
        assert np.array_equal(_run(ooc, 2048, 1536, 5000, S, synth.LOGSPREAD, 4.0, mb=mb, nb=nb, budget=4 << 30)[3],
                              many)


@pytest.mark.parametrize("uplo", "LU")
def test_triangular_update(ooc, uplo):
    """Masked stores of the wide kernel: the rest comes back as it was."""
    N, K = 300, 500
    A, C = pinned_from(98, 0, N, K, synth.NORMAL), pinned_from(98, 2, N, N, synth.NORMAL)
    keep = np.triu(np.ones((N, N), bool), 1) if uplo == "L" else np.tril(np.ones((N, N), bool), -1)
    C.numpy()[keep] = np.nan
    c0 = np64(C)
    rc = ooc.ooc_dsyrk(uplo, "N", N, K, 1.5, A, K, 0.5, C, N, 1 << 30,
                       ooc.make_opts(form=ooc.OOC_FORM_OZAKI, slices=10), None)
    assert rc == 0, ooc.ooc_last_error()
    a, got = np64(A), np64(C)
    ref = oracle.gemm("N", "T", 1.5, a, a, 0.5, np.nan_to_num(c0))
    bd = bounds.ozaki_bound(a, a.T, 1.5, 0.5, np.nan_to_num(c0), 10)
    assert bounds.worst_ratio(got[~keep], ref[~keep], bd[~keep]) <= 1.0
    assert np.array_equal(got[keep], c0[keep], equal_nan=True)


@pytest.mark.parametrize("S", [8, 9])
def test_six_planes_beyond_one_unit(ooc, S):
    K = (1 << 18) + 200
    A, B, c0, got, st = _run(ooc, 40, 30, K, S, synth.LOGSPREAD, 4.0, alpha=-2.5, beta=0.5, budget=4 << 30, kb=K)
    ref = oracle.gemm("N", "N", -2.5, A, B, 0.5, c0)
    assert bounds.worst_ratio(got, ref, bounds.ozaki_bound(A, B, -2.5, 0.5, c0, S)) <= 1.0


# one unit and two: sums beyond the largest FP64 number are infinite with the sum's sign, whatever
# the signs of its coarse and fine parts
@pytest.mark.parametrize("S,K", [(8, 200), (10, 200), (9, 5000), (8, (1 << 18) + 200)])
def test_overflow_is_infinite(ooc, S, K):
    M, N = 12, 10
    A, B = pinned_from(94, 0, M, K, synth.NORMAL), pinned_from(94, 1, K, N, synth.NORMAL)
    C = pinned_from(94, 2, M, N, synth.NORMAL)
    exact = A.numpy().astype(np.longdouble) @ B.numpy().astype(np.longdouble)
    assert np.abs(exact).min() > 1e-6
    A.mul_(2.0 ** 560)
    B.mul_(2.0 ** 560)
    rc = ooc.ooc_dgemm("N", "N", M, N, K, 1.0, A, K, B, N, 0.5, C, N, 4 << 30,
                       ooc.make_opts(form=ooc.OOC_FORM_OZAKI, slices=S, kb=K), None)
    assert rc == 0, ooc.ooc_last_error()
    assert np.array_equal(np64(C), np.where(exact > 0, np.inf, -np.inf))


def test_stretches(ooc):
    """K beyond 2^24: a second launch that adds into C (three rows of digit planes, 52 GB of them)."""
    K = (1 << 24) + 200
    A, B, c0, got, _ = _run(ooc, 3, 2, K, 8, synth.NORMAL, alpha=-2.5, beta=0.5, budget=80 << 30, kb=K)
    ref = oracle.gemm("N", "N", -2.5, A, B, 0.5, c0)
    assert bounds.worst_ratio(got, ref, bounds.ozaki_bound(A, B, -2.5, 0.5, c0, 8)) <= 1.0


@pytest.mark.parametrize("S", [9, 10])
def test_signs_and_ties_of_the_low_bits(ooc, S):
    """Sums whose leading part is small, zero or negative, and results half way between two FP64
    numbers: integers with few bits, exact in every digit, against exact integers rounded once."""
    M, N, K = 64, 48, 5000
    rng = np.random.default_rng(S)
    a = np.zeros((M, K))
    b = np.zeros((K, N))
    a[:, :8] = rng.integers(-2 ** 26, 2 ** 26, (M, 8))
    b[:8] = rng.integers(-2 ** 26, 2 ** 26, (8, N))
    a[:, 8], b[8] = 2.0 ** 27, 0.0                    # the rows' and columns' largest entries
    a[:, 9], b[9] = 0.0, 2.0 ** 27
    a[::3, 10], b[10] = 1.0, 1.0                      # odd sums above 2^53
    a[:5, :8] = 0.0                                   # 1 or 0 alone: fine diagonals only
    A, B, C = (pinned_from(93, s, *x, synth.NORMAL) for s, x in ((0, a.shape), (1, b.shape), (2, (M, N))))
    A.numpy()[:], B.numpy()[:] = a, b
    for alpha in (1.0, -1.0):
        rc = ooc.ooc_dgemm("N", "N", M, N, K, alpha, A, K, B, N, 0.0, C, N, 1 << 30,
                           ooc.make_opts(form=ooc.OOC_FORM_OZAKI, slices=S, kb=K), None)
        assert rc == 0, ooc.ooc_last_error()
        ia, ib = a[:, :11].astype(np.int64).astype(object), b[:11].astype(np.int64).astype(object)
        exact = ia.dot(ib)
        assert np.array_equal(np64(C), alpha * np.array([[float(x) for x in r] for r in exact]))

"""CPU pin of the Ozaki kernels' number format (csrc/ozaki_gemm.cu), in exact integers.

Operands rounded to 8 s - 1 fractional bits and cut into s = ceil(3 S / 4) balanced digits of 8
bits; the digit products with i + j <= s + 1 summed in one integer of unit 2^-frac, the sums of
the finest diagonals rounded to it.  The result must lie inside the componentwise bound stated
for S digits of 6 bits (tests/bounds.py) without its slack factor, on random and on worst-case
inputs, and every partial sum the tensor cores would hold must be exact in FP32.
"""
import math
from fractions import Fraction

import numpy as np
import pytest

import bounds


def digits(x, e, s):
    """Balanced digits of x 2^(8 s - 1 - e) rounded to nearest (ties away), most significant first."""
    f = abs(Fraction(x)) * Fraction(2) ** (8 * s - 1 - e)
    F = int(f + Fraction(1, 2)) * (-1 if x < 0 else 1)
    d = []
    for _ in range(s - 1):
        low = (F & 255) - 256 * ((F >> 7) & 1)
        d.append(low)
        F = (F - low) >> 8
    return [F] + d[::-1]


def emulate(a, b, S):
    """sum_k a_k b_k as the kernels form it (K <= 1024: each digit product one FP32 sum)."""
    s, K = math.ceil(3 * S / 4), len(a)
    e, f = (int(bounds._exps(np.array([max(abs(v))]))[0]) for v in (a, b))
    da, db = [digits(x, e, s) for x in a], [digits(x, f, s) for x in b]
    assert all(abs(d) <= 128 for x in da + db for d in x)
    frac = 64 - max(6, math.ceil(math.log2(64 * math.ceil(K / 64))))
    total = 0
    for m in range(2, s + 2):
        for i in range(1, m):
            if i > s or m - i > s:
                continue
            p = sum(x[i - 1] * y[m - i - 1] for x, y in zip(da, db))
            assert abs(p) <= 2 ** 24
            q = frac - 8 * m
            total += p << q if q >= 0 else round(Fraction(p, 2 ** -q))
            assert abs(total) < 2 ** 63
    return Fraction(total) * Fraction(2) ** (e + f + 2 - frac)


@pytest.mark.parametrize("S", range(2, 11))
@pytest.mark.parametrize("kind", ["normal", "spread", "largest", "same"])
def test_inside_the_bound_of_six_bit_digits(S, kind):
    rng = np.random.default_rng(S)
    K = 200
    a, b = rng.standard_normal(K), rng.standard_normal(K)
    if kind == "spread":
        a, b = (np.sign(x) * 10.0 ** rng.uniform(-4, 4, K) for x in (a, b))
    elif kind == "largest":
        a, b = np.full(1024, 1 - 2.0 ** -53), np.full(1024, -(1 - 2.0 ** -53))
    elif kind == "same":  # every digit rounds the same way, every dropped product has one sign
        a = b = np.full(K, 1 / 3)
    got = emulate(a, b, S)
    ref = sum(Fraction(x) * Fraction(y) for x, y in zip(a, b))
    bound = bounds.ozaki_bound(a[None, :], b[:, None], 1.0, 0.0, None, S)[0, 0] / bounds.SLACK
    assert abs(float(got - ref)) <= bound

"""FP64 tile kernel at the edges of its 16 x 16 tiles, 8 x 8 fragments and 16-long K steps.

Every element must be within the rounding of a K-term sum in either order: the oracle and the
kernel each add K products (2K + 4 roundings of 2^-53 of |alpha| |A||B| + |beta C| between them),
and the elements beyond C's columns must keep their values.
"""
import numpy as np
import pytest
import torch

import oracle
from gpu_util import np64

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("ta,tb", [("N", "N"), ("N", "T"), ("T", "N"), ("T", "T")])
@pytest.mark.parametrize("M,N,K", [(1, 1, 1), (7, 9, 3), (8, 16, 4), (15, 17, 15), (16, 8, 16), (17, 33, 17),
                                   (33, 15, 129), (250, 130, 31)])
def test_tile_and_k_edges(ooc, ta, tb, M, N, K):
    rng = np.random.default_rng(M * 1000 + N * 10 + K)
    even = lambda x: x + x % 2
    sa, sb = ((M, K) if ta == "N" else (K, M)), ((K, N) if tb == "N" else (N, K))
    # operands inside wider rows of NaN: nothing beyond a row's end may be used
    host = [np.full((r, even(c) + 2), np.nan) for r, c in (sa, sb, (M, N))]
    for h, (r, c) in zip(host, (sa, sb, (M, N))):
        h[:, :c] = rng.standard_normal((r, c))
    A, B, C = (torch.from_numpy(h).cuda() for h in host)
    torch.cuda.synchronize()
    rc = ooc.ooc_dgemm_device(ta, tb, M, N, K, 1.5, A, A.shape[1], B, B.shape[1], -0.5, C, C.shape[1])
    assert rc == 0, ooc.ooc_last_error()
    torch.cuda.synchronize()
    got = np64(C.cpu())
    a, b, c0 = host[0][:, :sa[1]], host[1][:, :sb[1]], host[2][:, :N]
    ref = oracle.gemm(ta, tb, 1.5, a.copy(), b.copy(), -0.5, c0.copy())
    opa, opb = (a if ta == "N" else a.T), (b if tb == "N" else b.T)
    bound = (2 * K + 4) * 2.0 ** -53 * (1.5 * (np.abs(opa) @ np.abs(opb)) + 0.5 * np.abs(c0))
    assert (np.abs(got[:, :N] - ref) <= bound).all()
    assert np.isnan(got[:, N:]).all()

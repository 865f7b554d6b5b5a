"""LU statistics: the interchanges that the device makes in host memory count as link traffic."""
import numpy as np
import pytest

import synth
from gpu_util import pinned_from

pytestmark = pytest.mark.gpu


def _bytes(ooc, monkeypatch, n, by_host):
    monkeypatch.setenv("OOC_LU_HOST_ROWS", str(by_host))
    a, piv, st = pinned_from(96, 0, n, n, synth.NORMAL), np.zeros(n, dtype=np.int64), ooc.ooc_stats()
    rc, info = ooc.ooc_dgetrf(n, a, n, piv, 64 << 20, None, st)
    assert rc == 0 and info == 0, ooc.ooc_last_error()
    return st.h2d_bytes, st.d2h_bytes, piv


def test_interchanges_are_counted(ooc, monkeypatch):
    n, t = 1500, 1024   # two panels, the first of 1024 columns
    host, dev = _bytes(ooc, monkeypatch, n, 1), _bytes(ooc, monkeypatch, n, 0)
    assert np.array_equal(host[2], dev[2])
    moved = 0
    for c0, tk in ((0, t), (t, n - t)):
        for k0 in range(c0, c0 + tk, 512):              # rows gathered at once
            k1 = min(k0 + 512, c0 + tk)
            rows = set(range(k0, k1)) | {int(p) for p in dev[2][k0:k1]}
            moved += 8 * len(rows) * (n - tk)           # the other columns
    assert dev[0] - host[0] == moved and dev[1] - host[1] == moved

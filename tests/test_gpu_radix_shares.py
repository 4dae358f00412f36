"""The build's radix sorts where their shares change: whole and partial tiles
and rows, the sizes around one tile per CTA, and the round-robin tiles of wide
digits (20-bit ids).  The arrays are compared with stable sorts by numpy:
equal, element by element."""
import numpy as np
import pytest

import paper_1910_00692_gb300 as wt

pytestmark = pytest.mark.gpu
TT = 5632  # records of a tile


def graph(n, m, seed):
    """m distinct pairs of n vertices, weights with many ties."""
    rng = np.random.default_rng(seed)
    key = np.empty(0, np.int64)
    while key.size < m:
        a, b = rng.integers(0, n, (2, m + m // 4 + 64))
        x = np.minimum(a, b) * n + np.maximum(a, b)
        key = np.unique(np.concatenate([key, x[a != b]]))
    key = rng.permutation(key)[:m]
    u, v = (key // n).astype(np.int32), (key % n).astype(np.int32)
    flip = rng.random(m) < 0.5
    u[flip], v[flip] = v[flip], u[flip]
    return u, v, rng.integers(1, 1500, m).astype(np.int32)


@pytest.mark.parametrize("n, m", [
    (40, 1), (700, 511), (700, 512), (700, 513), (3000, 16 * 1024 + 1),
    (5000, 152 * TT // 2 - 7), (5000, 152 * TT // 2), (5000, 152 * TT // 2 + 33),
    (600000, 152 * 8 * TT - 1), (600000, 152 * 8 * TT),  # just below the spread sizes (on 152 SMs), at them
    (1000000, 152 * 8 * TT + 3 * TT + 45),
])
def test_sorted_structures(n, m):
    u, v, w = graph(n, m, m)
    g = wt.build_csr(n, u, v, w)
    try:
        order = np.argsort(-w, kind="stable")
        assert np.array_equal(g.array("order_u"), u[order])
        assert np.array_equal(g.array("order_v"), v[order])
        assert np.array_equal(g.array("order_w"), w[order])
        row = np.stack([u[order], v[order]], 1).ravel()
        col = np.stack([v[order], u[order]], 1).ravel()
        at = np.argsort(row, kind="stable")
        assert np.array_equal(g.array("wcol"), col[at])
        assert np.array_equal(g.array("wwt"), np.repeat(w[order], 2)[at])
        assert np.array_equal(g.array("wrank"), (at // 2).astype(np.int32))
        assert np.array_equal(g.array("rowptr"), np.concatenate([[0], np.cumsum(np.bincount(row, minlength=n))]))
    finally:
        g.free()

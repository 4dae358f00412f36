"""The row sorts' key widths: the same graph with its ids spread over 2^20,
2^24, 2^27 and 2^30 vertices (32-bit keys with the entry's index, ids alone,
64-bit keys, class by class) gives the same oriented rows, ids scaled."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu

wt = pytest.importorskip("paper_1910_00692_gb300")


def _cliques(sizes, seed):
    u, v, base = [], [], 0
    for s in sizes:
        a, b = np.triu_indices(s + 1, 1)  # oriented degrees s, s - 1, ..., 0
        u.append(a + base)
        v.append(b + base)
        base += s + 1
    u, v = np.concatenate(u), np.concatenate(v)
    rng = np.random.default_rng(seed)
    perm = rng.permutation(u.size)
    flip = rng.random(u.size) < 0.5
    u, v = np.where(flip, v, u)[perm], np.where(flip, u, v)[perm]
    return base, u.astype(np.int64), v.astype(np.int64), rng.integers(1, 1000, u.size).astype(np.int32)


@pytest.mark.parametrize("bits", [20, 24, 27, 30])
def test_oriented_rows_at_every_key_width(bits):
    n0, u, v, w = _cliques([8, 16, 17, 32, 33, 64, 65, 128, 129, 256, 257, 512, 520], 11)
    _, ocol, owt, oeid = oracle.oriented_csr(n0, u.astype(np.int32), v.astype(np.int32), w)
    rank = np.empty(w.size, np.int64)
    rank[oracle.edge_order(w)] = np.arange(w.size)
    n = 1 << bits
    step = (n - 1) // (n0 - 1)
    # the largest id is all ones: next to the padding of a row
    ids = n - 1 - step * np.arange(n0, dtype=np.int64)[::-1]
    d = wt.build_csr(n, ids[u].astype(np.int32), ids[v].astype(np.int32), w)
    try:
        assert np.array_equal(d.array("ocol"), ids[ocol].astype(np.int32))
        assert np.array_equal(d.array("owt"), owt)
        assert np.array_equal(d.array("orank"), rank[oeid])
    finally:
        d.free()


@pytest.mark.parametrize("bits", [20, 27])
@pytest.mark.parametrize("size", [8, 64, 400])
def test_repeated_pair_at_every_key_width(bits, size):
    n0, u, v, w = _cliques([size], 3)
    ids = (1 << bits) - n0 + np.arange(n0)
    u = ids[np.append(u, v[5])].astype(np.int32)
    v2 = ids[np.append(v, u[5] - ids[0])].astype(np.int32)
    with pytest.raises(wt.WtriError) as ei:
        wt.build_csr(1 << bits, u, v2, np.append(w, 7).astype(np.int32))
    assert ei.value.code == -1 and "repeated" in str(ei.value)

"""Cliques on graphs of more edges than whose bitmap is walked (2^17): the
drawn edges go through a filter to a work list.  Books of pages around the
longest row that is filtered (and of both table sizes, and past them), and
random cliques, in a large random graph; few draws, many and every edge."""
import math

import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu

wt = pytest.importorskip("paper_1910_00692_gb300")


def _graph(m, seed):
    """m edges: sparse background, books (an edge and its common neighbours,
    some of them joined) and cliques of 5 to 9 vertices."""
    rng = np.random.default_rng(seed)
    n, parts = 40_000, []

    def add(a, b):
        parts.append(np.stack([np.asarray(a), np.asarray(b)], 1))

    at = 0
    for pages in (1, 2, 3, 61, 62, 63, 64, 65, 127, 128, 129, 253, 254, 255, 256, 257, 400, 700):
        page = np.arange(at + 2, at + 2 + pages)
        add([at], [at + 1])
        add(np.full(pages, at), page)
        add(np.full(pages, at + 1), page)
        a, b = np.triu_indices(min(pages, 40), 1)
        keep = rng.random(a.size) < 0.3
        add(page[a[keep]], page[b[keep]])
        at += pages + 2
    for size in range(5, 10):
        for _ in range(40):
            c = rng.choice(n, size, replace=False)
            a, b = np.triu_indices(size, 1)
            add(c[a], c[b])
    add(rng.integers(0, n, 2 * m), rng.integers(0, n, 2 * m))
    e = np.concatenate(parts)
    key = np.minimum(e[:, 0], e[:, 1]) * n + np.maximum(e[:, 0], e[:, 1])
    _, first = np.unique(key[e[:, 0] != e[:, 1]], return_index=True)
    key = key[e[:, 0] != e[:, 1]][np.sort(first)][:m]
    perm = rng.permutation(key.size)
    w = rng.integers(1, 200, key.size) * np.where(rng.random(key.size) < 0.02, 50, 1)
    return n, (key // n)[perm].astype(np.int32), (key % n)[perm].astype(np.int32), w.astype(np.int32)


@pytest.mark.parametrize("m", [(1 << 17) - 1, 1 << 17, (1 << 17) + 1, 200_003])
@pytest.mark.parametrize("q", [4, 5])
def test_cliques_of_large_graphs(m, q):
    n, u, v, w = _graph(m, m)
    assert u.size == m
    d = wt.build_csr(n, u, v, w)
    try:
        for p, ns in ((1.0, -1), (2.0, -1), (-math.inf, -1), (math.inf, -1), (1.0, 1), (1.0, 300), (2.0, 20_000),
                      (1.0, 400_000)):
            k = 500
            flags = None if ns < 0 else oracle.sampled_edge_flags(w, p, ns, 5)
            want = oracle.clique_topk(n, u, v, w, q, p, k, flags)
            ids, _, keys = wt.sample_cliques(d, q, p, k, ns, 5)
            ctx = f"m={m} q={q} p={p} draws={ns}"
            assert ids.shape[0] == want["count"], ctx
            assert np.array_equal(ids, want["ids"]) and np.array_equal(keys, want["key"]), ctx
    finally:
        d.free()

"""Cliques on edges whose common neighbourhoods lie at the edges of the
enumeration's table sizes (128 and 256 kept neighbours) and past them, dense
and sparse, and selections cut inside a long tie."""
import math

import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu

wt = pytest.importorskip("paper_1910_00692_gb300")


def _book(pages, q, wmax, seed):
    """Vertices 0 and 1 joined to each other and to `pages` more, with a few
    hundred random edges and one clique among those."""
    rng = np.random.default_rng(seed)
    n = pages + 2
    a, b = np.triu_indices(pages, 1)
    keep = rng.random(a.size) < min(1.0, 600.0 / max(a.size, 1))
    keep |= b < q + 3
    u = np.concatenate([[0], np.zeros(pages), np.ones(pages), a[keep] + 2]).astype(np.int32)
    v = np.concatenate([[1], np.arange(2, n), np.arange(2, n), b[keep] + 2]).astype(np.int32)
    perm = rng.permutation(u.size)
    w = rng.integers(1, wmax + 1, u.size).astype(np.int32)
    return n, u[perm], v[perm], w


@pytest.mark.parametrize("pages", [3, 127, 128, 129, 255, 256, 257, 400])
@pytest.mark.parametrize("q", [4, 5])
def test_clique_table_sizes(pages, q):
    n, u, v, w = _book(pages, q, 50, pages + q)
    d = wt.build_csr(n, u, v, w)
    try:
        for p, ns in ((1.0, -1), (2.0, 40), (1.0, 2000), (math.inf, -1), (-math.inf, -1)):
            k = 300
            flags = None if ns < 0 else oracle.sampled_edge_flags(w, p, ns, 3)
            want = oracle.clique_topk(n, u, v, w, q, p, k, flags)
            ids, wts, keys = wt.sample_cliques(d, q, p, k, ns, 3)
            ctx = f"pages={pages} q={q} p={p} draws={ns}"
            assert ids.shape[0] == want["count"], ctx
            assert np.array_equal(ids, want["ids"]), ctx
            assert np.array_equal(keys, want["key"]), ctx
    finally:
        d.free()


def test_clique_ties():
    """Equal weights: every clique ties, so the selection is by vertex ids."""
    n, u, v, w = _book(60, 5, 1, 7)
    d = wt.build_csr(n, u, v, w)
    try:
        for q in (4, 5):
            for k in (1, 17, 4000):
                want = oracle.clique_topk(n, u, v, w, q, 1.0, k)
                ids, _, _ = wt.sample_cliques(d, q, 1.0, k, -1, 0)
                assert ids.shape[0] == want["count"] and np.array_equal(ids, want["ids"]), (q, k)
    finally:
        d.free()

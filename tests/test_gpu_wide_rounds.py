"""Sweeps that visit most of a graph (fewer triangles than asked for, so no
threshold): rounds of more edges than there are items, with short live ranges
scanned by their warp, long ones left as items, and more long ones than items."""
import numpy as np
import pytest

import oracle
from wtri_testutil import GEN_TOL, PS, assert_topk_close, assert_topk_equal

pytestmark = pytest.mark.gpu

wt = pytest.importorskip("paper_1910_00692_gb300")
torch = pytest.importorskip("torch")


def _sparse(n, m, bipartite, planted, seed):
    """m edges at random (between two halves if bipartite) and `planted`
    triangles of fresh vertices; weights 1..50."""
    rng = np.random.default_rng(seed)
    half = n // 2
    a = rng.integers(0, half if bipartite else n, 2 * m)
    b = rng.integers(half if bipartite else 0, n, 2 * m)
    key = np.unique(np.minimum(a, b)[a != b] * n + np.maximum(a, b)[a != b])
    key = rng.permutation(key)[:m]
    t = n + 3 * np.arange(planted)
    u = np.concatenate([key // n, t, t + 1, t])
    v = np.concatenate([key % n, t + 1, t + 2, t + 2])
    at = rng.permutation(u.size)
    w = rng.integers(1, 51, u.size)
    return n + 3 * planted, u[at].astype(np.int32), v[at].astype(np.int32), w.astype(np.int32)


def _device(fn, d, p, k):
    dev = torch.device("cuda:0")
    t = torch.zeros((k, 3), dtype=torch.int32, device=dev)
    w = torch.zeros(k, dtype=torch.float64, device=dev)
    c = torch.zeros(1, dtype=torch.int32, device=dev)
    fn(d, p, k, t, w, c)
    n = int(c.item())
    assert n >= 0, n
    return t[:n].cpu().numpy(), w[:n].cpu().numpy()


# rows of about eight entries; of 150 (no threshold: most live ranges are long,
# far more of them than items); of 130, whose suffixes lie on both sides of the
# longest range that is not left as an item
@pytest.mark.parametrize("n,m,bipartite", [(250_000, 1_000_000, False), (8_000, 600_000, True), (5_200, 340_000, True)])
def test_sweep_of_the_whole_graph(n, m, bipartite):
    n, u, v, w = _sparse(n, m, bipartite, 500, seed=m)
    d = wt.build_csr(n, u, v, w)
    try:
        for p in PS:
            want = oracle.topk(n, u, v, w, p, 2000)
            assert want["count"] >= 500
            for first in (64, 200_000):
                d.set_tune(first, 8, 32)
                ctx = f"n={n} m={m} p={p} first={first}"
                for name, got in (("host", d.topk(p, 2000)), ("noalloc", _device(wt.topk_device_noalloc, d, p, 2000))):
                    assert_topk_equal(*got, want, p, f"{ctx} {name}")
                parts = [wt.topk_shard(d, p, 2000, s, 3) for s in range(3)]
                assert_topk_equal(*wt.merge_topk(parts, 2000)[:2], want, p, f"{ctx} shards")
            (got,) = wt.topk_batch([d], [p], [2000])
            assert_topk_equal(*got, want, p, f"batch p={p}")
            res = wt.topk_batch([d] * 330, [p] * 330, [2000] * 330) if m < 500_000 and p == 1.0 else []  # one per part
            for got in res:
                assert_topk_equal(*got, want, p, f"parts p={p}")
        for p in (-1.0, 3.0):
            want = oracle.topk(n, u, v, w, p, 2000)
            assert_topk_close(*d.topk(p, 2000), want["tri"], want["value"], f"p={p}", rel=GEN_TOL)
        # the k-th key exists but hardly moves: rounds stay wide under a threshold
        want = oracle.topk(n, u, v, w, 1.0, 450)
        assert_topk_equal(*d.topk(1.0, 450), want, 1.0, "k=450")
        # sampled: nearly every edge drawn
        for p in (0.0, 1.0):
            want = oracle.sample_topk(n, u, v, w, p, 2000, 4 * u.size, 5)
            assert want["sampled_edges"] > 0.5 * u.size
            assert_topk_equal(*d.sample_topk(p, 2000, 4 * u.size, 5), want, p, f"sampled p={p}")
    finally:
        d.free()


def _late(heavy, m, n, seed):
    """heavy triangle-free heavy edges, then a light random graph of m edges on n
    vertices: every triangle lies in the last edges of the edge order."""
    rng = np.random.default_rng(seed)
    key = np.unique(rng.integers(0, 200_000, 2 * heavy) * 400_000 + rng.integers(200_000, 400_000, 2 * heavy))
    key = rng.permutation(key)[:heavy]
    a, b = rng.integers(0, n, 2 * m), rng.integers(0, n, 2 * m)
    light = np.unique(np.minimum(a, b)[a != b] * n + np.maximum(a, b)[a != b])
    light = rng.permutation(light)[:m]
    u = np.concatenate([key // 400_000, 400_000 + light // n])
    v = np.concatenate([key % 400_000, 400_000 + light % n])
    w = np.concatenate([rng.integers(1000, 1100, key.size), rng.integers(1, 21, light.size)])
    return 400_000 + n, u.astype(np.int32), v.astype(np.int32), w.astype(np.int32)


@pytest.mark.parametrize("p", [0.0, 1.0, 2.0, np.inf])
def test_wide_round_that_fills_the_candidates(p):
    """1.3 million triangles in the edges of one wide round, more than the
    1,048,576 candidates of the fixed scratch; rounds of as many edges as items
    (46,592) hold them.  (p = -inf and the allocating device form take all these
    edges in one round whatever the items, and report WTRI_ENOMEM.)"""
    n, u, v, w = _late(600_000, 200_000, 2000, 3)
    d = wt.build_csr(n, u, v, w)
    try:
        for k in (16_384, 3000):
            want = oracle.topk(n, u, v, w, p, k)
            assert want["ntri"] > 1 << 20
            assert_topk_equal(*_device(wt.topk_device_noalloc, d, p, k), want, p, f"noalloc p={p} k={k}")
            assert_topk_equal(*d.topk(p, k), want, p, f"host p={p} k={k}")
            for got in wt.topk_batch([d] * 3, [p] * 3, [k] * 3):
                assert_topk_equal(*got, want, p, f"batch p={p} k={k}")
    finally:
        d.free()

"""How a batched call deals the SMs: equal queries that share them unevenly,
more queries than one launch has teams (k above what a part of a block ranks
needs one each), and both beside small ones; with the graph launch built anew
and updated."""
import numpy as np
import pytest

import oracle
import synth
from wtri_testutil import PS, assert_topk_equal

pytestmark = pytest.mark.gpu

wt = pytest.importorskip("paper_1910_00692_gb300")

SIZES = [(120, 500), (400, 3000), (1500, 12_000), (6000, 60_000)]


@pytest.fixture(scope="module")
def pool():
    gs = [synth.scaled_mid_graph(n, m, seed=70 + i) for i, (n, m) in enumerate(SIZES)]
    ds = [wt.build_csr(g.n, g.u, g.v, g.w) for g in gs]
    wants = {(i, p): oracle.topk(g.n, g.u, g.v, g.w, p, 4100) for i, g in enumerate(gs) for p in PS}
    yield ds, wants
    for d in ds:
        d.free()


def _check(pool, queries):
    ds, wants = pool
    for call in range(2):
        res = wt.topk_batch([ds[i] for i, _, _ in queries], [p for _, p, _ in queries], [k for _, _, k in queries])
        for (i, p, k), (tris, wts) in zip(queries, res):
            w = wants[i, p]
            part = {"tri": w["tri"][:k], "value": w["value"][:k], "count": min(k, w["count"])}
            assert_topk_equal(tris, wts, part, p, f"call={call} graph={i} p={p} k={k}")


# one k each; then k above 2,048, so that every query has a team: fewer than
# there are SMs, one too many for 64, two launches' worth and more
@pytest.mark.parametrize("count", [1, 2, 16, 64, 65, 153, 330])
@pytest.mark.parametrize("k", [500, 2100])
def test_equal_queries(pool, count, k):
    _check(pool, [(2, PS[count % 5], k)] * count)


def test_more_teams_than_a_launch_has_beside_parts(pool):
    rng = np.random.default_rng(8)
    queries = [(i % 4, PS[i % 5], 2100) for i in range(70)]
    queries += [(int(rng.integers(0, 4)), PS[int(rng.integers(0, 5))], int(rng.integers(1, 1001))) for _ in range(300)]
    queries = [queries[i] for i in rng.permutation(len(queries))]
    _check(pool, queries)
    _check(pool, queries[:200] + [(3, p, 4100) for p in PS])


@pytest.fixture(scope="module")
def ties():
    """Weights 1..3 only: most candidates tie, the vertex triple decides."""
    g = synth.scaled_mid_graph(8000, 90_000, seed=77)
    g.w = (1 + np.random.default_rng(6).integers(0, 3, g.m)).astype(np.int32)
    d = wt.build_csr(g.n, g.u, g.v, g.w)
    yield d, {p: oracle.topk(g.n, g.u, g.v, g.w, p, 65_536) for p in PS}
    d.free()


# On both sides of a sorted run (2,048), of two candidates per warp of the
# whole GPU (9,728), of 32 runs, and the largest k; alone, in a team of a few
# SMs, and on a part of one.
@pytest.mark.parametrize("p", PS)
def test_rankings_of_many(ties, p):
    d, wants = ties
    w = wants[p]

    def check(got, k, ctx):
        part = {"tri": w["tri"][:k], "value": w["value"][:k], "count": min(k, w["count"])}
        assert_topk_equal(*got, part, p, f"p={p} k={k} {ctx}")

    assert w["count"] == 65_536
    for k in (2049, 4096, 4097, 9727, 9728, 9729, 9730, 63_488, 65_535, 65_536):
        check(d.topk(p, k), k, "alone")
    for k in (2049, 4097, 20_000):
        for got in wt.topk_batch([d] * 20, [p] * 20, [k] * 20):
            check(got, k, "team")
    for k in (2049, 4096, 6145):
        for got in wt.topk_batch([d] * 310, [p] * 310, [k] * 310):
            check(got, k, "part")
    ks = [65_536] + [50] * 400
    for k, got in zip(ks, wt.topk_batch([d] * len(ks), [p] * len(ks), ks)):
        check(got, k, "beside small ones")


@pytest.mark.parametrize("p", PS)
def test_fewer_results_than_asked_for(p):
    """k above 2,048 on graphs with fewer triangles: ranked by counting on the
    whole GPU, by one block's sort on a few SMs and on a part."""
    for n, m, seed in ((60, 400, 1), (2000, 20_000, 2)):
        g = synth.scaled_mid_graph(n, m, seed=seed)
        d = wt.build_csr(g.n, g.u, g.v, g.w)
        try:
            want = oracle.topk(g.n, g.u, g.v, g.w, p, 3000)
            for k in (2049, 3000):
                w = {"tri": want["tri"][:k], "value": want["value"][:k], "count": min(k, want["count"])}
                assert_topk_equal(*d.topk(p, k), w, p, f"m={m} k={k}")
                for count in (1, 40, 320):
                    for got in wt.topk_batch([d] * count, [p] * count, [k] * count):
                        assert_topk_equal(*got, w, p, f"m={m} k={k} batch of {count}")
        finally:
            d.free()

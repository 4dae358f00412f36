"""The one-kernel sweep at the edges of its rules: results ranked by the sort
in shared memory and by counting, tie-heavy selects, batched queries answered
by one block and by a team of blocks (and several launches of teams), and the
fp32 pruning of the fp64 means over a wide range of p."""
import math

import numpy as np
import pytest

import oracle
import synth
from wtri_testutil import GEN_TOL, PS, assert_topk_close, assert_topk_equal

pytestmark = pytest.mark.gpu

wt = pytest.importorskip("paper_1910_00692_gb300")


@pytest.fixture(scope="module")
def ties():
    """Weights 1..3 only: thousands of triangles tie at the k-th key."""
    g = synth.scaled_mid_graph(20_000, 200_000, seed=3)
    g.w = (1 + np.random.default_rng(5).integers(0, 3, g.m)).astype(np.int32)
    d = wt.build_csr(g.n, g.u, g.v, g.w)
    yield g, d
    d.free()


@pytest.mark.parametrize("p", PS)
def test_rank_by_sort_and_by_counting(ties, p):
    """k at and around the largest sorted in shared memory (2,048)."""
    g, d = ties
    want = oracle.topk(g.n, g.u, g.v, g.w, p, 4097)
    for k in (1, 2, 2047, 2048, 2049, 4097):
        part = {"tri": want["tri"][:k], "value": want["value"][:k], "count": min(k, want["count"])}
        tris, wts = d.topk(p, k)
        assert_topk_equal(tris, wts, part, p, f"p={p} k={k}")
        (tris, wts), = wt.topk_batch([d], [p], [k])
        assert_topk_equal(tris, wts, part, p, f"batch p={p} k={k}")


def test_batch_blocks_and_teams():
    """One batch over graphs on both sides of the largest answered by one
    block (2^18 edges), with more large queries than one launch has teams."""
    sizes = [(300, 1000), (30_000, (1 << 18) - 1), (30_000, 1 << 18), (30_000, (1 << 18) + 1)]
    gs = [synth.scaled_mid_graph(n, m, seed=40 + i) for i, (n, m) in enumerate(sizes)]
    ds = [wt.build_csr(g.n, g.u, g.v, g.w) for g in gs]
    try:
        which, ps, ks = [], [], []
        for i in range(60):
            which.append(3 if i < 35 else i % 4)
            ps.append(PS[i % 5])
            ks.append((10, 500, 2100)[i % 3])
        res = wt.topk_batch([ds[i] for i in which], ps, ks)
        want = {}
        for i, p, k, (tris, wts) in zip(which, ps, ks, res):
            if (i, p) not in want:
                g = gs[i]
                want[i, p] = oracle.topk(g.n, g.u, g.v, g.w, p, 2100)
            w = want[i, p]
            part = {"tri": w["tri"][:k], "value": w["value"][:k], "count": min(k, w["count"])}
            assert_topk_equal(tris, wts, part, p, f"graph {i} p={p} k={k}")
    finally:
        for d in ds:
            d.free()


# on both sides of the smallest and largest |p| pruned in fp32 (0.05, 1000)
@pytest.mark.parametrize("p", [0.04, 0.06, -0.04, -0.06, -8.0, 12.0, 60.0, -60.0, 1001.0])
@pytest.mark.parametrize("real", [False, True])
def test_general_means_prune_nothing_due(p, real):
    g = synth.scaled_mid_graph(5_000, 50_000, seed=9)
    w = np.random.default_rng(4).lognormal(0.0, 2.0, g.m).astype(np.float32) if real else g.w
    d = wt.build_csr(g.n, g.u, g.v, w)
    try:
        for k in (5, 1000):
            want = oracle.topk_real(g.n, g.u, g.v, w, p, k) if real else oracle.topk(g.n, g.u, g.v, w, p, k)
            tris, wts = d.topk(p, k)
            # a mean of three powers carries the rounding of the power divided by p
            assert_topk_close(tris, wts, want["tri"], want["value"], f"p={p} k={k} real={real}", rel=GEN_TOL)
    finally:
        d.free()


def test_first_round_of_any_size():
    """Rounds that start with the filtered p = -inf scan, with a thread per
    edge, and past the item buffer, with no threshold yet."""
    g = synth.scaled_mid_graph(50_000, 400_000, seed=10)
    d = wt.build_csr(g.n, g.u, g.v, g.w)
    try:
        for first in (1, 5_000, 10_000, 300_000, 400_000):
            d.set_tune(first, 3, 32)
            for p in PS:
                want = oracle.topk(g.n, g.u, g.v, g.w, p, 300)
                tris, wts = d.topk(p, 300)
                assert_topk_equal(tris, wts, want, p, f"first={first} p={p}")
        assert math.isinf(PS[0])
    finally:
        d.free()

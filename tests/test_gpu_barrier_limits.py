"""Bounded waits of the sweep's grid barrier that run out at any moment: the
first wait's poll limit is lowered to a few polls, so that a block marks the
query as timed out while the others are already past the barrier.  Every
call either reports WTRI_ETIMEOUT or returns the exact answer, and the next
one with the default limit is exact."""
import math

import pytest

import oracle
import synth
from wtri_testutil import PS, assert_topk_equal

pytestmark = pytest.mark.gpu

wt = pytest.importorskip("paper_1910_00692_gb300")

ETIMEOUT = -4


@pytest.fixture(scope="module")
def scaled():
    g = synth.scaled_mid_graph(20_000, 200_000, seed=17)
    d = wt.build_csr(g.n, g.u, g.v, g.w)
    yield g, d, {p: oracle.topk(g.n, g.u, g.v, g.w, p, 2100) for p in PS}
    d.free()


def _part(want, k):
    return {"tri": want["tri"][:k], "value": want["value"][:k], "count": min(k, want["count"])}


# first rounds that leave items, that are scanned directly at p = -inf, and
# that hold the whole graph
@pytest.mark.parametrize("first", [64, 10_000, 200_000])
@pytest.mark.parametrize("p", PS)
def test_first_wait_of_a_few_polls(scaled, p, first):
    g, d, wants = scaled
    d.set_tune(first, 8, 32)
    try:
        for polls in (1, 2, 3, 5, 8, 15, 30, 60, 120, 1000):
            for k in (100, 2100):
                wt.debug_set_wait_limit(polls)
                try:
                    tris, wts = d.topk(p, k)
                except wt.WtriError as e:
                    assert e.code == ETIMEOUT
                else:
                    assert_topk_equal(tris, wts, _part(wants[p], k), p, f"polls={polls} p={p} k={k}")
        wt.debug_set_wait_limit(-1)
        tris, wts = d.topk(p, 2100)
        assert_topk_equal(tris, wts, _part(wants[p], 2100), p, f"after timeouts p={p}")
    finally:
        wt.debug_set_wait_limit(-1)
        d.set_tune(64, 8, 32)
    assert math.isinf(PS[0])

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


def _calls(d, torch):
    """Every call whose kernel has a grid barrier: name, the call."""
    dev = torch.device("cuda:0")

    def device(fn, k):
        t = torch.zeros((k, 3), dtype=torch.int32, device=dev)
        w = torch.zeros(k, dtype=torch.float64, device=dev)
        c = torch.full((1,), 7, dtype=torch.int32, device=dev)  # what an earlier call left
        fn(d, 1.0, k, t, w, c)
        torch.cuda.synchronize()
        if int(c.item()) < 0:
            raise wt.WtriError(int(c.item()), "device status")
        return t[:int(c.item())].cpu().numpy(), w[:int(c.item())].cpu().numpy()

    def served(p, k):
        s = wt.Server(8 << 30, 16)
        try:
            gid = s.add_graph(d)
            ticket = s.submit(gid, p, k)
            while True:
                r = s.poll(ticket, k)
                if r is not None:
                    return r[:2]
        finally:
            s.free()

    yield from ((f"topk p={p} k={k}", lambda p=p, k=k: d.topk(p, k)) for p in PS + [-1.0] for k in (100, 2100))
    yield "device", lambda: device(wt.topk_device, 100)
    yield "device, ranked by counting", lambda: device(wt.topk_device, 2100)
    yield "noalloc", lambda: device(wt.topk_device_noalloc, 100)
    yield "shard", lambda: wt.topk_shard(d, 1.0, 100, 1, 2)
    yield "sampled", lambda: d.sample_topk(1.0, 100, 50_000, 3)
    yield "wedges, ranked by counting", lambda: wt.wedge_topk(d, 1.0, 2100, 50_000, 3)
    yield "batch", lambda: wt.topk_batch([d, d, d], [1.0, -math.inf, 2.0], [100, 100, 2100])[0]
    yield "server", lambda: served(-math.inf, 100)
    yield "cliques", lambda: wt.sample_cliques(d, 4, 1.0, 100, 20_000, 3)


def test_waits_that_run_out_for_good(scaled):
    """No block waits for another: each leaves at its first barrier (later
    limit 0) or as soon as one is a few polls late.  The status says so,
    whatever the count held, and the same call is exact afterwards."""
    torch = pytest.importorskip("torch")
    _, d, _ = scaled
    for name, call in _calls(d, torch):
        wt.debug_set_wait_limits(-1, -1)
        before = call()
        try:
            wt.debug_set_wait_limits(0, 0)
            with pytest.raises(wt.WtriError) as ei:
                call()
            assert ei.value.code == ETIMEOUT, name
            for first, later in ((50, 0), (0, 50), (50, 50), (400, 400), (3000, 10)):
                wt.debug_set_wait_limits(first, later)
                try:
                    got = call()
                except wt.WtriError as e:
                    assert e.code == ETIMEOUT, name
                else:
                    assert all((a == b).all() for a, b in zip(got, before)), name
        finally:
            wt.debug_set_wait_limits(-1, -1)
        assert all((a == b).all() for a, b in zip(call(), before)), name


def test_status_is_written_once(scaled):
    """A count that the host reads while the query runs holds what it held, or
    the answer: no status of a query that has not given up shows."""
    torch = pytest.importorskip("torch")
    _, d, _ = scaled
    dev = torch.device("cuda:0")
    t = torch.zeros((100, 3), dtype=torch.int32, device=dev)
    w = torch.zeros(100, dtype=torch.float64, device=dev)
    c = torch.zeros(1, dtype=torch.int32, pin_memory=True)  # the device writes host memory
    seen = set()
    for i in range(200):
        c[0] = 7777
        wt.topk_device(d, PS[i % 5], 100, t, w, c)
        done = torch.cuda.Event()
        done.record()
        while not done.query():
            seen.add(int(c[0]))
        seen.add(int(c[0]))
    torch.cuda.synchronize()
    assert seen <= {7777, 100}, seen

"""Queries of small graphs, whose sweep takes some of the SMs: around the sizes
where their number changes, where it reaches its largest, and where the whole
GPU takes over; every mean, alone, sampled, in shards and without allocation."""
import numpy as np
import pytest

import oracle
import synth
from wtri_testutil import GEN_TOL, PS, assert_topk_close, assert_topk_equal

pytestmark = pytest.mark.gpu

wt = pytest.importorskip("paper_1910_00692_gb300")
torch = pytest.importorskip("torch")


def _noalloc(d, p, k):
    dev = torch.device("cuda:0")
    t = torch.zeros((k, 3), dtype=torch.int32, device=dev)
    w = torch.zeros(k, dtype=torch.float64, device=dev)
    c = torch.zeros(1, dtype=torch.int32, device=dev)
    wt.topk_device_noalloc(d, p, k, t, w, c)
    n = int(c.item())
    return t[:n].cpu().numpy(), w[:n].cpu().numpy()


@pytest.mark.parametrize("m", [1, 3, 15, 16, 17, 63, 64, 65, 129, 2432, 2433, 3007, 3008, 3073, 65_535, 65_536, 65_537])
def test_sizes_around_the_rule(m):
    n = max(3, int(np.ceil((1 + np.sqrt(1 + 8 * m)) / 2)), m // 12)
    if m < 200:  # dense: the first m pairs of a random order
        a, b = np.triu_indices(n, 1)
        at = np.random.default_rng(m).permutation(a.size)[:m]
        u, v = a[at].astype(np.int32), b[at].astype(np.int32)
        w = np.random.default_rng(m + 1).integers(1, 9, m).astype(np.int32)
    else:
        g = synth.scaled_mid_graph(n, m, seed=m)
        u, v, w = g.u, g.v, g.w
    d = wt.build_csr(n, u, v, w)
    try:
        for first in (64, 5):
            d.set_tune(first, 8, 32)
            for p in PS:
                for k in (1, 300, 2500):
                    want = oracle.topk(n, u, v, w, p, k)
                    assert_topk_equal(*d.topk(p, k), want, p, f"p={p} k={k} first={first}")
                assert_topk_equal(*_noalloc(d, p, 2500), want, p, f"noalloc p={p}")
                parts = [wt.topk_shard(d, p, 300, s, 2) for s in range(2)]
                want = oracle.topk(n, u, v, w, p, 300)
                assert_topk_equal(*wt.merge_topk(parts, 300)[:2], want, p, f"shards p={p}")
        for p in (-1.0, 3.0):
            want = oracle.topk(n, u, v, w, p, 300)
            assert_topk_close(*d.topk(p, 300), want["tri"], want["value"], f"p={p}", rel=GEN_TOL)
        want = oracle.sample_topk(n, u, v, w, 1.0, 300, 2 * m, 3)
        assert_topk_equal(*d.sample_topk(1.0, 300, 2 * m, 3), want, 1.0, "sampled")
    finally:
        d.free()

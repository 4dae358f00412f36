"""The general means' pruning weight on real weights at the ends of fp32's
range: subnormal weights, and weights that span more than sixty decades, where
fp32 quotients and powers underflow or overflow.  No triangle that is due may
be dropped (the oracle ranks every triangle by its fp64 mean)."""
import numpy as np
import pytest

import oracle
import synth
from wtri_testutil import GEN_TOL, assert_topk_close

pytestmark = pytest.mark.gpu

wt = pytest.importorskip("paper_1910_00692_gb300")


def _check(n, u, v, w, p, ks, ctx):
    d = wt.build_csr(n, u, v, w)
    try:
        for first in (8, 64):  # several rounds under a threshold
            d.set_tune(first, 2, 32)
            for k in ks:
                want = oracle.topk_real(n, u, v, w, p, k)
                tris, wts = d.topk(p, k)
                assert_topk_close(tris, wts, want["tri"], want["value"], f"{ctx} first={first} k={k}", rel=GEN_TOL)
    finally:
        d.free()


def _subnormal(units):
    return np.asarray(units, np.int32).view(np.float32)  # units of 2^-149


@pytest.mark.parametrize("p", [-1.0, -0.06, 0.0, 0.06, 0.5, 1.0, 2.0, 3.0])
def test_subnormal_weights(p):
    for seed in range(4):
        g = synth.random_small_graph(70, 0.5, 5, 900 + seed)
        rng = np.random.default_rng(seed)
        for top in (10, 1000, 1 << 22):
            w = _subnormal(rng.integers(1, top + 1, g.m))
            _check(g.n, g.u, g.v, w, p, (1, 7, 200), f"subnormal top={top} seed={seed} p={p}")


@pytest.mark.parametrize("p", [-8.0, -1.0, -0.12, -0.1, -0.06, -0.05, 0.0, 0.05, 0.06, 0.1, 0.12, 1.0, 3.0])
@pytest.mark.parametrize("decades", [30, 37])
def test_weights_of_many_decades(p, decades):
    for seed in range(4):
        g = synth.random_small_graph(70, 0.5, 5, 950 + seed)
        w = (10.0 ** np.random.default_rng(seed).uniform(-decades, decades, g.m)).astype(np.float32)
        _check(g.n, g.u, g.v, w, p, (1, 7, 200), f"decades={decades} seed={seed} p={p}")


# Two triangles, the better one second in the edge order and past the first
# round: the first sets the threshold that must not drop it.
@pytest.mark.parametrize("p,worse,better", [
    (2.0, (9, 7, 7), (9, 8, 6)),  # units of 2^-149
    (0.05, (1.07e21, 6.5e20, 7.6e-29), (1.07e21, 6.6e20, 7.7e-29)),
    (-0.1, (1.65e24, 3.1e15, 1.8e-32), (1.65e24, 3.2e15, 1.9e-32)),
])
def test_second_triangle_is_better(p, worse, better):
    fill = 80  # single edges of the heaviest weight between the triangles
    u = [0, 1, 0] + [6 + 2 * i for i in range(fill)] + [3, 4, 3]
    v = [1, 2, 2] + [7 + 2 * i for i in range(fill)] + [4, 5, 5]
    w = list(worse) + [worse[0]] * fill + list(better)
    w = _subnormal(w) if max(w) < 100 else np.asarray(w, np.float32)
    u, v = np.asarray(u, np.int32), np.asarray(v, np.int32)
    assert oracle.topk_real(6 + 2 * fill, u, v, w, p, 1)["tri"].tolist() == [[3, 4, 5]]
    _check(6 + 2 * fill, u, v, w, p, (1,), f"p={p}")

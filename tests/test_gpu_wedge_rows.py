"""The wedge sampler's row tables at the row lengths where their loops change
(64 entries and multiples of a warp's step), drawn from by the oracle's draws;
and rows whose sum does not fit 64 bits, short and long."""
import numpy as np
import pytest

import oracle
from wtri_testutil import assert_topk_equal

pytestmark = pytest.mark.gpu

wt = pytest.importorskip("paper_1910_00692_gb300")


def _rows(lengths, seed):
    """A hub per length: joined to that many of 600 vertices, which are joined
    at random among themselves."""
    rng = np.random.default_rng(seed)
    base, hubs = 600, len(lengths)
    u, v = [], []
    for i, n in enumerate(lengths):
        u += [base + i] * n
        v += rng.choice(base, n, replace=False).tolist()
    a, b = np.triu_indices(base, 1)
    keep = rng.random(a.size) < 0.02
    u, v = np.concatenate([u, a[keep]]), np.concatenate([v, b[keep]])
    at = rng.permutation(u.size)
    w = rng.integers(1, 100_000, u.size)
    return base + hubs, u[at].astype(np.int32), v[at].astype(np.int32), w.astype(np.int32)


@pytest.mark.parametrize("p", [0.0, 1.0, 2.0])
def test_rows_around_the_steps(p):
    n, u, v, w = _rows([1, 2, 31, 32, 33, 63, 64, 65, 66, 127, 128, 129, 130, 255, 256, 257, 260, 384, 385, 512, 513, 599], 3)
    d = wt.build_csr(n, u, v, w)
    try:
        got = wt.sample_wedges(d, p, 100_000, 11)
        want = oracle.wedge_samples(n, u, v, w, p, 100_000, 11)
        for a, b in zip(got, want):
            assert np.array_equal(np.asarray(a).reshape(-1), np.asarray(b).reshape(-1))
        top = oracle.wedge_topk(n, u, v, w, p, 500, 100_000, 11)
        assert_topk_equal(*wt.wedge_topk(d, p, 500, 100_000, 11), top, p, f"p={p}")
    finally:
        d.free()


@pytest.mark.parametrize("length", [4, 64, 65, 200])
def test_row_sums_above_64_bits_are_refused(length):
    n, u, v, w = _rows([length], 4)
    d = wt.build_csr(n, u, v, np.where(u >= 600, 2**31 - 1, w).astype(np.int32))
    try:
        if length == 4:  # 4 (2^31 - 1)^2 still fits
            assert len(wt.wedge_topk(d, 2.0, 10, 1000, 1)[1]) <= 10
        else:
            with pytest.raises(wt.WtriError):
                wt.wedge_topk(d, 2.0, 10, 1000, 1)
        assert len(wt.wedge_topk(d, 1.0, 10, 1000, 1)[1]) <= 10
    finally:
        d.free()

"""wtri_topk_device_noalloc from several host threads and streams at once: the
calls share one fixed array, so the library orders them on the device; every
answer is the allocating query's, and no barrier wait runs out."""
import threading

import numpy as np
import pytest

import synth
from wtri_testutil import PS

pytestmark = pytest.mark.gpu

wt = pytest.importorskip("paper_1910_00692_gb300")
torch = pytest.importorskip("torch")


def _outputs(k, dev):
    return (torch.zeros((k, 3), dtype=torch.int32, device=dev),
            torch.zeros(k, dtype=torch.float64, device=dev),
            torch.zeros(1, dtype=torch.int32, device=dev))


@pytest.mark.parametrize("threads", [1, 4])
def test_overlapping_calls(threads):
    """Each thread keeps two streams busy; nothing is waited for in between."""
    dev = torch.device("cuda:0")
    gs = [synth.tiny_graph(0), synth.scaled_mid_graph(20_000, 200_000, seed=23)]
    ds = [wt.build_csr(g.n, g.u, g.v, g.w) for g in gs]
    try:
        want = {}
        for i, d in enumerate(ds):
            for p in PS:
                for k in (100, 2100):
                    out = _outputs(k, dev)
                    wt.topk_device(d, p, k, *out)
                    torch.cuda.synchronize()
                    want[i, p, k] = [x.cpu().numpy() for x in out]
        jobs = sorted(want) * 3
        got, errors = {}, []

        def work(t):
            try:
                torch.cuda.set_device(0)
                streams = [torch.cuda.Stream(device=dev) for _ in range(2)]
                outs = []
                for j in range(t, len(jobs), threads):
                    i, p, k = jobs[j]
                    s = streams[len(outs) % 2]
                    with torch.cuda.stream(s):
                        out = _outputs(k, dev)
                    wt.topk_device_noalloc(ds[i], p, k, *out, stream=s)
                    outs.append((j, out))
                for s in streams:
                    s.synchronize()
                for j, out in outs:
                    got[j] = [x.cpu().numpy() for x in out]
            except Exception as e:  # reported by the test's thread
                errors.append(e)

        ts = [threading.Thread(target=work, args=(t,)) for t in range(threads)]
        for t in ts:
            t.start()
        for t in ts:
            t.join()
        assert not errors, errors
        assert sorted(got) == list(range(len(jobs)))
        for j, job in enumerate(jobs):
            assert all(np.array_equal(a, b) for a, b in zip(got[j], want[job])), job
    finally:
        for d in ds:
            d.free()


def test_captured_call():
    """A captured call takes no part in the ordering and can be replayed."""
    dev = torch.device("cuda:0")
    g = synth.tiny_graph(0)
    d = wt.build_csr(g.n, g.u, g.v, g.w)
    try:
        ref, out = _outputs(100, dev), _outputs(100, dev)
        wt.topk_device(d, 1.0, 100, *ref)
        wt.topk_device_noalloc(d, 1.0, 100, *out)
        torch.cuda.synchronize()
        graph = torch.cuda.CUDAGraph()
        s = torch.cuda.Stream(device=dev)
        with torch.cuda.graph(graph, stream=s):
            wt.topk_device_noalloc(d, 1.0, 100, *out, stream=s)
        for _ in range(3):
            for x in out:
                x.zero_()
            graph.replay()
            torch.cuda.synchronize()
            assert all(torch.equal(a, b) for a, b in zip(ref, out))
    finally:
        d.free()

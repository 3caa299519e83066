"""Restores and closes that the caller captures into a CUDA graph: the readers
return what the last replay or call found, with replays queued behind other work
and between calls that are not captured."""
import numpy as np
import pytest

import synth
from gpu_util import sp_rows, to_device

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def mods():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1807_01527_gb300 import asse, build
    build.build()
    return asse, torch


def lists(asse, torch, pool):
    """Report and candidates, the report from a device buffer too."""
    rep, cand = sp_rows(pool.report()), sp_rows(pool.candidates())
    out = torch.zeros(4096 * 4, dtype=torch.int32, device="cuda")
    torch.cuda.current_stream().synchronize()
    n = pool.report(out=out)
    assert sp_rows(out.cpu().numpy().view(asse.SP_DTYPE)[:n]) == rep
    return rep, cand


@pytest.mark.parametrize("counter", ["at", "hist"])
def test_captured_peek_between_closes(mods, counter):
    """scan + restore captured once and replayed in every slice, closes in
    between; the same calls uncaptured on a second pool are the reference."""
    asse, torch = mods
    w = synth.workload("tiny_b")
    s = torch.cuda.Stream()
    pool, ref = (asse.Pool(w.params, counter=counter, stream=s.cuda_stream) for _ in range(2))
    other = asse.Pool(w.params, stream=s.cuda_stream)
    big = torch.randint(-(1 << 31), 1 << 31, (8 << 20, 2), device="cuda", dtype=torch.int64).to(torch.int32)
    slices = [to_device(w.pairs(t)) for t in range(5)]
    torch.cuda.synchronize()
    for p in (pool, ref):
        p.ingest(slices[0])
        p.close_slice()
    assert lists(asse, torch, pool) == lists(asse, torch, ref)
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=s, capture_error_mode="thread_local"):
        pool.scan()
        pool.restore()
    seen = set()
    for x in slices[1:]:
        pool.ingest(x)
        for _ in range(4):
            other.ingest(big)          # the replay waits a while in the stream
        with torch.cuda.stream(s):
            graph.replay()
        got = lists(asse, torch, pool)
        ref.ingest(x)
        ref.scan()
        ref.restore()
        assert got == lists(asse, torch, ref)
        assert np.array_equal(pool.counts(), ref.counts())
        for p in (pool, ref):
            p.close_slice()
        closed = lists(asse, torch, pool)
        assert closed == lists(asse, torch, ref)
        seen.add(tuple(closed[0]))
    assert len(seen) > 1
    for p in (pool, ref, other):
        p.close()


@pytest.mark.parametrize("kps", [(4,), (4, 2, 1)])
def test_captured_close(mods, kps):
    """A close captured and replayed once, then closes that are not."""
    asse, torch = mods
    w = synth.workload("tiny_b")
    s = torch.cuda.Stream()
    pool, ref = (asse.Pool(w.params, stream=s.cuda_stream) for _ in range(2))
    slices = [to_device(w.pairs(t)) for t in range(4)]
    torch.cuda.synchronize()

    def close(p):
        p.close_slice_multi(kps) if len(kps) > 1 else p.close_slice(kps[0])

    graph = torch.cuda.CUDAGraph()
    for t, x in enumerate(slices):
        for p in (pool, ref):
            p.ingest(x)
        close(ref)
        if t == 1:
            torch.cuda.synchronize()
            with torch.cuda.graph(graph, stream=s, capture_error_mode="thread_local"):
                close(pool)
            with torch.cuda.stream(s):
                graph.replay()
        else:
            close(pool)
        for i in range(len(kps)):
            pool.select_window(i)
            ref.select_window(i)
            assert lists(asse, torch, pool) == lists(asse, torch, ref), (t, i)
    assert np.array_equal(pool.read_pool(), ref.read_pool())
    assert pool.info()["slice"] == ref.info()["slice"]
    pool.close()
    ref.close()

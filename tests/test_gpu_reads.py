"""Lists read into device memory are there when the call returns, whatever
stream reads them next and whatever is queued behind the close."""
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


@pytest.mark.parametrize("change_stream", [False, True])
def test_device_lists_are_complete_on_return(mods, change_stream):
    """The next slice's ingests (several ms of them) are queued after the close;
    the lists then go into device buffers and are read on another stream at
    once.  With change_stream the pool has moved to that stream in between."""
    asse, torch = mods
    w = synth.workload("tiny_b")
    one, two = torch.cuda.Stream(), torch.cuda.Stream()
    pool = asse.Pool(w.params, stream=one.cuda_stream)
    big = torch.randint(-(1 << 31), 1 << 31, (8 << 20, 2), device="cuda", dtype=torch.int64).to(torch.int32)
    slices = [to_device(w.pairs(t)) for t in range(6)]
    torch.cuda.synchronize()
    plain = asse.Pool(w.params, stream=one.cuda_stream)   # the same slices, read on the host
    for t, x in enumerate(slices):
        plain.ingest(x)
        plain.close_slice()
    want = {"report": sp_rows(plain.report()), "candidates": sp_rows(plain.candidates())}
    assert len(want["report"]) > 0
    for t, x in enumerate(slices):
        pool.ingest(x)
        pool.close_slice()
    for name in ("report", "candidates"):
        if change_stream:
            one.synchronize()
            pool.set_stream(two.cuda_stream)
        for _ in range(8):
            pool.ingest(big)
        out = torch.full((4096 * 4,), -1, dtype=torch.int32, device="cuda")
        torch.cuda.current_stream().synchronize()
        n = getattr(pool, name)(out=out)
        with torch.cuda.stream(two):
            got = out.cpu().numpy()
        assert sp_rows(got.view(asse.SP_DTYPE)[:n]) == want[name]
        assert (got[4 * n:] == -1).all()
    torch.cuda.synchronize()
    pool.close()
    plain.close()

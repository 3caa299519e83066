"""Host input at the sizes where its chunks change (a last chunk in two
parts, the two staging buffers in turn across calls), against the same pairs ingested
from device memory.  Integer state, compared exactly."""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu

MI = 1 << 20


@pytest.fixture(scope="module")
def mods():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1807_01527_gb300 import asse, build
    build.build()
    return asse, torch


@pytest.mark.parametrize("max_batch,pinned,sizes", [
    (0, True, (2 * MI - 1, 2 * MI, 2 * MI + 1, 1)),         # two parts of one chunk, even and odd, a lone pair
    (0, True, (5 * MI // 4, 5 * MI // 4 + 1, MI + 1)),      # one part, two parts, one part
    (0, True, (4 * MI, 4 * MI + 1, 6 * MI + 3, 9 * MI + 5)),  # one, two and three chunks, the last one short, split or not
    (3 * MI - 1, True, (3 * MI, 6 * MI + 1, 5 * MI + 7)),   # a buffer of an odd size; halves, whole buffers
    (65_001, True, (5 * MI // 4 + 3, 131_072, 65_003)),     # a buffer smaller than the parts and their alignment
    (0, False, (2 * MI + 1, 5 * MI + 3)),                    # pageable memory
    (1, True, (1, 2, 7))])
def test_host_chunks_equal_device_input(mods, max_batch, pinned, sizes):
    """The calls follow one another without a wait, and each batch is
    overwritten as soon as its call returns."""
    asse, torch = mods
    w = synth.workload("tiny_b")
    host, dev = asse.Pool(w.params, max_batch=max_batch), asse.Pool(w.params)
    gen = torch.Generator(device="cuda").manual_seed(sum(sizes))
    batches = []
    for n in sizes:
        x = torch.randint(-(1 << 31), 1 << 31, (n, 2), generator=gen, device="cuda", dtype=torch.int64).to(torch.int32)
        x[:, 0] %= 4096      # few hosts, so that not every field of the pool is set
        x[:, 0] += 1         # (the address 0 in none of them)
        x[:, 1] %= 48
        batches.append(x)
    for t in range(2):
        bufs = [x.cpu().pin_memory() if pinned else x.cpu() for x in batches]
        for b in bufs:
            host.ingest(b)
            b.zero_()
        for x in batches:
            dev.ingest(x)
        assert np.array_equal(host.read_pool(), dev.read_pool()), "slice %d" % t
        host.close_slice()
        dev.close_slice()
        assert np.array_equal(host.counts(), dev.counts())
    assert (host.counts() > 0).any()
    host.close()
    dev.close()

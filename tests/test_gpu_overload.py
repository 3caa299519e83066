"""Slices of more pairs than the pool has ATs, where the ingest stops using a key
table that it could do without: batches on both sides of that line, against the
oracle.  Integer state, compared exactly."""
import numpy as np
import pytest

import synth
from gpu_util import state, to_device

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def mods():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import oracle
    from paper_1807_01527_gb300 import asse, build
    build.build()
    oracle.build()
    return asse, oracle, torch


@pytest.mark.parametrize("counter,k,g,per_at", [("at", 4, 33, 2), ("ace", 1, 40, 2), ("at", 10, 65, 2), ("at", 40, 80, 4),
                                                ("at", 100, 200, 4), ("hist", 4, 33, 2)])
def test_batches_across_the_line(mods, counter, k, g, per_at):
    """Two batches that end at the line, one pair past it, batches beyond, from
    the device and from the host, and a next slice that starts below it again;
    keys of one batch come again in the others."""
    asse, oracle, torch = mods
    p = dict(k=k, theta=g, g=g, r=4, c=8, u=0, s=8, **synth.method_keys(k + g))
    pool = asse.Pool(p, counter=counter)
    orc = oracle.Oracle.from_params(p, mode={"ace": 1}.get(counter, 0))
    line = per_at * g * 256
    rng = np.random.default_rng(g)
    for t in range(2):
        x = rng.integers(0, 1 << 32, (line + 5001, 2), dtype=np.uint64).astype(np.uint32)
        x[:, 0] %= 97                         # of few hosts, so that fields stay unset
        cuts = [0, line // 3, line, line + 1, line + 5001]
        batches = [x[a:b] for a, b in zip(cuts, cuts[1:])] + [x[: 4001]]
        for i, b in enumerate(batches):
            b = np.ascontiguousarray(b)
            pool.ingest(b if i == 4 else to_device(b))
            orc.ingest(b)
        np.testing.assert_array_equal(state(pool), orc.at(), err_msg="slice %d" % t)
        assert ((state(pool) == (2 * k if counter != "ace" else 0)).any())
        pool.scan()
        pool.advance()
        orc.advance()
        np.testing.assert_array_equal(state(pool), orc.at(), err_msg="after slice %d" % t)
    pool.close()


@pytest.mark.parametrize("counter,k,g,elog,ats_per_pair", [("at", 60, 288, 17, 5), ("at", 10, 512, 17, 10),
                                                           ("ace", 10, 512, 18, 10)])
def test_large_pool_across_its_line(mods, counter, k, g, elog, ats_per_pair):
    """A pool larger than the L2 cache, whose claimed keys are set blind up to a
    line and read first past it, equals one without a key table; the keys of one
    batch come again in the others."""
    asse, oracle, torch = mods
    c, u, s = synth.column_split(elog, 4)
    p = dict(k=k, theta=g, g=g, r=4, c=c, u=u, s=s, **synth.method_keys(k + g))
    pools = [asse.Pool(p, counter=counter, key_table=kt) for kt in ("auto", "off")]
    l2 = torch.cuda.get_device_properties(0).L2_cache_size
    assert 4 * pools[0].info()["pool_words"] > l2
    line = (g << elog) // ats_per_pair
    gen = torch.Generator(device="cuda").manual_seed(k)
    for t in range(2):
        x = torch.randint(-(1 << 31), 1 << 31, (line + 300_001, 2), generator=gen, device="cuda",
                          dtype=torch.int64).to(torch.int32)
        x[:, 0] %= 5003
        x[:, 1] %= 2003
        batches = [x[: line // 2], x[line // 2: line], x[line: line + 1], x[line + 1:], x[: 100_001]]
        for b in batches:
            b = b.clone()               # from a 16-byte boundary
            for pool in pools:
                pool.ingest(b)
            torch.cuda.synchronize()
        a, b = (pool.read_pool() for pool in pools)
        np.testing.assert_array_equal(a, b, err_msg="slice %d" % t)
        for pool in pools:
            pool.close_slice()
        np.testing.assert_array_equal(pools[0].counts(), pools[1].counts())
        assert (pools[0].counts() > 0).any()
    for pool in pools:
        pool.close()

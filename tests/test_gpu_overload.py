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

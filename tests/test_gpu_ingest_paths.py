"""The ways an ingest sets fields (with and without a key table, and with
slice counts) at every packed field width, against the oracle: blind byte
stores and clear-and-set atomics must end at the same counters as a read
followed by a change.  Integer state, compared exactly."""
import numpy as np
import pytest

import synth
from gpu_util import check_close, mixed_pairs, state, to_device

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


@pytest.mark.parametrize("key_table", ["auto", "on", "off"])
@pytest.mark.parametrize("counter,k,g", [
    ("ace", 1, 96), ("at", 1, 130), ("at", 3, 97), ("at", 7, 200), ("at", 15, 333), ("at", 31, 301),
    ("at", 60, 400), ("at", 100, 801), ("ace", 100, 500), ("hist", 10, 257), ("hist", 40, 300), ("hist", 100, 500),
    ("aligned", 5, 4096)])
def test_field_sets_at_every_width(mods, counter, k, g, key_table):
    """Widths 1 to 6 and 8 (with and without the byte's guard bit), r = 4 and
    another r, the largest g, odd batch sizes, repeats within and across
    batches, the address 0, and slices of one pair."""
    asse, oracle, torch = mods
    r = 3 if k in (7, 60) else 4
    p = dict(k=k, theta=g, g=g, r=r, c=11, u=1, s=10, **synth.method_keys(k + g))
    pool = asse.Pool(p, counter=counter, key_table=key_table, restore_cap=1 << 14)
    orc = oracle.Oracle.from_params(p, mode={"ace": 1, "aligned": 2}.get(counter, 0))
    for t in range(3):
        x = mixed_pairs(k + g, t, 9001 + 2 * t, [g // 2, g, 3 * g])
        x[::37, 0] = 0
        for batch in (x, x[:1], x[1::2], x[::-1][:4097]):
            batch = np.ascontiguousarray(batch)
            pool.ingest(to_device(batch))
            orc.ingest(batch)
        np.testing.assert_array_equal(state(pool), orc.at(), err_msg="after ingest, slice %d" % t)
        check_close(pool, orc, k)
        orc.advance()
        np.testing.assert_array_equal(state(pool), orc.at(), err_msg="after refresh, slice %d" % t)
    pool.close()

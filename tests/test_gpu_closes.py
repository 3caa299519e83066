"""Closes in a row with nothing between them, fused and stepwise, against the
oracle: each kernel of a close reads the slice state that the close before wrote,
started while that one was still ending."""
import numpy as np
import pytest

import synth
from gpu_util import compare_lists, mixed_pairs, state, to_device

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
    return asse, oracle


@pytest.mark.parametrize("counter,k,g", [("at", 4, 128), ("hist", 4, 128), ("ace", 5, 200), ("aligned", 3, 96),
                                         ("at", 60, 400), ("hist", 60, 400)])
def test_closes_in_a_row(mods, counter, k, g):
    asse, oracle = mods
    p = dict(k=k, theta=g // 4, g=g, r=4, c=9, u=2, s=7, **synth.method_keys(k + g))
    fused, steps, multi = (asse.Pool(p, counter=counter, restore_cap=1 << 14) for _ in range(3))
    orc = oracle.Oracle.from_params(p, mode={"ace": 1, "aligned": 2}.get(counter, 0))
    t = 0
    for run in (1, 2, 5, k, 2 * k + 1):   # closes after each batch
        x = mixed_pairs(k, t, 3001, [g // 4, g // 2, g])
        for pool in (fused, steps, multi):
            pool.ingest(to_device(x))
        orc.ingest(x)
        for i in range(run):
            fused.close_slice()
            multi.close_slice_multi([k, 1])
            steps.scan()
            steps.restore()
            if i + 1 < run:
                steps.advance()
                orc.advance()
        res = orc.close_report(k, cap=1 << 14)
        for pool in (fused, multi, steps):
            np.testing.assert_array_equal(pool.counts(), res["counts"])
            np.testing.assert_array_equal(pool.loads(), res["aat"])
            compare_lists(pool.candidates(), res["candidates"], orc.theta, "after %d closes" % run)
        np.testing.assert_array_equal(state(steps), orc.at())
        steps.advance()
        orc.advance()
        for pool in (fused, multi, steps):
            np.testing.assert_array_equal(state(pool), orc.at(), err_msg="after %d closes" % run)
        t += run
    for pool in (fused, steps, multi):
        pool.close()

"""Synthetic training states of ATVs larger than a pool's: rows of every AT up to
the largest g, and the sizes that are refused."""
import ctypes
import os

import numpy as np
import pytest

import synth
from paper_1807_01527_gb300 import asse


def _cfg(k, g):
    keys = synth.method_keys(2)
    return dict(k=k, g=g, r=4, n_max_log2=16, bg_max=0.05, seed=3, bh_a=keys["bh_a"], bh_b=keys["bh_b"])


@pytest.mark.skipif(not os.path.exists(asse.LIB_PATH), reason="libasse.so is not built")
@pytest.mark.parametrize("k,g", [(32, 3713), (64, 4096)])
def test_sizes_beyond_the_limit_are_invalid(k, g):
    """Refused by rule, before any CUDA call: the status names the argument."""
    c = _cfg(k, g)
    cfg = asse.SynthCfg(c["k"], c["g"], c["r"], c["n_max_log2"], c["bg_max"], 0, c["seed"], c["bh_a"], c["bh_b"])
    some = ctypes.c_void_p(16)    # no buffer is reached
    call = asse.lib().asse_synth_states
    assert call(ctypes.byref(cfg), 0, 1, some, some, some, None) == asse.EINVAL
    assert call(ctypes.byref(cfg), 0, 0, some, some, some, None) == asse.OK


@pytest.mark.gpu
@pytest.mark.parametrize("k,g", [(10, 3073), (10, 4096), (40, 2049), (64, 3712)])
def test_rows_of_every_at(k, g):
    """513 words and more: counts, ages and Eq. 2 are those of the state's draws."""
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1807_01527_gb300 import build
    build.build()
    c, n = _cfg(k, g), 12
    x, ln, lc = (v.float().cpu().numpy() for v in asse.synth_states(c, 77, n))
    inv = np.float32(1) / np.float32(g)
    for si in range(n):
        d = synth.training_state_draws(3, 77 + si, k, g, 16, 0.05)
        last = np.full(g, -1)
        for s in range(k):
            with np.errstate(over="ignore"):
                h = d["bips"][s].astype(np.uint64) * np.uint64(c["bh_a"]) + np.uint64(c["bh_b"])
            last[((h >> np.uint64(32)) * np.uint64(g) >> np.uint64(32)).astype(np.int64)] = s
            last[d["bg"][s]] = s
        ages = np.bincount(k - 1 - last[last >= 0], minlength=64)[:64]
        want = torch.from_numpy(np.concatenate([[(last >= 0).sum()], ages]).astype(np.float32) * inv)
        np.testing.assert_array_equal(x[si, :65], want.to(torch.bfloat16).float().numpy(), err_msg="state %d" % si)
        assert ln[si] == np.float32(np.log(d["card"]))
        eq2 = -g * np.log((g - min(float((last >= 0).sum()), g - 0.5)) / g)
        assert abs(lc[si] - eq2) <= 1e-6 * eq2 + 1e-6

"""asse_estimate (NAT and Eq. 4 of given hosts) at the sizes where a warp's
share of the hosts, a host's share of the lanes or the range tables change,
against the oracle.  NAT is an integer and the estimate FP64 stored in FP32, so
both are compared as the parity tests do."""
import numpy as np
import pytest

import synth
from gpu_util import EST_ATOL, EST_RTOL, mixed_pairs, to_device

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


@pytest.mark.parametrize("counter,k,g,r,c,u,s", [
    ("ace", 1, 2, 4, 11, 1, 10), ("at", 1, 33, 3, 11, 1, 10), ("at", 10, 512, 4, 9, 2, 7), ("hist", 31, 301, 5, 9, 2, 6),
    ("at", 60, 1024, 4, 9, 4, 7), ("ace", 100, 500, 8, 9, 0, 4), ("at", 100, 801, 2, 16, 0, 16),
    ("aligned", 5, 2560, 4, 9, 2, 7)])
def test_estimates_of_hosts(mods, counter, k, g, r, c, u, s):
    """1 to 40,001 hosts (4 to 32 a warp), those of the traffic, unseen ones and
    the address 0, for the full window and a shorter one."""
    asse, oracle, torch = mods
    p = dict(k=k, theta=g, g=g, r=r, c=c, u=u, s=s, **synth.method_keys(k + g))
    pool = asse.Pool(p, counter=counter, restore_cap=1 << 14)
    orc = oracle.Oracle.from_params(p, mode={"ace": 1, "aligned": 2}.get(counter, 0))
    for t in range(3):
        x = mixed_pairs(k + g, t, 4001, [max(1, g // 4), max(1, g // 2), 2 * g])
        pool.ingest(to_device(x))
        orc.ingest(x)
        if t < 2:
            pool.advance()
            orc.advance()
    hosts = np.concatenate([np.unique(x[:, 0])[:60], [0, 1, 0xFFFFFFFF]]).astype(np.uint32)
    for kp in {k, max(1, k // 2)}:
        pool.scan(kp)
        aat = orc.aat(orc.counts(kp))
        want = [orc.estimate(aat, int(a), kp) for a in hosts]
        for n in (1, 3, 5, 33, 1025, 40001):
            pick = np.arange(n) % hosts.size
            got = pool.estimate(hosts[pick])
            assert np.array_equal(got["aip"], hosts[pick])
            assert np.array_equal(got["nat"], np.array([w[1] for w in want])[pick])
            est = np.array([w[0] for w in want])[pick]
            np.testing.assert_allclose(got["est"], est, rtol=EST_RTOL, atol=EST_ATOL)
            assert np.array_equal((got["flags"] & 2) != 0, est >= p["theta"])
        rec = pool.estimate(torch.from_numpy(hosts.view(np.int32)).cuda()).view(-1, 4).cpu().numpy()
        assert np.array_equal(rec[:, 1], [w[1] for w in want])
    pool.close()

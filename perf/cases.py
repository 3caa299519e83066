"""The work that users of this library have it do, as measurable cases.

``listed()`` names them, ``draw()`` gives more of the same ranges, ``prepare()`` makes what a
program holds before the call (on the GPU, from a seed), ``run()`` is one pass through the public
Python entry points, ``work()`` the bytes and operations a pass cannot do without, and ``exact()``
the computed numbers of the first pass in 64 bits, by plain torch and numpy.

Every pool case works on traffic of the shape of the synthetic workloads: Zipf hosts whose opposite
hosts come from sets with a power-law size (or of 1 to 16 members), plus planted super points whose
window cardinalities are log-uniform around the threshold.  A pool is prepared with RING slices
already in its window, and a pass takes the next batch of the ring.
"""
import math

import numpy as np
import torch

from paper_1807_01527_gb300 import asse

P32 = (1 << 32) + 15          # the mangling modulus
M32 = 0xFFFFFFFF
RING = 4                      # distinct slice batches a state holds
DISTINCT = 1.0 / 6.0          # distinct (aip, bip) pairs per pair of a batch, about
LIST = 4096                   # records of the buffer a list of super points comes back in


def listed():
    link = dict(k=10, theta=1024, g=512, r=4, elog=16, hosts=1 << 20, zipf=1.1, sets="power", n=8 << 20)
    long = dict(k=60, theta=4096, g=1024, r=4, elog=18, hosts=1 << 22, zipf=1.2, sets="power", n=32 << 20)
    return [
        # the smallest link: one slice of 64 Ki packets, where launches and waits are all there is
        dict(name="tiny_slice", kind="slice", counter="at", host=False, k=4, theta=64, g=128, r=4, elog=10,
             hosts=4096, zipf=1.1, sets="small", n=65536),
        # a slice of an edge link, packets already on the device: ingest, close, read the report
        dict(name="link_slice", kind="slice", counter="at", host=False, **link),
        # the same slice arriving in pinned host memory, as from a capture card
        dict(name="link_slice_host", kind="slice", counter="at", host=True, **link),
        # aging counters, the paper's other counter: every close decrements the whole pool
        dict(name="link_slice_aging", kind="slice", counter="ace", host=False, **link),
        # one slice answered for several windows at once (the last second, the half and the full window)
        dict(name="link_windows", kind="windows", counter="at", kps="10,5,1", **link),
        # a long window over a pool much larger than L2, with slice counts, the kind advised for it
        dict(name="long_slice", kind="slice", counter="hist", host=False, **long),
        # the same window with the library's default counter
        dict(name="long_slice_plain", kind="slice", counter="at", host=False, **long),
        # four differently shaped links served side by side: submit each its slice, poll until all reported
        dict(name="serve_four", kind="serve", streams=4, scale=16),
        # a look into the open slice without ending it: stepwise scan and restore, a watch list estimated
        dict(name="link_peek", kind="peek", counter="at", watch=100_003, **link),
        # learned estimate of every estimator of the pool: feature rows, tensor-core MLP, fallback rule
        dict(name="link_learned", kind="learned", counter="at", **link),
        # training of that model: Adam steps at the batch size of the training runs
        dict(name="train_steps", kind="train", rows=4096, steps=4, loss="log_mse"),
        # synthetic training states of the link pool's shape for that training
        dict(name="train_states", kind="states", rows=16384, k=10, g=512, r=4, n_max_log2=20, bg=0.08),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["slice", "slice", "slice", "windows", "serve", "peek", "learned", "train", "states"])
    if kind == "serve":
        return dict(kind=kind, streams=rng.randint(2, 6), scale=_log(rng, 12, 64))
    if kind == "train":
        return dict(kind=kind, rows=_log(rng, 1024, 16384), steps=rng.randint(1, 6), loss="log_mse")
    if kind == "states":
        k = _log(rng, 4, 60)
        return dict(kind=kind, rows=_log(rng, 1024, 16384), k=k, g=_log(rng, max(128, 2 * k), 1024), r=4,
                    n_max_log2=rng.randint(12, 20), bg=round(rng.uniform(0.01, 0.1), 3))
    k = _log(rng, 3, 60)
    g = _log(rng, max(128, 2 * k), 1024)
    elog = rng.randint(13, 18)
    r = rng.choice([4, 4, 4, 3, 5]) if elog >= 15 else 4
    # between a thirtieth and a fifth of a pair per AT of a row and slice, as the workloads have
    n = min(32 << 20, max(50_000, int((g << elog) * math.exp(rng.uniform(math.log(1 / 30), math.log(1 / 5)))) | 1))
    c = dict(kind=kind, counter="at", k=k, theta=int(g * rng.uniform(1.5, 4)), g=g, r=r, elog=elog,
             hosts=max(4096, n // 8), zipf=round(rng.uniform(1.05, 1.25), 3), sets="power", n=n)
    if kind == "slice":
        c["counter"] = rng.choice(["at", "at", "hist", "ace"])
        c["host"] = rng.random() < 0.25
    elif kind == "windows":
        c["counter"] = rng.choice(["at", "at", "hist"])
        c["kps"] = "%d,%d" % (k, max(1, k // 2))
    elif kind == "peek":
        c["counter"] = rng.choice(["at", "hist"])
        c["watch"] = _log(rng, 1000, 200_000)
    else:
        c["counter"] = rng.choice(["at", "hist"])
    return c


# ------------------------------------------------------------------ inputs

def _mix(x):
    """A bijection of 32-bit values held in int64 tensors (the murmur3 finaliser)."""
    x = x ^ (x >> 16)
    x = (x * 0x85EBCA6B) & M32
    x = x ^ (x >> 13)
    x = (x * 0xC2B2AE35) & M32
    return x ^ (x >> 16)


def _column_split(elog, r):
    for u in (4, 0):
        c, w = elog - u, 32 - u
        if c >= 1 and r * c >= w and c <= w:
            s = max(1, -(-(w - c) // (r - 1)))
            if s <= c and s * (r - 1) < w:
                return c, u, s
    raise ValueError("no column split for 2^%d ATVs and %d rows" % (elog, r))


def _params(case, seed):
    c, u, s = _column_split(case["elog"], case["r"])
    rs = np.random.RandomState(seed % (1 << 31))
    return dict(k=case["k"], theta=case["theta"], g=case["g"], r=case["r"], c=c, u=u, s=s,
                A=int(rs.randint(2, 1 << 32, dtype=np.uint64)),
                bh_a=int(rs.randint(0, 1 << 63, dtype=np.uint64)) | 1,
                bh_b=int(rs.randint(0, 1 << 63, dtype=np.uint64)))


def _as_pairs(a, b):
    """(n, 2) int32 tensor of two int64 columns of 32-bit values."""
    return torch.stack([a, b], 1).view(torch.int32)[:, ::2].contiguous()


def _batches(case, seed):
    """RING batches of (aip, bip) pairs on the GPU."""
    gen = torch.Generator(device="cuda").manual_seed(seed)
    n, hosts, theta = case["n"], case["hosts"], case["theta"]
    salt = (seed * 0x9E3779B1 + 12345) & M32
    nb = min(case["k"], RING)
    cdf = torch.arange(1, hosts + 1, dtype=torch.float64, device="cuda").pow_(-case["zipf"]).cumsum_(0)
    cdf /= cdf[-1].clone()
    # planted hosts: window cardinalities log-uniform in [theta/2, 20 theta], at most 8 % of the pairs
    n_pl = max(3, min((1 << case["elog"]) // 328, int(0.08 * n * nb / (5.3 * theta))))
    card = torch.exp(torch.rand(n_pl, generator=gen, device="cuda", dtype=torch.float64) * math.log(40.0)) * theta / 2
    per = torch.ceil(card / nb).long()
    pl = torch.repeat_interleave(torch.arange(n_pl, device="cuda"), per)
    pl_j = torch.arange(pl.numel(), device="cuda") - torch.repeat_interleave(per.cumsum(0) - per, per)
    pl_aip = _mix((pl + hosts + salt) & M32)
    out = []
    for t in range(nb):
        m = max(0, n - pl.numel())
        rank = torch.searchsorted(cdf, torch.rand(m, generator=gen, device="cuda", dtype=torch.float64), right=True)
        rank.clamp_(max=hosts - 1)
        v = _mix((rank + (salt ^ 0x51ED270B)) & M32)
        size = 1 + v % 16 if case["sets"] == "small" else ((1 << 32) // (v + 1)).clamp_(1, 1 << 20)
        j = (torch.rand(m, generator=gen, device="cuda", dtype=torch.float64) * size).long()
        aip = torch.cat([pl_aip, _mix((rank + salt) & M32)])
        bip = _mix((_mix(aip ^ 0x5BD1E995) + torch.cat([pl_j + t * per[pl], j])) & M32)
        order = torch.randperm(aip.numel(), generator=gen, device="cuda")[:n]
        out.append(_as_pairs(aip[order], bip[order]))
    return out


class _Words:
    """The packed words of a pool, for a tensor of them without a copy (the tensor keeps this object, and so the pool)."""

    def __init__(self, pool):
        info = pool.info()
        self.pool = pool
        self.__cuda_array_interface__ = {"shape": (info["pool_words"],), "typestr": "<i4",
                                         "data": (info["pool"], False), "version": 3}


def _pool_state(case, seed):
    params = _params(case, seed)
    pool = asse.Pool(params, counter=case["counter"])
    batches = _batches(case, seed)
    for b in batches:                      # the slices already in the window
        pool.ingest(b)
        pool.close_slice()
    if case.get("host"):
        batches = [b.cpu().pin_memory() for b in batches]
    return dict(case=case, params=params, pool=pool, batches=batches, t=0,
                words=torch.as_tensor(_Words(pool), device="cuda"))


SHAPES = ((256, asse.FEAT), (256,), (256, 256), (256,), (256,), (1,))  # W1, b1, W2, b2, w3, b3


def _weights(seed, b3=0.0):
    """A model's parameters: uniform weights scaled by their fan-in (unused features zero), zero biases but the last."""
    rs = np.random.RandomState((seed + 1) % (1 << 31))
    w = [np.zeros(s) for s in SHAPES]
    for i, fan in ((0, 68), (2, 256), (4, 256)):
        w[i][...] = rs.uniform(-1, 1, SHAPES[i]) * math.sqrt(6.0 / fan)
    w[0][:, 68:] = 0.0
    w[5][0] = b3
    return np.concatenate([v.ravel() for v in w]).astype(np.float32)


def _model(seed, b3=0.0):
    mlp = asse.MLP(seed=seed)
    mlp.set_params(_weights(seed, b3))
    return mlp


def _feature_rows(rows, seed):
    """Rows shaped like the estimator's features (ages, count, loads) and their ln n targets."""
    gen = torch.Generator(device="cuda").manual_seed(seed)
    k, g = 10, 512
    rnd = lambda *s: torch.rand(*s, generator=gen, device="cuda", dtype=torch.float64)  # noqa: E731
    ln = rnd(rows) * 20 * math.log(2.0)
    share = -torch.log(rnd(rows, k) + 1e-12)
    load = share / share.sum(1, keepdim=True) * torch.exp(ln)[:, None] / g + 0.08 * rnd(rows)[:, None]
    older = load.cumsum(1) - load
    ages = torch.floor(g * torch.exp(-older) * -torch.expm1(-load)) / g
    p = -torch.expm1(-0.08 * k * rnd(rows))
    x = torch.zeros(rows, asse.FEAT, dtype=torch.float64, device="cuda")
    x[:, 0] = ages.sum(1)
    x[:, 1:1 + k] = ages
    x[:, 65], x[:, 66], x[:, 67] = p, p ** 4, p
    return x.to(torch.bfloat16), ln.to(torch.float32)


def _stream_cases(case):
    shapes = [(10, 16, 512), (4, 14, 128), (30, 15, 512), (60, 17, 1024), (4, 15, 512), (10, 14, 1024)]
    for k, elog, g in shapes[: case["streams"]]:
        n = (g << elog) // case["scale"] | 1
        yield dict(k=k, theta=2 * g, g=g, r=4, elog=elog, hosts=max(4096, n // 8), zipf=1.1, sets="power", n=n)


def _states_cfg(case, seed):
    rs = np.random.RandomState(seed % (1 << 31))
    return dict(k=case["k"], g=case["g"], r=case["r"], n_max_log2=case["n_max_log2"], bg_max=case["bg"], seed=seed,
                bh_a=int(rs.randint(0, 1 << 63, dtype=np.uint64)) | 1,
                bh_b=int(rs.randint(0, 1 << 63, dtype=np.uint64)))


def prepare(case, seed):
    kind = case["kind"]
    if kind == "train":
        mlp = _model(seed)
        mlp.set_loss(case["loss"])
        return dict(case=case, mlp=mlp, data=[_feature_rows(case["rows"], seed * 16 + i) for i in range(case["steps"])])
    if kind == "states":
        return dict(case=case, cfg=_states_cfg(case, seed), first=0)
    if kind == "serve":
        server = asse.Server(64 << 30)
        streams = []
        for i, c in enumerate(_stream_cases(case)):
            batches = _batches(c, seed * 16 + i)
            sid = server.open(_params(c, seed * 16 + i), c["k"], max_batch=c["n"])
            streams.append((sid, batches))
        torch.cuda.synchronize()
        for t in range(RING):
            _serve(server, streams, t)
        return dict(case=case, server=server, streams=streams, t=0)
    s = _pool_state(case, seed)
    if kind in ("peek", "learned"):
        s["pool"].ingest(s["batches"][0])  # the open slice's packets so far
    if kind == "peek":
        gen = torch.Generator(device="cuda").manual_seed(seed + 7)
        some = torch.randint(0, case["n"], (case["watch"],), generator=gen, device="cuda")
        s["watch"] = s["batches"][1][some, 0].contiguous()
    if kind == "learned":
        s["mlp"] = _model(seed, 5.0)  # outputs about e^5, inside the training range
    return s


# ------------------------------------------------------------------ one pass

def _listing(rec):
    """A list of super points by address (its own order is unspecified), in a buffer of LIST records."""
    out = np.zeros(LIST, dtype=rec.dtype)
    rec = rec[np.argsort(rec["aip"], kind="stable")][:LIST]
    out[: rec.size] = rec
    return {"n": rec.size, "aip": out["aip"].astype(np.int64), "nat": out["nat"].astype(np.int64), "est": out["est"],
            "flags": out["flags"].astype(np.int64)}


def _serve(server, streams, t):
    for sid, batches in streams:
        server.submit(sid, batches[t % len(batches)], True)
    reports = []
    for sid, _ in streams:
        got = None
        while got is None:
            got = server.poll(sid)
        reports.append(_listing(got[0]))
    return reports


def run(state):
    kind = state["case"]["kind"]
    if kind == "train":
        losses = [state["mlp"].train_step(x, t, 1e-3) for x, t in state["data"]]
        return {"loss": losses, "params": state["mlp"].params()}
    if kind == "states":
        n = state["case"]["rows"]
        x, ln, lc = asse.synth_states(state["cfg"], state["first"], n)
        state["first"] += n
        return {"x": x, "ln": ln, "lc": lc}
    if kind == "serve":
        state["t"] += 1
        return _serve(state["server"], state["streams"], state["t"] - 1)
    pool = state["pool"]
    if kind == "peek":
        pool.scan()
        pool.restore()
        est = pool.estimate(state["watch"])
        rec = est.view(-1, 4)
        return {"loads": pool.loads().astype(np.int64), "candidates": _listing(pool.candidates()), "nat": rec[:, 1],
                "est": rec[:, 2].view(torch.float32)}
    if kind == "learned":
        pool.scan()
        est, fallbacks, x = pool.estimate_learned(state["mlp"], 20 * math.log(2.0))
        return {"est": est, "x": x, "fallbacks": fallbacks}
    batch = state["batches"][state["t"] % len(state["batches"])]
    state["t"] += 1
    pool.ingest(batch)
    if kind == "windows":
        kps = [int(v) for v in state["case"]["kps"].split(",")]
        pool.close_slice_multi(kps)
        out = []
        for i in range(len(kps)):
            pool.select_window(i)
            out.append(_listing(pool.report()))
        return {"reports": out, "pool": state["words"]}
    pool.close_slice()
    return {"report": _listing(pool.report()), "pool": state["words"]}


def _pool_bytes(case):
    values = case["k"] + 1 if case.get("counter") == "ace" else 2 * case["k"] + 1
    return case["r"] * (1 << case["elog"]) * 4 * math.ceil(case["g"] / (32 // math.ceil(math.log2(values))))


def _slice_bytes(case):
    pool = _pool_bytes(case)
    atv = case["r"] << case["elog"]
    # the pairs, one word of each row read and written for every distinct pair, and the close: every
    # counter read (slice counts: one sum per ATV), the two refreshed blocks of 2k written, or, with
    # aging counters, every counter written
    batch = 8 * case["n"] + DISTINCT * case["n"] * case["r"] * 8
    if case.get("counter") == "hist":
        return batch + 6 * atv + 2 * pool / (2 * case["k"])
    return batch + pool + (pool if case.get("counter") == "ace" else pool / (2 * case["k"]))


def work(case):
    kind = case["kind"]
    mac = 80 * 256 + 256 * 256 + 256
    if kind == "train":
        return {"bytes": case["steps"] * (case["rows"] * 164 + 6 * 4 * mac), "flops": case["steps"] * case["rows"] * 6 * mac}
    if kind == "states":
        return {"bytes": case["rows"] * 168, "flops": 0}
    if kind == "serve":
        return {"bytes": sum(_slice_bytes(c) for c in _stream_cases(case)), "flops": 0}
    if kind == "peek":
        return {"bytes": _pool_bytes(case) + 20 * case["watch"], "flops": 0}
    if kind == "learned":
        atv = case["r"] << case["elog"]
        return {"bytes": _pool_bytes(case) + 164 * atv, "flops": 2 * atv * mac}
    return {"bytes": _slice_bytes(case), "flops": 0}


# ------------------------------------------------------------------ the same in 64 bits

class _Exact:
    """The pool by its definition: for every AT the slice that last set it."""

    def __init__(self, case, seed):
        self.case, self.p = case, _params(case, seed)
        self.r, self.g, self.e = case["r"], case["g"], 1 << case["elog"]
        self.w = 32 - self.p["u"]
        self.last = torch.full((self.r, self.e, self.g), -1, dtype=torch.int8, device="cuda")
        self.now = 0
        batches = _batches(case, seed)
        self.batches = batches
        for t, b in enumerate(batches + [batches[0]]):  # the window before, then the first pass's slice
            self.now = t
            for part in b.split(1 << 23):
                self._set(part.long() & M32, t)

    def rows(self, aip):
        p = self.p
        y = aip
        for first in (True, False, False):
            z = ((y * (p["A"] >> 16)) % P32 * 65536 + y * (p["A"] & 0xFFFF)) % P32
            y = z if first else torch.where(y >> 32 > 0, z, y)
        frame = y & ((1 << p["u"]) - 1)
        lbs = y >> p["u"]
        twice = (lbs << self.w) | lbs
        cols = [(twice >> self.shift(i)) & ((1 << p["c"]) - 1) for i in range(self.r)]
        return frame, [(frame << p["c"]) | x for x in cols]

    def shift(self, i):
        return 2 * self.w - self.p["c"] - self.p["s"] * i

    def _set(self, pairs, t):
        wrap = lambda v: v - (1 << 64) if v >> 63 else v  # noqa: E731
        h = pairs[:, 1] * wrap(self.p["bh_a"]) + wrap(self.p["bh_b"])
        h = (((h >> 32) & M32) * self.g) >> 32
        _, atvs = self.rows(pairs[:, 0])
        for i, a in enumerate(atvs):
            self.last[i].view(-1)[a * self.g + h] = t

    def window(self, kp):
        self.on = (self.last >= 0) & (self.last > self.now - kp)
        self.count = self.on.sum(2, dtype=torch.int64)
        loads = self.count.view(self.r, 1 << self.p["u"], -1).sum(2)
        self.load = loads.double() / (self.g * float(1 << self.p["c"]))
        self.up = self.load.prod(0)

    def eq4(self, nat, frame):
        ratio = (self.g - nat.double()) / (self.g * (1.0 - self.up[frame]))
        n = -self.g * torch.log(ratio.clamp(max=1.0))
        return torch.where((nat >= self.g) | (self.up[frame] >= 1.0), torch.full_like(n, math.inf), n)

    def nat(self, atvs):
        return torch.cat([torch.stack([self.on[i, a] for i, a in enumerate(part)]).all(0).sum(1)
                          for part in zip(*[a.split(1 << 15) for a in atvs])])

    def restored(self):
        """Every candidate: addresses by the join of the super ATVs of each frame."""
        p = self.p
        need = math.ceil(self.g - self.g * math.exp(-p["theta"] / self.g))
        full = np.uint64((1 << self.w) - 1)
        sup = (self.count >= need).cpu().numpy().reshape(self.r, 1 << p["u"], -1)
        inv = pow(p["A"], -1, P32)
        found = []
        for j in range(1 << p["u"]):
            val, known = np.zeros(1, np.uint64), np.zeros(1, np.uint64)
            for i in range(self.r):
                sh = np.uint64(self.shift(i))
                put = lambda x: ((x << sh) >> np.uint64(self.w)) | ((x << sh) & full)  # noqa: E731
                v = put(np.nonzero(sup[i, j])[0].astype(np.uint64))
                m = put(np.array([(1 << p["c"]) - 1], np.uint64))[0]
                a, b = np.nonzero(((val[:, None] ^ v[None, :]) & m & known[:, None]) == 0)
                val, known = val[a] | v[b], known[a] | m
            for y in ((int(x) << p["u"]) | j for x in val):
                x = inv * y % P32
                while x >> 32:
                    x = inv * x % P32
                found.append(x)
        return torch.tensor(sorted(found), dtype=torch.int64, device="cuda")

    def listing(self, reported):
        aip, out = self.restored(), np.zeros(LIST)
        if aip.numel():
            frame, atvs = self.rows(aip)
            est = self.eq4(self.nat(atvs), frame)
            est = (est[est >= self.p["theta"]] if reported else est)[:LIST]
            out[: est.numel()] = est.cpu().numpy()
        return {"n": None, "aip": None, "nat": None, "est": out, "flags": None}

    def features(self, kp):
        """Feature rows [r*E][80] in 64 bits."""
        x = torch.zeros(self.r * self.e, asse.FEAT, dtype=torch.float64, device="cuda")
        for a in range(min(kp, self.now + 1)):
            x[:, 1 + a] = (self.last == self.now - a).sum(2).view(-1).double() / self.g
        x[:, 0] = self.count.view(-1).double() / self.g
        cols = 1 << self.p["c"]
        x[:, 65] = self.load.repeat_interleave(cols, 1).view(-1)
        x[:, 66] = self.up.repeat_interleave(cols).repeat(self.r)
        x[:, 67] = self.load.mean(0).repeat_interleave(cols).repeat(self.r)
        return x


def _unpack(p):
    """W1, b1, W2, b2, w3, b3 of a flat parameter tensor."""
    out, at = [], 0
    for shape in SHAPES:
        n = math.prod(shape)
        out.append(p[at: at + n].view(shape))
        at += n
    return out


def _forward(p, x):
    w1, b1, w2, b2, w3, b3 = _unpack(p)
    return torch.relu(torch.relu(x @ w1.T + b1) @ w2.T + b2) @ w3 + b3


def _weights64(seed, b3=0.0):
    return torch.from_numpy(_weights(seed, b3)).cuda().double()


def _exact_train(case, seed):
    p = _weights64(seed)
    m, v, losses = torch.zeros_like(p), torch.zeros_like(p), []
    for i in range(case["steps"]):
        x, t = _feature_rows(case["rows"], seed * 16 + i)
        p = p.detach().requires_grad_(True)
        d = _forward(p, x.double()) - t.double()
        loss = d.square().mean()
        grad, = torch.autograd.grad(loss, p)
        losses.append(loss.detach().view(1))
        m, v = 0.9 * m + 0.1 * grad, 0.999 * v + 0.001 * grad.square()
        p = p.detach() - 1e-3 * (m / (1 - 0.9 ** (i + 1))) / (torch.sqrt(v / (1 - 0.999 ** (i + 1))) + 1e-8)
    return {"loss": losses, "params": p}


def _splitmix(x):
    srl = lambda z, n: (z >> n) & ((1 << (64 - n)) - 1)  # noqa: E731
    wrap = lambda v: v - (1 << 64)  # noqa: E731
    z = x + wrap(0x9E3779B97F4A7C15)
    z = (z ^ srl(z, 30)) * wrap(0xBF58476D1CE4E5B9)
    z = (z ^ srl(z, 27)) * wrap(0x94D049BB133111EB)
    return z ^ srl(z, 31)


def _exact_states(case, seed):
    """ln n and the Eq. 2 estimate of states 0 .. rows-1, from the generator's published draws."""
    cfg = _states_cfg(case, seed)
    unit = lambda key, i: ((_splitmix(key ^ _splitmix(i)) >> 11) & ((1 << 53) - 1)).double() / (1 << 53)  # noqa: E731
    n, k, g = case["rows"], case["k"], case["g"]
    at = lambda v: torch.tensor(v, dtype=torch.int64, device="cuda")  # noqa: E731
    key = _splitmix(at(seed) ^ _splitmix(torch.arange(n, device="cuda") + 0x51ED270B27))
    card = torch.floor(torch.exp(unit(key, at(1)) * (case["n_max_log2"] * 0.6931471805599453))).clamp(min=1).long()
    pbg = (unit(key, at(2)) * float(np.float32(case["bg"]))).float().double()
    on = torch.zeros(n, g, dtype=torch.bool, device="cuda")
    for s in range(k):
        i = (s << 32) | torch.arange(g, device="cuda")
        on |= unit((key ^ 0xB5)[:, None], i[None, :]) < pbg[:, None]
    base, ends = (key >> 32) & M32, card.cumsum(0)
    wrap = lambda v: v - (1 << 64) if v >> 63 else v  # noqa: E731
    for lo in range(0, int(ends[-1]), 1 << 25):
        e = torch.arange(lo, min(lo + (1 << 25), int(ends[-1])), device="cuda")
        i = torch.searchsorted(ends, e, right=True)
        h = _mix((base[i] + e - (ends[i] - card[i])) & M32) * wrap(cfg["bh_a"]) + wrap(cfg["bh_b"])
        on.view(-1)[i * g + ((((h >> 32) & M32) * g) >> 32)] = True
    c = on.sum(1).double()
    c = torch.where(c >= g, torch.full_like(c, g - 0.5), c)
    return {"x": None, "ln": torch.log(card.double()), "lc": -g * torch.log((g - c) / g)}


def exact(case, seed):
    kind = case["kind"]
    if kind == "train":
        return _exact_train(case, seed)
    if kind == "states":
        return _exact_states(case, seed)
    if kind == "serve":
        out = []
        for i, c in enumerate(_stream_cases(case)):
            e = _Exact(c, seed * 16 + i)
            e.window(c["k"])
            out.append(e.listing(True))
        return out
    e = _Exact(case, seed)
    if kind == "windows":
        out = []
        for kp in (int(v) for v in case["kps"].split(",")):
            e.window(kp)
            out.append(e.listing(True))
        return {"reports": out, "pool": None}
    e.window(case["k"])
    if kind == "learned":
        x = e.features(case["k"])
        w = _weights64(seed, 5.0)
        y = torch.cat([_forward(w, part) for part in x.split(1 << 16)])
        cc = e.count.view(-1).double()
        cc = torch.where(cc >= e.g, torch.full_like(cc, e.g - 0.5), cc)
        eq2 = -e.g * torch.log((e.g - cc) / e.g)
        inside = (e.count.view(-1) > 0) & (y <= 20 * math.log(2.0))
        return {"est": torch.where(inside, torch.exp(y.clamp(min=0.0)), eq2), "x": x, "fallbacks": None}
    if kind == "peek":
        gen = torch.Generator(device="cuda").manual_seed(seed + 7)
        some = torch.randint(0, case["n"], (case["watch"],), generator=gen, device="cuda")
        frame, atvs = e.rows(e.batches[1][some, 0].long() & M32)
        return {"loads": None, "candidates": e.listing(False), "nat": None, "est": e.eq4(e.nat(atvs), frame)}
    return {"report": e.listing(True), "pool": None}

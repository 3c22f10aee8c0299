"""Workloads of the super point library whose speed is watched.

A case is one pass of work as a program that uses the library has it done,
through the binding's public entry points (``paper_1901_07306_gb300.sp``) or
the serving engine.  ``listed`` gives the watched cases, ``draw`` more of the
same ranges, ``prepare`` what a program holds before the call, ``run`` one
pass and its outputs, ``work`` the bytes a pass cannot do without, and
``exact`` the estimates of Eq. 4 from a plain 64-bit evaluation of the scheme.

Traffic is shaped like the benchmark's core link (``workloads.core_link``):
Zipf(1.1) background sources, planted hosts with log-uniform numbers of
peers, one pair in ten a duplicate, shuffled.  It is drawn on the GPU, where
2^28 pairs take a fraction of a second.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_1901_07306_gb300 import serving, sp

# Parameter sets.  D: the library's default; D3 and S: the benchmark's
# distributed and serving profiles; K12: the tests' wide estimators (k = 4096,
# which the binned scan does not take); R3: the tests' three-row profile with
# k = 256, at a core-link LDCA width; M: the benchmark's many-results profile.
PROFILES = {
    "D": dict(r=14, isb=(0, 5, 10, 15), ibn=(7, 7, 7, 7), k_log2=10, lr=4, lc_log2=16),
    "D3": dict(r=16, isb=(0, 4, 8, 12), ibn=(7, 7, 7, 7), k_log2=10, lr=4, lc_log2=18),
    "S": dict(r=12, isb=(0, 5, 10, 15), ibn=(7, 7, 7, 7), k_log2=10, lr=4, lc_log2=14),
    "K12": dict(r=14, isb=(0, 5, 10, 15), ibn=(7, 7, 7, 7), k_log2=12, lr=4, lc_log2=14),
    "R3": dict(r=12, isb=(0, 7, 14), ibn=(8, 8, 8), k_log2=8, lr=3, lc_log2=16),
    "M": dict(r=16, isb=(0, 8), ibn=(9, 9), k_log2=10, lr=4, lc_log2=16),
}
HASH_SEED = 0x5EED
BINNED_MIN = 1 << 22                      # updates from here on need the reserved lists


def listed():
    return [
        # the smallest call: a quiet link's window, where launches and the wait count
        dict(name="window_4k", kind="window", profile="S", n=4099, off=0, theta=128),
        # the single-router configuration: 2^20 pairs, one window
        dict(name="window_1m", kind="window", profile="D", n=1 << 20, off=0, theta=1024),
        # estimators too wide for the binned scan, an odd number of pairs
        dict(name="window_k4096", kind="window", profile="K12", n=1500001, off=1, theta=2048),
        # the benchmark's headline: a core link's window
        dict(name="window_64m", kind="window", profile="D", n=1 << 26, off=0, theta=1024),
        # a watch point that ships its sketch to the global server (Sec. 4.2):
        # odd size, a stream that starts off a 16-byte boundary
        dict(name="ship_5m", kind="ship", profile="D", n=5000011, off=1, theta=1024),
        # the watch point's host path (Sec. 4.1): pairs in pinned host memory
        dict(name="host_16m", kind="host", profile="D", n=(1 << 24) - 77, off=0, theta=1024),
        # the distributed configuration: 16 routers' uneven batches, merge, detect
        dict(name="distributed_16x16m", kind="batched", profile="D3", routers=16, n=1 << 24, batches=64, theta=1024),
        # many small batches named in a device table (the form a CUDA graph replays)
        dict(name="table_64", kind="table", profile="S", routers=64, lo=10, hi=15, batches=256, theta=1024),
        # the global server: OR of 16 watch points' shipped sketches, detect
        dict(name="gs_merge_16", kind="gs", profile="D", images=16, n=1 << 20, theta=1024),
        # sliding window (Sec. 5): slices of uneven size, a detection per slice
        dict(name="sliding_8", kind="sliding", profile="D", slices=8, window=4, n=1 << 21, theta=1024),
        # the serving engine: pinned requests of 2^12 - 2^22 pairs from 64 routers
        dict(name="serving_64", kind="serving", profile="S", routers=64, requests=48, lo=12, hi=22, theta=1024),
        # a detection that returns about 150,000 hosts (the benchmark's many results)
        dict(name="detect_150k", kind="many", profile="M", hosts=150000, peers=64, theta=32),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["window"] * 4 + ["ship"] * 2 + ["host", "batched", "batched", "table", "gs", "sliding",
                                                       "serving", "many"])
    theta = rng.choice([512, 1024])
    if kind in ("window", "ship"):
        profile = rng.choice(["D", "D", "S", "D3", "K12", "R3"] if kind == "window" else ["D", "S", "R3"])
        n = _log(rng, 1 << 12, 1 << (26 if kind == "window" else 25))
        return dict(kind=kind, profile=profile, n=n, off=rng.randrange(2), theta=theta if n >= 1 << 15 else 128)
    if kind == "host":
        return dict(kind=kind, profile=rng.choice(["D", "S"]), n=_log(rng, 1 << 16, 1 << 25), off=0, theta=theta)
    if kind == "batched":
        return dict(kind=kind, profile=rng.choice(["D", "D3"]), routers=rng.randint(2, 16),
                    n=_log(rng, 1 << 19, 1 << 24), batches=rng.randint(1, 64), theta=theta)
    if kind == "table":
        return dict(kind=kind, profile="S", routers=rng.randint(8, 64), lo=8, hi=rng.randint(12, 16),
                    batches=_log(rng, 16, 1024), theta=theta)
    if kind == "gs":
        return dict(kind=kind, profile=rng.choice(["D", "S"]), images=rng.randint(2, 40), n=_log(rng, 1 << 17, 1 << 20),
                    theta=theta)
    if kind == "sliding":
        return dict(kind=kind, profile=rng.choice(["D", "S"]), slices=rng.randint(3, 8), window=rng.choice([2, 4, 32, 128]),
                    n=_log(rng, 1 << 18, 1 << 22), theta=theta)
    if kind == "serving":
        return dict(kind=kind, profile="S", routers=rng.randint(8, 64), requests=rng.randint(16, 64), lo=12,
                    hi=rng.randint(16, 21), theta=theta)
    return dict(kind="many", profile="M", hosts=_log(rng, 2000, 150000), peers=64, theta=32)


# ---- inputs ------------------------------------------------------------------
def _gen(seed, stream=0):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed) * 1000003 + stream)
    return g


def _addresses(g, n):
    return torch.randint(0, 1 << 32, (n,), generator=g, device="cuda")


def _traffic(n, g, off=0, shared=None):
    """n pairs as one int32 tensor of 2 n values, its start ``off`` pairs into
    its allocation.  ``shared``: hosts (and their weights) common to several
    routers, 30% of each router's sources."""
    sources = max(256, n // 16)
    hosts = _addresses(g, sources)
    if shared is not None:
        m = min(shared.numel(), sources * 3 // 10)
        hosts[:m] = shared[:m]
    # relative degrees: Zipf(1.1) truncated at 2^12, by its continuous inverse
    tail = float((1 << 12) + 1) ** -0.1
    u = torch.rand(sources, generator=g, device="cuda", dtype=torch.float64)
    ends = torch.cumsum(torch.floor((1.0 - u * (1.0 - tail)) ** -10.0), 0)
    # planted hosts, 500 in 2^26 pairs, 1,500 - 50,000 peers each
    hi = min(50000, max(8, n // 8))
    lo = min(1500, hi)
    planted = max(2, n * 500 >> 26)
    v = torch.rand(planted, generator=g, device="cuda", dtype=torch.float64)
    degree = (lo * torch.exp(v * math.log(hi / lo))).to(torch.int64)
    heavy = torch.repeat_interleave(_addresses(g, planted), degree)
    distinct = n - n // 10
    heavy = heavy[: distinct // 2]
    w = torch.rand(distinct - heavy.numel(), generator=g, device="cuda", dtype=torch.float64) * ends[-1]
    hip = torch.cat([heavy, hosts[torch.searchsorted(ends, w, right=True).clamp_(max=sources - 1)]])
    del w
    oip = _addresses(g, distinct)
    again = torch.randint(0, distinct, (n - distinct,), generator=g, device="cuda")
    order = torch.cat([torch.arange(distinct, device="cuda"), again])
    order = order[torch.randperm(n, generator=g, device="cuda")]
    out = torch.empty(2 * (n + off), dtype=torch.int32, device="cuda")[2 * off:]
    out[0::2] = hip[order].to(torch.int32)
    out[1::2] = oip[order].to(torch.int32)
    return out


def _sizes(count, lo, hi):
    """Batch sizes, log-uniform in [2^lo, 2^hi], the same for every seed (the
    serving engine's windows then close at the same requests)."""
    rng = np.random.default_rng(11)
    return [int(x) for x in np.exp(rng.uniform(lo * math.log(2), hi * math.log(2), count))]


def _cuts(n, parts, seed):
    """[0, n) in uneven parts (weights log-uniform in [1, 16])."""
    rng = np.random.default_rng(int(seed))
    w = np.exp(rng.uniform(0, math.log(16.0), parts))
    at = np.floor(np.cumsum(w / w.sum())[:-1] * n).astype(np.int64).tolist()
    return list(zip([0, *at], [*at, n]))


def _streams(case, seed):
    """[(router, pairs on the GPU)] of a case, in the order they are sent."""
    kind, out = case["kind"], []
    if kind in ("window", "ship", "host"):
        return [(0, _traffic(case["n"], _gen(seed), case["off"]))]
    if kind == "batched":
        common = _addresses(_gen(seed, 99991), 1 << 19)
        for r in range(case["routers"]):
            t = _traffic(case["n"], _gen(seed, r), 0, common)
            out += [(r, t[2 * a:2 * b]) for a, b in _cuts(case["n"], case["batches"], seed * 64 + r)]
        order = np.random.default_rng(int(seed)).permutation(len(out))
        return [out[i] for i in order]
    if kind in ("table", "serving"):
        count = case["batches"] if kind == "table" else case["requests"]
        sizes = _sizes(count, case["lo"], case["hi"])
        routers = np.random.default_rng(int(seed) + 1).integers(0, case["routers"], count)
        total = _traffic(sum(sizes), _gen(seed))
        at = 0
        for r, n in zip(routers, sizes):
            out.append((int(r), total[2 * at:2 * (at + n)]))
            at += n
        return out
    if kind == "gs":
        return [(i, _traffic(case["n"], _gen(seed, i))) for i in range(case["images"])]
    if kind == "sliding":
        common = _addresses(_gen(seed, 99991), 1 << 16)
        return [(t, _traffic(max(1024, b - a), _gen(seed, t), 0, common))
                for t, (a, b) in enumerate(_cuts(case["n"] * case["slices"], case["slices"], seed))]
    g = _gen(seed)                                     # many results: distinct peers per host, shuffled
    hip = torch.repeat_interleave(_addresses(g, case["hosts"]), case["peers"])
    hip = hip[torch.randperm(hip.numel(), generator=g, device="cuda")]
    out = torch.stack([hip, _addresses(g, hip.numel())], 1).to(torch.int32).reshape(-1)
    return [(0, out)]


def _context(case, routers=1, window=1):
    return sp.SuperPoint(sp.make_params(theta=case["theta"], seed=HASH_SEED, n_routers=routers, window_slices=window,
                                        **PROFILES[case["profile"]]))


# ---- one case ------------------------------------------------------------------
def prepare(case, seed):
    kind, streams = case["kind"], _streams(case, seed)
    s = dict(kind=kind, rows=_rows(case))
    if kind == "serving":
        # pinned requests, all arrived when the run starts (offered load above capacity)
        s["server"] = serving.SketchServer(case["routers"], dict(PROFILES[case["profile"]], theta=case["theta"],
                                                                 seed=HASH_SEED),
                                           budget_bytes=2 << 30, detect_every=1 << 24)
        s["requests"] = [serving.Request(router=r, pairs=t.cpu().pin_memory(), arrival=0.0) for r, t in streams]
        return s
    routers = case["routers"] + 1 if kind in ("batched", "table") else 1
    ctx = s["ctx"] = _context(case, routers, case.get("window", 1))
    if kind in ("batched", "host") or case.get("n", 0) >= BINNED_MIN:
        sp.sp_reserve(ctx.ctx)
    if kind == "host":
        s["pairs"] = streams[0][1].cpu().pin_memory()
    elif kind in ("window", "ship"):
        s["pairs"] = streams[0][1]
        if kind == "ship":
            s["image"] = torch.zeros(sp.sp_copy_sketch_bytes(ctx.ctx), dtype=torch.uint8, device="cuda")
    elif kind in ("batched", "table"):
        s["routers"], s["batches"], s["gs"] = [r for r, _ in streams], [t for _, t in streams], case["routers"]
        if kind == "table":
            rows = np.zeros(len(streams), sp.BATCH)
            for i, (r, t) in enumerate(streams):
                rows[i] = (t.data_ptr(), t.numel() // 2, r, 0)
            s["table"] = torch.from_numpy(rows.view(np.uint8)).cuda()
    elif kind == "gs":
        size = sp.sp_copy_sketch_bytes(ctx.ctx)
        s["images"] = [torch.zeros(size, dtype=torch.uint8, device="cuda") for _ in streams]
        for image, (_, t) in zip(s["images"], streams):
            sp.sp_reset(ctx.ctx, 0)
            sp.sp_update(ctx.ctx, 0, t)
            sp.sp_copy_sketch(ctx.ctx, 0, image)
    elif kind == "sliding":
        s["slices"] = [t for _, t in streams]
    else:
        ctx.update(streams[0][1])
        torch.cuda.synchronize()
    return s


def _answer(s, recs, found):
    """A detection's records in a table of the case's fixed length, as a
    report keeps them (rows past the last record are zero)."""
    out = np.zeros(s["rows"], sp.CANDIDATE)
    m = min(len(recs), s["rows"])
    out[:m] = recs[:m]
    return dict(ip=out["ip"], z0=out["z0"], est=out["est"], flags=out["flags"], found=int(found))


def _rows(case):
    return case["hosts"] * 5 // 4 if case["kind"] == "many" else 4096 if case.get("n", 1 << 20) > 1 << 16 else 256


def run(s):
    kind = s["kind"]
    if kind == "serving":
        return [_answer(s, w.records, w.n_found) for w in s["server"].run(s["requests"])]
    c = s["ctx"].ctx
    if kind in ("window", "ship"):
        sp.sp_reset(c, 0)
        sp.sp_update(c, 0, s["pairs"])
        if kind == "ship":
            sp.sp_copy_sketch(c, 0, s["image"])
            return s["image"]
    elif kind == "host":
        sp.sp_reset(c, 0)
        sp.sp_update_host(c, 0, s["pairs"])
    elif kind in ("batched", "table"):
        gs = s["gs"]
        sp.sp_reset_range(c, 0, gs + 1)
        if kind == "batched":
            sp.sp_update_batched(c, s["routers"], s["batches"])
        else:
            sp.sp_update_batched_device(c, s["table"], len(s["batches"]))
        sp.sp_merge(c, list(range(gs)), gs)
        return _answer(s, *sp.sp_detect(c, gs, 0)[:2])
    elif kind == "gs":
        sp.sp_reset(c, 0)
        sp.sp_merge_device(c, s["images"], 0)
    elif kind == "sliding":
        sp.sp_reset(c, 0)
        out = []
        for t, pairs in enumerate(s["slices"]):
            if t:
                sp.sp_slide(c, 0)
            sp.sp_update(c, 0, pairs)
            out.append(_answer(s, *sp.sp_detect(c, 0, 0)[:2]))
        return out
    if kind == "many":                                   # a caller's table of `rows` records, filled by the call
        recs, found, _ = sp.sp_detect(c, 0, 0, cap=s["rows"])
        table = recs.base
        return dict(ip=table["ip"], z0=table["z0"], est=table["est"], flags=table["flags"], found=int(found))
    return _answer(s, *sp.sp_detect(c, 0, 0)[:2])


def _sketch_bytes(case):
    p = PROFILES[case["profile"]]
    return (sum(1 << b for b in p["ibn"]) << p["r"]) + (p["lr"] << (p["lc_log2"] + p["k_log2"])) // 8


def work(case):
    """Bytes of a pass: every pair (8 bytes) or image read once, the sketch a
    pass makes written once, every result record (24 bytes) written once."""
    kind, sketch = case["kind"], _sketch_bytes(case)
    if kind == "many":
        p = PROFILES[case["profile"]]
        lines = p["lr"] << (p["k_log2"] - 3)             # the LDC lines a reported host is tested on
        return {"bytes": (sum(1 << b for b in p["ibn"]) << p["r"]) + case["hosts"] * (24 + lines), "flops": 0}
    if kind == "gs":
        return {"bytes": (case["images"] + 1) * sketch, "flops": 0}
    if kind in ("window", "ship", "host"):
        pairs = case["n"]
    elif kind == "batched":
        pairs = case["n"] * case["routers"]
    elif kind == "sliding":
        pairs = case["n"] * case["slices"]
    else:                                                # mean of a log-uniform size times the batches
        lo, hi = 2.0 ** case["lo"], 2.0 ** case["hi"]
        pairs = (hi - lo) / math.log(hi / lo) * case.get("batches", case.get("requests"))
    return {"bytes": int(8 * pairs) + sketch, "flops": 0}


# ---- the estimates in 64 bits ------------------------------------------------------
def _hash_words(count):
    s, out = HASH_SEED, []
    for _ in range(2 * count):                           # SplitMix64
        s = (s + 0x9E3779B97F4A7C15) & (2 ** 64 - 1)
        z = s
        z = ((z ^ (z >> 30)) * 0xBF58476D1CE4E5B9) & (2 ** 64 - 1)
        z = ((z ^ (z >> 27)) * 0x94D049BB133111EB) & (2 ** 64 - 1)
        z ^= z >> 31
        out.append(z - (1 << 64) if z >> 63 else z)
    return list(zip(out[0::2], out[1::2]))


def _mas(ab, x):
    return ((x * ab[0] + ab[1]) >> 32) & 0xFFFFFFFF


def _estimates(case, streams):
    """Eq. 4's estimates of the hosts reported for the union of the streams,
    by ascending address: every (RP, LP) whose SEs agree is tried, no pruning."""
    p, theta = PROFILES[case["profile"]], case["theta"]
    r, rows, k_log2, lr, lc_log2 = p["r"], list(zip(p["isb"], p["ibn"])), p["k_log2"], p["lr"], p["lc_log2"]
    L, k = 32 - r, 1 << k_log2
    h = _hash_words(2 + lr)
    tau = max(0, math.ceil(math.log2(theta / 8)))
    sea, offs = sum(1 << b for _, b in rows), []
    for _, b in rows:
        offs.append(sum(1 << x for _, x in rows[:len(offs)]))
    idx = lambda lp, i: ((lp | (lp << L)) >> rows[i][0]) & ((1 << rows[i][1]) - 1)  # noqa: E731  Eq. 2
    bits = torch.zeros((1 << r) * sea * 8, dtype=torch.bool, device="cuda")
    ldca = torch.zeros(lr, (1 << lc_log2) * k, dtype=torch.bool, device="cuda")
    for t in streams:
        for part in torch.split(t.reshape(-1, 2), 1 << 23):
            hip, oip = (part[:, j].to(torch.int64) & 0xFFFFFFFF for j in (0, 1))
            h1 = _mas(h[0], oip)
            b3 = _mas(h[1], oip) >> (32 - k_log2)
            for i in range(lr):
                ldca[i][((_mas(h[2 + i], hip) >> (32 - lc_log2)) << k_log2) + b3] = True
            on = (h1 & ((1 << tau) - 1)) == 0
            hs, bit = hip[on], h1[on] >> 29
            for i in range(len(rows)):
                bits[((hs & ((1 << r) - 1)) * sea + offs[i] + idx(hs >> r, i)) * 8 + bit] = True
    weights = (1 << torch.arange(8, device="cuda")).to(torch.uint8)
    seav = torch.empty(1 << r, sea, dtype=torch.uint8, device="cuda")
    for a in range(0, 1 << r, 1024):
        part = bits[a * sea * 8:(a + 1024) * sea * 8].view(-1, 8)
        seav[a:a + 1024] = (part * weights).sum(1, dtype=torch.int64).to(torch.uint8).view(-1, sea)
    lp = torch.arange(1 << L, device="cuda")
    at = [offs[i] + idx(lp, i) for i in range(len(rows))]
    hot = torch.tensor([bin(x).count("1") >= 3 for x in range(256)], device="cuda")
    step, found = max(1, 1 << (25 - L)), []
    for a in range(0, 1 << r, step):
        block = seav[a:a + step]
        seu = block[:, at[0]]
        for i in range(1, len(rows)):
            seu &= block[:, at[i]]
        rp, lps = torch.nonzero(hot[seu.to(torch.int64)], as_tuple=True)
        found.append((lps << r) | (rp + a))
    ips = torch.sort(torch.cat(found)).values
    z0 = []
    for part in torch.split(ips, 1 << 17):
        u = None
        for i in range(lr):
            line = ldca[i].view(1 << lc_log2, k)[_mas(h[2 + i], part) >> (32 - lc_log2)]
            u = line if u is None else u & line
        z0.append(k - u.sum(1))
    z0 = torch.cat(z0).to(torch.float64)
    est = torch.where(z0 == 0, k * math.log(k), -k * torch.log(z0.clamp(min=1) / k))
    return est[est >= theta].cpu().numpy()


def exact(case, seed):
    def answer(streams):
        est, out = _estimates(case, streams), np.zeros(_rows(case))
        out[:min(est.size, out.size)] = est[:out.size]
        return dict(ip=None, z0=None, est=out, flags=None, found=None)

    kind, streams = case["kind"], [t for _, t in _streams(case, seed)]
    if kind == "ship":
        return None                                      # a sketch is bits, no computed numbers
    if kind == "sliding":
        return [answer(streams[max(0, t - case["window"] + 1):t + 1]) for t in range(len(streams))]
    if kind == "serving":
        out, part, pairs = [], [], 0
        for t in streams:                                # a window closes at 2^24 admitted pairs
            part.append(t)
            pairs += t.numel() // 2
            if pairs >= 1 << 24:
                out.append(answer(part))
                part, pairs = [], 0
        return out + ([answer(part)] if part else [])
    return answer(streams)

"""The work that is timed: sessions classified against a prefix list and
histogrammed by time and direction, through the package's public entry points.

``listed()`` names the cases, ``draw()`` gives more of the same ranges,
``prepare()`` makes what a program holds before the call, ``run()`` is one
pass and ``exact()`` the same outputs from plain torch in 64 bits.

Records are made on the GPU from the seed alone, with the distributions of
the synthetic workloads in ``gen/``: 40 % of the records leave the listed
networks, 40 % enter them, 10 % stay inside and 10 % outside; byte counts are
log-normal (mu 8, sigma 2).
"""
import math

import numpy as np
import torch

import paper_2106_12863_gb300 as sinet

DAY_MS = 86_400_000
CHUNK = 1 << 25  # records made at a time
POLICIES = {"exclusive": sinet.EXCLUSIVE, "paper": sinet.PAPER_ALG1, "inclusive": sinet.INCLUSIVE}


def _fused(name, **over):
    case = {"name": name, "kind": "fused", "records": 1_000_000, "order": "uniform", "from_ms": 0,
            "span_ms": DAY_MS, "t0_ms": 0, "width_ms": 1, "bins": DAY_MS, "prefixes": 2000, "len_lo": 8,
            "len_hi": 30, "weighted": True, "watch": 0, "policy": "exclusive", "strategy": "auto",
            "accumulate": False, "offset": 0}
    case.update(over)
    return case


def listed():
    return [
        # one minute of a paper-scale day, added to the day's resident histogram
        # as it arrives (400 M sessions a day are 278 K a minute): the smallest call
        _fused("minute into the day", records=278_001, order="sorted", from_ms=50_400_000, span_ms=60_000,
               accumulate=True),
        # the tiny workload: an hour of a small network at 1 ms
        _fused("hour of 1 M", records=1_000_000, span_ms=3_600_000, bins=3_600_000, prefixes=64, len_lo=16,
               len_hi=24, weighted=False),
        # a slice the size of the largest of the batch workload as a call of its own:
        # unsorted, six hours at 1 ms, starting off a 16-byte boundary
        _fused("six hours of 20 M unsorted", records=19_999_999, from_ms=18_000_000, span_ms=21_600_000,
               t0_ms=18_000_000, bins=21_600_000, prefixes=4000, len_hi=32, weighted=False, offset=3),
        # an hour at 1 s for a dashboard; sessions inside the network count in both directions
        _fused("hour in seconds, inclusive", records=50_000_007, span_ms=3_600_000, width_ms=1000, bins=3600,
               prefixes=1000, policy="inclusive", offset=1),
        # the paper-scale day: 400 M records sorted by time up to +-500 ms
        _fused("day of 400 M sorted", records=400_000_000, order="sorted"),
        # the heavy day: 1.6 B records, Zipf-skewed bins and hosts
        _fused("heavy day of 1.6 B", records=1_600_000_000, order="zipf", prefixes=8000, len_hi=32,
               weighted=False),
        # the paper's own structure (discriminate, sort, reduce by key), asked for by name
        _fused("plain path of 16 M", records=16_000_001, span_ms=3_600_000, bins=3_600_000, prefixes=64,
               len_lo=16, len_hi=24, weighted=False, strategy="sort_reduce"),
        # Algorithm 1 alone, with the class of every record: a filter in front of other tools
        {"name": "classify 200 M", "kind": "classify", "records": 200_000_003, "prefixes": 2000, "len_lo": 8,
         "len_hi": 30, "weighted": True, "hosts": "prefix", "offset": 0},
        # records classified earlier, histogrammed at another width (10 ms)
        {"name": "classified 100 M at 10 ms", "kind": "classified", "records": 100_000_001, "order": "sorted",
         "from_ms": 0, "span_ms": DAY_MS, "t0_ms": 0, "width_ms": 10, "bins": 8_640_000,
         "policy": "exclusive", "accumulate": False, "offset": 0},
        # 256 uneven slices with a list, window and width each, in one launch
        {"name": "batch of 256", "kind": "batch", "slices": 256, "lo": 10_000, "hi": 20_000_000, "plan": 4},
        # requests of eight tenants from pinned host memory into their resident
        # day histograms (1 s bins), which are read back for a dashboard
        {"name": "eight requests served", "kind": "serve", "tenants": 8, "requests": 8, "median": 1_000_000,
         "cap": 4_000_000, "width_ms": 1000, "plan": 5},
        # the day's report: ten-minute totals and the non-empty milliseconds
        {"name": "report of a day", "kind": "report", "bins": DAY_MS, "filled": 82_000_001, "factor": 600_000},
    ]


def _log(rng, lo, hi):
    return int(math.exp(rng.uniform(math.log(lo), math.log(hi))))


def _draw_table(rng):
    lo, hi, weighted = rng.choice([(16, 24, False), (8, 30, True), (8, 32, False)])
    return {"prefixes": _log(rng, 16, 8000), "len_lo": lo, "len_hi": hi, "weighted": weighted}


def _draw_window(rng, width):
    span = min(_log(rng, 60_000, DAY_MS) // width + 1, DAY_MS // width) * width
    start = rng.randrange(0, DAY_MS - span + 1)
    return {"from_ms": start, "span_ms": span, "t0_ms": start, "width_ms": width, "bins": span // width}


def draw(rng):
    kind = rng.choice(["fused"] * 6 + ["plain", "classify", "classify", "classified", "batch", "serve", "report"])
    policy = rng.choice(["exclusive", "exclusive", "paper", "inclusive"])
    offset = rng.choice([0, 0, 1, 2, 3])
    width = rng.choice([1, 1, 10, 1000])
    if kind in ("fused", "plain"):
        plain = kind == "plain"
        case = _fused("", records=_log(rng, 10_000, 30_000_000 if plain else 200_000_000),
                      order=rng.choice(["uniform", "sorted", "zipf"]), policy=policy, offset=offset,
                      accumulate=rng.random() < 0.25, strategy="sort_reduce" if plain else "auto",
                      watch=0 if plain or rng.random() < 0.85 else _log(rng, 16, 2000),
                      **_draw_table(rng), **_draw_window(rng, width))
        if plain and case["records"] < 500_000:
            case["strategy"] = "noalloc"
    elif kind == "classify":
        case = {"kind": kind, "records": _log(rng, 10_000, 200_000_000), "hosts": rng.choice(["prefix", "zipf"]),
                "offset": offset, **_draw_table(rng)}
    elif kind == "classified":
        case = {"kind": kind, "records": _log(rng, 10_000, 200_000_000),
                "order": rng.choice(["uniform", "sorted", "zipf"]), "policy": policy,
                "accumulate": rng.random() < 0.25, "offset": offset, **_draw_window(rng, width)}
    elif kind == "batch":
        case = {"kind": kind, "slices": rng.randrange(8, 129), "lo": 10_000,
                "hi": _log(rng, 100_000, 20_000_000), "plan": rng.randrange(1 << 30)}
    elif kind == "serve":
        case = {"kind": kind, "tenants": rng.randrange(2, 17), "requests": rng.randrange(4, 25),
                "median": _log(rng, 50_000, 1_000_000), "cap": 4_000_000, "width_ms": 1000,
                "plan": rng.randrange(1 << 30)}
    else:
        bins = _log(rng, 100_000, DAY_MS)
        case = {"kind": "report", "bins": bins, "filled": max(1, int(bins * rng.uniform(0.01, 0.98))),
                "factor": rng.choice([10, 1000, 60_000, 600_000])}
    case.pop("name", None)
    return case


# --------------------------------------------------------------------------
# Inputs


def _table(seed, prefixes, len_lo, len_hi, weighted):
    """A prefix list within 0.0.0.0/1 (host bits clear); lengths 16-24 are four times as likely when weighted."""
    rng = np.random.default_rng(seed)
    lens = np.arange(len_lo, len_hi + 1)
    p = np.where(weighted & (lens >= 16) & (lens <= 24), 4.0, 1.0)
    ln = rng.choice(lens, prefixes, p=p / p.sum()).astype(np.uint8)
    mask = (0xFFFFFFFF << (32 - ln.astype(np.int64))) & 0xFFFFFFFF
    net = (rng.integers(0, 1 << 31, prefixes) & mask).astype(np.uint32)
    return net, ln


def _zipf(n, ranks, g, dev):
    """Ranks 0 .. ranks - 1 under Zipf's law with s = 1.1, by inverting the integral of x^-s."""
    a, b = 0.5 ** -0.1, (ranks + 0.5) ** -0.1
    v = torch.rand(n, generator=g, device=dev, dtype=torch.float64).mul_(b - a).add_(a)
    v2 = v * v
    v4 = v2 * v2
    x = (v4 * v4).mul_(v2).reciprocal_()  # v^-10
    return x.add_(0.5).floor_().clamp_(1, ranks).to(torch.int64) - 1


def _inside(n, net, host, g, dev):
    k = torch.randint(0, len(net), (n,), generator=g, device=dev)
    return net[k] | (torch.randint(0, 1 << 32, (n,), generator=g, device=dev) & host[k])


def _outside(n, g, dev):
    return torch.randint(1 << 31, 0xE0000000, (n,), generator=g, device=dev)


class _Hosts:
    """Addresses inside and outside a list: uniform, or Zipf-ranked from two pools of 25,000."""

    def __init__(self, net, ln, zipf, g, dev):
        self.net = torch.from_numpy(net.astype(np.int64)).to(dev)
        self.host = torch.from_numpy((1 << (32 - ln.astype(np.int64))) - 1).to(dev)
        self.g, self.dev, self.pools = g, dev, None
        if zipf:
            self.pools = _inside(25_000, self.net, self.host, g, dev), _outside(25_000, g, dev)

    def pick(self, inside):
        n = inside.numel()
        if self.pools:
            k = _zipf(n, 25_000, self.g, self.dev)
            a, b = self.pools[0][k], self.pools[1][k]
        else:
            a, b = _inside(n, self.net, self.host, self.g, self.dev), _outside(n, self.g, self.dev)
        return torch.where(inside, a, b)


def _classes(n, g, dev):
    """0 neither, 1 source inside, 2 destination inside, 3 both: 10, 40, 40 and 10 %."""
    u = torch.rand(n, generator=g, device=dev)
    return (u >= 0.1).to(torch.uint8) + (u >= 0.5).to(torch.uint8) + (u >= 0.9).to(torch.uint8)


def _sizes(n, g, dev):
    x = torch.randn(n, generator=g, device=dev).mul_(2).add_(8).exp_()
    return x.double().floor_().clamp_(max=4294967295.0).to(torch.int64)


def _times(case, first, n, g, dev):
    lo, span = case["from_ms"], case["span_ms"]
    if case["order"] == "uniform":
        return torch.randint(lo, lo + span, (n,), generator=g, device=dev)
    if case["order"] == "zipf":
        w, bins = case["width_ms"], max(1, span // case["width_ms"])
        a = 48_271 * 7919 % bins | 1
        while math.gcd(a, bins) != 1:
            a += 2
        b = (_zipf(n, bins, g, dev) * a + bins // 3) % bins  # hot bins spread over the window
        return lo + b * w + (torch.randint(0, w, (n,), generator=g, device=dev) if w > 1 else 0)
    # sorted up to +-500 ms; over a whole day the rate is 2 + cos(2 pi (t - 14 h) / 24 h)
    u = (torch.arange(first, first + n, device=dev, dtype=torch.float64) + 0.5) / case["records"]
    if span == DAY_MS:
        t = torch.linspace(0, DAY_MS, 86_401, device=dev, dtype=torch.float64)
        k = 2 * math.pi / DAY_MS
        cdf = 2 * t + (torch.sin(k * t - k * 14 * 3_600_000) + math.sin(k * 14 * 3_600_000)) / k
        cdf = cdf / cdf[-1].clone()
        i = torch.searchsorted(cdf, u).clamp_(1, 86_400)
        u = t[i - 1] + (u - cdf[i - 1]) / (cdf[i] - cdf[i - 1]) * 1000.0
    else:
        u = u * span
    t = u.floor_().to(torch.int64) + torch.randint(-500, 501, (n,), generator=g, device=dev)
    return t.clamp_(0, span - 1).add_(lo)


def _buffers(n, offset, dev, **kinds):
    """Record streams of n records, `offset` records into their allocation."""
    return {k: torch.empty(n + offset, dtype=t, device=dev)[offset:] for k, t in kinds.items()}


def _fill(case, rec, hosts, g, dev, first=0, n=None):
    """Make records [first, first + n) of a case in the streams that `rec` holds."""
    n = case["records"] if n is None else n
    for i in range(0, n, CHUNK):
        m = min(CHUNK, n - i)
        cls = _classes(m, g, dev)
        at = slice(first + i, first + i + m)
        if "src" in rec:
            rec["src"][at] = hosts.pick((cls & 1).bool()).to(torch.int32)
            rec["dst"][at] = hosts.pick((cls & 2).bool()).to(torch.int32)
        if "cls" in rec:
            rec["cls"][at] = cls
        if "ts" in rec:
            rec["ts"][at] = _times(case, i, m, g, dev)
            rec["bytes"][at] = _sizes(m, g, dev).to(torch.int32)


RECORD = {"ts": torch.int64, "src": torch.int32, "dst": torch.int32, "bytes": torch.int32}


def _slices(case):
    """The slice plan of a batch: sizes, windows (1 min - 6 h), widths and list sizes."""
    rng = np.random.default_rng(case["plan"])
    out = []
    for _ in range(case["slices"]):
        n = int(math.exp(rng.uniform(math.log(case["lo"]), math.log(case["hi"]))))
        w = int(rng.choice([1, 10, 1000]))
        span = -(-int(math.exp(rng.uniform(math.log(60_000), math.log(21_600_000)))) // w) * w
        t0 = int(rng.integers(0, DAY_MS - span))
        out.append({"records": n, "order": "uniform", "from_ms": t0, "span_ms": span, "t0_ms": t0, "width_ms": w,
                    "bins": span // w, "policy": "exclusive",
                    "prefixes": int(math.exp(rng.uniform(math.log(16), math.log(4000))))})
    return out


def _requests(case):
    """The requests of a serving pass: log-normal sizes (median, p99 = 50 medians), windows of 1 min - 6 h."""
    rng = np.random.default_rng(case["plan"])
    lists = [int(rng.integers(500, 4001)) for _ in range(case["tenants"])]
    out = []
    for i in range(case["requests"]):
        n = min(case["cap"], max(1000, int(case["median"] * math.exp(rng.normal() * math.log(50) / 2.326))))
        span = int(math.exp(rng.uniform(math.log(60_000), math.log(21_600_000))))
        out.append({"tenant": i % case["tenants"], "records": n, "order": "uniform",
                    "from_ms": int(rng.integers(0, DAY_MS - span)), "span_ms": span})
    return lists, out


def _inputs(case, seed):
    """Everything a case's call reads, from the seed alone (no call of the package)."""
    dev = torch.device("cuda")
    g = torch.Generator(dev)
    g.manual_seed(seed)
    kind = case["kind"]
    if kind == "fused":
        net, ln = _table(seed, case["prefixes"], case["len_lo"], case["len_hi"], case["weighted"])
        hosts = _Hosts(net, ln, case["order"] == "zipf", g, dev)
        rec = _buffers(case["records"], case["offset"], dev, **RECORD)
        _fill(case, rec, hosts, g, dev)
        watch = None
        if case["watch"]:  # hosts and small networks out of both address ranges
            wl = np.random.default_rng(seed + 1)
            length = wl.integers(16, 33, case["watch"]).astype(np.uint8)
            base = np.where(wl.random(case["watch"]) < 0.5, net[wl.integers(0, len(net), case["watch"])].astype(np.int64),
                            wl.integers(1 << 31, 0xE0000000, case["watch"]))
            watch = (base.astype(np.uint32), length)
        return {"table": (net, ln), "rec": rec, "watch": watch}
    if kind == "classify":
        net, ln = _table(seed, case["prefixes"], case["len_lo"], case["len_hi"], case["weighted"])
        hosts = _Hosts(net, ln, case["hosts"] == "zipf", g, dev)
        rec = _buffers(case["records"], case["offset"], dev, src=torch.int32, dst=torch.int32)
        _fill(case, rec, hosts, g, dev)
        return {"table": (net, ln), "rec": rec}
    if kind == "classified":
        rec = _buffers(case["records"], case["offset"], dev, ts=torch.int64, bytes=torch.int32, cls=torch.uint8)
        _fill(case, rec, None, g, dev)
        return {"rec": rec}
    if kind == "batch":
        plan = _slices(case)
        rec = _buffers(sum(s["records"] for s in plan), 0, dev, **RECORD)
        tables, first = [], 0
        for i, s in enumerate(plan):
            tables.append(_table(seed * 1000 + i, s["prefixes"], 8, 32, False))
            _fill(s, rec, _Hosts(*tables[-1], False, g, dev), g, dev, first, s["records"])
            first += s["records"]
        return {"plan": plan, "tables": tables, "rec": rec}
    if kind == "serve":
        lists, plan = _requests(case)
        tables = [_table(seed * 1000 + i, p, 8, 32, False) for i, p in enumerate(lists)]
        recs = []
        for q in plan:
            rec = _buffers(q["records"], 0, dev, **RECORD)
            _fill(q, rec, _Hosts(*tables[q["tenant"]], False, g, dev), g, dev)
            recs.append(rec)
        return {"plan": plan, "tables": tables, "recs": recs}
    # report: a histogram with `filled` non-empty bins spread over the window
    n, k = case["bins"], case["filled"]
    a = int(torch.randint(n // 3, n, (1,), generator=g, device=dev)) | 1
    while math.gcd(a, n) != 1:
        a += 2
    at = (torch.arange(k, device=dev) * a + seed) % n
    count = torch.zeros((2, n), dtype=torch.int32, device=dev)
    nbytes = torch.zeros((2, n), dtype=torch.int64, device=dev)
    side = torch.randint(1, 4, (k,), generator=g, device=dev)  # one direction or both
    for d in (0, 1):
        c = torch.randint(1, 6, (k,), generator=g, device=dev) * ((side >> d) & 1)
        count[d, at] = c.to(torch.int32)
        nbytes[d, at] = c * _sizes(k, g, dev)
    return {"count": count, "bytes": nbytes}


# --------------------------------------------------------------------------
# A program's state, and one pass


class _View:
    """A slice's outputs as views of the batch's flat output arrays."""

    def __init__(self, count, nbytes, stats, first, bins):
        self.n_bins = bins
        self.count = count[2 * first:2 * (first + bins)].view(2, bins)
        self.bytes = nbytes[2 * first:2 * (first + bins)].view(2, bins)
        self.stats = stats

    c = sinet.Histogram.c


def _params(case, **more):
    return sinet.HistParams(case["t0_ms"], case["width_ms"], case["bins"], policy=POLICIES[case["policy"]],
                            hints=sinet.HINT_TIME_SORTED if case["order"] == "sorted" else 0, **more)


def prepare(case, seed):
    x = _inputs(case, seed)
    kind, s = case["kind"], {"kind": case["kind"]}
    if kind == "fused":
        watch = sinet.PrefixTable(*x["watch"]) if x["watch"] else None
        noalloc = case["strategy"] == "noalloc"
        s.update(table=sinet.PrefixTable(*x["table"]), rec=x["rec"], out=sinet.Histogram(case["bins"]), noalloc=noalloc,
                 params=_params(case, accumulate=case["accumulate"], watch=watch,
                                strategy="auto" if noalloc else case["strategy"]))
    elif kind == "classify":
        s.update(table=sinet.PrefixTable(*x["table"]), rec=x["rec"],
                 cls=torch.empty(case["records"], dtype=torch.uint8, device="cuda"))
    elif kind == "classified":
        s.update(rec=x["rec"], out=sinet.Histogram(case["bins"]), params=_params(case, accumulate=case["accumulate"]))
    elif kind == "batch":
        bins = sum(p["bins"] for p in x["plan"])
        s["count"] = torch.zeros(2 * bins, dtype=torch.int32, device="cuda")
        s["bytes"] = torch.zeros(2 * bins, dtype=torch.int64, device="cuda")
        s["stats"] = torch.zeros((len(x["plan"]), 8), dtype=torch.int64, device="cuda")
        slices, first, b = [], 0, 0
        for i, (p, t) in enumerate(zip(x["plan"], x["tables"])):
            r = [x["rec"][k][first:first + p["records"]] for k in RECORD]
            out = _View(s["count"], s["bytes"], s["stats"][i], b, p["bins"])
            slices.append((sinet.PrefixTable(*t), *r, _params(p), out))
            first += p["records"]
            b += p["bins"]
        s["batch"] = sinet.Batch(slices, autotune=True)
    elif kind == "serve":
        tables = [sinet.PrefixTable(*t) for t in x["tables"]]
        p = sinet.HistParams(0, case["width_ms"], DAY_MS // case["width_ms"])
        s["server"] = sinet.Server([(t, p) for t in tables], budget_bytes=1 << 30)
        s["requests"] = []
        for q, rec in zip(x["plan"], x["recs"]):
            host = [torch.empty(v.shape, dtype=v.dtype, pin_memory=True).copy_(v) for v in rec.values()]
            s["requests"].append((q["tenant"], host))
    else:
        s["hist"] = sinet.Histogram(case["bins"])
        s["hist"].count, s["hist"].bytes, s["factor"] = x["count"], x["bytes"], case["factor"]
    return s


def run(s):
    kind = s["kind"]
    if kind == "fused":
        r, out = s["rec"], s["out"]
        if s["noalloc"]:
            sinet.sinet_discriminate_histogram_noalloc(s["table"].handle, r["ts"], r["src"], r["dst"], r["bytes"],
                                                       r["ts"].numel(), s["params"].c(), out.c())
        else:
            sinet.discriminate_histogram(s["table"], r["ts"], r["src"], r["dst"], r["bytes"], s["params"], out)
        return {"count": out.count, "bytes": out.bytes, "stats": out.stats}
    if kind == "classify":
        return {"counts": sinet.discriminate(s["table"], s["rec"]["src"], s["rec"]["dst"], s["cls"]), "class": s["cls"]}
    if kind == "classified":
        out = sinet.histogram(s["rec"]["ts"], s["rec"]["bytes"], s["rec"]["cls"], s["params"], s["out"])
        return {"count": out.count, "bytes": out.bytes, "stats": out.stats}
    if kind == "batch":
        s["batch"].run()
        return {"count": s["count"], "bytes": s["bytes"], "stats": s["stats"]}
    if kind == "serve":
        tickets = [s["server"].submit(tenant, *host) for tenant, host in s["requests"]]
        for t in tickets:
            s["server"].wait(t)
        hists = [s["server"].export(i) for i in range(len(s["server"].n_bins))]
        # the bits of the unsigned arrays
        return [{"count": h["count"].view(np.int32), "bytes": h["bytes"].view(np.int64),
                 "stats": h["stats"].view(np.int64)} for h in hists]
    coarse = sinet.rollup(s["hist"], s["factor"])
    dense = sinet.sparse(s["hist"])
    return {"coarse_count": coarse.count, "coarse_bytes": coarse.bytes, "present": dense["n"], "bin": dense["bin"],
            "count": dense["count"], "bytes": dense["bytes"]}


def _bin_bytes(records, bins, accumulate):
    """Every bin written once; a running histogram reads and writes only the bins that are hit."""
    return 48 * min(records, 2 * bins) // 2 if accumulate else 24 * bins


def work(case):
    kind = case["kind"]
    if kind == "fused":
        b = 20 * case["records"] + _bin_bytes(case["records"], case["bins"], case["accumulate"])
    elif kind == "classify":
        b = 9 * case["records"]
    elif kind == "classified":
        b = 13 * case["records"] + _bin_bytes(case["records"], case["bins"], case["accumulate"])
    elif kind == "batch":
        b = sum(20 * p["records"] + 24 * p["bins"] for p in _slices(case))
    elif kind == "serve":
        b = sum(20 * q["records"] for q in _requests(case)[1]) + case["tenants"] * 24 * (DAY_MS // case["width_ms"])
    else:
        b = 24 * case["bins"] + 28 * case["filled"] + 24 * -(-case["bins"] // case["factor"])
    return {"bytes": b, "flops": 0}


# --------------------------------------------------------------------------
# The same outputs from plain torch


def _intervals(net, ln, dev):
    """The union of a prefix list as sorted disjoint ranges."""
    size = 1 << (32 - ln.astype(np.int64))
    lo = net.astype(np.int64) & -size
    order = np.lexsort((lo + size, lo))
    a, b = [], []
    for x, y in zip(lo[order].tolist(), (lo + size - 1)[order].tolist()):
        if a and x <= b[-1] + 1:
            b[-1] = max(b[-1], y)
        else:
            a.append(x)
            b.append(y)
    return torch.tensor(a, device=dev), torch.tensor(b, device=dev)


def _member(addr, iv):
    a = addr.to(torch.int64) & 0xFFFFFFFF
    k = torch.searchsorted(iv[0], a, right=True) - 1
    return (k >= 0) & (a <= iv[1][k.clamp(min=0)])


def _class_of(rec, at, iv):
    return _member(rec["src"][at], iv).to(torch.int64) + 2 * _member(rec["dst"][at], iv).to(torch.int64)


def _plain(case, rec, first, n, iv, watch=None):
    """count[2, bins], bytes[2, bins] and stats[8] of records [first, first + n), in 64 bits."""
    dev = rec["ts"].device
    bins, t0, w = case["bins"], case["t0_ms"], case["width_ms"]
    count = torch.zeros((2, bins), dtype=torch.int64, device=dev)
    total = torch.zeros((2, bins), dtype=torch.int64, device=dev)
    stats = torch.zeros(8, dtype=torch.int64, device=dev)
    policy = torch.tensor(POLICIES[case["policy"]], device=dev)
    for i in range(first, first + n, CHUNK):
        at = slice(i, min(i + CHUNK, first + n))
        cls = rec["cls"][at].to(torch.int64) if iv is None else _class_of(rec, at, iv)
        ts, by = rec["ts"][at], rec["bytes"][at].to(torch.int64) & 0xFFFFFFFF
        if watch is not None:
            keep = _member(rec["src"][at], watch) | _member(rec["dst"][at], watch)
            stats[6] += (~keep).sum()
            cls, ts, by = cls[keep], ts[keep], by[keep]
        stats[:4] += torch.bincount(cls, minlength=4)
        inside = (ts >= t0) & (ts < t0 + bins * w)
        for d in (0, 1):
            routed = (policy[cls] >> d & 1).bool()
            stats[4 + d] += (routed & ~inside).sum()
            hit = routed & inside
            b = (ts[hit] - t0) // w
            count[d].index_add_(0, b, torch.ones_like(b))
            total[d].index_add_(0, b, by[hit])
    return {"count": count, "bytes": total, "stats": stats}


def exact(case, seed):
    x = _inputs(case, seed)
    dev, kind = torch.device("cuda"), case["kind"]
    if kind == "fused":
        watch = _intervals(*x["watch"], dev) if x["watch"] else None
        return _plain(case, x["rec"], 0, case["records"], _intervals(*x["table"], dev), watch)
    if kind == "classify":
        iv = _intervals(*x["table"], dev)
        cls = torch.cat([_class_of(x["rec"], slice(i, i + CHUNK), iv).to(torch.uint8)
                         for i in range(0, case["records"], CHUNK)])
        return {"counts": torch.bincount(cls.to(torch.int64), minlength=4), "class": cls}
    if kind == "classified":
        return _plain(case, x["rec"], 0, case["records"], None)
    if kind == "batch":
        parts, first = [], 0
        for p, t in zip(x["plan"], x["tables"]):
            parts.append(_plain(p, x["rec"], first, p["records"], _intervals(*t, dev)))
            first += p["records"]
        return {"count": torch.cat([p["count"].reshape(-1) for p in parts]),
                "bytes": torch.cat([p["bytes"].reshape(-1) for p in parts]),
                "stats": torch.stack([p["stats"] for p in parts])}
    if kind == "serve":
        day = {"t0_ms": 0, "width_ms": case["width_ms"], "bins": DAY_MS // case["width_ms"], "policy": "exclusive"}
        ivs = [_intervals(*t, dev) for t in x["tables"]]
        got = [None] * case["tenants"]
        for q, rec in zip(x["plan"], x["recs"]):
            h = _plain(day, rec, 0, q["records"], ivs[q["tenant"]])
            old = got[q["tenant"]]
            got[q["tenant"]] = h if old is None else {k: h[k] + old[k] for k in h}
        return [h if h is not None else None for h in got]
    f, n = case["factor"], case["bins"]
    to = torch.arange(n, device=dev) // f
    c, b = x["count"].to(torch.int64), x["bytes"]
    coarse = [torch.zeros((2, -(-n // f)), dtype=torch.int64, device=dev).index_add_(1, to, v) for v in (c, b)]
    at = ((c != 0).any(0) | (b != 0).any(0)).nonzero().reshape(-1)
    return {"coarse_count": coarse[0], "coarse_bytes": coarse[1], "present": int(at.numel()), "bin": at,
            "count": c[:, at], "bytes": b[:, at]}

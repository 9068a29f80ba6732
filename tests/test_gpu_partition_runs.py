"""The partition's runs: ranges summed directly and split by tile, edges of
tiles and ranges, and inputs whose sample misleads it (runs that overflow, and
an overflow list that overflows), all bit-exact against the oracle."""
import numpy as np
import pytest

import paper_2106_12863_gb300 as sinet
from helpers import assert_hist_equal, to_dev

pytestmark = pytest.mark.gpu

NET = np.array([0x0A000000, 0xC0A80000], np.uint32), np.array([8, 16], np.uint8)


def _records(ts, seed):
    """Records at the given times, 40 % outgoing, 40 % ingoing, 10 % inside, 10 % outside."""
    rng = np.random.default_rng(seed)
    n = len(ts)
    cls = rng.choice(4, n, p=[0.1, 0.4, 0.4, 0.1])
    inside = lambda: np.where(rng.random(n) < 0.5, 0x0A000000 | rng.integers(0, 1 << 24, n), 0xC0A80000 | rng.integers(0, 1 << 16, n))
    outside = lambda: rng.integers(0x80000000, 0xB0000000, n)
    return {"ts": ts.astype(np.uint64), "src": np.where(cls & 1, inside(), outside()).astype(np.uint32),
            "dst": np.where(cls & 2, inside(), outside()).astype(np.uint32),
            "bytes": rng.integers(0, 1 << 32, n, dtype=np.uint32)}


def _check(orc, rec, n_bins, width=1, policy=sinet.EXCLUSIVE, **params):
    table = sinet.PrefixTable(*NET)
    d = to_dev(rec)
    out = sinet.Histogram(n_bins)
    out.count.fill_(-1)  # every bin is stored
    out.bytes.fill_(-1)
    p = sinet.HistParams(7, width, n_bins, policy=policy, strategy="partition", **params)
    sinet.discriminate_histogram(table, d["ts"], d["src"], d["dst"], d["bytes"], p, out)
    ref = orc.discriminate_histogram(*NET, rec, 7, width, n_bins, policy=policy)
    assert_hist_equal(out.to_numpy(), ref, f"bins={n_bins}")
    # and once more on top of it
    p.accumulate = True
    sinet.discriminate_histogram(table, d["ts"], d["src"], d["dst"], d["bytes"], p, out)
    twice = {"count": (2 * ref["count"].astype(np.uint64)).astype(np.uint32), "bytes": 2 * ref["bytes"],
             "stats": 2 * ref["stats"]}
    assert_hist_equal(out.to_numpy(), twice, f"bins={n_bins}, accumulated")
    assert sinet.sinet_device_status() == 0


# one tile; tiles of 2^8 bins; 303, 304 and 305 tiles of 2^13; ranges of four
# tiles; just past the largest histogram summed without a split, and well past it
@pytest.mark.parametrize("n_bins", [1, 256, 257, 77_825, 303 * 8192, 304 * 8192, 304 * 8192 + 1, 8_640_000,
                                    4 * 384 * 8192, 4 * 384 * 8192 + 1, 20_000_001])
def test_histogram_sizes(orc, n_bins):
    rng = np.random.default_rng(n_bins)
    ts = 7 + rng.integers(0, n_bins, 300_007)
    ts[:5] = [0, 6, 7, 6 + n_bins, 7 + n_bins]  # around the window's ends
    _check(orc, _records(ts, 1), n_bins)


@pytest.mark.parametrize("n", [1, 31, 1984, 152 * 1984 + 5, 1_500_000])
@pytest.mark.parametrize("policy", [sinet.PAPER_ALG1, sinet.INCLUSIVE], ids=["paper", "inclusive"])
def test_record_counts_and_policies(orc, n, policy):
    ts = 7 + np.random.default_rng(n).integers(0, 13_000_000 * 3, n)
    _check(orc, _records(ts, 2), 13_000_000, width=3, policy=policy)


@pytest.mark.parametrize("n_bins", [1_000_000, 20_000_000])
@pytest.mark.parametrize("elsewhere", [0.03, 1.0], ids=["list overflows not", "list overflows"])
def test_misleading_sample(orc, n_bins, elsewhere):
    """The sampled chunks (512 records, every n / 65,536-th or more often) are
    spread over the window; a share of the others falls into 2,000 bins for
    which they give no room."""
    n = 3_000_000
    rng = np.random.default_rng(3)
    ts = 7 + rng.integers(0, n_bins, n)
    tiles = next(-(-n_bins // (1 << b)) for b in range(13, 7, -1) if -(-n_bins // (1 << b)) >= 304 or b == 8)
    chunks = -(-n // 512)
    stride = chunks * 512 // max(65_536, min(1 << 20, n // 16, 40 * tiles))
    far = (np.arange(n) // 512 % stride != 0) & (rng.random(n) < elsewhere)
    ts[far] = 7 + n_bins // 2 + rng.integers(0, 2000, int(far.sum()))
    _check(orc, _records(ts, 4), n_bins)


@pytest.mark.parametrize("accumulate", [False, True])
@pytest.mark.parametrize("n_bins", [4_000_000, 12_000_000], ids=["96 MB", "288 MB"])
def test_auto_without_room_for_scratch(orc, free_memory, n_bins, accumulate):
    """AUTO's partition, and the cells that replace it, do not fit: the call runs without scratch."""
    import torch

    table = sinet.PrefixTable(*NET)
    rng = np.random.default_rng(n_bins)
    rec = _records(rng.integers(0, n_bins, 10_000_001), 3)
    d = to_dev(rec)
    p = sinet.HistParams(0, 1, n_bins, accumulate=accumulate)
    assert sinet.auto_strategy(table, len(rec["ts"]), p) == "partition"
    out = sinet.Histogram(n_bins)
    if not accumulate:
        out.count.fill_(-1)
        out.bytes.fill_(-1)
    free_memory(48 << 20)  # the partition takes over 100 MB, the cells 32 bytes a bin
    sinet.discriminate_histogram(table, d["ts"], d["src"], d["dst"], d["bytes"], p, out)
    torch.cuda.synchronize()
    assert_hist_equal(out.to_numpy(), orc.discriminate_histogram(*NET, rec, 0, 1, n_bins))
    assert sinet.sinet_device_status() == 0


def test_streams_accumulating_into_one_histogram():
    """A large call and small ones, on two streams, that add to the same outputs at once lose nothing."""
    import torch

    table = sinet.PrefixTable(np.array([0], np.uint32), np.array([1], np.uint8))
    n, n_bins, calls = 10_200_001, 4_000_000, 40
    g = torch.Generator(device="cuda").manual_seed(1)
    p = sinet.HistParams(0, 1, n_bins, accumulate=True)
    assert [sinet.auto_strategy(table, k, p) for k in (n, 300_000)] == ["partition", "global_atomic"]
    ip = [torch.randint(-(1 << 31), 1 << 31, (n,), dtype=torch.int64, device="cuda", generator=g).to(torch.int32)
          for _ in range(2)]
    rec = (torch.randint(0, n_bins, (n,), dtype=torch.int64, device="cuda", generator=g), *ip,
           torch.randint(0, 1 << 30, (n,), dtype=torch.int32, device="cuda", generator=g))
    parts = [[v[i:i + 300_000] for v in rec] for i in range(0, n - 1, 300_000)]
    last = [v[n - 1:] for v in rec]
    out, once = sinet.Histogram(n_bins), sinet.Histogram(n_bins)
    sinet.discriminate_histogram(table, *rec, sinet.HistParams(0, 1, n_bins, strategy="atomic_noagg"), once)
    torch.cuda.synchronize()
    large, small = torch.cuda.Stream(), torch.cuda.Stream()
    for _ in range(calls):
        sinet.discriminate_histogram(table, *rec, p, out, stream=large)
        for r in (*parts, last):
            sinet.discriminate_histogram(table, *r, p, out, stream=small)
    torch.cuda.synchronize()
    for k in ("count", "bytes", "stats"):
        assert torch.equal(getattr(out, k), getattr(once, k) * (2 * calls)), k
    assert sinet.sinet_device_status() == 0


def test_auto_lines_of_the_partition():
    """From 90 MiB on: 6 M records, 10 M where the outputs are added to."""
    table = sinet.PrefixTable(*NET)
    auto = lambda n, bins, acc: sinet.auto_strategy(table, n, sinet.HistParams(0, 1, bins, accumulate=acc))
    for acc, line in ((False, 6_000_000), (True, 10_000_000)):
        assert [auto(n, 3_932_160, acc) for n in (line - 1, line)] == ["global_atomic", "partition"]
        assert auto(line, 3_932_159, acc) == "global_atomic"

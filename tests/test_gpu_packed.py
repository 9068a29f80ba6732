"""Warp combining through packed cells (count << 40 | byte sum): cells whose
fields overflow into one another must be noticed and the call redone, bit-exact
against the oracle; and warps that stop combining, start again or never do."""
import numpy as np
import pytest

import paper_2106_12863_gb300 as sinet
from helpers import assert_hist_equal, to_dev

pytestmark = pytest.mark.gpu

NET = np.array([0x0A000000], np.uint32), np.array([8], np.uint8)


def _records(ts, nbytes, seed):
    rng = np.random.default_rng(seed)
    n = len(ts)
    cls = rng.choice(4, n, p=[0.1, 0.4, 0.4, 0.1])
    host = lambda inside: np.where(inside, 0x0A000000 | rng.integers(0, 1 << 24, n), rng.integers(1 << 31, 1 << 32, n))
    return {"ts": ts.astype(np.uint64), "src": host(cls & 1).astype(np.uint32), "dst": host(cls & 2).astype(np.uint32),
            "bytes": nbytes.astype(np.uint32)}


def _check(orc, rec, n_bins, **params):
    table = sinet.PrefixTable(*NET)
    d = to_dev(rec, offsets=params.pop("offsets", None))
    out = sinet.Histogram(n_bins)
    out.count.fill_(-1)
    out.bytes.fill_(-1)
    p = sinet.HistParams(0, 1, n_bins, strategy="global_atomic", **params)
    sinet.discriminate_histogram(table, d["ts"], d["src"], d["dst"], d["bytes"], p, out)
    ref = orc.discriminate_histogram(*NET, rec, 0, 1, n_bins, policy=p.policy)
    assert_hist_equal(out.to_numpy(), ref, f"bins={n_bins}")
    assert sinet.sinet_device_status() == 0


# 16 bytes a bin fit 60 MiB (3,932,160 bins); sizes that are and are not multiples of four
@pytest.mark.parametrize("n_bins", [1, 3, 4, 1001, 4097, 100_000, 3_932_160, 3_932_161])
@pytest.mark.parametrize("policy", [sinet.EXCLUSIVE, sinet.INCLUSIVE], ids=["exclusive", "inclusive"])
def test_packed_sizes(orc, n_bins, policy):
    rng = np.random.default_rng(n_bins)
    n = 1_000_003
    ts = rng.integers(0, n_bins + 1, n)  # some past the window
    _check(orc, _records(ts, rng.integers(0, 1 << 32, n), 1), n_bins, policy=policy,
           offsets={"ts": 1, "src": 1, "dst": 1, "bytes": 1})


@pytest.mark.parametrize("hot", [255, 256, 257, 300, 2000])
def test_byte_sums_past_the_field(orc, hot):
    """A bin whose byte sum is just below, at and far past 2^40."""
    n, n_bins = 1_000_003, 10_000
    rng = np.random.default_rng(hot)
    ts, nbytes = rng.integers(0, n_bins, n), rng.integers(0, 1000, n)
    rec = _records(ts, nbytes, 2)
    out = np.flatnonzero((rec["src"] >> 24 == 10) & (rec["dst"] >> 24 != 10))[:hot]
    rec["ts"][out], rec["bytes"][out] = 1234, 0xFFFFFFFF
    _check(orc, rec, n_bins)


def test_counts_past_the_field(orc):
    """More than 2^24 records of no bytes in one bin: the count field wraps."""
    n = (1 << 24) + 5
    rec = {"ts": np.full(n, 3, np.uint64), "src": np.full(n, 0x0A000001, np.uint32),
           "dst": np.full(n, 0xC0000001, np.uint32), "bytes": np.zeros(n, np.uint32)}
    _check(orc, rec, 5000)


@pytest.mark.parametrize("order", ["uniform then hot", "hot then uniform", "alternating"])
def test_warps_change_their_mind(orc, order):
    n, n_bins = 2_000_003, 50_000
    rng = np.random.default_rng(5)
    hot = {"uniform then hot": np.arange(n) > n // 2, "hot then uniform": np.arange(n) < n // 2,
           "alternating": np.arange(n) // 100_000 % 2 == 0}[order]
    ts = np.where(hot, rng.integers(0, 8, n), rng.integers(0, n_bins, n))
    _check(orc, _records(ts, rng.integers(0, 1 << 20, n), 6), n_bins)


def test_batch_slices(orc):
    """Slices with packed cells in one batch, one of which overflows a cell; replayed, since the cells are kept."""
    import torch

    table = sinet.PrefixTable(*NET)
    slices, want = [], []
    for i, (strategy, n_bins, big) in enumerate([("atomic_noagg", 10_001, False), ("atomic_noagg", 10_000, True),
                                                 ("global_atomic", 70_000, False), ("global_atomic", 20_000, True),
                                                 ("atomic_noagg", 140_000, False)]):
        rng = np.random.default_rng(i)
        rec = _records(rng.integers(0, n_bins + 1, 60_000), rng.integers(0, 1 << 30, 60_000), i)
        if big:
            rec["ts"][:600], rec["bytes"][:600] = 77, 0xFFFFFFFF
        d = to_dev(rec, offsets={k: i for k in ("ts", "src", "dst", "bytes")})
        out = sinet.Histogram(n_bins)
        slices.append((table, d["ts"], d["src"], d["dst"], d["bytes"],
                       sinet.HistParams(0, 1, n_bins, strategy=strategy), out))
        want.append(orc.discriminate_histogram(*NET, rec, 0, 1, n_bins))
    batch = sinet.Batch(slices)
    for _ in range(3):
        for s in slices:
            s[-1].count.fill_(-1)
            s[-1].bytes.fill_(-1)
        batch.run()
        torch.cuda.synchronize()
        for i, (s, ref) in enumerate(zip(slices, want)):
            assert_hist_equal(s[-1].to_numpy(), ref, f"slice {i}")
    assert sinet.sinet_device_status() == 0
    batch.close()


@pytest.mark.parametrize("strategy", ["global_atomic", "partition", "sort_reduce", "owner"])
def test_two_threads_with_tables_of_two_sizes(strategy):
    """Calls from two host threads whose tables need different amounts of shared memory."""
    import threading

    import torch
    from test_host_plans import prefixes

    n, n_bins, errors = 1_000_003, 10_000, []
    g = torch.Generator(device="cuda").manual_seed(1)
    ts = torch.randint(0, n_bins, (n,), dtype=torch.int64, device="cuda", generator=g)
    ip = [torch.randint(-(1 << 31), 1 << 31, (n,), dtype=torch.int64, device="cuda", generator=g).to(torch.int32)
          for _ in range(2)]
    by = torch.randint(0, 1500, (n,), dtype=torch.int32, device="cuda", generator=g)
    p = sinet.HistParams(0, 1, n_bins, strategy=strategy)
    tables = [sinet.PrefixTable(*prefixes(k, 16, 24, 4)) for k in (6000, 9000)]  # one lookup form
    torch.cuda.synchronize()

    def work(table):
        try:
            with torch.cuda.stream(torch.cuda.Stream()):
                out = sinet.Histogram(n_bins)
                for _ in range(400):
                    sinet.discriminate_histogram(table, ts, *ip, by, p, out)
                torch.cuda.current_stream().synchronize()
                assert int(out.stats[:4].sum()) == n
        except Exception as e:  # noqa: BLE001 - reported by the test's thread
            errors.append(e)

    threads = [threading.Thread(target=work, args=(t,)) for t in tables]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors, errors
    assert sinet.sinet_device_status() == 0


@pytest.mark.parametrize("n,n_bins", [(953_520, 3_932_160), (953_519, 3_932_160), (1_949_999, 3_600_001),
                                      (275_011, 600_002), (300_000, 600_000), (299_999, 600_000), (300_001, 333_333)])
def test_packed_at_the_edges_of_the_rule(orc, n, n_bins):
    """Calls on both sides of the lines in records and bins from which packed cells are taken."""
    rng = np.random.default_rng(n)
    _check(orc, _records(rng.integers(0, n_bins + 1, n), rng.integers(0, 1 << 32, n), 1), n_bins, policy=sinet.INCLUSIVE)

"""Packed cells in a batch large enough for them: on both sides of the line that
sums the packed slices' records, with a cell that overflows its byte sum; replayed."""
from __future__ import annotations

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover - collected on CPU too
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_2106_12863_gb300 as sinet  # noqa: E402


@pytest.mark.parametrize("total", [7_999_999, 8_000_000])
def test_batches_around_the_line(total):
    table = sinet.PrefixTable(np.array([0], np.uint32), np.array([1], np.uint8))
    g = torch.Generator(device="cuda").manual_seed(total)
    slices, want = [], []
    for n, n_bins, strategy in ((3_000_001, 1_000_003, "global_atomic"), (total - 3_000_001, 70_001, "atomic_noagg")):
        ts = torch.randint(0, n_bins, (n,), dtype=torch.int64, device="cuda", generator=g)
        src = torch.randint(1, 1 << 31, (n,), dtype=torch.int64, device="cuda", generator=g).to(torch.int32)
        dst = torch.full((n,), -1, dtype=torch.int32, device="cuda")  # outside
        by = torch.randint(0, 1 << 30, (n,), dtype=torch.int32, device="cuda", generator=g)
        ts[:2000], by[:2000] = 77, -1  # 2,000 times 2^32 - 1 bytes in one bin: past 2^40
        out = sinet.Histogram(n_bins)
        slices.append((table, ts, src, dst, by, sinet.HistParams(0, 1, n_bins, strategy=strategy), out))
        want.append((torch.bincount(ts, minlength=n_bins),
                     torch.zeros(n_bins, dtype=torch.int64, device="cuda").index_add_(0, ts, by.to(torch.int64) & 0xFFFFFFFF)))
    batch = sinet.Batch(slices)
    for _ in range(2):
        for s in slices:
            s[-1].count.fill_(-1)
            s[-1].bytes.fill_(-1)
        batch.run()
        torch.cuda.synchronize()
        for s, (c, b) in zip(slices, want):
            got = s[-1].to_numpy()
            # inside to outside is the outgoing direction; the other one stays empty
            d = 0 if got["count"][0].any() else 1
            assert np.array_equal(got["count"][d], c.cpu().numpy().astype(got["count"].dtype))
            assert np.array_equal(got["bytes"][d], b.cpu().numpy().astype(got["bytes"].dtype))
            assert not got["count"][1 - d].any() and not got["bytes"][1 - d].any()
    batch.close()


@pytest.mark.parametrize("n_bins", [2_000_003, 300_001], ids=["shared area", "areas of their own"])
def test_tuning_a_slice_that_overflows_a_cell(n_bins):
    """The tuner times copies of a slice whose cells overflow; no wait of theirs runs out."""
    table = sinet.PrefixTable(np.array([0], np.uint32), np.array([1], np.uint8))
    n = 1_000_003
    g = torch.Generator(device="cuda").manual_seed(n_bins)
    # ten copies of 40 bytes a bin: beyond the tuner's 512 MB with the larger histogram
    ts = torch.randint(0, n_bins, (n,), dtype=torch.int64, device="cuda", generator=g)
    src = torch.randint(1, 1 << 31, (n,), dtype=torch.int64, device="cuda", generator=g).to(torch.int32)
    dst = torch.full((n,), -1, dtype=torch.int32, device="cuda")  # outside
    by = torch.randint(0, 1 << 30, (n,), dtype=torch.int32, device="cuda", generator=g)
    ts[:2000], by[:2000] = 77, -1
    out = sinet.Histogram(n_bins)
    # a width of 7 ms, which no other test of this size has: a class not tuned before
    batch = sinet.Batch([(table, ts * 7, src, dst, by, sinet.HistParams(0, 7, n_bins), out)], autotune=True)
    batch.run()
    torch.cuda.synchronize()
    assert sinet.sinet_device_status() == 0
    assert torch.equal(out.count[0].long() + out.count[1], torch.bincount(ts, minlength=n_bins))
    batch.close()


def test_cells_give_way_to_the_plain_path(free_memory):
    """Memory for the plain path's scratch or for packed cells, not for both: the cells are left out."""
    table = sinet.PrefixTable(np.array([0], np.uint32), np.array([1], np.uint8))
    n, n_bins = 20_000_003, 20_000_000
    g = torch.Generator(device="cuda").manual_seed(9)
    ts = torch.randint(0, n_bins, (n,), dtype=torch.int64, device="cuda", generator=g)
    src = torch.randint(1, 1 << 31, (n,), dtype=torch.int64, device="cuda", generator=g).to(torch.int32)
    dst = torch.full((n,), -1, dtype=torch.int32, device="cuda")  # outside
    by = torch.randint(0, 1 << 30, (n,), dtype=torch.int32, device="cuda", generator=g)
    outs = [sinet.Histogram(n_bins) for _ in range(2)]
    # 320 MB of cells, 330 MB of scratch
    free_memory(480 << 20)
    batch = sinet.Batch([(table, ts, src, dst, by, sinet.HistParams(0, 1, n_bins, strategy=s), o)
                         for s, o in zip(("global_atomic", "sort_reduce"), outs)])
    batch.run()
    torch.cuda.synchronize()
    assert sinet.sinet_device_status() == 0
    for k in ("count", "bytes", "stats"):
        assert torch.equal(getattr(outs[0], k), getattr(outs[1], k)), k
    assert int(outs[0].stats[:4].sum()) == n
    batch.close()


def _uniform(n, n_bins, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    ts = torch.randint(0, n_bins, (n,), dtype=torch.int64, device="cuda", generator=g)
    ip = [torch.randint(-(1 << 31), 1 << 31, (n,), dtype=torch.int64, device="cuda", generator=g).to(torch.int32)
          for _ in range(2)]
    return ts, *ip, torch.randint(0, 1 << 30, (n,), dtype=torch.int32, device="cuda", generator=g)


def test_slices_that_fill_one_histogram():
    """Slices whose outputs are the same rows, overlap in part, or are added to by another slice."""
    table = sinet.PrefixTable(np.array([0], np.uint32), np.array([1], np.uint8))
    n, n_bins = 3_000_001, 100_000
    recs = [_uniform(n, n_bins, i) for i in range(5)]
    apart = [sinet.Histogram(n_bins) for _ in recs]
    for r, o in zip(recs, apart):
        sinet.discriminate_histogram(table, *r, sinet.HistParams(0, 1, n_bins, strategy="atomic_noagg"), o)
    one, alone = sinet.Histogram(n_bins), sinet.Histogram(n_bins)
    day = sinet.Histogram(150_000)

    class Part:  # bins [first, first + n_bins) of the day
        def __init__(self, first):
            self.h = sinet.Histogram(1)
            self.h.count, self.h.bytes = day.count[:, first:first + n_bins], day.bytes[:, first:first + n_bins]

        def c(self):
            return self.h.c()

    parts = [Part(0), Part(50_000)]
    p = sinet.HistParams(0, 1, n_bins, strategy="atomic_noagg")
    add = sinet.HistParams(0, 1, n_bins, strategy="global_atomic", accumulate=True)
    batch = sinet.Batch([(table, *recs[0], p, one), (table, *recs[1], add, one), (table, *recs[2], p, parts[0]),
                         (table, *recs[3], p, parts[1]), (table, *recs[4], p, alone)])
    for _ in range(2):
        batch.run()
    torch.cuda.synchronize()
    for k in ("count", "bytes"):
        a = [getattr(h, k) for h in apart]
        assert torch.equal(getattr(one, k), a[0] + a[1]), k
        want = torch.zeros_like(getattr(day, k))
        want[:, :n_bins] += a[2]
        want[:, 50_000:] += a[3]
        assert torch.equal(getattr(day, k), want), k
        assert torch.equal(getattr(alone, k), a[4]), k
    batch.close()


@pytest.mark.parametrize("strategy,n,n_bins", [("global_atomic", 1_000_003, 100_000), ("auto", 1_000_003, 100_000),
                                               ("auto", 6_000_001, 4_000_000)])
def test_both_directions_in_one_row(strategy, n, n_bins):
    table = sinet.PrefixTable(np.array([0], np.uint32), np.array([1], np.uint8))
    rec = _uniform(n, n_bins, 7)
    two, one = sinet.Histogram(n_bins), sinet.Histogram(n_bins)
    sinet.discriminate_histogram(table, *rec, sinet.HistParams(0, 1, n_bins, strategy="atomic_noagg"), two)
    count, nbytes = one.count[0], one.bytes[0]
    one.count, one.bytes = [count, count], [nbytes, nbytes]
    sinet.discriminate_histogram(table, *rec, sinet.HistParams(0, 1, n_bins, strategy=strategy), one)
    assert torch.equal(count, two.count.sum(0, dtype=torch.int32))
    assert torch.equal(nbytes, two.bytes.sum(0))


def test_packed_slices_beside_others(orc):
    """Both-direction policies, unaligned streams, records outside the window, several cells that
    overflow, widths, and tile, accumulating and plain-path neighbours in one batch; replayed."""
    from helpers import assert_hist_equal, to_dev

    net, ln = np.array([10 << 24], np.uint32), np.array([8], np.uint8)
    table = sinet.PrefixTable(net, ln)
    kinds = [  # records, bins, width, strategy, policy, overflowing cells, accumulate
        (2_500_003, 300_001, 1, "atomic_noagg", sinet.INCLUSIVE, 3, False),
        (2_000_001, 70_000, 10, "global_atomic", sinet.INCLUSIVE, 1, False),
        (1_500_002, 140_003, 7, "atomic_noagg", sinet.PAPER_ALG1, 2, False),
        (2_100_000, 1_000_000, 1, "global_atomic", sinet.EXCLUSIVE, 0, False),
        (60_000, 10_001, 1, "atomic_noagg", sinet.EXCLUSIVE, 1, False),
        (100_001, 3_000, 1, "smem_full", sinet.INCLUSIVE, 1, False),
        (100_002, 90_000, 1, "atomic_noagg", sinet.EXCLUSIVE, 1, True),
        (100_003, 80_000, 1, "sort_reduce", sinet.INCLUSIVE, 1, False),
    ]
    slices, want = [], []
    for i, (n, n_bins, width, strategy, policy, hot, accumulate) in enumerate(kinds):
        rng = np.random.default_rng(i)
        cls = rng.choice(4, n, p=[0.1, 0.4, 0.4, 0.1])
        host = lambda inside: np.where(inside, 0x0A000000 | rng.integers(0, 1 << 24, n), rng.integers(1 << 31, 1 << 32, n))
        span = n_bins * width
        rec = {"ts": 1000 + rng.integers(-span // 20, span + span // 20, n).clip(-1000), "src": host(cls & 1),
               "dst": host(cls & 2), "bytes": rng.integers(0, 1 << 30, n)}
        for k in range(hot):
            at = slice(700 * k, 700 * (k + 1))
            rec["ts"][at], rec["bytes"][at] = 1000 + (span // 3) * k, 0xFFFFFFFF
        rec = {k: v.astype(np.uint64 if k == "ts" else np.uint32) for k, v in rec.items()}
        d = to_dev(rec, offsets={k: (i + j) % 4 for j, k in enumerate(rec)})
        out = sinet.Histogram(n_bins)
        slices.append((table, d["ts"], d["src"], d["dst"], d["bytes"],
                       sinet.HistParams(1000, width, n_bins, policy=policy, strategy=strategy, accumulate=accumulate), out))
        want.append(orc.discriminate_histogram(net, ln, rec, 1000, width, n_bins, policy=policy))
    batch = sinet.Batch(slices)
    for run in range(1, 4):
        for s, kind in zip(slices, kinds):
            if not kind[-1]:
                s[-1].count.fill_(-1)
                s[-1].bytes.fill_(-1)
        batch.run()
        torch.cuda.synchronize()
        for i, (s, ref, kind) in enumerate(zip(slices, want, kinds)):
            if kind[-1]:
                ref = {k: v * np.array(run, v.dtype) for k, v in ref.items()}
            assert_hist_equal(s[-1].to_numpy(), ref, f"slice {i}, run {run}")
    assert sinet.sinet_device_status() == 0
    batch.close()

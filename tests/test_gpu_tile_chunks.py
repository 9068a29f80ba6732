"""Tile chunks longer than three records a tile bin: many records per bin, on both
sides of the limits, against a histogram counted by torch."""
from __future__ import annotations

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover - collected on CPU too
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_2106_12863_gb300 as sinet  # noqa: E402


@pytest.mark.parametrize("n,n_bins", [(40_000_003, 833_333), (40_000_003, 200_001), (40_000_003, 78_200), (40_000_003, 78_000)])
def test_long_chunks(n, n_bins):
    table = sinet.PrefixTable(np.array([0], np.uint32), np.array([1], np.uint8))
    g = torch.Generator(device="cuda").manual_seed(n_bins)
    ts = torch.arange(n, dtype=torch.int64, device="cuda") * n_bins // n
    ts = (ts + torch.randint(-500, 501, (n,), device="cuda", generator=g)).clamp_(0, n_bins - 1)
    src = torch.randint(1, 1 << 31, (n,), dtype=torch.int64, device="cuda", generator=g).to(torch.int32)
    dst = torch.full((n,), -1, dtype=torch.int32, device="cuda")  # outside
    by = torch.randint(-(1 << 31), 1 << 31, (n,), dtype=torch.int64, device="cuda", generator=g).to(torch.int32)
    out = sinet.Histogram(n_bins)
    p = sinet.HistParams(0, 1, n_bins, hints=sinet.HINT_TIME_SORTED, strategy="priv_tile")
    sinet.discriminate_histogram(table, ts, src, dst, by, p, out)
    got = out.to_numpy()
    d = 0 if got["count"][0].any() else 1  # the one direction that inside to outside takes
    c = torch.bincount(ts, minlength=n_bins)
    b = torch.zeros(n_bins, dtype=torch.int64, device="cuda").index_add_(0, ts, by.to(torch.int64) & 0xFFFFFFFF)
    assert np.array_equal(got["count"][d], c.cpu().numpy().astype(np.uint32))
    assert np.array_equal(got["bytes"][d], b.cpu().numpy().astype(np.uint64))
    assert not got["count"][1 - d].any() and not got["bytes"][1 - d].any()
    table.close()


def test_whole_histogram_short_chunks(orc):
    """A whole-histogram tile that leaves one CTA an SM, each with several chunks of one
    quad a thread: every chunk's bins flushed, though consecutive chunks lie far apart."""
    from helpers import assert_hist_equal, to_dev
    from test_host_plans import prefixes

    net, ln = prefixes(8000, 16, 24, 4)
    n, n_bins = 600_001, 5000
    rng = np.random.default_rng(1)
    at = np.arange(n) // 2048 // 152 % 2  # a CTA's chunks in turn: the first bins, the last ones
    rec = {"ts": (at * 4990 + rng.integers(0, 10, n)).astype(np.uint64), "src": rng.choice(net, n),
           "dst": rng.integers(1 << 31, 1 << 32, n).astype(np.uint32),
           "bytes": rng.integers(0, 1 << 32, n).astype(np.uint32)}
    want = orc.discriminate_histogram(net, ln, rec, 0, 1, n_bins)
    table, d = sinet.PrefixTable(net, ln), to_dev(rec)
    for i in range(20):
        out = sinet.Histogram(n_bins)
        sinet.discriminate_histogram(table, d["ts"], d["src"], d["dst"], d["bytes"],
                                     sinet.HistParams(0, 1, n_bins, strategy="smem_full"), out)
        assert_hist_equal(out.to_numpy(), want, f"call {i}")
    table.close()

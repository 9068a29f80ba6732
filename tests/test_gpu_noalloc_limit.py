"""The allocation-free call's largest accepted input.

Its scratch is a fixed 32 MiB array, so the layout of the plain path's scratch
decides which inputs it takes. The limit is part of the interface: the largest
input that fits is accepted and gives the allocating call's result, one more
record is refused before anything is launched.
"""
from __future__ import annotations

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover - collected on CPU too
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_2106_12863_gb300 as sinet  # noqa: E402


def _scratch(n, dirs):
    """Bytes of the plain path's scratch: counters, digit counts, look-back words
    of the emit tiles (4,096 records), 8 bytes a digit and sort tile (4,096
    keys), two key and two value arrays; each part rounded up to 256 bytes."""
    al = lambda x: (x + 255) & ~255
    m = n * dirs
    emit = (n // 4 + 2 + 1023) // 1024
    tiles = max((m + 4095) // 4096, 1)
    return al(128) + al(4096) + al(8 * (emit + 1)) + al(2048 * tiles) + 4 * al(4 * m + 4)


@pytest.mark.parametrize("policy,dirs", [("EXCLUSIVE", 1), ("INCLUSIVE", 2)])
def test_the_largest_input_stays_the_largest(policy, dirs):
    lo, hi = 1, 4_000_000
    while lo < hi:
        mid = (lo + hi + 1) // 2
        lo, hi = (mid, hi) if _scratch(mid, dirs) <= 32 << 20 else (lo, mid - 1)
    n = lo
    table = sinet.PrefixTable(np.array([10 << 24], np.uint32), np.array([8], np.uint8))
    params = sinet.HistParams(0, 1, 1000, policy=getattr(sinet, policy))
    g = torch.Generator(device="cuda").manual_seed(3)
    ts = torch.randint(0, 1000, (n + 1,), dtype=torch.int64, device="cuda", generator=g)
    ip = [torch.randint(9 << 24, 12 << 24, (n + 1,), dtype=torch.int32, device="cuda", generator=g)
          for _ in range(2)]
    by = torch.randint(40, 1500, (n + 1,), dtype=torch.int32, device="cuda", generator=g)

    def run(fn, m):
        out = sinet.Histogram(params.n_bins)
        fn(table.handle, ts[:m], ip[0][:m], ip[1][:m], by[:m], m, params.c(), out.c())
        torch.cuda.synchronize()
        return out.to_numpy()

    got = run(sinet.sinet_discriminate_histogram_noalloc, n)
    want = run(sinet.sinet_discriminate_histogram, n)
    for k in want:
        assert np.array_equal(got[k], want[k]), k
    with pytest.raises(sinet.SinetError, match="BUDGET"):
        run(sinet.sinet_discriminate_histogram_noalloc, n + 1)
    table.close()


@pytest.mark.parametrize("policy,dirs", [("EXCLUSIVE", 1), ("INCLUSIVE", 2)])
@pytest.mark.parametrize("tiles", [1, 2, 511, 512, 513, 1500])
@pytest.mark.parametrize("over", [-1, 0, 1])
def test_plain_path_at_the_edges_of_tiles(tiles, over, policy, dirs):
    """One kernel a radix pass up to 512 sort tiles of 4,096 pairs, three beyond: equal to plain reductions."""
    n, n_bins = tiles * 4096 // dirs + over, 70_001
    table = sinet.PrefixTable(np.array([0], np.uint32), np.array([1], np.uint8))
    g = torch.Generator(device="cuda").manual_seed(tiles)
    ts = torch.randint(0, n_bins + 5, (n,), dtype=torch.int64, device="cuda", generator=g)
    # every record routed: inside to outside, or (both directions) inside to inside
    src = torch.randint(1, 1 << 31, (n,), dtype=torch.int64, device="cuda", generator=g).to(torch.int32)
    dst = src.clone() if dirs == 2 else torch.full((n,), -1, dtype=torch.int32, device="cuda")
    by = torch.randint(-(1 << 31), 1 << 31, (n,), dtype=torch.int64, device="cuda", generator=g).to(torch.int32)
    outs = []
    for strategy in ("sort_reduce", "atomic_noagg"):
        outs.append(sinet.Histogram(n_bins))
        p = sinet.HistParams(0, 1, n_bins, policy=getattr(sinet, policy), strategy=strategy)
        sinet.discriminate_histogram(table, ts, src, dst, by, p, outs[-1])
    for k in ("count", "bytes", "stats"):
        assert torch.equal(getattr(outs[0], k), getattr(outs[1], k)), k
    assert sinet.sinet_device_status() == 0
    table.close()

"""Slices that share a prefix list and stage it in different forms: a list whose
larger form leaves no room for the longer window's whole-histogram tile, in one
batch and in one server. Every CTA goes from one form to the other many times."""
from __future__ import annotations

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover - collected on CPU too
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_2106_12863_gb300 as sinet  # noqa: E402
from helpers import assert_hist_equal, to_dev  # noqa: E402
from test_host_plans import prefixes  # noqa: E402

NET = prefixes(2500, 16, 24, 1)  # see test_host_plans.py for the two forms
KINDS = [(3600, "smem_full"), (5400, "smem_full"), (5400, "global_atomic"), (3600, "auto"), (5400, "auto")]


def _records(n, seed):
    rng = np.random.default_rng(seed)
    net, ln = NET
    k = rng.integers(0, len(net), (2, n))
    host = rng.integers(0, 1 << 32, (2, n)) & ((1 << (32 - ln[k].astype(np.int64))) - 1)
    inside = rng.random((2, n)) < 0.5
    ip = np.where(inside, net[k].astype(np.int64) | host, rng.integers(0, 1 << 32, (2, n))).astype(np.uint32)
    return {"ts": rng.integers(0, 5_500_000, n).astype(np.uint64), "src": ip[0], "dst": ip[1],
            "bytes": rng.integers(0, 1 << 32, n).astype(np.uint32)}


@pytest.mark.parametrize("kinds", [KINDS[:2], KINDS], ids=["tiles", "tiles and reductions"])
def test_batch_alternating_forms(orc, kinds):
    table = sinet.PrefixTable(*NET)
    sets = [_records(2500, 10 + i) for i in range(len(kinds))]
    devs = [to_dev(r) for r in sets]
    want = [orc.discriminate_histogram(*NET, r, 0, 1000, b) for r, (b, _) in zip(sets, kinds)]
    slices = []
    for i in range(1200):  # an item each, four a CTA
        d, (bins, strategy) = devs[i % len(kinds)], kinds[i % len(kinds)]
        slices.append((table, d["ts"], d["src"], d["dst"], d["bytes"],
                       sinet.HistParams(0, 1000, bins, strategy=strategy), sinet.Histogram(bins, zero=False)))
    batch = sinet.Batch(slices)
    for _ in range(2):
        batch.run()
    torch.cuda.synchronize()
    for i, s in enumerate(slices):
        assert_hist_equal(s[-1].to_numpy(), want[i % len(kinds)], f"slice {i}")
    assert sinet.sinet_device_status() == 0
    batch.close()


def test_server_tenants_sharing_a_list(orc):
    table = sinet.PrefixTable(*NET)
    params = [sinet.HistParams(0, 1000, bins, accumulate=True) for bins in (3600, 5400)]
    sets = [_records(2500, 20 + i) for i in range(4)]
    server = sinet.Server([(table, p) for p in params], budget_bytes=64 << 20, max_requests_per_launch=512,
                          max_queued=2048)
    tickets = [server.submit(i % 2, *(sets[i // 2 % 4][k] for k in ("ts", "src", "dst", "bytes")))
               for i in range(1024)]
    for t in tickets:
        server.wait(t)
    for i, p in enumerate(params):
        want = orc.empty_hist(p.n_bins)
        for r in sets:
            orc.discriminate_histogram(*NET, r, 0, 1000, p.n_bins, into=want)
        got = server.export(i)
        with np.errstate(over="ignore"):
            for k in ("stats", "count", "bytes"):
                assert np.array_equal(got[k], want[k] * np.array(128, want[k].dtype)), f"tenant {i} {k}"
    assert sinet.sinet_device_status() == 0
    server.close()

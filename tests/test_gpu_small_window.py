"""Windows whose span is below 2^32 ms divide in 32 bits: every bin against
Python's integer division, at spans just below the limit, on it and past it."""
import numpy as np
import pytest

import paper_2106_12863_gb300 as sinet

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("t0", [0, 12_345_678_901])
@pytest.mark.parametrize("w", [1, 2, 3, 7, 10, 1000, 3600, 65_535, 65_536, 65_537, 1_000_003, (1 << 31) - 1, 1 << 31,
                               (1 << 32) - 1, 1 << 32])
def test_bins_of_small_windows(w, t0):
    import torch

    rng = np.random.default_rng(w)
    for n_bins in {max(1, min((1 << 31) - 1, ((1 << 32) - 1) // w + k)) for k in (-1, 0, 1)} | {1, 3}:
        span = n_bins * w
        rel = np.concatenate([rng.integers(0, span, 4000, dtype=np.uint64),
                              np.arange(0, min(span, 50), dtype=np.uint64), span - 1 - np.arange(min(span, 50)).astype(np.uint64),
                              np.uint64(w) * rng.integers(0, n_bins, 500, dtype=np.uint64), [span, span + 1]]).astype(np.uint64)
        rel = np.unique(np.concatenate([rel, rel + np.uint64(1), np.maximum(rel, 1) - np.uint64(1)]))
        ts = rel + np.uint64(t0)
        got = sinet.bin_index(torch.from_numpy(ts.view(np.int64)).cuda(), t0, w, n_bins).cpu().numpy().view(np.uint32)
        want = np.where(rel < span, rel // np.uint64(w), 0xFFFFFFFF).astype(np.uint32)
        assert np.array_equal(got, want), (w, n_bins)

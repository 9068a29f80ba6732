"""Roll-up and sparse form at the edges of their tiles (4,096 bins a compaction
tile, 256 a roll-up segment, 32 a row), against numpy on the same histogram."""
import numpy as np
import pytest

import paper_2106_12863_gb300 as sinet

pytestmark = pytest.mark.gpu


def _hist(n_bins, filled, seed):
    """A histogram with `filled` of its bins non-empty (some with one direction or bytes only), sums up to 2^64 - 1."""
    rng = np.random.default_rng(seed)
    count = rng.integers(0, 1 << 32, (2, n_bins), dtype=np.uint32)
    nbytes = rng.integers(0, 1 << 64, (2, n_bins), dtype=np.uint64, endpoint=False)
    kind = rng.integers(0, 4, n_bins)
    count[:, kind == 0] = 0
    nbytes[1, kind == 1] = 0
    count[1, kind == 2] = 0
    empty = rng.random(n_bins) >= filled
    count[:, empty] = 0
    nbytes[:, empty] = 0
    return count, nbytes


def _device(count, nbytes):
    import torch

    out = sinet.Histogram(count.shape[1])
    out.count.copy_(torch.from_numpy(count.view(np.int32)))
    out.bytes.copy_(torch.from_numpy(nbytes.view(np.int64)))
    return out


@pytest.mark.parametrize("factor", [1, 2, 31, 32, 33, 256, 1000, 1 << 40])
@pytest.mark.parametrize("n_bins", [1, 31, 33, 255, 256, 257, 2049, 100_003])
def test_rollup_edges(n_bins, factor):
    count, nbytes = _hist(n_bins, 0.7, n_bins + factor)
    edges = np.arange(0, n_bins, min(factor, n_bins))
    got = sinet.rollup(_device(count, nbytes), factor).to_numpy()
    assert np.array_equal(got["count"], np.add.reduceat(count, edges, axis=1, dtype=np.uint32))
    assert np.array_equal(got["bytes"], np.add.reduceat(nbytes, edges, axis=1, dtype=np.uint64))


@pytest.mark.parametrize("filled", [0.0, 0.01, 0.5, 1.0])
@pytest.mark.parametrize("n_bins", [1, 32, 2047, 4095, 4096, 4097, 8193, 1_000_003])
def test_sparse_edges(n_bins, filled):
    count, nbytes = _hist(n_bins, filled, n_bins)
    at = np.flatnonzero((count != 0).any(0) | (nbytes != 0).any(0))
    h = _device(count, nbytes)
    for cap in (None, len(at) // 2):
        got = sinet.sparse(h, cap)
        k = len(at) if cap is None else cap
        assert got["n"] == len(at)
        assert np.array_equal(got["bin"].cpu().numpy(), at[:k])
        assert np.array_equal(got["count"].cpu().numpy().view(np.uint32), count[:, at[:k]])
        assert np.array_equal(got["bytes"].cpu().numpy().view(np.uint64), nbytes[:, at[:k]])

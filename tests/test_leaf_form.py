"""The leaf form of a prefix table: the compiled image replayed on the host and
the kernels that stage it, against the oracle's loop over every entry."""
import numpy as np
import pytest

import paper_2106_12863_gb300 as sinet


def _spread(n, lo, hi, seed):
    """n prefixes of lengths lo..hi, uniform within 0.0.0.0/1."""
    rng = np.random.default_rng(seed)
    ln = rng.integers(lo, hi + 1, n)
    net = rng.integers(0, 1 << 31, n) & (0xFFFFFFFF << (32 - ln))
    return net.astype(np.uint32), ln.astype(np.uint8)


def _hosts(step):
    """Twenty /32 hosts `step` apart in one bucket."""
    return (0x0A000000 + step * np.arange(20)).astype(np.uint32), np.full(20, 32, np.uint8)


EMPTY = np.zeros(0, np.uint32), np.zeros(0, np.uint8)
EDGES = np.array([0, 0x80000000, 0xFFFFFFFF, 0x7FFFFFFF], np.uint32), np.array([8, 1, 32, 32], np.uint8)
# name: (table, words a leaf; 0 = no leaf form, the toggle form is staged)
TABLES = {
    "empty": (EMPTY, 2),
    "everything": ((np.zeros(1, np.uint32), np.zeros(1, np.uint8)), 2),
    "ends of the address range": (EDGES, 2),
    "one host": ((np.array([0xC0A80105], np.uint32), np.array([32], np.uint8)), 2),
    "every other host": (_hosts(2), 0),
    "long and short": (_spread(2000, 8, 32, 1), 2),
    "2,000 of /16-/24": (_spread(2000, 16, 24, 2), 4),
    "8,000 of /16-/24": (_spread(8000, 16, 24, 3), 0),
}


def _addresses(net, ln, seed, extra=2000):
    """Both ends of every prefix, their neighbours, and random addresses."""
    lo = net.astype(np.int64) & -(1 << (32 - ln.astype(np.int64)))
    hi = lo + (1 << (32 - ln.astype(np.int64))) - 1
    rng = np.random.default_rng(seed)
    a = np.concatenate([lo, lo - 1, hi, hi + 1, rng.integers(0, 1 << 32, extra), [0, (1 << 32) - 1]])
    return (a & 0xFFFFFFFF).astype(np.uint32)


def _leaf_lookup(img, addrs):
    off_leaves, off_desc, bits, words = (int(v) for v in img[-16:].view(np.uint32))
    desc = img[off_desc:off_desc + (4 << bits)].view(np.uint32)
    leaves = img[off_leaves:off_desc].view(np.uint32)
    off = addrs & np.uint32((1 << (32 - bits)) - 1)
    d = desc[addrs >> np.uint32(32 - bits)]
    at = (d >> np.uint32(8)).astype(np.int64) // 4 + (off >> (d & np.uint32(31))).astype(np.int64) * words
    assert at.max() + words <= len(leaves)  # every leaf read stays in the staged region
    x = np.zeros(len(addrs), np.uint32)
    for k in range(words):
        x ^= leaves[at + k] - off
    return (x >> np.uint32(31)).astype(np.uint8)


def _want(orc, net, ln, addrs):
    return (orc.classify(net, ln, addrs, np.zeros_like(addrs)) & 1).astype(np.uint8)


@pytest.mark.parametrize("name", TABLES)
def test_leaf_form_equals_oracle(orc, name):
    (net, ln), words = TABLES[name]
    img, lay = sinet.sinet_prefix_table_image(net, ln)
    assert int(img[-4:].view(np.uint32)[0]) == words
    if words:
        a = _addresses(net, ln, 5)
        got = _leaf_lookup(img, a)
        want = _want(orc, net, ln, a) if len(net) else np.zeros(len(a), np.uint8)
        assert np.array_equal(got, want)


def test_leaf_form_of_crowded_lists(orc):
    """Nested, adjacent and duplicate entries crowded into a few buckets."""
    rng = np.random.default_rng(11)
    for k in range(60):
        n = int(rng.integers(1, 120))
        ln = rng.integers(8, 33, n).astype(np.uint8)
        net = (0x0A000000 + rng.integers(0, 1 << int(rng.integers(4, 24)), n)).astype(np.uint32)
        img, lay = sinet.sinet_prefix_table_image(net, ln)
        if int(img[-4:].view(np.uint32)[0]) == 0:
            continue
        a = _addresses(net, ln, k, extra=200)
        assert np.array_equal(_leaf_lookup(img, a), _want(orc, net, ln, a))


@pytest.mark.gpu
@pytest.mark.parametrize("at", [(0, 0), (0, 1), (1, 0), (3, 2), (2, 3)], ids=lambda v: f"addr{v[0]}class{v[1]}")
@pytest.mark.parametrize("name", ["empty", "every other host", "long and short", "2,000 of /16-/24", "8,000 of /16-/24"])
def test_discriminate_forms_and_offsets(orc, name, at):
    """Every staged form, class bytes at another offset than the addresses, ragged ends."""
    import torch

    (net, ln), _ = TABLES[name]
    src = _addresses(net, ln, 6)
    dst = src[np.random.default_rng(8).permutation(len(src))]
    table = sinet.PrefixTable(net, ln)
    want = orc.classify(net, ln, src, dst) if len(net) else np.zeros(len(src), np.uint8)
    dev = {k: torch.zeros(len(v) + at[0], dtype=torch.int32, device="cuda")[at[0]:] for k, v in (("s", src), ("d", dst))}
    dev["s"].copy_(torch.from_numpy(src.view(np.int32)))
    dev["d"].copy_(torch.from_numpy(dst.view(np.int32)))
    for n in (1, 3, 4, 7, len(src)):
        cls = torch.full((n + at[1] + 4,), 9, dtype=torch.uint8, device="cuda")
        counts = sinet.discriminate(table, dev["s"][:n], dev["d"][:n], cls[at[1]:at[1] + n])
        got = cls.cpu().numpy()
        assert np.array_equal(got[at[1]:at[1] + n], want[:n])
        assert np.all(got[:at[1]] == 9) and np.all(got[at[1] + n:] == 9)  # nothing beside the records' bytes
        assert np.array_equal(counts.cpu().numpy(), np.bincount(want[:n], minlength=4))

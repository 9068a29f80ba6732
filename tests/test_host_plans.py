"""What the library plans on the host before a launch, from its own planning
functions with a GB300's facts; no GPU is used."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

from paper_2106_12863_gb300 import _build

HERE = os.path.dirname(os.path.abspath(__file__))
GLOBAL_ATOMIC, SMEM_FULL = 1, 4


@pytest.fixture(scope="module")
def plans(tmp_path_factory):
    lib = _build.build()
    out = str(tmp_path_factory.mktemp("plans") / "host_plans.so")
    subprocess.run([_build._nvcc(), *_build.ARCH, "-std=c++17", "-Xcompiler", "-fPIC", "--expt-relaxed-constexpr",
                    "-I", os.path.join(_build.ROOT, "include"), "-I", _build.CSRC, "-shared", "-o", out,
                    os.path.join(HERE, "host_plans.cu"), lib, "-Xlinker", "-rpath=" + os.path.dirname(lib)],
                   check=True)
    return ctypes.CDLL(out)


def prefixes(n, lo, hi, seed):
    rng = np.random.default_rng(seed)
    ln = rng.integers(lo, hi + 1, n)
    net = rng.integers(0, 1 << 31, n) & (0xFFFFFFFF << (32 - ln))
    return net.astype(np.uint32), ln.astype(np.uint8)


def _slice(plans, table, n, n_bins, strategy):
    out = np.zeros(6, np.int64)
    rc = plans.plan_batch_slice(*(ctypes.c_void_p(a.ctypes.data) for a in table), ctypes.c_uint32(len(table[0])),
                                ctypes.c_uint64(n), ctypes.c_uint64(n_bins), ctypes.c_int32(strategy),
                                ctypes.c_void_p(out.ctypes.data))
    assert rc == 0
    return dict(zip(("tile_fits", "lookup", "start", "bytes", "smem", "tile_bins"), out.tolist()))


def test_slices_of_one_list_in_both_forms(plans):
    """A list with a large leaf form: slices whose tile fits beside its smaller form only
    take that form on the tile alone, and what names a staged form tells the two apart."""
    table = prefixes(2500, 16, 24, 1)
    hour = _slice(plans, table, 100_000, 3600, SMEM_FULL)
    longer = _slice(plans, table, 100_000, 5400, SMEM_FULL)
    reduced = _slice(plans, table, 100_000, 5400, GLOBAL_ATOMIC)
    assert hour["tile_fits"] and longer["tile_fits"] and reduced["tile_fits"]
    assert longer["lookup"] != hour["lookup"] and longer["bytes"] < hour["bytes"]
    assert longer["start"] != hour["start"]
    assert (reduced["lookup"], reduced["start"]) == (hour["lookup"], hour["start"])
    for s in (hour, longer):
        assert s["bytes"] + 16 * s["tile_bins"] <= s["smem"]


@pytest.mark.parametrize("lean", [0, 1])
@pytest.mark.parametrize("n,n_bins", [(1, 1), (1_000_000, 10_000), (20_000_000, 21_600_000), (1_600_000_000, 86_400_000)])
def test_partition_run_counts_start_at_zero(plans, n, n_bins, lean):
    """A CTA of the main pass that leaves without storing its run counts leaves zeros, not stale memory."""
    out = np.zeros(5, np.uint64)
    assert plans.plan_partition_scratch(ctypes.c_uint64(n), ctypes.c_uint32(n_bins), lean, ctypes.c_void_p(out.ctypes.data)) == 0
    zero0, zero1, counts0, counts1, total = out.tolist()
    assert zero0 <= counts0 < counts1 <= zero1 <= total


def test_packed_cells_only_below_2_32_updates(plans):
    """The totals that check packed cells count bytes modulo 2^64: 2^32 updates at most, both directions' together."""
    packed = lambda n, two: plans.plan_packed_slice(ctypes.c_uint64(n), ctypes.c_uint32(1000), two)
    for two, limit in ((0, 1 << 32), (1, 1 << 31)):
        assert packed(limit - 1, two) and not packed(limit, two)
        assert (limit - 1) * (1 + two) * ((1 << 32) - 1) < 1 << 64


@pytest.mark.parametrize("seed", range(40))
def test_outputs_that_share_memory(plans, seed):
    """What keeps a slice or a call out of the schemes that store every bin, against every pair of rows."""
    rng = np.random.default_rng(seed)
    n = int(rng.integers(1, 9))
    bins = rng.integers(1, 50, n).astype(np.uint32)
    at = (4096 + 8 * rng.integers(0, (200, 2000)[seed % 2], (n, 4))).astype(np.uint64)
    shared, own = np.zeros(n, np.uint8), np.zeros(n, np.uint8)
    plans.output_overlaps(*(ctypes.c_void_p(a.ctypes.data) for a in (at, bins)), ctypes.c_uint32(n),
                          *(ctypes.c_void_p(a.ctypes.data) for a in (shared, own)))
    rows = [(i, int(at[i, k]), int(at[i, k]) + (4, 4, 8, 8)[k] * int(bins[i])) for i in range(n) for k in range(4)]
    meets = lambda a, b: a is not b and a[1] < b[2] and b[1] < a[2]
    for i in range(n):
        mine = [r for r in rows if r[0] == i]
        assert shared[i] == any(meets(a, b) for a in mine for b in rows)
        assert own[i] == any(meets(a, b) for a in mine for b in mine)


AUTO, NOAGG, SORT_REDUCE = 0, 5, 3
M = 1_000_000


@pytest.mark.parametrize("slices,want", [
    # (records, bins, strategy, accumulate, ready, as_first) of every slice; 8 M records are the line
    ([(20 * M, 21_600_000, AUTO, 0, 0, 0)], [1]),
    ([(7_999_999, M, AUTO, 0, 0, 0)], [0]),
    ([(7_999_999, M, NOAGG, 0, 0, 0), (1000, 6000, GLOBAL_ATOMIC, 0, 0, 0)], [1, 1]),
    # a slice that the rule puts on the tile does not count, but has cells if the tuner takes it off the tile
    ([(20 * M, 4000, AUTO, 0, 0, 0), (7_999_999, M, AUTO, 0, 0, 0)], [0, 0]),
    ([(20 * M, 4000, AUTO, 0, 0, 0), (8 * M, M, AUTO, 0, 0, 0)], [1, 1]),
    # too few records a bin; added to; waited for; outputs that another slice has too; other strategies
    ([(9 * M, M, NOAGG, 0, 0, 0), (16_666, 100_000, NOAGG, 0, 0, 0), (16_665, 100_000, NOAGG, 0, 0, 0)], [1, 1, 0]),
    ([(9 * M, 3_932_160, NOAGG, 0, 0, 0), (5 * M, 10 * M, NOAGG, 0, 0, 0), (5 * M - 1, 10 * M, NOAGG, 0, 0, 0)], [1, 1, 0]),
    ([(9 * M, M, NOAGG, 0, 0, 0), (9 * M, M, NOAGG, 1, 0, 0), (9 * M, M, NOAGG, 0, 1, 0)], [1, 0, 0]),
    ([(9 * M, M, NOAGG, 0, 0, 0), (9 * M, M, NOAGG, 0, 0, 1), (9 * M, M, NOAGG, 0, 0, 0)], [0, 0, 1]),
    ([(9 * M, M, SORT_REDUCE, 0, 0, 0), (9 * M, 4000, SMEM_FULL, 0, 0, 0), (7 * M, M, NOAGG, 0, 0, 0)], [0, 0, 0]),
])
def test_cells_are_decided_before_the_strategies(plans, slices, want):
    cols = [np.array(c, t) for c, t in zip(zip(*slices), (np.uint64, np.uint32, np.int32, np.uint8, np.uint8, np.uint8))]
    pack = np.zeros(len(slices), np.uint8)
    plans.plan_batch_cells(*(ctypes.c_void_p(c.ctypes.data) for c in cols), ctypes.c_uint32(len(slices)),
                           ctypes.c_void_p(pack.ctypes.data))
    assert pack.tolist() == want


def test_where_packed_cells_pay(plans):
    """The line in records over which a call takes packed cells, and that bench.py counts its kernels by it."""
    import bench

    pays = lambda bins, n: bool(plans.call_packed(ctypes.c_uint64(bins), ctypes.c_uint64(n)))
    lines = {1: 300_000, 600_000: 300_000, 600_002: 275_011, 1_000_000: 2_475_000, 1_500_000: 4_500_000,
             2_500_000: 4_500_000, 3_100_000: 3_450_000, 3_600_000: 1_950_000, 3_932_160: 953_520}
    for bins, line in lines.items():
        assert pays(bins, line) and not pays(bins, line - 1), bins
        assert [bench.kernels_per_step("global_atomic", n, bins) for n in (line - 1, line)] == [1, 3]
    assert not pays(3_932_161, 1 << 31) and bench.kernels_per_step("global_atomic", 1 << 31, 3_932_161) == 1

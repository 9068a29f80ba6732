// Host-side planning of the CUDA library, callable without a GPU: compiled by
// test_host_plans.py and linked against the library's own planning functions.
#include <cstdint>
#include <vector>

#include "batch_internal.h"
#include "partition.h"

using namespace sinet;

namespace {

// A GB300's facts, as device_state() reads them there.
DeviceState gb300() {
    DeviceState ds;
    ds.sm_count = 152;
    ds.smem_optin = 232448;
    ds.smem_per_sm = 233472;
    return ds;
}

bool host_table(const uint32_t *net, const uint8_t *len, uint32_t n, sinet_prefix_table &t) {
    if (compile_table(net, len, n, 0, t.host) != SINET_OK) return false;
    serialise(t.host, t.img);
    t.args = TableArgs{};
    t.args.image = reinterpret_cast<const uint8_t *>(uintptr_t(1) << 20);  // not read
    t.args.iv_bytes = t.img.iv_bytes;
    t.args.leaf_bytes = t.img.leaf_bytes;
    t.args.off_leaves = t.img.off_leaves;
    return true;
}

}  // namespace

extern "C" {

// One batch slice of n records and n_bins bins: {planned, lookup form, start of
// the staged form in the image (-1: none), its bytes, dynamic shared memory, tile bins}.
int plan_batch_slice(const uint32_t *net, const uint8_t *len, uint32_t n_net, uint64_t n, uint64_t n_bins,
                     int32_t strategy, int64_t *out) {
    sinet_prefix_table t{};
    if (!host_table(net, len, n_net, t)) return -1;
    const DeviceState ds = gb300();
    sinet_batch_slice u{};
    u.ts = reinterpret_cast<const uint64_t *>(uintptr_t(1) << 30);
    u.src = u.dst = u.bytes = reinterpret_cast<const uint32_t *>(uintptr_t(1) << 30);
    u.n = n;
    u.table = &t;
    u.params.bin_width_ms = 1;
    u.params.n_bins = n_bins;
    u.params.policy[1] = 1;
    u.params.policy[2] = 2;
    u.params.strategy = strategy;
    PlannedSlice ps;
    const uint32_t smem = batch_smem(&ds);
    const sinet_status st = plan_slice(u, &ds, smem, ps);
    if (st != SINET_OK) return (int)st;
    const uint8_t *form = staged_form(ps.d.t, ps.d.lk);
    out[0] = ps.tile_fits;
    out[1] = ps.d.lk;
    out[2] = form ? (int64_t)(form - t.args.image) : -1;
    out[3] = staged_form_bytes(ps.d.t, ps.d.lk);
    out[4] = smem;
    out[5] = ps.d.tile_bins;
    return 0;
}

// Whether a batch slice of n records and n_bins bins on plain reductions takes packed cells.
int plan_packed_slice(uint64_t n, uint32_t n_bins, int two_dir) {
    PlannedSlice ps;
    ps.d = BatchSlice{};
    ps.d.r.g = make_geom(n, {});
    ps.d.h.n_bins = n_bins;
    ps.d.h.two_dir = two_dir != 0;
    for (int d = 0; d < 2; ++d) {
        ps.d.h.cnt[d] = reinterpret_cast<uint32_t *>((uint64_t)(1 + d) << 40);
        ps.d.h.byt[d] = reinterpret_cast<uint64_t *>((uint64_t)(3 + d) << 40);
    }
    ps.d.zero = 1;
    ps.strategy = SINET_STRAT_ATOMIC_NOAGG;
    std::vector<PlannedSlice> v(1, ps);
    plan_cells(v);
    return slice_packed(v[0]);
}

int call_packed(uint64_t n_bins, uint64_t n) { return packed_pays(n_bins, n); }

// plan_cells for a batch of n_slices slices: records, bins, strategy, accumulate,
// ready word and "same outputs as slice 0" of each; pack[i] is its decision.
void plan_batch_cells(const uint64_t *n, const uint32_t *bins, const int32_t *strategy, const uint8_t *accumulate,
                      const uint8_t *ready, const uint8_t *as_first, uint32_t n_slices, uint8_t *pack) {
    std::vector<PlannedSlice> v(n_slices);
    for (uint32_t i = 0; i < n_slices; ++i) {
        PlannedSlice &ps = v[i];
        ps.d = BatchSlice{};
        ps.d.r.g = make_geom(n[i], {});
        const uintptr_t at = as_first[i] ? 1 : 1 + (uintptr_t)i;
        for (int d = 0; d < 2; ++d) {
            ps.d.h.cnt[d] = reinterpret_cast<uint32_t *>((2 * at + d) << 40);
            ps.d.h.byt[d] = reinterpret_cast<uint64_t *>(((2 * at + d) << 40) + (1ull << 39));
        }
        ps.d.h.n_bins = bins[i];
        ps.d.zero = !accumulate[i];
        ps.d.ready = ready[i] ? reinterpret_cast<const uint32_t *>(uintptr_t(64)) : nullptr;
        ps.tile_fits = bins[i] <= 4000;
        ps.strategy = strategy[i];
    }
    plan_cells(v);
    for (uint32_t i = 0; i < n_slices; ++i) pack[i] = v[i].pack;
}

// Which of n histograms' outputs (count[0], count[1], bytes[0], bytes[1] and
// bins each) overlap any other rows: by the batch's sweep, and each by itself.
void output_overlaps(const uint64_t *at, const uint32_t *bins, uint32_t n, uint8_t *shared, uint8_t *rows_overlap) {
    std::vector<OutputRange> v;
    std::vector<bool> mark(n);
    for (uint32_t i = 0; i < n; ++i) {
        HistArgs h{};
        for (int d = 0; d < 2; ++d) {
            h.cnt[d] = reinterpret_cast<uint32_t *>(at[4 * i + d]);
            h.byt[d] = reinterpret_cast<uint64_t *>(at[4 * i + 2 + d]);
        }
        h.n_bins = bins[i];
        output_ranges(h, i, v);
        rows_overlap[i] = !rows_apart(h);
    }
    mark_overlaps(v, mark);
    for (uint32_t i = 0; i < n; ++i) shared[i] = mark[i];
}

// The partition of n aligned records into n_bins bins: {zeroed bytes' start and
// end, run counts' start and end, scratch bytes}.
int plan_partition_scratch(uint64_t n, uint32_t n_bins, int lean, uint64_t *out) {
    RecArgs r{};
    r.g = make_geom(n, {});
    HistArgs h{};
    h.n_bins = n_bins;
    const DeviceState ds = gb300();
    PartPlan p;
    if (plan_partition(LK_LEAF2, 16384, r, h, 0, ds.sm_count, ds.smem_optin, lean != 0, &p) != cudaSuccess) return -1;
    out[0] = p.off_zero;
    out[1] = p.off_zero + p.bytes_zero;
    out[2] = p.off_counts;
    out[3] = p.off_counts + 4ull * p.d.n_buckets * p.d.g_main;
    out[4] = p.scratch_bytes;
    return 0;
}

}  // extern "C"

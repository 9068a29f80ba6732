// Host helpers shared by the C-ABI translation units.
#pragma once
#include <initializer_list>
#include <vector>

#include <nvtx3/nvToolsExt.h>

#include "launch.h"
#include "table_host.h"

struct sinet_prefix_table {
    int device;
    sinet::TableHost host;
    sinet::TableImage img;
    uint8_t *d_image;
    sinet::TableArgs args;
};

namespace sinet {

constexpr uint64_t kMaxN = 1ull << 40;

// Per-device facts and the device status word, set up on first use.
struct DeviceState {
    bool ready = false;
    int sm_count = 0;
    size_t smem_optin = 0;
    size_t smem_per_sm = 0;
    uint32_t *status = nullptr;  // device status word
};
sinet_status device_state(DeviceState **out);
// Map a failed CUDA call to a status (and remember it for sinet_last_cuda_error).
sinet_status cuda_fail(cudaError_t e);

#define SINET_CUDA(x)                                          \
    do {                                                       \
        cudaError_t e_ = (x);                                  \
        if (e_ != cudaSuccess) return ::sinet::cuda_fail(e_);  \
    } while (0)

// A profiler-visible range around a C-ABI call (NVTX; it costs nothing when
// no tool is attached).
struct TraceRange {
    explicit TraceRange(const char *name) { nvtxRangePushA(name); }
    ~TraceRange() { nvtxRangePop(); }
    TraceRange(const TraceRange &) = delete;
    TraceRange &operator=(const TraceRange &) = delete;
};
#define SINET_TRACE() ::sinet::TraceRange sinet_trace_range_(__func__)

struct Stream {
    const void *p;
    uint32_t esize;
};

Divider make_divider(uint64_t w);
QuadGeom make_geom(uint64_t n, std::initializer_list<Stream> streams);
bool aligned(const void *p, size_t a);
sinet_status check_params(const sinet_hist_params *p);
sinet_status check_out(const sinet_hist_out *o);
HistArgs make_hist(const sinet_hist_params *p, const sinet_hist_out *o);
// An update adds to its output words, so outputs may share memory: two slices
// of a batch that fill one histogram, both directions in one array. What stores
// every bin of its outputs instead asks here whether they stand apart.
struct OutputRange {
    uintptr_t lo, hi;
    uint32_t owner;
};
void output_ranges(const HistArgs &h, uint32_t owner, std::vector<OutputRange> &v);
// Sets mark[owner] for every owner of a range that overlaps another range.
void mark_overlaps(std::vector<OutputRange> &v, std::vector<bool> &mark);
bool rows_apart(const HistArgs &h);
// Whether the totals that check packed cells (HistArgs::packed) hold every total
// of n records: below 2^32 updates, whose bytes stay below 2^64. Past that the
// byte totals wrap, and cells that lost 2^64 bytes and a count could agree.
inline bool packed_countable(uint64_t n, bool two_dir) { return n < (two_dir ? 1ull << 31 : 1ull << 32); }
// Whether a call of n records over n_bins bins on warp combining gains by packed cells.
bool packed_pays(uint64_t n_bins, uint64_t n);
sinet_status zero_outputs(const sinet_hist_params *p, const sinet_hist_out *o, cudaStream_t s);
// The shared-memory form of a table that has one: its leaf form, else its toggle form.
int staged_lookup(const sinet_prefix_table *t);
int toggle_lookup(const sinet_prefix_table *t);
// The table's toggle form takes less shared memory than the form `lk`.
bool toggle_is_smaller(const sinet_prefix_table *t, int lk);
int pick_lookup(const sinet_prefix_table *t, int32_t lookup, sinet_status *err);

}  // namespace sinet

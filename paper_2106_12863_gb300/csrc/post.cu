// Histogram post-processing on the device: roll-up into coarser bins and
// sparse compaction of the non-empty bins (the downstream views of
// Section 6 use hourly and ten-minute bins; the reduce-by-key of Section 5
// yields only the present keys).
#include <algorithm>

#include "api_internal.h"

namespace sinet {
namespace {

constexpr uint32_t kPostBlock = 256;
constexpr uint32_t kPostWarps = kPostBlock / 32;
constexpr uint32_t kRollSteps = 8;                  // a warp's segment: this many rows of 32 bins
constexpr uint32_t kRollSeg = 32 * kRollSteps;
constexpr uint32_t kSparseBlock = 512;              // one CTA per SM
constexpr uint32_t kSparseWarps = kSparseBlock / 32;
constexpr uint32_t kSparseRows = 8;                 // a warp's share of a tile: this many rows of 32 bins
constexpr uint32_t kSparseTile = kSparseBlock * kSparseRows;  // bins per compaction tile

// One bin's four values.
struct Bin {
    uint32_t c0, c1;
    uint64_t b0, b1;
};

__device__ __forceinline__ Bin load_bin(const HistArgs &h, uint64_t i) {
    return {__ldcs(h.cnt[0] + i), __ldcs(h.cnt[1] + i),
            __ldcs(reinterpret_cast<const unsigned long long *>(h.byt[0] + i)),
            __ldcs(reinterpret_cast<const unsigned long long *>(h.byt[1] + i))};
}

__device__ __forceinline__ void add_bin(Bin &a, const Bin &b) {
    a.c0 += b.c0;
    a.c1 += b.c1;
    a.b0 += b.b0;
    a.b1 += b.b1;
}

__device__ __forceinline__ Bin shfl_down_bin(const Bin &a, int d) {
    return {__shfl_down_sync(kFull, a.c0, d), __shfl_down_sync(kFull, a.c1, d), __shfl_down_sync(kFull, a.b0, d),
            __shfl_down_sync(kFull, a.b1, d)};
}

__device__ __forceinline__ void red_bin(const HistArgs &out, uint32_t o, const Bin &v) {
    red_add_u32(out.cnt[0] + o, v.c0);
    red_add_u32(out.cnt[1] + o, v.c1);
    red_add_u64(out.byt[0] + o, v.b0);
    red_add_u64(out.byt[1] + o, v.b1);
}

// The whole warp's sum of v into output bin o (lane 0 adds it).
__device__ __forceinline__ void flush_warp(const HistArgs &out, uint32_t o, Bin v) {
#pragma unroll
    for (int d = 16; d; d >>= 1) add_bin(v, shfl_down_bin(v, d));
    if ((threadIdx.x & 31) == 0) red_bin(out, o, v);
}

// A read of the fine histogram (24 bytes a bin) is the whole cost. Each warp
// takes a contiguous run of segments of 256 bins and loads a segment as eight
// coalesced rows of 32, so 192 bytes a lane are in flight and no array needs
// more than its element's alignment. A segment inside one output bin is
// summed in registers, which carry over to the next segment of the same output
// bin; a segment that spans several is reduced row by row over the runs of
// equal output bins. One division per segment, or per bin where it spans
// several (by multiplication; the 64-bit divisions, one a bin, were most of
// the previous kernel's time: 960-1,050 us for 86.4 M bins to 144 or 86,400,
// 296-322 now).
__global__ void __launch_bounds__(kPostBlock) k_rollup(HistArgs in, Divider by, HistArgs out) {
    const uint32_t lane = threadIdx.x & 31;
    const uint64_t n = in.n_bins, segs = (n + kRollSeg - 1) / kRollSeg;
    const uint64_t warps = (uint64_t)gridDim.x * kPostWarps, w = (uint64_t)blockIdx.x * kPostWarps + (threadIdx.x >> 5);
    const uint64_t s1 = segs * (w + 1) / warps;
    Bin acc = {0, 0, 0, 0};
    uint32_t cur = kNoKey;  // output bin of acc
    for (uint64_t s = segs * w / warps; s < s1; ++s) {
        const uint64_t first = s * kRollSeg, last = min(first + kRollSeg, n) - 1;
        Bin v[kRollSteps];
#pragma unroll
        for (uint32_t k = 0; k < kRollSteps; ++k) {
            const uint64_t i = first + 32 * k + lane;
            v[k] = i <= last ? load_bin(in, i) : Bin{0, 0, 0, 0};
        }
        const uint32_t o = (uint32_t)divide(first, by);
        const bool one = (uint32_t)divide(last, by) == o;
        if (cur != kNoKey && (!one || cur != o)) {
            flush_warp(out, cur, acc);
            acc = {0, 0, 0, 0};
            cur = kNoKey;
        }
        if (one) {
#pragma unroll
            for (uint32_t k = 0; k < kRollSteps; ++k) add_bin(acc, v[k]);
            cur = o;
            continue;
        }
#pragma unroll
        for (uint32_t k = 0; k < kRollSteps; ++k) {
            const uint64_t i = first + 32 * k + lane;
            const uint32_t oi = i <= last ? (uint32_t)divide(i, by) : kNoKey;
            // suffix sums over the run of lanes with this output bin; its first lane adds the total
            Bin x = v[k];
#pragma unroll
            for (int d = 1; d < 32; d <<= 1) {
                const uint32_t od = __shfl_down_sync(kFull, oi, d);
                const Bin y = shfl_down_bin(x, d);
                if (lane + d < 32 && od == oi) add_bin(x, y);
            }
            const uint32_t before = __shfl_up_sync(kFull, oi, 1);
            if (oi != kNoKey && (lane == 0 || before != oi)) red_bin(out, oi, x);
        }
    }
    if (cur != kNoKey) flush_warp(out, cur, acc);
}

// A tile's status word: flag (2 bits) | bins kept (62 bits).
constexpr uint64_t kTileOwn = 1ull << 62;     // the tile's own bins
constexpr uint64_t kTilePrefix = 2ull << 62;  // the bins of every tile up to and including it
constexpr uint64_t kTileValue = (1ull << 62) - 1;

// Exclusive prefix of tile `tile` by the whole CTA: each thread reads the
// status word of one predecessor (thread 0 the nearest), back to the nearest
// one whose prefix is known; 512 a step, more than the tiles in flight, so one
// step (one L2 round trip) is the rule. Tiles are numbered as CTAs claim them,
// so every predecessor is held by a running CTA or done; the wait for each is
// bounded all the same. s_sum holds a word a warp.
__device__ __forceinline__ uint64_t tile_prefix(uint64_t *st, uint64_t tile, uint64_t *s_sum, uint32_t *status) {
    const uint32_t lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    volatile uint64_t *vst = st;
    uint64_t excl = 0;
    for (int64_t hi = (int64_t)tile; hi > 0; hi -= kSparseBlock) {
        const int64_t p = hi - 1 - (int64_t)threadIdx.x;
        uint64_t w = kTilePrefix;  // before the first tile: nothing
        if (p >= 0) {
            uint32_t it = 0;
            while ((w = vst[p]) < kTileOwn && ++it < kSpinLimit) {
            }
            if (w < kTileOwn) {
                latch_status(status, SINET_ERR_TIMEOUT);
                w = kTilePrefix;
            }
        }
        // the warp's sum up to its nearest known prefix
        const uint32_t known = __ballot_sync(kFull, (w & kTilePrefix) != 0);
        const uint32_t upto = known ? (uint32_t)__ffs(known) - 1 : 31u;
        uint64_t v = lane <= upto ? w & kTileValue : 0;
#pragma unroll
        for (int d = 16; d; d >>= 1) v += __shfl_down_sync(kFull, v, d);
        if (lane == 0) s_sum[warp] = v | (known ? kTilePrefix : 0);
        __syncthreads();
        bool done = false;
#pragma unroll
        for (uint32_t k = 0; k < kSparseWarps; ++k) {
            const uint64_t x = s_sum[k];
            if (!done) excl += x & kTileValue;
            done |= (x & kTilePrefix) != 0;
        }
        __syncthreads();
        if (done) break;
    }
    return excl;
}

// Sparse form in one pass: a CTA takes tile after tile of 4,096 bins (eight
// coalesced rows of 32 bins a warp, held in registers), ranks a tile's
// non-empty bins by ballots, learns how many precede the tile by looking back
// over the predecessors' status words, and writes the bins from registers. The
// loads of the next tile are in flight meanwhile (98 KB an SM), so the
// look-back's round trips hide behind them: one CTA per tile with no load ahead
// took 1,281 us for 82 M of 86.4 M bins, this 975. The traffic is the
// algorithmic one, 24 bytes read a bin and 28 written a kept bin (a counting
// pass before the writing one read the histogram twice: 1,680 us).
__global__ void __launch_bounds__(kSparseBlock, 1) k_sparse(HistArgs h, uint32_t tiles, uint64_t *tile_status,
                                                            uint32_t *ticket, uint64_t cap, uint32_t *o_bin,
                                                            uint32_t *o_c0, uint32_t *o_c1, uint64_t *o_b0,
                                                            uint64_t *o_b1, uint64_t *total, uint32_t *status) {
    __shared__ uint32_t s_next, s_warp[kSparseWarps];
    __shared__ uint64_t s_sum[kSparseWarps];
    const uint32_t lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const uint32_t mine = warp * (32 * kSparseRows) + lane;
    auto load = [&](uint32_t tile, Bin (&v)[kSparseRows]) {
#pragma unroll
        for (uint32_t k = 0; k < kSparseRows; ++k) {
            const uint64_t i = (uint64_t)tile * kSparseTile + mine + 32 * k;
            v[k] = tile < tiles && i < h.n_bins ? load_bin(h, i) : Bin{0, 0, 0, 0};
        }
    };
    if (threadIdx.x == 0) s_next = atomicAdd(ticket, 1u);
    __syncthreads();
    uint32_t tile = s_next;
    Bin v[kSparseRows], nv[kSparseRows];
    load(tile, v);
    while (tile < tiles) {
        uint32_t bal[kSparseRows], kept = 0;
#pragma unroll
        for (uint32_t k = 0; k < kSparseRows; ++k) {
            bal[k] = __ballot_sync(kFull, (v[k].c0 | v[k].c1) != 0 || (v[k].b0 | v[k].b1) != 0);
            kept += __popc(bal[k]);
        }
        if (lane == 0) s_warp[warp] = kept;
        __syncthreads();  // (the tile's number has been read, too)
        uint32_t ahead = 0, all = 0;
#pragma unroll
        for (uint32_t w = 0; w < kSparseWarps; ++w) {
            if (w < warp) ahead += s_warp[w];
            all += s_warp[w];
        }
        // the next tile is claimed only now: look-backs wait for claimed tiles,
        // and claimed while this tile's bins arrive it waits longer for its
        // turn (1,119 us; two tiles ahead 2,716)
        volatile uint64_t *vst = tile_status;
        if (threadIdx.x == 0) {
            vst[tile] = (tile ? kTileOwn : kTilePrefix) | all;
            s_next = atomicAdd(ticket, 1u);
        }
        __syncthreads();
        const uint32_t next = s_next;
        load(next, nv);
        const uint64_t before = tile_prefix(tile_status, tile, s_sum, status);
        if (threadIdx.x == 0) {
            if (tile) vst[tile] = kTilePrefix | (before + all);
            if (tile == tiles - 1) *total = before + all;
        }
        uint64_t pos = before + ahead;
#pragma unroll
        for (uint32_t k = 0; k < kSparseRows; ++k) {
            const uint64_t at = pos + __popc(bal[k] & ((1u << lane) - 1u));
            if ((bal[k] >> lane & 1u) && at < cap) {
                __stcs(o_bin + at, tile * kSparseTile + mine + 32 * k);
                __stcs(o_c0 + at, v[k].c0);
                __stcs(o_c1 + at, v[k].c1);
                __stcs(reinterpret_cast<unsigned long long *>(o_b0 + at), (unsigned long long)v[k].b0);
                __stcs(reinterpret_cast<unsigned long long *>(o_b1 + at), (unsigned long long)v[k].b1);
            }
            pos += __popc(bal[k]);
        }
#pragma unroll
        for (uint32_t k = 0; k < kSparseRows; ++k) v[k] = nv[k];
        tile = next;
    }
}

HistArgs view(const sinet_hist_out *o, uint64_t n_bins) {
    HistArgs h{};
    h.cnt[0] = o->count[0];
    h.cnt[1] = o->count[1];
    h.byt[0] = o->bytes[0];
    h.byt[1] = o->bytes[1];
    h.stats = o->stats;
    h.n_bins = (uint32_t)n_bins;
    return h;
}

bool out_arrays_ok(const sinet_hist_out *o) {
    return o && o->count[0] && o->count[1] && o->bytes[0] && o->bytes[1] && aligned(o->count[0], 4) &&
           aligned(o->count[1], 4) && aligned(o->bytes[0], 8) && aligned(o->bytes[1], 8);
}

}  // namespace
}  // namespace sinet

using namespace sinet;

extern "C" {

sinet_status sinet_histogram_rollup(const sinet_hist_out *in, uint64_t n_bins, uint64_t factor, int accumulate,
                                    const sinet_hist_out *out, sinet_stream_t stream) {
    SINET_TRACE();
    if (!out_arrays_ok(in) || !out_arrays_ok(out) || n_bins == 0 || n_bins > 0x7FFFFFFFull || factor == 0)
        return SINET_ERR_INVALID_ARG;
    DeviceState *ds = nullptr;
    sinet_status st = device_state(&ds);
    if (st != SINET_OK) return st;
    const uint64_t n_out = (n_bins + factor - 1) / factor;
    if (!accumulate) {
        SINET_CUDA(cudaMemsetAsync(out->count[0], 0, 4 * n_out, stream));
        SINET_CUDA(cudaMemsetAsync(out->count[1], 0, 4 * n_out, stream));
        SINET_CUDA(cudaMemsetAsync(out->bytes[0], 0, 8 * n_out, stream));
        SINET_CUDA(cudaMemsetAsync(out->bytes[1], 0, 8 * n_out, stream));
    }
    if (in->stats && out->stats && in->stats != out->stats)
        SINET_CUDA(cudaMemcpyAsync(out->stats, in->stats, 64, cudaMemcpyDeviceToDevice, stream));
    const uint64_t segs = (n_bins + kRollSeg - 1) / kRollSeg;
    const int grid = (int)std::min<uint64_t>((segs + kPostWarps - 1) / kPostWarps, 8ull * ds->sm_count);
    k_rollup<<<grid, kPostBlock, 0, stream>>>(view(in, n_bins), make_divider(factor), view(out, n_out));
    SINET_CUDA(cudaGetLastError());
    return SINET_OK;
}

sinet_status sinet_histogram_sparse(const sinet_hist_out *in, uint64_t n_bins, uint32_t *d_bin, uint32_t *d_count0,
                                    uint32_t *d_count1, uint64_t *d_bytes0, uint64_t *d_bytes1, uint64_t cap,
                                    uint64_t *d_n_out, sinet_stream_t stream) {
    SINET_TRACE();
    if (!out_arrays_ok(in) || n_bins == 0 || n_bins > 0x7FFFFFFFull || !d_n_out || !aligned(d_n_out, 8))
        return SINET_ERR_INVALID_ARG;
    if (cap && (!d_bin || !d_count0 || !d_count1 || !d_bytes0 || !d_bytes1 || !aligned(d_bin, 4) ||
                !aligned(d_count0, 4) || !aligned(d_count1, 4) || !aligned(d_bytes0, 8) || !aligned(d_bytes1, 8)))
        return SINET_ERR_INVALID_ARG;
    DeviceState *ds = nullptr;
    sinet_status st = device_state(&ds);
    if (st != SINET_OK) return st;
    const uint64_t tiles = (n_bins + kSparseTile - 1) / kSparseTile;
    // a status word per tile and the tile counter, zero at the start
    void *scratch = nullptr;
    const size_t bytes = 8 * tiles + 8;
    SINET_CUDA(cudaMallocAsync(&scratch, bytes, stream));
    uint64_t *tile_status = static_cast<uint64_t *>(scratch);
    cudaError_t e = cudaMemsetAsync(scratch, 0, bytes, stream);
    if (e == cudaSuccess) {
        const int grid = (int)std::min<uint64_t>(tiles, (uint64_t)ds->sm_count);
        k_sparse<<<grid, kSparseBlock, 0, stream>>>(view(in, n_bins), (uint32_t)tiles, tile_status,
                                                    reinterpret_cast<uint32_t *>(tile_status + tiles), cap, d_bin,
                                                    d_count0, d_count1, d_bytes0, d_bytes1, d_n_out, ds->status);
        e = cudaGetLastError();
    }
    const cudaError_t e2 = cudaFreeAsync(scratch, stream);
    if (e == cudaSuccess) e = e2;
    return e == cudaSuccess ? SINET_OK : cuda_fail(e);
}

}  // extern "C"

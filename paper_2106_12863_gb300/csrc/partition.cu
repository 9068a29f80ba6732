// Hot/cold partitioned histogram update (SINET_STRAT_PARTITION), for
// unsorted records over a histogram too large for shared memory.
//
// The update step of Section 5 (per-direction <timestamp, count> and
// <timestamp, bytes> sums) split by how often a bin is hit. A bin hit often
// lives in shared memory for the whole pass; a bin hit rarely becomes an entry
// of its bin range's run, and the runs are summed tile by tile in shared
// memory, so every output bin is stored once with plain stores and no sector
// of the histogram is ever read-modified-written in DRAM. See partition.h for
// the sequence.
#include <algorithm>

#include "combine.cuh"
#include "partition.h"

namespace sinet {

namespace {

// Fibonacci hashing: the top bits of bin * 2^32 / phi spread any run of bins
__device__ __forceinline__ uint32_t fib_hash(uint32_t b) { return b * 0x9E3779B1u; }

__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
}

__device__ __forceinline__ void mbar_expect_tx(uint32_t bar, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}

__device__ __forceinline__ void mbar_arrive(uint32_t bar) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}

// Bounded wait for the phase of `bar` with parity `parity` to complete.
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity) {
    for (uint32_t it = 0; it < kSpinLimit; ++it)
        if (mbar_try_wait(bar, parity)) return true;
    return false;
}

// TMA bulk copy (non-tensor) of `bytes` from global memory into this CTA's
// shared memory, completing on `bar`; 16-byte aligned ends, size a multiple of 16.
__device__ __forceinline__ void bulk_g2s(uint32_t dst, const void *src, uint32_t bytes, uint32_t bar) {
    asm volatile(
        "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(dst),
        "l"(src), "r"(bytes), "r"(bar)
        : "memory");
}

__device__ __forceinline__ uint32_t vload(const uint32_t *p) { return *reinterpret_cast<const volatile uint32_t *>(p); }

// Sample counts: linear probing over the open-addressing table. A key that
// finds no slot within the probe bound is dropped: the sample only ranks
// bins, it is not part of the result.
__device__ void hash_add(const PartDev &p, uint32_t key, uint32_t c) {
    uint32_t s = fib_hash(key) >> p.hash_shift;
    for (int probe = 0; probe < 64; ++probe) {
        const uint32_t k = atomicCAS(p.hash_keys + s, kNoKey, key);
        if (k == kNoKey || k == key) {
            atomicAdd(p.hash_cnt + s, c);
            return;
        }
        s = (s + 1) & p.hash_mask;
    }
}

}  // namespace

// ---------------------------------------------------------------------------
// 1. Sample: every sample_stride-th chunk of kPartSampleChunk records is
// classified and binned, a record per thread (the cost is the chain of round
// trips to the hash, not the loads); hits per bin (both directions together) are
// pre-aggregated in a per-CTA shared-memory cache, then counted in the hash.
template <int LK>
__global__ void __launch_bounds__(kPartSampleThreads) k_part_sample(RecArgs r, TableArgs t, HistArgs h, PartDev p,
                                                     uint32_t *status) {
    extern __shared__ __align__(16) uint8_t smem[];
    __shared__ uint64_t bar;
    Classifier<LK> C;
    if (!C.init(t, smem, &bar, status)) return;
    uint8_t *cm = smem + ((Classifier<LK>::smem_bytes(t) + 15u) & ~15u);
    const uint32_t slots = HotCache::kWays << kPartSampleSetBits;
    HotCache hc;
    hc.keys = reinterpret_cast<uint32_t *>(cm);
    hc.cnt = hc.keys + slots;
    hc.lo = hc.cnt + slots;
    hc.hi = hc.lo + slots;
    hc.set_bits = kPartSampleSetBits;
    for (uint32_t i = threadIdx.x; i < slots; i += blockDim.x) {
        hc.keys[i] = kNoKey;
        hc.cnt[i] = 0;
        hc.lo[i] = 0;
        hc.hi[i] = 0;
    }
    __syncthreads();
    const uint64_t total = p.sample_chunks * kPartSampleChunk;
    uint32_t oor[2] = {0, 0};
    for (uint64_t w = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; w < total;
         w += (uint64_t)gridDim.x * blockDim.x) {
        const uint64_t i = (w / kPartSampleChunk) * p.sample_stride * kPartSampleChunk + w % kPartSampleChunk;
        if (i >= r.g.n) continue;
        const uint32_t a[2] = {r.src[i], r.dst[i]};
        uint32_t in[2], bin;
        C.template in_n<2>(a, in);
        const uint32_t c = __popc(route(h, in[0] | in[1] << 1, r.ts[i], bin, oor));
        if (c && !hc.add(bin, c, 0)) hash_add(p, bin, c);
    }
    __syncthreads();
    for (uint32_t i = threadIdx.x; i < slots; i += blockDim.x)
        if (hc.cnt[i]) hash_add(p, hc.keys[i], hc.cnt[i]);
}

// 2a. Hash slots per log2 of their sample count, and the sample hits in all
// (levels[32], for the thresholds below).
__global__ void __launch_bounds__(256) k_part_levels(PartDev p) {
    __shared__ uint32_t s[33];
    if (threadIdx.x < 33) s[threadIdx.x] = 0;
    __syncthreads();
    uint32_t hits = 0;
    for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i <= p.hash_mask; i += gridDim.x * blockDim.x) {
        const uint32_t c = p.hash_cnt[i];
        hits += c;
        if (c) atomicAdd(&s[31 - __clz(c)], 1u);
    }
    hits = __reduce_add_sync(kFull, hits);
    if ((threadIdx.x & 31) == 0 && hits) atomicAdd(&s[32], hits);
    __syncthreads();
    if (threadIdx.x < 33 && s[threadIdx.x]) atomicAdd(p.levels + threadIdx.x, s[threadIdx.x]);
}

// 2b. Candidates: the bins with at least two hits of the highest count levels
// that together hold at most max_cand bins (twice the table's slots). And the sample hits of every
// tile of bins.
__global__ void __launch_bounds__(256) k_part_collect(PartDev p) {
    // the lowest level that fits, by every warp for itself: lane l holds the
    // bins of levels 31 - l and above
    const uint32_t lane = threadIdx.x & 31;
    uint32_t cum = p.levels[31 - lane];
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
        const uint32_t y = __shfl_up_sync(kFull, cum, d);
        if (lane >= (uint32_t)d) cum += y;
    }
    const uint32_t fits = __ballot_sync(kFull, cum <= p.max_cand && lane < 31);  // a prefix of the lanes
    const uint32_t thr = fits ? 1u << (31 - (31 - __clz(fits))) : 0xFFFFFFFFu;
    const uint32_t n_slots = p.hash_mask + 1;
    // warp-uniform trip count for the ballot
    for (uint32_t i0 = (blockIdx.x * blockDim.x + threadIdx.x) - lane; i0 < n_slots;
         i0 += gridDim.x * blockDim.x) {
        const uint32_t i = i0 + lane;
        const uint32_t c = i < n_slots ? p.hash_cnt[i] : 0u;
        const uint32_t key = c ? p.hash_keys[i] : 0u;
        if (c) atomicAdd(p.tile_hits + (key >> p.tile_bits), c);
        const bool take = c >= thr;
        const uint32_t m = __ballot_sync(kFull, take);
        if (!m) continue;
        uint32_t base = 0;
        if (lane == 0) base = atomicAdd(p.cand_n, (uint32_t)__popc(m));
        base = __shfl_sync(kFull, base, 0);
        if (take) {
            const uint32_t pos = base + __popc(m & ((1u << lane) - 1u));
            if (pos < p.max_cand) p.cand[pos] = make_uint2(key, c);
        }
    }
}

// Sum of v over the CTA (1,024 threads), in every thread. s holds 32 words.
__device__ __forceinline__ uint64_t cta_sum(uint64_t v, uint64_t *s) {
#pragma unroll
    for (int d = 16; d; d >>= 1) v += __shfl_down_sync(kFull, v, d);
    __syncthreads();
    if ((threadIdx.x & 31) == 0) s[threadIdx.x >> 5] = v;
    __syncthreads();
    uint64_t t = 0;
#pragma unroll
    for (int w = 0; w < 32; ++w) t += s[w];
    return t;
}

// Starts of n consecutive stretches from 0 on (start[n] = the end of the last)
// by the whole CTA: stretch i has room for hits(i) sample hits at `per_hit`
// entries each, as made likely by the sample: three standard deviations of the
// sample's own count and four of the entries' are added. Scaled down to `cap`
// in all. `room` is shared scratch of n words.
template <typename Hits>
__device__ void stretches(uint32_t n, Hits &&hits, float per_hit, uint64_t cap, uint32_t *room, uint32_t *start,
                          uint32_t *start2, uint64_t *s_sum) {
    uint64_t want = 0;
    for (uint32_t i = threadIdx.x; i < n; i += blockDim.x) {
        const float sh = (float)hits(i), e = sh * per_hit;
        const float w = (sh + 3.f * sqrtf(sh) + 3.f) * per_hit + 4.f * sqrtf(e) + 8.f;
        const uint32_t r = ((uint32_t)fminf(w, 4.0e9f) + 15u) & ~15u;  // whole 128-byte lines
        room[i] = r;
        want += r;
    }
    want = cta_sum(want, s_sum);
    const uint32_t per = (n + 1023) / 1024, i0 = threadIdx.x * per, i1 = min(i0 + per, n);
    uint32_t mine = 0;
    for (uint32_t i = i0; i < i1; ++i) {
        if (want > cap) room[i] = (uint32_t)((uint64_t)room[i] * cap / want) & ~15u;
        mine += room[i];
    }
    const uint32_t lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    uint32_t incl = mine;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
        const uint32_t y = __shfl_up_sync(kFull, incl, d);
        if (lane >= (uint32_t)d) incl += y;
    }
    __syncthreads();
    if (lane == 31) s_sum[warp] = incl;
    __syncthreads();
    uint32_t at = incl - mine;
    for (uint32_t w = 0; w < warp; ++w) at += (uint32_t)s_sum[w];
    for (uint32_t i = i0; i < i1; ++i) {
        const uint32_t r = room[i];  // (room may be start2)
        start[i] = at;
        if (start2) start2[i] = at;
        at += r;
        if (i == n - 1) start[n] = at;
    }
    __syncthreads();
}

// 2c. The hot table and the room of every run (one CTA).
//
// The table has sets of two ways. h = bin * 2^32 / phi is a bijection on 32
// bits, so its top set_bits name the set and the others the bin within it: the
// entry of a bin is h shifted left by set_bits, plus a code in the bits that
// frees. XORed with the shifted h of a record's bin an entry gives the code, or
// a value of at least 2^set_bits when it is another bin's, so the smaller of
// the two XORs is the whole probe (one 8-byte shared load; four ways of plain
// bins compared one by one took a 16-byte load and twice the instructions).
// Codes 0 and 1 name the way, and with it the slot of the sums; code 2 + g names
// group g of kPartRepCopies slots over which the lanes spread: the bins with at
// least 1/64 of the sampled updates, whose one slot would serialise its atomics.
//
// Candidates are inserted level by level, the highest sample counts first; one
// whose set is full stays cold. A table that would take less than 1/16 of the
// updates is left empty (n_hot = 0): the main pass then skips its probe, which
// every record would pay for.
//
// A CTA of the main pass keeps a run of entries per range, and the split a run
// per tile; their rooms come from the cold sample hits. An entry that finds its
// run full goes to the overflow list, so the rooms are never about correctness.
__global__ void __launch_bounds__(1024) k_part_build(PartDev p, uint32_t slots) {
    extern __shared__ __align__(16) uint8_t smem[];
    __shared__ uint64_t s_sum[32];
    __shared__ uint32_t s_lev[33], s_reps;
    uint32_t *keys = reinterpret_cast<uint32_t *>(smem);
    // [n_tiles] cold sample hits per tile, and scratch; in shared memory where it holds them
    uint32_t *hits = p.tiles_in_smem ? keys + slots : p.tile_hits;
    uint32_t *room = p.tiles_in_smem ? hits + p.n_tiles : p.tile_cur;
    for (uint32_t i = threadIdx.x; i < slots; i += blockDim.x) keys[i] = kNoKey;
    if (p.tiles_in_smem)
        for (uint32_t i = threadIdx.x; i < p.n_tiles; i += blockDim.x) hits[i] = p.tile_hits[i];
    if (threadIdx.x < 33) s_lev[threadIdx.x] = p.levels[threadIdx.x];
    if (threadIdx.x == 0) s_reps = 0;
    const uint32_t n = min(*p.cand_n, p.max_cand);
    constexpr int K = kPartMaxCand / 1024;
    uint32_t key[K], cnt[K];  // a candidate's bin and sample hits (at least two)
#pragma unroll
    for (int k = 0; k < K; ++k) {
        const uint32_t i = threadIdx.x + 1024u * k;
        const uint2 c = i < n ? p.cand[i] : make_uint2(kNoKey, 1u);
        key[k] = c.x;
        cnt[k] = c.y;
    }
    __syncthreads();
    const uint32_t shift = 32 - p.set_bits;
    uint32_t placed_mask = 0;
    const uint32_t total = s_lev[32];
    // a way holds bin | (group + 1) << 28 (bins are below 2^28)
    auto insert = [&](uint32_t bin, uint32_t v) {
        uint32_t *set = keys + 2 * (fib_hash(bin) >> shift);
        return atomicCAS(set, kNoKey, v) == kNoKey || atomicCAS(set + 1, kNoKey, v) == kNoKey;
    };
#pragma unroll
    for (int k = 0; k < K; ++k) {
        if (key[k] == kNoKey || (uint64_t)cnt[k] * 64 < (uint64_t)total) continue;
        const uint32_t g = atomicAdd(&s_reps, 1u);
        if (g < kPartReps && insert(key[k], key[k] | (g + 1) << 28)) placed_mask |= 1u << k;
    }
    __syncthreads();
    for (int l = 31; l >= 1; --l) {
        if (s_lev[l] == 0) continue;  // the same answer in every thread
#pragma unroll
        for (int k = 0; k < K; ++k) {
            if (1024u * k >= n) break;
            if (key[k] == kNoKey || 31 - __clz(cnt[k]) != l || (placed_mask >> k & 1u)) continue;
            if (insert(key[k], key[k])) placed_mask |= 1u << k;
        }
        __syncthreads();
    }
    uint32_t taken = 0;  // sample hits of the bins in the table
#pragma unroll
    for (int k = 0; k < K; ++k)
        if (placed_mask >> k & 1u) taken += cnt[k];
    const uint64_t hot = cta_sum(taken, s_sum);
    const bool use = hot * 16 >= total && hot > 0;
    if (threadIdx.x == 0) *p.n_hot = use ? 1u : 0u;
    for (uint32_t i = threadIdx.x; i < kPartReps * kPartRepCopies; i += blockDim.x) p.hot_keys[slots + i] = kNoKey;
    __syncthreads();
    for (uint32_t i = threadIdx.x; i < slots; i += blockDim.x) {
        const uint32_t v = keys[i], bin = v & 0x0FFFFFFFu, g = v >> 28;
        const bool have = use && v != kNoKey;
        p.hot_enc[i] = have ? fib_hash(bin) << p.set_bits | (g ? 1 + g : i & 1u) : kNoKey;
        p.hot_keys[i] = have && !g ? bin : kNoKey;
        if (have && g)
            for (uint32_t c = 0; c < kPartRepCopies; ++c) p.hot_keys[slots + (g - 1) * kPartRepCopies + c] = bin;
    }
    if (use) {
#pragma unroll
        for (int k = 0; k < K; ++k)
            if (placed_mask >> k & 1u) atomicSub(hits + (key[k] >> p.tile_bits), cnt[k]);
    }
    __syncthreads();
    const uint32_t S = 1u << (p.cb_shift - p.tile_bits);
    stretches(
        p.n_buckets,
        [&](uint32_t b) {
            uint32_t v = 0;
            for (uint32_t t = b * S; t < min((b + 1) * S, p.n_tiles); ++t) v += hits[t];
            return v;
        },
        p.entries_per_hit, p.region, room, p.base, nullptr, s_sum);
    if (p.split)
        stretches(p.n_tiles, [&](uint32_t t) { return hits[t]; }, p.entries_per_hit * (float)p.g_main, p.tile_room,
                  room, p.tile_base, p.tile_cur, s_sum);
}

// ---------------------------------------------------------------------------
// 3. Main pass.

namespace {

// Per-CTA state of the main pass, all in shared memory.
struct MainSmem {
    const uint32_t *enc;    // [slots] the hot table's entries
    uint32_t *sums;         // [slots + copies][2 directions] {count, byte sum low word, high word}
    uint32_t *cur;          // [n_buckets] next position of each range's run in the CTA's region
    const uint32_t *lim;    // [n_buckets] its end
    uint64_t *run;          // the CTA's region
    uint32_t slots, set_bits;
};

// An entry whose run is full: the shared list, positions claimed for all the
// lanes that are here at once. When the list is full too, nothing of the cold
// pass counts and the finishing kernel redoes the call (redo).
__device__ __noinline__ void cold_overflow(const PartDev &p, uint64_t e) {
    if (vload(p.redo)) return;
    const uint32_t m = __activemask(), lane = threadIdx.x & 31, lead = __ffs(m) - 1;
    uint32_t at = 0;
    if (lane == lead) at = atomicAdd(p.ovf_n, (uint32_t)__popc(m));
    at = __shfl_sync(m, at, lead) + __popc(m & ((1u << lane) - 1u));
    if (at < p.ovf_cap)
        p.ovf[at] = e;
    else
        *reinterpret_cast<volatile uint32_t *>(p.redo) = 1;
}

// Append one cold entry (key = bin << 1 | direction, the record's bytes) to
// the CTA's run of the bin's range: one shared-memory counter, one compare and
// one 8-byte store whose line collects 16 entries in L2.
__device__ __forceinline__ void cold_emit_entry(const PartDev &p, const MainSmem &m, uint64_t e) {
    const uint32_t bk = (uint32_t)(e >> 33) >> p.cb_shift;
    const uint32_t pos = atomicAdd(m.cur + bk, 1u);
    if (pos < m.lim[bk])
        m.run[pos] = e;
    else
        cold_overflow(p, e);
}

__device__ __forceinline__ void cold_emit(const PartDev &p, const MainSmem &m, uint32_t key, uint32_t by) {
    cold_emit_entry(p, m, (uint64_t)key << 32 | by);
}

// Hot slot of a bin, or kNoKey (see k_part_build).
__device__ __forceinline__ uint32_t hot_slot(const MainSmem &m, uint32_t bin) {
    const uint32_t hsh = fib_hash(bin), set = hsh >> (32 - m.set_bits), q = hsh << m.set_bits;
    const uint2 e = *reinterpret_cast<const uint2 *>(m.enc + 2 * set);
    const uint32_t x = min(e.x ^ q, e.y ^ q);
    const uint32_t slot = x < 2 ? 2 * set + x : m.slots + (x - 2) * kPartRepCopies + threadIdx.x % kPartRepCopies;
    return x < 2 + kPartReps ? slot : kNoKey;
}

__device__ __forceinline__ void hot_add(const MainSmem &m, uint32_t slot, uint32_t d, uint32_t by) {
    uint32_t *w = m.sums + 3 * (2 * slot + d);
    atomicAdd(w, 1u);
    smem_add_wide(w + 1, w + 2, by, 0u);
}

// One routed, in-window record: both directions share the bin's hot slot.
__device__ __forceinline__ void part_update(const PartDev &p, const MainSmem &m, bool hot, uint32_t bin,
                                            uint32_t dirs, uint32_t by) {
    const uint32_t slot = hot ? hot_slot(m, bin) : kNoKey;
    if (slot != kNoKey) {
        if (dirs & 1u) hot_add(m, slot, 0u, by);
        if (dirs & 2u) hot_add(m, slot, 1u, by);
        return;
    }
    if (dirs & 1u) cold_emit(p, m, bin << 1, by);
    if (dirs & 2u) cold_emit(p, m, bin << 1 | 1u, by);
}

template <bool W1>
__device__ __forceinline__ void part_record(const HistArgs &h, const PartDev &p, const MainSmem &m, bool hot, uint64_t ts,
                                            uint32_t by, uint32_t cls, uint64_t &ccp, uint32_t &oorp) {
    bump_class_packed(ccp, cls);
    const uint64_t rel = ts - h.t0;
    const bool inw = rel < h.span;
    const uint32_t bin = inw ? (W1 ? (uint32_t)rel : bin_of(h, rel)) : 0u;
    const uint32_t dirs = dirs_of_packed(h, cls, inw, oorp);
    if (dirs) part_update(p, m, hot, bin, dirs, by);
}

// First direction of a routed record: outgoing when its class routes there.
__device__ __forceinline__ uint32_t first_dir(uint32_t dirs) { return (dirs & 1u) ? 0u : 1u; }

__device__ __forceinline__ uint64_t cold_entry(uint32_t bin, uint32_t d, uint32_t by) {
    return (uint64_t)(bin << 1 | d) << 32 | by;
}

// Warp totals of 8-bit class counters and 16-bit out-of-window counters
// into the CTA's counters.
__device__ __forceinline__ void drain8(uint32_t &cc8, uint32_t &oorp, unsigned long long *s_cnt) {
    const uint32_t lane = threadIdx.x & 31;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        const uint32_t v = __reduce_add_sync(kFull, (cc8 >> (8 * k)) & 0xFFu);
        if (lane == 0 && v) atomicAdd(s_cnt + k, (unsigned long long)v);
    }
#pragma unroll
    for (int k = 0; k < 2; ++k) {
        const uint32_t v = __reduce_add_sync(kFull, (oorp >> (16 * k)) & 0xFFFFu);
        if (lane == 0 && v) atomicAdd(s_cnt + 4 + k, (unsigned long long)v);
    }
    cc8 = 0;
    oorp = 0;
}

}  // namespace

// One CTA per SM: warp 31 issues TMA bulk copies of stage after stage (a
// chunk of kPartStageRecords records of each stream: ts, src, dst, bytes);
// warps 0-30 take two records per thread from each stage, release it, and
// classify, bin and update. Chunks go to CTAs round-robin. With skewed input the
// pass is bound by instructions and shared-memory wavefronts (two stages, the
// rest of shared memory holds the hot table); with an empty table its room
// holds two more stages, since the pass then waits for its loads.
template <int LK, bool W1>
__global__ void __launch_bounds__(kPartThreads, 1) k_part_main(RecArgs r, TableArgs t, HistArgs h, PartDev p,
                                                               uint32_t *status) {
    extern __shared__ __align__(128) uint8_t smem[];
    __shared__ uint64_t tbar;
    __shared__ uint64_t full_bar[kPartMaxStages], empty_bar[kPartMaxStages];
    __shared__ unsigned long long s_cnt[6];
    __shared__ uint32_t s_abort;
    Classifier<LK> C;
    if (!C.init(t, smem, &tbar, status)) return;  // table not staged: the status word says so
    const uint32_t tsm = (Classifier<LK>::smem_bytes(t) + 127u) & ~127u;
    uint8_t *stage = smem + tsm;
    MainSmem m;
    m.set_bits = p.set_bits;
    m.slots = 2u << p.set_bits;
    m.run = p.entries + (uint64_t)blockIdx.x * p.region;
    const uint32_t n_sums = 2 * (m.slots + kPartReps * kPartRepCopies);
    // [table | stages | ranges' cursors and ends | hot table or more stages]
    m.cur = reinterpret_cast<uint32_t *>(stage + kPartStages * kPartStageBytes);
    uint32_t *lim = m.cur + p.n_buckets;
    m.lim = lim;
    uint8_t *extra = reinterpret_cast<uint8_t *>(m.cur) + ((8 * p.n_buckets + 127u) & ~127u);
    uint32_t *enc = reinterpret_cast<uint32_t *>(extra);
    m.enc = enc;
    m.sums = enc + m.slots;
    const bool hot = *p.n_hot != 0;  // the table holds bins: probe it
    const uint32_t n_stages =
        hot ? kPartStages : min(kPartMaxStages, kPartStages + (4 * m.slots + 12 * n_sums) / kPartStageBytes);
    auto stage_at = [&](uint32_t s) {
        return s < kPartStages ? stage + s * kPartStageBytes : extra + (s - kPartStages) * kPartStageBytes;
    };
    const uint32_t tid = threadIdx.x;
    if (hot) {
        for (uint32_t i = tid; i < m.slots; i += blockDim.x) enc[i] = p.hot_enc[i];
        for (uint32_t i = tid; i < 3 * n_sums; i += blockDim.x) m.sums[i] = 0;
    }
    for (uint32_t b = tid; b < p.n_buckets; b += blockDim.x) {
        m.cur[b] = p.base[b];
        lim[b] = p.base[b + 1];
    }
    if (tid < 6) s_cnt[tid] = 0;
    if (tid == 0) {
        s_abort = 0;
        for (uint32_t s = 0; s < kPartMaxStages; ++s) {
            mbar_init(smem_u32(&full_bar[s]), 1);
            mbar_init(smem_u32(&empty_bar[s]), kPartConsumers / 32);
        }
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    __syncthreads();

    const uint32_t warp = tid >> 5, lane = tid & 31;
    constexpr uint32_t R = kPartStageRecords;
    const uint32_t n_full = (uint32_t)p.n_full;  // records are below 2^32
    if (warp == kPartConsumers / 32) {
        // producer
        if (lane == 0) {
            uint32_t issued = 0, s = 0, turn = 0;  // turn: times round the ring
            for (uint32_t ch = blockIdx.x; ch < n_full; ch += gridDim.x) {
                if (turn && !mbar_wait(smem_u32(&empty_bar[s]), (turn - 1) & 1u)) {
                    latch_status(status, SINET_ERR_TIMEOUT);
                    *reinterpret_cast<volatile uint32_t *>(&s_abort) = 1;
                    break;
                }
                if (vload(&s_abort)) break;
                // the consumers' reads of this stage precede the copy's writes
                asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                const uint64_t i0 = p.i_lo + (uint64_t)ch * R;
                const uint32_t fb = smem_u32(&full_bar[s]);
                const uint32_t sb = smem_u32(stage_at(s));
                mbar_expect_tx(fb, kPartStageBytes);
                bulk_g2s(sb, r.ts + i0, 8 * R, fb);
                bulk_g2s(sb + 8 * R, r.src + i0, 4 * R, fb);
                bulk_g2s(sb + 12 * R, r.dst + i0, 4 * R, fb);
                bulk_g2s(sb + 16 * R, r.bytes + i0, 4 * R, fb);
                ++issued;
                if (++s == n_stages) {
                    s = 0;
                    ++turn;
                }
            }
            // every copy issued has landed before the CTA can exit
            for (uint32_t k = issued > n_stages ? issued - n_stages : 0; k < issued; ++k)
                mbar_wait(smem_u32(&full_bar[k % n_stages]), (k / n_stages) & 1u);
        }
    } else {
        uint32_t cc8 = 0;   // per-thread class counts, 8-bit fields
        uint32_t oorp = 0;  // per-thread out-of-window counts, 16-bit fields
        uint32_t since = 0, s = 0, phase = 0;
        // one stage per iteration: records 2 * tid and 2 * tid + 1 of the chunk
        static_assert(kPartRPT == 2, "two records per consumer thread and stage");
        for (uint32_t ch = blockIdx.x; ch < n_full; ch += gridDim.x) {
            uint64_t ts[2] = {0, 0};
            uint32_t a[4] = {0, 0, 0, 0}, by[2] = {0, 0};  // a: src, dst of record 0, then of record 1
            const bool ok = __all_sync(kFull, mbar_wait(smem_u32(&full_bar[s]), phase));
            if (ok) {
                const uint8_t *sp = stage_at(s);
                const uint4 t2 = *reinterpret_cast<const uint4 *>(sp + 16 * tid);
                const uint2 s2 = *reinterpret_cast<const uint2 *>(sp + 8 * R + 8 * tid);
                const uint2 d2 = *reinterpret_cast<const uint2 *>(sp + 12 * R + 8 * tid);
                const uint2 b2 = *reinterpret_cast<const uint2 *>(sp + 16 * R + 8 * tid);
                ts[0] = (uint64_t)t2.y << 32 | t2.x;
                ts[1] = (uint64_t)t2.w << 32 | t2.z;
                a[0] = s2.x;
                a[1] = d2.x;
                a[2] = s2.y;
                a[3] = d2.y;
                by[0] = b2.x;
                by[1] = b2.y;
                __syncwarp();
                if (lane == 0) mbar_arrive(smem_u32(&empty_bar[s]));
            }
            if (!ok) {
                if (lane == 0) {
                    latch_status(status, SINET_ERR_TIMEOUT);
                    *reinterpret_cast<volatile uint32_t *>(&s_abort) = 1;
                }
                break;
            }
            if (++s == n_stages) {
                s = 0;
                phase ^= 1u;
            }
            uint32_t in[4];
            C.template in_n_warp<4>(a, in);  // the warp is converged here
            uint32_t bin[2], dirs[2], slot[2];
            bool out[2];
#pragma unroll
            for (int j = 0; j < 2; ++j) {
                const uint32_t cls8 = 8 * (in[2 * j] | in[2 * j + 1] << 1);
                cc8 += 1u << cls8;
                const uint64_t rel = ts[j] - h.t0;
                out[j] = rel >= h.span;
                bin[j] = W1 ? (uint32_t)rel : bin_of(h, rel);
                dirs[j] = (h.policy >> cls8) & 3u;
            }
            if (__any_sync(kFull, out[0] || out[1])) {  // records outside the window are the exception
#pragma unroll
                for (int j = 0; j < 2; ++j)
                    if (out[j]) {
                        oorp += (dirs[j] & 1u) | ((dirs[j] >> 1) << 16);
                        dirs[j] = 0;
                    }
            }
#pragma unroll
            for (int j = 0; j < 2; ++j) slot[j] = hot && dirs[j] ? hot_slot(m, bin[j]) : kNoKey;
            // hot bins, first direction: one shared-memory add per record
#pragma unroll
            for (int j = 0; j < 2; ++j)
                if (slot[j] != kNoKey) hot_add(m, slot[j], first_dir(dirs[j]), by[j]);
            // classes routed to both directions: the second one
            if (h.two_dir && __any_sync(kFull, dirs[0] == 3u || dirs[1] == 3u)) {
#pragma unroll
                for (int j = 0; j < 2; ++j) {
                    if (dirs[j] != 3u) continue;
                    if (slot[j] != kNoKey) hot_add(m, slot[j], 1u, by[j]);
                    else cold_emit_entry(p, m, cold_entry(bin[j], 1u, by[j]));
                }
            }
            // cold bins, first direction: each lane appends its own entries (a
            // gather of the warp's entries onto its lanes first costs more
            // instructions than the second append it saves)
#pragma unroll
            for (int j = 0; j < 2; ++j)
                if (dirs[j] && slot[j] == kNoKey) cold_emit_entry(p, m, cold_entry(bin[j], first_dir(dirs[j]), by[j]));
            // at most two records per field per iteration: drain before 8 bits fill
            if (++since == 127) {
                drain8(cc8, oorp, s_cnt);
                since = 0;
            }
        }
        uint64_t ccp = 0;  // the records outside the staged chunks: 16-bit class fields
        // records outside the staged chunks, one by one
        const uint64_t tail_lo = p.i_lo + p.n_full * R;
        const uint64_t n_scalar = p.n_head + (r.g.n - tail_lo);
        for (uint64_t k = (uint64_t)blockIdx.x * kPartConsumers + tid; k < n_scalar;
             k += (uint64_t)gridDim.x * kPartConsumers) {
            const uint64_t i = k < p.n_head ? k : tail_lo + (k - p.n_head);
            uint32_t a[1] = {r.src[i]}, in_s[1], in_d[1];
            C.template in_n<1>(a, in_s);
            a[0] = r.dst[i];
            C.template in_n<1>(a, in_d);
            part_record<W1>(h, p, m, hot, r.ts[i], r.bytes[i], in_s[0] | in_d[0] << 1, ccp, oorp);
        }
        __syncwarp();
        drain_packed(ccp, oorp, s_cnt);
        drain8(cc8, oorp, s_cnt);
    }
    __syncthreads();

    // class and out-of-window counters
    if (tid < 6 && s_cnt[tid]) atomicAdd(reinterpret_cast<unsigned long long *>(h.stats) + tid, s_cnt[tid]);
    // this CTA's share of the hot table
    for (uint32_t i = tid; hot && i < n_sums; i += blockDim.x) {
        const uint32_t c = m.sums[3 * i];
        if (c) {
            red_add_u32(p.hot_cnt + i, c);
            red_add_u64(p.hot_bytes + i, (uint64_t)m.sums[3 * i + 2] << 32 | m.sums[3 * i + 1]);
        }
    }
    // the entries of its runs
    for (uint32_t b = tid; b < p.n_buckets; b += blockDim.x)
        p.counts[(uint64_t)b * p.g_main + blockIdx.x] = min(m.cur[b], lim[b]) - p.base[b];
}

// ---------------------------------------------------------------------------
// 4. Split: the entries of every run go on to the run of their tile. The main
// pass writes to few ranges (at most kPartMaxRuns), because every one of them is
// a half-written L2 line in each of its CTAs: with 165, 340, 660, 1,320 and 2,640
// ranges it takes 7.0, 7.2, 7.8, 8.6 and 10.2 ms on the heavy day, the last with
// 7.5 GB of DRAM traffic from lines evicted before they were full. A range of
// up to 64 tiles is then split here, where the warps at work at one time write
// to the tiles of a few ranges only.
//
// A warp works alone, without CTA barriers, on blocks of 512 entries: it ranks
// them per tile with its own counters in shared memory, sorts them there, claims
// room in each tile's run (one global atomic per tile and block) and writes
// them in order. (Sorting 2,048-entry pages in place under CTA barriers, for
// owners that gathered their shares of every page, took the larger part of the
// 3.55 ms that the cold pass of the heavy day's 400 M entries used to take;
// split and tiles together now take 3.0 ms.)
namespace {

constexpr uint32_t kSplitThreads = 768;  // 24 warps of up to 85 registers
constexpr uint32_t kSplitBlock = 512;    // entries a warp sorts at a time
constexpr uint32_t kSplitSubs = 64;      // tiles of a range at most
constexpr uint32_t kSplitShare = 4;      // warps that share a run
constexpr size_t kSplitWarpBytes = 8 * kSplitBlock + 12 * kSplitSubs;

constexpr uint32_t kColdThreads = 1024;
constexpr uint32_t kColdRuns = 5;   // runs a warp has in flight
constexpr uint32_t kColdAhead = 6;  // entries a thread loads ahead of its CTA's next tile

__device__ __forceinline__ uint64_t ld_entry(const uint64_t *p) {
    return __ldcs(reinterpret_cast<const unsigned long long *>(p));
}

// First of c places in tile t's run (at its end or beyond: the run is full).
// Where all updates in one tile could carry its 32-bit cursor round (split 2),
// a full run's cursor is left alone.
__device__ __forceinline__ uint32_t split_claim(const PartDev &p, uint32_t t, uint32_t c, uint32_t end) {
    if (p.split == 2 && vload(p.tile_cur + t) >= end) return end;
    return atomicAdd(p.tile_cur + t, c);
}

}  // namespace

__global__ void __launch_bounds__(kSplitThreads, 1) k_part_split(PartDev p) {
    extern __shared__ __align__(16) uint8_t smem[];
    const uint32_t warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    uint64_t *buf = reinterpret_cast<uint64_t *>(smem + warp * kSplitWarpBytes);
    uint32_t *cnt = reinterpret_cast<uint32_t *>(buf + kSplitBlock);  // per tile: entries, then their first place
    uint32_t *dst = cnt + kSplitSubs;                                  // place in the tile's run minus place in buf
    uint32_t *lim = dst + kSplitSubs;                                  // end of the tile's run
    constexpr int U = kSplitBlock / 32;
    const uint32_t G = p.g_main, sh = p.tile_bits + 1, S = 1u << (p.cb_shift - p.tile_bits);
    const uint64_t units = (uint64_t)p.n_buckets * G * kSplitShare;
    for (uint64_t u = (uint64_t)blockIdx.x * (kSplitThreads / 32) + warp; u < units;
         u += (uint64_t)gridDim.x * (kSplitThreads / 32)) {
        const uint32_t run = (uint32_t)(u / kSplitShare), r = run / G, c = run - r * G;
        const uint32_t n = p.counts[run];
        const uint64_t *src = p.entries + (uint64_t)c * p.region + p.base[r];
        const uint32_t t0 = r * S;
        for (uint32_t at = (uint32_t)(u % kSplitShare) * kSplitBlock; at < n; at += kSplitShare * kSplitBlock) {
            const uint32_t m = min(n - at, kSplitBlock);
            cnt[lane] = 0;
            cnt[lane + 32] = 0;
            uint64_t e[U];
            uint32_t pos[U];  // tile << 16 | rank among the tile's entries
#pragma unroll
            for (int j = 0; j < U; ++j)
                if (j * 32 < m) e[j] = j * 32 + lane < m ? ld_entry(src + at + j * 32 + lane) : 0ull;
            __syncwarp();
#pragma unroll
            for (int j = 0; j < U; ++j) {
                if (j * 32 >= m) break;  // the whole warp
                pos[j] = ((uint32_t)(e[j] >> 32) >> sh) - t0;
                if (j * 32 + lane < m) pos[j] = pos[j] << 16 | atomicAdd(cnt + pos[j], 1u);
            }
            __syncwarp();
            // each lane: two neighbouring tiles
            const uint32_t c0 = cnt[2 * lane], c1 = cnt[2 * lane + 1];
            uint32_t incl = c0 + c1;
#pragma unroll
            for (int d = 1; d < 32; d <<= 1) {
                const uint32_t y = __shfl_up_sync(kFull, incl, d);
                if (lane >= (uint32_t)d) incl += y;
            }
            const uint32_t o0 = incl - c0 - c1, o1 = incl - c1;
            cnt[2 * lane] = o0;  // (its own two words: nobody else reads them before the __syncwarp)
            cnt[2 * lane + 1] = o1;
            bool fits = true;
            if (c0) {
                const uint32_t t = t0 + 2 * lane, end = p.tile_base[t + 1], q = split_claim(p, t, c0, end);
                lim[2 * lane] = end;
                dst[2 * lane] = q - o0;
                fits = q <= end && end - q >= c0;
            }
            if (c1) {
                const uint32_t t = t0 + 2 * lane + 1, end = p.tile_base[t + 1], q = split_claim(p, t, c1, end);
                lim[2 * lane + 1] = end;
                dst[2 * lane + 1] = q - o1;
                fits = fits && q <= end && end - q >= c1;
            }
            fits = __all_sync(kFull, fits);
            __syncwarp();  // every lane's cnt before the scatter reads them (a vote orders no memory)
#pragma unroll
            for (int j = 0; j < U; ++j) {
                if (j * 32 >= m) break;
                if (j * 32 + lane < m) buf[cnt[pos[j] >> 16] + (pos[j] & 0xFFFFu)] = e[j];
            }
            __syncwarp();
            if (fits) {
#pragma unroll 8
                for (uint32_t i = lane; i < m; i += 32) {
                    const uint64_t v = buf[i];
                    p.tile_entries[dst[((uint32_t)(v >> 32) >> sh) - t0] + i] = v;
                }
            } else {
                for (uint32_t i = lane; i < m; i += 32) {
                    const uint64_t v = buf[i];
                    const uint32_t k = ((uint32_t)(v >> 32) >> sh) - t0, q = dst[k] + i;
                    if (q < lim[k])
                        p.tile_entries[q] = v;
                    else
                        cold_overflow(p, v);
                }
            }
            __syncwarp();
        }
    }
}

// 5. Tiles: each CTA takes tile after tile of 2^tile_bits bins, sums the tile's
// entries in shared memory and stores every bin once. After a split they are
// the tile's own run. Without one they lie in the runs of the tile's range (of
// at most eight tiles), a run per CTA of the main pass, which each of the
// range's tiles reads for itself; warp w then takes runs w, w + 32, ...: their
// counts in one step, the first 64 entries of all of them in flight together
// (runs are short where the input is small), then what is left of each.
namespace {

// The entry's update if its bin lies in the tile: [6][T] words, counts of
// directions 0 and 1, byte sums' low words of both, high words of both.
__device__ __forceinline__ void tile_add(uint32_t *tile, uint32_t T, uint32_t lo_key, uint64_t e) {
    const uint32_t k = (uint32_t)(e >> 32) - lo_key;  // (bin - first bin) << 1 | direction
    if (k >= 2 * T) return;
    uint32_t *w = tile + (k & 1u) * T + (k >> 1);
    atomicAdd(w, 1u);
    smem_add_wide(w + 2 * T, w + 4 * T, (uint32_t)e, 0u);
}

}  // namespace

__global__ void __launch_bounds__(kColdThreads, 1) k_part_cold(HistArgs h, PartDev p, uint32_t accumulate) {
    extern __shared__ __align__(128) uint8_t smem[];
    uint32_t *tile = reinterpret_cast<uint32_t *>(smem);
    const uint32_t T = 1u << p.tile_bits, G = p.g_main;
    const uint32_t warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    constexpr uint64_t kNone = ~0ull;  // not an entry: bins are below 2^28
    for (uint32_t i = threadIdx.x; i < 6 * T; i += kColdThreads) tile[i] = 0;
    const bool redo = *p.redo != 0;  // the tiles stay empty: zeros stored, or nothing added
    __syncthreads();
    // a tile's own run (split): its first entries are loaded while the tile
    // before it is stored
    uint64_t ahead[kColdAhead];
    uint32_t n_run = 0;
    const uint64_t *run = p.tile_entries;
    auto start_run = [&](uint32_t t) {
        if (!p.split || redo || t >= p.n_tiles) return;
        const uint32_t at = p.tile_base[t];
        n_run = min(p.tile_cur[t], p.tile_base[t + 1]) - at;
        run = p.tile_entries + at;
#pragma unroll
        for (uint32_t u = 0; u < kColdAhead; ++u)
            ahead[u] = threadIdx.x + u * kColdThreads < n_run ? ld_entry(run + threadIdx.x + u * kColdThreads) : kNone;
    };
    start_run(blockIdx.x);
    for (uint32_t t = blockIdx.x; t < p.n_tiles; t += gridDim.x) {
        const uint32_t lo_key = t << (p.tile_bits + 1);
        if (redo) {
        } else if (p.split) {
#pragma unroll
            for (uint32_t u = 0; u < kColdAhead; ++u) tile_add(tile, T, lo_key, ahead[u]);
            for (uint32_t i = threadIdx.x + kColdAhead * kColdThreads; i < n_run; i += 8 * kColdThreads) {
                uint64_t f[8];
#pragma unroll
                for (int u = 0; u < 8; ++u)
                    f[u] = i + u * kColdThreads < n_run ? ld_entry(run + i + u * kColdThreads) : kNone;
#pragma unroll
                for (int u = 0; u < 8; ++u) tile_add(tile, T, lo_key, f[u]);
            }
        } else {
            const uint32_t b = t >> (p.cb_shift - p.tile_bits);
            const uint64_t *runs = p.entries + p.base[b];
            const uint32_t *counts = p.counts + (uint64_t)b * G;
            for (uint32_t g0 = warp; g0 < G; g0 += 32 * kColdRuns) {
                uint32_t n[kColdRuns];
                uint64_t e[kColdRuns][2];
#pragma unroll
                for (uint32_t r = 0; r < kColdRuns; ++r) n[r] = g0 + 32 * r < G ? counts[g0 + 32 * r] : 0u;
#pragma unroll
                for (uint32_t r = 0; r < kColdRuns; ++r) {
                    const uint64_t *q = runs + (uint64_t)(g0 + 32 * r) * p.region;
                    e[r][0] = lane < n[r] ? ld_entry(q + lane) : kNone;
                    e[r][1] = lane + 32 < n[r] ? ld_entry(q + lane + 32) : kNone;
                }
#pragma unroll
                for (uint32_t r = 0; r < kColdRuns; ++r) {
                    tile_add(tile, T, lo_key, e[r][0]);
                    tile_add(tile, T, lo_key, e[r][1]);
                    const uint64_t *q = runs + (uint64_t)(g0 + 32 * r) * p.region;
                    for (uint32_t i = 64 + lane; i < n[r]; i += 256) {
                        uint64_t f[8];
#pragma unroll
                        for (int u = 0; u < 8; ++u) f[u] = i + 32 * u < n[r] ? ld_entry(q + i + 32 * u) : kNone;
#pragma unroll
                        for (int u = 0; u < 8; ++u) tile_add(tile, T, lo_key, f[u]);
                    }
                }
            }
        }
        __syncthreads();
        start_run(t + gridDim.x);
        const uint64_t lo_bin = (uint64_t)t << p.tile_bits;
        const uint32_t nb = (uint32_t)min((uint64_t)T, (uint64_t)h.n_bins - lo_bin);
        for (uint32_t i = threadIdx.x; i < nb; i += kColdThreads) {
            const uint64_t bin = lo_bin + i;
            const uint32_t c0 = tile[i], c1 = tile[T + i];
            const uint64_t s0 = (uint64_t)tile[4 * T + i] << 32 | tile[2 * T + i];
            const uint64_t s1 = (uint64_t)tile[5 * T + i] << 32 | tile[3 * T + i];
#pragma unroll
            for (uint32_t k = 0; k < 6; ++k) tile[k * T + i] = 0;  // ready for the next tile
            // added with reductions, since calls on other streams may be adding to
            // the same outputs, and only where the tile has updates (all bins read,
            // added and stored took 1,238 us for 30 M records into 86.4 M bins, this
            // 911; 20 M into 10 M 427, 400; 200 M skewed into 86.4 M 2,080, 1,706)
            if (accumulate) {
                if (c0) gadd(h, 0u, bin, c0, s0);
                if (c1) gadd(h, 1u, bin, c1, s1);
                continue;
            }
            h.cnt[0][bin] = c0;
            h.cnt[1][bin] = c1;
            h.byt[0][bin] = s0;
            h.byt[1][bin] = s1;
        }
        __syncthreads();  // every bin stored and zeroed before the next tile's adds
    }
}

// 6. Finish: the hot totals (a bin's copies sit in several slots, so the adds
// are reductions) and the overflow list into their bins. When the list itself
// was full (redo: the sample missed the distribution badly), the cold pass
// stored empty tiles and every record is added here instead, with one
// reduction each; the class and window counters stand from the main pass.
template <int LK>
__global__ void __launch_bounds__(256) k_part_finish(RecArgs r, TableArgs t, HistArgs h, PartDev p, uint32_t slots,
                                                     uint32_t *status) {
    extern __shared__ __align__(16) uint8_t smem[];
    __shared__ uint64_t bar;
    const uint32_t tid = blockIdx.x * blockDim.x + threadIdx.x, threads = gridDim.x * blockDim.x;
    if (*p.redo) {
        Classifier<LK> C;
        if (!C.init(t, smem, &bar, status)) return;  // table not staged: the status word says so
        const uint64_t pol = policy_evict_first();
        uint32_t oor[2] = {0, 0};
        for (uint64_t q = tid; q < r.g.quads; q += threads) {
            Quad Q;
            load_quad<true, true, true, false>(r, q, pol, Q);
            classify_quad<LK>(C, Q);
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                if (!(Q.valid >> j & 1u)) continue;
                uint32_t bin;
                const uint32_t dirs = route(h, Q.cls[j], Q.ts[j], bin, oor);
                if (dirs & 1u) gadd(h, 0, bin, 1u, Q.by[j]);
                if (dirs & 2u) gadd(h, 1, bin, 1u, Q.by[j]);
            }
        }
        return;
    }
    for (uint32_t i = tid; i < slots + kPartReps * kPartRepCopies; i += threads) {
        const uint32_t key = p.hot_keys[i];
        if (key == kNoKey || key >= h.n_bins) continue;
#pragma unroll
        for (uint32_t d = 0; d < 2; ++d) {
            const uint32_t c = p.hot_cnt[2 * i + d];
            if (c) gadd(h, d, key, c, p.hot_bytes[2 * i + d]);
        }
    }
    const uint32_t n = min(*p.ovf_n, p.ovf_cap);
    for (uint32_t i = tid; i < n; i += threads) {
        const uint64_t e = p.ovf[i];
        gadd(h, (uint32_t)(e >> 32) & 1u, (uint32_t)(e >> 33), 1u, (uint32_t)e);
    }
}

// ---------------------------------------------------------------------------
// Host side.

namespace {

uint32_t ceil_log2(uint64_t x) {
    uint32_t l = 0;
    while ((1ull << l) < x) ++l;
    return l;
}

size_t align256(size_t x) { return (x + 255) & ~(size_t)255; }

}  // namespace

Divider make_divider(uint64_t w);  // api.cu

static size_t main_smem(uint32_t tsm, uint32_t slots, uint32_t n_buckets) {
    return ((size_t)(tsm + 127u) & ~(size_t)127u) + (size_t)kPartStages * kPartStageBytes + 28ull * slots +
           24ull * kPartReps * kPartRepCopies + ((8ull * n_buckets + 127u) & ~127ull);
}

cudaError_t plan_partition(int lk, uint32_t table_smem, const RecArgs &r, const HistArgs &h, uint32_t bucket_bits,
                           int sm_count, size_t smem_optin, bool lean, PartPlan *out) {
    PartPlan P{};
    PartDev &d = P.d;
    if (lk == LK_CLASS_IN || sm_count <= 0) return cudaErrorNotSupported;
    const uint64_t n = r.g.n;
    const uint64_t routed_max = n * (h.two_dir ? 2ull : 1ull);
    if (routed_max >= 0xFFFFF000ull) return cudaErrorNotSupported;  // u32 positions
    if (h.n_bins > (1u << 28)) return cudaErrorNotSupported;
    const uint32_t G = (uint32_t)sm_count;
    // tiles: 2^13 bins (24 bytes each) fill an SM's shared memory; fewer where
    // that would leave SMs without a tile
    uint32_t tb = kPartTileBits;
    while (tb > 8 && ((h.n_bins - 1) >> tb) + 1 < 2 * G) --tb;
    const uint32_t tiles = ((h.n_bins - 1) >> tb) + 1;
    // ranges of 2^k tiles, at most kPartMaxRuns of them, and no more than give
    // runs of 48 entries (the cold pass loads 64 of a run in its first step).
    // Up to four tiles a range are summed straight from the range's runs, each
    // tile reading them all; more are split first, if the split's room may be
    // allocated (lean: it may not, and ranges stay at eight tiles).
    auto ranges = [&](uint32_t cb) { return ((h.n_bins - 1) >> cb) + 1; };
    uint32_t cb = tb;
    if (bucket_bits) {
        cb = std::min(std::max(bucket_bits, tb), tb + 3);
    } else {
        while (cb < tb + 2 && (ranges(cb) > kPartMaxRuns || n / ((uint64_t)G * ranges(cb)) < 48)) ++cb;
        const uint64_t room = routed_max + routed_max / 4 + std::min<uint64_t>(routed_max, 40000000ull) + 32ull * tiles;
        if (ranges(cb) > kPartMaxRuns + kPartMaxRuns / 2 && !lean && room < 0xFE000000ull) {
            while (cb < tb + 6 && ranges(cb) > kPartMaxRuns) ++cb;
            // (a warp in flight adds at most 512 to a cursor before it sees it full)
            d.split = room + routed_max + (1u << 24) < (1ull << 32) ? 1 : 2;
            d.tile_room = room;
        }
    }
    while (!d.split && cb < tb + 3 && ranges(cb) > 12 * kPartMaxRuns) ++cb;
    const uint32_t nb = ranges(cb);
    P.smem_cold = 24ull << tb;
    if (P.smem_cold + 1024 > smem_optin) return cudaErrorNotSupported;
    // hot table: as many sets of two as shared memory allows (at least 2^5)
    const uint32_t tsm = (table_smem + 127u) & ~127u;
    uint32_t sb = 13;
    while (sb > 5 && main_smem(tsm, 2u << sb, nb) + 1024 > smem_optin) --sb;
    if (main_smem(tsm, 2u << sb, nb) + 1024 > smem_optin) return cudaErrorNotSupported;
    P.slots = 2u << sb;
    P.smem_main = main_smem(tsm, P.slots, nb);
    P.smem_split = (kSplitThreads / 32) * kSplitWarpBytes;
    // sample: about n / 4096 records (at least 2^16 and 40 a tile, at most 2^20
    // or a sixteenth), in chunks: a bin holding 1 / 4,096 of the updates (a
    // slot's share of the table) gets at least a dozen hits
    const uint64_t chunks = (n + kPartSampleChunk - 1) / kPartSampleChunk;
    const uint64_t target = std::min<uint64_t>(n, std::min<uint64_t>({1ull << 20, std::max<uint64_t>(1ull << 16, n / 16), std::max<uint64_t>({1ull << 16, n >> 12, 40ull * tiles})}));
    uint64_t stride = target ? (chunks * kPartSampleChunk) / target : 1;
    if (stride < 1) stride = 1;
    const uint64_t s_chunks = (chunks + stride - 1) / stride;
    uint32_t hb = ceil_log2(2 * s_chunks * kPartSampleChunk);
    hb = std::min(23u, std::max(10u, hb));
    // records staged by TMA: from the first index at which all four streams
    // are 16-byte aligned, in whole stages
    if (r.g.vec) {
        const uint64_t i_lo = r.g.shift < 0 ? (uint64_t)(r.g.shift + 4) : 0ull;
        d.i_lo = std::min<uint64_t>(i_lo, n);
        d.n_full = n > d.i_lo ? (n - d.i_lo) / kPartStageRecords : 0;
        d.n_head = d.i_lo;
    } else {
        d.i_lo = 0;
        d.n_full = 0;
        d.n_head = 0;
    }
    d.set_bits = sb;
    d.cb_shift = cb;
    d.n_buckets = nb;
    d.g_main = G;
    d.tile_bits = tb;
    d.n_tiles = tiles;
    d.max_cand = std::min(kPartMaxCand, 2 * P.slots);
    d.hash_mask = (1u << hb) - 1u;
    d.hash_shift = 32 - hb;
    d.sample_chunks = s_chunks;
    d.sample_stride = stride;
    // a CTA's region: its share of every routed update and a quarter, more for
    // small inputs (whose sample is coarse), and a line per range. The overflow
    // list: a sixteenth of the routed updates
    d.entries_per_hit = (float)((double)n / (double)std::max<uint64_t>(1, std::min<uint64_t>(n, s_chunks * kPartSampleChunk)) / G);
    const uint64_t slack = std::min<uint64_t>(routed_max, 40000000ull);
    d.region = ((routed_max + routed_max / 8 + slack) / G + 64ull * nb + 15) & ~15ull;
    if (d.region >= 0xFFFFFF00ull) return cudaErrorNotSupported;
    d.ovf_cap = (uint32_t)(routed_max / 16 + 65536);
    P.grid_main = G;
    P.grid_sample = G;
    P.grid_cold = (int)std::min<uint32_t>(tiles, G);
    P.smem_build = 4ull * P.slots + 8ull * tiles;
    d.tiles_in_smem = P.smem_build + 1024 <= smem_optin;
    if (!d.tiles_in_smem) P.smem_build = 4ull * P.slots;
    P.smem_sample = ((table_smem + 15u) & ~15u) + (size_t)HotCache::kSlotBytes * (HotCache::kWays << kPartSampleSetBits);
    P.smem_finish = (table_smem + 15u) & ~15u;
    // scratch layout
    size_t o = 0;
    P.off_ff = o;
    P.off_hash_keys = o;
    o = align256(o + (4ull << hb));
    P.bytes_ff = o - P.off_ff;
    const uint64_t sums = 2ull * (P.slots + kPartReps * kPartRepCopies);
    P.off_hot_enc = o;
    o = align256(o + 4ull * P.slots);
    P.off_hot_keys = o;
    o = align256(o + 2ull * sums);
    P.off_zero = o;
    P.off_levels = o;
    o = align256(o + 4ull * 33);
    P.off_words = o;  // cand_n, n_hot, ovf_n, redo
    o = align256(o + 16);
    P.off_hot_cnt = o;
    o = align256(o + 4ull * sums);
    P.off_hot_bytes = o;
    o = align256(o + 8ull * sums);
    P.off_tile_hits = o;
    o = align256(o + 4ull * tiles);
    P.off_hash_cnt = o;
    o = align256(o + (4ull << hb));
    // zero, since a CTA whose table did not land leaves the main pass without
    // storing its counts: its runs are then empty, and nothing reads beyond them
    P.off_counts = o;
    o = align256(o + 4ull * nb * G);
    P.bytes_zero = o - P.off_zero;
    P.off_cand = o;
    o = align256(o + 8ull * kPartMaxCand);
    P.off_base = o;
    o = align256(o + 4ull * (nb + 1));
    P.off_tile_base = o;
    o = align256(o + 4ull * (tiles + 1));
    P.off_tile_cur = o;
    o = align256(o + 4ull * tiles);
    P.off_ovf = o;
    o = align256(o + 8ull * d.ovf_cap);
    P.off_entries = o;
    o = align256(o + 8ull * d.region * G);
    P.off_tile_entries = o;
    o = align256(o + 8ull * d.tile_room);
    P.scratch_bytes = o;
    *out = P;
    return cudaSuccess;
}

template <typename K>
static cudaError_t set_smem(K kernel, size_t smem) {
    return raise_smem_limit((const void *)kernel, smem);
}

template <int LK>
static cudaError_t launch_lk(const RecArgs &r, const TableArgs &t, const HistArgs &h, const PartPlan &P,
                             bool accumulate, const LaunchCfg &c) {
    cudaError_t e;
    if ((e = set_smem(k_part_sample<LK>, P.smem_sample)) != cudaSuccess) return e;
    k_part_sample<LK><<<P.grid_sample, kPartSampleThreads, P.smem_sample, c.stream>>>(r, t, h, P.d, c.status);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    const int scan_grid = std::min<int>(2 * P.grid_main, (int)((P.d.hash_mask + 1023) / 1024) + 1);
    k_part_levels<<<scan_grid, 256, 0, c.stream>>>(P.d);
    k_part_collect<<<scan_grid, 256, 0, c.stream>>>(P.d);
    if ((e = set_smem(k_part_build, P.smem_build)) != cudaSuccess) return e;
    k_part_build<<<1, 1024, P.smem_build, c.stream>>>(P.d, P.slots);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    if (h.w_is_one) {
        if ((e = set_smem(k_part_main<LK, true>, P.smem_main)) != cudaSuccess) return e;
        k_part_main<LK, true><<<P.grid_main, kPartThreads, P.smem_main, c.stream>>>(r, t, h, P.d, c.status);
    } else {
        if ((e = set_smem(k_part_main<LK, false>, P.smem_main)) != cudaSuccess) return e;
        k_part_main<LK, false><<<P.grid_main, kPartThreads, P.smem_main, c.stream>>>(r, t, h, P.d, c.status);
    }
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    if (P.d.split) {
        if ((e = set_smem(k_part_split, P.smem_split)) != cudaSuccess) return e;
        k_part_split<<<P.grid_main, kSplitThreads, P.smem_split, c.stream>>>(P.d);
        if ((e = cudaGetLastError()) != cudaSuccess) return e;
    }
    if ((e = set_smem(k_part_cold, P.smem_cold)) != cudaSuccess) return e;
    k_part_cold<<<P.grid_cold, kColdThreads, P.smem_cold, c.stream>>>(h, P.d, accumulate ? 1u : 0u);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    if ((e = set_smem(k_part_finish<LK>, P.smem_finish)) != cudaSuccess) return e;
    k_part_finish<LK><<<P.grid_main, 256, P.smem_finish, c.stream>>>(r, t, h, P.d, P.slots, c.status);
    return cudaGetLastError();
}

cudaError_t run_partition(int lk, const RecArgs &r, const TableArgs &t, const HistArgs &h, PartPlan P,
                          void *scratch, bool accumulate, const LaunchCfg &c) {
    uint8_t *base = static_cast<uint8_t *>(scratch);
    PartDev &d = P.d;
    d.hash_keys = reinterpret_cast<uint32_t *>(base + P.off_hash_keys);
    d.hash_cnt = reinterpret_cast<uint32_t *>(base + P.off_hash_cnt);
    d.levels = reinterpret_cast<uint32_t *>(base + P.off_levels);
    uint32_t *words = reinterpret_cast<uint32_t *>(base + P.off_words);
    d.cand_n = words;
    d.n_hot = words + 1;
    d.ovf_n = words + 2;
    d.redo = words + 3;
    d.cand = reinterpret_cast<uint2 *>(base + P.off_cand);
    d.hot_enc = reinterpret_cast<uint32_t *>(base + P.off_hot_enc);
    d.hot_keys = reinterpret_cast<uint32_t *>(base + P.off_hot_keys);
    d.hot_cnt = reinterpret_cast<uint32_t *>(base + P.off_hot_cnt);
    d.hot_bytes = reinterpret_cast<uint64_t *>(base + P.off_hot_bytes);
    d.tile_hits = reinterpret_cast<uint32_t *>(base + P.off_tile_hits);
    d.tile_base = reinterpret_cast<uint32_t *>(base + P.off_tile_base);
    d.tile_cur = reinterpret_cast<uint32_t *>(base + P.off_tile_cur);
    d.tile_entries = reinterpret_cast<uint64_t *>(base + P.off_tile_entries);
    d.base = reinterpret_cast<uint32_t *>(base + P.off_base);
    d.counts = reinterpret_cast<uint32_t *>(base + P.off_counts);
    d.ovf = reinterpret_cast<uint64_t *>(base + P.off_ovf);
    d.entries = reinterpret_cast<uint64_t *>(base + P.off_entries);
    cudaError_t e;
    if ((e = cudaMemsetAsync(base + P.off_ff, 0xFF, P.bytes_ff, c.stream)) != cudaSuccess) return e;
    if ((e = cudaMemsetAsync(base + P.off_zero, 0, P.bytes_zero, c.stream)) != cudaSuccess) return e;
    switch (lk) {
        case LK_INTERVAL: e = launch_lk<LK_INTERVAL>(r, t, h, P, accumulate, c); break;
        case LK_LEAF2: e = launch_lk<LK_LEAF2>(r, t, h, P, accumulate, c); break;
        case LK_LEAF4: e = launch_lk<LK_LEAF4>(r, t, h, P, accumulate, c); break;
        case LK_TOGGLE2: e = launch_lk<LK_TOGGLE2>(r, t, h, P, accumulate, c); break;
        case LK_PML: e = launch_lk<LK_PML>(r, t, h, P, accumulate, c); break;
        case LK_INTERVAL_GLOBAL: e = launch_lk<LK_INTERVAL_GLOBAL>(r, t, h, P, accumulate, c); break;
        default: return cudaErrorInvalidValue;
    }
    return e;
}

}  // namespace sinet

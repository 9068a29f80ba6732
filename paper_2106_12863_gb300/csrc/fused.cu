// Discriminate-only and fused discriminate + histogram kernels (sm_103a).
//
// One pass over the SoA records: 128-bit streaming loads of 4 records per
// thread, Algorithm 1 against the shared-memory-staged table, routing by the
// class policy, millisecond binning, and the histogram update of Section 5
// (a merge-scatter with the associative, commutative integer +).
#include <algorithm>
#include <map>
#include <mutex>
#include <utility>

#include "combine.cuh"
#include "launch.h"

namespace sinet {

// ---------------------------------------------------------------------------
// Algorithm 1 only. Each thread takes quads of records; a quad's eight
// memberships stay sign bits until they are packed into its four class bytes
// (byte permutes that replicate the sign), and the classes are counted by
// population counts of those bytes. `align`: log2 of the alignment of the class
// bytes of a full quad (2: one 32-bit store; 1, 0: smaller stores, when the
// class array starts at another offset than the addresses).
template <int LK>
__global__ void __launch_bounds__(512, LK == LK_INTERVAL ? 2 : 3) k_discriminate(RecArgs r, TableArgs t, uint32_t align, uint64_t *counts,
                                                         uint32_t *status) {
    extern __shared__ __align__(16) uint8_t smem[];
    __shared__ uint64_t bar;
    __shared__ unsigned long long s_cnt[4];
    if (threadIdx.x < 4) s_cnt[threadIdx.x] = 0;
    Classifier<LK> C;
    if (!C.init(t, smem, &bar, status)) return;  // table not staged: the status word says so
    __syncthreads();
    const uint64_t pol = policy_evict_first();
    uint32_t n_rec = 0, n_src = 0, n_dst = 0, n_both = 0;  // 8 x the thread's records of each kind
    const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
    for (uint64_t q = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; q < r.g.quads; q += stride) {
        Quad Q;
        load_quad<false, true, false, false>(r, q, pol, Q);
        uint32_t s[4], d[4];
        C.template sign_n<4>(Q.src, s);
        C.template sign_n<4>(Q.dst, d);
        uint32_t S = signs4(s[0], s[1], s[2], s[3]), D = signs4(d[0], d[1], d[2], d[3]);
        const int64_t base = quad_base(r.g, q);
        if (Q.valid == 0xFu) {
            if (r.cls_out) {
                const uint32_t w = (S & 0x01010101u) | (D & 0x02020202u);
                uint8_t *p = r.cls_out + base;
                if (align == 2) {
                    *reinterpret_cast<uint32_t *>(p) = w;
                } else if (align == 1) {
                    *reinterpret_cast<uint16_t *>(p) = (uint16_t)w;
                    *reinterpret_cast<uint16_t *>(p + 2) = (uint16_t)(w >> 16);
                } else {
#pragma unroll
                    for (int j = 0; j < 4; ++j) p[j] = (uint8_t)(w >> (8 * j));
                }
            }
        } else {
            const uint32_t m = signs4(Q.valid << 31, Q.valid << 30, Q.valid << 29, Q.valid << 28);
            S &= m;
            D &= m;
            if (r.cls_out) {
#pragma unroll
                for (int j = 0; j < 4; ++j)
                    if (Q.valid >> j & 1u) r.cls_out[base + j] = (uint8_t)(((S >> (8 * j)) & 1u) | ((D >> (8 * j)) & 2u));
            }
        }
        n_rec += 8 * __popc(Q.valid);
        n_src += __popc(S);
        n_dst += __popc(D);
        n_both += __popc(S & D);
    }
    // at most 2^40 records over at least one 512-thread CTA per SM: a thread's counts stay below 2^28
    const uint32_t v[4] = {(n_rec - n_src - n_dst + n_both) / 8, (n_src - n_both) / 8, (n_dst - n_both) / 8, n_both / 8};
    flush_cta(s_cnt, v, counts);
}

// Watch list (the blocklist views of Section 6, as a filter): a record whose
// src and dst are both outside the second list leaves the quad and counts in
// `flt` (stats[6]); the list is looked up in its global-memory interval form.
template <bool WATCH>
__device__ __forceinline__ void watch_filter(const Classifier<LK_INTERVAL_GLOBAL> &W, Quad &Q, uint32_t &flt) {
    if (!WATCH) return;
    uint32_t a[4], ws[4], wd[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) a[j] = Q.src[j];
    W.template in_n<4>(a, ws);
#pragma unroll
    for (int j = 0; j < 4; ++j) a[j] = Q.dst[j];
    W.template in_n<4>(a, wd);
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        if ((Q.valid >> j & 1u) && !(ws[j] | wd[j])) {
            Q.valid &= ~(1u << j);
            flt++;
        }
    }
}

// With AGG a warp combines its lanes' equal keys only while that saves global
// updates: combining costs about twice the instructions of a plain reduction,
// which uniform records over many bins would pay for nothing, and without it
// the hottest bin of skewed records serialises its reductions. Every kRecheck-th
// quad of a warp that goes without is combined all the same, and decides anew.
//   AGG 1: hot keys are kept in a shared-memory cache; fewer than a fifth of the
//          quad's routed updates saved, and the warp goes without.
//   AGG 2: a small cache that only keys which repeat within a warp enter (8 KB a
//          CTA leave its L1); none saved, and the warp goes without (a hot bin's
//          warps all save some). 10 M records over 100 K bins, packed cells:
//          uniform 85 us, skewed 133; always combining, into the output arrays,
//          159 and 199. run_fused_atomic says where each is taken.
enum : int { AGG_NONE = 0, AGG_CACHE = 1, AGG_REPEATS = 2 };
constexpr uint32_t kRecheck = 16;
constexpr uint32_t kRepeatSetBits = 7;

template <int LK, int AGG, bool WATCH>
__global__ void __launch_bounds__(256, 3) k_fused_atomic(RecArgs r, TableArgs t, HistArgs h,
                                                         uint32_t cache_set_bits, TableArgs wt, uint32_t *status) {
    extern __shared__ __align__(16) uint8_t smem[];
    __shared__ uint64_t bar;
    Classifier<LK> C;
    if (!C.init(t, smem, &bar, status)) return;  // table not staged: the status word says so
    Classifier<LK_INTERVAL_GLOBAL> W;
    if (WATCH) W.attach(wt, nullptr);
    __shared__ unsigned long long s_cnt[9];  // stats[0 .. 6], then updates and their bytes
    if (threadIdx.x < 9) s_cnt[threadIdx.x] = 0;
    __syncthreads();
    const uint64_t pol = policy_evict_first();
    uint32_t cc[4] = {0, 0, 0, 0}, oor[2] = {0, 0}, flt = 0;
    const uint32_t lane = threadIdx.x & 31;
    const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
    if (AGG == AGG_NONE) {
        for (uint64_t q = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; q < r.g.quads; q += stride) {
            Quad Q;
            load_quad<true, LK != LK_CLASS_IN, true, LK == LK_CLASS_IN>(r, q, pol, Q);
            watch_filter<WATCH>(W, Q, flt);
            classify_quad<LK>(C, Q);
            combine_quad(h, Q, cc, oor, [&](uint32_t key, uint32_t c, uint64_t s) {
                gadd(h, key & 1u, key >> 1, c, s);
            });
        }
        const uint32_t v[7] = {cc[0], cc[1], cc[2], cc[3], oor[0], oor[1], flt};
        flush_cta(s_cnt, v, h.stats);
        return;
    }
    // hot-key cache after the staged table
    uint8_t *cm = smem + ((Classifier<LK>::smem_bytes(t) + 15u) & ~15u);
    const uint32_t slots = HotCache::kWays << cache_set_bits;
    HotCache hc;
    hc.keys = reinterpret_cast<uint32_t *>(cm);
    hc.cnt = hc.keys + slots;
    hc.lo = hc.cnt + slots;
    hc.hi = hc.lo + slots;
    hc.set_bits = cache_set_bits;
    for (uint32_t i = threadIdx.x; i < slots; i += blockDim.x) {
        hc.keys[i] = kNoKey;
        hc.cnt[i] = 0;
        hc.lo[i] = 0;
        hc.hi[i] = 0;
    }
    __syncthreads();
    uint64_t sum = 0;  // bytes of the thread's updates, for the check of packed cells
    uint32_t plain = 0;  // quads the warp takes next without combining
    // warp-uniform trip count: every lane reaches the warp-synchronous updates
    for (uint64_t q0 = ((uint64_t)blockIdx.x * blockDim.x + threadIdx.x) - lane; q0 < r.g.quads;
         q0 += stride) {
        // a loop of its own: with both ways in one body Zipf-skewed records,
        // which never take this one, took a fifth longer
        for (; plain && q0 < r.g.quads; --plain, q0 += stride) {
            Quad Q;
            load_quad<true, LK != LK_CLASS_IN, true, LK == LK_CLASS_IN>(r, q0 + lane, pol, Q);
            watch_filter<WATCH>(W, Q, flt);
            classify_quad<LK>(C, Q);
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                if (!(Q.valid >> j & 1u)) continue;
                bump_class(cc, Q.cls[j]);
                uint32_t bin;
                const uint32_t dirs = route(h, Q.cls[j], Q.ts[j], bin, oor);
                if (h.packed) sum += (uint64_t)__popc(dirs) * Q.by[j];
                if (dirs & 1u) gadd(h, 0u, bin, 1u, Q.by[j]);
                if (dirs & 2u) gadd(h, 1u, bin, 1u, Q.by[j]);
            }
        }
        if (q0 >= r.g.quads) break;
        Quad Q;
        load_quad<true, LK != LK_CLASS_IN, true, LK == LK_CLASS_IN>(r, q0 + lane, pol, Q);
        watch_filter<WATCH>(W, Q, flt);
        classify_quad<LK>(C, Q);
        uint32_t saved = 0;  // and, from bit 16 on, the thread's routed records
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const bool v = Q.valid >> j & 1u;
            uint32_t bin = 0, dirs = 0;
            if (v) {
                bump_class(cc, Q.cls[j]);
                dirs = route(h, Q.cls[j], Q.ts[j], bin, oor);
            }
            if (h.packed) sum += (uint64_t)__popc(dirs) * Q.by[j];
            const uint32_t key = dirs ? (bin << 1 | (dirs & 1u ? 0u : 1u)) : kNoKey;
            if (AGG == AGG_CACHE && dirs) saved += 1u << 16;
            saved += update_agg<AGG>(h, hc, key, Q.by[j]);
            if (h.two_dir) {
                const bool both = dirs == 3u;
                if (__any_sync(kFull, both))
                    update_agg<AGG>(h, hc, both ? (bin << 1 | 1u) : kNoKey, Q.by[j]);
            }
        }
        saved = __reduce_add_sync(kFull, saved);
        const uint32_t routed = saved >> 16;
        if (AGG == AGG_CACHE ? routed >= 16 && 5 * (saved & 0xFFFFu) < routed : saved == 0) plain = kRecheck - 1;
    }
    if (h.packed) {
        uint64_t updates = 0;
#pragma unroll
        for (int k = 0; k < 4; ++k) updates += (uint64_t)cc[k] * __popc((h.policy >> (8 * k)) & 3u);
        updates -= oor[0] + (uint64_t)oor[1];
        warp_totals(updates, sum);
        if (lane == 0 && updates) {
            atomicAdd(s_cnt + 7, (unsigned long long)updates);
            atomicAdd(s_cnt + 8, (unsigned long long)sum);
        }
    }
    __syncthreads();
    for (uint32_t i = threadIdx.x; i < slots; i += blockDim.x) {
        const uint32_t c = hc.cnt[i];
        if (c) gadd(h, hc.keys[i] & 1u, hc.keys[i] >> 1, c, (uint64_t)hc.hi[i] << 32 | hc.lo[i]);
    }
    const uint32_t v[7] = {cc[0], cc[1], cc[2], cc[3], oor[0], oor[1], flt};
    flush_cta(s_cnt, v, h.stats);
    if (h.packed && threadIdx.x < 2) red_add_u64(h.pack_sums + threadIdx.x, s_cnt[7 + threadIdx.x]);
}

// One record into entry e of a tile: byte sum's low word, then count << 16 with
// the carry out of it (see below).
__device__ __forceinline__ void tile_add(uint32_t *tlo, uint32_t *thi, uint32_t e, uint32_t by) {
    const uint32_t old = atomicAdd(tlo + e, by);
    atomicAdd(thi + e, 0x10000u + (uint32_t)(old + by < old));
}

// ---------------------------------------------------------------------------
// Shared-memory privatised bins. A CTA takes chunks of blockDim * iters quads
// (at most 65,535 records); for each chunk it places a tile of `tile_bins`
// bins per direction just below the chunk's first record (time-sorted input
// keeps the chunk inside it). A tile entry is two 32-bit words updated with
// native shared atomics: the low 32 bits of the byte sum, and a high word
// holding the record count in its upper 16 bits and the byte sum's bits
// 32-47 in its lower 16 (a bin of one chunk holds at most 65,535 records,
// whose bytes sum below 2^48). The touched part of the tile is flushed with
// global atomics after the chunk. Records outside the tile go straight to
// global atomics. With `full`, the tile is the whole histogram (base 0).
//
// The kernel is bound by instructions and by its loads' latency in turn (59 %
// of issue slots, 32 warps an SM), so both were cut: classes, directions and
// counters are computed on bit masks of four records, windows below 2^32 ms
// divide in 32 bits, a quad that lies in the window and in the tile (the rule)
// takes no branch per record, and the next quad's loads overlap this one's
// adds. With `full`, chunks are as long as the 16-bit counts allow: the whole
// tile is flushed for each. 50 M records into 3,600 bins of 1 s, both
// directions: 327 -> 215 us; with the counters' sums per CTA (flush_cta), 100 M
// classified records at 10 ms 439 -> 372; the 400 M sorted day 2.53 -> 2.27-2.47 ms.
template <int LK, bool W1>
__global__ void __launch_bounds__(1024) k_fused_tile(RecArgs r, TableArgs t, HistArgs h, TileArgs ta,
                                                     uint32_t *status) {
    extern __shared__ __align__(16) uint8_t smem[];
    __shared__ uint64_t bar;
    __shared__ uint32_t s_base, s_lo, s_hi;
    __shared__ unsigned long long s_cnt[6];
    Classifier<LK> C;
    if (!C.init(t, smem, &bar, status)) return;  // table not staged: the status word says so
    const uint32_t T = ta.tile_bins;
    uint32_t *tlo = reinterpret_cast<uint32_t *>(smem + ((Classifier<LK>::smem_bytes(t) + 15u) & ~15u));
    uint32_t *thi = tlo + 2 * T;
    for (uint32_t i = threadIdx.x; i < 2 * T; i += blockDim.x) {
        tlo[i] = 0;
        thi[i] = 0;
    }
    if (threadIdx.x == 0) {
        s_lo = 0xFFFFFFFFu;
        s_hi = 0;
    }
    if (threadIdx.x < 6) s_cnt[threadIdx.x] = 0;
    const uint64_t pol = policy_evict_first();
    // per-thread counts: records, source inside, destination inside, both; routed outside the window
    uint32_t n_rec = 0, n_src = 0, n_dst = 0, n_both = 0, oor[2] = {0, 0};
    const DirMasks out_of(h.policy, 0), in_of(h.policy, 1);
    const uint64_t qpc = (uint64_t)blockDim.x * ta.iters;
    const uint64_t n_chunks = (r.g.quads + qpc - 1) / qpc;
    const uint32_t lane = threadIdx.x & 31;
    // thread 0 places each chunk's tile from the chunk's first timestamp,
    // loaded one chunk ahead so the CTA does not wait on it at the barrier
    uint64_t ts_first = 0;
    if (!ta.full && threadIdx.x == 0 && blockIdx.x < n_chunks) {
        int64_t i0 = quad_base(r.g, (uint64_t)blockIdx.x * qpc);
        ts_first = r.ts[i0 < 0 ? 0 : i0];
    }
    Quad N;  // the quad loaded ahead
    load_quad<true, LK != LK_CLASS_IN, true, LK == LK_CLASS_IN>(r, (uint64_t)blockIdx.x * qpc + threadIdx.x, pol, N);
    __syncthreads();

    for (uint64_t ch = blockIdx.x; ch < n_chunks; ch += gridDim.x) {
        if (!ta.full && threadIdx.x == 0) {
            uint32_t b = 0;
            const uint64_t rel = ts_first - h.t0;
            if (rel < h.span) {
                b = h.w_is_one ? (uint32_t)rel : bin_of(h, rel);
                b = b > ta.margin ? b - ta.margin : 0u;
            }
            s_base = b;
            if (ch + gridDim.x < n_chunks) {
                const int64_t i1 = quad_base(r.g, (ch + gridDim.x) * qpc);
                ts_first = r.ts[i1 < 0 ? 0 : i1];
            }
        }
        // the tile is placed; and with `full` too, thread 0 has reset s_lo and
        // s_hi before any warp adds this chunk's range to them
        __syncthreads();
        const uint32_t base = ta.full ? 0u : s_base;
        uint32_t omin = 0xFFFFFFFFu, omax = 0;
        for (uint32_t it = 0; it < ta.iters; ++it) {
            uint32_t off[4], by[4], src, dst;
            const uint32_t inr = bin_quad<W1>(h, N, off), valid = N.valid;
            class_masks<LK>(C, N, src, dst);
#pragma unroll
            for (int j = 0; j < 4; ++j) by[j] = N.by[j];
            // the loaded quad is used up: the next one's loads overlap the adds
            // (and the flush, at the end of a chunk)
            const uint64_t q = it + 1 < ta.iters ? ch * qpc + (uint64_t)(it + 1) * blockDim.x : (ch + gridDim.x) * qpc;
            load_quad<true, LK != LK_CLASS_IN, true, LK == LK_CLASS_IN>(r, q + threadIdx.x, pol, N);
            src &= valid;
            dst &= valid;
            n_rec += __popc(valid);
            n_src += __popc(src);
            n_dst += __popc(dst);
            n_both += __popc(src & dst);
            uint32_t d0 = out_of.of(src, dst) & valid, d1 = in_of.of(src, dst) & valid;
#pragma unroll
            for (int j = 0; j < 4; ++j) off[j] -= base;
            const uint32_t most = max(max(off[0], off[1]), max(off[2], off[3]));
            if (inr == 0xFu && most < T) {
                // the rule: the whole quad lies in the window and in the tile
                omin = min(omin, min(min(off[0], off[1]), min(off[2], off[3])));
                omax = max(omax, most);
                const uint32_t both = d0 & d1, any = d0 | d1;
#pragma unroll
                for (int j = 0; j < 4; ++j)
                    if (any >> j & 1u) tile_add(tlo, thi, (d0 >> j & 1u) ? off[j] : T + off[j], by[j]);
                if (both) {
#pragma unroll
                    for (int j = 0; j < 4; ++j)
                        if (both >> j & 1u) tile_add(tlo, thi, T + off[j], by[j]);
                }
                continue;
            }
            oor[0] += __popc(d0 & ~inr);  // routed, outside the window
            oor[1] += __popc(d1 & ~inr);
            d0 &= inr;
            d1 &= inr;
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                if (!((d0 | d1) >> j & 1u)) continue;
                if (off[j] < T) {
                    omin = min(omin, off[j]);
                    omax = max(omax, off[j]);
                    if (d0 >> j & 1u) tile_add(tlo, thi, off[j], by[j]);
                    if (d1 >> j & 1u) tile_add(tlo, thi, T + off[j], by[j]);
                } else {
                    if (d0 >> j & 1u) gadd(h, 0u, base + off[j], 1u, by[j]);
                    if (d1 >> j & 1u) gadd(h, 1u, base + off[j], 1u, by[j]);
                }
            }
        }
        // touched range of the tile, then flush it
        omin = __reduce_min_sync(kFull, omin);
        omax = __reduce_max_sync(kFull, omax);
        if (lane == 0 && omin <= omax) {
            atomicMin(&s_lo, omin);
            atomicMax(&s_hi, omax);
        }
        __syncthreads();
        const uint32_t lo = s_lo, hi = s_hi;
        if (lo <= hi) {
            // consecutive lanes take consecutive bins, so each warp-wide global
            // atomic covers as few sectors as possible
            const uint32_t n = hi - lo + 1;
            for (uint32_t i = threadIdx.x; i < 2 * n; i += blockDim.x) {
                const uint32_t d = i >= n;
                const uint32_t off = lo + i - d * n;
                const uint32_t e = d * T + off;
                const uint32_t vh = thi[e];
                if (vh) {
                    gadd(h, d, base + off, vh >> 16, (uint64_t)(vh & 0xFFFFu) << 32 | tlo[e]);
                    tlo[e] = 0;
                    thi[e] = 0;
                }
            }
        }
        __syncthreads();
        if (threadIdx.x == 0) {
            s_lo = 0xFFFFFFFFu;
            s_hi = 0;
        }
    }
    // (a thread's counts stay far below 2^32: at most 2^40 records over the grid)
    const uint32_t cc[6] = {n_rec - n_src - n_dst + n_both, n_src - n_both, n_dst - n_both, n_both, oor[0], oor[1]};
    flush_cta(s_cnt, cc, h.stats);
}

// ---------------------------------------------------------------------------
// Binning alone: the bin of each record, or kNoKey outside the window.
__global__ void __launch_bounds__(256) k_bin(const uint64_t *ts, uint64_t n, HistArgs h, uint32_t *bin) {
    const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
    for (uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += stride) {
        const uint64_t rel = ts[i] - h.t0;
        bin[i] = rel < h.span ? bin_of(h, rel) : kNoKey;
    }
}

cudaError_t run_bin(const uint64_t *ts, uint64_t n, const HistArgs &h, uint32_t *bin, const LaunchCfg &c) {
    k_bin<<<8 * c.sm_count, 256, 0, c.stream>>>(ts, n, h, bin);
    return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// Cell expansion: one thread per bin reads its 32-byte cell and writes (or
// adds to) the four output arrays; consecutive threads write consecutive bins.
__global__ void __launch_bounds__(256) k_cells_expand(HistArgs h, uint32_t accumulate) {
    const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
    for (uint64_t b = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; b < h.n_bins; b += stride) {
        const ulonglong2 sums = __ldcs(reinterpret_cast<const ulonglong2 *>(h.cells + 4 * b));
        const ulonglong2 cnts = __ldcs(reinterpret_cast<const ulonglong2 *>(h.cells + 4 * b + 2));
        const uint32_t c0 = (uint32_t)cnts.x, c1 = (uint32_t)(cnts.x >> 32);
        const uint64_t s0 = sums.x, s1 = sums.y;
        if (accumulate) {  // reductions: calls on other streams may be adding to the same outputs
            if (c0) red_add_u32(h.cnt[0] + b, c0);
            if (c1) red_add_u32(h.cnt[1] + b, c1);
            if (s0) red_add_u64(h.byt[0] + b, s0);
            if (s1) red_add_u64(h.byt[1] + b, s1);
            continue;
        }
        h.cnt[0][b] = c0;
        h.cnt[1][b] = c1;
        h.byt[0][b] = s0;
        h.byt[1][b] = s1;
    }
}

// ---------------------------------------------------------------------------
// Packed cells (HistArgs::packed): expansion into the output arrays, and the
// totals of what it wrote.
// VEC: four bins a thread in 16-byte loads and stores (every array 16-byte
// aligned and n_bins a multiple of four); else one, four rows in flight.
template <bool VEC>
__global__ void __launch_bounds__(256) k_pack_expand(HistArgs h) {
    __shared__ unsigned long long s_sum[2];
    if (threadIdx.x < 2) s_sum[threadIdx.x] = 0;
    __syncthreads();
    uint64_t updates = 0, bytes = 0;
    constexpr uint64_t kMask = (1ull << kPackBits) - 1;
    const uint64_t stride = (uint64_t)gridDim.x * blockDim.x, first = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (VEC) {
        for (uint64_t q = first; q < h.n_bins / 4; q += stride) {
            ulonglong2 x[2][2];
#pragma unroll
            for (int d = 0; d < 2; ++d) {
                const ulonglong2 *p = reinterpret_cast<const ulonglong2 *>(h.packed + (uint64_t)d * h.n_bins) + 2 * q;
                x[d][0] = __ldcs(p);
                x[d][1] = __ldcs(p + 1);
            }
#pragma unroll
            for (int d = 0; d < 2; ++d) {
                const uint64_t v[4] = {x[d][0].x, x[d][0].y, x[d][1].x, x[d][1].y};
                uint32_t c[4];
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    c[k] = (uint32_t)(v[k] >> kPackBits);
                    updates += c[k];
                    bytes += v[k] & kMask;
                }
                reinterpret_cast<uint4 *>(h.cnt[d])[q] = make_uint4(c[0], c[1], c[2], c[3]);
                ulonglong2 *o = reinterpret_cast<ulonglong2 *>(h.byt[d]) + 2 * q;
                o[0] = make_ulonglong2(v[0] & kMask, v[1] & kMask);
                o[1] = make_ulonglong2(v[2] & kMask, v[3] & kMask);
            }
        }
    } else {
        for (uint64_t b0 = first; b0 < h.n_bins; b0 += 4 * stride) {
            uint64_t x[4][2];
#pragma unroll
            for (int k = 0; k < 4; ++k)
#pragma unroll
                for (int d = 0; d < 2; ++d) {
                    const uint64_t b = b0 + k * stride;
                    x[k][d] = b < h.n_bins ? h.packed[(uint64_t)d * h.n_bins + b] : 0ull;
                }
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                const uint64_t b = b0 + k * stride;
                if (b >= h.n_bins) break;
#pragma unroll
                for (int d = 0; d < 2; ++d) {
                    const uint32_t c = (uint32_t)(x[k][d] >> kPackBits);
                    h.cnt[d][b] = c;
                    h.byt[d][b] = x[k][d] & kMask;
                    updates += c;
                    bytes += x[k][d] & kMask;
                }
            }
        }
    }
    warp_totals(updates, bytes);
    if ((threadIdx.x & 31) == 0 && updates) {
        atomicAdd(s_sum, (unsigned long long)updates);
        atomicAdd(s_sum + 1, (unsigned long long)bytes);
    }
    __syncthreads();  // one global add a CTA (see flush_cta)
    if (threadIdx.x < 2) red_add_u64(h.pack_sums + 2 + threadIdx.x, s_sum[threadIdx.x]);
}

__device__ __forceinline__ bool pack_right(const uint64_t *s) {
    return s[0] == s[2] && s[1] == s[3];
}

// What follows when the totals disagree, in a cooperative launch: the outputs
// are zeroed, and once every CTA has done its share (a bounded wait) every
// record is added to them with plain reductions (the class and window counters
// stand). Otherwise it returns at once.
template <int LK, bool WATCH>
__global__ void __launch_bounds__(256) k_pack_redo(RecArgs r, TableArgs t, HistArgs h, TableArgs wt, uint32_t *status) {
    extern __shared__ __align__(16) uint8_t smem[];
    __shared__ uint64_t bar;
    if (pack_right(h.pack_sums)) return;
    for (uint64_t b = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; b < h.n_bins;
         b += (uint64_t)gridDim.x * blockDim.x)
#pragma unroll
        for (int d = 0; d < 2; ++d) {
            h.cnt[d][b] = 0;
            h.byt[d][b] = 0;
        }
    __threadfence();
    __syncthreads();
    __shared__ bool s_zeroed;
    if (threadIdx.x == 0) {
        uint32_t *arrived = reinterpret_cast<uint32_t *>(h.pack_sums + 4);
        atomicAdd(arrived, 1u);
        bool ok = false;
        for (uint32_t k = 0; k < kSpinLimit && !ok; ++k)
            ok = *reinterpret_cast<volatile uint32_t *>(arrived) == gridDim.x;
        if (!ok) latch_status(status, SINET_ERR_TIMEOUT);
        s_zeroed = ok;
    }
    __syncthreads();
    if (!s_zeroed) return;
    h.packed = nullptr;
    Classifier<LK> C;
    if (!C.init(t, smem, &bar, status)) return;  // table not staged: the status word says so
    Classifier<LK_INTERVAL_GLOBAL> W;
    if (WATCH) W.attach(wt, nullptr);
    const uint64_t pol = policy_evict_first();
    uint32_t oor[2] = {0, 0}, flt = 0;
    for (uint64_t q = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; q < r.g.quads;
         q += (uint64_t)gridDim.x * blockDim.x) {
        Quad Q;
        load_quad<true, LK != LK_CLASS_IN, true, LK == LK_CLASS_IN>(r, q, pol, Q);
        watch_filter<WATCH>(W, Q, flt);
        classify_quad<LK>(C, Q);
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            if (!(Q.valid >> j & 1u)) continue;
            uint32_t bin;
            const uint32_t dirs = route(h, Q.cls[j], Q.ts[j], bin, oor);
            if (dirs & 1u) gadd(h, 0u, bin, 1u, Q.by[j]);
            if (dirs & 2u) gadd(h, 1u, bin, 1u, Q.by[j]);
        }
    }
}

// ---------------------------------------------------------------------------
// Host launchers.

size_t smem_optin_limit() {
    int dev = 0, v = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&v, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
    return (size_t)v;
}

// What the runtime was told and answered about a kernel on a device: the
// shared-memory limit set so far (only ever raised, so no launch finds it lowered
// by another thread's) and resident CTAs per SM by block and shared memory. The
// two calls took a third of a small launch's host time.
struct KernelFacts {
    size_t smem_limit = 0;
    std::map<std::pair<int, size_t>, int> per_sm;
};
static std::mutex g_facts_mu;
static std::map<std::pair<const void *, int>, KernelFacts> g_facts;

// (g_facts_mu is held)
static cudaError_t raise_limit(KernelFacts &f, const void *kernel, size_t smem) {
    if (smem <= f.smem_limit) return cudaSuccess;
    const cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e == cudaSuccess) f.smem_limit = smem;
    return e;
}

cudaError_t raise_smem_limit(const void *kernel, size_t smem) {
    int dev = 0;
    const cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    std::lock_guard<std::mutex> lk(g_facts_mu);
    return raise_limit(g_facts[{kernel, dev}], kernel, smem);
}

template <typename K>
static cudaError_t launch(K kernel, size_t smem, const LaunchCfg &c, int &grid) {
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    std::lock_guard<std::mutex> lk(g_facts_mu);
    KernelFacts &f = g_facts[{(const void *)kernel, dev}];
    if ((e = raise_limit(f, (const void *)kernel, smem)) != cudaSuccess) return e;
    grid = c.grid;
    if (grid > 0) return cudaSuccess;
    if (f.per_sm.size() > 256) f.per_sm.clear();  // tables of many sizes
    int &per_sm = f.per_sm[{c.block, smem}];
    if (per_sm == 0) {
        e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel, c.block, smem);
        if (e != cudaSuccess) {
            per_sm = 0;
            return e;
        }
    }
    if (per_sm < 1) return cudaErrorInvalidConfiguration;
    grid = per_sm * c.sm_count;
    return cudaSuccess;
}

cudaError_t run_cells_expand(const HistArgs &h, bool accumulate, const LaunchCfg &c) {
    const int grid = 8 * c.sm_count;
    k_cells_expand<<<grid, 256, 0, c.stream>>>(h, accumulate ? 1u : 0u);
    return cudaGetLastError();
}

cudaError_t run_pack_finish(int lk, const RecArgs &r, const TableArgs &t, const HistArgs &h, const LaunchCfg &c,
                            const TableArgs *watch) {
    const int grid = (int)std::min<uint64_t>(8ull * c.sm_count, ((uint64_t)h.n_bins + 1023) / 1024);
    const uintptr_t all = (uintptr_t)h.cnt[0] | (uintptr_t)h.cnt[1] | (uintptr_t)h.byt[0] | (uintptr_t)h.byt[1];
    if (all % 16 == 0 && h.n_bins % 4 == 0)
        k_pack_expand<true><<<grid, 256, 0, c.stream>>>(h);
    else
        k_pack_expand<false><<<grid, 256, 0, c.stream>>>(h);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    RecArgs ra = r;
    TableArgs ta = t, wa = watch ? *watch : TableArgs{};
    HistArgs ha = h;
    uint32_t *status = c.status;
    void *args[] = {&ra, &ta, &ha, &wa, &status};
#define SINET_REDO(L, WA)                                                                                     \
    if (lk == L && (watch != nullptr) == WA) {                                                                \
        const size_t smem = Classifier<L>::smem_bytes(t);                                                     \
        const void *f = (const void *)k_pack_redo<L, WA>;                                                     \
        if ((e = raise_smem_limit(f, smem)) != cudaSuccess) return e;                                         \
        return cudaLaunchCooperativeKernel(f, dim3(c.sm_count), dim3(256), args, smem, c.stream);             \
    }
    SINET_REDO(LK_INTERVAL, false)
    SINET_REDO(LK_LEAF2, false)
    SINET_REDO(LK_LEAF4, false)
    SINET_REDO(LK_TOGGLE2, false)
    SINET_REDO(LK_PML, false)
    SINET_REDO(LK_INTERVAL_GLOBAL, false)
    SINET_REDO(LK_CLASS_IN, false)
    SINET_REDO(LK_INTERVAL, true)
    SINET_REDO(LK_LEAF2, true)
    SINET_REDO(LK_LEAF4, true)
    SINET_REDO(LK_TOGGLE2, true)
    SINET_REDO(LK_INTERVAL_GLOBAL, true)
#undef SINET_REDO
    return cudaErrorInvalidValue;
}

cudaError_t run_discriminate(int lk, const RecArgs &r, const TableArgs &t, uint64_t *counts,
                             const LaunchCfg &c) {
    int grid = 0;
    cudaError_t e;
    // full quads start 4-record aligned in the addresses, not always in the class array
    const uintptr_t at = (uintptr_t)r.cls_out + (uintptr_t)(intptr_t)r.g.shift;
    const uint32_t align = at % 4 == 0 ? 2u : at % 2 == 0 ? 1u : 0u;
    switch (lk) {
#define SINET_DISC(L)                                                                           \
    case L: {                                                                                   \
        size_t smem = Classifier<L>::smem_bytes(t);                                             \
        if ((e = launch(k_discriminate<L>, smem, c, grid)) != cudaSuccess) return e;            \
        k_discriminate<L><<<grid, c.block, smem, c.stream>>>(r, t, align, counts, c.status);    \
        break;                                                                                  \
    }
        SINET_DISC(LK_INTERVAL)
        SINET_DISC(LK_LEAF2)
        SINET_DISC(LK_LEAF4)
        SINET_DISC(LK_TOGGLE2)
        SINET_DISC(LK_PML)
        SINET_DISC(LK_INTERVAL_GLOBAL)
#undef SINET_DISC
        default:
            return cudaErrorInvalidValue;
    }
    return cudaGetLastError();
}

cudaError_t run_fused_atomic(int lk, bool agg, const RecArgs &r, const TableArgs &t,
                             const HistArgs &h, uint32_t cache_set_bits, const LaunchCfg &c,
                             const TableArgs *watch) {
    int grid = 0;
    cudaError_t e;
    const TableArgs none{};
    // The large cache pays where updates miss L2 (outputs beyond about 90 MB) and
    // hot keys therefore must not reach memory, from half a million records on:
    // small and large, us (uniform; skewed), 1.2 M records over 5.7 M bins 78, 83;
    // 73, 64. 5 M 183, 187; 132, 117. 8 M over 40 M 667, 666; 346, 301. In L2 the
    // small one is better or equal: 1.2 M over 600 K 32, 40; 42, 42. 13 M over
    // 100 K 104, 112; 168, 184. 130 M over 600 K 811, 769; 1,382, 1,530. And with a
    // watch list, whose lookups want the L1 that the large one takes: 60 M over
    // 600 K with 1,500 entries 775, 2,465
    const bool large = !watch && 24ull * h.n_bins > (90ull << 20) && r.g.n >= 500000;
    const int mode = !agg ? AGG_NONE : large ? AGG_CACHE : AGG_REPEATS;
    const uint32_t bits = large ? cache_set_bits : std::min<uint32_t>(cache_set_bits, kRepeatSetBits);
#define SINET_ATOM(L, A, WA)                                                                    \
    if (lk == L && mode == A && (watch != nullptr) == WA) {                                     \
        size_t smem = ((Classifier<L>::smem_bytes(t) + 15u) & ~15u) +                           \
                      (A ? (size_t)HotCache::kSlotBytes * (HotCache::kWays << bits) : 0ull);    \
        if ((e = launch(k_fused_atomic<L, A, WA>, smem, c, grid)) != cudaSuccess) return e;     \
        k_fused_atomic<L, A, WA><<<grid, c.block, smem, c.stream>>>(r, t, h, bits,               \
                                                                   WA ? *watch : none, c.status); \
        return cudaGetLastError();                                                              \
    }
#define SINET_ATOM2(L) SINET_ATOM(L, AGG_CACHE, false) SINET_ATOM(L, AGG_REPEATS, false) SINET_ATOM(L, AGG_NONE, false)
#define SINET_ATOM3(L) SINET_ATOM(L, AGG_REPEATS, true) SINET_ATOM(L, AGG_NONE, true)
    SINET_ATOM2(LK_INTERVAL)
    SINET_ATOM2(LK_LEAF2)
    SINET_ATOM2(LK_LEAF4)
    SINET_ATOM2(LK_TOGGLE2)
    SINET_ATOM2(LK_PML)
    SINET_ATOM2(LK_INTERVAL_GLOBAL)
    SINET_ATOM2(LK_CLASS_IN)
    SINET_ATOM3(LK_INTERVAL)
    SINET_ATOM3(LK_LEAF2)
    SINET_ATOM3(LK_LEAF4)
    SINET_ATOM3(LK_TOGGLE2)
    SINET_ATOM3(LK_INTERVAL_GLOBAL)
#undef SINET_ATOM3
#undef SINET_ATOM2
#undef SINET_ATOM
    return cudaErrorInvalidValue;
}

cudaError_t run_fused_tile(int lk, const RecArgs &r, const TableArgs &t, const HistArgs &h,
                           const TileArgs &ta, const LaunchCfg &c) {
    int grid = 0;
    cudaError_t e;
    const bool w1 = h.w_is_one != 0;
#define SINET_TILE(L, W)                                                                        \
    if (lk == L && w1 == W) {                                                                   \
        size_t smem = ((Classifier<L>::smem_bytes(t) + 15u) & ~15u) + 16ull * ta.tile_bins;     \
        if ((e = launch(k_fused_tile<L, W>, smem, c, grid)) != cudaSuccess) return e;           \
        k_fused_tile<L, W><<<grid, c.block, smem, c.stream>>>(r, t, h, ta, c.status);           \
        return cudaGetLastError();                                                              \
    }
    SINET_TILE(LK_INTERVAL, true)
    SINET_TILE(LK_INTERVAL, false)
    SINET_TILE(LK_LEAF2, true)
    SINET_TILE(LK_LEAF2, false)
    SINET_TILE(LK_LEAF4, true)
    SINET_TILE(LK_LEAF4, false)
    SINET_TILE(LK_TOGGLE2, true)
    SINET_TILE(LK_TOGGLE2, false)
    SINET_TILE(LK_PML, true)
    SINET_TILE(LK_PML, false)
    SINET_TILE(LK_INTERVAL_GLOBAL, true)
    SINET_TILE(LK_INTERVAL_GLOBAL, false)
    SINET_TILE(LK_CLASS_IN, true)
    SINET_TILE(LK_CLASS_IN, false)
#undef SINET_TILE
    return cudaErrorInvalidValue;
}

}  // namespace sinet

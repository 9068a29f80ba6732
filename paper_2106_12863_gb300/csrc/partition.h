// Hot/cold partitioned histogram update (SINET_STRAT_PARTITION): host-side
// plan of the launch sequence and its scratch layout.
//
// The scheme, for unsorted records over a histogram too large for shared
// memory:
//   1. sample: classify and bin a strided sample of the records and count
//      sample hits per bin in an L2-resident hash table;
//   2. select: the bins with the most sample hits form a static hot table
//      (sets of two ways, hottest first), the same in every CTA; the other hits give
//      the room that every bin range's run of entries gets;
//   3. main pass (one read of the records, staged into shared memory by TMA
//      bulk copies): hot bins are accumulated in each CTA's shared-memory copy
//      of the hot table; every other routed update becomes an 8-byte entry
//      (bin << 1 | direction, bytes) appended to the CTA's run of its bin range;
//   4. split (large histograms): the entries of the ranges' runs go on to runs of
//      their tile of bins;
//   5. cold pass: each CTA takes tile after tile of bins, sums its entries in
//      shared memory and stores every bin of the tile once;
//   6. finish: the hot table's totals and the entries that found their run full
//      are added to their bins.
// Every update is counted exactly once: in a hot slot, as an entry of a run, or
// in the overflow list (or, where that is full, by the finishing kernel over
// the records themselves).
#pragma once
#include "launch.h"

namespace sinet {

// Main pass: 31 consumer warps and one producer warp, 1,024 threads (64
// registers each fit the register file), two adjacent records per consumer
// per stage (read with one 16-byte and three 8-byte shared-memory loads), two
// stages of 39 KB in flight.
constexpr int kPartConsumers = 992;                 // consumer threads of the main pass
constexpr int kPartThreads = kPartConsumers + 32;   // plus one producer warp (TMA)
constexpr int kPartRPT = 2;                         // records per consumer per stage
constexpr uint32_t kPartStageRecords = kPartRPT * kPartConsumers;  // records per TMA stage
static_assert((4 * kPartStageRecords) % 16 == 0, "every stage starts 16-byte aligned in every stream");
constexpr uint32_t kPartStages = 2;                 // more, in the hot table's room, when that is empty
constexpr uint32_t kPartMaxStages = 4;
constexpr uint32_t kPartStageBytes = 20 * kPartStageRecords;
constexpr uint32_t kPartTileBits = 13;              // bins of a cold tile: 24 bytes each, one CTA per SM
constexpr uint32_t kPartMaxRuns = 256;              // ranges that the main pass writes to (see k_part_split)
constexpr uint32_t kPartMaxCand = 16384;            // hot candidates taken from the sample
constexpr uint32_t kPartReps = 14;                  // bins whose sums are kept in several copies
constexpr uint32_t kPartRepCopies = 8;
constexpr uint32_t kPartSampleChunk = 512;          // records per sampled chunk
constexpr uint32_t kPartSampleThreads = 1024;
constexpr uint32_t kPartSampleSetBits = 9;          // sample pass: per-CTA pre-aggregation cache

// Device view of the scheme's scratch (all device pointers).
struct PartDev {
    // sample counts: open-addressing hash table over bins
    uint32_t *hash_keys;  // kNoKey when empty
    uint32_t *hash_cnt;
    uint32_t hash_mask;   // slots - 1
    uint32_t hash_shift;  // 32 - log2(slots): slot = top bits of the hash
    uint32_t *levels;     // [32] hash slots per log2 of their count; [32] sample hits in all
    uint32_t *cand_n;     // candidates collected
    uint2 *cand;          // [max_cand] (bin, sample count)
    uint32_t max_cand;    // at most kPartMaxCand
    // hot table (slot = 2 * set + way, then the copies of the replicated
    // bins), the same in every CTA; see k_part_build
    uint32_t *hot_enc;    // [slots] entries
    uint32_t *hot_keys;   // [slots + copies] bin of each slot's sums or kNoKey
    uint32_t *hot_cnt;    // [slots + copies][2]
    uint64_t *hot_bytes;  // [slots + copies][2]
    uint32_t set_bits;
    uint32_t *n_hot;      // 0: the table is empty
    // cold entries: CTA c's region is entries[c * region .. (c + 1) * region);
    // in it the run of range b starts at base[b] and has room up to base[b + 1]
    uint32_t *tile_hits;    // [n_tiles] sample hits per tile
    uint32_t tiles_in_smem; // k_part_build keeps two words per tile in shared memory
    float entries_per_hit;  // entries a CTA expects for each of them
    uint32_t *base;         // [n_buckets + 1]
    uint64_t *entries;      // [g_main][region]
    uint64_t region;
    uint32_t *counts;       // [n_buckets][g_main] entries of every run (zero until its CTA stores them)
    uint64_t *ovf;          // [ovf_cap] entries that found their run full
    uint32_t *ovf_n;
    uint32_t ovf_cap;
    uint32_t *redo;         // not 0: the overflow list is full, see k_part_finish
    uint32_t cb_shift;      // range of a bin = bin >> cb_shift
    uint32_t n_buckets;     // ranges
    uint32_t g_main;        // CTAs of the main pass
    uint32_t tile_bits;     // bins of a cold tile = 1 << tile_bits (<= cb_shift)
    uint32_t n_tiles;
    // split: the tiles' own runs, entries tile_base[t] .. tile_base[t + 1) of tile_entries
    uint32_t split;         // 1, 2: the runs of a range are split by tile before they are summed (2: see split_claim)
    uint64_t tile_room;     // entries in all
    uint32_t *tile_base;    // [n_tiles + 1]
    uint32_t *tile_cur;     // [n_tiles] next position of each
    uint64_t *tile_entries;
    // main pass geometry: full TMA stages [i_lo, i_lo + n_full * R); the
    // other records (head, tail, or all when the streams cannot be staged)
    // are loaded one by one
    uint64_t i_lo, n_full;
    uint64_t n_head;        // records before i_lo
    // sample geometry: chunk k * sample_stride for k < sample_chunks
    uint64_t sample_chunks, sample_stride;
};

struct PartPlan {
    PartDev d;                 // pointers filled once the scratch exists
    uint32_t slots;            // 2 << set_bits
    int grid_main, grid_sample, grid_cold;
    size_t smem_main, smem_sample, smem_build, smem_split, smem_cold, smem_finish;
    size_t scratch_bytes;
    // scratch layout (byte offsets)
    size_t off_ff, bytes_ff;   // region set to 0xFF (hash keys)
    size_t off_zero, bytes_zero;  // region set to zero
    size_t off_hash_keys, off_hot_enc, off_hot_keys, off_levels, off_words, off_hot_cnt, off_hot_bytes, off_tile_hits,
        off_hash_cnt, off_cand, off_base, off_counts, off_tile_base, off_tile_cur, off_ovf, off_entries,
        off_tile_entries;
};

// Plan for n records into h.n_bins bins with table lookup `lk`; returns
// cudaErrorNotSupported when the histogram or the input is beyond the
// scheme's limits (more than 2^28 bins, 2^32 routed updates).
cudaError_t plan_partition(int lk, uint32_t table_smem, const RecArgs &r, const HistArgs &h,
                           uint32_t bucket_bits, int sm_count, size_t smem_optin, bool lean, PartPlan *out);

// Enqueue the whole sequence; `scratch` holds plan.scratch_bytes.
cudaError_t run_partition(int lk, const RecArgs &r, const TableArgs &t, const HistArgs &h,
                          PartPlan plan, void *scratch, bool accumulate, const LaunchCfg &c);

}  // namespace sinet

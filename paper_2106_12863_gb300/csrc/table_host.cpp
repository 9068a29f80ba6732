// Host compilation of a CIDR list (step a-1 of the hot path; runs once per table).
//
// Algorithm 1 compares bitmask(X, Z) with bitmask(Y, Z) for each entry Y/Z of
// the CIDR list. Everything the kernels need is derived here, exactly:
//   * canonical entries: net &= bitmask(len) (the CB of Algorithm 1), deduped,
//     grouped by length and sorted -> per-mask-length binary search;
//   * the union of the entries as disjoint intervals [lo, hi] (nested and
//     duplicate entries merged, adjacent ranges coalesced) with a direct index
//     over the top k address bits -> one index probe plus a short search.
// Membership in the list is membership in the union, so both forms answer
// the same question as the per-entry loop of Algorithm 1.
#include <algorithm>
#include <cmath>
#include <cstring>

#include "sinet.h"
#include "table_host.h"

namespace sinet {

static inline uint32_t prefix_mask(uint32_t len) { return len == 0 ? 0u : (0xFFFFFFFFu << (32 - len)); }

static uint32_t pad16(uint32_t b) { return (b + 15u) & ~15u; }

static uint32_t iv_image_bytes(uint32_t n_iv, uint32_t k) {
    return pad16(4 * n_iv) * 2 + pad16(2 * ((1u << k) + 1));
}

// Where membership flips: the addresses in (0, 2^32) at which an interval
// starts or has just ended, ascending.
static std::vector<uint32_t> toggles(const TableHost &t) {
    std::vector<uint32_t> tog;
    tog.reserve(2 * t.lo.size());
    for (size_t i = 0; i < t.lo.size(); i++) {
        if (t.lo[i]) tog.push_back(t.lo[i]);
        if (t.hi[i] != 0xFFFFFFFFu) tog.push_back(t.hi[i] + 1);
    }
    return tog;
}

// Fills the leaf form (table_host.h) if it fits `budget` bytes: two words a
// leaf where that fits, else four; within a width, the bucket bits that take
// the least room. The budget is never below the toggle form's size plus one
// block, so a one-block toggle table always has a four-word leaf form (its
// buckets need no cut, and the second pure leaf is the extra block).
static void build_leaves(TableHost &t, const std::vector<uint32_t> &tog, size_t budget) {
    const bool first_in = !t.lo.empty() && t.lo[0] == 0;
    const size_t n = tog.size();
    t.leaf_words = 0;
    for (uint32_t words : {2u, 4u}) {
        // a leaf of 2^s addresses holds tog[i] .. tog[i + words] strictly inside
        // (a toggle on its first address is the start state instead) exactly
        // when tog[i] - 1 and tog[i + words] agree above bit s: it must be cut
        // to the highest bit in which they differ
        std::vector<uint8_t> cut(n > words ? n - words : 0);
        for (size_t i = 0; i < cut.size(); i++) {
            uint32_t d = (tog[i] - 1) ^ tog[i + words], s = 31;
            while (!(d >> s)) s--;
            cut[i] = (uint8_t)s;
        }
        uint32_t best_bits = 0;
        size_t best = budget + 1;
        // one walk over the toggles per bucket count: done(bucket, log2 of its
        // leaves' size) for every bucket that is not pure, until it says false. A
        // bucket that holds a toggle off its first address is one leaf, or as many
        // as its smallest cut asks for
        auto walk = [&](uint32_t sh, auto &&done) {
            const uint32_t m = (1u << sh) - 1;
            for (size_t i = 0; i < n;) {
                const uint32_t b = tog[i] >> sh;
                uint32_t s = 0xFF;
                for (; i < n && tog[i] >> sh == b; i++) {
                    if (tog[i] & m) s = std::min(s, sh);
                    if (i >= words && cut[i - words] < sh) s = std::min<uint32_t>(s, cut[i - words]);
                }
                if (s != 0xFF && !done(b, s)) return;
            }
        };
        for (uint32_t kb = 6; kb <= 14; kb++) {
            const uint32_t sh = 32 - kb;
            size_t leaves = 2;
            walk(sh, [&](uint32_t, uint32_t s) {
                leaves += (size_t)1 << (sh - s);
                return 4 * words * leaves < best;
            });
            const size_t bytes = ((4 * words * leaves + 15) & ~(size_t)15) + (4ull << kb);
            if (bytes < best) {
                best = bytes;
                best_bits = kb;
            }
        }
        if (!best_bits) continue;
        const uint32_t sh = 32 - best_bits;
        std::vector<uint8_t> best_log2(1u << best_bits, 0xFF);  // per bucket: leaf size, or 0xFF when pure
        walk(sh, [&](uint32_t b, uint32_t s) {
            best_log2[b] = (uint8_t)s;
            return true;
        });
        t.leaf_bits = best_bits;
        t.leaf_words = words;
        t.leaf_desc.assign(1u << best_bits, 0);
        t.leaves.assign(2 * words, 0x7FFFFFFFu);
        t.leaves[words] = 0xFFFFFFFFu;  // the pure leaf that is inside
        size_t j = 0;  // toggles at or below the current leaf's first address
        for (uint32_t b = 0; b < (1u << best_bits); b++) {
            const uint64_t start = (uint64_t)b << sh, end = start + (1ull << sh);
            while (j < n && tog[j] <= start) j++;
            if (best_log2[b] == 0xFF) {
                t.leaf_desc[b] = (((j & 1) != 0) != first_in ? 4 * words : 0u) << 8 | sh;
                continue;
            }
            const uint32_t s = best_log2[b];
            t.leaf_desc[b] = (uint32_t)(4 * t.leaves.size()) << 8 | s;
            for (uint64_t a = start; a < end; a += 1ull << s) {
                while (j < n && tog[j] <= a) j++;
                const uint32_t in = ((j & 1) != 0) != first_in;
                for (uint32_t k = 0; k < words; k++) {
                    const bool here = j + k < n && tog[j + k] < a + (1ull << s);
                    const uint32_t w = here ? (uint32_t)(tog[j + k] - start - 1) : 0x7FFFFFFFu;
                    t.leaves.push_back(w ^ (k == 0 ? in << 31 : 0u));
                }
            }
        }
        return;
    }
}

int compile_table(const uint32_t *net, const uint8_t *len, uint32_t n, uint32_t index_bits,
                  TableHost &t) {
    if (n > (1u << 24)) return SINET_ERR_TABLE_TOO_LARGE;
    if (n && (!net || !len)) return SINET_ERR_INVALID_ARG;
    if (index_bits > 20) return SINET_ERR_INVALID_ARG;
    for (uint32_t i = 0; i < n; i++)
        if (len[i] > 32) return SINET_ERR_INVALID_ARG;

    // canonicalise, then sort by (len, net) and dedup
    std::vector<uint64_t> keyed(n);
    for (uint32_t i = 0; i < n; i++)
        keyed[i] = (uint64_t)len[i] << 32 | (net[i] & prefix_mask(len[i]));
    std::sort(keyed.begin(), keyed.end());
    keyed.erase(std::unique(keyed.begin(), keyed.end()), keyed.end());
    t.nets.resize(keyed.size());
    std::memset(t.len_offset, 0, sizeof t.len_offset);
    for (size_t i = 0; i < keyed.size(); i++) {
        t.nets[i] = (uint32_t)keyed[i];
        t.len_offset[(keyed[i] >> 32) + 1]++;
    }
    for (int L = 1; L < 34; L++) t.len_offset[L] += t.len_offset[L - 1];

    t.groups.clear();
    for (uint32_t L = 0; L <= 32; L++) {
        uint32_t c = t.len_offset[L + 1] - t.len_offset[L];
        if (c) t.groups.push_back({L, t.len_offset[L], c});
    }
    // probe the lengths that cover the most addresses first (early exit on a hit)
    std::stable_sort(t.groups.begin(), t.groups.end(), [](const TableHost::Group &a, const TableHost::Group &b) {
        long double ca = (long double)a.cnt * std::ldexp(1.0L, 32 - (int)a.len);
        long double cb = (long double)b.cnt * std::ldexp(1.0L, 32 - (int)b.len);
        return ca > cb;
    });

    // union as intervals: sort by start, merge overlapping or adjacent ranges
    std::vector<std::pair<uint32_t, uint32_t>> r(keyed.size());
    for (size_t i = 0; i < keyed.size(); i++) {
        uint32_t L = (uint32_t)(keyed[i] >> 32), s = (uint32_t)keyed[i];
        r[i] = {s, s | ~prefix_mask(L)};
    }
    std::sort(r.begin(), r.end());
    t.lo.clear();
    t.hi.clear();
    for (auto &iv : r) {
        if (!t.lo.empty() && (uint64_t)iv.first <= (uint64_t)t.hi.back() + 1) {
            t.hi.back() = std::max(t.hi.back(), iv.second);
        } else {
            t.lo.push_back(iv.first);
            t.hi.push_back(iv.second);
        }
    }
    const uint32_t n_iv = (uint32_t)t.lo.size();

    // direct index bits: the fewest (>= 6) whose buckets hold at most four
    // candidate intervals (two halving steps), else as many as fit the
    // shared-memory budget
    auto build_index = [&](uint32_t k) {
        const uint32_t nb = 1u << k;
        t.index.assign(nb + 1, n_iv);
        uint32_t j = 0;  // index[b] = first interval with hi >= bucket start
        for (uint32_t b = 0; b < nb; b++) {
            uint64_t start = (uint64_t)b << (32 - k);
            while (j < n_iv && (uint64_t)t.hi[j] < start) j++;
            t.index[b] = j;
        }
        t.index[nb] = n_iv;
        uint32_t mr = 0;
        for (uint32_t b = 0; b < nb && n_iv; b++) {
            uint32_t e = std::min(t.index[b + 1], n_iv - 1);
            uint32_t s0 = t.index[b];
            mr = std::max(mr, e >= s0 ? e - s0 + 1 : 0u);
        }
        return mr;
    };
    uint32_t k = index_bits;
    if (k == 0) {
        uint32_t best = 0;
        for (uint32_t c = 6; c <= 16; c++) {
            if (iv_image_bytes(n_iv, c) > kSmemTableBudget) break;
            best = c;
            if (build_index(c) <= 4) break;
        }
        k = best ? best : 16;  // nothing fits shared memory: global lookups
    }
    t.index_bits = k;
    t.max_range = build_index(k);

    // toggle form `form` (1, 2 or 0, see table_host.h) at kb bucket bits: its
    // image bytes, or ~0 when the form cannot hold this table
    const std::vector<uint32_t> tog = toggles(t);
    auto toggle_size = [&](uint32_t kb, uint32_t form) {
        const uint32_t sh = 32 - kb, m = (1u << sh) - 1;
        const uint32_t most = form ? form : 15, last = form == 1 ? 0x7FFFu : form == 2 ? 0x7FFEu : 0xFFFFFFu;
        size_t blocks = 1;
        for (size_t i = 0; i < tog.size();) {
            const uint32_t b = tog[i] >> sh;
            uint32_t inside = 0;
            for (; i < tog.size() && tog[i] >> sh == b; i++) inside += (tog[i] & m) != 0;
            const uint32_t need = (inside + 3) / 4;
            if (need > most || (need && blocks > last)) return ~size_t(0);
            blocks += need;
        }
        return 16 * blocks + ((size_t)4 << kb);
    };
    auto build_toggles = [&](uint32_t kb, uint32_t form) {
        const uint32_t nb = 1u << kb, sh = 32 - kb, m = (1u << sh) - 1;
        t.desc.assign(nb, 0);
        t.blocks.assign(4, 0x7FFFFFFFu);
        t.max_blocks = 1;
        size_t j = 0;
        bool in = n_iv && t.lo[0] == 0;  // membership just below toggle j
        for (uint32_t b = 0; b < nb; b++) {
            if (j < tog.size() && tog[j] == b << sh) {  // flips on the bucket's first address
                in = !in;
                j++;
            }
            const uint32_t s0 = in;
            const uint32_t first = (uint32_t)t.blocks.size() / 4;
            for (; j < tog.size() && tog[j] >> sh == b; j++) {
                t.blocks.push_back((tog[j] & m) - 1);
                in = !in;
            }
            while (t.blocks.size() % 4) t.blocks.push_back(0x7FFFFFFFu);
            const uint32_t need = (uint32_t)t.blocks.size() / 4 - first, at = need ? first : 0;
            t.max_blocks = std::max(t.max_blocks, need);
            if (form == 1) t.desc[b] = at | (s0 << 31);
            else if (form == 2) t.desc[b] = at | ((need == 2 ? at + 1 : 0u) << 15) | (s0 << 31);
            else t.desc[b] = at | (std::max(need, 1u) << 24) | (s0 << 31);
        }
        t.desc_bits = kb;
        t.toggle_form = form;
    };
    // one block per bucket if some bit count allows it, else two, else as
    // many as needed; within a form, the fewest bits that fit the budget
    uint32_t kb = 0, form = 0;
    for (uint32_t f : {1u, 2u}) {
        for (uint32_t c = 8; c <= 14 && !kb; c++) {
            if (toggle_size(c, f) <= kSmemTableBudget) {
                kb = c;
                form = f;
            }
        }
        if (kb) break;
    }
    if (!kb) {
        size_t best = ~size_t(0);
        for (uint32_t c = 8; c <= 14; c++) {
            const size_t size = toggle_size(c, 0);
            if (size < best) {
                best = size;
                kb = c;
            }
        }
        form = 0;
    }
    if (kb) build_toggles(kb, form);  // (else global lookups)
    const size_t toggle_bytes = pad16(4 * (uint32_t)t.blocks.size()) + pad16(4 * (uint32_t)t.desc.size());
    if (t.max_blocks <= 15 && toggle_bytes <= kSmemTableBudget) build_leaves(t, tog, std::max<size_t>(kLeafBudget, toggle_bytes + 16));
    return SINET_OK;
}

std::vector<uint8_t> serialise(const TableHost &t, TableImage &img) {
    const uint32_t n_iv = (uint32_t)t.lo.size();
    const uint32_t n_pairs = n_iv ? n_iv : 1;  // an empty table keeps one empty interval
    const uint32_t nb1 = (1u << t.index_bits) + 1;
    img = TableImage{};
    uint32_t off = 0;
    img.off_blocks = off;
    off += pad16(4 * (uint32_t)t.blocks.size());
    img.off_desc = off;
    off += pad16(4 * (uint32_t)t.desc.size());
    img.iv_bytes = off;
    img.iv_fits_smem = !t.desc.empty() && t.max_blocks <= 15 && img.iv_bytes <= kSmemTableBudget;
    img.off_nets = off;
    off += pad16(4 * (uint32_t)t.nets.size());
    img.off_groups = off;
    off += 16 * (uint32_t)t.groups.size();
    img.pml_bytes = off - img.off_nets;
    img.pml_fits_smem = img.pml_bytes <= kSmemTableBudget;
    img.off_lo = off;
    off += pad16(4 * n_pairs);
    img.off_hi = off;
    off += pad16(4 * n_pairs);
    img.off_idx32 = off;
    off += pad16(4 * nb1);
    // the leaf form, and after it a trailer of four words saying where it is:
    // {off_leaves, off_leaf_desc, leaf_bits, leaf_words}
    if (t.leaf_words) {
        img.off_leaves = off;
        off += pad16(4 * (uint32_t)t.leaves.size());
        img.off_leaf_desc = off;
        off += pad16(4 * (uint32_t)t.leaf_desc.size());
        img.leaf_bytes = off - img.off_leaves;
    }
    off += 16;
    img.total = off;

    std::vector<uint8_t> buf(img.total, 0);
    uint32_t *lo = reinterpret_cast<uint32_t *>(buf.data() + img.off_lo);
    uint32_t *hi = reinterpret_cast<uint32_t *>(buf.data() + img.off_hi);
    if (n_iv) {
        std::memcpy(lo, t.lo.data(), 4 * n_iv);
        std::memcpy(hi, t.hi.data(), 4 * n_iv);
    } else {
        lo[0] = 1;  // lo > hi: contains nothing
        hi[0] = 0;
    }
    if (!t.blocks.empty()) std::memcpy(buf.data() + img.off_blocks, t.blocks.data(), 4 * t.blocks.size());
    if (!t.desc.empty()) std::memcpy(buf.data() + img.off_desc, t.desc.data(), 4 * t.desc.size());
    if (!t.nets.empty()) std::memcpy(buf.data() + img.off_nets, t.nets.data(), 4 * t.nets.size());
    uint32_t *g = reinterpret_cast<uint32_t *>(buf.data() + img.off_groups);
    for (size_t i = 0; i < t.groups.size(); i++) {
        g[4 * i + 0] = t.groups[i].len;
        g[4 * i + 1] = t.groups[i].off;
        g[4 * i + 2] = t.groups[i].cnt;
        g[4 * i + 3] = 0;
    }
    std::memcpy(buf.data() + img.off_idx32, t.index.data(), 4 * nb1);
    if (t.leaf_words) {
        std::memcpy(buf.data() + img.off_leaves, t.leaves.data(), 4 * t.leaves.size());
        std::memcpy(buf.data() + img.off_leaf_desc, t.leaf_desc.data(), 4 * t.leaf_desc.size());
    }
    const uint32_t trailer[4] = {img.off_leaves, img.off_leaf_desc, t.leaf_bits, t.leaf_words};
    std::memcpy(buf.data() + img.total - 16, trailer, 16);
    return buf;
}

}  // namespace sinet

extern "C" sinet_status sinet_compile_prefix_table(const uint32_t *h_net, const uint8_t *h_len,
                                                   uint32_t n, uint32_t index_bits,
                                                   uint32_t *nets_by_len, uint32_t *len_offset,
                                                   uint32_t *iv_lo, uint32_t *iv_hi,
                                                   uint32_t *index, uint32_t *counts) {
    if (!len_offset || !counts) return SINET_ERR_INVALID_ARG;
    sinet::TableHost t;
    int rc = sinet::compile_table(h_net, h_len, n, index_bits, t);
    if (rc != SINET_OK) return (sinet_status)rc;
    if (nets_by_len && !t.nets.empty()) std::memcpy(nets_by_len, t.nets.data(), 4 * t.nets.size());
    std::memcpy(len_offset, t.len_offset, sizeof t.len_offset);
    if (iv_lo && !t.lo.empty()) std::memcpy(iv_lo, t.lo.data(), 4 * t.lo.size());
    if (iv_hi && !t.hi.empty()) std::memcpy(iv_hi, t.hi.data(), 4 * t.hi.size());
    if (index) std::memcpy(index, t.index.data(), 4 * t.index.size());
    counts[0] = (uint32_t)t.nets.size();
    counts[1] = (uint32_t)t.lo.size();
    counts[2] = t.index_bits;
    counts[3] = t.max_range;
    return SINET_OK;
}

extern "C" sinet_status sinet_prefix_table_image(const uint32_t *h_net, const uint8_t *h_len,
                                                 uint32_t n, uint8_t *image, size_t capacity,
                                                 uint32_t *layout, size_t *bytes) {
    if (!layout || !bytes) return SINET_ERR_INVALID_ARG;
    sinet::TableHost t;
    int rc = sinet::compile_table(h_net, h_len, n, 0, t);
    if (rc != SINET_OK) return (sinet_status)rc;
    sinet::TableImage img;
    std::vector<uint8_t> buf = sinet::serialise(t, img);
    *bytes = buf.size();
    const uint32_t v[16] = {img.off_blocks, img.off_desc, t.desc_bits, img.iv_bytes,
                            img.off_nets, img.off_groups, (uint32_t)t.groups.size(), img.pml_bytes,
                            img.off_lo, img.off_hi, img.off_idx32, t.index_bits,
                            (uint32_t)t.lo.size(), t.max_blocks | (t.toggle_form << 8),
                            img.iv_fits_smem ? 1u : 0u, img.pml_fits_smem ? 1u : 0u};
    std::memcpy(layout, v, sizeof v);
    if (image) {
        if (capacity < buf.size()) return SINET_ERR_INVALID_ARG;
        std::memcpy(image, buf.data(), buf.size());
    }
    return SINET_OK;
}

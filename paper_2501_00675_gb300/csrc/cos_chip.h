// Row schedule of the on-chip walk (cos_chip.cu): host-only, no CUDA.
//
// The on-chip walk keeps the node values of a level and the propagators of a chunk of
// samples in shared memory, one row of RB bytes per node and per propagator slot.  A
// warp reads the rows of 128 / RB nodes in one shared-memory phase, so those rows'
// parents (and slots) should lie in different 128 / RB bank groups, at every step of
// the rows' in-edge lists.  The order in which the rows of a level are processed, and
// with it their place in the level buffer, is free: no result depends on it, since a
// row adds its in-edges in the graph's order wherever it is processed.  build_chip()
// orders each level by decreasing in-edge count and, inside one count, fills a phase with
// rows whose bank groups are still unused (chip_order_class): random order costs 1.5 / 2.1
// / 2.6 passes per phase with 2 / 4 / 8 rows per phase, this order 1.08 / 1.37 / 1.8 on
// the medium graph's level sizes, for about 60 ns of host time per row.
#pragma once

#include <algorithm>
#include <cstdint>
#include <numeric>
#include <vector>

namespace cosgpu {

// Rows are processed in groups of 64 with one in-edge count, a lane summing rows r and
// r + 32 of a group side by side (control and edge-word loads are then paid once for two
// rows: 2.29 -> 1.73 ms on the medium graph in FP32 against one row per lane).  A row with
// fewer in-edges than its group (at the boundary between two counts, or behind the level's
// end) has its list filled up with the word (place 0, slot P), whose node and propagator
// rows hold zeros: such a step adds 0 * 0.
constexpr int kChipGroup = 64;
constexpr int kChipMaxFanin = 1024;
constexpr int kChipMaxTables = 4096;          // 16-byte units of levels and group descriptors, kept in shared memory

struct ChipLevel {
    int32_t width;
    int32_t groups;
    int32_t first;    // number of the level's first group
    int32_t pad;
};

struct ChipSchedule {
    int phase_rows = 0;              // rows per shared-memory phase the order was made for (128 / RB)
    int max_width = 0;               // widest level kept on chip (every level but the sink's)
    std::vector<ChipLevel> lev;      // [L], levels 1 .. L-2 used
    std::vector<uint32_t> grp;       // per group: edge words per row (1 ..) | (first word / 64) << 11
    std::vector<uint32_t> words;     // edge words: parent's place in its level (from 1) | slot << 16
    std::vector<uint32_t> sink;      // the sink's in-edges, in the graph's order
};

// Edge words of a group with n words per row, in blocks of the rows' next four: n = 1 left
// [32][row r, row r + 32], 2 left [32][2 of row r, 2 of row r + 32], more [row r's, row
// r + 32's half][32][4] (three take the room of four), so that a lane loads both its rows'
// next words with one 8- or one or two 16-byte loads.
inline uint32_t chip_block(uint32_t n) { return (n >= 3 ? 4 : n) * kChipGroup; }   // words of a block with n left
inline uint32_t chip_word_at(uint32_t first, uint32_t n, int row, uint32_t e) {
    for (; e >= 4; e -= 4, n -= 4) first += chip_block(4);
    const uint32_t half = (uint32_t)row / 32, r = (uint32_t)row % 32;
    return n >= 3 ? first + half * 128 + r * 4 + e : first + (2 * r + half) * n + e;
}
inline uint32_t chip_words_of(uint32_t n) { return (n - 1) / 4 * chip_block(4) + chip_block((n - 1) % 4 + 1); }

// Candidates a place of a phase is chosen from.
constexpr int kWindow = 24;

// Appends the rows of one in-edge count n to `out` in processing order.  `words` are the
// rows' edge words (n per row, row-major).  Rows wait in B * B buckets by the bank groups
// of their first parent and slot; a place of a phase takes candidates from the buckets
// whose two groups the phase has not used, and of these the row with the fewest clashes at
// the other steps (one bit per step, table and group).
inline void chip_order_class(int n, int B, const std::vector<int32_t>& rows, const uint32_t* words,
                             std::vector<int32_t>& out) {
    const int cnt = (int)rows.size();
    // phases of 16 and 32 rows (rows of 8 and 4 bytes) keep the order: such graphs run on
    // chip for small sample counts only, which the ordering's time would outweigh
    if (B <= 1 || B > 8 || n == 0 || cnt <= 1) {
        out.insert(out.end(), rows.begin(), rows.end());
        return;
    }
    const int steps = std::min(n, 64 / (2 * B));   // steps whose clashes one 64-bit mask holds
    const int nb = B * B;
    std::vector<uint64_t> mask((size_t)cnt);   // by bucket
    std::vector<int32_t> id((size_t)cnt);
    int begin[65] = {0}, end[64];
    auto bucket = [&](int r) {
        const uint32_t q = words[(size_t)r * (size_t)n];
        return (int)(q & 0xffffu) % B * B + (int)(q >> 16) % B;
    };
    for (int r = 0; r < cnt; ++r) begin[bucket(r) + 1]++;
    for (int b = 0; b < nb; ++b) begin[b + 1] += begin[b];
    for (int b = 0; b < nb; ++b) end[b] = begin[b];
    // rows enter their buckets in a scattered order (a step coprime to their number, near
    // the golden section): a place's bank group must not go with the row's number, by which
    // the next level's in-edge lists may be sorted
    int step = (int)(0.618 * cnt) | 1;
    while (std::gcd(step, cnt) != 1) step += 2;
    for (int k = 0, r = 0; k < cnt; ++k, r = (int)(((int64_t)r + step) % cnt)) {
        uint64_t m = 0;
        for (int e = 0; e < steps; ++e) {
            const uint32_t q = words[(size_t)r * (size_t)n + (size_t)e];
            m |= 1ull << (2 * e * B + (int)(q & 0xffffu) % B) | 1ull << ((2 * e + 1) * B + (int)(q >> 16) % B);
        }
        const int at = end[bucket(r)]++;
        mask[(size_t)at] = m;
        id[(size_t)at] = rows[(size_t)r];
    }
    int left = cnt, start = (int)(out.size() % (size_t)B);   // (a phase begun by the rows of a larger count)
    const unsigned all = (1u << B) - 1u;
    while (left > 0) {
        uint64_t used = 0;
        unsigned free_p = all, free_g = all;
        const int places = B - start;
        start = 0;
        for (int k = 0; k < places && left > 0; ++k) {
            int best_b = -1, best_at = 0, best_cost = 1 << 30, best_size = 0;
            if (k == 0) {   // the fullest bucket
                for (int b = 0; b < nb; ++b)
                    if (best_b < 0 || end[b] - begin[b] > end[best_b] - begin[best_b]) best_b = b;
                best_at = end[best_b] - 1;
            } else {
                // fewest clashes, then the fullest bucket (so that none is left over); no
                // clash and a bucket of average size end the search
                const int each = std::max(1, kWindow / (__builtin_popcount(free_p) * __builtin_popcount(free_g)));
                bool done = false;
                for (unsigned fp = free_p; fp && !done; fp &= fp - 1)
                    for (unsigned fg = free_g; fg && !done; fg &= fg - 1) {
                        const int b = __builtin_ctz(fp) * B + __builtin_ctz(fg), size = end[b] - begin[b];
                        for (int c = end[b] - 1; c >= begin[b] && c >= end[b] - each; --c) {
                            const uint64_t clash = used & mask[(size_t)c];
                            const int cost = clash ? __builtin_popcountll(clash) : 0;
                            if (cost > best_cost || (cost == best_cost && size <= best_size)) continue;
                            best_cost = cost;
                            best_size = size;
                            best_b = b;
                            best_at = c;
                            if (cost == 0) {
                                done = size * nb >= left;
                                break;
                            }
                        }
                    }
                for (int b = 0; b < nb && best_b < 0; ++b)   // those buckets are empty: any row
                    if (end[b] > begin[b]) {
                        best_b = b;
                        best_at = end[b] - 1;
                    }
            }
            const int last = --end[best_b], row = id[(size_t)best_at];
            used |= mask[(size_t)best_at];
            mask[(size_t)best_at] = mask[(size_t)last];
            id[(size_t)best_at] = id[(size_t)last];
            --left;
            free_p &= ~(1u << (best_b / B));
            free_g &= ~(1u << (best_b % B));
            if (!free_p) free_p = all;
            if (!free_g) free_g = all;
            out.push_back(row);
        }
    }
}

// Schedule of a graph in destination-sorted CSR form.  off[L+1]: first node of each
// level; row_ptr[N+1]; src(q), slot(q): parent (index inside the previous level) and
// slot of in-edge q.  Returns false (schedule not usable) when an index does not fit
// 16 bits, a row has more than kChipMaxFanin in-edges or the tables are too long.
template <class Src, class Slot>
bool build_chip(int32_t L, const int64_t* off, const int32_t* row_ptr, int64_t P, int phase_rows, const Src& src,
                const Slot& slot, ChipSchedule& s) {
    if (P > 65534) return false;
    int64_t wmax = 1;
    for (int32_t l = 0; l + 1 < L; ++l) wmax = std::max(wmax, off[l + 1] - off[l]);
    if (wmax > 65534) return false;
    s.phase_rows = phase_rows;
    s.max_width = (int)wmax;
    s.lev.assign((size_t)L, ChipLevel{0, 0, 0, 0});
    s.grp.clear();
    s.words.clear();
    s.sink.clear();
    std::vector<uint16_t> place_prev(1, 1), place;   // place of each node in its level's buffer (0: the zero row)
    std::vector<std::vector<int32_t>> classes;
    std::vector<int32_t> order;
    std::vector<uint32_t> cw;
    for (int32_t l = 1; l < L; ++l) {
        const int64_t W = off[l + 1] - off[l];
        const int32_t* rp = row_ptr + off[l];
        auto word = [&](int32_t q) { return (uint32_t)place_prev[(size_t)src(q)] | (uint32_t)slot(q) << 16; };
        if (l == L - 1) {
            for (int32_t r = 0; r < (int32_t)W; ++r) {
                if (rp[r + 1] - rp[r] > kChipMaxFanin) return false;
                for (int32_t q = rp[r]; q < rp[r + 1]; ++q) s.sink.push_back(word(q));
            }
            break;
        }
        int maxn = 0;
        for (int32_t r = 0; r < (int32_t)W; ++r) maxn = std::max(maxn, rp[r + 1] - rp[r]);
        if (maxn > kChipMaxFanin) return false;
        if ((int)classes.size() <= maxn) classes.resize((size_t)maxn + 1);
        for (auto& c : classes) c.clear();
        for (int32_t r = 0; r < (int32_t)W; ++r) classes[(size_t)(rp[r + 1] - rp[r])].push_back(r);
        order.clear();
        for (int n = maxn; n >= 0; --n) {
            const std::vector<int32_t>& rows = classes[(size_t)n];
            if (rows.empty()) continue;
            cw.resize(rows.size() * (size_t)n);
            for (size_t r = 0; r < rows.size(); ++r)
                for (int e = 0; e < n; ++e) cw[r * (size_t)n + (size_t)e] = word(rp[rows[r]] + e);
            chip_order_class(n, phase_rows, rows, cw.data(), order);
        }
        place.assign((size_t)W, 0);
        for (size_t k = 0; k < order.size(); ++k) place[(size_t)order[k]] = (uint16_t)(k + 1);
        ChipLevel& lv = s.lev[(size_t)l];
        lv.width = (int32_t)W;
        lv.groups = (int32_t)((W + kChipGroup - 1) / kChipGroup);
        lv.first = (int32_t)s.grp.size();
        for (int64_t g = 0; g < lv.groups; ++g) {
            const int64_t k0 = g * kChipGroup, k1 = std::min<int64_t>(W, k0 + kChipGroup);
            auto fanin = [&](int64_t k) { return rp[order[(size_t)k] + 1] - rp[order[(size_t)k]]; };
            const uint32_t n = (uint32_t)std::max(fanin(k0), 1);   // the first row has the most
            const uint32_t first = (uint32_t)s.words.size();
            if (first / kChipGroup >= (1u << 21)) return false;
            s.grp.push_back(n | first / kChipGroup << 11);
            s.words.resize(s.words.size() + (size_t)chip_words_of(n), (uint32_t)P << 16);
            for (int64_t k = k0; k < k1; ++k)
                for (int32_t e = 0; e < fanin(k); ++e)
                    s.words[chip_word_at(first, n, (int)(k - k0), (uint32_t)e)] = word(rp[order[(size_t)k]] + e);
        }
        place_prev.swap(place);
    }
    return s.lev.size() + (s.grp.size() + 3) / 4 <= (size_t)kChipMaxTables;
}

}  // namespace cosgpu

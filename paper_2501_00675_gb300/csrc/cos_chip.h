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
// the medium graph's level sizes, for about 35 ns of host time per row (Grace; medium graph,
// whole schedule: 0.79 ms, before the shared inner loops below 1.32).
#pragma once

#include <algorithm>
#include <cstdint>
#include <future>
#include <numeric>
#include <system_error>
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

// Rows of one in-edge count that are worth a thread (some 40 us) while others are ordered: a
// place of a phase of 8 rows takes twice the time of one of 4 (80 / 35 ns).
constexpr int kOrderThread = 8192;   // rows x rows per phase

// Candidates a place of a phase is chosen from.
constexpr int kWindow = 24;

// Processing order of the rows of one in-edge count n, written to out[0, cnt); `start`: rows of
// a larger count that begin the first phase.  Row r's n edge words are words[at[r] .. ].  Rows
// wait in B * B buckets by the bank groups of their first parent and slot; a place of a
// phase takes candidates from the buckets whose two groups the phase has not used, and of
// these the row with the fewest clashes at the other steps (one bit per step, table and
// group).
struct ChipOrderScratch {
    std::vector<uint64_t> mask, by_bucket;
    std::vector<int32_t> id;
    std::vector<uint8_t> bucket;
};
template <int B>
inline void chip_order_phases(int n, int cnt, int start, const int32_t* rows, const int32_t* at, const uint32_t* words,
                              ChipOrderScratch& sc, int32_t* out) {
    constexpr int nb = B * B, LOG = B == 2 ? 1 : B == 4 ? 2 : 3;
    const int steps = std::min(n, 64 / (2 * B));   // steps whose clashes one 64-bit mask holds
    sc.mask.resize((size_t)cnt);
    sc.by_bucket.resize((size_t)cnt);
    sc.id.resize((size_t)cnt);
    sc.bucket.resize((size_t)cnt);
    uint64_t* const mask = sc.by_bucket.data();   // by bucket
    int32_t* const id = sc.id.data();
    int begin[nb + 1] = {0}, end[nb];
    for (int r = 0; r < cnt; ++r) {
        const uint32_t* w = words + at[rows[r]];
        uint64_t m = 0;
        for (int e = 0; e < steps; ++e)
            m |= (1ull << (w[e] & (B - 1)) | 1ull << (B + (w[e] >> 16 & (B - 1)))) << 2 * B * e;
        sc.mask[(size_t)r] = m;
        const int b = (int)((w[0] & (B - 1)) << LOG | (w[0] >> 16 & (B - 1)));
        sc.bucket[(size_t)r] = (uint8_t)b;
        begin[b + 1]++;
    }
    for (int b = 0; b < nb; ++b) begin[b + 1] += begin[b];
    for (int b = 0; b < nb; ++b) end[b] = begin[b];
    // rows enter their buckets in a scattered order (a step coprime to their number, near
    // the golden section): a place's bank group must not go with the row's number, by which
    // the next level's in-edge lists may be sorted
    int step = (int)(0.618 * cnt) | 1;
    while (std::gcd(step, cnt) != 1) step += 2;
    step %= cnt;
    for (int k = 0, r = 0; k < cnt; ++k) {
        const int to = end[sc.bucket[(size_t)r]]++;
        mask[to] = sc.mask[(size_t)r];
        id[to] = rows[r];
        if ((r += step) >= cnt) r -= cnt;
    }
    const unsigned all = (1u << B) - 1u;
    int32_t* const last_out = out + cnt;
    while (out < last_out) {
        uint64_t used = 0;
        unsigned free_p = all, free_g = all;
        const int places = B - start;
        start = 0;
        for (int k = 0; k < places && out < last_out; ++k) {
            const int left = (int)(last_out - out);
            int best_b = -1, best_at = 0, best_cost = 1 << 30, best_size = 0;
            if (k == 0) {   // the fullest bucket
                for (int b = 0; b < nb; ++b)
                    if (end[b] - begin[b] > best_size) {
                        best_size = end[b] - begin[b];
                        best_b = b;
                    }
                best_at = end[best_b] - 1;
            } else {
                // fewest clashes, then the fullest bucket (so that none is left over); no
                // clash and a bucket of average size end the search
                static constexpr int8_t kEach[9] = {0, 24, 12, 8, 6, 4, 4, 3, 3};   // kWindow / n
                const int np = __builtin_popcount(free_p), ng = __builtin_popcount(free_g);
                const int each = std::max(1, (ng == 1 ? kEach[np] : np == 1 ? kEach[ng] : kWindow / (np * ng)));
                bool done = false;
                for (unsigned fp = free_p; fp && !done; fp &= fp - 1)
                    for (unsigned fg = free_g; fg && !done; fg &= fg - 1) {
                        const int b = __builtin_ctz(fp) << LOG | __builtin_ctz(fg), size = end[b] - begin[b];
                        if (size == 0) continue;
                        // the bucket's first candidate with the fewest clashes
                        const uint64_t* c = mask + end[b] - 1;
                        const int nc = std::min(size, each);
                        int cost = 1 << 20, which = 0;
                        for (int q = 0; q < nc; ++q) {
                            const uint64_t clash = used & c[-q];
                            if (clash == 0) {
                                cost = 0;
                                which = q;
                                break;
                            }
                            const int x = __builtin_popcountll(clash);
                            which = x < cost ? q : which;
                            cost = std::min(cost, x);
                        }
                        if (cost > best_cost || (cost == best_cost && size <= best_size)) continue;
                        best_cost = cost;
                        best_size = size;
                        best_b = b;
                        best_at = end[b] - 1 - which;
                        done = cost == 0 && size * nb >= left;
                    }
                for (int b = 0; b < nb && best_b < 0; ++b)   // those buckets are empty: any row
                    if (end[b] > begin[b]) {
                        best_b = b;
                        best_at = end[b] - 1;
                    }
            }
            const int last = --end[best_b];
            used |= mask[best_at];
            *out++ = id[best_at];
            mask[best_at] = mask[last];
            id[best_at] = id[last];
            free_p &= ~(1u << (best_b >> LOG));
            free_g &= ~(1u << (best_b & (B - 1)));
            if (!free_p) free_p = all;
            if (!free_g) free_g = all;
        }
    }
}

inline void chip_order_class(int n, int B, int cnt, int start, const int32_t* rows, const int32_t* at, const uint32_t* words,
                             ChipOrderScratch& sc, int32_t* out) {
    // phases of 16 and 32 rows (rows of 8 and 4 bytes) keep the order: such graphs run on
    // chip for small sample counts only, which the ordering's time would outweigh
    if (n == 0 || cnt <= 1 || (B != 2 && B != 4 && B != 8)) std::copy(rows, rows + cnt, out);
    else if (B == 2) chip_order_phases<2>(n, cnt, start, rows, at, words, sc, out);
    else if (B == 4) chip_order_phases<4>(n, cnt, start, rows, at, words, sc, out);
    else chip_order_phases<8>(n, cnt, start, rows, at, words, sc, out);
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
    s.max_width = (int)wmax;
    s.lev.assign((size_t)L, ChipLevel{0, 0, 0, 0});
    s.grp.clear();
    s.words.clear();
    s.sink.clear();
    std::vector<uint16_t> place_prev(1, 1), place;   // place of each node in its level's buffer (0: the zero row)
    std::vector<int32_t> classes, order, begin, at;
    std::vector<uint32_t> words;   // of the level's in-edges, in the graph's order
    ChipOrderScratch scratch;
    for (int32_t l = 1; l < L; ++l) {
        const int32_t W = (int32_t)(off[l + 1] - off[l]);
        const int32_t* rp = row_ptr + off[l];
        const int32_t q0 = rp[0], ne = rp[W] - q0;
        int maxn = 0;
        for (int32_t r = 0; r < W; ++r) maxn = std::max(maxn, rp[r + 1] - rp[r]);
        if (maxn > kChipMaxFanin) return false;
        words.resize((size_t)ne);
        for (int32_t q = 0; q < ne; ++q)
            words[(size_t)q] = (uint32_t)place_prev[(size_t)src(q0 + q)] | (uint32_t)slot(q0 + q) << 16;
        if (l == L - 1) {
            s.sink = words;
            break;
        }
        // rows by decreasing in-edge count; begin[m]: first with maxn - m in-edges
        begin.assign((size_t)maxn + 2, 0);
        for (int32_t r = 0; r < W; ++r) begin[(size_t)(maxn - (rp[r + 1] - rp[r])) + 1]++;
        for (int m = 0; m <= maxn; ++m) begin[(size_t)m + 1] += begin[(size_t)m];
        classes.resize((size_t)W);
        order.resize((size_t)W);
        at.resize((size_t)W);
        for (int32_t r = 0; r < W; ++r) {
            classes[(size_t)begin[(size_t)(maxn - (rp[r + 1] - rp[r]))]++] = r;
            at[(size_t)r] = rp[r] - q0;
        }
        // the classes do not depend on one another: all but the last long one on threads of their own
        std::vector<std::future<void>> others;
        int last_long = -1;
        auto rows_of = [&](int m) { return begin[(size_t)m] - (m ? begin[(size_t)m - 1] : 0); };   // (one past each class by now)
        for (int m = 0; m <= maxn; ++m)
            if (rows_of(m) * phase_rows >= kOrderThread && m < maxn) last_long = m;
        for (int m = 0; m <= maxn; ++m) {
            const int cnt = rows_of(m), first = begin[(size_t)m] - cnt;
            if (cnt == 0) continue;
            auto run = [&, m, cnt, first](ChipOrderScratch& sc) {
                chip_order_class(maxn - m, phase_rows, cnt, first % phase_rows, classes.data() + first, at.data(), words.data(), sc,
                                 order.data() + first);
            };
            if (cnt * phase_rows >= kOrderThread && m != last_long && m < maxn && phase_rows > 1 && phase_rows <= 8) {
                try {
                    others.push_back(std::async(std::launch::async, [run] {
                        ChipOrderScratch own;
                        run(own);
                    }));
                    continue;
                } catch (const std::system_error&) {   // no thread to be had
                }
            }
            run(scratch);
        }
        for (std::future<void>& f : others) f.get();
        place.resize((size_t)W);
        for (int32_t k = 0; k < W; ++k) place[(size_t)order[(size_t)k]] = (uint16_t)(k + 1);
        ChipLevel& lv = s.lev[(size_t)l];
        lv.width = W;
        lv.groups = (W + kChipGroup - 1) / kChipGroup;
        lv.first = (int32_t)s.grp.size();
        for (int32_t k0 = 0; k0 < W; k0 += kChipGroup) {
            const int32_t k1 = std::min(W, k0 + kChipGroup);
            auto fanin = [&](int32_t r) { return (uint32_t)(rp[r + 1] - rp[r]); };
            const uint32_t n = std::max(fanin(order[(size_t)k0]), 1u);   // the first row has the most
            const uint32_t first = (uint32_t)s.words.size();
            if (first / kChipGroup >= (1u << 21)) return false;
            s.grp.push_back(n | first / kChipGroup << 11);
            s.words.resize(s.words.size() + (size_t)chip_words_of(n), (uint32_t)P << 16);
            for (int32_t k = k0; k < k1; ++k) {
                const int32_t r = order[(size_t)k];
                const uint32_t *w = words.data() + at[(size_t)r], *w_end = w + fanin(r);
                uint32_t block = first;
                for (uint32_t m = n; w < w_end; m -= 4, block += chip_block(4))   // (the row's next four)
                    for (uint32_t e = 0; e < 4 && w < w_end; ++e) s.words[chip_word_at(block, m, k - k0, e)] = *w++;
            }
        }
        place_prev.swap(place);
    }
    return s.lev.size() + (s.grp.size() + 3) / 4 <= (size_t)kChipMaxTables;
}

}  // namespace cosgpu

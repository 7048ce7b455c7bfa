// Host-only probe of the on-chip walk's row schedule (build_chip in csrc/cos_chip.h).
// Reads a graph in destination-sorted form from standard input ("L P phase_rows", the
// level widths, row_ptr[N+1], then "src slot" per in-edge), builds the schedule, and
// walks it with the kernel's index arithmetic for every launch shape (threads, row
// bytes, lane bytes), checking that groups, edge words, places and staging columns stay
// in bounds.  A node's value is an order-sensitive fold of its in-edges modulo 2^64
// (v = v * 1000003 + parent * (slot + 1)), so a lost, repeated or reordered in-edge
// shows.  Prints the sink's value, one line per launch shape, or an error and exits 1.
#include <cstdio>
#include <cstdlib>
#include <vector>

#include "../../paper_2501_00675_gb300/csrc/cos_chip.h"

using namespace cosgpu;

static void fail(const char* what) {
    std::printf("error: %s\n", what);
    std::exit(1);
}

int main() {
    long long L, P, B;
    if (std::scanf("%lld %lld %lld", &L, &P, &B) != 3) return 2;
    std::vector<int64_t> off(1, 0);
    for (long long l = 0; l < L; ++l) {
        long long w;
        if (std::scanf("%lld", &w) != 1) return 2;
        off.push_back(off.back() + w);
    }
    std::vector<int32_t> rp((size_t)off.back() + 1);
    for (auto& x : rp)
        if (std::scanf("%d", &x) != 1) return 2;
    std::vector<int> src((size_t)rp.back()), slot((size_t)rp.back());
    for (size_t q = 0; q < src.size(); ++q)
        if (std::scanf("%d %d", &src[q], &slot[q]) != 2) return 2;
    ChipSchedule s;
    if (!build_chip((int32_t)L, off.data(), rp.data(), P, (int)B, [&](int32_t q) { return src[(size_t)q]; },
                    [&](int32_t q) { return slot[(size_t)q]; }, s)) {
        std::printf("none\n");
        return 0;
    }
    for (int T = 128; T <= 512; T *= 2)
        for (int rb = 4; rb <= 128; rb *= 2)
            for (int lb = 4; lb <= 16; lb *= 2) {
                if (lb > rb || rb / lb > 8 || T / 32 < rb / lb || (long long)s.max_width * rb > 512LL * T) continue;
                const int lanes = rb / lb, gstep = T / 32 / lanes;
                // place 0 is the zero row; slot P is the zero slot (its fold factor is 0)
                std::vector<unsigned long long> lev((size_t)s.max_width + 1, 0), child;
                lev[1] = 1;
                auto fold = [&](unsigned long long v, uint32_t m) {
                    if ((m & 0xffffu) >= lev.size() || (long long)(m >> 16) > P) fail("edge word out of range");
                    if (((m & 0xffffu) == 0) != ((long long)(m >> 16) == P)) fail("half of a filling word");
                    return (m & 0xffffu) == 0 ? v : v * 1000003ull + lev[m & 0xffffu] * (unsigned long long)((m >> 16) + 1);
                };
                for (int l = 1; l + 1 < (int)L; ++l) {
                    const ChipLevel& lv = s.lev[(size_t)l];
                    const int W = lv.width;
                    if (lv.groups != (W + kChipGroup - 1) / kChipGroup) fail("groups of a level");
                    child.assign((size_t)s.max_width + 1, 0);
                    std::vector<int> seen((size_t)W, 0);
                    for (int tid = 0; tid < T; ++tid) {
                        const int warp = tid / 32, lane = tid % 32;
                        const int r32 = (warp & (lanes - 1)) * (32 / lanes) + lane / lanes;
                        int k = 0;
                        for (int g = warp / lanes; g < lv.groups; g += gstep, ++k) {
                            if ((size_t)(lv.first + g) >= s.grp.size()) fail("group out of range");
                            const uint32_t d = s.grp[(size_t)(lv.first + g)], n = d & 0x7ffu, first = d >> 11 << 6;
                            if ((k + 1) * (lb / 2) > 128) fail("staging columns");
                            for (int half = 0; half < 2; ++half) {
                                unsigned long long v = 0;
                                for (uint32_t e = 0; e < n; ++e) {
                                    const uint32_t w = chip_word_at(first, n, r32 + 32 * half, e);
                                    if (w >= s.words.size()) fail("word out of range");
                                    v = fold(v, s.words[w]);
                                }
                                const int row = g * kChipGroup + r32 + 32 * half;
                                if (row < W) {
                                    child[(size_t)row + 1] = v;
                                    seen[(size_t)row]++;
                                } else if (v != 0) fail("in-edges behind the level");
                            }
                        }
                    }
                    for (int x : seen)
                        if (x != lanes) fail("row not covered once per piece");
                    lev.swap(child);
                }
                unsigned long long v = 0;
                for (uint32_t m : s.sink) v = fold(v, m);
                std::printf("%llu\n", v);
            }
    return 0;
}

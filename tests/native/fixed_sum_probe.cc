// Host-only probe of the integer sums (cos_fixed.h): reads "extra n" and n doubles as
// 64-bit hexadecimal words, prints the sum as one (or "range" where the values need the
// floating-point sum), until the end of the input.
#include <cinttypes>
#include <cstdio>
#include <vector>

#include "../../paper_2501_00675_gb300/csrc/cos_fixed.h"

int main() {
    int extra, n;
    while (std::scanf("%d %d", &extra, &n) == 2) {
        std::vector<uint64_t> x((size_t)n);
        int emax = 0;
        for (auto& v : x) {
            if (std::scanf("%" SCNx64, &v) != 1) return 1;
            const int e = (int)((v >> 52) & 0x7ff);
            emax = e > emax ? e : emax;
        }
        if (emax < cosgpu::kFixedMin || emax > cosgpu::kFixedMax) {
            std::puts("range");
            continue;
        }
        cosgpu::Fixed f{{0, 0, 0, 0}};
        for (uint64_t v : x) cosgpu::fixed_add_double(f, (uint32_t)(v >> 32), (uint32_t)v, emax + extra);
        uint32_t hi, lo;
        cosgpu::fixed_to_double(f, emax + extra, hi, lo);
        std::printf("%016" PRIx64 "\n", (uint64_t)hi << 32 | lo);
    }
    return 0;
}

// Sums of doubles in 128-bit integers: no CUDA, shared with a host test.
//
// A warp-wide FP64 operation occupies a quarter of an SM for 64 cycles on GB300, and a
// compensated addition is five of them: one warp took 15,800 cycles (8 us) for the sum of
// a block of 1,024 samples, longer than the whole walk of a small graph.  Here every
// value is shifted to a common binary point (given by the largest exponent) and added
// with 32-bit integer instructions, some 35 per value, which any number of lanes share:
// integer addition is associative, so the result depends on no order.  The bits of a
// value below 2^-116 of the largest one's leading bit are dropped (2^-96 for `extra` =
// 20): at most n 2^-116 of the largest value, against n^2 2^-106 of the sum of magnitudes
// for the compensated sum, and the total is rounded once.
#pragma once

#include <cstdint>

#ifdef __CUDACC__
#define COS_HD __host__ __device__ __forceinline__
#else
#define COS_HD inline
#endif

namespace cosgpu {

// Exponent fields of the largest value for which the arithmetic below neither meets a
// subnormal, an infinity or NaN nor can overflow; outside (also all zeros) the
// compensated floating-point sum is used.
constexpr int kFixedMin = 200, kFixedMax = 2000;

// Two's complement, least significant word first.
struct Fixed {
    uint32_t w[4];
};

// Low word of (hi:lo) >> r, r in [0, 31].
COS_HD uint32_t funnel_right(uint32_t lo, uint32_t hi, int r) {
#ifdef __CUDA_ARCH__
    return __funnelshift_r(lo, hi, r);
#else
    return (uint32_t)((((uint64_t)hi << 32) | lo) >> r);
#endif
}
COS_HD int leading_zeros(uint32_t x) {
#ifdef __CUDA_ARCH__
    return __clz((int)x);
#else
    return x ? __builtin_clz(x) : 32;
#endif
}

// a += b + (m & 1), m 0 or all ones.
COS_HD void fixed_add(Fixed& a, const Fixed& b, uint32_t m) {
#ifdef __CUDA_ARCH__
    asm("{\n\t.reg .u32 t;\n\tadd.cc.u32 t, %4, %4;\n\taddc.cc.u32 %0, %0, %5;\n\taddc.cc.u32 %1, %1, %6;\n\t"
        "addc.cc.u32 %2, %2, %7;\n\taddc.u32 %3, %3, %8;\n\t}"
        : "+r"(a.w[0]), "+r"(a.w[1]), "+r"(a.w[2]), "+r"(a.w[3])
        : "r"(m), "r"(b.w[0]), "r"(b.w[1]), "r"(b.w[2]), "r"(b.w[3]));
#else
    uint64_t c = m & 1u;
    for (int i = 0; i < 4; ++i) {
        c += (uint64_t)a.w[i] + b.w[i];
        a.w[i] = (uint32_t)c;
        c >>= 32;
    }
#endif
}

// Adds the double (hi:lo); `top` = largest exponent field + extra, extra in {0, 20}: room
// for 2^(10 + extra) values.
COS_HD void fixed_add_double(Fixed& f, uint32_t hi, uint32_t lo, int top) {
    const int e = (int)((hi >> 20) & 0x7ffu), d = top - e;   // (a subnormal is below every kept bit)
    const bool in = e != 0 && d < 128;
    const uint32_t a = in ? (hi & 0xfffffu) | 0x100000u : 0u, b = in ? lo : 0u;
    const int q = (d >> 5) & 3, r = d & 31;
    const uint32_t x2 = a >> r, x1 = funnel_right(b, a, r), x0 = funnel_right(0u, b, r);
    const uint32_t neg = (uint32_t)((int32_t)hi >> 31);
    Fixed y;   // the mantissa's 53 bits at 116 .. 64, d places to the right
    y.w[3] = (q == 0 ? x2 : 0u) ^ neg;
    y.w[2] = (q == 0 ? x1 : q == 1 ? x2 : 0u) ^ neg;
    y.w[1] = (q == 0 ? x0 : q == 1 ? x1 : q == 2 ? x2 : 0u) ^ neg;
    y.w[0] = (q == 1 ? x0 : q == 2 ? x1 : q == 3 ? x2 : 0u) ^ neg;
    fixed_add(f, y, neg);
}

// The value as a double (hi:lo), rounded to nearest even.
COS_HD void fixed_to_double(const Fixed& f, int top, uint32_t& hi, uint32_t& lo) {
    const uint32_t neg = (uint32_t)((int32_t)f.w[3] >> 31);
    Fixed m{{0u, 0u, 0u, 0u}};
    const Fixed x{{f.w[0] ^ neg, f.w[1] ^ neg, f.w[2] ^ neg, f.w[3] ^ neg}};
    fixed_add(m, x, neg);
    const int q = m.w[3] ? 0 : m.w[2] ? 1 : m.w[1] ? 2 : m.w[0] ? 3 : 4;   // leading zero words
    if (q == 4) {
        hi = lo = 0u;
        return;
    }
    const uint32_t y3 = q == 0 ? m.w[3] : q == 1 ? m.w[2] : q == 2 ? m.w[1] : m.w[0];
    const uint32_t y2 = q == 0 ? m.w[2] : q == 1 ? m.w[1] : q == 2 ? m.w[0] : 0u;
    const uint32_t y1 = q == 0 ? m.w[1] : q == 1 ? m.w[0] : 0u;
    const uint32_t y0 = q == 0 ? m.w[0] : 0u;
    const int z = leading_zeros(y3), s = (32 - z) & 31;   // shifted left by z: the leading bit at 127
    const uint32_t z3 = z ? funnel_right(y2, y3, s) : y3, z2 = z ? funnel_right(y1, y2, s) : y2;
    const uint32_t rest = (z ? funnel_right(y0, y1, s) : y1) | y0;   // (y0's shifted bits: zero or not is all that counts)
    const uint32_t mh = z3 >> 11, ml = (z3 << 21) | (z2 >> 11);
    const uint32_t sticky = (z2 & 0x3ffu) | rest;
    const uint32_t up = (z2 >> 10) & 1u & ((sticky ? 1u : 0u) | (ml & 1u));
    const int e = top + 11 - (32 * q + z);
    lo = ml + up;
    hi = (((uint32_t)(e - 1) << 20) + mh + (lo < up ? 1u : 0u)) | (neg & 0x80000000u);
}

}  // namespace cosgpu

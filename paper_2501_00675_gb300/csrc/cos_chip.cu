// On-chip walk: a CTA carries a chunk of samples through the whole evaluation --
// exponentials, propagators, every level, sink -- in shared memory.
//
// The general kernels keep node values and propagators in global memory: every edge and
// sample moves a parent value and a propagator (8 bytes in FP32) from L2 to an SM, and
// the node values of the samples in flight, which exceed L2, move to HBM and back at
// every level.  Here a chunk has only as many samples as the widest level and the
// propagator slots of the graph allow in 227 KB of shared memory (8 float or 4 double
// samples on the medium graph), so neither leaves the SM; global memory serves the
// times, the edge words (4 bytes per edge and chunk, from L2) and one result per sample.
//   level buffer  [row][RB bytes]: node values of the current level, RB bytes per row; the
//                 next level goes to its free end, or, when both do not fit, to
//   TMEM          until every row has read its parents: a second level buffer would halve
//                 RB.  A thread stores and later loads only its own values (tcgen05.st /
//                 ld, its warp's lanes), 256 KB per SM.
//   propagators   [slot][RB bytes] of the chunk
// A lane owns one 16-byte piece (8 or 4 when rows are that narrow) of two destination rows
// and sums their in-edges in CSR order with the arithmetic of the general kernels, so the
// results are bitwise theirs.
//
// What bounds it (ncu, medium graph, FP32, 16,384 samples): the shared-memory pipe, two
// 16-byte reads per edge and lane, 68 % of all cycles busy, a quarter of the load wavefronts
// bank conflicts that the row order of cos_chip.h leaves; issue slots 41 %, DRAM 0.  A chunk of 8 samples
// takes 64,600 cycles, 43,000 of them in its four levels of 4,096 rows, 9,000 in the
// propagators; a small level costs some 900 cycles whatever it holds.  Medium graph, 65,536
// samples, before (general kernels) and after: FP32 2.35 -> 1.62 ms, with A 3.89 -> 2.86,
// count 3.2 -> 1.85.  The FP64 walk is bound by the FP64 pipe on both paths (6.3 / 6.9 ms).
//
// CTAs never wait for one another: a CTA that has no chunk left sums its share of the
// blocks of kReduceBlock samples that are complete, the last CTA the others, and it forms
// the mean.  A block is summed by the whole CTA in 128-bit integers (cos_fixed.h): 2,800
// cycles from the first load to the partial sum, most of them latency, against 15,800 for
// one warp's compensated additions, which the end of every launch waits for.  Tiny graph,
// 1,000 samples, mixed, one launch: 20.5 -> 14.3 us; order 2, 1,000 nodes, 10,007 samples:
// 96 -> 84 us (66 with the exponentials below and two CTAs per SM).
#include <algorithm>
#include <atomic>
#include <cstdio>
#include <type_traits>

#include "cos_chip.cuh"
#include "cos_chip.h"
#include "cos_items.cuh"

namespace cosgpu {
namespace {

// ---------------------------------------------------------------- tensor memory

__device__ __forceinline__ void tmem_alloc(unsigned* smem_dst, unsigned cols) {
    if (cols)
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(smem_dst)), "r"(cols)
                     : "memory");
    // (also by a CTA that allocates nothing: while one holds the permit, no second CTA of the
    // kernel runs on its SM -- order 2, two CTAs per SM: 66 / 105 us)
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void tmem_dealloc(unsigned addr, unsigned cols) {
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(addr), "r"(cols) : "memory");
}

// A lane's pieces of its two rows as 32-bit registers.
template <int LB>
struct alignas(16) Pair {
    unsigned w[LB / 2];
};

template <int LB>
__device__ __forceinline__ void tmem_put(unsigned addr, const Pair<LB>& x) {
    if constexpr (LB == 16)
        asm volatile("tcgen05.st.sync.aligned.32x32b.x8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"r"(addr), "r"(x.w[0]),
                     "r"(x.w[1]), "r"(x.w[2]), "r"(x.w[3]), "r"(x.w[4]), "r"(x.w[5]), "r"(x.w[6]), "r"(x.w[7])
                     : "memory");
    else if constexpr (LB == 8)
        asm volatile("tcgen05.st.sync.aligned.32x32b.x4.b32 [%0], {%1, %2, %3, %4};" ::"r"(addr), "r"(x.w[0]), "r"(x.w[1]),
                     "r"(x.w[2]), "r"(x.w[3])
                     : "memory");
    else
        asm volatile("tcgen05.st.sync.aligned.32x32b.x2.b32 [%0], {%1, %2};" ::"r"(addr), "r"(x.w[0]), "r"(x.w[1])
                     : "memory");
}
// (the values may be used after tmem_wait_ld)
template <int LB>
__device__ __forceinline__ void tmem_get(unsigned addr, Pair<LB>& x) {
    if constexpr (LB == 16)
        asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
                     : "=r"(x.w[0]), "=r"(x.w[1]), "=r"(x.w[2]), "=r"(x.w[3]), "=r"(x.w[4]), "=r"(x.w[5]), "=r"(x.w[6]),
                       "=r"(x.w[7])
                     : "r"(addr)
                     : "memory");
    else if constexpr (LB == 8)
        asm volatile("tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0, %1, %2, %3}, [%4];"
                     : "=r"(x.w[0]), "=r"(x.w[1]), "=r"(x.w[2]), "=r"(x.w[3])
                     : "r"(addr)
                     : "memory");
    else
        asm volatile("tcgen05.ld.sync.aligned.32x32b.x2.b32 {%0, %1}, [%2];" : "=r"(x.w[0]), "=r"(x.w[1]) : "r"(addr) : "memory");
}
// Ties the loaded registers to the wait, so that no use of them moves ahead of it.
template <int LB>
__device__ __forceinline__ void tmem_wait_ld(Pair<LB>& x) {
    if constexpr (LB == 16)
        asm volatile("tcgen05.wait::ld.sync.aligned;"
                     : "+r"(x.w[0]), "+r"(x.w[1]), "+r"(x.w[2]), "+r"(x.w[3]), "+r"(x.w[4]), "+r"(x.w[5]), "+r"(x.w[6]),
                       "+r"(x.w[7])::"memory");
    else if constexpr (LB == 8)
        asm volatile("tcgen05.wait::ld.sync.aligned;" : "+r"(x.w[0]), "+r"(x.w[1]), "+r"(x.w[2]), "+r"(x.w[3])::"memory");
    else
        asm volatile("tcgen05.wait::ld.sync.aligned;" : "+r"(x.w[0]), "+r"(x.w[1])::"memory");
}
__device__ __forceinline__ void tmem_wait_st() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }

// ---------------------------------------------------------------- shared-memory layout

// Scratch of the propagator phase, in the level buffer behind the zero row and the root's
// (256 bytes): one word per pair (i, j) whose bit b says t_i >= t_j for sample b, then
// three arrays [kinds][D][pitch] of 8 bytes.
constexpr int kScratchAt = 256;
__host__ __device__ constexpr int chip_pair_bytes(int D) { return (4 * D * D + 15) / 16 * 16; }
// Values between the rows (kind, time) of a scratch array: two more than the samples, so
// that the rows of neighbouring slots start in different banks (and stay 16-byte aligned).
__host__ __device__ constexpr int chip_pitch(int s) { return s > 1 ? s + 2 : 1; }

// A level before the sink of at most this many rows has a place of its own, so that the
// sink is summed while the next chunk's exponentials are formed in the level buffer.
constexpr int kTailRows = 64;

// Constants of the graph: the mode's 2^{j/64} table (128 values of 8 bytes), then per
// kind coef+ and coef- as doubles, the same as float-float pairs, eps, and one word per
// kind (1: float-float arithmetic applies).
__host__ __device__ constexpr int chip_coef_bytes(int K) { return 1024 + 44 * K; }
struct Consts {
    const double* tab;
    const double* cf;
    const float2* cff;
    const double* eps;
    const int* ff;
    __device__ __forceinline__ Consts(const unsigned char* sm, int off, int K)
        : tab(reinterpret_cast<const double*>(sm + off)), cf(tab + 128), cff(reinterpret_cast<const float2*>(cf + 2 * K)),
          eps(reinterpret_cast<const double*>(cff + 2 * K)), ff(reinterpret_cast<const int*>(eps + K)) {}
};

__host__ __device__ constexpr int round128(int64_t x) { return (int)((x + 127) / 128 * 128); }

struct ChipArgs {
    ChipParams one;
    const ChipParams* list;   // nullptr: `one`, chunks dealt out by CTA number
    unsigned* ticket;
    unsigned long long* exits;   // CTAs that have left
    unsigned long long tag;
    int n, total;
    int tmem_cols;            // 0: no level goes through TMEM
    int few;                  // so few blocks of samples that the last CTA sums them all
};

// ---------------------------------------------------------------- propagators of a chunk

// Once per graph and CTA: constants of every kind, level and group tables, the zero
// propagator row.
template <int MODE>
__device__ __forceinline__ void chip_setup(const ChipParams& p, unsigned char* sm) {
    int4* tab = reinterpret_cast<int4*>(sm + p.tab_off);
    for (int x = threadIdx.x; x < p.g.tables; x += blockDim.x)
        if (x >= p.L) tab[x] = __ldg(p.g.lev + x);
    if (threadIdx.x == 0) {
        // where each level goes: a free part of the level buffer, or through TMEM (sign bit)
        // to its start once every parent is read; the level before the sink to its own place
        const int rb = 1 << p.rb_log2;
        int cur = p.L == 2 ? p.tail_off : 0, before = round128(2 * rb);
        for (int l = 0; l + 1 < p.L; ++l) {
            int4 lv = l ? __ldg(p.g.lev + l) : make_int4(1, 1, 0, 0);
            if (l > 0) {
                const int need = round128((int64_t)(lv.x + 1) * rb);
                const bool tail = l + 2 == p.L && p.tail_off >= 0;
                const bool staged = !tail && before + need > p.lev_bytes;
                cur = tail ? p.tail_off : staged || cur != 0 ? 0 : p.lev_bytes - need;
                before = need;
                lv.w = cur | (staged ? (int)0x80000000 : 0);
            } else {
                lv.w = cur;
            }
            tab[l] = lv;
        }
    }
    if constexpr (!Traits<MODE>::kCount) {
        const int gb = (1 << p.rb_log2) >> (Traits<MODE>::kAbs ? 1 : 0);
        if ((int)threadIdx.x * 4 < gb) reinterpret_cast<unsigned*>(sm + p.g_off + (size_t)p.P * gb)[threadIdx.x] = 0u;
        const Consts c(sm, p.coef_off, p.K);
        const double* tab64 = p.exp_tab + (Traits<MODE>::kBase == COS_MODE_FP32_MIXED ? 128 : 0);
        for (int x = threadIdx.x; x < 128; x += blockDim.x) const_cast<double*>(c.tab)[x] = __ldg(tab64 + x);
        // kinds from the last thread downwards, a thread per prefactor
        for (int x = blockDim.x - 1 - threadIdx.x; x < 2 * p.K; x += blockDim.x) {
            const int k = x < p.K ? x : x - p.K;
            const double e = __ldg(p.eps + k), be = p.beta * e;
            // -1/(1+e^{-beta eps}) (tau >= 0), 1/(1+e^{beta eps}) (tau < 0)
            const double v = (x < p.K ? -1.0 : 1.0) / (1.0 + exp(x < p.K ? -be : be));
            const_cast<double*>(c.cf)[x] = v;
            const_cast<float2*>(c.cff)[x] = split_ff(v);
            if (x >= p.K) continue;
            const_cast<double*>(c.eps)[k] = e;
            const_cast<int*>(c.ff)[k] = fabs(e) * p.beta <= 30.0 ? 1 : 0;
        }
    }
}

// Start the copy of a chunk's times into the times buffer [D][s].
template <int MODE>
__device__ __forceinline__ void chip_times(const ChipParams& p, unsigned char* sm, int chunk) {
    if constexpr (!Traits<MODE>::kCount) {
        double* st = reinterpret_cast<double*>(sm + p.times_off);
        const int sl = p.s_log2, n = p.D << sl;
        const double* t = p.t + ((int64_t)chunk << sl);
        for (int x = threadIdx.x; x < n; x += blockDim.x)
            cp_async_lane<8>(st + x, t + (int64_t)(x >> sl) * p.t_ld + (x & ((1 << sl) - 1)));
        cp_async_commit();
    }
}

// What bounds the propagators is the instructions of the exponentials (some 115 each, one of
// them FP64; 38 % of the issue slots used) and fetching them: the loops have one copy of
// their code, and a graph whose kinds need no double arithmetic never enters its loop.  Order
// 2, 32 kinds, 32 samples a chunk: exponentials 18,000 -> 14,000 cycles, slots 15,700 ->
// 10,900, of 50,000 -> 45,000 (84 -> 72 us for 10,007 samples in this shape; 66 in two CTAs
// per SM).
//
// Exponentials of the kinds [k0, k0 + kn), times and samples of the chunk, with the
// arithmetic of item_props of the general kernels.  Returns whether a time lies so far
// outside [-beta, beta] that float-float arithmetic does not apply (then the caller
// repeats the pass in double).
template <int MODE>
__device__ __forceinline__ bool chip_exps(const ChipParams& p, unsigned char* sm, int k0, int kn, bool in_double) {
    using Tr = Traits<MODE>;
    const int sl = p.s_log2, s = 1 << sl, D = p.D, DS = D << sl, n = kn * DS, pitch = chip_pitch(s), np = kn * D * pitch;
    const double* st = reinterpret_cast<const double*>(sm + p.times_off);
    const Consts c(sm, p.coef_off, p.K);
    double* fa = reinterpret_cast<double*>(sm + kScratchAt + chip_pair_bytes(D));   // [kn][D][pitch]: coef+ e^{-eps t}
    double* fb = fa + np;                                                           // coef- e^{-eps t}
    double* fc = fb + np;                                                           // e^{+eps t}
    const int T = blockDim.x;
    constexpr bool kMixed = Tr::kBase == COS_MODE_FP32_MIXED;
    const FmaConst fma_ = fma_const(p.D);
    bool far = false, rest = true;   // rest: this thread has exponentials to form in double
    if (kMixed && !in_double) {
        rest = false;
        // two independent chains per thread, their arguments (the FP64 part) formed a round
        // ahead; warp 0, which has a sink to sum, comes last
        const int half = (n + 1) / 2;
        struct Item {
            int k, at;
            double arg;
        };
        auto fetch = [&](int x) {
            const unsigned r = (unsigned)x >> sl;
            const int kk = D == 1 ? (int)r : (int)__umulhi(r, p.d_magic);
            return Item{k0 + kk, (int)r * pitch + (x & (s - 1)), c.eps[k0 + kk] * st[x - kk * DS]};
        };
        auto second = [&](int x) { return x + half < n ? x + half : x; };
        int x = T - 1 - (int)threadIdx.x;
        Item next[2];
        if (x < half) {
            next[0] = fetch(x);
            next[1] = fetch(second(x));
        }
        for (; x < half; x += T) {
            const Item it[2] = {next[0], next[1]};
            if (x + T < half) {
                next[0] = fetch(x + T);
                next[1] = fetch(second(x + T));
            }
#pragma unroll
            for (int u = 0; u < 2; ++u) {
                const bool ok = within_30(it[u].arg);
                float2 em, ep;
                exp_pair_ff(ok ? it[u].arg : 0.0, reinterpret_cast<const float2*>(c.tab), em, ep);
                if (!c.ff[it[u].k]) {
                    rest = true;
                    continue;
                }
                if (!ok) far = true;
                reinterpret_cast<float2*>(fa)[it[u].at] = mul_ff2(c.cff[it[u].k], em);
                reinterpret_cast<float2*>(fb)[it[u].at] = mul_ff2(c.cff[p.K + it[u].k], em);
                reinterpret_cast<float2*>(fc)[it[u].at] = ep;
            }
        }
    }
    if (!rest) return far;
    // (the same exponentials as above, one after another)
    const int half = kMixed ? (n + 1) / 2 : n;
    for (int x0 = T - 1 - (int)threadIdx.x; x0 < half; x0 += T)
#pragma unroll 1
        for (int x = x0; x < n; x += half) {
            const unsigned r = (unsigned)x >> sl;
            const int kk = D == 1 ? (int)r : (int)__umulhi(r, p.d_magic), k = k0 + kk;
            if (kMixed && !in_double && c.ff[k]) continue;
            const double arg = fma_.mul(c.eps[k], st[x - kk * DS]);
            double em, ep;
            if constexpr (kMixed) exp_pair(arg, p.exp_tab, fma_, em, ep);   // (rare: the table at hand is the other)
            else exp_pair_at(arg, c.tab, fma_, em, ep);
            const int at = (int)r * pitch + (x & (s - 1));
            fa[at] = fma_.mul(c.cf[k], em);
            fb[at] = fma_.mul(c.cf[p.K + k], em);
            fc[at] = ep;
        }
    return far;
}

// Bit b of pair (i, j): t_i >= t_j of the chunk's sample b.
__device__ __forceinline__ void chip_pairs(const ChipParams& p, unsigned char* sm) {
    const int sl = p.s_log2, s = 1 << sl, D = p.D, n = (D * D) << sl, lane = threadIdx.x & 31;
    const double* st = reinterpret_cast<const double*>(sm + p.times_off);
    unsigned* pair = reinterpret_cast<unsigned*>(sm + kScratchAt);
    for (int x0 = ((int)threadIdx.x & ~31); x0 < n; x0 += blockDim.x) {
        const int x = min(x0 + lane, n - 1), q = x >> sl, b = x & (s - 1);
        const int i = D == 1 ? q : (int)__umulhi((unsigned)q, p.d_magic), j = q - i * D;
        const bool ge = key_ge(time_order_key(st[(i << sl) + b]), time_order_key(st[(j << sl) + b]));
        const unsigned bits = __ballot_sync(0xffffffffu, ge);
        if (x0 + lane < n && b == 0) pair[q] = s == 32 ? bits : (bits >> lane) & ((1u << s) - 1u);
    }
}

// This thread's slots of the kinds [k0, k0 + kn): pieces x, x + T, ... below `end`, the
// next kAhead descriptors loaded (the first ahead of the exponentials).
constexpr int kAhead = 2;
struct SlotRange {
    int x, end;
    uint2 sd[kAhead];
    __device__ __forceinline__ void open(const ChipParams& p, int k0, int kn, int pl) {
        const bool all = kn == p.K;
        x = (all ? 0 : __ldg(p.kind_slot + k0) << pl) + (int)threadIdx.x;
        end = (all ? p.P : __ldg(p.kind_slot + k0 + kn)) << pl;
#pragma unroll
        for (int u = 0; u < kAhead; ++u)
            if (x + u * (int)blockDim.x < end) sd[u] = __ldg(p.g.slots + ((x + u * (int)blockDim.x) >> pl));
    }
};

// V doubles from shared memory, two per access, the second two `half` further.
template <int V>
__device__ __forceinline__ VecT<double, V> load_pair(const double* x, int half) {
    VecT<double, V> r;
    if constexpr (V == 1) {
        r.v[0] = x[0];
    } else {
#pragma unroll
        for (int v = 0; v < V; v += 2) {
            const double2 d = *reinterpret_cast<const double2*>(x + (v ? half : 0));
            r.v[v] = d.x;
            r.v[v + 1] = d.y;
        }
    }
    return r;
}
// A scratch value that holds a float-float pair.
__device__ __forceinline__ float2 as_ff(double x) {
    return make_float2(__int_as_float(__double2loint(x)), __int_as_float(__double2hiint(x)));
}

// Propagators of the slots of kinds [k0, k0 + kn); a thread forms V samples of a slot.
template <int MODE, int V>
__device__ __forceinline__ void chip_slots(const ChipParams& p, unsigned char* sm, int k0, int kn, bool in_double, SlotRange& r) {
    using Tr = Traits<MODE>;
    using Prop = typename Tr::Prop;
    constexpr bool kMixed = Tr::kBase == COS_MODE_FP32_MIXED;
    constexpr int VL = V == 4 ? 2 : V == 2 ? 1 : 0;
    const int sl = p.s_log2, D = p.D, pitch = chip_pitch(1 << sl), np = kn * D * pitch;
    const int pl = sl - VL, T = blockDim.x;   // pl: log2 pieces per slot
    const FmaConst fma_ = fma_const(p.D);
    const Consts c(sm, p.coef_off, p.K);
    const unsigned* pair = reinterpret_cast<const unsigned*>(sm + kScratchAt);
    const double* fa = reinterpret_cast<const double*>(sm + kScratchAt + chip_pair_bytes(D));
    const double* fb = fa + np;
    const double* fc = fb + np;
    Prop* G = reinterpret_cast<Prop*>(sm + p.g_off);
    const int ahi = p.abs_weights ? 0x7fffffff : -1;
    // a thread's samples: V = 4 takes two at smp and two half a row on, so that the threads
    // of a row read 16 neighbouring bytes each (four in a row: two of eight threads in the
    // same banks)
    const int part = (int)threadIdx.x & ((1 << pl) - 1), smp = V == 4 ? part << 1 : part << VL, half = V == 4 ? 1 << (sl - 1) : 0;
    fa += smp - k0 * D * pitch;
    fb += smp - k0 * D * pitch;
    fc += smp - k0 * D * pitch;
    while (r.x < r.end) {   // (one copy of the code: unrolled, the warps wait for instructions)
        const int x = r.x;
        const uint2 d = r.sd[0];
#pragma unroll
        for (int u = 0; u + 1 < kAhead; ++u) r.sd[u] = r.sd[u + 1];
        if (x + kAhead * T < r.end) r.sd[kAhead - 1] = __ldg(p.g.slots + ((x + kAhead * T) >> pl));
        r.x += T;
        unsigned ge = pair[d.y & 0xffffu] >> smp;   // tau = t_i - t_j >= 0 ?
        if constexpr (V == 4) ge = (ge & 3u) | (ge >> half & 3u) << 2;
        const int shi = (int)(d.y & 0x80000000u);
        const int xi = (int)(d.x & 0xffffu) * pitch, xj = (int)(d.x >> 16) * pitch;
        // V values of 8 bytes, aligned to 16 when there are more than one; neighbouring slots
        // share (kind, i), so fetching both prefactors' rows costs few wavefronts
        const VecT<double, V> vp = load_pair<V>(fa + xi, half), vn = load_pair<V>(fb + xi, half), ve = load_pair<V>(fc + xj, half);
        VecT<Prop, V> out;
        if (kMixed && !in_double && c.ff[(d.y >> 16) & 0x7fff]) {
#pragma unroll
            for (int v = 0; v < V; ++v) {
                const float g = mul_ff(as_ff((ge >> v) & 1u ? vp.v[v] : vn.v[v]), as_ff(ve.v[v]));
                out.v[v] = (Prop)__uint_as_float((__float_as_uint(g) ^ (unsigned)shi) & (unsigned)ahi);
            }
        } else {
#pragma unroll
            for (int v = 0; v < V; ++v)
                out.v[v] = (Prop)sign_ops(fma_.mul((ge >> v) & 1u ? vp.v[v] : vn.v[v], ve.v[v]), shi, ahi);
        }
        Prop* g = G + (((size_t)x - part) << VL) + smp;
        if constexpr (V == 4) {
            *reinterpret_cast<VecT<Prop, 2>*>(g) = VecT<Prop, 2>{{out.v[0], out.v[1]}};
            *reinterpret_cast<VecT<Prop, 2>*>(g + half) = VecT<Prop, 2>{{out.v[2], out.v[3]}};
        } else {
            *reinterpret_cast<VecT<Prop, V>*>(g) = out;
        }
    }
}

// As chip_slots for user-tabulated propagators (see item_props).
template <int MODE>
__device__ __forceinline__ void chip_slots_table(const ChipParams& p, unsigned char* sm) {
    using Prop = typename Traits<MODE>::Prop;
    const int sl = p.s_log2, D = p.D, PT = p.ptab_T, n = p.P << sl, T = blockDim.x;
    const FmaConst fc = fma_const(p.D);
    const double* st = reinterpret_cast<const double*>(sm + p.times_off);
    Prop* G = reinterpret_cast<Prop*>(sm + p.g_off);
    const int ahi = p.abs_weights ? 0x7fffffff : -1;
    int x = threadIdx.x;
    uint2 sd = x < n ? __ldg(p.g.slots + (x >> sl)) : make_uint2(0, 0);
    while (x < n) {
        uint2 next = sd;
        if (x + T < n) next = __ldg(p.g.slots + ((x + T) >> sl));
        const int smp = x & ((1 << sl) - 1);
        const int k = (sd.y >> 16) & 0x7fff, i = (int)(sd.x & 0xffffu) - k * D, j = (int)(sd.x >> 16) - k * D;
        const int shi = (int)(sd.y & 0x80000000u);
        const double2* tk = reinterpret_cast<const double2*>(p.ptab) + (int64_t)k * 2 * PT;
        G[x] = (Prop)sign_ops(table_value(st[(i << sl) + smp], st[(j << sl) + smp], tk, PT, p.ptab_inv_h, fc), shi, ahi);
        x += T;
        sd = next;
    }
}

// ---------------------------------------------------------------- rows

// This lane's words (two rows) of a block with n words per row left (see cos_chip.h).
struct Words {
    uint4 a, b;
};
__device__ __forceinline__ void load_words(Words& m, const uint32_t* block, unsigned n, int r32) {
    if (n == 1) {
        const uint2 q = __ldg(reinterpret_cast<const uint2*>(block) + r32);
        m.a.x = q.x;
        m.a.y = q.y;
    } else {
        m.a = __ldg(reinterpret_cast<const uint4*>(block) + r32);
        if (n > 2) m.b = __ldg(reinterpret_cast<const uint4*>(block) + 32 + r32);
    }
}

// A lane's pieces of two destination rows: the in-edges in order, one multiply-add each.
// par and pro: byte offsets in shared memory of this lane's piece of place 0 and slot 0.
template <int MODE, int LB>
struct RowSum {
    using Tr = Traits<MODE>;
    using Val = typename Tr::Val;
    using Prop = typename Tr::Prop;
    static constexpr int V = LB / (int)sizeof(Val);
    using VecV = VecT<Val, V>;
    using VecG = VecT<Prop, V>;

    int par, pro;
    int rb, gb;                       // row bytes of a node and of a slot
    bool use_abs;                     // this lane sums A (|G|)
    VecV acc[2];

    __device__ __forceinline__ VecV parent(const unsigned char* sm, unsigned m) const {
        return *reinterpret_cast<const VecV*>(sm + ((int)(m & 0xffffu) * rb + par));
    }
    __device__ __forceinline__ VecG factor(const unsigned char* sm, unsigned m) const {
        if constexpr (Tr::kCount) return VecG{};
        else return *reinterpret_cast<const VecG*>(sm + ((int)(m >> 16) * gb + pro));
    }
    __device__ __forceinline__ void add(VecV& s, const VecV& a, const VecG& g) {
#pragma unroll
        for (int v = 0; v < V; ++v) {
            if constexpr (Tr::kCount) s.v[v] += a.v[v];
            else if constexpr (Tr::kAbs) s.v[v] = fmaf(a.v[v], use_abs ? abs_to_float(g.v[v]) : g.v[v], s.v[v]);
            else s.v[v] = madd(a.v[v], g.v[v], s.v[v]);
        }
    }
    // the next N in-edges of both rows, their loads ahead of the multiply-adds
    template <int N>
    __device__ __forceinline__ void steps(const unsigned char* sm, const unsigned (&w0)[N], const unsigned (&w1)[N]) {
        VecV a0[N], a1[N];
        VecG g0[N], g1[N];
#pragma unroll
        for (int e = 0; e < N; ++e) {
            a0[e] = parent(sm, w0[e]);
            g0[e] = factor(sm, w0[e]);
            a1[e] = parent(sm, w1[e]);
            g1[e] = factor(sm, w1[e]);
        }
#pragma unroll
        for (int e = 0; e < N; ++e) {
            add(acc[0], a0[e], g0[e]);
            add(acc[1], a1[e], g1[e]);
        }
    }
    __device__ __forceinline__ void block(const unsigned char* sm, const Words& m, unsigned n) {
        const uint4 &a = m.a, &b = m.b;
        if (n == 1) {
            const unsigned w0[1] = {a.x}, w1[1] = {a.y};
            steps<1>(sm, w0, w1);
        } else if (n == 2) {
            const unsigned w0[2] = {a.x, a.y}, w1[2] = {a.z, a.w};
            steps<2>(sm, w0, w1);
        } else if (n == 3) {
            const unsigned w0[3] = {a.x, a.y, a.z}, w1[3] = {b.x, b.y, b.z};
            steps<3>(sm, w0, w1);
        } else {
            const unsigned w0[2] = {a.x, a.y}, w1[2] = {b.x, b.y};
            steps<2>(sm, w0, w1);
            const unsigned w2[2] = {a.z, a.w}, w3[2] = {b.z, b.w};
            steps<2>(sm, w2, w3);
        }
    }
    // n in-edges whose first words are m and whose first block is b
    __device__ __forceinline__ void rows(const unsigned char* sm, const Words& m, unsigned n, const uint32_t* b, int r32) {
#pragma unroll
        for (int v = 0; v < V; ++v) acc[0].v[v] = acc[1].v[v] = (Val)0;
        block(sm, m, n);
        while (n > 4) {
            n -= 4;
            b += 4 * kChipGroup;
            Words q;
            load_words(q, b, n, r32);
            block(sm, q, n);
        }
    }
};

// ---------------------------------------------------------------- sample reduction

// For values outside the integers' range.
template <typename T>
__device__ __noinline__ double block_sum_compensated(const T* x, int64_t S, int64_t b, int lane) {
    constexpr int per_lane = kReduceBlock / 32;
    constexpr int AHEAD = 8;
    const int64_t s0 = b * kReduceBlock + lane;
    double sum = 0.0, comp = 0.0;
#pragma unroll 1
    for (int u0 = 0; u0 < per_lane; u0 += AHEAD) {
        double v[AHEAD];
#pragma unroll
        for (int u = 0; u < AHEAD; ++u) {
            const int64_t s = s0 + (int64_t)(u0 + u) * 32;
            v[u] = s < S ? load_value(x + s) : 0.0;
        }
#pragma unroll
        for (int u = 0; u < AHEAD; ++u) neumaier_add(sum, comp, v[u]);
    }
    warp_sum(sum, comp);
    return sum + comp;
}

// Sums of blocks of kReduceBlock samples by the whole CTA, its threads sharing a block's
// values; same result as block_sum of the general kernels.
static_assert(kScratchAt <= 320, "the level buffer has room for either");
struct CtaSum {
    unsigned mx[16];
    Fixed f[16];
};
constexpr int kPerThread = 8;   // values of a thread, 128 threads

template <typename T>
__device__ __forceinline__ void cta_load(double (&v)[kPerThread], const T* x, int64_t S, int64_t b) {
    const int64_t s0 = b * kReduceBlock + threadIdx.x;
#pragma unroll
    for (int u = 0; u < kPerThread; ++u) {
        const int at = u * (int)blockDim.x;
        v[u] = at < kReduceBlock && s0 + at < S ? load_value(x + s0 + at) : 0.0;
    }
}
// (two barriers; the partial sum is written by thread 0)
template <typename T>
__device__ __forceinline__ void cta_sum(double (&v)[kPerThread], const T* x, double* partials, int64_t S, int64_t b,
                                        CtaSum& c) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5, T_ = blockDim.x;
    unsigned mx = 0;
#pragma unroll
    for (int u = 0; u < kPerThread; ++u) mx = max(mx, magnitude_word(v[u]));
    mx = __reduce_max_sync(0xffffffffu, mx);
    if (lane == 0) c.mx[warp] = mx;
    __syncthreads();
    const int emax = warp_exponent(lane < nw ? c.mx[lane] : 0u);
    if (!fixed_in_range(emax)) {
        if (warp == 0) {
            const double sum = block_sum_compensated(x, S, b, lane);
            if (lane == 0) partials[b] = sum;
        }
        __syncthreads();
        return;
    }
    Fixed f{{0u, 0u, 0u, 0u}};
#pragma unroll 1
    for (int u = 0; u * T_ < kReduceBlock; ++u) {   // (one copy of the code: it runs cold)
        fixed_add_value(f, v[0], emax);
#pragma unroll
        for (int h = 0; h + 1 < kPerThread; ++h) v[h] = v[h + 1];
    }
    f = warp_fixed_sum(f);
    if (lane == 0) c.f[warp] = f;
    __syncthreads();
    if (warp == 0) {
        f = lane < nw ? c.f[lane] : Fixed{{0u, 0u, 0u, 0u}};
        const double sum = fixed_value(warp_fixed_sum(f), emax);
        if (lane == 0) partials[b] = sum;
    }
}
constexpr unsigned kBlockSummed = 0xffffffffu;   // arrival word of a block whose partial sum is written

// The first block from q on whose arrival word is not kBlockSummed; 32 words at a time, read by
// one warp for all -- the callers' loop has block barriers, and a launch that overlaps on the
// same words changes them.  (Out of line: short launches sum every block, and fetch the code
// behind it cold.)
__device__ __noinline__ int next_open(const unsigned* arrive, int q, int nblk, bool first) {
    __shared__ unsigned s_open;
    __shared__ int s_base;
    int base = first ? -1 : s_base;
    unsigned open = first ? 0u : s_open;
    while (q < nblk) {
        if ((q & ~31) != base) {
            base = q & ~31;
            const int at = base + (int)(threadIdx.x & 31);
            __syncthreads();   // everyone has the words before
            if (threadIdx.x < 32) {
                const unsigned left = __ballot_sync(0xffffffffu, at < nblk && __ldcg(arrive + at) != kBlockSummed);
                if (threadIdx.x == 0) {
                    s_open = left;
                    s_base = base;
                }
            }
            __syncthreads();
            open = s_open;
        }
        const unsigned left = open >> (q - base);
        if (left) return q + __ffs((int)left) - 1;
        q = base + 32;
    }
    return nblk;
}

// Partial sums of blocks [b, nblk) whose arrival word is not kBlockSummed (arrive
// nullptr: of all).
template <typename T>
__device__ __forceinline__ void cta_sums(const T* x, double* partials, int64_t S, int b, int nblk, const unsigned* arrive, CtaSum& c) {
    if (arrive) b = next_open(arrive, b, nblk, true);
    double v[kPerThread], next[kPerThread];
    if (b < nblk) cta_load(v, x, S, b);
    while (b < nblk) {
        const int n = arrive ? next_open(arrive, b + 1, nblk, false) : b + 1;
        if (n < nblk) cta_load(next, x, S, n);   // a block ahead
        cta_sum(v, x, partials, S, b, c);
#pragma unroll
        for (int u = 0; u < kPerThread; ++u) v[u] = next[u];
        b = n;
    }
}
template <int MODE>
__device__ __noinline__ void chip_sums(const ChipParams& p, unsigned char* sm, int b, int nblk, const unsigned* arrive) {
    CtaSum& c = *reinterpret_cast<CtaSum*>(sm);   // (the level buffer, free by now)
    if constexpr (Traits<MODE>::kCount) cta_sums(static_cast<const long long*>(p.R), p.partials, p.S, b, nblk, arrive, c);
    else cta_sums(static_cast<const double*>(p.R), p.partials, p.S, b, nblk, arrive, c);
    if constexpr (Traits<MODE>::kAbs) cta_sums(p.Rabs, p.partials_abs, p.S, b, nblk, arrive, c);
}


__device__ __forceinline__ unsigned long long ld_relaxed_gpu(const unsigned long long* p) {
    unsigned long long v;
    asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ unsigned long long tagged(unsigned long long tag, unsigned n) { return tag << kTagShift | n; }

// Count a chunk's results in (one thread, after the writes and, unless it is one of theirs, a
// block barrier).
__device__ __forceinline__ void chip_arrive(const ChipParams& p, int chunk) {
    const int64_t s0 = (int64_t)chunk << p.s_log2;
    const unsigned mine = (unsigned)min((int64_t)1 << p.s_log2, p.S - s0);
    asm volatile("red.release.gpu.global.add.u32 [%0], %1;" ::"l"(p.arrive + s0 / kReduceBlock), "r"(mine) : "memory");
}

__device__ __forceinline__ int chip_blocks(const ChipParams& p) { return (int)((p.S + kReduceBlock - 1) / kReduceBlock); }

// A CTA that has no chunk left sums its share of the evaluation's blocks, as far as
// they are complete; `first`: number of this evaluation's block 0 in the launch.
template <int MODE>
__device__ __forceinline__ void chip_sum_own(const ChipParams& p, unsigned char* sm, int first, const unsigned long long* exits,
                                             unsigned long long tag) {
    __shared__ int s_full;
    const int nblk = chip_blocks(p), grid = gridDim.x;
    for (int b = (int)((blockIdx.x + grid - first % grid) % grid); b < nblk; b += grid) {
        if (threadIdx.x == 0) {   // (two loads in flight together)
            const unsigned long long e = tag ? ld_relaxed_gpu(exits) : 0;
            const unsigned n = ld_acquire_gpu_u32(p.arrive + b);
            s_full = e >> kTagShift == tag && !(e & kExitsUntrusted) &&
                     n == (unsigned)min((int64_t)kReduceBlock, p.S - (int64_t)b * kReduceBlock);
        }
        __syncthreads();
        const bool full = s_full != 0;
        __syncthreads();
        if (!full) continue;
        chip_sums<MODE>(p, sm, b, b + 1, nullptr);
        if (threadIdx.x == 0) p.arrive[b] = kBlockSummed;   // (read by the last CTA, after this one's release)
    }
}

// The last CTA of the launch: the blocks nobody has summed (`all`: every block), then the
// means.
template <int MODE>
__device__ __forceinline__ void chip_sum_rest(const ChipParams& p, unsigned char* sm, bool all) {
    chip_sums<MODE>(p, sm, 0, chip_blocks(p), all ? nullptr : p.arrive);
}
template <int MODE>
__device__ __noinline__ void chip_mean(const ChipParams& p, int lane) {
    const int64_t nblk = (p.S + kReduceBlock - 1) / kReduceBlock;
    double sum, comp, sa = 0.0, ca = 0.0;
    partials_sum(p.partials, nblk, lane, sum, comp);
    if constexpr (Traits<MODE>::kAbs) partials_sum(p.partials_abs, nblk, lane, sa, ca);
    if (lane == 0) {
        const double mean = (sum + comp) / (double)p.S, mean_abs = Traits<MODE>::kAbs ? (sa + ca) / (double)p.S : 0.0;
        p.ctrl->sum = sum;
        p.ctrl->comp = comp;
        p.ctrl->mean = mean;
        p.ctrl->mean_abs = mean_abs;
        if (p.clear_err) {
            p.ctrl->err = 0;
            p.ctrl->err_detail = 0;
        }
        if (p.mean_out) {
            p.mean_out[0] = mean;
            if constexpr (Traits<MODE>::kAbs) p.mean_out[1] = mean_abs;
        }
    }
}

// ---------------------------------------------------------------- kernel

// A float as a double, by 32-bit integer instructions but for subnormals, infinities and
// NaN (a conversion takes as long as an FP64 operation, and the sink's in-edges are a
// serial chain).
__device__ __forceinline__ double widen(float f) {
    const unsigned u = __float_as_uint(f), e = (u >> 23) & 0xffu;
    if (e - 1u >= 254u && (u << 1) != 0) return (double)f;
    const unsigned hi = (u & 0x80000000u) | (e ? ((u & 0x7fffffffu) >> 3) + (896u << 20) : 0u);
    return __hiloint2double((int)hi, (int)(e ? u << 29 : 0u));
}

// Sink of chunk `chunk` by one warp: one lane per sample, in-edges in order; parents at
// byte `base` of shared memory.
template <int MODE>
__device__ __forceinline__ void chip_sink(const ChipParams& p, unsigned char* sm, int base, int chunk, unsigned word) {
    using Tr = Traits<MODE>;
    using Val = typename Tr::Val;
    using Prop = typename Tr::Prop;
    using Out = typename Tr::SinkAcc;
    const int lane = threadIdx.x & 31, s = 1 << p.s_log2, smp = lane & (s - 1);
    const int rb = 1 << p.rb_log2, gb = Tr::kAbs ? rb / 2 : rb;
    const unsigned char* G = sm + p.g_off;
    Out acc = (Out)0, acca = (Out)0;
    for (int e = 0; e < p.g.nsink; ++e) {
        const unsigned m = e < 32 ? __shfl_sync(0xffffffffu, word, e) : __ldg(p.g.sink + e);
        const Val* pr = reinterpret_cast<const Val*>(sm + base + (int)(m & 0xffffu) * rb);
        if constexpr (Tr::kCount) {
            acc += pr[smp];
        } else {
            const Prop g = reinterpret_cast<const Prop*>(G + (int)(m >> 16) * gb)[smp];
            if constexpr (Tr::kBase == COS_MODE_FP32_MIXED) {
                const double gd = widen(g);
                acc = fma(widen(pr[smp]), gd, acc);   // exact product
                if constexpr (Tr::kAbs) acca = fma(widen(pr[s + smp]), sign_ops(gd, 0, 0x7fffffff), acca);
            } else {
                acc = madd(pr[smp], g, acc);
            }
        }
    }
    const int64_t at = ((int64_t)chunk << p.s_log2) + lane;
    if (lane < s && at < p.S) {
        static_cast<Out*>(p.R)[at] = acc;
        if constexpr (Tr::kAbs) p.Rabs[at] = acca;
    }
}

// State of a CTA between chunks.
struct ChipState {
    int pending;        // chunk whose sink has not been summed (-1: none); its tail level is in place
    int written;        // chunk whose results are written but not counted in
    unsigned word;      // this lane's sink word
    bool counts;        // results are counted in block by block
};

// One chunk of samples: propagators (and the previous chunk's sink), then every level.
// The chunk's times are in the times buffer; those of chunk `next` (< 0: none) follow.
// `next_of` is called after a block barrier.
template <int MODE, int LB, class Next>
__device__ __forceinline__ void chip_chunk(const ChipParams& p, int chunk, unsigned char* sm, unsigned tmem, ChipState& cs,
                                           const Next& next_of) {
    using Tr = Traits<MODE>;
    using Val = typename Tr::Val;
    using RS = RowSum<MODE, LB>;
    constexpr int V = RS::V;
    constexpr bool kMixed = Tr::kBase == COS_MODE_FP32_MIXED;
    const int tid = threadIdx.x, T = blockDim.x, lane = tid & 31, warp = __shfl_sync(0xffffffffu, tid >> 5, 0);
    const int RB = 1 << p.rb_log2;
    // the previous chunk's sink beside the exponentials
    if (warp == 0 && cs.pending >= 0) {
        chip_sink<MODE>(p, sm, p.tail_off, cs.pending, cs.word);
    }
    if (cs.pending >= 0) cs.written = cs.pending;
    int cur = p.L == 2 ? p.tail_off : 0;   // where the current level is
    if (tid * 4 < RB) reinterpret_cast<unsigned*>(sm + cur)[tid] = 0u;                        // the zero row
    if (tid * (int)sizeof(Val) < RB) reinterpret_cast<Val*>(sm + cur + RB)[tid] = (Val)1;     // the root holds 1
    if constexpr (Tr::kCount) {
        __syncthreads();
    } else if (p.ptab) {
        __syncthreads();   // the previous sink has read its propagators
        chip_slots_table<MODE>(p, sm);
        __syncthreads();
    } else {
        for (int k0 = 0; k0 < p.K; k0 += p.kinds_per_pass) {
            const int kn = min(p.kinds_per_pass, p.K - k0);
            SlotRange range;
            range.open(p, k0, kn, p.s_log2 - (V == 4 ? 2 : V == 2 ? 1 : 0));
            bool far = !kMixed;
            for (;;) {   // again in double, where a time lies too far outside [-beta, beta]
                const bool again = chip_exps<MODE>(p, sm, k0, kn, far);
                if (k0 == 0 && far == !kMixed) chip_pairs(p, sm);
                if (!__syncthreads_or(again)) break;
                far = true;
            }
            chip_slots<MODE, V>(p, sm, k0, kn, far, range);
            __syncthreads();   // the propagators are complete, the scratch is free
        }
    }
    const int next = next_of();
    if (next >= 0) chip_times<MODE>(p, sm, next);

    const int lsh = p.rb_log2 - (LB == 16 ? 4 : LB == 8 ? 3 : 2);   // log2 lanes per row
    const int lanes = 1 << lsh, piece = lane & (lanes - 1);
    const int r32 = ((warp & (lanes - 1)) << (5 - lsh)) + (lane >> lsh);   // rows r32, r32 + 32 of a group
    const int g0 = warp >> lsh, gstep = T >> (5 + lsh);
    RS rs;
    rs.rb = RB;
    rs.gb = Tr::kAbs ? RB / 2 : RB;
    rs.pro = p.g_off + (Tr::kAbs ? piece & (lanes / 2 - 1) : piece) * LB;
    rs.use_abs = Tr::kAbs && piece >= lanes / 2;
    const int mine = RB + r32 * RB + piece * LB;   // this lane's first piece in a level's rows
    const int4* levt = reinterpret_cast<const int4*>(sm + p.tab_off);
    const unsigned* grp = reinterpret_cast<const unsigned*>(levt + p.L);
    const uint32_t* words = p.g.words;
    int4 lv = make_int4(0, 0, 0, 0);   // width, groups, first group, place | staged
    unsigned d = 0;                    // descriptor of this warp's next group, and this lane's words
    Words m{};
    auto open = [&](int l) {
        lv = levt[l];
        if (g0 >= lv.y) return;
        d = __shfl_sync(0xffffffffu, grp[lv.z + g0], 0);
        load_words(m, words + (d >> 11 << 6), d & 0x7ffu, r32);
    };
    if (p.L > 2) open(1);
    // In count mode, where no propagators lie between, the release waits for the sink's writes,
    // and not in warp 0, which has had the sink to sum: by it medium count took 1.8 % longer.
    // Elsewhere the last warp, which has formed the most exponentials, would be the wrong one
    // (14 levels of 8 rows, FP32, 1.5 % longer).
    if (cs.counts && tid == (Tr::kCount ? T - 32 : 0) && cs.written >= 0) chip_arrive(p, cs.written);
    cs.written = -1;
    for (int l = 1; l + 1 < p.L; ++l) {
        const int W = lv.x, groups = lv.y, dst = lv.w & 0x7fffffff;
        const bool staged = lv.w < 0;
        const unsigned* gd = grp + lv.z;
        rs.par = cur + piece * LB;
        unsigned col = tmem;
        for (int g = g0; g < groups; g += gstep) {
            const unsigned dc = d;
            const Words mc = m;
            if (g + gstep < groups) {   // the next group's words, a round ahead
                d = __shfl_sync(0xffffffffu, gd[g + gstep], 0);   // (uniform, known to be)
                load_words(m, words + (d >> 11 << 6), d & 0x7ffu, r32);
            }
            rs.rows(sm, mc, dc & 0x7ffu, words + (dc >> 11 << 6), r32);
            if (staged) {
                Pair<LB> x;
                memcpy(&x, &rs.acc, 2 * LB);
                __syncwarp();
                tmem_put<LB>(col, x);
                col += LB / 2;
            } else {
                const int row = g * kChipGroup + r32, at = dst + g * (kChipGroup * RB) + mine;
                if (row < W) *reinterpret_cast<typename RS::VecV*>(sm + at) = rs.acc[0];
                if (row + 32 < W) *reinterpret_cast<typename RS::VecV*>(sm + (at + 32 * RB)) = rs.acc[1];
            }
        }
        const int first = g0 * kChipGroup + r32, step = gstep * kChipGroup;
        if (l + 2 < p.L) open(l + 1);   // ahead of the barriers
        else cp_async_wait<0>();        // the next chunk's times
        if (staged) {
            tmem_wait_st();
            __syncthreads();   // every row has read its parents
            constexpr int U = 2;   // rounds per wait (a warp's 128 columns hold a multiple)
            unsigned from = tmem;
            const int warp_first = g0 * kChipGroup;
            for (int row = first, wrow = warp_first; wrow < W; row += U * step, wrow += U * step) {
                Pair<LB> x[U];
                __syncwarp();
#pragma unroll
                for (int u = 0; u < U; ++u) tmem_get<LB>(from + (unsigned)u * (LB / 2), x[u]);
                from += U * (LB / 2);
#pragma unroll
                for (int u = 0; u < U; ++u) tmem_wait_ld<LB>(x[u]);
                const int at = dst + RB + row * RB + piece * LB;
#pragma unroll
                for (int u = 0; u < U; ++u) {
                    typename RS::VecV v[2];
                    memcpy(&v, &x[u], 2 * LB);
                    if (row + u * step < W) *reinterpret_cast<typename RS::VecV*>(sm + (at + u * step * RB)) = v[0];
                    if (row + u * step + 32 < W) *reinterpret_cast<typename RS::VecV*>(sm + (at + (u * step + 32) * RB)) = v[1];
                }
            }
        }
        if (tid * 4 < RB) reinterpret_cast<unsigned*>(sm + dst)[tid] = 0u;   // its zero row
        __syncthreads();
        cur = dst;
    }
    if (p.L == 2) {
        cp_async_wait<0>();
        __syncthreads();
    }
    if (p.tail_off >= 0) {
        cs.pending = chunk;   // its sink is summed beside the next chunk's exponentials
    } else {
        if (warp == 0) {
            chip_sink<MODE>(p, sm, cur, chunk, cs.word);
        }
        cs.written = chunk;
        __syncthreads();
    }
}

// After the last chunk of a graph: its sink, and the results counted in.
template <int MODE>
__device__ __forceinline__ void chip_finish(const ChipParams& p, unsigned char* sm, ChipState& cs) {
    if ((threadIdx.x >> 5) == 0) {
        if (cs.counts && cs.written >= 0 && threadIdx.x == 0) chip_arrive(p, cs.written);
        if (cs.pending >= 0) {
            chip_sink<MODE>(p, sm, p.tail_off, cs.pending, cs.word);
            __syncwarp();
            if (cs.counts && threadIdx.x == 0) chip_arrive(p, cs.pending);
        }
    }
    cs.pending = cs.written = -1;
    __syncthreads();
}

// The exit word does not belong to this launch when one of its CTAs leaves: those that claim it
// have not started yet.  Takes it over, or counts on what another CTA made of it.  (Out of
// line: the last CTA fetches the code behind it cold.)
__device__ __noinline__ unsigned long long chip_exit_early(unsigned long long* exits, unsigned long long tag) {
    unsigned long long before = 0;
    __threadfence();
    for (int q = 0; q < (1 << 20); ++q) {   // (a try fails when another CTA's succeeds)
        const unsigned long long now = ld_relaxed_gpu(exits);
        if (now >> kTagShift == tag) {
            before = atomicAdd(exits, 1ull);
            break;
        }
        if (atomicCAS(exits, now, tagged(tag, kExitsUntrusted | 1u)) == now) {
            before = tagged(tag, kExitsUntrusted);
            break;
        }
    }
    __threadfence();
    return before;
}

template <int MODE, int LB>
__global__ void __launch_bounds__(512, 1) chip_kernel(const __grid_constant__ ChipArgs a) {
    extern __shared__ __align__(128) unsigned char sm[];
    __shared__ unsigned s_tmem;
    __shared__ int s_next[2];
    __shared__ int s_last;
    __shared__ ChipParams s_p;
    const int warp = threadIdx.x >> 5;
    // the first CTAs take the exit word over for this launch, by a compare-and-swap that nobody
    // waits for (by every CTA it cost 1.2 us, hundreds at one address)
    const bool claims = a.tag && blockIdx.x < 4 && threadIdx.x == 32;
    unsigned long long found = 0;
    if (claims) found = ld_relaxed_gpu(a.exits);
    if (warp == 0) tmem_alloc(&s_tmem, (unsigned)a.tmem_cols);
    if (a.list && threadIdx.x == 0) s_next[0] = (int)atomicAdd(a.ticket, 1u);
    __syncthreads();
    const unsigned base = a.tmem_cols ? s_tmem : 0u;
    // a warp reaches the TMEM lanes of its number mod 4; the warps that share them take
    // 128 columns each
    const unsigned tmem = base + ((unsigned)(warp & 3) << 21) + (unsigned)(warp >> 2) * 128u;
    const int lane = threadIdx.x & 31;
    ChipState cs{-1, -1, 0u, !a.few};
    if (!a.list) {
        chip_setup<MODE>(a.one, sm);
        cs.word = lane < a.one.g.nsink ? __ldg(a.one.g.sink + lane) : 0u;
        chip_times<MODE>(a.one, sm, blockIdx.x);   // (the grid has no CTA without a chunk)
        cp_async_wait<0>();
        __syncthreads();
        if (claims && found >> kTagShift != a.tag) {
            const bool clean = found == 0 || ((unsigned)found & ((1u << kTagShift) - 1u)) == kExitsDone;
            atomicCAS(a.exits, found, tagged(a.tag, clean ? 0u : kExitsUntrusted));
        }
        for (int c = blockIdx.x; c < a.one.nchunks; c += gridDim.x)
            chip_chunk<MODE, LB>(a.one, c, sm, tmem, cs, [&] {
                const int n = c + (int)gridDim.x;
                return n < a.one.nchunks ? n : -1;
            });
        chip_finish<MODE>(a.one, sm, cs);
        if (!a.few) chip_sum_own<MODE>(a.one, sm, 0, a.exits, a.tag);
    } else {
        int g = -1;
        for (int buf = 0;; buf ^= 1) {
            const int c = s_next[buf];
            if (c >= a.total) break;
            if (threadIdx.x == 0) s_next[buf ^ 1] = (int)atomicAdd(a.ticket, 1u);   // read after a barrier
            int h = max(g, 0);
            while (h + 1 < a.n && a.list[h + 1].first_chunk <= c) ++h;
            if (h != g) {
                if (g >= 0) chip_finish<MODE>(s_p, sm, cs);
                g = h;
                static_assert(sizeof(ChipParams) % 4 == 0, "copied as words");
                for (int q = threadIdx.x; q < (int)(sizeof(ChipParams) / 4); q += blockDim.x)
                    reinterpret_cast<unsigned*>(&s_p)[q] = __ldg(reinterpret_cast<const unsigned*>(a.list + h) + q);
                __syncthreads();
                chip_setup<MODE>(s_p, sm);
                cs.word = lane < s_p.g.nsink ? __ldg(s_p.g.sink + lane) : 0u;
                chip_times<MODE>(s_p, sm, c - s_p.first_chunk);
                cp_async_wait<0>();
                __syncthreads();
            }
            chip_chunk<MODE, LB>(s_p, c - s_p.first_chunk, sm, tmem, cs, [&] {
                const int n = s_next[buf ^ 1] - s_p.first_chunk;
                return n < s_p.nchunks ? n : -1;
            });
        }
        if (g >= 0) chip_finish<MODE>(s_p, sm, cs);
        int first = 0;
        for (int h = 0; h < a.n && !a.few; ++h) {
            chip_sum_own<MODE>(a.list[h], sm, first, a.exits, kClearedTag);
            first += (int)((a.list[h].S + kReduceBlock - 1) / kReduceBlock);
        }
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        // (one atomic with both orders: between two fences it took 1,000 cycles longer)
        unsigned long long before;
        asm volatile("atom.add.acq_rel.gpu.global.u64 %0, [%1], 1;" : "=l"(before) : "l"(a.exits) : "memory");
        if (before >> kTagShift != a.tag) before = chip_exit_early(a.exits, a.tag);
        const unsigned n = (unsigned)(before - tagged(a.tag, 0u)) + 1u;   // CTAs that have left, or more than all
        s_last = n == gridDim.x ? 1 : n == (gridDim.x | kExitsUntrusted) ? 2 : 0;
    }
    __syncthreads();
    if (s_last) {   // every other CTA has counted its chunks in and left
        const int n = a.list ? a.n : 1;
        for (int h = 0; h < n; ++h) {
            const ChipParams& p = a.list ? a.list[h] : a.one;
            chip_sum_rest<MODE>(p, sm, a.few || s_last == 2);
        }
        __syncthreads();
        for (int h = warp; h < n; h += blockDim.x >> 5) chip_mean<MODE>(a.list ? a.list[h] : a.one, threadIdx.x & 31);
        if (!a.list && warp > 0) {   // beside the mean (a batch's words are cleared before each launch)
            const int words = s_last == 2 ? a.one.arrive_cap : a.few ? 0 : chip_blocks(a.one);
            for (int b = threadIdx.x - 32; b < words; b += blockDim.x - 32) a.one.arrive[b] = 0;
            if (threadIdx.x == 32)
                atomicCAS(a.exits, tagged(a.tag, (s_last == 2 ? kExitsUntrusted : 0u) | gridDim.x), tagged(a.tag, kExitsDone));
        }
    }
    __syncthreads();
    if (warp == 0 && a.tmem_cols) tmem_dealloc(base, (unsigned)a.tmem_cols);
}

template <int MODE, int LB>
const void* ck() {
    return reinterpret_cast<const void*>(&chip_kernel<MODE, LB>);
}

const void* select_chip(int kmode, int lb) {
    switch (kmode * 32 + lb) {
        case COS_MODE_FP64 * 32 + 16: return ck<COS_MODE_FP64, 16>();
        case COS_MODE_FP64 * 32 + 8: return ck<COS_MODE_FP64, 8>();
        case COS_MODE_FP32_MIXED * 32 + 16: return ck<COS_MODE_FP32_MIXED, 16>();
        case COS_MODE_FP32_MIXED * 32 + 8: return ck<COS_MODE_FP32_MIXED, 8>();
        case COS_MODE_FP32_MIXED * 32 + 4: return ck<COS_MODE_FP32_MIXED, 4>();
        case COS_MODE_COUNT_I64 * 32 + 16: return ck<COS_MODE_COUNT_I64, 16>();
        case COS_MODE_COUNT_I64 * 32 + 8: return ck<COS_MODE_COUNT_I64, 8>();
        case kModeMixedAbs * 32 + 16: return ck<kModeMixedAbs, 16>();
        case kModeMixedAbs * 32 + 8: return ck<kModeMixedAbs, 8>();
        case kModeMixedAbs * 32 + 4: return ck<kModeMixedAbs, 4>();
        default: return nullptr;
    }
}

// Bytes of one sample in a node's row and in a slot's row.
int node_bytes(int kmode) { return kmode == COS_MODE_FP32_MIXED ? 4 : 8; }
int slot_bytes(int kmode) {
    return kmode == COS_MODE_COUNT_I64 ? 0 : base_mode(kmode) == COS_MODE_FP32_MIXED ? 4 : 8;
}

// Shared memory of one CTA when `ctas` share an SM (1 KB of 228 KB reserved per CTA, and
// the kernel's static shared memory).
int smem_limit(int ctas) { return 228 * 1024 / ctas - 1024 - 512; }

struct ChipLayout {
    int lev_bytes, g_off, times_off, tab_off, coef_off, tail_off, total, kinds;
};

// Shared-memory layout of a CTA; total > limit when it does not fit.
ChipLayout chip_layout(const ChipGraph& g, int kmode, int P, int K, int D, bool table, int rb, int limit) {
    ChipLayout y;
    const bool count = kmode == COS_MODE_COUNT_I64;
    const int s = rb / node_bytes(kmode);
    const int64_t gbytes = count ? 0 : round128((int64_t)(P + 1) * s * slot_bytes(kmode));
    const int64_t times = count ? 0 : round128(8LL * D * s), tab = round128(16LL * g.tables);
    const int64_t coef = count ? 0 : round128(chip_coef_bytes(K));
    const int64_t tail = g.tail_width <= kTailRows ? round128((int64_t)(g.tail_width + 1) * rb) : 0;
    const int64_t level = std::max<int64_t>(round128((int64_t)(g.max_width + 1) * rb), round128(sizeof(CtaSum)));
    const int64_t rest = gbytes + times + tab + coef + tail;
    int64_t lev = level;
    y.kinds = K;
    if (!count && !table) {
        const int64_t fixed = kScratchAt + chip_pair_bytes(D), kind = 24LL * D * chip_pitch(s);
        y.kinds = (int)std::max<int64_t>(1, std::min<int64_t>(K, (std::max<int64_t>(level, limit - rest) - fixed) / kind));
        lev = std::max<int64_t>(level, round128(fixed + kind * y.kinds));
    }
    // room for a level and the next beside it, where there is some: no staging
    lev = std::max<int64_t>(lev, std::min<int64_t>(2 * level, (limit - rest) / 128 * 128));
    y.lev_bytes = (int)std::min<int64_t>(lev, 1 << 28);
    y.g_off = y.lev_bytes;
    y.times_off = y.g_off + (int)gbytes;
    y.tab_off = y.times_off + (int)times;
    y.coef_off = y.tab_off + (int)tab;
    y.tail_off = tail ? y.coef_off + (int)coef : -1;
    y.total = (int)(y.lev_bytes + rest);
    return y;
}

}  // namespace

int chip_phase_rows(int64_t max_width, int64_t P, int32_t K, int32_t D) {
    ChipGraph g;
    g.max_width = (int32_t)std::min<int64_t>(max_width, INT32_MAX - 1);
    g.tail_width = kTailRows;
    if (max_width > 65534 || P > 65534) return 0;
    for (int rb = 128; rb >= 4; rb /= 2)
        if (chip_layout(g, COS_MODE_FP32_MIXED, (int)P, K, D, false, rb, smem_limit(1)).total <= smem_limit(1)) return 128 / rb;
    return 0;
}

// Model of the time of an evaluation in microseconds, fitted to 16 graphs (1,000 to 117,000
// nodes, 300 to 65,536 samples, every mode) in every shape that fits them, 6 % rms.  Per
// chunk: the busiest of the shared-memory pipe (128 bytes per cycle, times the passes per
// phase that the row order leaves), the issue slots and the FP64 pipe, then the propagators,
// four tenths of whose time CTAs that share an SM hide from one another, then what a chunk
// waits for by itself -- barriers, fetch and L2 latency, mostly per level -- which they hide
// almost wholly.  Order 2, 1,000 nodes, 10,007 samples, FP32: one CTA with 32 samples 72
// us, two with 16 or 8 samples 66, four with 8 samples 70; medium, FP32: one with 8 samples
// 1.61 ms, two with 4 samples 1.99.
double chip_time_us(const ChipGraph& g, int kmode, int32_t L, int32_t P, int32_t K, int32_t D, bool table, int64_t S, int sms,
                    int rb, int lane, int ctas, int members) {
    const int s = rb / node_bytes(kmode), mode = base_mode(kmode);
    const double B = 128.0 / rb;
    double conf = B <= 1 ? 1.0 : B <= 2 ? 1.15 : B <= 4 ? 1.5 : B <= 8 ? 2.0 : B <= 16 ? 2.4 : 2.5;
    const double tables = mode == COS_MODE_COUNT_I64 ? 1.0 : kmode == kModeMixedAbs ? 1.65 : 2.0;
    const double lds = (double)g.edges * rb / 128.0 * conf * tables + (double)g.rows * rb / 128.0 * 1.3;
    const double issue = ((double)g.edges * 15.2 + (double)g.rows * 47.9) * rb / lane / 32.0 / 4.0;
    const double f64 = mode == COS_MODE_FP64 ? (double)g.edges * s / 2.0 * 1.1 : 0.0;
    double props = 0.0;
    if (table) props = (double)P * s * 4.0;
    else if (mode == COS_MODE_FP64) props = ((double)K * D * s * 19.9 + (double)P * s) / 2.0 * 1.1;
    else if (mode == COS_MODE_FP32_MIXED) props = (double)K * D * s * 0.68 + (double)P * s * 0.62;
    const double busy = std::max(lds, std::max(issue, f64)), alone = 3000.0 + 590.0 * L;
    const int64_t chunks = (S + s - 1) / s, slots = (int64_t)ctas * sms;
    const double wave = ctas * (busy + 0.59 * props) + 0.41 * props + alone * (1.0 + 0.03 * (ctas - 1));
    // (the chunks of a batch's members fill one another's last rounds)
    const double rounds = members > 1 ? (double)chunks / (double)slots : (double)((chunks + slots - 1) / slots);
    return rounds * wave / 1930.0 + 13.9 / members;
}

// The same for the general kernels: launch and barriers or task planning, edges at the
// rate they reach on graphs of this kind, propagator slots (through L2, and back).
double general_time_us(const ChipGraph& g, int kmode, int32_t L, int32_t P, int64_t S, int members) {
    const double es = (double)g.edges * (double)S, ps = (double)P * (double)S, fixed = (45.0 + 3.0 * L) / members;
    if (kmode == COS_MODE_COUNT_I64) return fixed + es / 9.5e5;
    if (kmode == COS_MODE_FP64) return fixed + es / 5.4e5 + ps / 1.5e5;
    return fixed + es / (kmode == kModeMixedAbs ? 8.5e5 : 1.65e6) + ps / 3e5;
}

// The shape with the least model time; on chip when that is below the general kernels'.
// Measured on both sides of the line, general / on-chip: medium graph, 65,536 samples, 2.35 /
// 1.62 ms (FP32), 3.89 / 2.86 ms (with A), 3.1 / 1.85 ms (count), FP64, 16,384 samples, 1.60 / 1.63 ms
// (both held by the FP64 pipe; general), 10,000 nodes of order 4, FP64, 2,000 samples 226 /
// 169 us; FP32 with two samples per chunk: 100,000 nodes, levels of 12,200, 4,000 samples 868 /
// 988 us (general), 500 samples 198 / 131; levels of 19,500 5.44 / 5.80 ms (general), but
// 3,000 samples of the latter 0.48 / 0.42 ms and 300 samples of levels of 30,000 102 / 63 us.
// The members of a batch share the fixed times of either side and the last rounds.
bool chip_plan(const ChipGraph& g, int kmode, int32_t L, int32_t P, int32_t K, int32_t D, bool table, int64_t S, int sms,
               int members, ChipPlan* out) {
    if (g.max_width <= 0 || S <= 0 || sms <= 0 || kmode == kModeFp64Abs) return false;
    const int nb = node_bytes(kmode);
    bool found = false;
    for (int rb = std::max(nb, 4); rb <= 128; rb *= 2) {
        const int lane = std::min(kmode == kModeMixedAbs ? rb / 2 : rb, 16);   // (a piece is wholly R or wholly A)
        // the chunks of a launch, those of a batch's members together, are counted in 32 bits
        if ((S + rb / nb - 1) / (rb / nb) > (INT32_MAX - (1 << 20)) / std::max(members, 1)) continue;
        for (int ctas = 1; ctas <= 4; ctas *= 2) {
            const ChipLayout y = chip_layout(g, kmode, P, K, D, table, rb, smem_limit(ctas));
            if (y.total > smem_limit(ctas) || 512 / ctas / 32 < rb / lane) continue;   // (a group needs rb / lane warps)
            const double cost = chip_time_us(g, kmode, L, P, K, D, table, S, sms, rb, lane, ctas, members);
            if (found && cost >= out->cost) continue;
            found = true;
            out->rb_log2 = 31 - __builtin_clz((unsigned)rb);
            out->lane_bytes = lane;
            out->threads = 512 / ctas;
            out->ctas = ctas;
            out->smem = y.total;
            out->cost = cost;
        }
    }
    return found && out->cost < 0.97 * general_time_us(g, kmode, L, P, S, members);
}

void chip_shape(int kmode, const ChipPlan& plan, ChipParams* p) {
    const int rb = 1 << plan.rb_log2, s = rb / node_bytes(kmode);
    const ChipLayout y = chip_layout(p->g, kmode, p->P, p->K, p->D, p->ptab != nullptr, rb, smem_limit(plan.ctas));
    p->rb_log2 = plan.rb_log2;
    p->s_log2 = 31 - __builtin_clz((unsigned)s);
    p->kinds_per_pass = y.kinds;
    p->lev_bytes = y.lev_bytes;
    p->g_off = y.g_off;
    p->times_off = y.times_off;
    p->tab_off = y.tab_off;
    p->coef_off = y.coef_off;
    p->tail_off = y.tail_off;
    p->d_magic = p->D > 1 ? (uint32_t)(((1ull << 32) + (uint64_t)p->D - 1) / (uint64_t)p->D) : 0;
    p->nchunks = (int32_t)((p->S + s - 1) / s);
}

namespace {

// Blocks of samples up to which the last CTA sums them all, one after another: 2 for a CTA of
// 128 threads, 8 for one of 512.
int few_blocks(int threads) { return 2 * (threads / 128); }

int launch(int kmode, int lane_bytes, int threads, int smem, bool staged, ChipArgs& a, int chunks, int sms, cudaStream_t st) {
    const void* k = select_chip(kmode, lane_bytes);
    if (!k) return set_error(COS_ERR_INVALID, "no on-chip kernel for mode %d, %d bytes per lane", kmode, lane_bytes);
    // (always the same limit: calls of other threads may come between this one and the launch)
    if (prepare_kernel_attrs(k, smem_limit(1)) != COS_OK) return set_error(COS_ERR_CUDA, "cannot set dynamic shared memory");
    const int ctas = 512 / threads;
    a.tmem_cols = staged ? 512 / ctas : 0;
    void* args[] = {&a};
    const int grid = std::min(chunks, sms * ctas);
    const cudaError_t e = cudaLaunchKernel(k, dim3((unsigned)grid), dim3((unsigned)threads), args, (size_t)smem, st);
    if (e != cudaSuccess) {
        cudaGetLastError();
        return set_error(COS_ERR_CUDA, "on-chip walk launch: %s", cudaGetErrorString(e));
    }
    return COS_OK;
}

}  // namespace

unsigned long long next_chip_tag() {
    static std::atomic<unsigned long long> tag{kClearedTag};
    return ++tag;
}

int launch_chip(int kmode, const ChipPlan& plan, const ChipParams& p, int sms, bool waits, cudaStream_t st) {
    ChipArgs a{};
    a.one = p;
    const int64_t blocks = (p.S + kReduceBlock - 1) / kReduceBlock;
    cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
    if (!waits && cudaStreamIsCapturing(st, &cap) != cudaSuccess) cudaGetLastError();   // (the launch reports it)
    if (cap != cudaStreamCaptureStatusNone) {   // replays carry one tag
        a.one.tag = kClearedTag;
        cudaError_t e = cudaMemsetAsync(p.arrive, 0, sizeof(*p.arrive) * (size_t)p.arrive_cap, st);
        if (e == cudaSuccess) e = cudaMemsetAsync(p.exits, 0, sizeof(*p.exits), st);
        if (e != cudaSuccess) return set_error(COS_ERR_CUDA, "clear arrival counters: %s", cudaGetErrorString(e));
    }
    a.exits = p.exits;
    a.tag = a.one.tag;
    a.few = blocks <= few_blocks(plan.threads);
    // with room for any two levels none goes through TMEM, whose allocation takes 700 cycles
    const bool staged = p.lev_bytes < 2 * round128(((int64_t)p.g.max_width + 1) << p.rb_log2);
    return launch(kmode, plan.lane_bytes, plan.threads, plan.smem, staged, a, p.nchunks, sms, st);
}

int launch_chip_list(int kmode, int lane_bytes, int threads, int smem, const ChipParams* list, int n, int total,
                     unsigned* ticket, unsigned long long* exits, int sms, cudaStream_t st) {
    ChipArgs a{};
    a.exits = exits;
    a.tag = kClearedTag;
    a.list = list;
    a.n = n;
    a.total = total;
    a.ticket = ticket;
    return launch(kmode, lane_bytes, threads, smem, true, a, total, sms, st);
}

}  // namespace cosgpu

// On-chip walk: host interface shared by cos_graph.cu, cos_batch.cu and cos_noalloc.cu
// (kernel and planner in cos_chip.cu, row schedule in cos_chip.h).
#pragma once

#include <cstdint>
#include <cuda_runtime.h>

#include "cos_internal.cuh"

namespace cosgpu {

// Device form of a graph's ChipSchedule, owned by the graph's shared arrays.
struct ChipGraph {
    const int4* lev = nullptr;      // [L] ChipLevel, then the group descriptors (4 per unit)
    const uint32_t* words = nullptr;
    const uint32_t* sink = nullptr;
    const uint2* slots = nullptr;   // [P]: (k*D+i) | (k*D+j) << 16,  (i*D+j) | k << 16 | sign << 31
    int32_t nsink = 0;
    int32_t max_width = 0;          // 0: the graph has no schedule
    int32_t tail_width = 0;         // width of the level before the sink
    int32_t tables = 0;             // 16-byte units of lev
    int64_t edges = 0, rows = 0;
};

// A launch leaves the block words at zero.  Launches that share them and overlap (which
// spoils their own results) do not, so that the exit word also tells whether they can be
// trusted: its upper 44 bits are the number of the launch that counts its CTAs there, a
// number that no other launch of the process has, and the last CTA of a launch that
// nothing came between marks it kExitsDone.  A launch that finds neither this nor zero
// counts under kExitsUntrusted: its last CTA sums every block itself and clears all block words.
// A CTA of an overlapping launch that wrote a block word after that leaves later still, and
// its count spoils the mark again.  Clearing the words on the stream before each launch instead
// would cost a node of some 2 us in front of a tiny graph's 14; that is what a captured
// launch has, whose replays carry one number, and a batch's.
constexpr int kTagShift = 20;
constexpr unsigned long long kClearedTag = 0;   // of launches whose words are cleared before
constexpr unsigned kExitsDone = 1u << 19, kExitsUntrusted = 1u << 18;
unsigned long long next_chip_tag();

constexpr int kChipMaxTimes = 48;   // D: the sign masks of all (i, j) pairs are kept in shared memory

// Everything the kernel needs about one evaluation.
struct ChipParams {
    ChipGraph g;
    const int32_t* kind_slot;
    const double* exp_tab;
    const double* t;
    const double* eps;
    const double* ptab;
    void* R;
    double* Rabs;
    double* partials;
    double* partials_abs;
    Ctrl* ctrl;
    double* mean_out;          // optional second destination of the mean(s)
    unsigned* arrive;          // [blocks of kReduceBlock samples]: samples that are written
    unsigned long long* exits; // CTAs of the launch that have left (see kTagShift)
    unsigned long long tag;    // this launch's number
    double beta, ptab_inv_h;
    int64_t S, t_ld;
    int32_t L, P, K, D, ptab_T, abs_weights;
    int32_t clear_err;         // 1: a completed evaluation clears ctrl->err
    int32_t arrive_cap;        // words at `arrive`
    int32_t nchunks, first_chunk;
    int32_t rb_log2, s_log2;   // bytes of a node's row; samples per chunk
    uint32_t d_magic;          // ceil(2^32 / D): r / D = mulhi(r, d_magic) for r < 65536 (D > 1)
    int32_t kinds_per_pass;    // kinds whose exponentials fit the scratch at once
    // shared memory: level buffer [0, lev_bytes), then propagator rows, times, level and
    // group tables, constants, and the tail level (-1: it is in the level buffer)
    int32_t lev_bytes, g_off, times_off, tab_off, coef_off, tail_off;
    int32_t pad;
};

// Launch shape of one evaluation.
struct ChipPlan {
    int rb_log2, lane_bytes, threads, ctas, smem;
    double cost;               // model time of the evaluation, in SM cycles
};

// Best launch shape for `kmode` on S samples of a graph (max D of the kinds' times,
// P slots, K kinds), one of `members` evaluations that run together; false when the graph
// does not fit on chip or the general kernels are expected to be faster.
bool chip_plan(const ChipGraph& g, int kmode, int32_t L, int32_t P, int32_t K, int32_t D, bool table, int64_t S, int sms,
               int members, ChipPlan* out);
// Fill the shape-dependent fields of p (rb_log2 .. coef_off, nchunks).
void chip_shape(int kmode, const ChipPlan& plan, ChipParams* p);
// One evaluation, parameters by value; waits: the caller waits for it (which no capture
// survives).
int launch_chip(int kmode, const ChipPlan& plan, const ChipParams& p, int sms, bool waits, cudaStream_t st);
// Evaluations of n graphs that share (lane_bytes, threads): parameters in device
// memory, chunks [0, total) drawn from *ticket, leaving CTAs counted in *exits (both zero
// at launch, the block words of every member too).
int launch_chip_list(int kmode, int lane_bytes, int threads, int smem, const ChipParams* list, int n, int total,
                     unsigned* ticket, unsigned long long* exits, int sms, cudaStream_t st);
// Parameters and launch shape of an evaluation of g in kernel mode `kmode` (cos_graph.cu);
// *on_chip = 0 when it is the general kernels' (no schedule, no fit, or a launch shape set).
int prepare_chip(cos_graph_t g, int kmode, void* per_sample_out, int members, ChipParams* out, ChipPlan* plan, int* sms,
                 int* on_chip);
// The handle's row schedule.
void chip_view(cos_graph_t g, ChipGraph* out);
// Phase rows the row schedule of a graph is made for: the widest rows that fit on chip
// (0: no width fits).
int chip_phase_rows(int64_t max_width, int64_t P, int32_t K, int32_t D);

}  // namespace cosgpu

// grid.cuh -- what the planners for batches of a few large traces share: the
// dataflow over the whole GPU (grid.cu) and the placement in phases by one CTA
// per trace (grid_phases.cuh).
#pragma once

#include "common.cuh"
#include "launch.h"
#include "phases.cuh"

namespace mp {
namespace grid {

constexpr int32_t kGridLong = 32;  // lives above this many steps: long-lived
constexpr int32_t kMaxLongPerThread = 2;
constexpr int32_t kFarMaxLong = 2048;  // long-lived tensors of a trace placed in phases
static_assert(kGridLong == phases::kLong, "both planners split lifetimes alike");

// ---- placement in phases by one CTA per trace (grid_phases.cuh)
constexpr int32_t kFarThreads = 1024;
constexpr int32_t kPrepareThreads = 512;  // the flow kernel's
static_assert(kFarMaxLong <= kMaxLongPerThread * kFarThreads, "a thread's share of the long-lived tensors");
constexpr int32_t kFarMaxTensors = 32767;  // positions and ranks are 16-bit words below phases::kIsLong
constexpr int32_t kPer = 4;                // buckets of addresses per thread, while a long-lived tensor is placed
constexpr int32_t kBuckets = kPer * kFarThreads;
constexpr int32_t kSegments = kBuckets / 8;  // address ranges looked at more closely at a time
constexpr int32_t kFlowPairs = 9216;       // predecessors of a long-lived tensor that the dataflow's shared memory holds
constexpr int32_t kLeastRoom = 128;        // no more than it costs to find out how long the chains are
constexpr int32_t kEdges = 1024;           // positions before a window's core whose overlap is kept as bits

// Shared memory of k_far_place for n tensors, nl of them long-lived.
struct FarLayout {
    size_t oe, lg_oe, lg_af, heads, edge, mn, mx, flags, seg, total;
    __host__ __device__ FarLayout(int32_t n, int32_t nl) {
        auto a16 = [](size_t x) { return (x + 15) & ~size_t(15); };
        oe = 0;
        lg_oe = oe + a16((size_t)n * 8);
        lg_af = lg_oe + a16((size_t)nl * 8);
        heads = lg_af + a16((size_t)nl * 4);
        edge = heads + (size_t)phases::kHeads * 2;
        mn = edge + kEdges / 8;
        mx = mn + (size_t)kBuckets * 4;
        flags = mx + (size_t)kBuckets * 4;
        seg = flags + 2 * kBuckets / 8;
        total = seg + 2 * (size_t)kSegments * 8;
    }
};
constexpr size_t kFarSmem = 225 * 1024;  // of the 227 KB a CTA may have; the rest is static

// The longest chain (alloc-order positions from the first to the last member of a
// component of short lifetimes) with which one SM is expected to place a checked
// trace in phases sooner than the whole GPU's dataflow would; -1 if it cannot or
// is not whatever the chains, INT32_MAX if they do not matter (a small trace in a
// batch of large ones).  Estimates, in us, of what was measured over traces of
// 2,000 to 20,000 tensors, 2 to 6 a step, with long-lived ones that span the trace
// or a part of it (dataflow / phases, ms: 20,000, 1,000 of them long, 2 a step 30.4 /
// 12.0 FIRST, 33.8 / 42.9 BEST, 6 a step 32.8 / 44.1 FIRST; 2,000, 4 a step 1.54 /
// 1.74 and 1.94 / 4.56; 20,000 in one chain, 10 that span it 2.2 / 6.8, 100 that do
// 33.6 / 5.3):
//   - the dataflow places long-lived tensors that are live together one after
//     another, at most some 2.7 times as many in a row as are live on average,
//     each after looking at the tensors allocated during its life, several times
//     as slowly where these do not fit its shared memory;
//   - one SM pays for every long-lived tensor with the run before it; BEST looks at
//     every gap, of which long-lived tensors that overlap in part leave more; and
//     for the short-lived ones where their number is large;
//   - one warp walks a chain, member by member: 0.9 us each, more where many are
//     live at a step.
// Without long-lived tensors, or with more neighbours than are listed per short
// one, the dataflow's width wins.
__host__ __device__ inline int64_t chain_room(int64_t n, int64_t nlong, int64_t long_steps, int64_t short_steps,
                                              int64_t T, int32_t policy) {
    if (n > kFarMaxTensors || nlong > kFarMaxLong || T > 65535 || 2 * short_steps > (int64_t)phases::kNear * T)
        return -1;
    if (FarLayout((int32_t)n, (int32_t)nlong).total > kFarSmem) return -1;
    if (n <= 1024) return INT32_MAX;
    if (nlong == 0) return -1;
    // (in floating point: a thread of k_grid_prep does it with everybody waiting)
    const bool first = policy == MP_FIT_FIRST;
    const float nf = (float)n, longs = (float)nlong, live_long = (float)long_steps / (float)T;
    const float hops = fminf(2.7f * live_long, longs);
    const float seen = nf * live_long / longs;  // tensors allocated during a long-lived one's life
    float flow = hops * (15.0f + seen * (1.0f / 130.0f));
    if (!first) flow *= 1.15f;
    if (seen > (float)kFlowPairs) flow *= first ? 2.0f : 4.0f;
    float phased = 150.0f + nf * nf * (1.0f / 120000.0f);
    if (first) phased += longs * (5.0f + nf * (1.0f / 5000.0f));
    else phased += longs * (7.0f + nf * (1.0f / 1500.0f)) + (longs - live_long) * (3.0f + nf * (1.0f / 900.0f));
    const float live = (float)short_steps / (float)T;
    const float member = first ? 0.93f + 0.11f * fmaxf(live - 9.0f, 0.0f) : 0.4f + 0.29f * live;
    const float room = (flow - phased) / member;
    return room < (float)kLeastRoom ? -1 : (int64_t)room;
}

// Queues and counters shared by the whole grid.
struct GridCtl {
    int32_t head_s, tail_s;  // warp items: next slot to take, next slot to fill
    int32_t head_l, tail_l;  // CTA items
    int32_t total;           // tensors of the traces that passed their checks
    int32_t placed;          // tensors placed so far
    int32_t fail;            // a CTA gave up waiting
    int32_t checked;         // traces that passed their checks ...
    int32_t votes, neutral;  // ... for which phases may pay, and which fit them (chain_room)
    int32_t against;         // ... whose chains turned out too long for them
    int32_t arrived;         // CTAs that reached the grid's barriers, all told
    int32_t finished;        // CTAs of k_grid_finish that are done
};

// Whether the batch's traces are placed by one CTA each in phases
// (grid_phases.cuh) instead of by the dataflow: all of them or none, since the
// two would run one after the other.  Once k_grid_prep has finished this says
// whether it may be; once the chains are known (far_comps) whether it is.
__device__ __forceinline__ bool in_phases(const GridCtl* ctl) {
    return ctl->votes > 0 && ctl->votes + ctl->neutral == ctl->checked && *(const volatile int32_t*)&ctl->against == 0;
}

// Per-trace state.
struct TraceInfo {
    int64_t lo;               // first tensor of the trace in the batch arrays
    unsigned long long peak;  // largest offset + size
    unsigned long long key;   // smallest conflicting (min id, max id), packed; ~0 if none
    int32_t n, T, lw, nlong;  // tensors, steps, longest short life, long-lived tensors
    int32_t ok;               // 1 once the trace passed its checks
    int32_t incomplete;       // a tensor was left unplaced
    int32_t shift;            // every size is a multiple of 1 << shift (a unit)
    int32_t room;             // the longest chain for which phases pay (chain_room)
};

// A tensor in alloc-step order (16 bytes: one vector load).
struct GRec {
    int64_t s;
    int32_t a, f;
};

struct GridWs {
    GridCtl* ctl;
    TraceInfo* ti;
    int32_t* bend;   // [B][max_steps]: bucket ends by alloc step
    GRec* rec;       // [B][max_tensors]: alloc-ordered records
    int32_t* rid;    // tensor id of each record
    int64_t* off;    // offset of each record (-1 until placed)
    int32_t* cnt;    // signed predecessor counts
    int32_t* cls;    // 1: a CTA item (long-lived, or more predecessors than a warp's buffer)
    int32_t* qs;     // queue of ready warp items (1 + slot id, 0 = not filled)
    int32_t* ql;     // queue of ready CTA items
    int32_t* ll;     // [B][max_tensors]: positions of the long-lived records, ascending
    int64_t* ovf;    // per long-capable CTA: pairs beyond the shared region
    int64_t ovf_pairs;
    int32_t M;       // max_tensors: the slot stride of a trace
    int32_t TS;      // max_steps: the bucket stride of a trace
    int64_t hold;    // test hook: the slot that is never queued, or kHoldBarrier (-1: none)
    // For traces placed in phases, by slot (stable: alloc step, then id), or
    // by rank: null if no trace of the batch can be.
    uint32_t* p_af;  // lifetime: alloc | free << 16
    uint32_t* p_sz;  // size in units
    uint16_t* p_at;  // the record's position in rec / off
    uint32_t* p_cs;  // 1 + first position of its component of short lifetimes (0: long-lived)
    uint32_t* p_rk;  // priority rank
    phases::Rec* p_rec;    // by rank
    phases::Win* p_win;    // by rank
    uint16_t* p_near;      // by rank: phases::kNear positions
    uint16_t* p_lr;        // [B][kFarMaxLong]: ranks of the long-lived tensors, ascending
};

}  // namespace grid
}  // namespace mp

// phases.cuh -- greedy placement of one trace by one CTA in phases, for traces
// whose lifetimes link many tensors (components past the warp tier): the
// deferred traces of greedy_by_size (plan.cuh) and of greedy by breadth
// (breadth.cu).
//
// The sequential definition takes tensors in priority order and gives each a
// gap among the placed tensors whose lifetimes overlap its own.  Tensors that
// live longer than kLong steps ("long") overlap nearly everything; the others
// ("short") only a few neighbours in alloc order, and long ones.  The long
// tensors cut the priority order into runs of short ones:
//   - a run's short tensors depend on each other only inside components of
//     short lifetimes linked by overlap, which are small where the long tensors
//     held the trace together: the warps take one such chain each and walk it
//     in priority order, with no waits between warps (run_chains).  A short
//     tensor's obstacles are its window of alloc order, a lane each, and the
//     placed long tensors, kept sorted by offset: a prefix maximum of the ends
//     over 32 of them at a time exposes the gaps between them, and only gaps
//     that fit are searched among the window's tensors (place_short);
//   - a long tensor is placed by the whole CTA over the list of every placed
//     tensor, kept sorted by offset: one prefix maximum of the ends of those
//     that overlap its lifetime exposes every gap at once (place_long).  The
//     list takes the run's tensors just before it is needed (insert_pending),
//     by one shift of its entries.
// Each tensor sees exactly the tensors of lower rank that overlap it, placed,
// so the offsets are the sequential definition's.
//
// Bytes are counted in units of the largest power of two that divides every
// size of the trace: every offset and end is a sum of sizes, so nothing is
// rounded, and all arithmetic is 32-bit when the sizes sum below 2^32 units
// (otherwise, and past the limits below, the callers' general paths place the
// trace).
#pragma once

#include <type_traits>

#include "common.cuh"
#include "launch.h"

namespace mp {
namespace phases {

constexpr int32_t kLong = 32;          // lives above this many steps are long
constexpr int32_t kMaxLong = 768;      // long tensors a trace may have here
constexpr int32_t kMaxTensors = 4080;  // tensors a trace may have here: no more fit the shared memory (Layout)
constexpr uint32_t kLongestChain = 1024;  // positions a chain may span beside long tensors: one warp walks it, the
                                       // general paths' queues place its members side by side
constexpr int32_t kMixedTensors = 1024;  // most tensors a trace may have on average in a batch of mixed lengths (smem_bytes)
constexpr int32_t kBatch = 512;        // tensors inserted into the sorted list at a time
constexpr int32_t kHeads = 1024;       // chains of a run listed at a time
constexpr int32_t kChunk = 8;          // sorted-list entries per thread, at most: the callers have 512 threads, or 256
                                       // where an SM holds two CTAs, whose traces have 2,048 tensors at most
constexpr int32_t kNear = 32;          // neighbours listed per short tensor of a large trace (grid_phases.cuh)
constexpr int32_t kThreadChain = 8;    // chains up to this long within a run can be walked by one thread
constexpr int32_t kTeamChain = 64;     // chains from this length on are walked by the whole CTA together ...
constexpr int32_t kTeams = 4;          // ... up to this many of a run
#ifdef MP_TEST_SPIN_CYCLES
constexpr int32_t kTeamPolls = 1 << 17;  // test builds: some 6 ms
#else
constexpr int32_t kTeamPolls = 1 << 23;  // polls of a wait there (some 0.2 s) in which some member has to be placed
#endif
constexpr int32_t kListRun = 64;       // runs from this length on list the gaps between the long tensors first
constexpr int32_t kFewPending = 8;     // up to this many are inserted by comparison with every entry
constexpr uint32_t kScanChain = 128;  // chains are linked member by member up to this many looks per thread, else by a sort
constexpr uint64_t kLongKey = 0xfffffffffffffffeull;  // sort key of a long tensor among the chains: last
constexpr uint16_t kNone = 0xffff;     // no such rank
constexpr uint16_t kIsLong = 0xfffe;   // in Rec::prev: the tensor is long

// A tensor by priority rank.
struct __align__(16) Rec {
    uint32_t s;           // size in units
    uint16_t a, f;        // lifetime [a, f)
    uint16_t pos;         // alloc-order position
    uint16_t next, prev;  // ranks of the neighbours in its chain (component of short lifetimes)
    union {
        uint16_t many;  // kFar: more than kNear neighbours, not listed
        uint16_t comp;  // otherwise: its component of short lifetimes
    };
};
// Alloc-order positions of the short tensors that can overlap it: [w0, w1);
// those from `core` on are allocated during its life.
// Ctx::mask has the short ones of lower rank that overlap it, as bits from w0
// on, unless there are more than 32 positions (`wide`).
struct __align__(8) Win {
    uint16_t w0, core, w1, wide;
};

// Shared memory of a trace of n tensors over T steps.  Regions are reused:
// sort keys, then the (offset, end) pairs; per-step arrays (the profile's
// differences, the operators' breadths), then the records; bucket ends, then
// the long tensors and the scratch of insertions; sizes, then the windows.
struct Layout {
    size_t oe = 0, rec = 0, win = 0, mask = 0, af = 0, id = 0, sl = 0, tmp = 0, bend = 0;
    size_t lg_oe = 0, lg_af = 0, lr = 0, pk = 0, heads = 0, total = 0;
    __host__ __device__ static constexpr size_t a16(size_t x) { return (x + 15) & ~size_t(15); }
    __host__ __device__ static constexpr int32_t keys_of(int32_t n) {  // sort length
        int32_t k = 512;  // a key per thread at least
        while (k < n) k <<= 1;
        return k;
    }
    __host__ __device__ constexpr Layout(int32_t n, int32_t T, size_t step_bytes) {
        oe = 0;
        rec = oe + (size_t)keys_of(n) * 8;
        const size_t recs = a16((size_t)n * sizeof(Rec)), steps = a16((size_t)T * step_bytes);
        win = rec + (recs > steps ? recs : steps);
        mask = win + a16((size_t)n * sizeof(Win));
        af = mask + a16((size_t)n * 4);
        id = af + a16((size_t)n * 4);
        sl = id + a16((size_t)n * 2);
        tmp = sl + a16((size_t)n * 2);
        bend = tmp + a16((size_t)n * 2);
        lg_oe = bend;  // the bucket ends are dead once the windows are known
        lg_af = lg_oe + (size_t)kMaxLong * 8;
        lr = lg_af + (size_t)kMaxLong * 4;
        pk = lr + (size_t)kMaxLong * 2;
        heads = pk + (size_t)kBatch * 8;
        const size_t end = heads + (size_t)kHeads * 2, bends = bend + a16((size_t)T * 4);
        total = align_up(end > bends ? end : bends);
    }
};

// Bytes per step of the per-step array: the 32-bit differences of the profile,
// or the 64-bit breadths of the operators.
template <bool kBreadth>
__host__ __device__ constexpr size_t step_bytes() {
    return kBreadth ? 8 : 4;
}

static_assert(Layout(kMaxTensors, 1, 4).total <= kSmemCeiling && Layout(kMaxTensors + 1, 1, 4).total > kSmemCeiling,
              "the most tensors a trace may have");
static_assert(kMaxTensors <= 512 * kChunk && Layout(256 * kChunk + 1, 1, 4).total > kTwoPerSm,
              "the sorted list's entries are held in registers while some are inserted");

// Whether a trace of n tensors over T steps can be placed here with that much
// dynamic shared memory.
template <bool kBreadth>
__host__ __device__ bool fits(int32_t n, int32_t T, size_t smem) {
    return n <= kMaxTensors && T <= 65535 && Layout(n, T, step_bytes<kBreadth>()).total <= smem;
}

// Dynamic shared memory that a launch for the batch's traces should have: enough
// for the longest; where that is too much, as in a batch of ordinary traces with
// a very long one among them, what leaves an SM as many CTAs as the batch can
// use, and the traces it holds are placed here (600 chains of 374 tensors and a
// trace of 2,000 over 20,000 steps: 1.32 ms by the general path, 0.46 so); 0 if few
// would be.
template <bool kBreadth>
size_t smem_bytes(const mp_batch& bt, int sms) {
    if (fits<kBreadth>(bt.max_tensors, bt.max_steps, kSmemCeiling))
        return Layout(bt.max_tensors, bt.max_steps, step_bytes<kBreadth>()).total;
    const size_t room = bt.n_traces > sms ? kTwoPerSm : kSmemCeiling;
    const int64_t n = bt.n_tensors / bt.n_traces, T = bt.n_steps / bt.n_traces;  // of the average trace
    return n <= kMixedTensors && T <= 65535 && fits<kBreadth>((int32_t)n, (int32_t)T, room) ? room : 0;
}

struct Shared {
    uint32_t red[33];
    unsigned long long hi, lo, bits, best;
    uint32_t best32, lb, far;
    int32_t bad, lw, nl, cnt, next, cnt1, next1, teams, fail;
    int32_t seen[16];  // by warp: members of its team placed when it last asked
    int32_t hold;      // test builds: alloc-order position of a team's member that is never placed (-1: none)
    uint16_t team[kTeams];
    uint32_t last_free;
    uint32_t before[kFewPending];
    unsigned long long key;
};

// Test builds (MP_TEST_HOOKS) can keep one member of a team from being placed,
// so that the others' bounded waits run out: {trace, alloc-order position}.
#ifdef MP_TEST_HOOKS
static __device__ int32_t g_test_team_hold[2] = {-1, -1};
__device__ __forceinline__ int32_t test_team_hold(int b) { return b == g_test_team_hold[0] ? g_test_team_hold[1] : -1; }
__device__ __forceinline__ bool test_held(const Shared& sh, int32_t pos) { return pos == sh.hold; }
#else
__device__ __forceinline__ int32_t test_team_hold(int) { return -1; }
__device__ __forceinline__ bool test_held(const Shared&, int32_t) { return false; }
#endif

__device__ __forceinline__ uint32_t umax2(uint32_t a, uint32_t b) { return a > b ? a : b; }

// Inclusive prefix maximum over the warp.
__device__ __forceinline__ uint32_t warp_incl_max(uint32_t v) {
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t u = __shfl_up_sync(0xffffffffu, v, o);
        if (lane >= o) v = umax2(v, u);
    }
    return v;
}

// Exclusive prefix maximum (identity 0) over the block; the maximum in *total.
// Ends with a barrier before red may be written again by the caller's next
// call (each call starts with its own writes after the previous one's barrier).
__device__ __forceinline__ uint32_t block_excl_max(uint32_t v, uint32_t* red, uint32_t* total) {
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, nw = blockDim.x >> 5;
    const uint32_t incl = warp_incl_max(v);
    if (lane == 31) red[w] = incl;
    __syncthreads();
    const uint32_t x = lane < nw ? red[lane] : 0u;  // every warp scans the warp totals for itself
    const uint32_t xs = warp_incl_max(x);
    *total = __shfl_sync(0xffffffffu, xs, 31);
    const uint32_t wex = w == 0 ? 0u : __shfl_sync(0xffffffffu, xs, w == 0 ? 0 : w - 1);
    const uint32_t up = __shfl_up_sync(0xffffffffu, incl, 1);
    __syncthreads();
    return lane == 0 ? wex : umax2(wex, up);
}

__device__ __forceinline__ uint32_t block_excl_sum(uint32_t v, uint32_t* red, uint32_t* total) {
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, nw = blockDim.x >> 5;
    const uint32_t incl = warp_incl_scan(v);
    if (lane == 31) red[w] = incl;
    __syncthreads();
    const uint32_t x = lane < nw ? red[lane] : 0u;
    const uint32_t xs = warp_incl_scan(x);
    *total = __shfl_sync(0xffffffffu, xs, 31);
    const uint32_t wex = w == 0 ? 0u : __shfl_sync(0xffffffffu, xs, w == 0 ? 0 : w - 1);
    __syncthreads();
    return wex + incl - v;
}

// Ascending bitonic sort of a key per lane.
__device__ __forceinline__ uint64_t warp_sort(uint64_t k) {
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int kk = 2; kk <= 32; kk <<= 1) {
#pragma unroll
        for (int j = kk >> 1; j > 0; j >>= 1) {
            const uint64_t o = __shfl_xor_sync(0xffffffffu, k, j);
            const bool keep_min = ((lane & kk) == 0) == ((lane & j) == 0);
            k = (o < k) == keep_min ? o : k;
        }
    }
    return k;
}

// Ascending bitonic sort of E * blockDim keys (a power of two), E per thread:
// thread t holds elements t E .. t E + E - 1.  Strides below E stay in the
// thread's registers, strides inside a warp are shuffles, and only the wider
// ones go through shared memory (buf: E * blockDim words).
template <int E>
__device__ void block_sort(uint64_t (&k)[E], uint64_t* buf) {
    const int32_t t = (int32_t)threadIdx.x, nt = (int32_t)blockDim.x;
    const int32_t len = E * nt;
    for (int32_t kk = 2; kk <= len; kk <<= 1) {
        for (int32_t j = kk >> 1; j > 0; j >>= 1) {
            if (j >= E) {
                const int32_t d = j / E;  // partner thread: t ^ d
                const bool lower = (t & d) == 0;
                const bool up = ((t * E) & kk) == 0;  // kk > j >= E: the same for all E elements
                const bool keep_min = up == lower;
                if (d < 32) {
#pragma unroll
                    for (int e = 0; e < E; ++e) {
                        const uint64_t o = __shfl_xor_sync(0xffffffffu, k[e], d);
                        k[e] = (o < k[e]) == keep_min ? o : k[e];
                    }
                } else {
                    __syncthreads();  // the previous stage's reads are done
#pragma unroll
                    for (int e = 0; e < E; ++e) buf[e * nt + t] = k[e];
                    __syncthreads();
#pragma unroll
                    for (int e = 0; e < E; ++e) {
                        const uint64_t o = buf[e * nt + (t ^ d)];
                        k[e] = (o < k[e]) == keep_min ? o : k[e];
                    }
                }
            } else {
#pragma unroll
                for (int jj = E >> 1; jj > 0; jj >>= 1) {  // (j is one of these: indices stay compile-time)
                    if (j == jj) {
#pragma unroll
                        for (int e = 0; e < E; ++e) {
                            const int l = e ^ jj;
                            if (l > e) {
                                const bool up = ((t * E + e) & kk) == 0;
                                const uint64_t a = k[e], b = k[l];
                                const bool swap = (b < a) == up;
                                k[e] = swap ? b : a;
                                k[l] = swap ? a : b;
                            }
                        }
                    }
                }
            }
        }
    }
    __syncthreads();
}

// The trace being placed.  kFar: a large trace whose records by rank and
// lifetimes are in global memory, with the neighbours of its short tensors
// listed beforehand (grid_phases.cuh).
template <bool kFar>
struct Ctx {
    uint2* oe;            // by position: (offset, end) in units; (0, 0) until placed
    const uint32_t* af;   // by position: alloc step | free step << 16
    uint16_t* sl;         // positions of placed tensors by ascending offset
    uint2* lg_oe;         // placed long tensors by ascending offset: (offset, end)
    uint32_t* lg_af;      // ... and lifetimes
    const Rec* rec;       // by rank
    const Win* win;       // by rank
    const uint32_t* mask; // by rank
    uint64_t* pk;         // kBatch keys of tensors being inserted; gaps (start << 32 | length) otherwise
    uint16_t* heads;      // kHeads ranks
    uint16_t* list;       // ranks of the members of one chain (not kFar)
    const uint16_t* near; // kFar, by rank: positions of the kNear short tensors it overlaps (kNone: no more)
    int32_t policy;
};

// The placed long tensors as short tensors meet them: nlp of them, all live
// during [late, early) -- the latest alloc and the earliest free step.  When
// that spans every short tensor's life, the gaps between all of the long ones
// are every short tensor's gaps: ng of them are listed in Ctx::pk, ascending,
// up to `top` (ng < 0: no list).
struct Longs {
    int32_t nlp, ng;
    uint32_t late, early, top;
};

// The window obstacles of a short tensor as one thread walks them: the set
// bits of `mask` are positions from w0 on ((0, 0) entries never conflict).
struct Near {
    const uint2* oe;  // at w0
    uint32_t mask, s;

    // FIRST: the lowest offset from `from` on that meets none of them, or one
    // from which the tensor would not end by `lim`.
    __device__ __forceinline__ uint32_t settle(uint32_t from, uint32_t lim) const {
        uint32_t o = from;
        for (;;) {
            uint32_t m = 0;
            for (uint32_t b = mask; b; b &= b - 1) {
                const uint2 v = oe[__ffs(b) - 1];
                m = (v.x < o + s) & (o < v.y) & (v.y > m) ? v.y : m;
            }
            if (m <= o) return o;
            o = m;
            if (o + s > lim) return o;
        }
    }
    // BEST: the holes between them in [from, lim).
    __device__ __forceinline__ void holes(uint32_t from, uint32_t lim, uint32_t& best, uint32_t& best_len) const {
        uint32_t o = from;
        while (o < lim) {
            uint32_t m = 0, ns = lim;
            for (uint32_t b = mask; b; b &= b - 1) {
                const uint2 v = oe[__ffs(b) - 1];
                m = (v.x <= o) & (o < v.y) & (v.y > m) ? v.y : m;
                ns = (v.x > o) & (v.x < ns) ? v.x : ns;
            }
            if (m > o) {  // covered: past it
                o = m;
                continue;
            }
            const uint32_t len = ns - o;
            if (len >= s && len < best_len) {
                best_len = len;
                best = o;
            }
            o = ns;
        }
    }
    __device__ __forceinline__ uint32_t top(uint32_t at_least) const {
        uint32_t t = at_least;
        for (uint32_t b = mask; b; b &= b - 1) t = umax2(t, oe[__ffs(b) - 1].y);
        return t;
    }
};

// Places the short tensor of rank r, whose gaps between long ones are listed
// and whose window has a mask, with one thread; returns its end.
__device__ __forceinline__ uint32_t place_short_alone(const Ctx<false>& c, int32_t r, const Longs& lg) {
    const Rec rc = c.rec[r];
    const Near nr = {c.oe + c.win[r].w0, c.mask[r], rc.s};
    const uint32_t s = rc.s;
    uint32_t best = 0, best_len = 0xffffffffu;
    if (c.policy == MP_FIT_FIRST) {
        bool found = false;
        for (int32_t k = 0; k < lg.ng && !found; ++k) {
            const uint64_t v = c.pk[k];
            if ((uint32_t)v < s) continue;
            const uint32_t g0 = (uint32_t)(v >> 32), g1 = g0 + (uint32_t)v;
            best = nr.settle(g0, g1);
            found = best + s <= g1;
        }
        if (!found) best = nr.settle(lg.top, 0xffffffffu);
    } else {
        for (int32_t k = 0; k < lg.ng; ++k) {
            const uint64_t v = c.pk[k];
            const uint32_t g0 = (uint32_t)(v >> 32);
            if ((uint32_t)v >= s) nr.holes(g0, g0 + (uint32_t)v, best, best_len);
        }
        const uint32_t top = nr.top(lg.top);
        nr.holes(lg.top, top, best, best_len);
        if (best_len == 0xffffffffu) best = top;
    }
    c.oe[rc.pos] = make_uint2(best, best + s);
    return best + s;
}

// The same with one warp, a gap per lane.
__device__ __forceinline__ uint32_t place_short_listed(const Ctx<false>& c, int32_t r, const Longs& lg) {
    const unsigned full = 0xffffffffu;
    const int lane = threadIdx.x & 31;
    const Rec rc = c.rec[r];
    const Near nr = {c.oe + c.win[r].w0, c.mask[r], rc.s};
    const uint32_t s = rc.s;
    uint32_t best = 0, best_len = 0xffffffffu;
    if (c.policy == MP_FIT_FIRST) {
        bool found = false;
        for (int32_t k0 = 0; k0 < lg.ng && !found; k0 += 32) {
            const uint64_t v = k0 + lane < lg.ng ? c.pk[k0 + lane] : 0;
            bool ok = false;
            uint32_t o = 0;
            if ((uint32_t)v >= s) {
                const uint32_t g0 = (uint32_t)(v >> 32), g1 = g0 + (uint32_t)v;
                o = nr.settle(g0, g1);
                ok = o + s <= g1;
            }
            const unsigned m = __ballot_sync(full, ok);
            if (m) {
                best = __shfl_sync(full, o, __ffs(m) - 1);
                found = true;
            }
        }
        if (!found) best = nr.settle(lg.top, 0xffffffffu);
    } else {
        for (int32_t k0 = 0; k0 < lg.ng; k0 += 32) {
            const uint64_t v = k0 + lane < lg.ng ? c.pk[k0 + lane] : 0;
            const uint32_t g0 = (uint32_t)(v >> 32);
            if ((uint32_t)v >= s) nr.holes(g0, g0 + (uint32_t)v, best, best_len);
        }
        const uint32_t ln = __reduce_min_sync(full, best_len);
        best = __reduce_min_sync(full, best_len == ln ? best : 0xffffffffu);
        best_len = ln;
        const uint32_t top = nr.top(lg.top);
        nr.holes(lg.top, top, best, best_len);
        if (best_len == 0xffffffffu) best = top;
    }
    __syncwarp();
    if (lane == 0) c.oe[rc.pos] = make_uint2(best, best + s);
    __syncwarp();
    return best + s;
}

// Places the short tensor of rank r with one warp; returns its end.
template <bool kFar>
__device__ __forceinline__ uint32_t place_short(const Ctx<kFar>& c, int32_t r, const Longs& lg) {
    const unsigned full = 0xffffffffu;
    const int32_t nlp = lg.nlp;
    const int lane = threadIdx.x & 31;
    const Rec rc = c.rec[r];
    const Win w = c.win[r];
    const uint32_t s = rc.s, a = rc.a, f = rc.f;
    const int32_t w0 = w.w0, core = w.core, w1 = w.w1;
    auto load = [&](int32_t q) -> uint2 {  // (0, 0): not an obstacle
        uint2 v = c.oe[q];
        if (q < core && (c.af[q] >> 16) <= a) v = make_uint2(0, 0);
        return v;
    };
    uint2 p0 = make_uint2(0, 0), p1 = make_uint2(0, 0);
    int32_t rest = w0 + 64;  // window positions from here on are not held in p0, p1
    if constexpr (kFar) {
        const uint32_t q = c.near[(size_t)r * kNear + lane];  // (loaded with the record, whatever it says)
        if (!rc.many && q != kNone) p0 = c.oe[q];
        rest = rc.many ? w0 : w1;
    } else {
        if (w0 + lane < w1) p0 = load(w0 + lane);
        if (w0 + 32 + lane < w1) p1 = load(w0 + 32 + lane);
    }
    const bool wide = rest < w1;
    auto each = [&](auto&& fn) {
        fn(p0.x, p0.y);
        if (!kFar) fn(p1.x, p1.y);
        if (wide)
            for (int32_t q = rest + lane; q < w1; q += 32) {
                const uint2 v = load(q);
                fn(v.x, v.y);
            }
    };
    // FIRST: the lowest offset from `from` on that meets no window tensor, or
    // one from which the tensor would not end by `lim`.
    auto settle = [&](uint32_t from, uint32_t lim) -> uint32_t {
        uint32_t o = from;
        for (;;) {
            uint32_t m = 0;
            each([&](uint32_t po, uint32_t pe) {
                m = (po < o + s) & (o < pe) & (pe > m) ? pe : m;
            });
            m = __reduce_max_sync(full, m);
            if (m <= o) return o;
            o = m;
            if (o + s > lim) return o;
        }
    };
    uint32_t best = 0, best_len = 0xffffffffu;
    // BEST: the holes between window tensors in [from, lim).
    auto holes = [&](uint32_t from, uint32_t lim) {
        uint32_t o = from;
        while (o < lim) {
            uint32_t m = 0;
            each([&](uint32_t po, uint32_t pe) {
                m = (po <= o) & (o < pe) & (pe > m) ? pe : m;
            });
            m = __reduce_max_sync(full, m);
            if (m > o) {
                o = m;
                continue;
            }
            uint32_t ns = lim;
            each([&](uint32_t po, uint32_t) {
                ns = (po > o) & (po < ns) ? po : ns;
            });
            ns = __reduce_min_sync(full, ns);
            const uint32_t len = ns - o;
            if (len >= s && len < best_len) {
                best_len = len;
                best = o;
            }
            o = ns;
        }
    };
    const bool first = c.policy == MP_FIT_FIRST;
    uint32_t carry = 0;  // largest end of the long obstacles so far
    bool found = false;
    uint32_t lane_best = 0, lane_len = 0xffffffffu;  // BEST: the best untouched gap this lane saw
    const unsigned near0 = __ballot_sync(full, p0.y != 0), near1 = __ballot_sync(full, p1.y != 0);
    for (int32_t k0 = 0; k0 < nlp && !found; k0 += 32) {
        const int32_t k = k0 + lane;
        bool hit = false;
        uint2 v = make_uint2(0, 0);
        if (k < nlp) {
            const uint32_t x = c.lg_af[k];
            hit = (x & 0xffffu) < f && (x >> 16) > a;
            if (hit) v = c.lg_oe[k];
        }
        if (!__any_sync(full, hit)) continue;
        // the largest end before each: that of the obstacle before it, as they
        // lie side by side unless two that never meet overlap in address
        const unsigned hm = __ballot_sync(full, hit), before = hm & ((1u << lane) - 1u);
        uint32_t prev = __shfl_sync(full, v.y, before ? 31 - __clz(before) : 0);
        prev = before ? umax2(prev, carry) : carry;
        if (__any_sync(full, hit && v.y < prev)) {
            const uint32_t incl = warp_incl_max(v.y);
            prev = __shfl_up_sync(full, incl, 1);
            prev = lane == 0 ? carry : umax2(prev, carry);
        }
        bool fits = hit && v.x >= prev && v.x - prev >= s;
        if (!first && !wide) {
            // most gaps meet no window tensor: those are compared as they
            // are, a lane each (looking into every one takes a warp reduction
            // or two per gap: 47.2 against 42.9 ms on a long tail of 20,000)
            bool touched = false;
            for (unsigned b = near0; b; b &= b - 1) {
                const int src = __ffs(b) - 1;
                touched |= (__shfl_sync(full, p0.x, src) < v.x) & (__shfl_sync(full, p0.y, src) > prev);
            }
            if (!kFar)
                for (unsigned b = near1; b; b &= b - 1) {
                    const int src = __ffs(b) - 1;
                    touched |= (__shfl_sync(full, p1.x, src) < v.x) & (__shfl_sync(full, p1.y, src) > prev);
                }
            if (fits && !touched) {
                if (v.x - prev < lane_len) {
                    lane_len = v.x - prev;
                    lane_best = prev;
                }
                fits = false;
            }
        }
        unsigned g = __ballot_sync(full, fits);
        while (g) {  // gaps between long obstacles that hold the tensor, ascending
            const int src = __ffs(g) - 1;
            g &= g - 1;
            const uint32_t g0 = __shfl_sync(full, prev, src), g1 = __shfl_sync(full, v.x, src);
            if (first) {
                best = settle(g0, g1);
                if (best + s <= g1) {
                    found = true;
                    break;
                }
            } else {
                holes(g0, g1);
            }
        }
        carry = umax2(carry, __reduce_max_sync(full, v.y));
    }
    if (!found) {
        if (first) {
            best = settle(carry, 0xffffffffu);
        } else {
            uint32_t top = 0;
            each([&](uint32_t, uint32_t pe) { top = umax2(top, pe); });
            top = umax2(__reduce_max_sync(full, top), carry);
            holes(carry, top);
            const uint32_t ln = __reduce_min_sync(full, lane_len);
            const uint32_t at = __reduce_min_sync(full, lane_len == ln ? lane_best : 0xffffffffu);
            if (ln < best_len || (ln == best_len && at < best)) {  // (both none: best is overwritten below)
                best_len = ln;
                best = at;
            }
            if (best_len == 0xffffffffu) best = top;
        }
    }
    if (lane == 0) c.oe[rc.pos] = make_uint2(best, best + s);
    __syncwarp();
    return best + s;
}

// The offset of a short tensor of s units whose placed predecessors (an
// obstacle per lane; (0, 0): none) and lg.top are all it meets, by one warp:
// FIRST jumps past whatever conflicts, BEST walks the holes.
__device__ __forceinline__ uint32_t fit_plain(uint2 v, uint32_t s, uint32_t base, int32_t policy) {
    const unsigned full = 0xffffffffu;
    uint32_t o = base;
    if (policy == MP_FIT_FIRST) {
        for (;;) {
            const uint32_t m = __reduce_max_sync(full, (v.x < o + s) & (o < v.y) ? v.y : 0u);
            if (m <= o) return o;
            o = m;
        }
    }
    const uint32_t top = umax2(o, __reduce_max_sync(full, v.y));
    uint32_t at = o, best_len = 0xffffffffu;
    o = top;
    while (at < top) {
        const uint32_t m = __reduce_max_sync(full, (v.x <= at) & (at < v.y) ? v.y : 0u);
        const uint32_t ns = __reduce_min_sync(full, v.x > at ? v.x : top);
        if (m > at) {
            at = m;
            continue;
        }
        if (ns - at >= s && ns - at < best_len) {
            best_len = ns - at;
            o = at;
        }
        at = ns;
    }
    return o;
}

// Walks the chain from rank r up to rank r1 with one warp, a window position
// per lane, when no gap between long tensors needs a look: everything goes
// above lg.top.  The next member's entries (which depend on no offset) are
// loaded while the current one is placed.  (Testing every possible start
// against all predecessors at once, without jumps, took a third longer: one
// warp is bound by the number of its dependent instructions.)
__device__ __forceinline__ uint32_t walk_plain(const Ctx<false>& c, int32_t r, int32_t r1, const Longs& lg) {
    const int lane = threadIdx.x & 31;
    uint32_t mx = 0;
    Rec rc = c.rec[r];
    Win w = c.win[r];
    uint32_t mask = c.mask[r];
    for (;;) {
        const int32_t rn = rc.next;
        const bool more = rn < r1;  // (kNone is past every rank)
        const Rec rc1 = c.rec[more ? rn : r];
        const Win w1 = c.win[more ? rn : r];
        const uint32_t mask1 = c.mask[more ? rn : r];
        if (w.wide) {
            mx = umax2(mx, place_short(c, r, lg));
        } else {
            const uint2 v = (mask >> lane) & 1u ? c.oe[w.w0 + lane] : make_uint2(0, 0);
            const uint32_t o = fit_plain(v, rc.s, lg.top, c.policy);
            if (lane == 0) c.oe[rc.pos] = make_uint2(o, o + rc.s);
            __syncwarp();
            mx = umax2(mx, o + rc.s);
        }
        if (!more) return mx;
        r = rn;
        rc = rc1;
        w = w1;
        mask = mask1;
    }
}

// Walks the run's long chains (of the components of sh.team[0, teams), their
// members among ranks [r0, r1)) with every warp of the CTA, no gap between long
// tensors needing a look: the warps are dealt out to the chains, take their
// chain's members in rank order in turn, each waits until its member's
// predecessors are placed (the offsets it needs are what it polls), and places
// it.  The lowest unplaced member's predecessors are placed and its warp has
// nothing earlier left to do, so every wait ends; it is bounded all the same: a
// warp that has polled kTeamPolls times counts the members that are placed, and
// leaves (sh.fail) if they are no more than when it last did.  (One member may
// keep the others waiting for some ms: one whose window is thousands of positions
// wide goes through it once for every level it is stacked above.)  A chain of
// equal sizes is deep but not a single path: 262 and 112 activations of a residual
// network, 172 K cycles by a warp each, 100 K this way.
__device__ __forceinline__ uint32_t walk_teams(const Ctx<false>& c, int32_t teams, int32_t r0, int32_t r1,
                                               const Longs& lg, Shared& sh) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const unsigned full = 0xffffffffu;
    const int32_t nwarps = (int32_t)(blockDim.x >> 5) / teams;  // per chain
    const int32_t mine = min(warp / nwarps, teams);             // (warps left over take none)
    int32_t n = 0, first = 0, end = 0;
    for (int32_t k = 0; k < teams; ++k) {
        const uint32_t comp = c.rec[sh.team[k]].comp;
        if (k == mine) first = n;
        for (int32_t b0 = r0; b0 < r1; b0 += (int32_t)blockDim.x) {
            const int32_t r = b0 + (int32_t)threadIdx.x;
            const uint32_t flag = r < r1 && c.rec[r].comp == comp && c.rec[r].prev != kIsLong ? 1u : 0u;
            uint32_t tot;
            const uint32_t at = (uint32_t)n + block_excl_sum(flag, sh.red, &tot);
            if (flag) c.list[at] = (uint16_t)r;
            n += (int32_t)tot;
        }
        if (k == mine) end = n;
    }
    __syncthreads();
    uint32_t mx = 0;
    volatile unsigned long long* oe = reinterpret_cast<volatile unsigned long long*>(c.oe);
    if (lane == 0) sh.seen[warp] = -1;
    __syncwarp();
    auto stuck = [&]() -> bool {  // (nothing of it is kept between calls: registers are short here)
        int32_t now = 0;
        for (int32_t x = first + lane; x < end; x += 32) now += oe[c.rec[c.list[x]].pos] != 0 ? 1 : 0;
        now = __reduce_add_sync(full, now);
        const bool out = __any_sync(full, now == *(volatile int32_t*)&sh.seen[warp] || *(volatile int32_t*)&sh.fail);
        *(volatile int32_t*)(out ? &sh.fail : &sh.seen[warp]) = out ? 1 : now;
        return out;
    };
    for (int32_t i = first + warp % nwarps; i < end; i += nwarps) {
        const int32_t r = c.list[i];
        const Rec rc = c.rec[r];
        const Win w = c.win[r];
        bool out = false;
        if (w.wide) {  // no mask of its predecessors: every earlier member's turn first
            for (int32_t x0 = first; x0 < i && !out; x0 += 32) {
                const bool pred = x0 + lane < i;
                const int32_t q = pred ? c.rec[c.list[x0 + lane]].pos : 0;
                for (int32_t polls = 0; !out && __any_sync(full, pred && oe[q] == 0); ++polls)
                    if (polls > kTeamPolls) {
                        out = stuck();
                        polls = 0;
                    }
            }
            if (out) break;
            if (test_held(sh, rc.pos)) continue;
            mx = umax2(mx, place_short(c, r, lg));
            continue;
        }
        const bool pred = (c.mask[r] >> lane) & 1u;
        const int32_t q = w.w0 + lane;
        unsigned long long v = 0;
        for (int32_t polls = 0;; ++polls) {
            if (pred) v = oe[q];
            if (!__any_sync(full, pred && v == 0)) break;
            if (polls > kTeamPolls) {
                out = stuck();
                if (out) break;
                polls = 0;
            }
        }
        if (out) break;
        if (test_held(sh, rc.pos)) continue;
        const uint32_t o = fit_plain(make_uint2((uint32_t)v, (uint32_t)(v >> 32)), rc.s, lg.top, c.policy);
        if (lane == 0) oe[rc.pos] = ((unsigned long long)(o + rc.s) << 32) | o;
        mx = umax2(mx, o + rc.s);
    }
    __syncthreads();
    return mx;
}

// Places the short tensors of ranks [r0, r1), every lower rank being placed:
// the first of each chain among them starts a walk up to rank r1.  With the
// long tensors' gaps listed (lg.ng >= 0: every tensor of the run meets all of
// them) a thread walks a chain of up to kThreadChain members, and a warp a
// longer one with a gap per lane; otherwise a warp walks every chain, a window
// position or a long tensor per lane.  (1,960 short tensors between 40 that
// span the trace, 16 warps: 164 K cycles by warps alone, 78 K with threads: a
// thread's walk costs about 20 times fewer issue slots.)  The caller puts a barrier after it.  Returns the largest
// end this thread or its warp placed.
template <bool kFar>
__device__ __forceinline__ uint32_t run_chains(const Ctx<kFar>& c, int32_t r0, int32_t r1, const Longs& lg, Shared& sh) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarps = blockDim.x >> 5;
    uint32_t mx = 0;
    auto is_head = [&](int32_t r) {
        const uint16_t p = c.rec[r].prev;
        return p == kNone || p < r0;
    };
    auto warp_walk = [&](int32_t r) {
        if constexpr (!kFar) {
            if (lg.ng == 0) {  // no long tensors' gaps to look at
                mx = umax2(mx, walk_plain(c, r, r1, lg));
                return;
            }
        }
        while (r < r1) {  // (kNone is past every rank)
            bool listed = false;
            if constexpr (!kFar) {
                listed = lg.ng >= 0 && !c.win[r].wide;
                if (listed) mx = umax2(mx, place_short_listed(c, r, lg));
            }
            if (!listed) mx = umax2(mx, place_short(c, r, lg));
            r = c.rec[r].next;
        }
    };
    if (r1 - r0 <= nwarps) {  // a warp per rank, no list
        const int32_t r = r0 + warp;
        if (r < r1 && is_head(r)) warp_walk(r);
        return mx;
    }
    for (int32_t b0 = r0; b0 < r1; b0 += kHeads) {
        __syncthreads();  // the previous list is done with
        if (threadIdx.x == 0) sh.cnt = sh.next = sh.cnt1 = sh.next1 = sh.teams = 0;
        __syncthreads();
        // chains for warps from the front of the list, for threads from its back
        const int32_t b1 = min(r1, b0 + kHeads);
        for (int32_t r = b0 + (int32_t)threadIdx.x; r < b1; r += (int32_t)blockDim.x) {
            if (!is_head(r)) continue;
            int32_t len = lg.ng >= 0 ? 0 : 2 * kTeamChain;  // members, if all have masks
            for (int32_t x = r; len < kTeamChain && x < r1; x = c.rec[x].next) len = c.win[x].wide ? 2 * kTeamChain : len + 1;
            if (len <= kThreadChain) {
                c.heads[kHeads - 1 - atomicAdd(&sh.cnt1, 1)] = (uint16_t)r;
            } else {
                int32_t k = kTeams;
                if constexpr (!kFar)
                    if (len == kTeamChain && lg.ng == 0) k = atomicAdd(&sh.teams, 1);
                if (k < kTeams) sh.team[k] = (uint16_t)r;
                else c.heads[atomicAdd(&sh.cnt, 1)] = (uint16_t)r;
            }
        }
        __syncthreads();
        if constexpr (!kFar) {
            const int32_t teams = min(sh.teams, kTeams);
            if (teams > 0 && !sh.fail) mx = umax2(mx, walk_teams(c, teams, r0, r1, lg, sh));
        }
        const int32_t nh = sh.cnt, nh1 = sh.cnt1;
        // half of the warps begin with the long chains, half with the others
        for (int32_t part = 0; part < 2; ++part) {
            const bool alone = (part == 0) == (warp >= (nwarps >> 1));
            for (;;) {
                int32_t i = 0;
                if (lane == 0) i = alone ? atomicAdd(&sh.next1, 32) : atomicAdd(&sh.next, 1);
                i = __shfl_sync(0xffffffffu, i, 0);
                if (i >= (alone ? nh1 : nh)) break;
                if (alone) {
                    if constexpr (!kFar) {
                        if (i + lane < nh1)
                            for (int32_t r = c.heads[kHeads - 1 - i - lane]; r < r1; r = c.rec[r].next)
                                mx = umax2(mx, place_short_alone(c, r, lg));
                    }
                    __syncwarp();
                } else {
                    warp_walk(c.heads[i]);
                }
            }
        }
    }
    return mx;
}

// Inserts m placed tensors, pend(i) being the position of the i-th, into the
// sorted list of len entries; ends with a barrier.
template <typename Pend>
__device__ __forceinline__ void insert_pending(const Ctx<false>& c, int32_t len, int32_t m, Pend&& pend, Shared& sh) {
    const int32_t t = (int32_t)threadIdx.x, nt = (int32_t)blockDim.x;
    for (int32_t done = 0; done < m; done += kBatch) {
        const int32_t mb = min(kBatch, m - done);
        for (int32_t i = t; i < mb; i += nt) {
            const uint32_t p = (uint32_t)pend(done + i);
            c.pk[i] = ((uint64_t)c.oe[p].x << 32) | p;
        }
        if (t < kFewPending) sh.before[t] = 0;
        __syncthreads();
        const int32_t chunk = (len + nt - 1) / nt;
        const int32_t i0 = min(len, t * chunk), cnt = min(len, i0 + chunk) - i0;
        uint32_t mv[kChunk];  // position | new index << 16
        if (mb <= kFewPending) {  // every entry against every new one
            uint32_t less[kFewPending];  // entries of this thread that stay before new tensor j
#pragma unroll
            for (int j = 0; j < kFewPending; ++j) less[j] = 0;
#pragma unroll
            for (int e = 0; e < kChunk; ++e) {
                if (e >= cnt) break;
                const uint32_t p = c.sl[i0 + e], o = c.oe[p].x;
                uint32_t up = 0;
#pragma unroll
                for (int j = 0; j < kFewPending; ++j) {
                    if (j >= mb) break;
                    const bool after = (uint32_t)(c.pk[j] >> 32) < o;
                    up += after ? 1u : 0u;
                    less[j] += after ? 0u : 1u;
                }
                mv[e] = p | ((uint32_t)(i0 + e) + up) << 16;
            }
#pragma unroll
            for (int j = 0; j < kFewPending; ++j) {
                if (j >= mb) break;
                const uint32_t w = __reduce_add_sync(0xffffffffu, less[j]);
                if ((t & 31) == 0 && w) atomicAdd(&sh.before[j], w);
            }
            __syncthreads();
            if (t < mb) {
                const uint64_t k = c.pk[t];
                uint32_t at = sh.before[t];
                for (int j = 0; j < mb; ++j) at += c.pk[j] < k ? 1u : 0u;
                c.sl[at] = (uint16_t)k;  // the keys' low half is the position
            }
        } else {
            // each new tensor's place among the entries (binary search) and
            // among the new ones: the warps sort 32 keys each, then every key
            // looks its place up in each of these runs
            const int32_t runs = (mb + 31) >> 5;
            uint64_t kx[kBatch / 256];
            uint32_t at[kBatch / 256], rk[kBatch / 256];
#pragma unroll
            for (int x = 0; x < kBatch / 256; ++x) {
                const int32_t i = t + x * nt;
                kx[x] = i < mb ? c.pk[i] : ~0ull;
                if ((i & ~31) < mb) {
                    kx[x] = warp_sort(kx[x]);
                    c.pk[i] = kx[x];  // (a run is read and written by one warp)
                }
            }
            __syncthreads();
#pragma unroll
            for (int x = 0; x < kBatch / 256; ++x) {
                const int32_t i = t + x * nt;
                if ((i & ~31) >= mb) break;
                const uint32_t o = (uint32_t)(kx[x] >> 32);
                int32_t lo = 0, hi = len;
                while (lo < hi) {
                    const int32_t mid = (lo + hi) >> 1;
                    if (c.oe[c.sl[mid]].x <= o) lo = mid + 1;
                    else hi = mid;
                }
                at[x] = (uint32_t)lo;
                uint32_t less = 0;
                for (int32_t w = 0; w < runs; ++w) {
                    const uint64_t* run = c.pk + 32 * w;
                    uint32_t l = 0;  // keys of the run below mine (0..32; the keys are distinct)
#pragma unroll
                    for (int step = 16; step > 0; step >>= 1) l += run[l + step - 1] < kx[x] ? step : 0;
                    l += run[l] < kx[x] ? 1 : 0;
                    less += l;
                }
                rk[x] = less;
            }
            __syncthreads();
#pragma unroll
            for (int x = 0; x < kBatch / 256; ++x) {
                if (kx[x] == ~0ull) continue;  // past the end
                c.pk[rk[x]] = ((uint64_t)at[x] << 32) | (uint32_t)(kx[x] & 0xffffu);  // by offset: (place, position)
            }
            __syncthreads();
            // an entry moves up by the number of new ones placed at or before it
            int32_t k = 0;
            {
                int32_t lo = 0, hi = mb;
                while (lo < hi) {
                    const int32_t mid = (lo + hi) >> 1;
                    if ((int32_t)(c.pk[mid] >> 32) <= i0) lo = mid + 1;
                    else hi = mid;
                }
                k = lo;
            }
#pragma unroll
            for (int e = 0; e < kChunk; ++e) {
                if (e >= cnt) break;
                while (k < mb && (int32_t)(c.pk[k] >> 32) <= i0 + e) ++k;
                mv[e] = (uint32_t)c.sl[i0 + e] | (uint32_t)(i0 + e + k) << 16;
            }
            __syncthreads();
            for (int32_t i = t; i < mb; i += nt) {
                const uint64_t v = c.pk[i];
                c.sl[(uint32_t)(v >> 32) + i] = (uint16_t)v;
            }
        }
#pragma unroll
        for (int e = 0; e < kChunk; ++e) {
            if (e >= cnt) break;
            c.sl[mv[e] >> 16] = (uint16_t)mv[e];
        }
        len += mb;
        __syncthreads();
    }
}

// Adds the long tensor x, placed at o, to the nlp placed long ones (at most
// kPer per thread), whose entries above it move up by one; ends with a barrier.
template <int kPer, bool kFar>
__device__ __forceinline__ void add_long(const Ctx<kFar>& c, const Rec& rc, uint32_t o, int32_t nlp) {
    const int32_t t = (int32_t)threadIdx.x, nt = (int32_t)blockDim.x;
    const uint32_t s = rc.s;
    uint2 v[kPer];
    uint32_t af[kPer];
#pragma unroll
    for (int x = 0; x < kPer; ++x) {
        const int32_t k = t + x * nt;
        if (k < nlp) {
            v[x] = c.lg_oe[k];
            af[x] = c.lg_af[k];
        }
    }
    // its own place: after the last entry at or below it
    bool mine = t == 0 && (nlp == 0 || v[0].x > o);
    int32_t here = 0;
#pragma unroll
    for (int x = 0; x < kPer; ++x) {
        const int32_t k = t + x * nt;
        if (k < nlp && v[x].x <= o && (k + 1 == nlp || c.lg_oe[k + 1].x > o)) {
            mine = true;
            here = k + 1;
        }
    }
    __syncthreads();
#pragma unroll
    for (int x = 0; x < kPer; ++x) {
        const int32_t k = t + x * nt;
        if (k < nlp && v[x].x > o) {
            c.lg_oe[k + 1] = v[x];
            c.lg_af[k + 1] = af[x];
        }
    }
    if (mine) {
        c.lg_oe[here] = make_uint2(o, o + s);
        c.lg_af[here] = (uint32_t)rc.a | ((uint32_t)rc.f << 16);
    }
    if (t == 0) c.oe[rc.pos] = make_uint2(o, o + s);
    __syncthreads();
}

// Places the long tensor of rank r with the whole CTA over the sorted list of
// len placed tensors, and adds it to the nlp placed long ones; ends with a
// barrier.  Returns its end.
__device__ __forceinline__ uint32_t place_long(const Ctx<false>& c, int32_t r, int32_t len, int32_t nlp, Shared& sh) {
    const int32_t t = (int32_t)threadIdx.x, nt = (int32_t)blockDim.x;
    const unsigned full = 0xffffffffu;
    const Rec rc = c.rec[r];
    const Win w = c.win[r];
    const uint32_t s = rc.s, a = rc.a;
    const int32_t core = w.core, w1 = w.w1;
    const bool first = c.policy == MP_FIT_FIRST;
    const int32_t chunk = (len + nt - 1) / nt;
    const int32_t i0 = min(len, t * chunk), cnt = min(len, i0 + chunk) - i0;
    if (t == 0) {
        sh.best32 = 0xffffffffu;
        sh.best = ~0ull;
    }
    uint32_t hits = 0, mx = 0;  // entries that overlap its lifetime; their largest end
    for (int32_t e = 0; e < cnt; ++e) {
        const int32_t p = c.sl[i0 + e];
        if (p < w1 && (p >= core || (c.af[p] >> 16) > a)) {
            hits |= 1u << e;
            mx = umax2(mx, c.oe[p].y);
        }
    }
    uint32_t top;
    uint32_t prev = block_excl_max(mx, sh.red, &top);  // (its barriers also cover sh.best)
    uint32_t gap = 0xffffffffu, at = 0xffffffffu;      // the best gap of this thread's entries
    for (uint32_t h = hits; h; h &= h - 1) {
        const uint2 v = c.oe[c.sl[i0 + __ffs(h) - 1]];
        if (v.x >= prev && v.x - prev >= s) {
            if (first) {
                at = prev;
                break;
            }
            if (v.x - prev < gap) {  // the lowest on ties: entries ascend
                gap = v.x - prev;
                at = prev;
            }
        }
        prev = umax2(prev, v.y);
    }
    if (first) {
        at = __reduce_min_sync(full, at);
        if ((t & 31) == 0 && at != 0xffffffffu) atomicMin(&sh.best32, at);
    } else {
        const uint32_t g = __reduce_min_sync(full, gap);
        at = __reduce_min_sync(full, gap == g ? at : 0xffffffffu);
        if ((t & 31) == 0 && g != 0xffffffffu) atomicMin(&sh.best, ((unsigned long long)g << 32) | at);
    }
    __syncthreads();
    uint32_t o;
    if (first) o = sh.best32 != 0xffffffffu ? sh.best32 : top;
    else o = sh.best != ~0ull ? (uint32_t)sh.best : top;
    add_long<(kMaxLong + 255) / 256>(c, rc, o, nlp);
    return o + s;
}

// Lists the gaps between the placed long tensors that hold the smallest tensor
// of the run [r0, r1) (ascending) in Ctx::pk with one warp; every thread gets
// the count (-1: more than kBatch) and the largest end.  Ends with a barrier.
__device__ __forceinline__ void list_long_gaps(const Ctx<false>& c, int32_t r0, int32_t r1, Longs& lg, Shared& sh) {
    const unsigned full = 0xffffffffu;
    const int lane = threadIdx.x & 31;
    if (threadIdx.x == 0) sh.best32 = 0xffffffffu;
    __syncthreads();
    uint32_t least = 0xffffffffu;
    for (int32_t r = r0 + (int32_t)threadIdx.x; r < r1; r += (int32_t)blockDim.x)
        least = c.rec[r].s < least ? c.rec[r].s : least;
    least = __reduce_min_sync(full, least);
    if (lane == 0) atomicMin(&sh.best32, least);
    __syncthreads();
    least = sh.best32;
    __syncthreads();
    if (threadIdx.x < 32) {
        uint32_t carry = 0;
        int32_t ng = 0;
        for (int32_t k0 = 0; k0 < lg.nlp; k0 += 32) {
            const uint2 v = k0 + lane < lg.nlp ? c.lg_oe[k0 + lane] : make_uint2(0, 0);
            const uint32_t incl = warp_incl_max(v.y);
            uint32_t prev = __shfl_up_sync(full, incl, 1);
            prev = lane == 0 ? carry : umax2(prev, carry);
            const bool gap = v.x > prev && v.x - prev >= least;
            const unsigned m = __ballot_sync(full, gap);
            const int32_t at = ng + __popc(m & ((1u << lane) - 1u));
            if (gap && at < kBatch) c.pk[at] = ((uint64_t)prev << 32) | (v.x - prev);
            ng += __popc(m);
            carry = umax2(carry, __shfl_sync(full, incl, 31));
        }
        if (lane == 0) {
            sh.cnt = ng <= kBatch ? ng : -1;
            sh.best32 = carry;
        }
    }
    __syncthreads();
    lg.ng = sh.cnt;
    lg.top = sh.best32;
    __syncthreads();
}

// Places g long tensors of ranks [r, r + g) that all share one lifetime: their
// obstacles differ only by each other, so the gaps of the first (at least as
// large as the smallest of them) are listed once, over the sorted list of len
// placed tensors as in place_long, and one warp hands them out in rank order,
// each tensor taking the bottom of its gap.  (40 tensors that span a trace of
// 2,000, in 4 groups: 280 K cycles one by one, 120 K in groups.)  Returns false, with nothing placed, if there are more
// than kBatch such gaps; ends with a barrier.
__device__ __forceinline__ bool place_group(const Ctx<false>& c, int32_t r, int32_t g, int32_t len, int32_t nlp, Shared& sh,
                                            uint32_t* end) {
    const int32_t t = (int32_t)threadIdx.x, nt = (int32_t)blockDim.x;
    const unsigned full = 0xffffffffu;
    const int lane = t & 31;
    const Win w = c.win[r];
    const uint32_t a = c.rec[r].a;
    const int32_t core = w.core, w1 = w.w1;
    const int32_t chunk = (len + nt - 1) / nt;
    const int32_t i0 = min(len, t * chunk), cnt = min(len, i0 + chunk) - i0;
    if (t == 0) sh.best32 = 0xffffffffu;
    uint32_t hits = 0, mx = 0;
    for (int32_t e = 0; e < cnt; ++e) {
        const int32_t p = c.sl[i0 + e];
        if (p < w1 && (p >= core || (c.af[p] >> 16) > a)) {
            hits |= 1u << e;
            mx = umax2(mx, c.oe[p].y);
        }
    }
    uint32_t top;
    const uint32_t before = block_excl_max(mx, sh.red, &top);
    for (int32_t i = t; i < g; i += nt) atomicMin(&sh.best32, c.rec[r + i].s);
    __syncthreads();
    const uint32_t least = sh.best32;
    uint32_t gaps = 0, prev = before;
    for (uint32_t h = hits; h; h &= h - 1) {
        const uint2 v = c.oe[c.sl[i0 + __ffs(h) - 1]];
        gaps += v.x >= prev && v.x - prev >= least ? 1u : 0u;
        prev = umax2(prev, v.y);
    }
    uint32_t ng;
    uint32_t at = block_excl_sum(gaps, sh.red, &ng);
    if (ng > (uint32_t)kBatch) return false;
    prev = before;
    for (uint32_t h = gaps ? hits : 0; h; h &= h - 1) {
        const uint2 v = c.oe[c.sl[i0 + __ffs(h) - 1]];
        if (v.x >= prev && v.x - prev >= least) c.pk[at++] = ((uint64_t)prev << 32) | (v.x - prev);
        prev = umax2(prev, v.y);
    }
    __syncthreads();
    if (t < 32) {
        const bool first = c.policy == MP_FIT_FIRST;
        uint32_t mxe = 0;
        for (int32_t i = 0; i < g; ++i) {
            const uint32_t s = c.rec[r + i].s;
            uint32_t best_len = 0xffffffffu, pick = 0xffffffffu;  // this lane's best gap (its index)
            for (int32_t k = lane; k < (int32_t)ng; k += 32) {
                const uint32_t ln = (uint32_t)c.pk[k];
                if (ln >= s && (first ? pick == 0xffffffffu : ln < best_len)) {
                    best_len = ln;
                    pick = (uint32_t)k;
                }
            }
            if (!first) {  // the smallest gap; the lowest (they ascend by index) on ties
                const uint32_t b = __reduce_min_sync(full, best_len);
                if (best_len != b) pick = 0xffffffffu;
            }
            pick = __reduce_min_sync(full, pick);
            uint32_t o = top;
            if (pick != 0xffffffffu) o = (uint32_t)(c.pk[pick] >> 32);
            else top += s;
            __syncwarp();
            if (lane == 0) {
                if (pick != 0xffffffffu) c.pk[pick] += ((uint64_t)s << 32) - s;  // start up, length down
                c.oe[c.rec[r + i].pos] = make_uint2(o, o + s);
            }
            mxe = umax2(mxe, o + s);
            __syncwarp();
        }
        if (lane == 0) sh.best32 = mxe;
    }
    __syncthreads();
    *end = sh.best32;
    // the placed long tensors by offset: an entry moves up by the new ones
    // below it, a new one goes behind the entries at or below it
    constexpr int kPer = (kMaxLong + 255) / 256;
    uint2 v[kPer];
    uint32_t af[kPer];
    int32_t to[kPer];
#pragma unroll
    for (int x = 0; x < kPer; ++x) {
        const int32_t k = t + x * nt;
        if (k >= nlp) continue;
        v[x] = c.lg_oe[k];
        af[x] = c.lg_af[k];
        to[x] = k;
        for (int32_t i = 0; i < g; ++i) to[x] += c.oe[c.rec[r + i].pos].x < v[x].x ? 1 : 0;
    }
    uint2 nv[kPer];
    int32_t nto[kPer];
#pragma unroll
    for (int x = 0; x < kPer; ++x) {
        const int32_t i = t + x * nt;
        if (i >= g) continue;
        nv[x] = c.oe[c.rec[r + i].pos];
        nto[x] = 0;
        for (int32_t k = 0; k < nlp; ++k) nto[x] += c.lg_oe[k].x <= nv[x].x ? 1 : 0;
        for (int32_t j = 0; j < g; ++j) {  // (they are live together: no two offsets are equal)
            nto[x] += c.oe[c.rec[r + j].pos].x < nv[x].x ? 1 : 0;
        }
    }
    __syncthreads();
#pragma unroll
    for (int x = 0; x < kPer; ++x) {
        if (t + x * nt < nlp) {
            c.lg_oe[to[x]] = v[x];
            c.lg_af[to[x]] = af[x];
        }
        if (t + x * nt < g) {
            const Rec& y = c.rec[r];
            c.lg_oe[nto[x]] = nv[x];
            c.lg_af[nto[x]] = (uint32_t)y.a | ((uint32_t)y.f << 16);
        }
    }
    __syncthreads();
    return true;
}

// Places every tensor of ranks [0, n): runs of short tensors between the long
// ones, whose ranks are lr[0, nl), ascending.  Returns the largest end this
// thread knows of.
__device__ __forceinline__ uint32_t place_all(const Ctx<false>& c, int32_t n, const uint16_t* lr, int32_t nl, Shared& sh) {
    uint32_t mx = 0;
    int32_t r0 = 0, len = 0, pending = 0;  // ranks [pending, r0) are placed but not in the sorted list
    Longs lg = {0, -1, 0, 0xffffffffu, 0};
    const uint32_t first_alloc = c.af[0] & 0xffffu;
    for (int32_t k = 0; k <= nl;) {
        const int32_t r1 = k < nl ? lr[k] : n;
        if (r1 > r0) {
            lg.ng = -1;
            if (r1 - r0 >= kListRun && lg.late <= first_alloc && lg.early >= sh.last_free)
                list_long_gaps(c, r0, r1, lg, sh);
            mx = umax2(mx, run_chains(c, r0, r1, lg, sh));
            __syncthreads();
        }
        if (k == nl) break;
        insert_pending(c, len, r1 - pending, [&](int32_t i) { return c.rec[pending + i].pos; }, sh);
        len += r1 - pending;
        pending = r1;
        // long tensors of consecutive ranks and one lifetime go together
        const Rec x = c.rec[r1];
        int32_t g = 1;
        while (k + g < nl && lr[k + g] == r1 + g && c.rec[r1 + g].a == x.a && c.rec[r1 + g].f == x.f) ++g;
        uint32_t end = 0;
        if (g == 1 || !place_group(c, r1, g, len, k, sh, &end)) {
            g = 1;
            end = place_long(c, r1, len, k, sh);
        }
        mx = umax2(mx, end);
        lg.late = umax2(lg.late, x.a);
        lg.early = lg.early < x.f ? lg.early : x.f;
        k += g;
        lg.nlp = k;
        r0 = r1 + g;
    }
    return mx;
}

// Outputs of a trace (b's slices of the batch outputs; null: not wanted).
struct Out {
    int64_t* offsets;    // of the trace
    int64_t* plan_peak;  // ... and the rest: one entry per trace
    int32_t* status;
    int64_t* profile;    // of the trace
    int64_t* peak_lb;
    int32_t* verdict;
    int32_t* conflict;   // a pair
    int32_t hold;        // test_team_hold of the trace
};

template <int E>
__device__ __forceinline__ void load_keys(uint64_t (&k)[E], const uint64_t* buf, int32_t n) {
#pragma unroll
    for (int e = 0; e < E; ++e) {
        const int32_t i = (int32_t)threadIdx.x * E + e;
        k[e] = i < n ? buf[i] : ~0ull;
    }
}

// Sorts the n keys (below ~0) at the start of the dynamic shared memory,
// ascending, in place.
static __device__ __noinline__ void sort_keys(int32_t n) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    uint64_t* buf = reinterpret_cast<uint64_t*>(smem_raw);
    const int32_t nt = (int32_t)blockDim.x;
    auto go = [&](auto e_const) {
        constexpr int E = decltype(e_const)::value;
        uint64_t k[E];
        load_keys<E>(k, buf, n);
        __syncthreads();
        block_sort<E>(k, buf);
#pragma unroll
        for (int e = 0; e < E; ++e) {
            const int32_t i = (int32_t)threadIdx.x * E + e;
            if (i < n) buf[i] = k[e];
        }
        __syncthreads();
    };
    if (n <= nt) go(std::integral_constant<int, 1>());
    else if (n <= 2 * nt) go(std::integral_constant<int, 2>());
    else if (n <= 4 * nt) go(std::integral_constant<int, 4>());
    else go(std::integral_constant<int, 8>());  // (kChunk)
}

// The whole trace by the whole CTA (256 or 512 threads): checks, profile (when
// out.profile is set), priority order (greedy_by_size, or greedy by breadth
// with kBreadth), placement, validation (kCheck) and outputs.  Returns false,
// with nothing written, when the trace is not one for this path: an invalid
// tensor, sizes summing to 2^32 units or more, too many long tensors, or a long
// chain beside some.  That is known before the sorts, so that a trace for the
// general path loses little here, and no thread touches the dynamic shared memory
// any more when another one returns.
template <bool kBreadth, bool kCheck>
__device__ __forceinline__ bool plan(const mp_batch& bt, const TraceView& tv, int32_t policy, const Out& out) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    unsigned char* smem = smem_raw;
    __shared__ Shared sh;
    const int32_t t = (int32_t)threadIdx.x, nt = (int32_t)blockDim.x, lane = t & 31, warp = t >> 5, nwarps = nt >> 5;
    const int32_t n = tv.n, T = tv.T;
    const Layout L(n, T, step_bytes<kBreadth>());
    uint2* OE = reinterpret_cast<uint2*>(smem + L.oe);
    uint64_t* KEY = reinterpret_cast<uint64_t*>(smem + L.oe);
    Rec* REC = reinterpret_cast<Rec*>(smem + L.rec);
    Win* WIN = reinterpret_cast<Win*>(smem + L.win);
    uint32_t* SZ = reinterpret_cast<uint32_t*>(smem + L.win);  // until the windows are written
    uint32_t* MASK = reinterpret_cast<uint32_t*>(smem + L.mask);
    uint32_t* AF = reinterpret_cast<uint32_t*>(smem + L.af);
    uint32_t* AF0 = SZ + n;  // by id, until the tensors are sorted by alloc step (with their sizes in KEY)
    uint16_t* ID = reinterpret_cast<uint16_t*>(smem + L.id);
    uint16_t* SL = reinterpret_cast<uint16_t*>(smem + L.sl);
    uint16_t* TMP = reinterpret_cast<uint16_t*>(smem + L.tmp);
    int32_t* BEND = reinterpret_cast<int32_t*>(smem + L.bend);
    const int32_t* __restrict__ Ag = bt.alloc_step + tv.lo;
    const int32_t* __restrict__ Fg = bt.free_step + tv.lo;
    const int64_t* __restrict__ Sg = bt.size_bytes + tv.lo;

    // ---- checks, size sum and unit, alloc-step histogram
    for (int32_t i = t; i < T; i += nt) BEND[i] = 0;
    if (t == 0) {
        sh.bad = sh.nl = 0;
        sh.lw = 1;
        sh.fail = 0;
        sh.hold = out.hold;
        sh.hi = sh.lo = sh.bits = 0;
        sh.lb = sh.far = sh.last_free = 0;
        sh.key = ~0ull;
    }
    __syncthreads();
    {
        bool bad = false;
        uint64_t sum = 0, bits = 0;
        int32_t longs = 0;
        for (int32_t k = t; k < n; k += nt) {
            const int32_t a = __ldg(Ag + k), f = __ldg(Fg + k);
            const int64_t s = __ldg(Sg + k);
            if (!tensor_ok(a, f, s, T)) {
                bad = true;
                continue;
            }
            longs += f - a > kLong ? 1 : 0;
            sum = sat_add(sum, (uint64_t)s);
            bits |= (uint64_t)s;
            KEY[k] = (uint64_t)s;
            AF0[k] = (uint32_t)a | ((uint32_t)f << 16);
            atomicAdd(BEND + a, 1);
        }
        block_add_size_sum(sum, &sh.hi, &sh.lo);
        const unsigned b0 = __reduce_or_sync(0xffffffffu, (unsigned)bits);
        const unsigned b1 = __reduce_or_sync(0xffffffffu, (unsigned)(bits >> 32));
        longs = __reduce_add_sync(0xffffffffu, longs);
        if (lane == 0) {
            atomicOr(&sh.bits, ((unsigned long long)b1 << 32) | b0);
            if (longs) atomicAdd(&sh.nl, longs);
        }
        if (bad) sh.bad = 1;
    }
    __syncthreads();
    const int32_t nl = sh.nl;
    if (sh.bad || n == 0 || size_sum_overflows(sh.hi, sh.lo) || nl > kMaxLong) return false;
    const int shift = __ffsll((long long)sh.bits) - 1;
    if ((((sh.hi << 32) + sh.lo) >> shift) > 0xffffffffull) return false;

    // ---- counting sort by alloc step, stable in the id: position = rank by
    // (alloc step, id)
    block_excl_scan_array<int32_t, 8>(BEND, T, reinterpret_cast<int32_t*>(sh.red));
    for (int32_t k = t; k < n; k += nt) TMP[atomicAdd(BEND + (AF0[k] & 0xffffu), 1)] = (uint16_t)k;
    constexpr bool kProfile = kCheck;
    const bool want_profile = kProfile && out.profile != nullptr;
    uint32_t* D = reinterpret_cast<uint32_t*>(smem + L.rec);             // profile differences, in units
    int64_t* BR = reinterpret_cast<int64_t*>(smem + L.rec);              // operators' breadths, in units
    if (want_profile)
        for (int32_t i = t; i < T; i += nt) D[i] = 0;
    if (kBreadth)
        for (int32_t i = t; i < T; i += nt) BR[i] = 0;
    __syncthreads();
    {
        int32_t lw = 1, last = 0;
        for (int32_t p = t; p < n; p += nt) {
            const int32_t k = TMP[p];
            const uint32_t af = AF0[k], s = (uint32_t)(KEY[k] >> shift);
            const int32_t a = (int32_t)(af & 0xffffu), f = (int32_t)(af >> 16);
            const int32_t lo = a ? BEND[a - 1] : 0, hi = BEND[a];
            int32_t q = lo;
            for (int32_t x = lo; x < hi; ++x) q += TMP[x] < k ? 1 : 0;
            ID[q] = (uint16_t)k;
            AF[q] = af;
            SZ[q] = s;
            if (f - a <= kLong) {
                lw = max(lw, f - a);
                last = max(last, f);
            }
            if (want_profile) {
                atomicAdd(D + a, s);
                if (f < T) atomicAdd(D + f, 0u - s);
            }
            if (kBreadth) {  // outputs of the operator at a, inputs of the one at f - 1
                atomic_add_u64_split(BR + a, s);
                if (f - 1 != a) atomic_add_u64_split(BR + (f - 1), s);
            }
        }
        lw = __reduce_max_sync(0xffffffffu, lw);
        last = __reduce_max_sync(0xffffffffu, last);
        if (lane == 0) {
            atomicMax(&sh.lw, lw);
            atomicMax(&sh.last_free, (uint32_t)last);
        }
    }
    __syncthreads();

    // ---- components of short lifetimes linked by overlap: one starts at a short
    // tensor allocated when every earlier short one is freed.  SL[q]: 1 + the first
    // position of q's component (0: q is long).
    {
        const int32_t chunk = (n + nt - 1) / nt, q0 = min(n, t * chunk), q1 = min(n, q0 + chunk);
        auto is_short = [](uint32_t af) { return (int32_t)(af >> 16) - (int32_t)(af & 0xffffu) <= kLong; };
        uint32_t live = 0;
        for (int32_t q = q0; q < q1; ++q)
            if (is_short(AF[q])) live = umax2(live, AF[q] >> 16);
        uint32_t tot;
        const uint32_t before = block_excl_max(live, sh.red, &tot);
        uint32_t run = before, start = 0;  // start: 1 + position of the last component start
        for (int32_t q = q0; q < q1; ++q) {
            const uint32_t af = AF[q];
            if (!is_short(af)) continue;
            if (run <= (af & 0xffffu)) start = (uint32_t)q + 1;
            run = umax2(run, af >> 16);
        }
        start = block_excl_max(start, sh.red, &tot);
        run = before;
        // the longest stretch of positions of one component bounds the work of
        // looking through it member by member
        uint32_t far = 0;
        for (int32_t q = q0; q < q1; ++q) {
            const uint32_t af = AF[q];
            SL[q] = 0;
            if (!is_short(af)) continue;
            if (run <= (af & 0xffffu)) start = (uint32_t)q + 1;
            run = umax2(run, af >> 16);
            SL[q] = (uint16_t)start;
            far = umax2(far, (uint32_t)q + 1 - start);
        }
        far = __reduce_max_sync(0xffffffffu, far);
        if (lane == 0 && far) atomicMax(&sh.far, far);
    }
    __syncthreads();
    if (nl > 0 && sh.far > kLongestChain) return false;

    // ---- live profile: prefix sums of the differences
    if (want_profile) {
        uint32_t carry = 0, mx = 0;
        const bool vec = (reinterpret_cast<uintptr_t>(out.profile) & 15) == 0;
        for (int32_t base = 0; base < T; base += nt * 4) {
            const int32_t i = base + 4 * t;
            uint4 d = make_uint4(0, 0, 0, 0);
            if (i + 4 <= T) {
                d = *reinterpret_cast<const uint4*>(D + i);
            } else {
                if (i < T) d.x = D[i];
                if (i + 1 < T) d.y = D[i + 1];
                if (i + 2 < T) d.z = D[i + 2];
            }
            d.y += d.x;
            d.z += d.y;
            d.w += d.z;
            uint32_t tot;
            const uint32_t pre = carry + block_excl_sum(d.w, sh.red, &tot);
            carry += tot;
            const uint32_t v[4] = {d.x + pre, d.y + pre, d.z + pre, d.w + pre};
            if (vec && i + 4 <= T) {
                longlong2* o = reinterpret_cast<longlong2*>(out.profile + i);
                o[0] = make_longlong2((int64_t)v[0] << shift, (int64_t)v[1] << shift);
                o[1] = make_longlong2((int64_t)v[2] << shift, (int64_t)v[3] << shift);
            }
#pragma unroll
            for (int x = 0; x < 4; ++x) {
                if (i + x >= T) break;
                mx = umax2(mx, v[x]);
                if (!vec || i + 4 > T) out.profile[i + x] = (int64_t)v[x] << shift;
            }
        }
        mx = __reduce_max_sync(0xffffffffu, mx);
        if (lane == 0) atomicMax(&sh.lb, mx);
    }

    // ---- priority order: size descending, alloc step, id (the position)
    for (int32_t p = t; p < n; p += nt) KEY[p] = ((uint64_t)(0xffffffffu - SZ[p]) << 32) | (uint32_t)p;
    __syncthreads();
    sort_keys(n);
    if (kBreadth) {  // the wider operator's breadth descending and its step (the earlier on ties) come first
        for (int32_t r = t; r < n; r += nt) {
            const uint32_t p = (uint32_t)KEY[r], af = AF[p], a = af & 0xffffu, z = (af >> 16) - 1;
            const uint64_t ba = (uint64_t)BR[a], bz = (uint64_t)BR[z];
            const uint64_t m = bz > ba ? bz : ba;  // below 2^33: a size counts twice at most
            const uint32_t st = bz > ba ? z : a;
            TMP[r] = (uint16_t)p;
            KEY[r] = (((1ull << 33) - 1 - m) << 31) | ((uint64_t)st << 15) | (uint32_t)r;
        }
        __syncthreads();
        sort_keys(n);
        for (int32_t r = t; r < n; r += nt) KEY[r] = TMP[KEY[r] & 0x7fffu];
        __syncthreads();
    }

    // ---- records by rank (over the per-step arrays), then the windows (over the sizes)
    for (int32_t r = t; r < n; r += nt) {
        const uint32_t p = (uint32_t)KEY[r], af = AF[p];
        Rec x;
        x.s = SZ[p];
        x.a = (uint16_t)af;
        x.f = (uint16_t)(af >> 16);
        x.pos = (uint16_t)p;
        x.next = kNone;
        x.prev = (int32_t)x.f - (int32_t)x.a > kLong ? kIsLong : kNone;
        x.many = 0;
        REC[r] = x;
        TMP[p] = (uint16_t)r;
    }
    __syncthreads();
    const int32_t lw = sh.lw;
    for (int32_t r = t; r < n; r += nt) {
        const Rec x = REC[r];
        Win w;
        w.w0 = (uint16_t)((int32_t)x.a >= lw ? BEND[(int32_t)x.a - lw] : 0);
        w.core = (uint16_t)(x.a ? BEND[x.a - 1] : 0);
        w.w1 = (uint16_t)BEND[x.f - 1];
        w.wide = w.w1 - w.w0 > 32 ? 1 : 0;
        WIN[r] = w;
        uint32_t mask = 0;
        if (!w.wide)
            for (int32_t q = w.w0; q < w.w1; ++q) {
                const int32_t qa = (int32_t)(AF[q] & 0xffffu), qf = (int32_t)(AF[q] >> 16);
                if (TMP[q] < r && qf - qa <= kLong && (q >= w.core || qf > x.a)) mask |= 1u << (q - w.w0);
            }
        MASK[r] = mask;
    }

    // ---- chains: the components, each in rank order
    for (int32_t q = t; q < n; q += nt) KEY[q] = SL[q] ? ((uint64_t)SL[q] << 16) | TMP[q] : kLongKey;
    __syncthreads();
    if (sh.far * (uint32_t)((n + nt - 1) / nt) < kScanChain) {  // each member looks for its neighbours in rank among the others
        for (int32_t q = t; q < n; q += nt) {
            const uint64_t k = KEY[q];
            if (k == kLongKey) continue;
            const uint32_t mine = (uint32_t)(k & 0xffffu);
            uint32_t up = kNone, dn = kNone;
            for (int32_t x = (int32_t)(k >> 16) - 1; x < n; ++x) {
                const uint64_t o = KEY[x];
                if (o == kLongKey) continue;
                if ((o >> 16) != (k >> 16)) break;
                const uint32_t r = (uint32_t)(o & 0xffffu);
                if (r > mine) up = r < up ? r : up;
                if (r < mine && (dn == kNone || r > dn)) dn = r;
            }
            REC[mine].next = (uint16_t)up;
            REC[mine].prev = (uint16_t)dn;
            REC[mine].comp = (uint16_t)(k >> 16);
        }
    } else {
        sort_keys(n);
        for (int32_t i = t; i < n; i += nt) {
            const uint64_t k = KEY[i];
            if (k == kLongKey) continue;
            const uint64_t up = i + 1 < n ? KEY[i + 1] : ~0ull, dn = i ? KEY[i - 1] : ~0ull;
            Rec& x = REC[k & 0xffffu];
            x.comp = (uint16_t)(k >> 16);
            if ((up >> 16) == (k >> 16)) x.next = (uint16_t)up;
            if ((dn >> 16) == (k >> 16)) x.prev = (uint16_t)dn;
        }
    }
    __syncthreads();
    // ---- ranks of the long tensors (the bucket ends are dead), offsets cleared
    uint16_t* LR = reinterpret_cast<uint16_t*>(smem + L.lr);
    for (int32_t r0 = 0, at0 = 0; r0 < n; r0 += nt) {
        const int32_t r = r0 + t;
        const uint32_t flag = r < n && REC[r].prev == kIsLong ? 1u : 0u;
        uint32_t tot;
        const uint32_t at = (uint32_t)at0 + block_excl_sum(flag, sh.red, &tot);
        if (flag) LR[at] = (uint16_t)r;
        at0 += (int32_t)tot;
    }
    for (int32_t p = t; p < n; p += nt) OE[p] = make_uint2(0, 0);
    __syncthreads();

    Ctx<false> c = {};
    c.oe = OE;
    c.af = AF;
    c.sl = SL;
    c.lg_oe = reinterpret_cast<uint2*>(smem + L.lg_oe);
    c.lg_af = reinterpret_cast<uint32_t*>(smem + L.lg_af);
    c.rec = REC;
    c.win = WIN;
    c.mask = MASK;
    c.pk = reinterpret_cast<uint64_t*>(smem + L.pk);
    c.heads = reinterpret_cast<uint16_t*>(smem + L.heads);
    c.list = TMP;
    c.policy = policy;
    uint32_t top = place_all(c, n, LR, nl, sh);

    // ---- outputs, and every lifetime-overlapping pair checked once, from its
    // earlier member in alloc order
    for (int32_t p = t; p < n; p += nt) out.offsets[ID[p]] = (int64_t)OE[p].x << shift;
    if (kCheck) {
        __syncthreads();
        if (t == 0) sh.cnt = 0;
        __syncthreads();
        // the pairs are tested without branches; a window with a conflict is
        // gone over again to report it
        auto clash = [&](uint2 v, int32_t q) {
            const uint2 u = OE[q];
            return (v.x < u.y) & (u.x < v.y);
        };
        auto report = [&](int32_t p, int32_t q) {
            const uint32_t i = ID[p], j = ID[q];
            atomicMin(&sh.key, ((unsigned long long)(i < j ? i : j) << 32) | (i < j ? j : i));
        };
        auto window = [&](int32_t p, int32_t q0, int32_t stop, int32_t step) {
            const uint2 v = OE[p];
            bool any = false;
#pragma unroll 4
            for (int32_t q = q0; q < stop; q += step) any |= clash(v, q);
            if (any)
                for (int32_t q = q0; q < stop; q += step)
                    if (clash(v, q)) report(p, q);
        };
        for (int32_t r = t; r < n; r += nt) {
            const int32_t p = REC[r].pos, stop = WIN[r].w1;
            if (stop - p - 1 > 64) TMP[atomicAdd(&sh.cnt, 1)] = (uint16_t)r;  // long windows: a warp each
            else window(p, p + 1, stop, 1);
        }
        __syncthreads();
        const int32_t nwide = sh.cnt;
        for (int32_t k = warp; k < nwide; k += nwarps) {
            const int32_t r = TMP[k], p = REC[r].pos;
            window(p, p + 1 + lane, WIN[r].w1, 32);
        }
    }
    top = __reduce_max_sync(0xffffffffu, top);
    if (t == 0) sh.best32 = 0;
    __syncthreads();
    if (lane == 0) atomicMax(&sh.best32, top);
    __syncthreads();
    if (t == 0) {
        *out.plan_peak = (int64_t)sh.best32 << shift;
        if (kCheck) {
            if (want_profile && out.peak_lb) *out.peak_lb = (int64_t)sh.lb << shift;
            const unsigned long long key = sh.key;
            const bool good = key == ~0ull;
            if (out.verdict) *out.verdict = good ? 1 : 0;
            if (out.conflict) {
                out.conflict[0] = good ? -1 : (int32_t)(key >> 32);
                out.conflict[1] = good ? -1 : (int32_t)(key & 0xffffffffu);
            }
        }
        *out.status = sh.fail ? MP_ETIMEOUT : MP_OK;
    }
    __syncthreads();
    return true;
}

}  // namespace phases
}  // namespace mp

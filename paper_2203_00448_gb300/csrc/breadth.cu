// breadth.cu -- greedy by breadth, the strategy of Pisarchyk et al. that
// Sec. 6 discusses: operators are taken by breadth (the sizes of their input
// and output tensors) descending, and each assigns offsets to its tensors not
// yet placed, largest first, by greedy_by_size's gap search.  A trace has one
// operator per step and no consumer lists, so the operator at step t is read
// as producing the tensors allocated at t and using for the last time the
// tensors freed at t + 1: its breadth is the bytes of both (a tensor of one
// step counts once), and a tensor is placed by the wider of its producer and
// its last user.  The order is therefore: that breadth descending, that
// operator's step (the earlier on ties), then size descending, alloc step
// ascending, id ascending.
//
// GPU form: one CTA per trace.  k_breadth_comp places every trace whose working
// set fits in shared memory by lifetime components (see its comment below): a
// thread, a warp or the whole CTA per component.  Of the traces it leaves (a
// component past kBBigComp tensors, or too large or too many for it)
//   - k_breadth_rest places short-lived tensors by chains and long-lived ones by
//     the whole CTA over a list sorted by offset (phases.cuh): 256 traces of 2,000
//     tensors take 0.32 ms instead of 38.5 ms;
//   - what that path does not take (sizes past 2^32 units, too many long-lived
//     tensors, traces past its limits) or is no gain for (comp_rule) is placed
//     tensor by tensor (breadth_trace), there or by k_breadth_tensor: the breadths
//     (two integer atomics per tensor, order-independent), each tensor's wider
//     operator, an in-place odd-even merge sort of the ids by that order, then for
//     each tensor all warps gather the placed tensors whose lifetimes overlap it (one
//     shared counter update per warp) and warp 0 runs the gap search with warp
//     reductions.
#include <algorithm>

#include "common.cuh"
#include "launch.h"
#include "phases.cuh"

namespace mp {

namespace {

constexpr int32_t kBDeferred = -2;  // status of a trace left by k_breadth_comp: in phases, or tensor by tensor
constexpr int32_t kBTensor = -3;    // ... tensor by tensor
__device__ __forceinline__ bool left_over(int32_t status) { return status == kBDeferred || status == kBTensor; }

// Per-trace working set: the breadth of the operator at each step; per tensor
// (by id) its operator's breadth and step, (alloc, free), size and offset; the priority order; the
// gathered predecessors' offsets and ends.
struct BreadthLayout {
    size_t prof, km, kt, ord, af, sz, off, pb, pe, total;
    __host__ __device__ BreadthLayout(int64_t n, int64_t T) {
        prof = 0;
        km = prof + align_up((size_t)T * 8);
        kt = km + align_up((size_t)n * 8);
        ord = kt + align_up((size_t)n * 4);
        af = ord + align_up((size_t)n * 4);
        sz = af + align_up((size_t)n * 8);
        off = sz + align_up((size_t)n * 8);
        pb = off + align_up((size_t)n * 8);
        pe = pb + align_up((size_t)n * 8);
        total = pe + align_up((size_t)n * 8);
    }
};

__device__ __forceinline__ int64_t warp_max_nonneg(int64_t v) {
    const unsigned hi = __reduce_max_sync(0xffffffffu, (unsigned)((uint64_t)v >> 32));
    const unsigned lo = __reduce_max_sync(0xffffffffu, (unsigned)((uint64_t)v >> 32) == hi ? (unsigned)v : 0u);
    return (int64_t)(((uint64_t)hi << 32) | lo);
}
__device__ __forceinline__ int64_t warp_min_nonneg(int64_t v) {
    const unsigned hi = __reduce_min_sync(0xffffffffu, (unsigned)((uint64_t)v >> 32));
    const unsigned lo = __reduce_min_sync(0xffffffffu, (unsigned)((uint64_t)v >> 32) == hi ? (unsigned)v : ~0u);
    return (int64_t)(((uint64_t)hi << 32) | lo);
}

// Gap search by one warp over P predecessors (pb / pe), each lane taking every
// 32nd: FIRST jumps to the largest end among the conflicting ones until none
// conflicts; BEST walks the free holes below the top and keeps the smallest
// that fits (the lowest on ties), else the top.  Every lane returns the offset.
__device__ int64_t warp_gap_search(int32_t policy, int64_t s, const int64_t* pb, const int64_t* pe, int32_t P) {
    const int lane = threadIdx.x & 31;
    int64_t o = 0;
    if (policy == MP_FIT_FIRST) {
        for (;;) {
            int64_t next = 0;
            for (int32_t k = lane; k < P; k += 32)
                if (pb[k] < o + s && o < pe[k] && pe[k] > next) next = pe[k];
            next = warp_max_nonneg(next);
            if (next <= o) return o;
            o = next;
        }
    }
    int64_t top = 0;
    for (int32_t k = lane; k < P; k += 32) top = pe[k] > top ? pe[k] : top;
    top = warp_max_nonneg(top);
    int64_t c = 0, best_len = INT64_MAX;
    o = top;
    while (c < top) {
        for (;;) {  // move c off any predecessor that covers it
            int64_t next = 0;
            for (int32_t k = lane; k < P; k += 32)
                if (pb[k] <= c && c < pe[k] && pe[k] > next) next = pe[k];
            next = warp_max_nonneg(next);
            if (next <= c) break;
            c = next;
        }
        if (c >= top) break;
        int64_t ns = INT64_MAX;
        for (int32_t k = lane; k < P; k += 32)
            if (pb[k] > c && pb[k] < ns) ns = pb[k];
        ns = warp_min_nonneg(ns);
        const int64_t len = ns - c;
        if (len >= s && len < best_len) {
            best_len = len;
            o = c;
        }
        c = ns;
    }
    return o;
}

// Odd-even merge sort (Batcher) of keys[0, n) in place by `before`, for any n
// (a comparator whose upper index falls past n would only meet padding that
// sorts last).  Every thread of the block must call it.
template <typename Before>
__device__ void block_sort_ids(int32_t* keys, int32_t n, Before&& before) {
    for (int32_t lp = 0; (1 << lp) < n; ++lp) {
        const int32_t p = 1 << lp;
        for (int32_t lk = lp; lk >= 0; --lk) {
            const int32_t k = 1 << lk, j0 = k == p ? 0 : k;
            const int32_t umax = ((n >> (lk + 1)) + 1) << lk;
            for (int32_t u = threadIdx.x; u < umax; u += blockDim.x) {
                const int32_t m = j0 + ((u >> lk) << (lk + 1)) + (u & (k - 1));
                if (m + k < n && (m >> (lp + 1)) == ((m + k) >> (lp + 1))) {
                    const int32_t x = keys[m], y = keys[m + k];
                    if (before(y, x)) {
                        keys[m] = y;
                        keys[m + k] = x;
                    }
                }
            }
            __syncthreads();
        }
    }
}

// Places trace b tensor by tensor with the whole CTA.
template <bool kSmem>
__device__ __forceinline__ void breadth_trace(const int b, const mp_batch& bt, int32_t policy,
                                              int64_t* __restrict__ offsets, int64_t* __restrict__ plan_peak,
                                              int32_t* __restrict__ status, unsigned char* __restrict__ ws,
                                              size_t ws_stride) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ int64_t red[72];
    __shared__ int32_t s_cnt, s_bad;
    __shared__ unsigned long long s_hi, s_lo;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const unsigned lt = (1u << lane) - 1u;
    const TraceView tv = load_trace(bt, b, false);
    if (tv.st != MP_OK) {
        if (threadIdx.x == 0) {
            status[b] = tv.st;
            plan_peak[b] = 0;
        }
        return;
    }
    const int32_t n = tv.n, T = tv.T;
    const BreadthLayout L(kSmem ? n : bt.max_tensors, kSmem ? T : bt.max_steps);
    unsigned char* base = kSmem ? smem_raw : ws + (size_t)b * ws_stride;
    int64_t* PROF = reinterpret_cast<int64_t*>(base + L.prof);
    int64_t* KM = reinterpret_cast<int64_t*>(base + L.km);
    int32_t* KT = reinterpret_cast<int32_t*>(base + L.kt);
    int32_t* ORD = reinterpret_cast<int32_t*>(base + L.ord);
    int2* AF = reinterpret_cast<int2*>(base + L.af);
    int64_t* SZ = reinterpret_cast<int64_t*>(base + L.sz);
    int64_t* OFF = reinterpret_cast<int64_t*>(base + L.off);
    int64_t* PB = reinterpret_cast<int64_t*>(base + L.pb);
    int64_t* PE = reinterpret_cast<int64_t*>(base + L.pe);

    for (int t = threadIdx.x; t < T; t += blockDim.x) PROF[t] = 0;
    if (threadIdx.x == 0) {
        s_bad = 0;
        s_hi = s_lo = 0;
    }
    __syncthreads();
    bool bad = false;
    uint64_t sum = 0;
    for (int k = threadIdx.x; k < n; k += blockDim.x) {
        const int32_t a = __ldg(bt.alloc_step + tv.lo + k), f = __ldg(bt.free_step + tv.lo + k);
        const int64_t s = __ldg(bt.size_bytes + tv.lo + k);
        if (!tensor_ok(a, f, s, T)) {
            bad = true;
            continue;
        }
        sum = sat_add(sum, (uint64_t)s);
        AF[k] = make_int2(a, f);
        SZ[k] = s;
        ORD[k] = k;
        // outputs of the operator at a, inputs of the operator at f - 1 (a
        // tensor counts for two operators at most: the sums stay below 2^64)
        atomic_add_u64_split(PROF + a, (uint64_t)s);
        if (f - 1 != a) atomic_add_u64_split(PROF + (f - 1), (uint64_t)s);
    }
    block_add_size_sum(sum, &s_hi, &s_lo);
    if (bad) s_bad = 1;
    __syncthreads();
    if (s_bad || size_sum_overflows(s_hi, s_lo)) {
        if (threadIdx.x == 0) {
            status[b] = s_bad ? MP_EINVAL : MP_EOVERFLOW;
            plan_peak[b] = 0;
        }
        return;
    }
    // PROF[t] (as uint64): the breadth of the operator at step t.  Each
    // tensor's operator: the wider of its producer and its last user, the
    // earlier one on ties
    const uint64_t* BR = reinterpret_cast<const uint64_t*>(PROF);
    for (int k = threadIdx.x; k < n; k += blockDim.x) {
        const int2 af = AF[k];
        uint64_t m = BR[af.x];
        int32_t tm = af.x;
        if (BR[af.y - 1] > m) {
            m = BR[af.y - 1];
            tm = af.y - 1;
        }
        KM[k] = (int64_t)m;
        KT[k] = tm;
    }
    __syncthreads();
    block_sort_ids(ORD, n, [&](int32_t x, int32_t y) {
        if (KM[x] != KM[y]) return (uint64_t)KM[x] > (uint64_t)KM[y];
        if (KT[x] != KT[y]) return KT[x] < KT[y];
        if (SZ[x] != SZ[y]) return SZ[x] > SZ[y];
        if (AF[x].x != AF[y].x) return AF[x].x < AF[y].x;
        return x < y;
    });

    // placement in that order
    for (int32_t r = 0; r < n; ++r) {
        if (threadIdx.x == 0) s_cnt = 0;
        __syncthreads();  // the previous offset is written, the counter reset
        const int32_t i = ORD[r];
        const int2 me = AF[i];
        for (int32_t x0 = warp * 32; x0 < r; x0 += blockDim.x) {
            const int32_t x = x0 + lane;
            bool ov = false;
            int32_t j = 0;
            if (x < r) {
                j = ORD[x];
                const int2 o = AF[j];
                ov = o.x < me.y && me.x < o.y;
            }
            const unsigned m = __ballot_sync(0xffffffffu, ov);
            if (m == 0) continue;
            const int leader = __ffs(m) - 1;
            int32_t at = 0;
            if (lane == leader) at = atomicAdd(&s_cnt, __popc(m));
            at = __shfl_sync(0xffffffffu, at, leader) + __popc(m & lt);
            if (ov) {
                PB[at] = OFF[j];
                PE[at] = OFF[j] + SZ[j];
            }
        }
        __syncthreads();  // the predecessors are gathered
        if (warp == 0) {
            const int64_t o = warp_gap_search(policy, SZ[i], PB, PE, s_cnt);
            if (lane == 0) OFF[i] = o;
        }
    }
    __syncthreads();
    int64_t mx = 0;
    for (int k = threadIdx.x; k < n; k += blockDim.x) {
        offsets[tv.lo + k] = OFF[k];
        mx = OFF[k] + SZ[k] > mx ? OFF[k] + SZ[k] : mx;
    }
    mx = block_max_i64(mx, red);
    if (threadIdx.x == 0) {
        plan_peak[b] = mx;
        status[b] = MP_OK;
    }
}

bool breadth_fits_smem(const mp_batch& bt) {
    return BreadthLayout(bt.max_tensors, bt.max_steps).total <= kSmemCeiling;
}

// ------------------------------------------------------------- components
// Lifetime components are independent under any placement order (a tensor's
// offset depends only on placed tensors whose lifetimes overlap its own), so
// traces are placed by k_breadth_comp: one CTA per trace counting-sorts the
// tensors by alloc step into records carrying their order keys, finds the
// components (a run starts where no earlier tensor is still live), and places
// each component in the breadth order -- one thread for up to kBThreadComp
// members, one warp (a member per lane) for up to kBWarpComp, the whole CTA
// beyond.  Traces with more than kBBigComps such large components, or one that is
// better placed in phases or too large for the CTA tier's scratch, and batches whose
// working set does not fit in shared memory, are left to the other kernels
// (status kBDeferred or kBTensor in between).

// Exclusive prefix maximum (identity 0) of one non-negative value per thread
// over the block; ends with a barrier.  red: >= 33 slots.
__device__ int32_t block_excl_max_i32(int32_t v, int32_t* red) {
    const int lane = threadIdx.x & 31, wp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    int32_t incl = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int32_t u = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl = max(incl, u);
    }
    if (lane == 31) red[wp] = incl;
    __syncthreads();
    if (wp == 0) {
        const int32_t x = lane < nw ? red[lane] : 0;
        int32_t xi = x;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int32_t u = __shfl_up_sync(0xffffffffu, xi, o);
            if (lane >= o) xi = max(xi, u);
        }
        const int32_t ex = __shfl_up_sync(0xffffffffu, xi, 1);
        if (lane < nw) red[lane] = lane == 0 ? 0 : ex;
    }
    __syncthreads();
    const int32_t up = __shfl_up_sync(0xffffffffu, incl, 1);
    const int32_t r = lane == 0 ? red[wp] : max(up, red[wp]);
    __syncthreads();
    return r;
}
constexpr int32_t kBThreadComp = 8;
constexpr int32_t kBWarpComp = 32;
constexpr int32_t kBBigComps = 64;  // components of more than kBWarpComp members a trace may have here
constexpr int32_t kBBigComp = 64;   // the most members of one, where the trace can be placed in phases ...
constexpr int32_t kBMidComp = 128;  // ... and where no trace of a very large batch has more tensors (comp_rule)
constexpr int32_t kBLongLife = 32;  // lives above this many steps are long

// Which traces with large components the component kernel leaves to the phases:
// those with one of more than `comp` members, or whose components it cannot place
// itself; but none that has `dense` or more short-lived tensors live at a step and
// no long-lived ones.
struct CompRule {
    int32_t comp, dense;
};

// A tensor in alloc-step order with the keys of the breadth order.
struct BRec {
    uint64_t m;    // breadth of its wider operator
    int64_t s;     // size
    int32_t a, f;  // lifetime [a, f)
    int32_t t;     // that operator's step
    int32_t id;    // tensor id in the trace
};

// x comes before y: breadth descending, operator step, size descending, alloc
// step, id.
__device__ __forceinline__ bool b_before(const BRec& x, const BRec& y) {
    if (x.m != y.m) return x.m > y.m;
    if (x.t != y.t) return x.t < y.t;
    if (x.s != y.s) return x.s > y.s;
    if (x.a != y.a) return x.a < y.a;
    return x.id < y.id;
}

struct BCompLayout {
    size_t br, bend, rec, off, rk, sb, lst, byr, total;
    __host__ __device__ BCompLayout(int64_t n, int64_t T) {
        br = 0;
        bend = br + align16b((size_t)T * 8);
        rec = bend + align16b((size_t)T * 4);
        off = rec + align16b((size_t)n * sizeof(BRec));
        rk = off + align16b((size_t)n * 8);
        sb = rk + align16b((size_t)n * 4);
        lst = sb + align16b((size_t)((n + 31) / 32) * 4);
        byr = lst + align16b((size_t)n * 4);
        total = byr + align16b((size_t)n);
    }
    __host__ __device__ static size_t align16b(size_t x) { return (x + 15) / 16 * 16; }
};

// The CTA tier's scratch (the per-step arrays, 12 bytes a step) holds a
// component of c members: its order and the gathered (offset, end) pairs.
__device__ __forceinline__ bool big_fits(int32_t c, int32_t T) {
    return BCompLayout::align16b((size_t)c * 4) + (size_t)c * 16 <=
           BCompLayout::align16b((size_t)T * 8) + BCompLayout::align16b((size_t)T * 4);
}

// One thread places a component of c <= kBThreadComp members at positions
// [p0, p0 + c), whose ranks in the breadth order and predecessor masks (the
// earlier-ranked members whose lifetimes overlap, as bits of the member
// index) were computed per member (RK[p] = mask << 8 | rank; BYR[p0 + r]: the
// member of rank r).  Each member in rank order: FIRST jumps to the largest
// conflicting end; BEST walks the free holes below the top in address order
// (the smallest that fits, the lowest on ties, else the top).
__device__ void place_comp_thread(const BRec* __restrict__ R, int64_t* __restrict__ OFF,
                                  const int32_t* __restrict__ RK, const uint8_t* __restrict__ BYR, int32_t p0,
                                  int32_t c, int32_t policy) {
    for (int32_t r = 0; r < c; ++r) {
        const int32_t i = BYR[p0 + r];
        const int64_t s = R[p0 + i].s;
        const uint32_t mask = (uint32_t)RK[p0 + i] >> 8;
        int64_t o = 0;
        if (mask != 0) {
            if (policy == MP_FIT_FIRST) {
                for (;;) {
                    int64_t nx = 0;
                    for (uint32_t m = mask; m; m &= m - 1) {
                        const int32_t j = p0 + __ffs(m) - 1;
                        const int64_t oj = OFF[j], ej = oj + R[j].s;
                        if (oj < o + s && o < ej && ej > nx) nx = ej;
                    }
                    if (nx <= o) break;
                    o = nx;
                }
            } else {
                int64_t top = 0;
                for (uint32_t m = mask; m; m &= m - 1) {
                    const int32_t j = p0 + __ffs(m) - 1;
                    top = max(top, OFF[j] + R[j].s);
                }
                int64_t cc = 0, best = -1, best_gap = 0;
                for (;;) {
                    for (;;) {  // move cc past every member that covers it
                        int64_t nx = cc;
                        for (uint32_t m = mask; m; m &= m - 1) {
                            const int32_t j = p0 + __ffs(m) - 1;
                            const int64_t oj = OFF[j], ej = oj + R[j].s;
                            if (oj <= cc && cc < ej) nx = max(nx, ej);
                        }
                        if (nx == cc) break;
                        cc = nx;
                    }
                    if (cc >= top) break;
                    int64_t ns = INT64_MAX;
                    for (uint32_t m = mask; m; m &= m - 1) {
                        const int32_t j = p0 + __ffs(m) - 1;
                        if (OFF[j] > cc) ns = min(ns, OFF[j]);
                    }
                    const int64_t gap = ns - cc;
                    if (gap >= s && (best < 0 || gap < best_gap)) {
                        best = cc;
                        best_gap = gap;
                    }
                    cc = ns;
                }
                o = best >= 0 ? best : top;
            }
        }
        OFF[p0 + i] = o;
    }
}

// One warp places a component of kBThreadComp < c <= kBWarpComp members, a
// member per lane: each lane counts the members before it, then the lanes
// place rank 0, 1, ... in turn with warp reductions over the earlier-ranked
// members that overlap the placed one (the same FIRST and BEST as above).
__device__ void place_comp_warp(const BRec* __restrict__ R, int64_t* __restrict__ OFF, int32_t p0, int32_t c,
                                int32_t policy) {
    const unsigned full = 0xffffffffu;
    const int lane = threadIdx.x & 31;
    const bool act = lane < c;
    BRec me{};
    if (act) me = R[p0 + lane];
    int32_t rank = 0;
    for (int32_t j = 0; j < c; ++j) {
        const BRec o = R[p0 + j];
        if (act && j != lane && b_before(o, me)) ++rank;
    }
    int64_t myoff = 0;
    for (int32_t r = 0; r < c; ++r) {
        const int L = __ffs(__ballot_sync(full, act && rank == r)) - 1;
        const int32_t La = __shfl_sync(full, me.a, L), Lf = __shfl_sync(full, me.f, L);
        const int64_t Ls = __shfl_sync(full, me.s, L);
        const bool pred = act && rank < r && me.a < Lf && La < me.f;
        const int64_t pe = myoff + me.s;
        int64_t o = 0;
        if (policy == MP_FIT_FIRST) {
            for (;;) {
                const int64_t nx = warp_max_nonneg(pred && myoff < o + Ls && o < pe ? pe : 0);
                if (nx <= o) break;
                o = nx;
            }
        } else {
            const int64_t top = warp_max_nonneg(pred ? pe : 0);
            int64_t cc = 0, best = -1, best_gap = 0;
            for (;;) {
                for (;;) {
                    const int64_t nx = warp_max_nonneg(pred && myoff <= cc && cc < pe ? pe : cc);
                    if (nx == cc) break;
                    cc = nx;
                }
                if (cc >= top) break;
                const int64_t ns = warp_min_nonneg(pred && myoff > cc ? myoff : INT64_MAX);
                const int64_t gap = ns - cc;
                if (gap >= Ls && (best < 0 || gap < best_gap)) {
                    best = cc;
                    best_gap = gap;
                }
                cc = ns;
            }
            o = best >= 0 ? best : top;
        }
        if (lane == L) myoff = o;
    }
    if (act) OFF[p0 + lane] = myoff;
}

__global__ void __launch_bounds__(kBreadthThreads)
k_breadth_comp(mp_batch bt, int32_t policy, int64_t* __restrict__ offsets, int64_t* __restrict__ plan_peak,
               int32_t* __restrict__ status, CompRule rule) {
    // once every CTA of this grid runs, those of k_breadth_rest may take what
    // room is left; they wait for this grid to finish
    asm volatile("griddepcontrol.launch_dependents;");
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ int64_t red[72];
    __shared__ int32_t s_bad, s_defer, s_nt, s_nw, s_nb, s_cnt, s_mid, s_lives, s_bin[kBThreadComp - 1], s_base[kBThreadComp];
    __shared__ int32_t s_mbase[kBThreadComp];    // the thread tier's members, by size class
    __shared__ uint32_t s_magic[kBThreadComp - 1];  // ceil(2^32 / c) of each size class
    __shared__ int32_t s_big[kBBigComps];
    __shared__ unsigned long long s_hi, s_lo;
    const int b = blockIdx.x;
    const int tid = threadIdx.x, nthr = blockDim.x, warp = tid >> 5, nwarps = nthr >> 5;
    const TraceView tv = load_trace(bt, b, false);
    if (tv.st != MP_OK) {
        if (tid == 0) {
            status[b] = tv.st;
            plan_peak[b] = 0;
        }
        return;
    }
    const int32_t n = tv.n, T = tv.T;
    const BCompLayout L(n, T);
    uint64_t* BR = reinterpret_cast<uint64_t*>(smem_raw + L.br);
    int32_t* BEND = reinterpret_cast<int32_t*>(smem_raw + L.bend);
    BRec* R = reinterpret_cast<BRec*>(smem_raw + L.rec);
    int64_t* OFF = reinterpret_cast<int64_t*>(smem_raw + L.off);
    int32_t* RK = reinterpret_cast<int32_t*>(smem_raw + L.rk);
    uint32_t* SB = reinterpret_cast<uint32_t*>(smem_raw + L.sb);
    int32_t* LST = reinterpret_cast<int32_t*>(smem_raw + L.lst);
    uint8_t* BYR = reinterpret_cast<uint8_t*>(smem_raw + L.byr);
    const int32_t* Ag = bt.alloc_step + tv.lo;
    const int32_t* Fg = bt.free_step + tv.lo;
    const int64_t* Sg = bt.size_bytes + tv.lo;
    const int32_t nwords = (n + 31) >> 5;
    for (int32_t t = tid; t < T; t += nthr) {
        BR[t] = 0;
        BEND[t] = 0;
    }
    for (int32_t w = tid; w < nwords; w += nthr) SB[w] = 0;
    if (tid == 0) {
        s_bad = s_defer = s_nt = s_nw = s_nb = s_mid = s_lives = 0;
        s_hi = s_lo = 0;
    }
    if (tid < kBThreadComp - 1) s_bin[tid] = 0;
    __syncthreads();
    // checks, operator breadths (as in breadth_trace) and the alloc-step histogram
    bool bad = false;
    uint64_t sum = 0;
    for (int32_t k = tid; k < n; k += nthr) {
        const int32_t a = __ldg(Ag + k), f = __ldg(Fg + k);
        const int64_t sz = __ldg(Sg + k);
        if (!tensor_ok(a, f, sz, T)) {
            bad = true;
            continue;
        }
        sum = sat_add(sum, (uint64_t)sz);
        atomic_add_u64_split(reinterpret_cast<int64_t*>(BR) + a, (uint64_t)sz);
        if (f - 1 != a) atomic_add_u64_split(reinterpret_cast<int64_t*>(BR) + (f - 1), (uint64_t)sz);
        atomicAdd(BEND + a, 1);
    }
    block_add_size_sum(sum, &s_hi, &s_lo);
    if (bad) s_bad = 1;
    __syncthreads();
    if (s_bad || size_sum_overflows(s_hi, s_lo)) {
        if (tid == 0) {
            status[b] = s_bad ? MP_EINVAL : MP_EOVERFLOW;
            plan_peak[b] = 0;
        }
        return;
    }
    block_excl_scan_array<int32_t, 8>(BEND, T, reinterpret_cast<int32_t*>(red));
    // records in alloc-step order, each with its wider operator (the earlier
    // one on ties)
    for (int32_t k = tid; k < n; k += nthr) {
        BRec r;
        r.a = __ldg(Ag + k);
        r.f = __ldg(Fg + k);
        r.s = __ldg(Sg + k);
        r.id = k;
        r.m = BR[r.a];
        r.t = r.a;
        if (BR[r.f - 1] > r.m) {
            r.m = BR[r.f - 1];
            r.t = r.f - 1;
        }
        R[atomicAdd(BEND + r.a, 1)] = r;
    }
    __syncthreads();
    // component starts: position p starts one when every earlier tensor is
    // freed by a_p (prefix maximum of the free steps over contiguous chunks)
    {
        const int32_t chunk = (n + nthr - 1) / nthr;
        const int32_t q0 = min(n, tid * chunk), q1 = min(n, q0 + chunk);
        int32_t local = 0;
        for (int32_t q = q0; q < q1; ++q) local = max(local, R[q].f);
        int32_t run = block_excl_max_i32(local, reinterpret_cast<int32_t*>(red));
        for (int32_t q = q0; q < q1; ++q) {
            if (q == 0 || run <= R[q].a) atomicOr(SB + (q >> 5), 1u << (q & 31));
            run = max(run, R[q].f);
        }
    }
    __syncthreads();
    // every component start finds its size: a single tensor sits at 0; the
    // components are counted by tier and size
    auto size_from = [&](int32_t p0) {  // distance from a start to the next one
        int32_t w = p0 >> 5;
        uint32_t m = SB[w] & ~((2u << (p0 & 31)) - 1u);
        while (m == 0 && ++w < nwords) m = SB[w];
        return (m ? (w << 5) + __ffs(m) - 1 : n) - p0;
    };
    for (int32_t p = tid; p < n; p += nthr) {
        if (!((SB[p >> 5] >> (p & 31)) & 1u)) continue;
        const int32_t c = size_from(p);
        if (c == 1) {
            OFF[p] = 0;
        } else if (c <= kBThreadComp) {
            atomicAdd(&s_bin[kBThreadComp - c], 1);
        } else if (c <= kBWarpComp) {
            LST[n - 1 - atomicAdd(&s_nw, 1)] = p * 64 + c;
        } else {  // the CTA tier, while its scratch holds the component
            const int32_t at = atomicAdd(&s_nb, 1);
            if (at < kBBigComps && big_fits(c, T)) s_big[at] = p;
            else s_defer = 1;
            if (c > rule.comp) s_mid = 1;
        }
    }
    __syncthreads();
    if (s_defer | s_mid) {  // (the same for every thread)
        int32_t lives = 0;
        bool any_long = false;
        for (int32_t k = tid; k < n; k += nthr) {
            const int32_t life = R[k].f - R[k].a;
            any_long |= life > kBLongLife;
            lives += life <= kBLongLife ? life : 0;
        }
        lives = __reduce_add_sync(0xffffffffu, lives);
        if ((tid & 31) == 0) atomicAdd(&s_lives, lives);
        const bool dense = !__syncthreads_or(any_long) && (int64_t)s_lives >= (int64_t)rule.dense * T;
        if (s_defer || !dense) {
            if (tid == 0) status[b] = dense ? kBTensor : kBDeferred;
            return;
        }
    }
    test_route(kRouteBreadthComp);
    if (tid == 0) {  // thread-tier components in descending size: bin starts, then cursors; member counts
        int32_t at = 0, mat = 0;
        for (int32_t k = 0; k < kBThreadComp - 1; ++k) {
            s_base[k] = at;
            s_mbase[k] = mat;
            s_magic[k] = 0xffffffffu / (uint32_t)(kBThreadComp - k) + 1u;
            at += s_bin[k];
            mat += s_bin[k] * (kBThreadComp - k);
            s_bin[k] = s_base[k];
        }
        s_nt = at;
        s_mbase[kBThreadComp - 1] = mat;
    }
    __syncthreads();
    for (int32_t p = tid; p < n; p += nthr) {
        if (!((SB[p >> 5] >> (p & 31)) & 1u)) continue;
        const int32_t c = size_from(p);
        if (c >= 2 && c <= kBThreadComp) LST[atomicAdd(&s_bin[kBThreadComp - c], 1)] = p * 64 + c;
    }
    __syncthreads();
    // members of the thread tier's components, one thread per member in the
    // size-sorted component list (so a warp's members mostly share one
    // component size): each gets its rank in the breadth order and the mask
    // of the earlier-ranked members that overlap its lifetime
    {
        int32_t mb[kBThreadComp];
#pragma unroll
        for (int k = 0; k < kBThreadComp; ++k) mb[k] = s_mbase[k];
        for (int32_t g = tid; g < mb[kBThreadComp - 1]; g += nthr) {
            int bin = 0;
            int32_t below = 0;  // members of the classes before bin
#pragma unroll
            for (int k = 1; k < kBThreadComp - 1; ++k) {
                if (g >= mb[k]) {
                    bin = k;
                    below = mb[k];
                }
            }
            const int32_t c = kBThreadComp - bin;
            const uint32_t r = (uint32_t)(g - below);
            const int32_t k = (int32_t)__umulhi(r, s_magic[bin]);  // r / c (r < 2^28)
            const int32_t p0 = LST[s_base[bin] + k] >> 6;
            const int32_t p = p0 + ((int32_t)r - k * c);
            const BRec me = R[p];
            uint32_t rank = 0, mask = 0;
            for (int32_t j = 0; j < c; ++j) {
                if (p0 + j == p) continue;
                const BRec o = R[p0 + j];
                if (b_before(o, me)) {
                    ++rank;
                    if (o.a < me.f && me.a < o.f) mask |= 1u << j;
                }
            }
            RK[p] = (int32_t)(mask << 8 | rank);
            BYR[p0 + rank] = (uint8_t)(p - p0);
        }
    }
    __syncthreads();
    for (int32_t i = warp; i < s_nw; i += nwarps) {
        const int32_t v = LST[n - 1 - i];
        place_comp_warp(R, OFF, v >> 6, v & 63, policy);
    }
    // the largest thread-tier components go to the last warp, which has the
    // fewest warp-tier components
    for (int32_t g = ((nwarps - 1 - warp) << 5) + (tid & 31); g < s_nt; g += nthr) {
        const int32_t v = LST[g];
        place_comp_thread(R, OFF, RK, BYR, v >> 6, v & 63, policy);
    }
    // components of more than kBWarpComp members: the whole CTA, one member at
    // a time in the breadth order (the per-step arrays, done with, are the
    // scratch: the order, then the gathered predecessors' offsets and ends)
    const int32_t nbig = min(s_nb, kBBigComps);
    for (int32_t k = 0; k < nbig; ++k) {
        __syncthreads();  // the previous component's scratch reads are done
        const int32_t p0 = s_big[k], c = size_from(p0);
        int32_t* ORDC = reinterpret_cast<int32_t*>(smem_raw + L.br);
        int64_t* PB = reinterpret_cast<int64_t*>(smem_raw + L.br + BCompLayout::align16b((size_t)c * 4));
        int64_t* PE = PB + c;
        for (int32_t i = tid; i < c; i += nthr) ORDC[i] = p0 + i;
        __syncthreads();
        block_sort_ids(ORDC, c, [&](int32_t x, int32_t y) { return b_before(R[x], R[y]); });
        const unsigned lt = (1u << (tid & 31)) - 1u;
        for (int32_t r = 0; r < c; ++r) {
            if (tid == 0) s_cnt = 0;
            __syncthreads();  // the previous member's offset is written, the counter reset
            const int32_t i = ORDC[r];
            const BRec me = R[i];
            for (int32_t x0 = warp * 32; x0 < r; x0 += nthr) {
                const int32_t x = x0 + (tid & 31);
                bool ov = false;
                int32_t j = 0;
                if (x < r) {
                    j = ORDC[x];
                    ov = R[j].a < me.f && me.a < R[j].f;
                }
                const unsigned m = __ballot_sync(0xffffffffu, ov);
                if (m == 0) continue;
                const int leader = __ffs(m) - 1;
                int32_t at = 0;
                if ((tid & 31) == leader) at = atomicAdd(&s_cnt, __popc(m));
                at = __shfl_sync(0xffffffffu, at, leader) + __popc(m & lt);
                if (ov) {
                    PB[at] = OFF[j];
                    PE[at] = OFF[j] + R[j].s;
                }
            }
            __syncthreads();  // the predecessors are gathered
            if (warp == 0) {
                const int64_t o = warp_gap_search(policy, me.s, PB, PE, s_cnt);
                if ((tid & 31) == 0) OFF[i] = o;
            }
        }
    }
    __syncthreads();
    int64_t mx = 0;
    for (int32_t p = tid; p < n; p += nthr) {
        const int64_t o = OFF[p];
        offsets[tv.lo + R[p].id] = o;
        mx = max(mx, o + R[p].s);
    }
    mx = block_max_i64(mx, red);
    if (tid == 0) {
        plan_peak[b] = mx;
        status[b] = MP_OK;
    }
}

// The traces k_breadth_comp deferred (or, with deferred_only false, all of
// them), in phases where they fit that path (phase_smem: the shared memory for
// it; 0: none does), else tensor by tensor (by_tensor; otherwise they are left
// deferred).  It waits for the kernel before it in the kernel.
template <bool kSmem>
__global__ void __launch_bounds__(kBreadthPhaseThreads, 1)
k_breadth_rest(mp_batch bt, int32_t policy, int64_t* __restrict__ offsets, int64_t* __restrict__ plan_peak,
               int32_t* __restrict__ status, unsigned char* __restrict__ ws, size_t ws_stride, bool deferred_only,
               uint32_t phase_smem, bool by_tensor) {
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;");
    // this CTA's traces are blockIdx.x + k * gridDim.x; their statuses are
    // read 32 at a time by one warp
    __shared__ unsigned s_todo;
    for (int64_t k0 = 0; blockIdx.x + k0 * gridDim.x < bt.n_traces; k0 += 32) {
        if (threadIdx.x < 32) {
            const int64_t b = blockIdx.x + (k0 + threadIdx.x) * gridDim.x;
            bool mine = b < bt.n_traces;
            if (mine && deferred_only) mine = by_tensor ? left_over(status[b]) : status[b] == kBDeferred;
            const unsigned m = __ballot_sync(0xffffffffu, mine);
            if (threadIdx.x == 0) s_todo = m;
        }
        __syncthreads();
        unsigned m = s_todo;
        __syncthreads();
        for (; m; m &= m - 1) {
            const int b = (int)(blockIdx.x + (k0 + __ffs(m) - 1) * gridDim.x);
            bool done = false;
            if (phase_smem > 0 && !(deferred_only && status[b] == kBTensor)) {
                const TraceView tv = load_trace(bt, b, false);
                if (tv.st == MP_OK && phases::fits<true>(tv.n, tv.T, phase_smem)) {
                    phases::Out o = {};
                    o.offsets = offsets + tv.lo;
                    o.plan_peak = plan_peak + b;
                    o.status = status + b;
                    o.hold = phases::test_team_hold(b);
                    done = phases::plan<true, false>(bt, tv, policy, o);
                    if (done) test_route(kRouteBreadthPhases);
                }
            }
            if (!done && by_tensor) test_route(kRouteBreadthTensor);
            if (!done && by_tensor) breadth_trace<kSmem>(b, bt, policy, offsets, plan_peak, status, ws, ws_stride);
            if (!done && !by_tensor && threadIdx.x == 0) status[b] = kBDeferred;  // left to the next launch
            __syncthreads();
        }
    }
}

// The traces k_breadth_comp and k_breadth_rest deferred (or all of them), tensor
// by tensor with small CTAs.
template <bool kSmem>
__global__ void __launch_bounds__(kBreadthThreads)
k_breadth_tensor(mp_batch bt, int32_t policy, int64_t* __restrict__ offsets, int64_t* __restrict__ plan_peak,
                 int32_t* __restrict__ status, unsigned char* __restrict__ ws, size_t ws_stride, bool deferred_only) {
    asm volatile("griddepcontrol.wait;" ::: "memory");
    __shared__ unsigned s_todo;  // as in k_breadth_rest
    for (int64_t k0 = 0; blockIdx.x + k0 * gridDim.x < bt.n_traces; k0 += 32) {
        if (threadIdx.x < 32) {
            const int64_t b = blockIdx.x + (k0 + threadIdx.x) * gridDim.x;
            const unsigned m = __ballot_sync(0xffffffffu, b < bt.n_traces && (!deferred_only || left_over(status[b])));
            if (threadIdx.x == 0) s_todo = m;
        }
        __syncthreads();
        unsigned m = s_todo;
        __syncthreads();
        for (; m; m &= m - 1) {
            const int b = (int)(blockIdx.x + (k0 + __ffs(m) - 1) * gridDim.x);
            test_route(kRouteBreadthTensor);
            breadth_trace<kSmem>(b, bt, policy, offsets, plan_peak, status, ws, ws_stride);
            __syncthreads();
        }
    }
}

bool breadth_comp_fits(const mp_batch& bt) {
    return BCompLayout(bt.max_tensors, bt.max_steps).total <= kSmemCeiling;
}

// Geometry of k_breadth_rest.
struct RestGeometry {
    size_t smem;
    int threads, resident;
};
template <bool kSmem>
cudaError_t rest_geometry(const mp_batch& bt, size_t phase_smem, bool by_tensor, int sms, RestGeometry* g) {
    g->smem = std::max(kSmem && by_tensor ? BreadthLayout(bt.max_tensors, bt.max_steps).total : 0, phase_smem);
    // more traces than SMs: half the threads, where an SM holds two of them
    g->threads = bt.n_traces > sms && g->smem <= kTwoPerSm ? kBreadthPhaseThreads / 2 : kBreadthPhaseThreads;
    const void* fn = (const void*)k_breadth_rest<kSmem>;
    const cudaError_t e = set_smem_limit(fn, g->smem);
    return e != cudaSuccess ? e : max_resident_ctas(fn, g->threads, g->smem, &g->resident);
}

// The component kernel places large components tensor by tensor with its 128
// threads, nine traces and more an SM, and k_breadth_tensor those it has no scratch
// for; the phases hold two.  While they hold the whole batch at once they are the
// faster ones (300 chains of 374 tensors 0.09 ms, 0.89 by components), except for
// very dense traces (300 of 1,000 tensors over 10 steps: 34.2 and 30.0 ms).  In
// larger batches they still are for chains (4,096: 1.00 and 1.94 ms), but not for
// traces with more than a few tensors live at a step (2,048 of 512 tensors over 100
// steps: 2.72 and 1.72 ms), nor, in very large ones, for traces little over the warp
// tier (4,096 chains of 94: 0.49 and 0.28 ms, best fit 0.55 and 0.41; 1,024:
// 0.14 and 0.13, 0.16 and 0.19).
CompRule comp_rule(const mp_batch& bt, int32_t policy, size_t phase_smem, int sms) {
    if (phase_smem == 0) return {INT32_MAX, 0};  // (what is left goes tensor by tensor either way)
    if (bt.n_traces <= (phase_smem <= kTwoPerSm ? 2 * sms : sms)) return {kBBigComp, 100};
    if (bt.max_tensors <= kBMidComp && bt.n_traces > (policy == MP_FIT_FIRST ? 6 : 12) * sms) return {kBMidComp, 0};
    return {kBBigComp, 8};
}

// A launch that waits in the kernel for the one before it in this call.
template <typename... Params, typename... Args>
cudaError_t launch_next(void (*kernel)(Params...), int grid, int threads, size_t smem, cudaStream_t stream, bool follows,
                        Args... args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)grid);
    cfg.blockDim = dim3((unsigned)threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = stream;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = follows ? 1 : 0;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kernel, args...);
}

constexpr int32_t kBApart = 1024;  // launch_rest
// Enough tensors a step for dense traces, as comp_rule has them.
bool crowded(const mp_batch& bt) { return 4 * (int64_t)bt.max_tensors >= 3 * (int64_t)bt.max_steps; }

// What k_breadth_comp leaves (comp; otherwise all traces).  Both ways in one launch
// where that holds the batch at once and what places tensor by tensor wants no
// shared memory that the phases do not leave it -- 256 traces of 2,000 tensors take
// 0.32 ms so, and 0.45 ms with the 160 KB that placing one of them tensor by tensor
// would need --, nor, with its data in the workspace, the L1 cache instead (40 chains
// and a trace of 5,000 tensors: 15.6 ms in one launch, 5.7 apart).  A batch
// that is more than one wave of its CTAs is placed tensor by tensor with small ones
// (1,000 traces of 1,500 tensors, none of them for the phases: 22.7 ms with the
// phases' registers, 18.2 so) where that may be for many of its traces or matters
// more than a launch: 1.6 us, 8% of the call for 500 traces of 60 tensors.
template <bool kSmem>
cudaError_t launch_rest(const mp_batch& bt, int32_t policy, int64_t* offsets, int64_t* plan_peak, int32_t* status,
                        void* workspace, bool comp, size_t phase_smem, int sms, cudaStream_t stream) {
    const size_t data = BreadthLayout(bt.max_tensors, bt.max_steps).total;
    unsigned char* ws = static_cast<unsigned char*>(workspace);
    bool deferred_only = comp;
    RestGeometry g;
    // (a CTA that an SM takes on while the phases still run there gets the little L1
    // cache that they leave, for as long as it runs: not where its data are in the
    // workspace)
    auto rest = [&](size_t phases_with, bool by_tensor) {
        return launch_next(k_breadth_rest<kSmem>, std::min(bt.n_traces, g.resident), g.threads, g.smem, stream,
                           deferred_only && (kSmem || phases_with > 0), bt, policy, offsets, plan_peak, status, ws,
                           data, deferred_only, (uint32_t)phases_with, by_tensor);
    };
    cudaError_t e = rest_geometry<kSmem>(bt, phase_smem, true, sms, &g);
    if (e != cudaSuccess) return e;
    if (phase_smem > 0) {
        const bool small_ctas = bt.n_traces > g.resident && (bt.max_tensors > kBApart || crowded(bt));
        if (!small_ctas && kSmem && data <= std::max(phase_smem, kTwoPerSm)) return rest(phase_smem, true);
        e = rest_geometry<kSmem>(bt, phase_smem, false, sms, &g);
        if (e == cudaSuccess) e = rest(phase_smem, false);
        deferred_only = true;
        if (e == cudaSuccess) e = rest_geometry<kSmem>(bt, 0, true, sms, &g);
        if (e != cudaSuccess) return e;
    }
    if (bt.n_traces <= g.resident) return rest(0, true);
    const size_t smem = kSmem ? data : 0;
    int resident = 0;
    e = set_smem_limit((const void*)k_breadth_tensor<kSmem>, smem);
    if (e == cudaSuccess)
        e = max_resident_ctas((const void*)k_breadth_tensor<kSmem>, kBreadthThreads, smem, &resident);
    if (e != cudaSuccess) return e;
    // (two waves of CTAs in a larger batch, so that the second evens the first out: a
    // whole CTA for every trace costs 1.5 us where 4,096 of them have nothing to do)
    const int64_t grid = std::min<int64_t>(bt.n_traces, bt.n_traces > 2 * sms ? 2 * (int64_t)resident : resident);
    return launch_next(k_breadth_tensor<kSmem>, (int)grid, kBreadthThreads, smem, stream,
                       deferred_only && kSmem, bt, policy, offsets, plan_peak, status, ws, data, deferred_only);
}

}  // namespace

size_t breadth_workspace_bytes(const mp_batch& bt) {
    if (bt.n_traces == 0 || breadth_fits_smem(bt)) return 0;
    return mul_sat((size_t)bt.n_traces, BreadthLayout(bt.max_tensors, bt.max_steps).total);
}

cudaError_t launch_breadth(const mp_batch& bt, int32_t policy, int64_t* offsets, int64_t* plan_peak, int32_t* status,
                           void* workspace, cudaStream_t stream) {
    if (bt.n_traces == 0) return cudaSuccess;
    const bool comp = breadth_comp_fits(bt);
    int sms = 0;
    cudaError_t e = sm_count(&sms);
    if (e != cudaSuccess) return e;
    const size_t phase_smem = phases::smem_bytes<true>(bt, sms);
    if (comp) {
        const size_t cbytes = BCompLayout(bt.max_tensors, bt.max_steps).total;
        e = set_smem_limit((const void*)k_breadth_comp, cbytes);
        if (e != cudaSuccess) return e;
        k_breadth_comp<<<(unsigned)bt.n_traces, kBreadthThreads, cbytes, stream>>>(bt, policy, offsets, plan_peak,
                                                                                  status,
                                                                                  comp_rule(bt, policy, phase_smem, sms));
        e = cudaGetLastError();
        if (e != cudaSuccess || bt.max_tensors <= kBWarpComp) return e;  // no component is too large for it
    }
    return breadth_fits_smem(bt)
               ? launch_rest<true>(bt, policy, offsets, plan_peak, status, workspace, comp, phase_smem, sms, stream)
               : launch_rest<false>(bt, policy, offsets, plan_peak, status, workspace, comp, phase_smem, sms, stream);
}

}  // namespace mp

#ifdef MP_TEST_HOOKS
// Test builds only: mp_plan_greedy_by_breadth, except that the member at
// alloc-order position hold_pos of trace hold_trace is never placed if a team
// of warps walks its chain, so that the team's bounded waits run out.
extern "C" __attribute__((visibility("default"))) mp_status mp_test_breadth_team_hold(
    const mp_batch* batch, mp_fit_policy policy, int64_t* offsets, int64_t* plan_peak, int32_t* trace_status,
    void* workspace, size_t workspace_bytes, int32_t hold_trace, int32_t hold_pos, void* stream) {
    if (batch == nullptr || workspace_bytes < mp::breadth_workspace_bytes(*batch)) return MP_EINVAL;
    const int32_t none[2] = {-1, -1}, held[2] = {hold_trace, hold_pos};
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    cudaError_t e = cudaMemcpyToSymbol(mp::phases::g_test_team_hold, held, sizeof(held));
    if (e == cudaSuccess) e = mp::launch_breadth(*batch, policy, offsets, plan_peak, trace_status, workspace, st);
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    const cudaError_t e2 = cudaMemcpyToSymbol(mp::phases::g_test_team_hold, none, sizeof(none));
    return e == cudaSuccess && e2 == cudaSuccess ? MP_OK : MP_ECUDA;
}
#endif

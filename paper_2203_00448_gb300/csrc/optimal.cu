// optimal.cu -- the exact optimum of Eq. 2.1 for traces of at most kOptMax
// tensors, by exhaustive search.  Every order of the tensors is considered,
// each tensor placed in turn at its lowest feasible offset among the lifetime-
// overlapping tensors placed before it, and the smallest resulting total_mem
// is the optimum: taking the tensors of any optimal packing by ascending
// offset, each lands at or below its optimal offset, so some order reaches
// the optimum.  Among equally good orders the first in lexicographic order
// gives the reported offsets.  It measures how far greedy_by_size (Sec. 2.3)
// is from optimal, the comparison of Sec. 3.2's strategy study.
//
// GPU form: branch and bound over the tree of orders, one CTA per trace.  The
// orders are cut by their first kOptDepth tensors; the warps take these
// prefixes in lexicographic order from a shared counter and walk the subtree
// of each depth first, also in lexicographic order, a tensor per lane: one
// pass over the placed tensors by ascending offset gives every remaining
// tensor's lowest feasible offset, and the unusable gaps at the step where
// each lane's tensor starts.  (With a thread per prefix the lanes of a warp
// stood at different nodes: 16.0 ms for the case below.)  Orders are left out
// only when they cannot be the answer:
//   - a tensor's lowest feasible offset never falls as more tensors are placed,
//     so a prefix is dropped once its peak, or the end any remaining tensor
//     would have if it were placed next, reaches the best total_mem so far
//     (that of greedy_by_size to begin with; ties stay while an earlier order
//     could still take them);
//   - the tensors live at one step end up side by side, so their sizes, and the
//     gaps between those placed that are too small for any of them still to be
//     placed, bound total_mem from below;
//   - two neighbours i, j of an order that do not overlap in lifetime can be
//     swapped without changing any offset, so an order in which such a pair
//     stands as (larger id, smaller id) has an equal, earlier one;
//   - the heaviest step's live bytes bound every plan from below: once an order
//     reaches them, no later one can win.
// A prefix dropped by its first tensors alone takes every later prefix that
// starts with them along.  4,096 traces of 9 tensors over 6 steps: placing all 9!
// orders took 184 ms, this search takes 1.8 ms, bound by the few traces with
// over 10,000 nodes.
//
// Bytes are counted in units of the largest power of two that divides every
// size of the trace: every offset is a sum of sizes, so nothing is rounded,
// and traces whose sizes then sum below 2^32 (all but the largest) use 32-bit
// words.
#include "common.cuh"
#include "launch.h"

namespace mp {

namespace {

constexpr int kOptMax = 10;
constexpr int kOptDepth = 3;  // tensors of a prefix: at most 720 subtrees of at most 7! orders a trace

// The workspace that the entry point asks its callers for: 16 bytes per
// kOptChunk orders of a trace.  The search itself needs none.
constexpr int64_t kOptChunk = 4096;

__host__ __device__ constexpr int64_t factorial(int n) { return n <= 1 ? 1 : n * factorial(n - 1); }

__device__ __forceinline__ int nib(uint64_t x, int k) { return (int)((x >> (4 * k)) & 15u); }

// Shared state of a trace: its tensors by id, and the best order so far.
struct OptShared {
    int64_t size[kOptMax];
    int32_t a[kOptMax], f[kOptMax];
    unsigned long long best;  // with 32-bit words total_mem << 32 | prefix, else total_mem
    unsigned long long sum_hi, sum_lo;
    unsigned long long bits;  // the sizes or-ed together
    unsigned int task, winner;
    int bad;
};

// One warp's search, lane j holding tensor j.  With 32-bit words the shared
// best holds the prefix too, so that prefixes after the best one's drop ties
// as well; with 64-bit words ties are settled at the end.
template <typename W>
struct Search {
    static constexpr bool kNarrow = sizeof(W) == 4;
    static constexpr unsigned kFull = 0xffffffffu;
    static constexpr W kNone = sizeof(W) == 4 ? (W)UINT32_MAX : (W)INT64_MAX;
    OptShared& sh;
    W (*fits)[32];  // by depth: the offset each remaining tensor had there
    const int lane, n;
    // this lane's tensor: size, ids that overlap it in lifetime, ids live when it starts and their bytes
    W size;
    uint32_t ov, live;
    W live_bytes;
    W lb;  // live bytes of the heaviest step
    // the prefix: ids placed, in order, by ascending offset; this lane's offset if placed
    uint32_t placed;
    uint64_t perm, by_off;
    W off;
    // lane d: state of depth d
    uint32_t left_d;
    W peak_d;
    uint64_t by_off_d;
    // the best order this warp found
    W v;
    uint32_t q_of_v;
    uint64_t perm_of_v;

    __device__ W all_max(W x) const {
        if constexpr (kNarrow) return __reduce_max_sync(kFull, x);
        return (W)warp_max_i64((int64_t)x);
    }
    __device__ void load(int shift) {
        size = lane < n ? (W)(sh.size[lane] >> shift) : (W)0;
        ov = live = 0;
        live_bytes = 0;
        for (int j = 0; j < n; ++j) {
            if (lane >= n) continue;
            if (j != lane && sh.a[lane] < sh.f[j] && sh.a[j] < sh.f[lane]) ov |= 1u << j;
            if (sh.a[j] <= sh.a[lane] && sh.a[lane] < sh.f[j]) {
                live |= 1u << j;
                live_bytes += (W)(sh.size[j] >> shift);
            }
        }
        lb = all_max(live_bytes);  // the heaviest step is one where some tensor starts
        reset();
        v = kNone;
        q_of_v = 0xffffffffu;
        perm_of_v = 0;
    }
    __device__ void reset() {
        placed = 0;
        perm = by_off = 0;
        off = 0;
    }
    // One pass over the placed tensors by ascending offset: fit is the lowest
    // feasible offset of this lane's tensor, bound a lower bound on the top of
    // the step where it starts.
    __device__ void pass(W& fit, W& bound) const {
        const uint32_t full = (1u << n) - 1u;
        W least = kNone;  // smallest tensor still to be placed among those live at this lane's step
        for (uint32_t t = full & ~placed; t; t &= t - 1) {
            const int k = __ffs(t) - 1;
            const W sk = __shfl_sync(kFull, size, k);
            if (((live >> k) & 1u) && sk < least) least = sk;
        }
        W o = 0, at = 0, lost = 0;
        bool done = false;
        const int np = __popc(placed);
        uint64_t list = by_off;
        for (int x = 0; x < np; ++x, list >>= 4) {
            const int k = (int)(list & 15u);
            const W ok = __shfl_sync(kFull, off, k), ek = ok + __shfl_sync(kFull, size, k);
            if ((ov >> k) & 1u) {
                done |= ok >= o + size;
                if (!done && ek > o) o = ek;
            }
            if ((live >> k) & 1u) {  // live at one step: side by side, ascending
                const W gap = ok - at;
                if (gap < least) lost += gap;
                at = ek;
            }
        }
        fit = o;
        bound = live_bytes + lost;
    }
    __device__ void place(int j, W o) {
        const bool below = ((placed >> lane) & 1u) && off <= o;
        const int at = 4 * __popc(__ballot_sync(kFull, below));
        const uint64_t low = by_off & ((1ull << at) - 1ull);
        by_off = low | ((uint64_t)j << at) | ((by_off ^ low) << 4);
        perm |= (uint64_t)j << (4 * __popc(placed));
        placed |= 1u << j;
        if (lane == j) off = o;
    }
    __device__ unsigned long long best() const { return *(volatile unsigned long long*)&sh.best; }
    // No order of prefix q with a total_mem of e or more can be the answer.
    __device__ bool hopeless(W e, uint32_t q, unsigned long long best) const {
        if constexpr (kNarrow) return (((unsigned long long)e << 32) | q) >= best;
        return e >= v || (unsigned long long)e > best;
    }
    // Whether the prefix leads nowhere; fit: this lane's lowest feasible offset.
    __device__ bool dead(uint32_t q, W& fit) const {
        W bound;
        pass(fit, bound);
        const unsigned long long b = __shfl_sync(kFull, best(), 0);
        const bool open = lane < n && !((placed >> lane) & 1u);
        return __any_sync(kFull, (lane < n && hopeless(bound, q, b)) || (open && hopeless((W)(fit + size), q, b)));
    }

    // The prefixes of q's block (of the given size) are done with.
    __device__ bool skip(uint32_t q, uint32_t block) {
        if (lane == 0) atomicMax(&sh.task, (q / block + 1) * block);
        return true;
    }

    // Walks the orders of prefix q; returns whether later prefixes matter.
    __device__ bool subtree(uint32_t q, int depth) {
        const uint32_t full = (1u << n) - 1u;
        reset();
        W peak = 0, fit;
        uint32_t rank = q;
        for (int d = 0; d < depth; ++d) {  // the prefix of that rank, placed
            uint32_t below = 1;            // ways to fill the prefix after position d
            for (int x = d + 1; x < depth; ++x) below *= (uint32_t)(n - x);
            uint32_t ids = full & ~placed;
            for (uint32_t x = rank / below; x > 0; --x) ids &= ids - 1;
            rank %= below;
            const int j = __ffs(ids) - 1;
            const int prev = d ? nib(perm, d - 1) : -1;
            // a prefix that leads nowhere takes all later ones with the same
            // first tensors with it
            if (prev > j && !((__shfl_sync(kFull, ov, j) >> prev) & 1u)) return skip(q, below);
            if (dead(q, fit)) return skip(q, below * (uint32_t)(n - d));
            const W o = __shfl_sync(kFull, fit, j), e = o + __shfl_sync(kFull, size, j);
            peak = e > peak ? e : peak;
            place(j, o);
        }
        int d = depth;
        bool fresh = true;  // the last tensor of the d placed ones was just placed
        for (;;) {
            if (fresh) {
                const unsigned long long b = __shfl_sync(kFull, best(), 0);
                // no order of this prefix or a later one can be the answer any more
                if (kNarrow ? b <= (((unsigned long long)lb << 32) | q) : v == lb) return false;
                const uint32_t rem = full & ~placed;
                uint32_t tries = 0;
                if (rem == 0) {
                    if (!hopeless(peak, q, b)) {  // a whole order, better than any before it
                        v = peak;
                        q_of_v = q;
                        perm_of_v = perm;
                        if (lane == 0)
                            atomicMin(&sh.best,
                                      kNarrow ? (((unsigned long long)peak << 32) | q) : (unsigned long long)peak);
                    }
                } else if (!dead(q, fit)) {
                    const int last = nib(perm, d - 1);
                    tries = __ballot_sync(kFull, ((rem >> lane) & 1u) && !(last > lane && !((ov >> last) & 1u)));
                    fits[d][lane] = fit;
                    __syncwarp();
                }
                if (lane == d) {
                    left_d = tries;
                    peak_d = peak;
                    by_off_d = by_off;
                }
            }
            fresh = false;
            const uint32_t tries = __shfl_sync(kFull, left_d, d);
            if (tries == 0) {  // back to the parent
                if (d == depth) return true;
                --d;
                placed &= ~(1u << nib(perm, d));
                perm &= ~(15ull << (4 * d));
                by_off = __shfl_sync(kFull, by_off_d, d);
                continue;
            }
            const int j = __ffs(tries) - 1;
            if (lane == d) left_d = tries & (tries - 1);
            const W o = fits[d][j], e = o + __shfl_sync(kFull, size, j), up = __shfl_sync(kFull, peak_d, d);
            const W p = e > up ? e : up;
            if (hopeless(p, q, __shfl_sync(kFull, best(), 0))) continue;
            place(j, o);
            peak = p;
            ++d;
            fresh = true;
        }
    }
};

// The search of one trace of n >= 1 valid tensors by the whole CTA; writes its
// offsets and returns its optimum (every thread).
template <typename W>
__device__ int64_t search_trace(OptShared& sh, W (*fits)[32], int n, int shift, int64_t* __restrict__ offsets) {
    const int lane = (int)(threadIdx.x & 31);
    constexpr unsigned kFull = 0xffffffffu;
    Search<W> s{sh, fits, lane, n};
    s.load(shift);
    if (threadIdx.x < 32) {  // greedy_by_size bounds the optimum from above
        int rank = 0;        // by size descending, alloc step, id
        for (int j = 0; j < n; ++j) {
            const W sj = __shfl_sync(kFull, s.size, j);
            if (lane < n && j != lane)
                rank += sj != s.size ? sj > s.size : sh.a[j] != sh.a[lane] ? sh.a[j] < sh.a[lane] : j < lane;
        }
        W peak = 0;
        for (int r = 0; r < n; ++r) {
            const int j = __ffs(__ballot_sync(kFull, lane < n && rank == r)) - 1;
            W fit, bound;
            s.pass(fit, bound);
            const W o = __shfl_sync(kFull, fit, j), e = o + __shfl_sync(kFull, s.size, j);
            peak = e > peak ? e : peak;
            s.place(j, o);
        }
        if (lane == 0)
            sh.best = sizeof(W) == 4 ? (((unsigned long long)peak << 32) | 0xffffffffull) : (unsigned long long)peak;
    }
    __syncthreads();
    const int depth = n < kOptDepth ? n : kOptDepth;
    uint32_t prefixes = 1;
    for (int x = 0; x < depth; ++x) prefixes *= (uint32_t)(n - x);
    for (;;) {
        uint32_t q = 0;
        if (lane == 0) q = atomicAdd(&sh.task, 1u);
        q = __shfl_sync(kFull, q, 0);
        if (q >= prefixes || !s.subtree(q, depth)) break;
    }
    __syncthreads();
    const unsigned long long best = sh.best;
    const W opt = (W)(sizeof(W) == 4 ? best >> 32 : best);
    if (lane == 0 && s.v == opt) atomicMin(&sh.winner, s.q_of_v);
    __syncthreads();
    if (s.v == opt && s.q_of_v == sh.winner) {  // one warp: a prefix is walked by one
        s.reset();
        for (int r = 0; r < n; ++r) {
            const int j = nib(s.perm_of_v, r);
            W fit, bound;
            s.pass(fit, bound);
            s.place(j, __shfl_sync(kFull, fit, j));
        }
        if (lane < n) offsets[lane] = (int64_t)s.off << shift;
    }
    return (int64_t)opt << shift;
}

template <int kThreads>
__global__ void __launch_bounds__(kThreads)
k_opt_search(mp_batch bt, int64_t* __restrict__ offsets, int64_t* __restrict__ opt_peak,
             int32_t* __restrict__ status) {
    __shared__ OptShared sh;
    __shared__ int64_t fits[kThreads / 32][kOptMax][32];  // (32-bit words use half of it)
    const int b = blockIdx.x;
    const int tid = (int)threadIdx.x;
    const TraceView tv = load_trace(bt, b, false);
    if (tv.st != MP_OK || tv.n > kOptMax) {
        if (tid == 0) {
            status[b] = MP_EINVAL;
            opt_peak[b] = 0;
        }
        return;
    }
    const int n = tv.n;
    if (tid == 0) {
        sh.bad = 0;
        sh.bits = sh.sum_hi = sh.sum_lo = 0;
        sh.task = 0;
        sh.winner = 0xffffffffu;
    }
    __syncthreads();
    if (tid < n) {
        const int32_t a = __ldg(bt.alloc_step + tv.lo + tid), f = __ldg(bt.free_step + tv.lo + tid);
        const int64_t s = __ldg(bt.size_bytes + tv.lo + tid);
        sh.a[tid] = a;
        sh.f[tid] = f;
        sh.size[tid] = s;
        if (!tensor_ok(a, f, s, tv.T)) {
            sh.bad = 1;
        } else {
            atomicAdd(&sh.sum_hi, (unsigned long long)s >> 32);
            atomicAdd(&sh.sum_lo, (unsigned long long)s & 0xffffffffull);
            atomicOr(&sh.bits, (unsigned long long)s);
        }
    }
    __syncthreads();
    const bool overflow = size_sum_overflows(sh.sum_hi, sh.sum_lo);
    if (sh.bad || overflow || n == 0) {
        if (tid == 0) {
            status[b] = sh.bad ? MP_EINVAL : overflow ? MP_EOVERFLOW : MP_OK;
            opt_peak[b] = 0;
        }
        return;
    }
    const int shift = __ffsll((long long)sh.bits) - 1;
    const unsigned long long units = ((sh.sum_hi << 32) + sh.sum_lo) >> shift;
    int64_t(*mine)[32] = fits[tid >> 5];
    const int64_t opt =
        units <= 0xffffffffull
            ? search_trace<uint32_t>(sh, reinterpret_cast<uint32_t(*)[32]>(mine), n, shift, offsets + tv.lo)
            : search_trace<int64_t>(sh, mine, n, shift, offsets + tv.lo);
    if (tid == 0) {
        opt_peak[b] = opt;
        status[b] = MP_OK;
    }
}

int32_t opt_chunks(const mp_batch& bt) {
    const int nmax = bt.max_tensors < kOptMax ? (bt.max_tensors > 0 ? bt.max_tensors : 1) : kOptMax;
    return (int32_t)((factorial(nmax) + kOptChunk - 1) / kOptChunk);
}

}  // namespace

size_t optimal_workspace_bytes(const mp_batch& bt) {
    if (bt.n_traces == 0) return 0;
    const size_t need = mul_sat(mul_sat((size_t)bt.n_traces, (size_t)opt_chunks(bt)), sizeof(longlong2));
    return need > SIZE_MAX - kAlign ? SIZE_MAX : align_up(need);
}

cudaError_t launch_optimal(const mp_batch& bt, int64_t* offsets, int64_t* opt_peak, int32_t* status,
                           cudaStream_t stream) {
    if (bt.n_traces == 0) return cudaSuccess;
    // The longer the traces, the longer the hardest of them holds the call up:
    // more warps shorten it, fewer leave room for more traces.  4,096 traces
    // with 128 / 256 / 512 threads: 6 tensors 85 / 124 / 226 us, 9 tensors 4.0 /
    // 2.3 / 1.8 ms; 1,000 of 8 tensors 272 / 158 / 170 us.
    const unsigned grid = (unsigned)bt.n_traces;
    if (bt.max_tensors <= 4) k_opt_search<64><<<grid, 64, 0, stream>>>(bt, offsets, opt_peak, status);
    else if (bt.max_tensors <= 6) k_opt_search<128><<<grid, 128, 0, stream>>>(bt, offsets, opt_peak, status);
    else if (bt.max_tensors <= 8) k_opt_search<256><<<grid, 256, 0, stream>>>(bt, offsets, opt_peak, status);
    else k_opt_search<512><<<grid, 512, 0, stream>>>(bt, offsets, opt_peak, status);
    return cudaGetLastError();
}

}  // namespace mp

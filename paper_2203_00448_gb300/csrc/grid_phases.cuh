// grid_phases.cuh -- one large trace per SM, placed in phases (phases.cuh), for
// the batches of a few large traces whose dependencies form a long chain.
//
// The dataflow over the whole GPU (grid.cu) pays two to three dependent trips
// to L2 for every hop of the chain of dependencies, and a long-lived tensor
// there gathers its predecessors from L2 and sorts them: about 30 us a hop, 867
// hops on a 20,000-tensor trace with 1,000 long-lived ones.  Placed in phases
// by one CTA, the offsets stay in that SM's shared memory, 8 bytes a tensor, so
// that the candidates of a long-lived tensor are one pass over a window there,
// and their gaps are found by buckets of addresses instead of a sort
// (place_far_long): about 12 us a hop with the run of short-lived ones before it.
// Everything that does not depend on an offset is prepared by the whole GPU
// first:
//
//   far_sort   stable alloc order (alloc step, then id) of every tensor;
//   far_comps  components of short lifetimes, a CTA per trace; with chains too
//              long for one SM the batch goes back to the dataflow;
//   far_rank   priority ranks, by counting (every pair of tensors once);
//   far_link   records by rank: windows, chain links, neighbour lists;
//   far_place  one CTA per trace.
//
// All but the last are stages of the cooperative launch that also runs the
// dataflow (k_grid_flow): as launches of their own they cost every batch that
// has no trace for them 30 us.
//
// A trace is placed in phases when its sizes sum below 2^32 units, it fits the
// shared memory, and one SM is likely to beat the dataflow (grid.cuh:
// chain_room, which k_grid_prep asks).
#pragma once

#include "grid.cuh"

namespace mp {
namespace grid {

using phases::kLong;
using phases::kNear;
using phases::kNone;

__device__ __forceinline__ void far_sort(const mp_batch& bt, const GridWs& w) {
    const int64_t slots = (int64_t)bt.n_traces * w.M;
    for (int64_t g = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; g < slots; g += (int64_t)gridDim.x * blockDim.x) {
        const int32_t b = (int32_t)(g / w.M), p = (int32_t)(g - (int64_t)b * w.M);
        const TraceInfo* ti = w.ti + b;
        if (!ti->ok || p >= ti->n) continue;
        const GRec r = w.rec[g];
        const int64_t base = (int64_t)b * w.M;
        const int32_t* bend = w.bend + (int64_t)b * w.TS;
        const int32_t lo = r.a ? bend[r.a - 1] : 0, hi = bend[r.a], id = w.rid[g];
        int32_t q = lo;
        for (int32_t x = lo; x < hi; ++x) q += w.rid[base + x] < id ? 1 : 0;
        w.p_af[base + q] = (uint32_t)r.a | ((uint32_t)r.f << 16);
        w.p_sz[base + q] = (uint32_t)(r.s >> ti->shift);
        w.p_at[base + q] = (uint16_t)p;
        w.p_rk[g] = 0;
    }
}

__device__ __forceinline__ void far_comps(const GridWs& w, int32_t b, uint32_t* red) {
    const int32_t n = w.ti[b].n, t = (int32_t)threadIdx.x, nt = (int32_t)blockDim.x;
    const int64_t base = (int64_t)b * w.M;
    const uint32_t* AF = w.p_af + base;
    const int32_t chunk = (n + nt - 1) / nt, q0 = min(n, t * chunk), q1 = min(n, q0 + chunk);
    auto life = [](uint32_t af) { return (int32_t)(af >> 16) - (int32_t)(af & 0xffffu); };
    uint32_t live = 0;
    for (int32_t q = q0; q < q1; ++q)
        if (life(AF[q]) <= kLong) live = max(live, AF[q] >> 16);
    uint32_t tot;
    const uint32_t before = phases::block_excl_max(live, red, &tot);
    uint32_t run = before, start = 0;
    for (int32_t q = q0; q < q1; ++q) {
        const uint32_t af = AF[q];
        if (life(af) > kLong) continue;
        if (run <= (af & 0xffffu)) start = (uint32_t)q + 1;
        run = max(run, af >> 16);
    }
    start = phases::block_excl_max(start, red, &tot);
    run = before;
    int32_t longest = 0;
    for (int32_t q = q0; q < q1; ++q) {
        const uint32_t af = AF[q];
        if (life(af) > kLong) {
            w.p_cs[base + q] = 0;
            continue;
        }
        if (run <= (af & 0xffffu)) start = (uint32_t)q + 1;
        run = max(run, af >> 16);
        w.p_cs[base + q] = start;
        longest = max(longest, q + 1 - (int32_t)start + 1);
    }
    if (__syncthreads_or(longest > w.ti[b].room) && t == 0) atomicAdd(&w.ctl->against, 1);
}

// Ranks by (size descending, position): every tensor against a slice of the
// others, the slices' counts added up.
constexpr int32_t kRankTile = 1024;
__device__ __forceinline__ void far_rank_tile(const GridWs& w, int32_t b, int32_t i0, int32_t j0, uint64_t* key) {
    const int32_t n = w.ti[b].n;
    const int64_t base = (int64_t)b * w.M;
    const int32_t nt = (int32_t)blockDim.x;
    constexpr int32_t kMine = kRankTile / kPrepareThreads;
    auto key_of = [&](int32_t p) { return ((uint64_t)(0xffffffffu - w.p_sz[base + p]) << 32) | (uint32_t)p; };
    __syncthreads();  // the previous tile's reads are done
    for (int32_t x = threadIdx.x; x < kRankTile; x += blockDim.x) key[x] = j0 + x < n ? key_of(j0 + x) : ~0ull;
    __syncthreads();
    uint64_t mine[kMine];
    uint32_t less[kMine];
#pragma unroll
    for (int e = 0; e < kMine; ++e) {
        const int32_t p = i0 + (int32_t)threadIdx.x + nt * e;
        mine[e] = p < n ? key_of(p) : 0;
        less[e] = 0;
    }
    const int32_t m = min(kRankTile, n - j0);
#pragma unroll 4
    for (int32_t x = 0; x < m; ++x) {
        const uint64_t k = key[x];
#pragma unroll
        for (int e = 0; e < kMine; ++e) less[e] += k < mine[e] ? 1u : 0u;
    }
#pragma unroll
    for (int e = 0; e < kMine; ++e) {
        const int32_t p = i0 + (int32_t)threadIdx.x + nt * e;
        if (p < n && less[e]) atomicAdd(w.p_rk + base + p, less[e]);
    }
}

__device__ __forceinline__ void far_link(const mp_batch& bt, const GridWs& w) {
    const int lane = threadIdx.x & 31;
    const unsigned lt = (1u << lane) - 1u, full = 0xffffffffu;
    const int64_t slots = (int64_t)bt.n_traces * w.M;
    const int64_t gw = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
    for (int64_t g = gw; g < slots; g += nw) {  // a warp per tensor
        const int32_t b = (int32_t)(g / w.M), p = (int32_t)(g - (int64_t)b * w.M);
        const TraceInfo* ti = w.ti + b;
        if (!ti->ok || p >= ti->n) continue;
        const int64_t base = (int64_t)b * w.M;
        const int32_t* bend = w.bend + (int64_t)b * w.TS;
        const uint32_t* AF = w.p_af + base;
        const uint32_t* RK = w.p_rk + base;
        const uint32_t* CS = w.p_cs + base;
        const uint32_t af = AF[p], rank = RK[p];
        const int32_t a = (int32_t)(af & 0xffffu), f = (int32_t)(af >> 16);
        phases::Win win;
        win.w0 = (uint16_t)(a >= ti->lw ? bend[a - ti->lw] : 0);
        win.core = (uint16_t)(a ? bend[a - 1] : 0);
        win.w1 = (uint16_t)bend[f - 1];
        win.wide = 0;
        phases::Rec rec;
        rec.s = w.p_sz[base + p];
        rec.a = (uint16_t)a;
        rec.f = (uint16_t)f;
        rec.pos = (uint16_t)p;
        rec.next = kNone;
        rec.prev = kNone;
        rec.many = 0;
        if (f - a > kLong) {
            rec.prev = phases::kIsLong;
            uint32_t below = 0;  // long-lived tensors that come before it
            for (int32_t k0 = 0; k0 < ti->nlong; k0 += 32) {
                const int32_t k = k0 + lane;
                bool first = false;
                if (k < ti->nlong) {  // (the list holds positions in rec, whose order inside a step differs)
                    const GRec o = w.rec[base + w.ll[base + k]];
                    const int32_t mine = w.rid[base + w.p_at[base + p]], theirs = w.rid[base + w.ll[base + k]];
                    const uint32_t os = (uint32_t)(o.s >> ti->shift);
                    first = os != rec.s ? os > rec.s : o.a != a ? o.a < a : theirs < mine;
                }
                below += __popc(__ballot_sync(full, first));
            }
            if (lane == 0) w.p_lr[(int64_t)b * kFarMaxLong + below] = (uint16_t)rank;
        } else {
            // its neighbours in rank inside its component
            const uint32_t cs = CS[p];
            uint32_t up = 0xffffffffu, dn = 0;  // dn: 1 + rank
            for (int32_t q0 = (int32_t)cs - 1;; q0 += 32) {
                const int32_t q = q0 + lane;
                const uint32_t c = q < ti->n ? CS[q] : 0xffffffffu;
                if (c == cs) {
                    const uint32_t r = RK[q];
                    if (r > rank) up = min(up, r);
                    if (r < rank) dn = max(dn, r + 1);
                }
                if (__any_sync(full, c != cs && c != 0)) break;  // past the component (0: long-lived ones between)
            }
            up = __reduce_min_sync(full, up);
            dn = __reduce_max_sync(full, dn);
            if (up != 0xffffffffu) rec.next = (uint16_t)up;
            if (dn) rec.prev = (uint16_t)(dn - 1);
            // the short-lived tensors it overlaps
            int32_t cnt = 0;
            uint16_t* near = w.p_near + (base + rank) * kNear;
            for (int32_t q0 = win.w0; q0 < win.w1; q0 += 32) {
                const int32_t q = q0 + lane;
                bool hit = false;
                if (q < win.w1 && q != p) {
                    const uint32_t o = AF[q];
                    const int32_t oa = (int32_t)(o & 0xffffu), of = (int32_t)(o >> 16);
                    hit = of - oa <= kLong && of > a && oa < f;
                }
                const unsigned m = __ballot_sync(full, hit);
                const int32_t at = cnt + __popc(m & lt);
                if (hit && at < kNear) near[at] = (uint16_t)q;
                cnt += __popc(m);
            }
            if (cnt > kNear) rec.many = 1;
            else if (lane >= cnt) near[lane] = kNone;
        }
        if (lane == 0) {
            w.p_rec[base + rank] = rec;
            w.p_win[base + rank] = win;
        }
    }
}

// Shared state of place_far_long.
struct FarShared {
    unsigned long long best;  // FIRST: the lowest start; BEST: (length << 32 | start)
    uint32_t resume, ns;
    int32_t warp_n[kFarThreads / 32];
    uint32_t high;
};

// Places the long-lived tensor rc with the whole CTA, nlp long ones
// being placed and no end being above `high`.  Its obstacles are the placed
// tensors of its window (a pass over their offsets, in position order) and the
// long ones that overlap it.  Their gaps are found without sorting them: the
// address space is cut into buckets, every obstacle leaves the least start and
// the largest end in the bucket it starts in, and a prefix maximum of the ends
// over the buckets gives, before each bucket's least start, the gap that ends
// there.  That is every gap of at least a bucket's length, since two starts of
// one bucket are closer; if the tensor is smaller, the buckets that can hold a
// gap between their own starts are looked at again the same way, cut into
// smaller buckets, until the tensor is as large as a bucket or a bucket is one
// address.  At most kSegments buckets at a time, ascending; the addresses of
// what is left then follow in another round.  Each level costs two passes over
// the obstacles and one over the buckets, whatever the offsets are.  Returns the
// offset (every thread); ends with a barrier.
__device__ __forceinline__ uint32_t place_far_long(const phases::Ctx<true>& c, const FarLayout& L, unsigned char* smem,
                                                   const phases::Rec& rc, const phases::Win& w, int32_t nlp,
                                                   uint32_t high, uint32_t* red, FarShared& fs) {
    const int32_t t = (int32_t)threadIdx.x, nt = kFarThreads;
    const int lane = t & 31, warp = t >> 5;
    const unsigned full = 0xffffffffu;
    uint32_t* MN = reinterpret_cast<uint32_t*>(smem + L.mn);
    uint32_t* MX = reinterpret_cast<uint32_t*>(smem + L.mx);
    uint32_t* FL = reinterpret_cast<uint32_t*>(smem + L.flags);
    uint32_t* FN = FL + kBuckets / 32;
    const uint32_t* EDGE = reinterpret_cast<const uint32_t*>(smem + L.edge);
    uint2* SEG = reinterpret_cast<uint2*>(smem + L.seg);  // (first address, largest end before it), two sets
    const uint32_t s = rc.s, a = rc.a, f = rc.f;
    const int32_t w0 = w.w0, core = w.core, w1 = w.w1;
    const bool first = c.policy == MP_FIT_FIRST;
    auto each = [&](auto&& fn) {  // fn(offset, end) for every obstacle, spread over the threads
        for (int32_t q = w0 + t; q < w1; q += nt) {
            const uint2 v = c.oe[q];
            if (v.y == 0) continue;
            if (q < core) {
                const int32_t i = q - w0;
                if (!(i < kEdges ? (EDGE[i >> 5] >> (i & 31)) & 1u : (c.af[q] >> 16) > a)) continue;
            }
            fn(v.x, v.y);
        }
        for (int32_t k = t; k < nlp; k += nt) {
            const uint32_t x = c.lg_af[k];
            if ((x & 0xffffu) < f && (x >> 16) > a) {
                const uint2 v = c.lg_oe[k];
                fn(v.x, v.y);
            }
        }
    };
    if (t == 0) fs.best = ~0ull;
    uint32_t top = 0, floor = 0;
    for (;;) {  // rounds: gaps between starts below `floor` are all found
        int32_t ns = 1, set = 0, sh1 = 0;
        int wb = 32 - __clz(high | 1u);  // a segment's addresses: [base, base + 2^wb)
        if (t == 0) {
            SEG[0] = make_uint2(0, 0);
            fs.resume = 0xffffffffu;
        }
        for (bool coarse = true;; coarse = false) {
            int sub = 31 - __clz(kBuckets / ns);  // log2 of the buckets per segment
            if (sub > wb) sub = wb;
            const int sh = wb - sub;
            const int32_t nb = ns << sub;
            if (coarse) sh1 = sh;
            const uint2* S = SEG + set * kSegments;
            // (every thread owns kPer buckets; those past nb stay empty)
#pragma unroll
            for (int v = 0; v < kPer / 4; ++v) {
                reinterpret_cast<uint4*>(MN)[t + v * nt] = make_uint4(~0u, ~0u, ~0u, ~0u);
                reinterpret_cast<uint4*>(MX)[t + v * nt] = make_uint4(0, 0, 0, 0);
            }
            __syncthreads();
            auto bucket = [&](uint32_t o) -> int32_t {  // -1: in no segment
                int32_t si = 0;
                if (!coarse) {
                    const uint32_t c1 = o >> sh1;  // most lie in no bucket that is looked at again
                    if (!((FL[c1 >> 5] >> (c1 & 31)) & 1u)) return -1;
                    int32_t lo = 0, hi = ns;  // the last segment that starts at or below o
                    while (lo < hi) {
                        const int32_t mid = (lo + hi) >> 1;
                        if (S[mid].x <= o) lo = mid + 1;
                        else hi = mid;
                    }
                    if (lo == 0) return -1;
                    si = lo - 1;
                    const uint32_t d = o - S[si].x;
                    if (wb < 32 && (d >> wb)) return -1;
                    return (si << sub) + (int32_t)(d >> sh);
                }
                return (int32_t)(o >> sh);
            };
            each([&](uint32_t o, uint32_t e) {
                const int32_t b = bucket(o);
                if (b < 0) return;
                // (many start in few buckets: most change nothing)
                if (o < *(volatile uint32_t*)(MN + b)) atomicMin(MN + b, o);
                if (e > *(volatile uint32_t*)(MX + b)) atomicMax(MX + b, e);
            });
            __syncthreads();
            // gaps that end at a bucket's least start; MX then holds the largest end before the bucket
            {
                const int32_t b0 = kPer * t;
                uint32_t m[kPer], e[kPer], seed[kPer];
#pragma unroll
                for (int v = 0; v < kPer / 4; ++v) {
                    const uint4 m4 = reinterpret_cast<const uint4*>(MN)[t * (kPer / 4) + v];
                    const uint4 e4 = reinterpret_cast<const uint4*>(MX)[t * (kPer / 4) + v];
                    m[4 * v] = m4.x, m[4 * v + 1] = m4.y, m[4 * v + 2] = m4.z, m[4 * v + 3] = m4.w;
                    e[4 * v] = e4.x, e[4 * v + 1] = e4.y, e[4 * v + 2] = e4.z, e[4 * v + 3] = e4.w;
                }
#pragma unroll
                for (int x = 0; x < kPer; ++x) seed[x] = b0 + x < nb ? S[(b0 + x) >> sub].y : 0u;
                uint32_t mx = 0;
#pragma unroll
                for (int x = 0; x < kPer; ++x) mx = max(mx, max(e[x], seed[x]));
                uint32_t tot;
                uint32_t prev = phases::block_excl_max(mx, red, &tot);
                if (coarse) top = tot;
                uint32_t at = 0xffffffffu, gap = 0xffffffffu, pv[kPer];
#pragma unroll
                for (int x = 0; x < kPer; ++x) {
                    prev = max(prev, seed[x]);
                    pv[x] = prev;
                    const bool fits = m[x] != 0xffffffffu && m[x] >= prev && m[x] - prev >= s;
                    if (fits && (first ? prev < at : m[x] - prev < gap)) {
                        gap = m[x] - prev;
                        at = prev;
                    }
                    prev = max(prev, e[x]);
                }
#pragma unroll
                for (int v = 0; v < kPer / 4; ++v)
                    reinterpret_cast<uint4*>(MX)[t * (kPer / 4) + v] =
                        make_uint4(pv[4 * v], pv[4 * v + 1], pv[4 * v + 2], pv[4 * v + 3]);
                if (first) {
                    at = __reduce_min_sync(full, at);
                    if (lane == 0 && at != 0xffffffffu) atomicMin(&fs.best, (unsigned long long)at);
                } else {
                    const uint32_t g = __reduce_min_sync(full, gap);
                    at = __reduce_min_sync(full, gap == g ? at : 0xffffffffu);
                    if (lane == 0 && g != 0xffffffffu) atomicMin(&fs.best, ((unsigned long long)g << 32) | at);
                }
            }
            if (sh == 0 || (sh < 32 && s >= (1u << sh))) break;  // no gap between two starts of one bucket holds it
            __syncthreads();
            // buckets that may hold one, as bits (FN); FL keeps the first level's
            if (t < kBuckets / 32) FN[t] = 0;
            __syncthreads();
            const uint32_t limit = first && fs.best != ~0ull ? (uint32_t)fs.best : 0xffffffffu;
            each([&](uint32_t o, uint32_t) {
                if (o < floor) return;
                const int32_t b = bucket(o);
                if (b < 0) return;
                const uint32_t prev = MX[b], m = MN[b];
                if (o >= s && o - s >= prev && o - s > m && prev < limit) {
                    if (!((*(volatile uint32_t*)(FN + (b >> 5)) >> (b & 31)) & 1u)) atomicOr(FN + (b >> 5), 1u << (b & 31));
                }
            });
            __syncthreads();
            // they become the next segments: kSegments of them, ascending
            int32_t mine = 0;
            if (t < kBuckets / 32) {
                mine = __popc(FN[t]);
                if (coarse) FL[t] = FN[t];
            }
            const int32_t incl = warp_incl_scan(mine);
            if (lane == 31) fs.warp_n[warp] = incl;
            __syncthreads();
            int32_t at = incl - mine, total = 0;
            for (int32_t x = 0; x < kBuckets / 1024; ++x) {
                if (x < warp) at += fs.warp_n[x];
                total += fs.warp_n[x];
            }
            uint2* N = SEG + (set ^ 1) * kSegments;
            if (t < kBuckets / 32)
                for (uint32_t fl = FN[t]; fl; fl &= fl - 1, ++at) {
                    const int32_t b = 32 * t + __ffs(fl) - 1;
                    const uint32_t base = S[b >> sub].x + ((uint32_t)(b & ((1 << sub) - 1)) << sh);
                    if (at < kSegments) N[at] = make_uint2(base, MX[b]);
                    else if (at == kSegments) fs.resume = min(fs.resume, base);
                }
            __syncthreads();
            if (total == 0) break;
            ns = min(total, kSegments);
            set ^= 1;
            wb = sh;
        }
        __syncthreads();
        const uint32_t resume = fs.resume;
        __syncthreads();
        if (resume == 0xffffffffu) break;
        floor = resume;
    }
    const unsigned long long best = fs.best;
    const uint32_t o = best == ~0ull ? top : (uint32_t)best;
    __syncthreads();
    phases::add_long<kMaxLongPerThread>(c, rc, o, nlp);
    return o;
}

// Places trace b (checked, in a batch placed in phases) with the whole CTA; smem: FarLayout bytes.
__device__ __forceinline__ void far_place(const GridWs& w, int32_t b, int32_t policy, unsigned char* smem_raw,
                                          phases::Shared& sh, FarShared& fs) {
    const TraceInfo* ti = w.ti + b;
    const int32_t n = ti->n, nl = ti->nlong, t = (int32_t)threadIdx.x, nt = (int32_t)blockDim.x;
    if (n == 0) return;  // an empty trace has no record to load ahead
    const int lane = t & 31, warp = t >> 5, nwarps = nt >> 5;
    const int64_t base = (int64_t)b * w.M;
    const FarLayout L(n, nl);
    const uint16_t* LR = w.p_lr + (int64_t)b * kFarMaxLong;
    phases::Ctx<true> c = {};
    c.oe = reinterpret_cast<uint2*>(smem_raw + L.oe);
    c.lg_oe = reinterpret_cast<uint2*>(smem_raw + L.lg_oe);
    c.lg_af = reinterpret_cast<uint32_t*>(smem_raw + L.lg_af);
    c.heads = reinterpret_cast<uint16_t*>(smem_raw + L.heads);
    uint32_t* edge = reinterpret_cast<uint32_t*>(smem_raw + L.edge);
    c.af = w.p_af + base;
    c.rec = w.p_rec + base;
    c.win = w.p_win + base;
    c.near = w.p_near + base * kNear;
    c.policy = policy;
    for (int32_t p = t; p < n; p += nt) c.oe[p] = make_uint2(0, 0);
    if (t == 0) fs.high = 0;
    __syncthreads();
    phases::Longs lg = {0, -1, 0, 0xffffffffu, 0};
    int32_t r0 = 0;
    uint32_t mx = 0;  // largest end this thread placed since it last added it to fs.high
    // the long tensor of this phase and the next, and the rank of the one after
    // that: loaded a phase ahead, as each is a trip to L2
    int32_t r1 = nl > 0 ? LR[0] : n, r2 = nl > 1 ? LR[1] : n;
    phases::Rec x = c.rec[min(r1, n - 1)];
    phases::Win xw = c.win[min(r1, n - 1)];
    for (int32_t k = 0; k <= nl; ++k) {
        const phases::Rec y = c.rec[min(r2, n - 1)];
        const phases::Win yw = c.win[min(r2, n - 1)];
        const int32_t r3 = k + 2 < nl ? LR[k + 2] : n;
        if (k < nl) {  // the overlap bits of the next long tensor, by warps that a short run leaves idle
            const uint32_t a = x.a;
            for (int32_t word = nwarps - 1 - warp; word < kEdges / 32 && xw.w0 + 32 * word < xw.core; word += nwarps) {
                const int32_t p = xw.w0 + 32 * word + lane;
                const unsigned bits = __ballot_sync(0xffffffffu, p < xw.core && (c.af[p] >> 16) > a);
                if (lane == 0) edge[word] = bits;
            }
        }
        lg.nlp = k;
        if (r1 > r0) mx = max(mx, phases::run_chains(c, r0, r1, lg, sh));
        if (k == nl) break;
        mx = __reduce_max_sync(0xffffffffu, mx);
        if (lane == 0 && mx) atomicMax(&fs.high, mx);
        mx = 0;
        __syncthreads();
        const uint32_t o = place_far_long(c, L, smem_raw, x, xw, k, fs.high, sh.red, fs);
        if (t == 0) mx = o + x.s;
        r0 = r1 + 1;
        r1 = r2;
        r2 = r3;
        x = y;
        xw = yw;
    }
    __syncthreads();
    const int shift = ti->shift;
    for (int32_t p = t; p < n; p += nt) w.off[base + w.p_at[base + p]] = (int64_t)c.oe[p].x << shift;
}

// Everything before far_place, by the whole cooperative grid: `sync` is a
// barrier over it, false when its bounded wait ran out.  Returns false if the
// batch's chains leave it to the dataflow after all (some 20 us for a trace of
// 2,000 tensors, 40 for 20,000).
template <typename Sync>
__device__ __forceinline__ bool far_prepare(const mp_batch& bt, const GridWs& w, unsigned char* smem, int64_t* red,
                                            Sync&& sync) {
    far_sort(bt, w);
    if (!sync()) return true;
    int32_t item = 0;
    for (int32_t b = 0; b < bt.n_traces; ++b) {
        if (!w.ti[b].ok) continue;
        const int32_t n = w.ti[b].n;
        if (item++ % (int32_t)gridDim.x == (int32_t)blockIdx.x) far_comps(w, b, reinterpret_cast<uint32_t*>(red));
        for (int32_t i0 = 0; i0 < n; i0 += kRankTile)
            for (int32_t j0 = 0; j0 < n; j0 += kRankTile, ++item)
                if (item % (int32_t)gridDim.x == (int32_t)blockIdx.x)
                    far_rank_tile(w, b, i0, j0, reinterpret_cast<uint64_t*>(smem));
    }
    if (!sync()) return true;
    if (!in_phases(w.ctl)) return false;
    far_link(bt, w);
    return true;
}

}  // namespace grid
}  // namespace mp

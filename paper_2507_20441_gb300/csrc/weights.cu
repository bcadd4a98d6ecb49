// Weight pass of TIMEST (Sec. 3.1): windows (Constraint 3, Alg. 1), the
// per-edge dynamic program over the rooted spanning tree (Claims 3.1-3.2,
// Alg. 2), segmented prefix sums of child weights, and the root CDF whose
// window totals give W (Claim 3.4).
//
// Windows [i*delta, (i+2)*delta) with the same parity of i are disjoint, so
// each edge has at most one window per parity ("layer" p = i mod 2) and one
// weight per (tree edge, layer).  The weight of tree node q for edge e in
// layer p is the product over q's children c of
//     sum of w_c over Lambda_z(time range of c) - sum over El(z, o)(same range)
// (the candidate list of Claim 3.1), where both ranges are clipped to e's
// window and the sums are differences of segmented prefix sums.
#include <cuda_runtime.h>
#include <stdint.h>
#include <string.h>

#include <algorithm>
#include <vector>

#include "scan.cuh"
#include "tm_device.cuh"
#include "tm_internal.h"

namespace timest {

namespace {

constexpr int TB = 256;
inline unsigned blocks_for(uint64_t n, int threads) { return (unsigned)((n + threads - 1) / threads); }

// Prefix arrays of the child nodes: per position the (layer 0, layer 1)
// prefix pair, so one 16-byte load serves both layers.  Slot i's prefix in the
// out/in order starts at base + 2 i stride, its prefix in the multi-edge order
// stride after that.
struct ChildPrefix {
    const ulonglong2 *base;
    size_t stride;
};

// Candidate ranges up to this many entries are scanned for the excluded
// neighbour; longer ones search the excluded multi-edge list instead.
constexpr uint32_t kScanLimit = 64;   // the bits of a RangeExcl
constexpr int kScanStep = 8;          // independent loads per step (4 and 16 measured 0.2 - 1 % slower)

// The candidate ranges of one kind (Claim 3.1) for every edge as the parent, in
// both layers.  Threads walk the meeting vertex's own list (out-list order for
// side 0, in-list order for side 1), so the lanes of a warp share the vertex,
// its candidate lists and nearby positions in them.  A range is galloped to
// from the parent edge's position in that list (or its cross rank into the
// vertex's other list).  Both layers share the unclipped range: the edge's
// windows of the two layers both contain t, so the bound on the side of the
// edge itself is common and only the far bound is clipped, in at most one
// layer, by a search inside the unclipped range.  The excluded entries are
// exactly the entries of the range whose other endpoint is the parent's other
// endpoint: short ranges are scanned for them in place (one pass serves both
// layers); long ones search the excluded multi-edge list.
// The instructions issued bound it, so time bounds are 32-bit compares, empty
// ranges (two thirds of a power-law graph's) leave early, and 32 registers let
// eight blocks run on an SM.  Kept, a range serves every tree node of its kind
// in the DP and every sample: 0.61 ms per kind on 5e7 edges, two kinds for the
// 5-cycle + chord, against 4.2 ms for the DP that searched them in each node.
__global__ void __launch_bounds__(256, 8) k_ranges(DevGraph g, int c2, int64_t delta, WinDiv wv, int side, int out,
                                                   int later, int inner, uint2 *__restrict__ rec, RangePtrs R)
{
    grid_wait();
    const uint32_t pos = blockIdx.x * blockDim.x + threadIdx.x;
    if (pos >= g.m) return;
    const uint32_t t = __ldg((side ? g.in_t : g.out_t) + pos);
    const uint32_t z = __ldg((side ? g.in_dst : g.out_src) + pos);
    // no earlier time than 0, no later one than the largest t'
    if (t == (later ? 0xFFFFFFFFu : 0u)) { rec[pos] = make_uint2(0, 0); return; }
    const uint32_t *off = out ? g.out_off : g.in_off;
    const uint32_t *tarr = out ? g.out_t : g.in_t;
    const uint32_t *nbr = out ? g.out_nbr : g.in_nbr;
    const uint32_t beg = __ldg(off + z), end = __ldg(off + z + 1);
    const uint32_t base = ((side == 0) == (out != 0)) ? gallop_back(tarr, beg, pos, t)
                                                      : __ldg((side == 0 ? g.out_xrank : g.in_xrank) + pos);
    // the unclipped range, [near, far) or [far, near)
    const uint64_t d = (uint64_t)delta;
    uint32_t near, far, lim;   // lim: the far end's time
    if (later) {
        const uint64_t hu = (uint64_t)t + d;
        lim = hu > 0xFFFFFFFFull ? 0xFFFFFFFFu : (uint32_t)hu;
        near = gallop_above(tarr, base, end, t);
        far = gallop_above(tarr, near, end, lim);
    } else {
        lim = (uint64_t)t >= d ? (uint32_t)((uint64_t)t - d) : 0u;
        near = base;
        far = gallop_back(tarr, beg, base, lim);
    }
    if (near == far) { rec[pos] = make_uint2(near, 0); return; }
    // window bounds as 32-bit times: wlo <= t fits, whi is clamped to the
    // largest t' (no time lies beyond it), which leaves every comparison
    // unchanged and keeps the bounds in half the registers
    const uint64_t wd = (uint64_t)wv.d;
    const uint32_t qt = wv.quot(t);
    uint32_t wlo[2], n[2];   // n: entries of the layer's range
#pragma unroll
    for (int p = 0; p < 2; ++p) {
        const int64_t wi = WinDiv::win_of(qt, p);
        const uint64_t whi64 = ((uint64_t)wi + 2) * wd - 1;
        const uint32_t whi = whi64 > 0xFFFFFFFFull ? 0xFFFFFFFFu : (uint32_t)whi64;
        wlo[p] = wi < 0 ? 0u : (uint32_t)((uint64_t)wi * wd);
        if (wi < 0) n[p] = 0;
        else if (later) n[p] = (whi >= lim ? far : above_idx(tarr, near, far, whi)) - near;
        else n[p] = near - (wlo[p] <= lim ? far : lower_idx(tarr, far, near, wlo[p]));
    }
    const uint32_t most = max(n[0], n[1]);
    if (most == 0) { rec[pos] = make_uint2(near, 0); return; }
    uint32_t y = 0;
#pragma unroll
    for (int p = 0; p < 2; ++p) {
        y |= n[p] << (16 * p);   // (of no use from kRangeLong entries on)
        if (inner && n[p]) {
            const uint32_t a = later ? near : near - n[p];
            if (a > beg && __ldg(tarr + a - 1) >= wlo[p]) y |= kRangeSame << (16 * p);
        }
    }
    // the excluded entries; without Constraint 2 nothing is
    uint4 ex = make_uint4(near, 0, 0, kExclBits);
    uint32_t has = 0;
    if (c2) {
        const uint32_t o = __ldg((side ? g.in_nbr : g.out_nbr) + pos);   // the parent's other endpoint
        if (most <= kScanLimit) {
            const uint32_t a = later ? near : near - most;
            for (uint32_t i0 = 0; i0 < most; i0 += kScanStep) {
                uint32_t hit = 0;   // entry a + i0 + i
#pragma unroll
                for (int i = 0; i < kScanStep; ++i)
                    hit |= (i0 + i < most && __ldg(nbr + a + i0 + i) == o) ? 1u << i : 0u;
                while (hit) {
                    const uint32_t i = i0 + (uint32_t)__ffs((int)hit) - 1, bit = later ? i : most - 1 - i;
                    if (bit < 32) ex.y |= 1u << bit; else ex.z |= 1u << (bit - 32);
                    has |= (bit < n[0] ? kRangeHasExcl : 0u) | (bit < n[1] ? kRangeHasExcl << 16 : 0u);
                    hit &= hit - 1;
                }
            }
        } else {
            // z -> o for a child leaving z, o -> z for one entering it
            const uint32_t pe = out ? pair_of(g, z, o) : pair_of(g, o, z);
            if (pe != kNone) {
                const uint32_t xb = __ldg(g.pair_off + pe), xe = __ldg(g.pair_off + pe + 1);
                ex.w = kExclList;
#pragma unroll
                for (int p = 0; p < 2; ++p) {
                    if (n[p] == 0) continue;
                    // the times of the layer's range: (t, hi] or [lo, t)
                    uint32_t ea, eb;
                    if (later) {
                        const int64_t wi = WinDiv::win_of(qt, p);
                        const uint64_t whi64 = ((uint64_t)wi + 2) * wd - 1;
                        ea = above_idx(g.multi_t, xb, xe, t);
                        eb = gallop_above(g.multi_t, ea, xe, whi64 < lim ? (uint32_t)whi64 : lim);
                        ex.y = ea;
                    } else {
                        ea = lower_idx(g.multi_t, xb, xe, max(lim, wlo[p]));
                        eb = gallop_idx(g.multi_t, ea, xe, t);
                        ex.y = eb;   // both layers' lists end together, a later child's start together
                    }
                    if (eb <= ea) continue;
                    has |= kRangeHasExcl << (16 * p);
                    ex.z |= (eb - ea) << (16 * p);   // (no more than the range's entries)
                    if (inner && ea > xb && __ldg(g.multi_t + ea - 1) >= wlo[p]) ex.z |= kExclSame << (16 * p);
                    n[p] -= eb - ea;   // (its candidates, from here on)
                }
            }
        }
    }
    if (most < kRangeLong) {
        if (!has) { rec[pos] = make_uint2(near, y); return; }
        const unsigned long long i = atomicAdd(R.excl_n, 1ull);
        if (i < R.excl_cap) {
            R.excl[i] = ex;
            rec[pos] = make_uint2((uint32_t)i, y | has);
            return;
        }
        const uint64_t bits = (uint64_t)ex.y | ((uint64_t)ex.z << 32);
#pragma unroll
        for (int p = 0; p < 2; ++p)
            if (ex.w == kExclBits && n[p]) n[p] -= (uint32_t)__popcll((long long)(bits & (~0ull >> (64 - n[p]))));
    }
    rec[pos] = range_counts(n[0], n[1]);
}

// The sum of child c's candidates for the edge at `pos` of the list of side
// `side`, in layer p, when the range is not kept.
static __device__ __noinline__ uint64_t search_sum(const DevGraph &g, const DevPlan &P, const WinDiv &wv, const ChildPrefix &cp,
                                            int c, uint32_t pos, int p)
{
    const bool side = P.tzside[c] != 0, out = P.tout[c] != 0, leaf = P.tleaf[c] != 0;
    const uint32_t t = __ldg((side ? g.in_t : g.out_t) + pos), z = __ldg((side ? g.in_dst : g.out_src) + pos);
    const int64_t wi = wv.win(t, p);
    if (wi < 0) return 0;
    const uint64_t whi64 = ((uint64_t)wi + 2) * (uint64_t)wv.d - 1;
    const uint32_t wlo = (uint32_t)((uint64_t)wi * (uint64_t)wv.d), whi = whi64 > 0xFFFFFFFFull ? 0xFFFFFFFFu : (uint32_t)whi64;
    const uint2 ab = search_range(g, P, c, z, pos, t, wlo, whi);
    if (ab.y <= ab.x) return 0;
    uint3 e = make_uint3(0, 0, 0);
    if (P.c2) e = search_excluded(g, P, c, z, __ldg((side ? g.in_nbr : g.out_nbr) + pos), t, wlo, whi);
    if (leaf) return (uint64_t)(ab.y - ab.x) - (e.z - e.y);
    const uint64_t *Pd = (const uint64_t *)(cp.base + 2 * P.tslot[c] * cp.stride) + p;
    const uint64_t *Pm = (const uint64_t *)(cp.base + (2 * P.tslot[c] + 1) * cp.stride) + p;
    const uint32_t beg = __ldg((out ? g.out_off : g.in_off) + z);
    uint64_t sum = __ldg(Pd + 2 * (size_t)(ab.y - 1));
    if (ab.x > beg && __ldg((out ? g.out_t : g.in_t) + ab.x - 1) >= wlo) sum -= __ldg(Pd + 2 * (size_t)(ab.x - 1));
    if (e.z > e.y) {
        sum -= __ldg(Pm + 2 * (size_t)(e.z - 1));
        if (e.y > e.x && __ldg(g.multi_t + e.y - 1) >= wlo) sum += __ldg(Pm + 2 * (size_t)(e.y - 1));
    }
    return sum;
}

// One side of tree node q (Claim 3.2): the product of the factors of q's
// children that meet q at its tail (side 0) or head (side 1), for every edge
// matched to q and both layers, in the order of the meeting vertex's lists.  A
// child's factor is the sum of its weights over the kept range: a count for a
// leaf, a difference of prefixes otherwise, minus the excluded entries'.
// Results are written in this list order, or through `scatter` into another
// order (a node whose parent scans the out-list order while its own DP runs
// in in-list order writes through the in -> out map).  A root with children at both ends
// runs side 0 (first) then side 1 (last), which reads side 0's partial
// product through the out->in position map, and its pending-overflow bits
// from two bit sets of m/32 words (one per layer; a warp of side 0 writes
// the word of its 32 positions with a ballot), small enough to stay in L2.
// Overflow rule: a factor >= 2^64, or an exact product >= 2^64 with no zero
// factor.
// LEAF: every child met on this side is a leaf, so no prefix sums are read.
// The work per edge is a few loads and little else, so a thread takes K edges
// (blockDim apart) whose loads are in flight together, and random accesses are
// made for weights that are not zero only (a third of them): with one edge per
// thread and every partial gathered, every weight scattered, the three launches
// of the 5-cycle + chord on 5e7 edges took 3.25 ms, like this 1.5 (the four of
// a 6-path on 1e7 edges 743 and 420 us).
constexpr int kDpLeaf = 4, kDpInner = 2;   // K (four and five blocks per SM)
template <bool LEAF, int K>
__global__ void __launch_bounds__(256, LEAF ? 4 : 5)
    k_dp(DevGraph g, const __grid_constant__ DevPlan P, WinDiv wv, int q, int side, int first, int last, ChildPrefix cp,
         RangePtrs ranges, ulonglong2 *__restrict__ wout, const uint32_t *__restrict__ scatter,
         uint32_t *__restrict__ nz, const ulonglong2 *__restrict__ in, const uint32_t *__restrict__ in_nz,
         const uint32_t *__restrict__ pin, uint32_t *__restrict__ pout, uint32_t *status)
{
    grid_wait();
    const uint64_t pos0 = (uint64_t)blockIdx.x * (256 * K) + threadIdx.x;
    auto at = [&](int k) { return (uint32_t)(pos0 + k * 256); };
    auto live = [&](int k) { return pos0 + k * 256 < g.m; };
    uint64_t prod[K][2];
    uint32_t zero = 0, ovf = 0;   // bit 2 k + p: edge k's product in layer p is zero / wrapped
    constexpr uint32_t kAll = (1u << (2 * K)) - 1u;
    uint2 r[K];
    int kind = -1;   // of the ranges in r
    auto load_ranges = [&](int kd) {
        kind = kd;
#pragma unroll
        for (int k = 0; k < K; ++k)
            if (((zero >> (2 * k)) & 3u) != 3u) r[k] = __ldg(ranges.base + (size_t)kind * ranges.stride + at(k));
    };
#pragma unroll
    for (int k = 0; k < K; ++k) {
        prod[k][0] = prod[k][1] = 1;
        r[k] = range_unknown();
        if (!live(k)) zero |= 3u << (2 * k);
    }
    if (P.nchild[q] == 0) {   // a root without children: one for each window that holds the edge
#pragma unroll
        for (int k = 0; k < K; ++k) {
            const uint32_t t = live(k) ? __ldg(g.out_t + at(k)) : 0u;
            zero |= ((wv.win(t, 0) < 0 ? 1u : 0u) | (wv.win(t, 1) < 0 ? 2u : 0u)) << (2 * k);
        }
    }
    if (!first) {
        // side 1 reads side 0's partial (both layers), a random access, where the
        // range of this side's first child holds something and, by its bit set,
        // the partial is not zero
        if (ranges.base) {
            int c = 0;
            while (P.tzside[P.child[q][c]] != side) ++c;
            load_ranges(P.tkind[P.child[q][c]]);
#pragma unroll
            for (int k = 0; k < K; ++k)
                zero |= (((r[k].y & kRangeLong) == 0 ? 1u : 0u) | (((r[k].y >> 16) & kRangeLong) == 0 ? 2u : 0u)) << (2 * k);
        }
        uint32_t xp[K];
#pragma unroll
        for (int k = 0; k < K; ++k) xp[k] = live(k) ? __ldg(g.in_to_out + at(k)) : 0u;
#pragma unroll
        for (int k = 0; k < K; ++k)
            if (((zero >> (2 * k)) & 3u) != 3u && !((__ldg(in_nz + (xp[k] >> 5)) >> (xp[k] & 31)) & 1u)) zero |= 3u << (2 * k);
        const uint32_t words = (g.m + 31) >> 5;
#pragma unroll
        for (int k = 0; k < K; ++k) {
            if (((zero >> (2 * k)) & 3u) == 3u) continue;
            const ulonglong2 pv = __ldg(in + xp[k]);
            prod[k][0] = pv.x;
            prod[k][1] = pv.y;
        }
#pragma unroll
        for (int k = 0; k < K; ++k) {
            if (((zero >> (2 * k)) & 3u) == 3u) continue;
            const uint32_t b0 = __ldg(pin + (xp[k] >> 5)) >> (xp[k] & 31), b1 = __ldg(pin + words + (xp[k] >> 5)) >> (xp[k] & 31);
            // (a partial that wrapped may be 0 as it stands and is none)
            const uint32_t wrapped = (b0 & 1u) | ((b1 & 1u) << 1);
            ovf |= wrapped << (2 * k);
            zero |= (((prod[k][0] == 0 ? 1u : 0u) | (prod[k][1] == 0 ? 2u : 0u)) & ~wrapped) << (2 * k);
        }
    }
    for (int ci = 0; ci < P.nchild[q] && zero != kAll; ++ci) {
        const int c = P.child[q][ci];
        if (P.tzside[c] != side) continue;
        const bool later = P.tlater[c] != 0, leaf = LEAF || P.tleaf[c] != 0;
        if (ranges.base && P.tkind[c] != kind) load_ranges(P.tkind[c]);
        // the range's weight with its excluded entries
        uint64_t sum[K][2];
        const uint64_t *Pd = leaf ? nullptr : (const uint64_t *)(cp.base + 2 * P.tslot[c] * cp.stride);
        if (!LEAF && !leaf) {
            uint32_t near[K];
#pragma unroll
            for (int k = 0; k < K; ++k)
                near[k] = (r[k].y & kRangeFlags) && ((zero >> (2 * k)) & 3u) != 3u ? __ldg(&ranges.excl[r[k].x].x) : r[k].x;
#pragma unroll
            for (int k = 0; k < K; ++k) {
#pragma unroll
                for (int p = 0; p < 2; ++p) {
                    const uint32_t half = (r[k].y >> (16 * p)) & 0xFFFFu, n = half & kRangeLong;
                    const bool on = !((zero >> (2 * k + p)) & 1u) && n && !range_searched(r[k]);
                    const uint32_t a = later ? near[k] : near[k] - n;
                    sum[k][p] = on ? __ldg(Pd + 2 * (size_t)(a + n - 1) + p) : 0;
                    if (on && (half & kRangeSame)) sum[k][p] -= __ldg(Pd + 2 * (size_t)(a - 1) + p);
                }
            }
        } else {
#pragma unroll
            for (int k = 0; k < K; ++k) {
                sum[k][0] = r[k].y & kRangeLong;
                sum[k][1] = (r[k].y >> 16) & kRangeLong;
            }
        }
#pragma unroll
        for (int k = 0; k < K; ++k) {
            if (((zero >> (2 * k)) & 3u) == 3u) continue;
            uint4 ex = make_uint4(r[k].x, 0, 0, kExclBits);
            if (r[k].y & kRangeFlags) ex = __ldg(ranges.excl + r[k].x);
#pragma unroll
            for (int p = 0; p < 2; ++p) {
                if ((zero >> (2 * k + p)) & 1u) continue;
                const uint32_t half = (r[k].y >> (16 * p)) & 0xFFFFu, n = half & kRangeLong;
                uint64_t &sm = sum[k][p];
                if (range_searched(r[k])) {
                    // (the search for both layers in one call takes more of the
                    // kernel's registers: 279 against 241 us on 1e7 edges, a 6-path)
                    sm = range_count(r[k], p);
                    if (leaf ? sm == kCountMany : sm != 0) sm = search_sum(g, P, wv, cp, c, at(k), p);
                } else if (half & kRangeHasExcl) {
                    const uint32_t a = later ? ex.x : ex.x - n;
                    const uint32_t h = (ex.z >> (16 * p)) & 0xFFFFu, ne = h & kExclCount;   // of a list
                    if (ex.w == kExclBits) {
                        uint64_t bits = ((uint64_t)ex.y | ((uint64_t)ex.z << 32)) & (~0ull >> (64 - n));
                        if (leaf) {
                            sm -= (uint32_t)__popcll((long long)bits);
                        } else {
                            for (; bits; bits &= bits - 1) {
                                // the entry's weight: its prefix minus the one before in its segment
                                const uint32_t i = (uint32_t)__ffsll((long long)bits) - 1;
                                const uint32_t x = later ? ex.x + i : ex.x - 1 - i;
                                sm -= __ldg(Pd + 2 * (size_t)x + p);
                                if (x > a || (half & kRangeSame)) sm += __ldg(Pd + 2 * (size_t)(x - 1) + p);
                            }
                        }
                    } else if (leaf) {
                        sm -= ne;
                    } else {
                        const uint64_t *Pm = (const uint64_t *)(cp.base + (2 * P.tslot[c] + 1) * cp.stride) + p;
                        const uint32_t ea = later ? ex.y : ex.y - ne;
                        sm -= __ldg(Pm + 2 * (size_t)(ea + ne - 1));
                        if (h & kExclSame) sm += __ldg(Pm + 2 * (size_t)(ea - 1));
                    }
                }
                bool o = false;
                prod[k][p] = mul_chk(prod[k][p], sm, o);
                ovf |= o ? 1u << (2 * k + p) : 0u;
                zero |= sm == 0 ? 1u << (2 * k + p) : 0u;
            }
        }
    }
    const uint32_t pend = ovf & ~zero;
#pragma unroll
    for (int k = 0; k < K; ++k) {
        // both layers, one store; through the scatter map, where one is given,
        // into an array of zeros
        const bool some = ((zero >> (2 * k)) & 3u) != 3u;
        if (live(k) && (some || !scatter))
            wout[scatter ? __ldg(scatter + at(k)) : at(k)] =
                make_ulonglong2((zero >> (2 * k)) & 1u ? 0 : prod[k][0], (zero >> (2 * k + 1)) & 1u ? 0 : prod[k][1]);
        if (nz) {   // which weights are not zero, a bit each
            const uint32_t w = __ballot_sync(0xffffffffu, some);
            if ((threadIdx.x & 31) == 0 && live(k)) nz[at(k) >> 5] = w;
        }
        if (!last) {   // side 0: the warp's pending bits, one word per layer
            const uint32_t b0 = __ballot_sync(0xffffffffu, (pend >> (2 * k)) & 1u);
            const uint32_t b1 = __ballot_sync(0xffffffffu, (pend >> (2 * k + 1)) & 1u);
            const uint32_t words = (g.m + 31) >> 5;
            if ((threadIdx.x & 31) == 0 && live(k)) {
                pout[at(k) >> 5] = b0;
                pout[words + (at(k) >> 5)] = b1;
            }
        }
    }
    if (last && pend) latch(status, ST_OVERFLOW);
}

// ---- scans over the three orders ----------------------------------------
// segment = (owner, window of layer p); owner boundaries come from a bit set.
// Whether the windows of layer p differ between two times.
__device__ __forceinline__ uint32_t win_change(const WinDiv &wv, uint32_t ta, uint32_t tb)
{
    const uint32_t qa = wv.quot(ta), qb = wv.quot(tb);
    return (WinDiv::win_of(qa, 0) != WinDiv::win_of(qb, 0) ? 1u : 0u) |
           (WinDiv::win_of(qa, 1) != WinDiv::win_of(qb, 1) ? 2u : 0u);
}

// Segment heads of one layer (exports rebuild weights from prefix sums).
struct DirHead {
    const uint32_t *tarr;       // position -> t'
    const uint32_t *ownbits;    // bit set: position starts a new owner
    int p;
    WinDiv wv;
    __device__ bool head(uint64_t i) const
    {
        if (i == 0) return true;
        if ((__ldg(ownbits + (i >> 5)) >> (i & 31)) & 1u) return true;
        return (win_change(wv, __ldg(tarr + i), __ldg(tarr + i - 1)) >> p) & 1u;
    }
};

struct RootHead {
    const uint32_t *tarr;       // g_t
    int p;
    WinDiv wv;
    __device__ bool head(uint64_t i) const
    {
        if (i == 0) return true;
        return (win_change(wv, __ldg(tarr + i), __ldg(tarr + i - 1)) >> p) & 1u;
    }
};

// Both layers at once (two-lane scans): the pair of weights of a position is
// one 16-byte gather; heads are per layer (bit p).
struct DirScan2 {
    const ulonglong2 *w;        // (layer 0, layer 1) weights
    const uint32_t *nz;         // bit set of the non-zero ones (null: none kept)
    const uint32_t *perm;       // scan position -> weight position (null: same order)
    const uint32_t *tarr;       // position -> t'
    const uint32_t *ownbits;    // bit set: position starts a new owner
    WinDiv wv;
    __device__ uint32_t owner_word(uint64_t w32) const { return __ldg(ownbits + w32); }
};

struct RootScan2 {
    const ulonglong2 *w;        // root weight pairs in list order
    const uint32_t *nz;         // bit set of the non-zero ones
    const uint32_t *tarr;       // g_t
    WinDiv wv;
    const uint32_t *perm;       // gid -> weight position
    __device__ uint32_t owner_word(uint64_t) const { return 0u; }
};

// ---- windows of both layers (Constraint 3, Alg. 1) ------------------------
// A window of layer p starts at GLOBAL position i when t'_i lies in a window
// of layer p and t'_{i-1} does not lie in the same one.  One pass: starts are
// counted over the rows of a warp, the warps of a tile and, by look-back, the
// tiles before it (both layers' counts in one word, 31 bits each: there are at
// most 2^31 windows of a layer), which gives each its place; then the windows'
// first positions and indices, the end sentinels beg[nwin] = m and the numbers
// of windows.  Nothing on the host waits for these numbers: the arrays are
// sized by what T / delta allows (a count, its scan, the host's wait for it and
// the fill were 250 us on 5e7 edges and 60 on 2e6).
struct WinOut {
    uint32_t *beg[2], *id[2];   // null: only the numbers are wanted
    uint32_t *nwin;             // [2]
};
constexpr int kWinChunk = 8;    // rows whose loads are in flight together
template <int ROWS>
__global__ void __launch_bounds__(256) k_windows(const uint32_t *__restrict__ t, uint32_t m, WinDiv wv,
                                                 unsigned long long *__restrict__ state, uint32_t *__restrict__ ticket,
                                                 WinOut W, uint32_t *status)
{
    grid_wait();
    __shared__ uint32_t s_h[2][8][ROWS], s_w[2][8], s_tile;
    __shared__ unsigned long long s_before;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (threadIdx.x == 0) s_tile = atomicAdd(ticket, 1u);
    __syncthreads();
    const uint32_t tile = s_tile;
    const uint64_t base = ((uint64_t)tile * 8 + warp) * (32 * ROWS);
    uint32_t mine[2] = {0, 0};
    for (int c = 0; c < ROWS; c += kWinChunk) {
        const uint64_t x0 = base + c * 32;
        uint32_t v[kWinChunk];
#pragma unroll
        for (int r = 0; r < kWinChunk; ++r) v[r] = x0 + r * 32 + lane < m ? __ldg(t + x0 + r * 32 + lane) : 0u;
        uint32_t qb = wv.quot(x0 > 0 && x0 <= m ? __ldg(t + x0 - 1) : 0u);   // the quotient before the row
#pragma unroll
        for (int r = 0; r < kWinChunk; ++r) {
            const uint64_t x = x0 + r * 32 + lane;
            const uint32_t q = wv.quot(v[r]);
            uint32_t qp = __shfl_up_sync(0xffffffffu, q, 1);
            if (lane == 0) qp = qb;
            qb = __shfl_sync(0xffffffffu, q, 31);
            // the windows of q are those of q / 2 (layer 0) and (q + 1) / 2 (layer 1; none for q = 0)
            const uint32_t h0 = __ballot_sync(0xffffffffu, x < m && (x == 0 || (q >> 1) != (qp >> 1)));
            const uint32_t h1 = __ballot_sync(0xffffffffu, x < m && q > 0 && (x == 0 || ((q + 1) >> 1) != ((qp + 1) >> 1)));
            mine[0] += __popc(h0);
            mine[1] += __popc(h1);
            if (lane == 0) { s_h[0][warp][c + r] = h0; s_h[1][warp][c + r] = h1; }
        }
    }
    if (lane == 0) { s_w[0][warp] = mine[0]; s_w[1][warp] = mine[1]; }
    __syncthreads();
    constexpr unsigned long long kSum = 1ull << 62, kPrefix = 2ull << 62, kCounts = kSum - 1;
    if (warp == 0) {
        unsigned long long sum = 0;
        for (int w = 0; w < 8; ++w) sum += s_w[0][w] | ((unsigned long long)s_w[1][w] << 31);
        if (lane == 0) *(volatile unsigned long long *)(state + tile) = (tile == 0 ? kPrefix : kSum) | sum;
        unsigned long long before = 0;
        for (int64_t j = (int64_t)tile - 1 - lane; tile != 0; j -= 32) {   // lane i at the i-th tile before
            unsigned long long x = 2ull << 62;
            if (j >= 0) {
                x = *(volatile unsigned long long *)(state + j);
                for (int it = 0; (x >> 62) == 0 && it < kLookbackPolls; ++it) {
                    __nanosleep(32);
                    x = *(volatile unsigned long long *)(state + j);
                }
                if ((x >> 62) == 0) { latch(status, ST_TIMEOUT); x = 2ull << 62; }
            }
            const unsigned end = __ballot_sync(0xffffffffu, (x >> 62) == 2);
            const int last = end ? __ffs((int)end) - 1 : 31;
            unsigned long long c = lane <= last ? x & kCounts : 0;
            for (int o = 16; o > 0; o >>= 1) c += __shfl_xor_sync(0xffffffffu, c, o);
            before += c;
            if (end) break;
        }
        if (lane == 0) {
            if (tile != 0) *(volatile unsigned long long *)(state + tile) = kPrefix | (before + sum);
            s_before = before;
        }
    }
    __syncthreads();
    uint32_t k[2] = {(uint32_t)(s_before & 0x7FFFFFFFu), (uint32_t)((s_before >> 31) & 0x7FFFFFFFu)};
    for (int w = 0; w < warp; ++w) { k[0] += s_w[0][w]; k[1] += s_w[1][w]; }
    for (int r = 0; r < ROWS; ++r) {
        const uint64_t x = base + r * 32 + lane;
        const uint32_t h[2] = {s_h[0][warp][r], s_h[1][warp][r]};
#pragma unroll
        for (int p = 0; p < 2; ++p) {
            const uint32_t at = k[p] + __popc(h[p] & ((1u << lane) - 1u)), mark = (h[p] >> lane) & 1u;
            if (mark && W.beg[p]) {
                W.beg[p][at] = (uint32_t)x;
                W.id[p][at] = (uint32_t)wv.win(__ldg(t + x), p);
            }
            if (x == (uint64_t)m - 1) {
                if (W.beg[p]) W.beg[p][at + mark] = m;
                W.nwin[p] = at + mark;
            }
            k[p] += __popc(h[p]);
        }
    }
}
// rows per warp: as the pair kernel's (a small array needs the blocks more than the fewer tiles)
constexpr int kWinRowsSmall = 8, kWinRowsLarge = 64;
constexpr uint32_t kWinSmall = 4000000;

// ---- guide table of the root search --------------------------------------
// Window kk of a layer gets about n/4 buckets of width 2^s over its draws
// [0, W_kk); the table holds, per bucket j, the first edge whose in-window
// CDF exceeds j 2^s, then the window's last edge.  count[kk] = buckets + 1.
__device__ __forceinline__ uint64_t ceil_shift(uint64_t c, uint32_t s) { return (c >> s) + ((c & ((1ull << s) - 1)) != 0); }

struct GuideLayer {
    const uint64_t *cdf;
    const uint32_t *win_beg;
    uint32_t nwin;
    uint32_t *gshift, *goff, *guide;
};
struct GuideArgs {
    GuideLayer L[2];
    const uint32_t *nwin;   // on the device [2] (null: those of L)
    __device__ __forceinline__ uint32_t windows(int p) const { return nwin ? __ldg(nwin + p) : p ? L[1].nwin : L[0].nwin; }
};

// Window totals W_i (last root-CDF entry of each window) and their 128-bit
// running sum over (layer 0 windows, layer 1 windows) by the blocks of y = 0,
// which also put their total at W; the guide table's bucket width and offset of
// each window by y = 1 + p for layer p.  A tile of kTotTile windows is a block,
// whose sum is looked back for as in the segmented scans: the number of windows
// is known on the device alone, so the grid is for the most there can be and
// the blocks past the last tile leave.  The loads of win_beg and of the CDF
// behind it are what takes the time (random sectors): one block for each y,
// eight windows per thread at a time, kept only three SMs' loads in flight.
// 5.6e4 windows: 61 us like that, 14 so; 1.7e4: 24 and 12.
constexpr int kTotItems = 4, kTotThreads = 256;
constexpr uint32_t kTotTile = kTotThreads * kTotItems;
__global__ void __launch_bounds__(kTotThreads) k_window_totals(GuideArgs A, uint64_t *__restrict__ wcum, uint64_t *__restrict__ W,
                                                               SegTile *__restrict__ tiles, uint32_t *__restrict__ ticket,
                                                               uint32_t *status)
{
    grid_wait();
    constexpr int kWarps = kTotThreads / 32;
    __shared__ u128 s_tot[kWarps];
    __shared__ u128 s_before;
    __shared__ uint32_t s_tile, s_stop;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const uint32_t nw0 = A.windows(0), nw1 = A.windows(1);
    const int b = blockIdx.y;
    const uint32_t n = b == 0 ? nw0 + nw1 : b == 1 ? nw0 : nw1, ntiles = n ? (n - 1) / kTotTile + 1 : 1;
    if (blockIdx.x >= ntiles) return;   // (as many blocks stay as there are tiles)
    tiles += (size_t)b * gridDim.x;
    if (threadIdx.x == 0) s_tile = atomicAdd(ticket + b, 1u);
    if (threadIdx.x == 32) s_stop = latched(status) & ST_TIMEOUT;
    __syncthreads();
    if (s_stop) {   // a wait ran out: win_beg may have holes; no tile waits for this one
        if (threadIdx.x == 0) seg_publish(tiles + s_tile, SegAgg2{0, 0, 0, 0}, 2);
        return;
    }
    const uint32_t tile = s_tile, k0 = tile * kTotTile + threadIdx.x * kTotItems;
    uint64_t v[kTotItems];
    u128 sum = 0;
#pragma unroll
    for (int j = 0; j < kTotItems; ++j) {
        const uint32_t k = k0 + j;
        v[j] = 0;
        if (k < n) {
            const bool second = b == 2 || (b == 0 && k >= nw0);
            const uint32_t *win_beg = second ? A.L[1].win_beg : A.L[0].win_beg;
            const uint32_t kk = b == 0 && second ? k - nw0 : k, wend = win_beg[kk + 1];
            const uint64_t W = (second ? A.L[1].cdf : A.L[0].cdf)[wend - 1];
            if (b == 0) {
                v[j] = W;
            } else {
                // about n / 4 buckets of 2^sh draws each over the window's W
                const uint32_t ne = wend - win_beg[kk], target = ne >> 2 ? ne >> 2 : 1;
                uint32_t sh = 0;
                if (W) {
                    const int d = __clz((int)target) - 32 + 64 - __clzll((long long)(W - 1));
                    sh = d > 1 ? d - 1 : 0;   // not above the least width, then stepped up to it
                    while (sh < 63 && ((W - 1) >> sh) + 1 > target) ++sh;
                }
                (second ? A.L[1].gshift : A.L[0].gshift)[kk] = sh;
                v[j] = (W ? ((W - 1) >> sh) + 1 : 0) + 1;
            }
        }
        sum += v[j];
    }
    // exclusive scan of the threads' sums (128-bit) across the block
    u128 incl = sum;
    for (int o = 1; o < 32; o <<= 1) {
        const uint64_t yl = __shfl_up_sync(0xffffffffu, (uint64_t)incl, o);
        const uint64_t yh = __shfl_up_sync(0xffffffffu, (uint64_t)(incl >> 64), o);
        if (lane >= o) incl += (u128)yl | ((u128)yh << 64);
    }
    if (lane == 31) s_tot[warp] = incl;
    __syncthreads();
    if (warp == 0) {
        u128 T = 0, before = 0;
        for (int w = 0; w < kWarps; ++w) T += s_tot[w];
        if (lane == 0) seg_publish(tiles + tile, SegAgg2{(uint64_t)T, (uint64_t)(T >> 64), 0, 0}, tile == 0 ? 2u : 1u);
        if (tile) {
            for (int64_t jb = (int64_t)tile - 1;; jb -= 32) {   // 32 tiles at a time, the closest in lane 0
                const int64_t j = jb - lane;
                SegAgg2 x{0, 0, 0, 0};
                uint32_t st = 2;
                if (j >= 0) {
                    st = seg_read(tiles + j, x);
                    for (int it = 0; st == 0 && it < kLookbackPolls; ++it) {
                        __nanosleep(64);
                        st = seg_read(tiles + j, x);
                    }
                    if (st == 0) { latch(status, ST_TIMEOUT); x = SegAgg2{0, 0, 0, 0}; }
                }
                const unsigned stop = __ballot_sync(0xffffffffu, st != 1);
                u128 y = !stop || lane < __ffs((int)stop) ? (u128)x.v0 | ((u128)x.v1 << 64) : 0;
                for (int o = 16; o; o >>= 1) {
                    const uint64_t yl = __shfl_xor_sync(0xffffffffu, (uint64_t)y, o);
                    const uint64_t yh = __shfl_xor_sync(0xffffffffu, (uint64_t)(y >> 64), o);
                    y += (u128)yl | ((u128)yh << 64);
                }
                before += y;
                if (stop) break;
            }
            const u128 P = before + T;
            if (lane == 0) seg_publish(tiles + tile, SegAgg2{(uint64_t)P, (uint64_t)(P >> 64), 0, 0}, 2);
        }
        if (lane == 0) {
            s_before = before;
            if (b == 0 && tile == ntiles - 1) {
                const u128 all = before + T;
                W[0] = wcum[2 * (size_t)n] = (uint64_t)all;
                W[1] = wcum[2 * (size_t)n + 1] = (uint64_t)(all >> 64);
            }
        }
    }
    __syncthreads();
    u128 run = s_before + incl - sum;
    for (int w = 0; w < warp; ++w) run += s_tot[w];
#pragma unroll
    for (int j = 0; j < kTotItems; ++j) {
        const uint32_t k = k0 + j;
        if (k < n) {
            if (b == 0) {
                wcum[2 * (size_t)k] = (uint64_t)run;
                wcum[2 * (size_t)k + 1] = (uint64_t)(run >> 64);
            } else {
                (b == 2 ? A.L[1].goff : A.L[0].goff)[k] = (uint32_t)run;
            }
        }
        run += v[j];
    }
}

// Guide table of the window pick: entry j is the window holding draw j 2^s
// (the last k with wcum[k] <= j 2^s), for the ceil(W / 2^s) buckets, then a
// sentinel (the last window).  A binary search per bucket j; W is read on the
// device (the last cumulative entry).
__device__ void wguide_entry(const uint64_t *__restrict__ wcum, uint32_t nw, uint32_t *__restrict__ guide, uint32_t j)
{
    const u128 W = (u128)wcum[2 * (size_t)nw] | ((u128)wcum[2 * (size_t)nw + 1] << 64);
    if (W == 0) return;
    const uint32_t s = wguide_shift((uint64_t)W, (uint64_t)(W >> 64), nw);
    const uint64_t nb = (uint64_t)((W + ((u128)1 << s) - 1) >> s);
    if (j > nb) return;
    if (j == nb) { guide[j] = nw - 1; return; }
    const u128 x = (u128)j << s;
    uint32_t lo = 0, hi = nw;   // wcum[0] = 0 <= x; find the last k with wcum[k] <= x
    while (hi - lo > 1) {
        const uint32_t mid = (lo + hi) >> 1;
        const u128 c = (u128)wcum[2 * (size_t)mid] | ((u128)wcum[2 * (size_t)mid + 1] << 64);
        if (c <= x) lo = mid; else hi = mid;
    }
    guide[j] = lo;
}

// Edges in GLOBAL order, kGuideItems consecutive ones per thread, layer p =
// blockIdx.y: the buckets whose lower bound falls in [cdf[x-1], cdf[x]) start
// at edge x.  A warp takes 32 x kGuideItems consecutive edges, lane l the
// edges l, l + 32, ... of them (coalesced CDF reads); the warp finds the
// window of its first edge by a binary search over the window starts, and a
// lane steps to the next window as its edges cross one, so a window of any
// size is spread over many threads.  blockIdx.y = 2: the window pick's guide,
// a bucket per thread.  A pass that has latched anything by now fills nothing:
// sums that wrapped 2^64 do not rise along a window, so their buckets need not
// lie in the room that the window's last sum was given.
#ifndef TM_GUIDE_ITEMS
#define TM_GUIDE_ITEMS 32   // measured: 32 edges per lane beat 8 (1.77 against 1.81 ms for the root phase) and 2
#endif
constexpr int kGuideItems = TM_GUIDE_ITEMS;
__global__ void __launch_bounds__(TB) k_guide_fill(GuideArgs A, uint32_t m, const uint64_t *__restrict__ wcum,
                                                   uint32_t *__restrict__ wguide, const uint32_t *status)
{
    grid_wait();
    const uint32_t bits = latched(status);   // (asked below, once the window is found)
    const int p = blockIdx.y;
    if (p == 2) {
        if (bits) return;
        const uint32_t nw = A.windows(0) + A.windows(1);
        if (nw == 0) return;
        for (uint64_t j = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; j <= 4 * (uint64_t)nw;
             j += (uint64_t)gridDim.x * blockDim.x)
            wguide_entry(wcum, nw, wguide, (uint32_t)j);
        return;
    }
    // per-field selects keep the parameter block out of local memory
    const uint32_t nwin = A.windows(p);
    const uint64_t *__restrict__ cdf = p ? A.L[1].cdf : A.L[0].cdf;
    const uint32_t *__restrict__ win_beg = p ? A.L[1].win_beg : A.L[0].win_beg;
    const uint32_t *__restrict__ gshift = p ? A.L[1].gshift : A.L[0].gshift;
    const uint32_t *__restrict__ goff = p ? A.L[1].goff : A.L[0].goff;
    uint32_t *__restrict__ guide = p ? A.L[1].guide : A.L[0].guide;
    const uint64_t gt = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const uint64_t xs = (gt >> 5) * (32u * kGuideItems) + (gt & 31u);
    if (xs >= m || nwin == 0) return;
    // kk = the last window starting at or before the warp's first edge x0
    // (none: x0 precedes every window); the same search in every lane, so
    // each probe is one broadcast load
    const uint32_t x0 = (uint32_t)(xs - (gt & 31u));
    uint32_t lo = 0, hi = nwin;
    while (lo < hi) {
        const uint32_t mid = (lo + hi) >> 1;
        if (win_beg[mid] <= x0) lo = mid + 1; else hi = mid;
    }
    if (bits) return;
    int64_t kk = (int64_t)lo - 1;
    const uint64_t xe = min((uint64_t)m, (uint64_t)(xs + 32u * kGuideItems));
    // kGuideBatch edges' CDF pairs loaded before any is used (independent
    // loads in flight), then the edges in order
    constexpr int kGuideBatch = 4;
    for (uint64_t xb = xs; xb < xe; xb += 32u * kGuideBatch) {
        uint64_t c1v[kGuideBatch], c0v[kGuideBatch];
#pragma unroll
        for (int u = 0; u < kGuideBatch; ++u) {
            const uint64_t xx = xb + 32u * u;
            c1v[u] = xx < xe ? cdf[xx] : 0;
            c0v[u] = (xx < xe && xx > 0) ? cdf[xx - 1] : 0;
        }
#pragma unroll
        for (int u = 0; u < kGuideBatch; ++u) {
            const uint64_t xx = xb + 32u * u;
            if (xx >= xe) break;
            const uint32_t x = (uint32_t)xx;
            while (kk + 1 < (int64_t)nwin && win_beg[kk + 1] <= x) ++kk;
            if (kk < 0) continue;   // before the layer's first window
            const uint32_t wbeg = win_beg[kk], wend = win_beg[kk + 1];
            const uint32_t sh = gshift[kk];
            uint32_t *G = guide + goff[kk];
            const uint64_t c1 = c1v[u], c0 = x > wbeg ? c0v[u] : 0;
            const uint64_t j1 = ceil_shift(c1, sh);
            for (uint64_t j = ceil_shift(c0, sh); j < j1; ++j) G[j] = x;
            if (x == wend - 1) G[j1] = x;
        }
    }
}

// Reconstruct w for one order from its segmented prefix (exports); the
// prefix of position i is pref[i * stride].
template <class F>
__global__ void k_unprefix(F f, const uint64_t *__restrict__ pref, int stride, const uint32_t *__restrict__ perm,
                           uint32_t m, uint64_t *__restrict__ out)
{
    grid_wait();
    uint32_t i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= m) return;
    uint64_t w = pref[(size_t)i * stride] - (f.head(i) ? 0 : pref[(size_t)(i - 1) * stride]);
    out[perm ? perm[i] : i] = w;
}

__global__ void k_leaf_weights(const uint32_t *__restrict__ t, uint32_t m, int p, WinDiv wv, uint64_t *__restrict__ out)
{
    grid_wait();
    uint32_t i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < m) out[i] = wv.win(t[i], p) >= 0 ? 1 : 0;
}

}  // namespace

static void *malloc_motif(tm_ctx *ctx, tm_motif *mo, size_t bytes)
{
    void *p = dalloc(ctx, bytes ? bytes : 8);
    if (p) { mo->bufs.push_back({p, bytes ? bytes : 8}); mo->bytes += bytes; }
    return p;
}

static void free_motif_weights(tm_ctx *ctx, tm_motif *mo)
{
    for (auto &b : mo->bufs) dfree(ctx, b.first, b.second);
    mo->bufs.clear();
    mo->bytes = 0;
    for (int p = 0; p < 2; ++p) mo->layer[p] = LayerData();
    for (int sl = 0; sl < kMaxTree; ++sl) mo->pref_dir[sl] = mo->pref_multi[sl] = nullptr;
    mo->range = RangePtrs{};
    mo->wcum = nullptr;
    mo->wguide = nullptr;
    mo->have_weights = false;
}

// A block of this size or more that is refused with candidate ranges is asked for
// without them.  A smaller one is reported as any other: scratch is taken in
// chunks of at least 64 MiB, so where 4 MiB are refused there is nothing to run with.
constexpr size_t kRangesOptional = (size_t)4 << 20;

// Sizes of the arrays that a motif keeps, each at a multiple of 256 bytes.
static size_t aligned(size_t b) { return (b + 255) / 256 * 256; }
static size_t guide_entries(uint64_t m, uint32_t nw) { return (size_t)m / 4 + 3 * (size_t)nw + 1; }
// window starts and indices of both layers
static size_t window_bytes(const uint32_t nw[2])
{
    return aligned(((size_t)nw[0] + 1) * 4) * 2 + aligned(((size_t)nw[1] + 1) * 4) * 2;
}
// room for excluded entries at 0.3 of the edges per kind: with bursts of repeated
// pairs a star's ranges have them at 0.2 - 0.3
static size_t excl_entries(uint64_t m, int kinds) { return (size_t)kinds * ((size_t)m * 3 / 10); }
static size_t range_bytes_of(uint64_t m, int kinds)
{
    return (size_t)kinds * aligned((size_t)m * sizeof(uint2)) + aligned(excl_entries(m, kinds) * sizeof(RangeExcl));
}
static size_t block_bytes(const DevPlan &P, uint64_t m, const uint32_t nw[2])   // without the ranges
{
    const size_t both = (size_t)nw[0] + nw[1];
    return 2 * window_bytes(nw) + 2 * aligned((size_t)m * 8) + (size_t)P.nslots * 2 * aligned((size_t)m * 16) +
           aligned((both + 1) * 16) + aligned(guide_entries(m, nw[0]) * 4) + aligned(guide_entries(m, nw[1]) * 4) +
           aligned((4 * both + 2) * 4);
}
// The most windows there can be: their indices go up to T / unit, the even ones in layer 0.
static void window_bounds(const DevPlan &P, uint64_t m, uint64_t T, uint32_t nw[2])
{
    const uint64_t qT = m ? T / (uint64_t)P.wdelta : 0;
    nw[0] = (uint32_t)std::min<uint64_t>(m, qT / 2 + 1);
    nw[1] = (uint32_t)std::min<uint64_t>(m, (qT + 1) / 2);
}

size_t weights_bytes(const DevPlan &P, uint64_t m, uint64_t T)
{
    uint32_t nw[2];
    window_bounds(P, m, T, nw);
    const uint64_t mm = m ? m : 1;
    return block_bytes(P, mm, nw) + range_bytes_of(mm, P.nkinds);
}

// Owner bit sets of the out-, in- and multi-edge orders (built with the graph).
struct OwnerBits { const uint32_t *out, *in, *multi; };

static GuideArgs guide_args(const tm_motif *mo, const uint32_t *nwin)
{
    GuideArgs ga{};
    ga.nwin = nwin;
    for (int p = 0; p < 2; ++p) {
        const LayerData &L = mo->layer[p];
        ga.L[p] = GuideLayer{L.root_cdf, L.win_beg, L.nwin, L.win_gshift, L.win_goff, L.guide};
    }
    return ga;
}

int fill_guides(tm_ctx *ctx, tm_motif *mo, const uint32_t *nwin)
{
    const uint64_t m = ctx->g.m;
    if (m == 0) return TM_OK;
    const uint64_t gwarps = (m + 32 * kGuideItems - 1) / (32 * kGuideItems);
    launch(ctx, k_guide_fill, dim3(blocks_for(gwarps * 32, TB), 3), TB, guide_args(mo, nwin), (uint32_t)m,
           (const uint64_t *)mo->wcum, mo->wguide, (const uint32_t *)ctx->status);
    return check_cuda(ctx, cudaGetLastError(), "guide tables");
}

int compute_weights(tm_ctx *ctx, tm_motif *mo, bool guides, SharedPass *sh)
{
    ScratchScope scope(ctx);
    free_motif_weights(ctx, mo);
    const DevGraph &g = ctx->g;
    assign_kinds(mo->plan);
    const DevPlan &P = mo->plan;
    cudaStream_t st = ctx->stream;
    const uint32_t m = g.m;
    const WinDiv wv = make_windiv(P.wdelta);   // window unit (delta, or one window without Constraint 3)
    int rc = TM_OK;
    const bool known = sh && sh->windows;      // the windows, from an earlier candidate
    cudaMemsetAsync(ctx->status, 0, kStatusBytes, st);
    uint32_t nwh[2];
    window_bounds(P, m, g.T, nwh);
    if (known) { nwh[0] = sh->nwin[0]; nwh[1] = sh->nwin[1]; }
    // cleared together: the tickets, the number of kept excluded ranges, the tile
    // words of the windows, of their totals and of every scan
    const bool win_small = m <= kWinSmall;
    const uint32_t win_tile = 256u * (win_small ? kWinRowsSmall : kWinRowsLarge), win_tiles = m ? (m - 1) / win_tile + 1 : 0;
    const size_t win_bytes = ((size_t)win_tiles * 8 + 64 + 255) / 256 * 256, scan_bytes = scan_state_bytes(m);
    const uint32_t tot_tiles = (uint32_t)(((uint64_t)nwh[0] + nwh[1]) / kTotTile) + 1;
    const size_t tot_bytes = (3 * (size_t)tot_tiles * sizeof(SegTile) + 255) / 256 * 256;
    const size_t clear_bytes = win_bytes + tot_bytes + (2 * (size_t)P.nslots + 1) * scan_bytes;
    char *clear = (char *)salloc(ctx, clear_bytes);
    if (!clear) return TM_E_NOMEM;
    cudaMemsetAsync(clear, 0, clear_bytes, st);
    uint32_t *ticket = (uint32_t *)clear;   // [0] the windows', [4..6] their totals'; [2] the excluded ranges' number
    unsigned long long *win_state = (unsigned long long *)(clear + 64);
    SegTile *tot_state = (SegTile *)(clear + win_bytes);
    char *scan_state = clear + win_bytes + tot_bytes;
    auto windows = [&](const WinOut &wo) {
        launch(ctx, win_small ? k_windows<kWinRowsSmall> : k_windows<kWinRowsLarge>, win_tiles, 256, g.g_t, m, wv,
               win_state, ticket, wo, ctx->status);
    };
    // ---- windows of each layer (K2); one block for everything the motif keeps
    if (!known && (uint64_t)nwh[0] + nwh[1] > (uint64_t)m / 8 + 4096) {
        // windows so short that most may be empty: counted before they take room
        PhaseScope ph(ctx, TM_PH_WINDOWS);
        windows(WinOut{{nullptr, nullptr}, {nullptr, nullptr}, ctx->status + 2});
        uint32_t bits = 0;
        rc = read_status(ctx, &bits);
        if (rc) return rc;
        if (bits) return set_err(ctx, TM_E_CUDA, "device status error in the window count");
        nwh[0] = ctx->status_host[2];
        nwh[1] = ctx->status_host[3];
        cudaMemsetAsync(clear, 0, win_bytes, st);
    }
    {
        const size_t mm = (size_t)(m ? m : 1);
        // the candidate ranges come last: a block that does not fit with them is
        // tried without (the DP and the samplers then search the ranges)
        const int nk = sh ? sh->max_kinds : P.nkinds;
        const size_t excl_cap = excl_entries(mm, nk), win_arrays = window_bytes(nwh);
        size_t range_bytes = range_bytes_of(mm, nk);
        char *blk = nullptr;
        size_t off = 0;
        auto take = [&](size_t bytes) { char *q = blk + off; off += aligned(bytes); return (void *)q; };
        auto take_windows = [&](uint32_t *beg[2], uint32_t *id[2]) {
            for (int p = 0; p < 2; ++p) {
                beg[p] = (uint32_t *)take(((size_t)nwh[p] + 1) * 4);
                id[p] = (uint32_t *)take(((size_t)nwh[p] + 1) * 4);
            }
        };
        auto take_ranges = [&](RangePtrs &r) {
            r.stride = aligned(mm * sizeof(uint2)) / sizeof(uint2);
            r.base = (uint2 *)take((size_t)nk * r.stride * sizeof(uint2));
            r.excl = (RangeExcl *)take(excl_cap * sizeof(RangeExcl));
            r.excl_cap = (uint32_t)std::min<size_t>(excl_cap, 0xFFFFFFFFu);
        };
        if (sh && !sh->block) {
            sh->bytes = win_arrays + range_bytes + 256;
            sh->block = blk = (char *)dalloc(ctx, sh->bytes);
            if (!blk) return TM_E_NOMEM;
            take_windows(sh->win_beg, sh->win_id);
            take_ranges(sh->range);
            sh->range.excl_n = (unsigned long long *)take(256);
            cudaMemsetAsync(sh->range.excl_n, 0, 8, st);
            off = 0;
        }
        if (sh) range_bytes = 0;
        size_t total = block_bytes(P, mm, nwh);
        if (sh) total -= win_arrays;
        bool with_ranges = true;
        blk = (char *)malloc_motif(ctx, mo, total + range_bytes);
        if (!blk && !sh && total + range_bytes >= kRangesOptional) {
            with_ranges = false;
            blk = (char *)malloc_motif(ctx, mo, total);
        }
        if (!blk) return TM_E_NOMEM;
        uint32_t *win_beg[2], *win_id[2];
        if (!sh) take_windows(win_beg, win_id);
        for (int p = 0; p < 2; ++p) {
            LayerData &L = mo->layer[p];
            L.nwin = nwh[p];
            L.win_beg = sh ? sh->win_beg[p] : win_beg[p];
            L.win_id = sh ? sh->win_id[p] : win_id[p];
            L.root_cdf = (uint64_t *)take(mm * 8);
            L.win_gshift = (uint32_t *)take(((size_t)nwh[p] + 1) * 4);
            L.win_goff = (uint32_t *)take(((size_t)nwh[p] + 1) * 4);
            L.guide = (uint32_t *)take(guide_entries(m, nwh[p]) * 4);
        }
        for (int sl = 0; sl < P.nslots; ++sl) {   // one after the other (ChildPrefix)
            mo->pref_dir[sl] = (ulonglong2 *)take(mm * 16);
            mo->pref_multi[sl] = (ulonglong2 *)take(mm * 16);
        }
        mo->wcum = (uint64_t *)take(((size_t)nwh[0] + nwh[1] + 1) * 16);
        mo->wguide = (uint32_t *)take((4 * ((size_t)nwh[0] + nwh[1]) + 2) * 4);
        if (sh) {
            mo->range = sh->range;
        } else if (with_ranges) {
            take_ranges(mo->range);
            mo->range.excl_n = (unsigned long long *)(ticket + 2);   // of this pass
        }
    }
    if (!known) {
        PhaseScope ph(ctx, TM_PH_WINDOWS);
        if (m)
            windows(WinOut{{mo->layer[0].win_beg, mo->layer[1].win_beg}, {mo->layer[0].win_id, mo->layer[1].win_id},
                           ctx->status + 2});
        else {
            cudaMemsetAsync(mo->layer[0].win_beg, 0, 4, st);
            cudaMemsetAsync(mo->layer[1].win_beg, 0, 4, st);
        }
    }
    // ---- DP over tree nodes in increasing height (K3) + prefixes (K4)
    const OwnerBits ob{g.own_out, g.own_in, g.own_multi};
    ulonglong2 *w = nullptr, *pw = nullptr;   // (layer 0, layer 1) weight pairs
    uint32_t *pend = nullptr;                 // per layer a bit set: pending overflow of a side-0 partial
    w = (ulonglong2 *)salloc(ctx, (size_t)(m ? m : 1) * 16);
    uint32_t *nz = (uint32_t *)salloc(ctx, ((size_t)m / 32 + 1) * 8);   // non-zero bits of w, then of pw
    if (!w || !nz) return TM_E_NOMEM;
    uint32_t *pw_nz = nz + (size_t)m / 32 + 1;
    const ChildPrefix cp{P.nslots ? mo->pref_dir[0] : nullptr, (size_t)((m ? m : 1) * (uint64_t)16 + 255) / 256 * 16};
    int maxh = 0;
    for (int q = 0; q < P.ntree; ++q) maxh = std::max(maxh, (int)P.height[q]);
    std::vector<int> order;
    for (int h = 1; h <= maxh; ++h)
        for (int q = P.ntree - 1; q >= 0; --q)
            if (P.height[q] == h) order.push_back(q);
    if (P.tleaf[0]) order.push_back(0);   // single-edge motif: the root is a leaf
    if (mo->range.base && m) {
        PhaseScope ph(ctx, TM_PH_DP);
        auto ranges = [&](int k, int at, int inner) {
            launch(ctx, k_ranges, blocks_for(m, TB), TB, g, P.c2, P.delta, wv, P.kside[k], P.kout[k], P.klater[k], inner,
                   mo->range.base + (size_t)at * mo->range.stride, mo->range);
        };
        int at[kMaxTree];   // where kind k's ranges are
        for (int k = 0; k < P.nkinds; ++k) {
            at[k] = k;
            if (!sh) { ranges(k, k, P.kinner[k]); continue; }
            int &i = at[k] = 0;
            while (i < sh->nkinds && (sh->side[i] != P.kside[k] || sh->out[i] != P.kout[k] || sh->later[i] != P.klater[k])) ++i;
            if (i < sh->nkinds) continue;
            sh->side[i] = P.kside[k]; sh->out[i] = P.kout[k]; sh->later[i] = P.klater[k];
            ++sh->nkinds;
            ranges(k, i, 1);   // with what inner nodes read: a later candidate may have one
        }
        for (int q = 1; q < P.ntree; ++q) mo->plan.tkind[q] = at[P.tkind[q]];
    }
    for (int q : order) {
        // sides of q that children meet; the weights come out in the order of
        // the last side run (out-list order for side 0, in-list for side 1)
        bool has[2] = {false, false};
        bool inner[2] = {false, false};   // a child with children meets this side
        for (int ci = 0; ci < P.nchild[q]; ++ci) {
            const int c = P.child[q][ci];
            has[P.tzside[c]] = true;
            if (!P.tleaf[c]) inner[P.tzside[c]] = true;
        }
        const bool in_order = has[1];
        {
            PhaseScope ph(ctx, TM_PH_DP);
            if (has[0] && has[1] && !pw) {
                pw = (ulonglong2 *)salloc(ctx, (size_t)(m ? m : 1) * 16);
                pend = (uint32_t *)salloc(ctx, ((size_t)m / 32 + 1) * 8);
                if (!pw || !pend) return TM_E_NOMEM;
            }
            if (m) {
                const uint32_t *none = nullptr;
                const ulonglong2 *no_in = nullptr;
                auto dp = [&](int side, int first, int last, ulonglong2 *wout, const uint32_t *scatter, uint32_t *out_nz,
                              const ulonglong2 *in, const uint32_t *in_nz, const uint32_t *pin, uint32_t *pout) {
                    auto go = [&](auto kernel, int per) {
                        launch(ctx, kernel, blocks_for(m, TB * per), TB, g, P, wv, q, side, first, last, cp, mo->range,
                               wout, scatter, out_nz, in, in_nz, pin, pout, ctx->status);
                    };
                    if (inner[side]) go(k_dp<false, kDpInner>, kDpInner);
                    else go(k_dp<true, kDpLeaf>, kDpLeaf);
                };
                if (has[0] && has[1]) {
                    dp(0, 1, 0, pw, none, pw_nz, no_in, none, none, pend);
                    dp(1, 0, 1, w, none, nz, pw, pw_nz, pend, nullptr);
                } else {
                    // a non-root node leaving its parent's meeting vertex runs in
                    // in-list order and is scanned by its parent in out-list
                    // order: it writes through the in -> out map
                    const bool to_out = q != 0 && P.tout[q] != 0 && in_order;
                    // (only what is not zero: 5e7 random 16-byte writes are 1.3 ms,
                    // clearing the array 0.13)
                    if (to_out) cudaMemsetAsync(w, 0, (size_t)m * 16, st);
                    dp(in_order ? 1 : 0, 1, 1, w, to_out ? g.in_to_out : none, to_out ? nullptr : nz, no_in, none, none,
                       nullptr);
                }
            }
        }
        rc = check_cuda(ctx, cudaGetLastError(), "weight DP");
        if (rc) return rc;
        if (q == 0) {
            PhaseScope ph(ctx, TM_PH_ROOT);
            RootScan2 f{w, nz, g.g_t, wv, in_order ? g.in_pos : g.out_pos};
            rc = segmented_scan2_u64(ctx, f, m, scan_state, mo->layer[0].root_cdf, mo->layer[1].root_cdf);
            if (rc) return rc;
        } else {
            PhaseScope ph(ctx, TM_PH_PREFIX);
            const int slot = P.tslot[q];
            const bool out = P.tout[q] != 0;
            // A non-root node's DP runs in the list order of its far endpoint,
            // never in the order its parent scans (out-list order when the node
            // leaves the meeting vertex, in-list order when it enters it).  A
            // node leaving it wrote its weights through the in -> out map, so
            // they are in out-list order already; for a node entering it the
            // in-list order is one gather through the same map.  Multi-edge
            // lists are grouped by source like the out-lists, so the multi-edge
            // prefix gathers, within each source's run, from the weights in
            // out-list order (w in both cases).
            const uint32_t *wnz = out && in_order ? nullptr : nz;   // (scattered weights have no bit set)
            DirScan2 fd{w, wnz, out ? nullptr : g.in_to_out, out ? g.out_t : g.in_t, out ? ob.out : ob.in, wv};
            rc = segmented_scan2_u64(ctx, fd, m, scan_state + (1 + 2 * slot) * scan_bytes, nullptr, nullptr, mo->pref_dir[slot]);
            if (rc) return rc;
            DirScan2 fm{w, wnz, g.multi_to_out, g.multi_t, ob.multi, wv};
            rc = segmented_scan2_u64(ctx, fm, m, scan_state + (2 + 2 * slot) * scan_bytes, nullptr, nullptr, mo->pref_multi[slot]);
            if (rc) return rc;
        }
    }
    // ---- window totals and their 128-bit running sum (K5)
    {
        PhaseScope ph(ctx, TM_PH_ROOT);
        const uint32_t tt = (uint32_t)(((uint64_t)nwh[0] + nwh[1]) / kTotTile) + 1;   // (not more than tot_tiles)
        launch(ctx, k_window_totals, dim3(tt, 3), kTotThreads, guide_args(mo, known ? nullptr : ctx->status + 2), mo->wcum,
               (uint64_t *)(ctx->status + 4), tot_state, ticket + 4, ctx->status);
        if (guides) {
            rc = fill_guides(ctx, mo, known ? nullptr : ctx->status + 2);
            if (rc) return rc;
        }
    }
    mo->range.excl_n = nullptr;   // (of the pass, or of the selection)
    uint32_t bits = 0;
    rc = read_status(ctx, &bits);
    if (rc) return rc;
    if (!known) for (int p = 0; p < 2; ++p) mo->layer[p].nwin = ctx->status_host[2 + p];
    if (sh && !known && !(bits & ~ST_OVERFLOW)) {
        for (int p = 0; p < 2; ++p) sh->nwin[p] = mo->layer[p].nwin;
        sh->windows = true;
    }
    if (bits & ST_OVERFLOW) return set_err(ctx, TM_E_OVERFLOW, "a weight, prefix sum or window total exceeds 2^64");
    if (bits) return set_err(ctx, TM_E_CUDA, "device status error in weight pass");
    memcpy(&mo->W, ctx->status_host + 4, 16);   // copied with the status
    mo->nwtot = mo->layer[0].nwin + mo->layer[1].nwin;
    mo->have_weights = true;
    mo->graph_epoch = ctx->epoch;
    return TM_OK;
}

// w_{q,e} by gid for one layer, rebuilt from the stored prefix arrays.
int export_weights(tm_ctx *ctx, tm_motif *mo, int q, int layer, uint64_t *host_out)
{
    ScratchScope scope(ctx);
    const DevGraph &g = ctx->g;
    const DevPlan &P = mo->plan;
    cudaStream_t st = ctx->stream;
    uint32_t m = g.m;
    if (m == 0) return TM_OK;
    uint64_t *out = (uint64_t *)salloc(ctx, (size_t)m * 8);
    if (!out) return TM_E_NOMEM;
    const WinDiv wv = make_windiv(P.wdelta);
    int rc = TM_OK;
    if (P.tleaf[q] && q != 0) {
        launch(ctx, k_leaf_weights, blocks_for(m, TB), TB, g.g_t, m, layer, wv, out);
    } else if (q == 0) {
        RootHead f{g.g_t, layer, wv};
        launch(ctx, k_unprefix<RootHead>, blocks_for(m, TB), TB, f, (const uint64_t *)mo->layer[layer].root_cdf, 1,
               (const uint32_t *)nullptr, m, out);
    } else {
        const OwnerBits ob{g.own_out, g.own_in, g.own_multi};
        bool o = P.tout[q] != 0;
        DirHead f{o ? g.out_t : g.in_t, o ? ob.out : ob.in, layer, wv};
        launch(ctx, k_unprefix<DirHead>, blocks_for(m, TB), TB, f,
               (const uint64_t *)mo->pref_dir[P.tslot[q]] + layer, 2, (const uint32_t *)(o ? g.out_gid : g.in_gid),
               m, out);
        rc = check_cuda(ctx, cudaStreamSynchronize(st), "export");
    }
    copy_d2h(ctx, host_out, out, (size_t)m * 8);
    int rc2 = check_cuda(ctx, cudaStreamSynchronize(st), "export copy");
    return rc ? rc : rc2;
}

void release_weights(tm_ctx *ctx, tm_motif *mo) { free_motif_weights(ctx, mo); }

}  // namespace timest

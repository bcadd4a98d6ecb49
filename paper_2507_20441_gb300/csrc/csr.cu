// Temporal CSR builder (Sec. 3 preamble; Defs. 3.1-3.3).
//
// From m raw tuples (u, v, t) it builds, all on the device:
//   GLOBAL order (t', src, dst)      -> gid, the edge id used everywhere
//   out-lists   (src | t', dst)      -> out_off / out_t / out_nbr / out_gid / out_pos
//   in-lists    (dst | t', src)      -> in_off / in_t / in_nbr / in_gid / in_pos / in_to_out
//   multi-edge  (src, dst | t')      -> pairs, pair_off / pair_dst / multi_t / multi_to_out
// with t' = t - t_min.  The orderings come from a stable LSD radix sort (up to
// 7-bit digits, up to four payload arrays) written here.  The GLOBAL order is
// a sort by t' after which each run of equal t' is put in (src, dst) order in
// place (one thread, one block, or, for a run of more than 4096 edges, the
// full three-key sort).  The OUT and IN orders are stable re-sorts of the
// GLOBAL order by one endpoint that carry gid, t' and the other endpoint as
// payloads, so no list array is gathered; each edge's list position by gid
// (the inverse of the sort's permutation) is then written through buckets of
// consecutive gids.  The IN sort carries each edge's out-list position too
// (read in GLOBAL order), which is the in -> out map, and the multi-edge
// order is a stable re-sort of the IN order by source carrying t', the
// destination and that map (-> multi_to_out).  The random accesses left are
// the cross ranks, found by searches in the owner's other list.
#include <cuda_runtime.h>
#include <stdint.h>
#include <string.h>

#include <algorithm>
#include <memory>
#include <string>

#include "scan.cuh"
#include "tm_device.cuh"
#include "tm_internal.h"

namespace timest {

namespace {

// ---- radix sort --------------------------------------------------------
// Keys are sorted least significant digit first, with up to 7-bit digits
// (a 21-bit vertex id takes three passes, a 27-bit time four; 9-bit digits,
// fewer passes of shorter runs, measured 6.2 against 5.4 ms for the sorts of
// 5e7 edges and the same at 2e6).  The digit counts of every pass of a sort are made once,
// before its first pass (for the build's sorts by the kernel that compacts the
// input, which reads the keys anyway), and a pass is one kernel: a tile of
// keys is ranked stably, the tile finds where its digits start in the output
// by looking back over the counts that the tiles before it have published, and
// writes its digit runs out (Adinets and Merrill, "Onesweep: A Faster Least
// Significant Digit Radix Sort for GPUs", 2022).
#ifndef TM_RS_ITEMS
#define TM_RS_ITEMS 16   // keys per thread (8 and 12 measured slower)
#endif
constexpr int OS_THREADS = 256;
constexpr int OS_ITEMS = TM_RS_ITEMS;
constexpr int OS_TILE = OS_THREADS * OS_ITEMS;     // 4096 keys per tile
constexpr int OS_WARPS = OS_THREADS / 32;
constexpr int OS_MAXBITS = 7;
constexpr int OS_MAXRADIX = 1 << OS_MAXBITS;
constexpr int OS_SCAN = 512;   // entries of the block scan of bucket counts (two per thread)
static_assert(OS_MAXRADIX <= OS_SCAN && OS_THREADS * 2 == OS_SCAN, "bucket scan layout");
constexpr int OS_MAXPASS = (32 + OS_MAXBITS - 1) / OS_MAXBITS;   // any 32-bit key
// Sorts of up to kSmallSort keys take tiles of 1024: a tile of 4096 would leave
// most SMs without one (20,000 keys: 5 tiles against 20).
constexpr int OS_SMALL_ITEMS = 4;
constexpr uint32_t kSmallSort = 300000;

// The digits of a key's passes: bits [sh, sh + bits) each.
struct DigitPlan {
    int npass = 0;
    int sh[OS_MAXPASS] = {}, bits[OS_MAXPASS] = {};
};
// counts[pass * OS_MAXRADIX + digit] of one key array
constexpr int OS_HIST = OS_MAXPASS * OS_MAXRADIX;

__device__ __forceinline__ void hist_key(const DigitPlan &D, uint32_t key, uint32_t *__restrict__ h)
{
#pragma unroll
    for (int p = 0; p < OS_MAXPASS; ++p)
        if (p < D.npass) atomicAdd(h + p * OS_MAXRADIX + ((key >> D.sh[p]) & ((1u << D.bits[p]) - 1u)), 1u);
}

__device__ __forceinline__ void hist_flush(const uint32_t *__restrict__ h, int n, uint32_t *__restrict__ out)
{
    for (int i = threadIdx.x; i < n; i += blockDim.x)
        if (h[i]) atomicAdd(out + i, h[i]);
}

// Digit counts of every pass over one key array.
__global__ void __launch_bounds__(OS_THREADS) k_rs_hist(const uint32_t *__restrict__ key, uint32_t n, DigitPlan D,
                                                        uint32_t *__restrict__ hist)
{
    grid_wait();
    __shared__ uint32_t h[OS_HIST];
    for (int i = threadIdx.x; i < OS_HIST; i += OS_THREADS) h[i] = 0;
    __syncthreads();
    for (uint64_t i = (uint64_t)blockIdx.x * OS_THREADS + threadIdx.x; i < n; i += (uint64_t)gridDim.x * OS_THREADS)
        hist_key(D, __ldg(key + i), h);
    __syncthreads();
    hist_flush(h, OS_HIST, hist);
}

// Inputs and outputs of a sort's pass: the key and up to four payloads.
struct RsSet {
    const uint32_t *kin = nullptr, *pin[4] = {};
    uint32_t *kout = nullptr, *pout[4] = {};
    uint32_t *inv = nullptr;   // when set: inv[payload 0] = output position (the inverse permutation)
};

// What a tile has published of a digit: its count, or the count of it and of
// every tile before it.
enum : unsigned long long { kTileSum = 1ull << 62, kTilePrefix = 2ull << 62 };

constexpr int kLookback = 4;   // tiles read at a time when looking back (2 measured 1 - 3 % slower, 8 the same)

// One pass.  Tiles are taken from a counter, so every tile before this one has
// been started and publishes its counts without waiting for anyone; waits for
// them are bounded all the same (ST_TIMEOUT).  After a wait that ran out the
// pass's output has holes, and the next pass's keys no longer match the digit
// counts that place them, so a position is checked before it is written (0.3 % of
// the passes on 5e7 keys; asking the status in each tile instead was 0.7).  A warp ranks 32 keys at a time:
// each lane marks its bit in its digit's word of shared memory and reads the
// word back, which gives the peers before it (a ballot per digit bit, which
// this replaces, was most of the pass's instructions).  The tile is staged
// through one shared array: keys first, then each payload in its own round.
// What bounds it is shared memory traffic (70 - 77 % of its throughput with
// ranks and output positions kept in shared arrays), so a thread's tile slots
// and output positions stay in registers (64, four blocks per SM; 48 and 80
// measured 4 - 28 % slower, tiles of 3072 and 5120 keys 3 - 40 %).
// 5e7 keys with three payloads: 395 us a pass, 421 with the shared arrays; with
// separate count, scan and scatter kernels 394 + 53 + 13 us.  2e6 keys: 29 us
// against 26 + 9 + 13 in four launches.
template <int NP, int ITEMS>
__global__ void __launch_bounds__(OS_THREADS, 4)
    k_rs_sweep(RsSet J, uint32_t n, int shift, int bits, const uint32_t *__restrict__ hist,
               unsigned long long *__restrict__ state, uint32_t *__restrict__ ticket, uint32_t *status)
{
    grid_wait();
    constexpr int TILE = OS_THREADS * ITEMS, WCHUNK = ITEMS * 32;
    static_assert(ITEMS % 2 == 0, "slots are kept two to a register");
    __shared__ uint32_t s_buf[TILE];                          // one array of the tile
    __shared__ uint32_t s_match[OS_WARPS * OS_MAXRADIX];      // [warp][digit] lanes of the digit
    __shared__ uint16_t s_wcnt[OS_WARPS * OS_MAXRADIX];       // [warp][digit] counts, then tile slots
    __shared__ uint32_t s_gpos[OS_MAXRADIX];                  // digit start in the output - in the tile
    __shared__ uint32_t s_wt[8];
    __shared__ uint32_t s_tile;
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    if (t == 0) s_tile = atomicAdd(ticket, 1u);
    for (int i = t; i < OS_WARPS * OS_MAXRADIX; i += OS_THREADS) { s_wcnt[i] = 0; s_match[i] = 0; }
    __syncthreads();
    const uint32_t tile = s_tile;
    const uint32_t radix = 1u << bits, dmask = radix - 1u;
    const uint32_t base = tile * (uint32_t)TILE;
    const uint32_t tile_n = min((uint32_t)TILE, n - base);
    const uint32_t lt = (1u << lane) - 1u;
    const uint32_t li0 = warp * WCHUNK + lane;   // this thread's inputs: li0, li0 + 32, ...
    uint16_t *wc = s_wcnt + warp * OS_MAXRADIX;
    uint32_t *wm = s_match + warp * OS_MAXRADIX;
    uint32_t kv[ITEMS];         // the keys, then one payload after the other
    uint32_t slot[ITEMS / 2] = {};   // rank in the warp's chunk, then tile slot, 16 bits each
    auto load = [&](const uint32_t *__restrict__ in) {
#pragma unroll
        for (int j = 0; j < ITEMS; ++j) {
            const uint32_t li = li0 + j * 32;
            kv[j] = li < tile_n ? (in ? __ldg(in + base + li) : base + li) : 0u;
        }
    };
    auto slot_of = [&](int j) { return j & 1 ? slot[j / 2] >> 16 : slot[j / 2] & 0xFFFFu; };
    load(J.kin);
    // ---- rank inside each warp's chunk (order: warp, item, lane)
#pragma unroll
    for (int j = 0; j < ITEMS; ++j) {
        const bool valid = li0 + j * 32 < tile_n;
        const uint32_t d = (kv[j] >> shift) & dmask;
        const uint32_t d0 = __shfl_sync(0xffffffffu, d, 0);
        uint32_t peers;
        if (__all_sync(0xffffffffu, valid && d == d0)) {
            peers = 0xffffffffu;
        } else {
            if (valid) atomicOr(wm + d, 1u << lane);
            __syncwarp();
            peers = valid ? wm[d] : 0u;
        }
        const uint32_t cur = valid ? wc[d] : 0;
        __syncwarp();
        const uint32_t r = cur + __popc(peers & lt);
        slot[j / 2] = j & 1 ? slot[j / 2] | (r << 16) : r;
        if (valid && (peers & lt) == 0) { wc[d] = (uint16_t)(cur + __popc(peers)); wm[d] = 0; }
        __syncwarp();
    }
    __syncthreads();
    // ---- per digit (thread d): the tile's count published, the exclusive scans
    // over the digits of it and of the whole array's counts, and where each
    // warp's keys of the digit go in the tile
    uint32_t cnt = 0, tot = 0, ci = 0, ti = 0;
    const bool digit = t < (int)radix;
    if (t < OS_MAXRADIX) {
        if (digit) {
            for (int w = 0; w < OS_WARPS; ++w) cnt += s_wcnt[w * OS_MAXRADIX + t];
            *(volatile unsigned long long *)(state + (size_t)tile * OS_MAXRADIX + t) =
                (tile == 0 ? kTilePrefix : kTileSum) | cnt;
            tot = __ldg(hist + t);
        }
        ci = cnt;
        ti = tot;
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t y = __shfl_up_sync(0xffffffffu, ci, o), z = __shfl_up_sync(0xffffffffu, ti, o);
            if (lane >= o) { ci += y; ti += z; }
        }
        if (lane == 31) { s_wt[warp] = ci; s_wt[4 + warp] = ti; }
    }
    __syncthreads();
    uint32_t tex = 0, gbase = 0;   // the digit's start in the tile and in the output
    if (digit) {
        for (int w = 0; w < warp; ++w) { ci += s_wt[w]; ti += s_wt[4 + w]; }
        tex = ci - cnt;
        gbase = ti - tot;
        uint32_t run = tex;
        for (int w = 0; w < OS_WARPS; ++w) {
            const uint32_t c = s_wcnt[w * OS_MAXRADIX + t];
            s_wcnt[w * OS_MAXRADIX + t] = (uint16_t)run;
            run += c;
        }
    }
    __syncthreads();
    // ---- keys into their tile slots
#pragma unroll
    for (int j = 0; j < ITEMS; ++j) {
        if (li0 + j * 32 < tile_n) {
            const uint32_t pos = wc[(kv[j] >> shift) & dmask] + slot_of(j);
            s_buf[pos] = kv[j];
            slot[j / 2] = j & 1 ? (slot[j / 2] & 0xFFFFu) | (pos << 16) : (slot[j / 2] & 0xFFFF0000u) | pos;
        }
    }
    if (NP > 0) load(J.pin[0]);   // on its way while the tile looks back
    // ---- look back: the digit's keys in the tiles before this one, kLookback
    // tiles' words in flight at a time
    if (digit) {
        uint32_t before = 0;
        bool done = tile == 0;
        for (int64_t j = (int64_t)tile - 1; !done; j -= kLookback) {
            unsigned long long v[kLookback];
#pragma unroll
            for (int i = 0; i < kLookback; ++i)
                v[i] = j - i >= 0 ? *(volatile unsigned long long *)(state + (size_t)(j - i) * OS_MAXRADIX + t)
                                  : (unsigned long long)kTilePrefix;
#pragma unroll
            for (int i = 0; i < kLookback; ++i) {
                if (done) break;
                for (int it = 0; (v[i] >> 62) == 0; ++it) {
                    if (it >= kLookbackPolls) { latch(status, ST_TIMEOUT); done = true; break; }
                    __nanosleep(32);
                    v[i] = *(volatile unsigned long long *)(state + (size_t)(j - i) * OS_MAXRADIX + t);
                }
                before += (uint32_t)v[i];
                if ((v[i] >> 62) == 2) done = true;
            }
        }
        if (tile != 0)
            *(volatile unsigned long long *)(state + (size_t)tile * OS_MAXRADIX + t) = kTilePrefix | (before + cnt);
        s_gpos[t] = gbase + before - tex;
    }
    __syncthreads();
    // ---- keys out; this thread's slots t, t + OS_THREADS, ... and their output
    // positions stay the same for the payloads
    uint32_t g[ITEMS];
#pragma unroll
    for (int j = 0; j < ITEMS; ++j) {
        const uint32_t p = t + j * OS_THREADS;
        if (p < tile_n) {
            const uint32_t k = s_buf[p];
            g[j] = s_gpos[(k >> shift) & dmask] + p;
            if (g[j] < n) J.kout[g[j]] = k;
        }
    }
    // ---- payloads, one round each
#pragma unroll
    for (int a = 0; a < NP; ++a) {
        uint32_t *__restrict__ pout = J.pout[a];
        __syncthreads();   // the previous round's reads of s_buf are done
#pragma unroll
        for (int j = 0; j < ITEMS; ++j)
            if (li0 + j * 32 < tile_n) s_buf[slot_of(j)] = kv[j];
        if (a + 1 < NP) load(J.pin[a + 1]);
        __syncthreads();
#pragma unroll
        for (int j = 0; j < ITEMS; ++j) {
            const uint32_t p = t + j * OS_THREADS;
            if (p < tile_n) {
                const uint32_t v = s_buf[p];
                if (g[j] < n) pout[g[j]] = v;
                if (a == 0 && J.inv && v < n) J.inv[v] = g[j];
            }
        }
    }
}

// block-wide exclusive scan of two values per thread (512 entries)
__device__ __forceinline__ void os_block_scan512(uint32_t *vals /* smem [512] in/out */, uint32_t *warp_tot /* smem [8] */)
{
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    uint32_t a = vals[2 * t], b = vals[2 * t + 1];
    uint32_t s = a + b, incl = s;
    for (int o = 1; o < 32; o <<= 1) {
        uint32_t y = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += y;
    }
    if (lane == 31) warp_tot[warp] = incl;
    __syncthreads();
    if (warp == 0) {
        uint32_t w = lane < OS_WARPS ? warp_tot[lane] : 0, wi = w;
        for (int o = 1; o < 32; o <<= 1) {
            uint32_t y = __shfl_up_sync(0xffffffffu, wi, o);
            if (lane >= o) wi += y;
        }
        if (lane < OS_WARPS) warp_tot[lane] = wi - w;
    }
    __syncthreads();
    uint32_t ex = warp_tot[warp] + incl - s;
    vals[2 * t] = ex;
    vals[2 * t + 1] = ex + a;
    __syncthreads();
}

// ---- inverse of a permutation, written through buckets -------------------
// inv[perm[i]] = i as one pass of random 4-byte writes costs a DRAM read and
// write of a whole sector per element once the array is larger than L2.
// Instead the (perm[i], i) pairs are first grouped into buckets of 2^shift
// consecutive values (unstable: the order inside a bucket does not matter),
// then written bucket after bucket, so the writes in flight cover a few
// buckets' worth of inv and every sector is complete before it leaves L2.
constexpr int IB_MAXB = 512;
__global__ void k_inv_cursor(uint32_t *__restrict__ cursor, uint32_t nb, int shift)
{
    grid_wait();
    const uint32_t b = blockIdx.x * blockDim.x + threadIdx.x;
    if (b < nb) cursor[b] = b << shift;
}

// (perm is no permutation when a wait of its sort ran out: nothing is written then)
__global__ void __launch_bounds__(OS_THREADS, 4) k_inv_bucket(const uint32_t *__restrict__ perm, uint32_t n, int shift,
                                                               uint32_t nb, uint32_t *__restrict__ cursor,
                                                               uint32_t *__restrict__ tkey, uint32_t *__restrict__ tpos,
                                                               const uint32_t *status)
{
    grid_wait();
    const uint32_t stop = latched(status) & ST_TIMEOUT;
    __shared__ uint32_t s_cnt[IB_MAXB], s_base[IB_MAXB], s_wt[OS_WARPS];
    __shared__ uint32_t s_key[OS_TILE], s_pos[OS_TILE];
    const int t = threadIdx.x;
    const uint32_t base = blockIdx.x * OS_TILE;
    const uint32_t tile_n = min((uint32_t)OS_TILE, n - base);
    for (int b = t; b < IB_MAXB; b += OS_THREADS) s_cnt[b] = 0;
    uint32_t v[OS_ITEMS];
#pragma unroll
    for (int j = 0; j < OS_ITEMS; ++j) {
        const uint32_t i = base + j * OS_THREADS + t;
        v[j] = i < n ? __ldg(perm + i) : 0u;
    }
    if (stop) return;
    __syncthreads();
    uint32_t r[OS_ITEMS];   // rank inside the tile's bucket (shared atomics: any order)
#pragma unroll
    for (int j = 0; j < OS_ITEMS; ++j) {
        const uint32_t i = base + j * OS_THREADS + t;
        r[j] = i < n ? atomicAdd(&s_cnt[v[j] >> shift], 1u) : 0u;
    }
    __syncthreads();
    for (uint32_t b = t; b < nb; b += OS_THREADS) {
        const uint32_t c = s_cnt[b];
        s_base[b] = c ? atomicAdd(cursor + b, c) : 0u;
    }
    __syncthreads();
    os_block_scan512(s_cnt, s_wt);   // bucket starts inside the tile
#pragma unroll
    for (int j = 0; j < OS_ITEMS; ++j) {
        const uint32_t i = base + j * OS_THREADS + t;
        if (i < n) {
            const uint32_t p = s_cnt[v[j] >> shift] + r[j];
            s_key[p] = v[j];
            s_pos[p] = i;
        }
    }
    __syncthreads();
    for (uint32_t p = t; p < tile_n; p += OS_THREADS) {
        const uint32_t k = s_key[p], b = k >> shift;
        const uint32_t dst = s_base[b] + (p - s_cnt[b]);
        tkey[dst] = k;
        tpos[dst] = s_pos[p];
    }
}

// 4 x TM_INV_VECS pairs per thread: TM_INV_VECS 16-byte loads of each work
// array (256-byte aligned) in flight, at vectors i, i + blockDim, ...
#ifndef TM_INV_VECS
#define TM_INV_VECS 1   // 2 and 4 measured no faster
#endif
__global__ void k_inv_fill(const uint32_t *__restrict__ tkey, const uint32_t *__restrict__ tpos, uint32_t n,
                           uint32_t *__restrict__ inv, const uint32_t *status)
{
    grid_wait();
    const uint32_t stop = latched(status) & ST_TIMEOUT;   // the pairs were not written
    const uint64_t v0 = (uint64_t)blockIdx.x * blockDim.x * TM_INV_VECS + threadIdx.x;
    uint4 k[TM_INV_VECS], p[TM_INV_VECS];
#pragma unroll
    for (int r = 0; r < TM_INV_VECS; ++r) {
        const uint64_t i = (v0 + (uint64_t)r * blockDim.x) * 4;
        if (i + 4 <= n) {
            k[r] = __ldg(reinterpret_cast<const uint4 *>(tkey + i));
            p[r] = __ldg(reinterpret_cast<const uint4 *>(tpos + i));
        }
    }
    if (stop) return;
#pragma unroll
    for (int r = 0; r < TM_INV_VECS; ++r) {
        const uint64_t i = (v0 + (uint64_t)r * blockDim.x) * 4;
        if (i + 4 <= n) {
            inv[k[r].x] = p[r].x; inv[k[r].y] = p[r].y; inv[k[r].z] = p[r].z; inv[k[r].w] = p[r].w;
        } else {
            for (uint64_t j = i; j < n; ++j) inv[__ldg(tkey + j)] = __ldg(tpos + j);
        }
    }
}

int bits_for(uint64_t maxval)
{
    int b = 0;
    while (b < 64 && (maxval >> b) != 0) ++b;
    return b;
}

DigitPlan digit_plan(int bits)
{
    DigitPlan D;
    D.npass = (bits + OS_MAXBITS - 1) / OS_MAXBITS;
    for (int pass = 0, sh = 0; pass < D.npass; ++pass) {
        const int left = D.npass - pass, pb = (bits - sh + left - 1) / left;
        D.sh[pass] = sh;
        D.bits[pass] = pb;
        sh += pb;
    }
    return D;
}

// inv[perm[i]] = i for a permutation perm of [0, n); tkey/tpos are n-entry
// work arrays (allocated here when null).
static int inverse_perm(tm_ctx *ctx, const uint32_t *perm, uint32_t n, uint32_t *inv, uint32_t *tkey, uint32_t *tpos)
{
    ScratchScope scope(ctx);
    if (n == 0) return TM_OK;
    if (!tkey) tkey = (uint32_t *)salloc(ctx, (size_t)n * 4);
    if (!tpos) tpos = (uint32_t *)salloc(ctx, (size_t)n * 4);
    uint32_t *cursor = (uint32_t *)salloc(ctx, IB_MAXB * 4);
    if (!tkey || !tpos || !cursor) return TM_E_NOMEM;
    int shift = 0;
    while (((uint64_t)(n - 1) >> shift) >= (uint64_t)IB_MAXB) ++shift;
    const uint32_t nb = (uint32_t)(((uint64_t)(n - 1) >> shift) + 1);
    launch(ctx, k_inv_cursor, 1, IB_MAXB, cursor, nb, shift);
    launch(ctx, k_inv_bucket, (n + OS_TILE - 1) / OS_TILE, OS_THREADS, perm, n, shift, nb, cursor, tkey, tpos,
           (const uint32_t *)ctx->status);
    launch(ctx, k_inv_fill, (unsigned)(((uint64_t)n + 1024 * TM_INV_VECS - 1) / (1024 * TM_INV_VECS)), 256,
           (const uint32_t *)tkey, (const uint32_t *)tpos, n, inv, (const uint32_t *)ctx->status);
    return check_cuda(ctx, cudaGetLastError(), "inverse permutation");
}
// Up to here the last pass writes the inverse itself, a random 4-byte store per
// element: the array stays in L2 (64 MB of it), where a partial sector costs
// nothing more, and two launches and 12 bytes per element are saved.
// (1e7 keys: 56 us more in the pass against 97 for the two kernels; 5e7: about
// 1.3 ms against 0.5.)
constexpr uint32_t kInvDirect = 16000000;

// A stable LSD sort of the key and up to four payloads by the low `bits` bits
// of the key, from read-only inputs into separate outputs (no copies): the
// passes alternate between the outputs and scratch so that the last one writes
// the outputs.  A null p[0] input with an output gives payload 0 = the input
// index (the sorting permutation).  Outputs must not alias inputs.
struct RsTo {
    const uint32_t *key_in = nullptr, *p_in[4] = {};
    uint32_t *key = nullptr, *p[4] = {};
    uint32_t *inv = nullptr;          // optional: inv[payload 0] = sorted position (payload 0 = the input index)
    const uint32_t *hist = nullptr;   // the key's digit counts (OS_HIST), when they are known
};

__global__ void k_iota(uint32_t *__restrict__ a, uint32_t m)
{
    grid_wait();
    uint32_t i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < m) a[i] = i;
}

template <int ITEMS>
static int rs_pass(tm_ctx *ctx, const RsSet &J, int np, uint32_t n, int sh, int pb, const uint32_t *hist,
                   unsigned long long *state, uint32_t *ticket)
{
    const unsigned ntiles = (n + OS_THREADS * ITEMS - 1) / (OS_THREADS * ITEMS);
    auto go = [&](auto kernel) {
        launch(ctx, kernel, ntiles, OS_THREADS, J, n, sh, pb, hist, state, ticket, ctx->status);
        return check_cuda(ctx, cudaGetLastError(), "radix pass");
    };
    switch (np) {
    case 0: return go(k_rs_sweep<0, ITEMS>);
    case 1: return go(k_rs_sweep<1, ITEMS>);
    case 2: return go(k_rs_sweep<2, ITEMS>);
    case 3: return go(k_rs_sweep<3, ITEMS>);
    default: return go(k_rs_sweep<4, ITEMS>);
    }
}

int radix_sort_to(tm_ctx *ctx, const RsTo &x, uint32_t n, int bits)
{
    ScratchScope scope(ctx);
    if (n == 0) return TM_OK;
    int np = 0;
    while (np < 4 && x.p[np]) ++np;
    if (x.inv && x.p_in[0]) return set_err(ctx, TM_E_ARG, "internal: inverse of a sort with explicit payload 0");
    cudaStream_t st = ctx->stream;
    if (n <= 1 || bits <= 0) {   // every key equal: the identity order
        cudaMemcpyAsync(x.key, x.key_in, (size_t)n * 4, cudaMemcpyDeviceToDevice, st);
        for (int a = 0; a < np; ++a) {
            if (x.p_in[a]) cudaMemcpyAsync(x.p[a], x.p_in[a], (size_t)n * 4, cudaMemcpyDeviceToDevice, st);
            else launch(ctx, k_iota, (n + 255) / 256, 256, x.p[a], n);
        }
        if (x.inv) launch(ctx, k_iota, (n + 255) / 256, 256, x.inv, n);
        return TM_OK;
    }
    const DigitPlan D = digit_plan(bits);
    if (D.npass > OS_MAXPASS) return set_err(ctx, TM_E_LIMIT, "radix key wider than 32 bits");
    const bool small = n <= kSmallSort;
    const size_t ntiles = (n + (small ? OS_THREADS * OS_SMALL_ITEMS : OS_TILE) - 1) /
                          (small ? OS_THREADS * OS_SMALL_ITEMS : OS_TILE);
    // one buffer of tile words for each pass, cleared at once; a large sort's
    // passes share one (8 bytes x 128 per tile)
    const size_t words = ntiles * OS_MAXRADIX;
    const bool share = words * 8 * D.npass > ((size_t)32 << 20);
    const size_t state_bytes = words * 8 * (share ? 1 : D.npass);
    char *blk = (char *)salloc(ctx, state_bytes + 64 + OS_HIST * 4);
    if (!blk) return TM_E_NOMEM;
    unsigned long long *state = (unsigned long long *)blk;
    uint32_t *ticket = (uint32_t *)(blk + state_bytes);
    uint32_t *own_hist = ticket + 16;
    RsSet scr;
    if (D.npass >= 2) {
        if (!(scr.kout = (uint32_t *)salloc(ctx, (size_t)n * 4))) return TM_E_NOMEM;
        for (int a = 0; a < np; ++a)
            if (!(scr.pout[a] = (uint32_t *)salloc(ctx, (size_t)n * 4))) return TM_E_NOMEM;
    }
    cudaMemsetAsync(blk, 0, state_bytes + 64 + (x.hist ? 0 : OS_HIST * 4), st);
    if (!x.hist)
        launch(ctx, k_rs_hist, (unsigned)std::min<uint64_t>(((uint64_t)n + 4095) / 4096, (uint64_t)ctx->num_sms * 8),
               OS_THREADS, x.key_in, n, D, own_hist);
    const uint32_t *hist = x.hist ? x.hist : own_hist;
    RsSet J;
    J.kin = x.key_in;
    for (int a = 0; a < np; ++a) J.pin[a] = x.p_in[a];
    int rc = TM_OK;
    for (int pass = 0; pass < D.npass && rc == TM_OK; ++pass) {
        const bool last = pass == D.npass - 1;
        // pass i writes the outputs when npass - 1 - i is even, else scratch
        const bool to_dst = ((D.npass - 1 - pass) & 1) == 0;
        J.kout = to_dst ? x.key : scr.kout;
        for (int a = 0; a < np; ++a) J.pout[a] = to_dst ? x.p[a] : scr.pout[a];
        J.inv = last && n <= kInvDirect ? x.inv : nullptr;
        unsigned long long *st_p = state + (share ? 0 : words * pass);
        if (share && pass) cudaMemsetAsync(state, 0, state_bytes, st);
        const uint32_t *h = hist + pass * OS_MAXRADIX;
        rc = small ? rs_pass<OS_SMALL_ITEMS>(ctx, J, np, n, D.sh[pass], D.bits[pass], h, st_p, ticket + pass)
                   : rs_pass<OS_ITEMS>(ctx, J, np, n, D.sh[pass], D.bits[pass], h, st_p, ticket + pass);
        J.kin = J.kout;
        for (int a = 0; a < np; ++a) J.pin[a] = J.pout[a];
    }
    // the inverse permutation of a large sort, through buckets; the scratch of
    // the passes (free once the last pass has written the outputs) holds the pairs
    if (rc == TM_OK && x.inv && n > kInvDirect) rc = inverse_perm(ctx, x.p[0], n, x.inv, scr.kout, scr.pout[0]);
    return rc;
}

// ---- input validation and t' -------------------------------------------
struct Stats {
    long long tmin, tmax;
    unsigned long long nself, nbad;
};

__global__ void k_input_stats(const uint32_t *__restrict__ src, const uint32_t *__restrict__ dst,
                              const int64_t *__restrict__ t, uint64_t m, uint32_t n, Stats *st)
{
    grid_wait();
    long long lo = LLONG_MAX, hi = LLONG_MIN;
    unsigned long long ns = 0, nb = 0;
    for (uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; i < m; i += (uint64_t)gridDim.x * blockDim.x) {
        uint32_t u = src[i], v = dst[i];
        if (u >= n || v >= n) { ++nb; continue; }
        if (u == v) { ++ns; continue; }
        long long x = t[i];
        lo = x < lo ? x : lo;
        hi = x > hi ? x : hi;
    }
    // warp, then block reduction: one set of atomics per block
    __shared__ long long s_lo[32], s_hi[32];
    __shared__ unsigned long long s_ns[32], s_nb[32];
    for (int pass = 0; pass < 2; ++pass) {
        for (int o = 16; o > 0; o >>= 1) {
            long long a = __shfl_down_sync(0xffffffffu, lo, o), b = __shfl_down_sync(0xffffffffu, hi, o);
            lo = a < lo ? a : lo; hi = b > hi ? b : hi;
            ns += __shfl_down_sync(0xffffffffu, ns, o);
            nb += __shfl_down_sync(0xffffffffu, nb, o);
        }
        if (pass == 1) break;
        const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = (blockDim.x + 31) >> 5;
        if (lane == 0) { s_lo[warp] = lo; s_hi[warp] = hi; s_ns[warp] = ns; s_nb[warp] = nb; }
        __syncthreads();
        if (warp != 0) return;
        lo = lane < nw ? s_lo[lane] : LLONG_MAX;
        hi = lane < nw ? s_hi[lane] : LLONG_MIN;
        ns = lane < nw ? s_ns[lane] : 0;
        nb = lane < nw ? s_nb[lane] : 0;
    }
    if (threadIdx.x == 0) {
        if (lo != LLONG_MAX) atomicMin(&st->tmin, lo);
        if (hi != LLONG_MIN) atomicMax(&st->tmax, hi);
        if (ns) atomicAdd(&st->nself, ns);
        if (nb) atomicAdd(&st->nbad, nb);
    }
}

// Elementwise kernels below take kElemItems elements per thread (i, i +
// blockDim, ...); one element per thread measured up to twice as slow.
#ifndef TM_ELEM_ITEMS
#define TM_ELEM_ITEMS 4
#endif
constexpr int kElemItems = TM_ELEM_ITEMS;

// keep flags for self-loop dropping
__global__ void k_keep_nonself(const uint32_t *__restrict__ src, const uint32_t *__restrict__ dst, uint64_t m,
                               uint32_t *__restrict__ keep)
{
    grid_wait();
    uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < m) keep[i] = src[i] != dst[i] ? 1u : 0u;
}

// Compact the kept tuples into (t', src, dst) u32 arrays, and count the digits
// of the sorts to come: of t' at hist, of src at hist + OS_HIST, of dst after
// that.  A few blocks per SM stride over the input, so that the counts of a
// block are added to the totals once.
__global__ void __launch_bounds__(OS_THREADS)
    k_compact_input(const uint32_t *__restrict__ src, const uint32_t *__restrict__ dst, const int64_t *__restrict__ t,
                    uint64_t m, const uint32_t *__restrict__ keep, const uint32_t *__restrict__ pos, long long tmin,
                    uint32_t *__restrict__ ot, uint32_t *__restrict__ os, uint32_t *__restrict__ od, DigitPlan Dt,
                    DigitPlan Dv, uint32_t *__restrict__ hist)
{
    grid_wait();
    __shared__ uint32_t h[3 * OS_HIST];
    for (int i = threadIdx.x; i < 3 * OS_HIST; i += OS_THREADS) h[i] = 0;
    __syncthreads();
    const uint64_t stride = (uint64_t)gridDim.x * OS_THREADS * kElemItems;
    for (uint64_t b = (uint64_t)blockIdx.x * OS_THREADS * kElemItems + threadIdx.x; b < m; b += stride) {
        uint32_t u[kElemItems], v[kElemItems];
        int64_t tt[kElemItems];
        bool k[kElemItems];
#pragma unroll
        for (int j = 0; j < kElemItems; ++j) {
            const uint64_t i = b + (uint64_t)j * OS_THREADS;
            k[j] = i < m && (!keep || keep[i]);
            if (k[j]) { u[j] = src[i]; v[j] = dst[i]; tt[j] = t[i]; }
        }
#pragma unroll
        for (int j = 0; j < kElemItems; ++j) {
            const uint64_t i = b + (uint64_t)j * OS_THREADS;
            if (!k[j]) continue;
            const uint32_t p = pos ? pos[i] : (uint32_t)i, x = (uint32_t)(tt[j] - tmin);
            ot[p] = x;
            os[p] = u[j];
            od[p] = v[j];
            hist_key(Dt, x, h);
            hist_key(Dv, u[j], h + OS_HIST);
            hist_key(Dv, v[j], h + 2 * OS_HIST);
        }
    }
    __syncthreads();
    hist_flush(h, 3 * OS_HIST, hist);
}

// After the GLOBAL sort: flag tuples equal to their predecessor.
// After a sort by t' alone: order each run of equal t' by (src, dst), and
// count the tuples equal to their predecessor (repeats lie inside a run), so
// the flags above are made only when there are repeats.  Runs
// of up to kRunMax edges are sorted by their head's thread; runs of up to
// kBlockRunMax are listed (start, length) for k_order_long_runs; a longer run
// is flagged and the caller sorts by all three keys instead.
constexpr uint32_t kRunMax = 32;
constexpr uint32_t kBlockRunMax = 4096;
__device__ __forceinline__ void order_run_at(uint32_t i, const uint32_t *__restrict__ t, uint32_t *__restrict__ s,
                                             uint32_t *__restrict__ d, uint32_t m, uint32_t *__restrict__ too_long,
                                             uint2 *__restrict__ long_runs, uint32_t *__restrict__ n_long,
                                             unsigned long long *__restrict__ ndup)
{
    if (i >= m || (i > 0 && t[i - 1] == t[i])) return;   // run heads only
    const uint32_t ti = t[i];
    uint32_t j = i + 1;
    while (j < m && t[j] == ti && j - i < kRunMax) ++j;
    if (j < m && t[j] == ti) {
        while (j < m && t[j] == ti && j - i <= kBlockRunMax) ++j;
        if (j - i > kBlockRunMax) atomicOr(too_long, 1u);
        else long_runs[atomicAdd(n_long, 1u)] = make_uint2(i, j - i);   // at most m / 33 runs
        return;
    }
    const uint32_t len = j - i;
    if (len < 2) return;
    if (len <= 4) {
        // most runs: a 4-key sorting network in registers (missing keys
        // padded with the largest value, which stay at the end)
        uint64_t k0 = ((uint64_t)s[i] << 32) | d[i], k1 = ((uint64_t)s[i + 1] << 32) | d[i + 1];
        uint64_t k2 = len > 2 ? ((uint64_t)s[i + 2] << 32) | d[i + 2] : ~0ull;
        uint64_t k3 = len > 3 ? ((uint64_t)s[i + 3] << 32) | d[i + 3] : ~0ull;
        auto cswap = [](uint64_t &a, uint64_t &b) { const uint64_t lo = a < b ? a : b, hi = a < b ? b : a; a = lo; b = hi; };
        cswap(k0, k1); cswap(k2, k3); cswap(k0, k2); cswap(k1, k3); cswap(k1, k2);
        s[i] = (uint32_t)(k0 >> 32); d[i] = (uint32_t)k0;
        s[i + 1] = (uint32_t)(k1 >> 32); d[i + 1] = (uint32_t)k1;
        if (len > 2) { s[i + 2] = (uint32_t)(k2 >> 32); d[i + 2] = (uint32_t)k2; }
        if (len > 3) { s[i + 3] = (uint32_t)(k3 >> 32); d[i + 3] = (uint32_t)k3; }
        const uint32_t dups = (k0 == k1) + (len > 2 && k1 == k2) + (len > 3 && k2 == k3);
        if (dups) atomicAdd(ndup, (unsigned long long)dups);
        return;
    }
    uint64_t key[kRunMax];
    for (uint32_t k = 0; k < len; ++k) key[k] = ((uint64_t)s[i + k] << 32) | d[i + k];
    for (uint32_t k = 1; k < len; ++k) {   // insertion sort
        const uint64_t x = key[k];
        uint32_t q = k;
        while (q > 0 && key[q - 1] > x) { key[q] = key[q - 1]; --q; }
        key[q] = x;
    }
    uint32_t dups = 0;
    for (uint32_t k = 0; k < len; ++k) {
        s[i + k] = (uint32_t)(key[k] >> 32); d[i + k] = (uint32_t)key[k];
        dups += k > 0 && key[k] == key[k - 1];
    }
    if (dups) atomicAdd(ndup, (unsigned long long)dups);
}

__global__ void k_order_runs(const uint32_t *__restrict__ t, uint32_t *__restrict__ s, uint32_t *__restrict__ d,
                             uint32_t m, uint32_t *__restrict__ too_long, uint2 *__restrict__ long_runs,
                             uint32_t *__restrict__ n_long, unsigned long long *__restrict__ ndup)
{
    grid_wait();
    const uint64_t i0 = (uint64_t)blockIdx.x * blockDim.x * kElemItems + threadIdx.x;
#pragma unroll
    for (int k = 0; k < kElemItems; ++k) {
        const uint64_t i = i0 + (uint64_t)k * blockDim.x;
        if (i >= m) break;
        order_run_at((uint32_t)i, t, s, d, m, too_long, long_runs, n_long, ndup);
    }
}

// One block per listed run (33 .. kBlockRunMax edges): bitonic sort of the
// (src, dst) keys in shared memory.  Blocks stride over the list, whose
// length is read on the device.
__global__ void __launch_bounds__(256) k_order_long_runs(uint32_t *__restrict__ s, uint32_t *__restrict__ d,
                                                         const uint2 *__restrict__ long_runs,
                                                         const uint32_t *__restrict__ n_long,
                                                         unsigned long long *__restrict__ ndup)
{
    grid_wait();
    __shared__ uint64_t key[kBlockRunMax];
    const uint32_t nl = *n_long;
    for (uint32_t r = blockIdx.x; r < nl; r += gridDim.x) {
        const uint2 run = long_runs[r];
        uint32_t P = 64;
        while (P < run.y) P <<= 1;
        for (uint32_t k = threadIdx.x; k < P; k += blockDim.x)
            key[k] = k < run.y ? (((uint64_t)s[run.x + k] << 32) | d[run.x + k]) : ~0ull;
        __syncthreads();
        for (uint32_t size = 2; size <= P; size <<= 1)
            for (uint32_t stride = size >> 1; stride > 0; stride >>= 1) {
                for (uint32_t k = threadIdx.x; k < P; k += blockDim.x) {
                    const uint32_t l = k ^ stride;
                    if (l > k) {
                        const bool up = (k & size) == 0;
                        const uint64_t a = key[k], b = key[l];
                        if ((a > b) == up) { key[k] = b; key[l] = a; }
                    }
                }
                __syncthreads();
            }
        uint32_t dups = 0;
        for (uint32_t k = threadIdx.x; k < run.y; k += blockDim.x) {
            s[run.x + k] = (uint32_t)(key[k] >> 32);
            d[run.x + k] = (uint32_t)key[k];
            dups += k > 0 && key[k] == key[k - 1];
        }
        if (dups) atomicAdd(ndup, (unsigned long long)dups);
        __syncthreads();
    }
}

__global__ void k_flag_unique(const uint32_t *__restrict__ t, const uint32_t *__restrict__ s,
                              const uint32_t *__restrict__ d, uint32_t m, uint32_t *__restrict__ keep,
                              unsigned long long *ndup)
{
    grid_wait();
    uint32_t i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= m) return;
    bool dup = i > 0 && t[i] == t[i - 1] && s[i] == s[i - 1] && d[i] == d[i - 1];
    keep[i] = dup ? 0u : 1u;
    if (dup) atomicAdd(ndup, 1ull);
}

__global__ void k_compact3(const uint32_t *__restrict__ a, const uint32_t *__restrict__ b,
                           const uint32_t *__restrict__ c, uint32_t m, const uint32_t *__restrict__ keep,
                           const uint32_t *__restrict__ pos, uint32_t *__restrict__ oa, uint32_t *__restrict__ ob,
                           uint32_t *__restrict__ oc)
{
    grid_wait();
    uint32_t i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= m || !keep[i]) return;
    uint32_t p = pos[i];
    oa[p] = a[i]; ob[p] = b[i]; oc[p] = c[i];
}


// The list offsets of a sorted key array, by the position at which a new key
// starts: off[v] = x for every v after the key before it and up to its own.
__device__ __forceinline__ void fill_offsets(uint32_t *__restrict__ off, uint32_t after, uint32_t upto, uint32_t n,
                                             uint32_t x)
{
    for (uint32_t v = after; v <= upto && v <= n; ++v) off[v] = x;
}

// Vertex lists of the out and in orders: the offsets of each vertex's list, and
// the owner-start bit sets (position x starts a new owner when its source
// (out) or destination (in) differs from position x - 1's).  A warp takes 32
// positions, whose ballots are one word of each set, and reads each key once
// (offsets and bit sets by separate kernels: 250 us on 5e7 edges, 164 like
// this; instructions bound it).
__global__ void k_owners(const uint32_t *__restrict__ out_src, const uint32_t *__restrict__ in_dst, uint32_t m,
                         uint32_t n, uint32_t words, uint32_t *__restrict__ out_off, uint32_t *__restrict__ in_off,
                         uint32_t *__restrict__ own_out, uint32_t *__restrict__ own_in,
                         const uint32_t *__restrict__ status)
{
    grid_wait();
    if (latched(status) & ST_TIMEOUT) return;   // a sort whose wait ran out: its keys are anything
    const int lane = threadIdx.x & 31;
    const uint64_t x0 = (uint64_t)blockIdx.x * blockDim.x * kElemItems + threadIdx.x;
    uint32_t k[2][kElemItems], kp[2][kElemItems];
#pragma unroll
    for (int r = 0; r < kElemItems; ++r) {
        const uint64_t x = x0 + (uint64_t)r * blockDim.x;
        k[0][r] = x < m ? __ldg(out_src + x) : 0u;
        k[1][r] = x < m ? __ldg(in_dst + x) : 0u;
        kp[0][r] = lane == 0 && x > 0 && x <= m ? __ldg(out_src + x - 1) : 0u;
        kp[1][r] = lane == 0 && x > 0 && x <= m ? __ldg(in_dst + x - 1) : 0u;
    }
#pragma unroll
    for (int r = 0; r < kElemItems; ++r) {
        // a warp's 32 positions are consecutive and start at a multiple of 32,
        // and words * 32 is a multiple of 32: whole warps leave together
        const uint64_t x = x0 + (uint64_t)r * blockDim.x;
        if (x >= (uint64_t)words * 32) break;
#pragma unroll
        for (int s = 0; s < 2; ++s) {
            const uint32_t up = __shfl_up_sync(0xffffffffu, k[s][r], 1);
            const uint32_t prev = lane == 0 ? kp[s][r] : up;
            const bool head = x < m && (x == 0 || k[s][r] != prev);
            const uint32_t w = __ballot_sync(0xffffffffu, head);
            if (lane == 0) (s ? own_in : own_out)[x >> 5] = w;
            if (head || x == m) fill_offsets(s ? in_off : out_off, x == 0 ? 0u : prev + 1u, x == m ? n : k[s][r], n, (uint32_t)x);
        }
    }
}

// The pairs of the multi-edge order (msrc, mdst: sorted source and destination
// of each position) in one pass: a position that starts a new pair is counted
// over the rows of its warp, the warps of its tile and, by look-back, the tiles
// before it, which numbers the pairs; their list starts, destinations, each
// source's first pair and the owner bits follow.  The number of pairs goes to
// *npairs.  The prefix moves through the tiles at about 32 per round trip to
// L2, so large arrays take tiles of 64 rows per warp and read the keys, which
// L2 still holds, again behind the look-back: 246 us on 5e7 edges (8 rows kept
// in registers 457; flags, their scan, fill and source offsets as separate
// kernels about 560).
constexpr int kPairChunk = 8;   // rows whose loads are in flight together
template <int ROWS>
__global__ void __launch_bounds__(256) k_pairs(const uint32_t *__restrict__ msrc, const uint32_t *__restrict__ mdst,
                                               uint32_t m, uint32_t n, unsigned long long *__restrict__ state,
                                               uint32_t *__restrict__ ticket, uint32_t *__restrict__ pair_off,
                                               uint32_t *__restrict__ pair_dst, uint32_t *__restrict__ vpair_off,
                                               uint32_t *__restrict__ own_multi, uint32_t *__restrict__ npairs,
                                               uint32_t *status)
{
    grid_wait();
    __shared__ uint32_t s_w[8], s_tile, s_before, s_h[8][ROWS];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (threadIdx.x == 0)   // a sort whose wait ran out: its keys are anything
        s_tile = (latched(status) & ST_TIMEOUT) ? 0xFFFFFFFFu : atomicAdd(ticket, 1u);
    __syncthreads();
    const uint32_t tile = s_tile;
    if (tile == 0xFFFFFFFFu) return;
    const uint64_t base = ((uint64_t)tile * 8 + warp) * (32 * ROWS);
    uint32_t u[kPairChunk], v[kPairChunk], pu, pv;   // a chunk of rows, and the keys before it
    auto load = [&](uint64_t x0) {
#pragma unroll
        for (int r = 0; r < kPairChunk; ++r) {
            const uint64_t x = x0 + r * 32 + lane;
            u[r] = x < m ? __ldg(msrc + x) : 0u;
            v[r] = x < m ? __ldg(mdst + x) : 0u;
        }
        pu = x0 > 0 && x0 <= m ? __ldg(msrc + x0 - 1) : 0u;
        pv = x0 > 0 && x0 <= m ? __ldg(mdst + x0 - 1) : 0u;
    };
    uint32_t mine = 0;
    for (int c = 0; c < ROWS; c += kPairChunk) {
        load(base + c * 32);
#pragma unroll
        for (int r = 0; r < kPairChunk; ++r) {
            const uint64_t x = base + (c + r) * 32 + lane;
            uint32_t a = __shfl_up_sync(0xffffffffu, u[r], 1), b = __shfl_up_sync(0xffffffffu, v[r], 1);
            if (lane == 0) { a = pu; b = pv; }
            pu = __shfl_sync(0xffffffffu, u[r], 31);
            pv = __shfl_sync(0xffffffffu, v[r], 31);
            const uint32_t h = __ballot_sync(0xffffffffu, x < m && (x == 0 || u[r] != a || v[r] != b));
            mine += __popc(h);
            if (lane == 0) {
                s_h[warp][c + r] = h;
                if (x <= m) own_multi[x >> 5] = h;
            }
        }
    }
    if (lane == 0) s_w[warp] = mine;
    __syncthreads();
    if (warp == 0) {
        uint32_t sum = 0;
        for (int w = 0; w < 8; ++w) sum += s_w[w];
        if (lane == 0) *(volatile unsigned long long *)(state + tile) = (tile == 0 ? kTilePrefix : kTileSum) | sum;
        uint32_t before = 0;
        for (int64_t j = (int64_t)tile - 1 - lane; tile != 0; j -= 32) {   // lane i at the i-th tile before
            unsigned long long x = kTilePrefix;
            if (j >= 0) {
                x = *(volatile unsigned long long *)(state + j);
                for (int it = 0; (x >> 62) == 0 && it < kLookbackPolls; ++it) {
                    __nanosleep(32);
                    x = *(volatile unsigned long long *)(state + j);
                }
                if ((x >> 62) == 0) { latch(status, ST_TIMEOUT); x = kTilePrefix; }
            }
            const unsigned end = __ballot_sync(0xffffffffu, (x >> 62) == 2);
            const int last = end ? __ffs((int)end) - 1 : 31;
            before += __reduce_add_sync(0xffffffffu, lane <= last ? (uint32_t)x : 0u);
            if (end) break;
        }
        if (lane == 0) {
            if (tile != 0) *(volatile unsigned long long *)(state + tile) = kTilePrefix | (before + sum);
            s_before = before;
        }
    }
    __syncthreads();
    uint32_t pid = s_before;   // pairs before the row
    for (int w = 0; w < warp; ++w) pid += s_w[w];
    for (int c = 0; c < ROWS; c += kPairChunk) {
        if (ROWS > kPairChunk || c > 0) load(base + c * 32);
        else pu = base > 0 && base <= m ? __ldg(msrc + base - 1) : 0u;
#pragma unroll
        for (int r = 0; r < kPairChunk; ++r) {
            const uint64_t x = base + (c + r) * 32 + lane;
            uint32_t a = __shfl_up_sync(0xffffffffu, u[r], 1);
            if (lane == 0) a = pu;
            pu = __shfl_sync(0xffffffffu, u[r], 31);
            const uint32_t h = s_h[warp][c + r];
            const uint32_t id = pid + __popc(h & ((1u << lane) - 1u));
            const bool head = (h >> lane) & 1u;
            if (head) {
                pair_off[id] = (uint32_t)x;
                pair_dst[id] = v[r];
                if (x == 0 || u[r] != a) fill_offsets(vpair_off, x == 0 ? 0u : a + 1u, u[r], n, id);
            }
            if (x == m - 1) {   // after the last pair
                const uint32_t end = id + (head ? 1u : 0u);
                pair_off[end] = m;
                *npairs = end;
                fill_offsets(vpair_off, u[r] + 1u, n, n, end);
            }
            pid += __popc(h);
        }
    }
}
// rows per warp: small arrays need the blocks more than the fewer tiles
constexpr int kPairRowsSmall = 8, kPairRowsLarge = 64;
constexpr uint32_t kPairSmall = 4000000;   // 244 tiles of the larger size: about one for each SM
inline uint32_t pair_tiles(uint32_t m) { return m / (256 * (m <= kPairSmall ? kPairRowsSmall : kPairRowsLarge)) + 1; }

// where each list time falls in the same vertex's other list
// Cross ranks of both lists (blockIdx.y = 0: out-list entries into the
// owner's in-list; 1: in-list entries into the owner's out-list).
struct XR {
    const uint32_t *own_t, *owner, *other_off, *other_t;
    uint32_t *xrank;
};
// A thread takes kXrItems consecutive entries: the first is searched for in the
// whole of its owner's other list, the next ones of the same owner from there
// on (their times do not fall), which takes a probe or two.
// 5e7 edges: 797 us with four separate searches in lockstep per thread, 566 with
// four consecutive entries, 481 with eight; 2e6 edges 34, 29 and 31.
template <int kXrItems>
__global__ void __launch_bounds__(256) k_cross_rank(XR a, XR b, uint32_t m, const uint32_t *status)
{
    grid_wait();
    const uint32_t stop = latched(status) & ST_TIMEOUT;   // the list offsets were not written
    const bool s1 = blockIdx.y != 0;
    const uint32_t *__restrict__ own_t = s1 ? b.own_t : a.own_t, *__restrict__ owner = s1 ? b.owner : a.owner;
    const uint32_t *__restrict__ other_off = s1 ? b.other_off : a.other_off, *__restrict__ other_t = s1 ? b.other_t : a.other_t;
    uint32_t *__restrict__ xrank = s1 ? b.xrank : a.xrank;
    const uint64_t i0 = ((uint64_t)blockIdx.x * blockDim.x + threadIdx.x) * kXrItems;
    if (i0 >= m) return;
    uint32_t z[kXrItems], t[kXrItems], r[kXrItems];
    const bool whole = i0 + kXrItems <= m;   // (the arrays are 256-byte aligned)
#pragma unroll
    for (int k = 0; k < kXrItems; k += 4) {
        if (whole) {
            const uint4 vz = __ldg(reinterpret_cast<const uint4 *>(owner + i0 + k)), vt = __ldg(reinterpret_cast<const uint4 *>(own_t + i0 + k));
            z[k] = vz.x; z[k + 1] = vz.y; z[k + 2] = vz.z; z[k + 3] = vz.w;
            t[k] = vt.x; t[k + 1] = vt.y; t[k + 2] = vt.z; t[k + 3] = vt.w;
        } else {
            for (int j = k; j < k + 4; ++j) {
                z[j] = __ldg(owner + min(i0 + j, (uint64_t)m - 1));
                t[j] = __ldg(own_t + min(i0 + j, (uint64_t)m - 1));
            }
        }
    }
    if (stop) return;
    uint32_t lo = 0, hi = 0;
#pragma unroll
    for (int k = 0; k < kXrItems; ++k) {
        if (k == 0 || z[k] != z[k - 1]) {
            lo = __ldg(other_off + z[k]);
            hi = __ldg(other_off + z[k] + 1);
            lo = lower_idx(other_t, lo, hi, t[k]);
        } else if (t[k] != t[k - 1]) {
            lo = gallop_idx(other_t, lo, hi, t[k]);
        }
        r[k] = lo;
    }
#pragma unroll
    for (int k = 0; k < kXrItems; k += 4) {
        if (whole) *reinterpret_cast<uint4 *>(xrank + i0 + k) = make_uint4(r[k], r[k + 1], r[k + 2], r[k + 3]);
        else
            for (int j = k; j < k + 4; ++j)
                if (i0 + j < m) xrank[i0 + j] = r[j];
    }
}

inline unsigned blocks_for(uint64_t n, int threads) { return (unsigned)((n + threads - 1) / threads); }

}  // namespace

// Graph arrays come from a few large blocks (one allocator call each), cut
// into 256-byte aligned arrays.
struct GraphBlock {
    char *base = nullptr;
    size_t size = 0, off = 0;
};

static size_t align256(size_t b) { return (b + 255) / 256 * 256; }

static bool gblock_open(tm_ctx *ctx, GraphBlock &b, size_t bytes)
{
    b.size = bytes ? bytes : 256;
    b.off = 0;
    b.base = (char *)dalloc(ctx, b.size);
    if (b.base) ctx->graph_bufs.push_back({b.base, b.size});
    return b.base != nullptr;
}

static uint32_t *gtake(GraphBlock &b, size_t count)
{
    size_t bytes = align256((count ? count : 1) * sizeof(uint32_t));
    if (b.off + bytes > b.size) return nullptr;
    uint32_t *p = (uint32_t *)(b.base + b.off);
    b.off += bytes;
    return p;
}

// The build's status as last copied.
static int build_status(tm_ctx *ctx)
{
    const uint32_t bits = *ctx->status_host;
    return bits ? set_err(ctx, TM_E_CUDA, "CSR build: device status " + std::to_string(bits)) : TM_OK;
}

int build_csr(tm_ctx *ctx)
{
    ScratchScope scope(ctx);
    GraphBlock gb;
    const int TB = 256;
    cudaStream_t st = ctx->stream;
    uint64_t m0 = ctx->m_in;
    uint32_t n = ctx->n;
    DevGraph &g = ctx->g;
    g = DevGraph();
    g.n = n;
    int rc = TM_OK;
    // ---- statistics: t range, self loops, bad ids
    std::unique_ptr<PhaseScope> sec(new PhaseScope(ctx, TM_PH_CSR_STATS));
    // (in the status block, which the copy clears: pinned both ways)
    static_assert(16 + sizeof(Stats) <= kStatusBytes, "the statistics fit the status block");
    Stats hs{LLONG_MAX, LLONG_MIN, 0, 0};
    Stats *ds = (Stats *)(ctx->status + 4);
    memset(ctx->status_host, 0, kStatusBytes);
    memcpy(ctx->status_host + 4, &hs, sizeof(Stats));
    copy_h2d(ctx, ctx->status, ctx->status_host, kStatusBytes);
    if (m0) {
        unsigned nb = std::min<uint64_t>(blocks_for(m0, TB), (uint64_t)ctx->num_sms * 8);
        launch(ctx, k_input_stats, nb, TB, ctx->in_src, ctx->in_dst, ctx->in_t, m0, n, ds);
    }
    copy_d2h(ctx, ctx->status_host, ctx->status, kStatusBytes);
    rc = check_cuda(ctx, cudaStreamSynchronize(st), "input statistics");
    if (rc) return rc;
    memcpy(&hs, ctx->status_host + 4, sizeof(Stats));
    if (hs.nbad) return set_err(ctx, TM_E_ARG, "vertex id >= n in input");
    if (hs.nself && !(ctx->load_flags & TM_DROP_SELF))
        return set_err(ctx, TM_E_SELFLOOP, "input has self loops (pass TM_DROP_SELF to drop them)");
    uint64_t m1 = m0 - hs.nself;
    if (m1 >= 0xFFFFFFFFull) return set_err(ctx, TM_E_LIMIT, "more than 2^32-2 edges");
    long long tmin = m1 ? hs.tmin : 0, tmax = m1 ? hs.tmax : 0;
    // the span as an unsigned difference: no signed overflow at the int64 extremes
    if ((unsigned long long)tmax - (unsigned long long)tmin >= 0xFFFFFFFFull)
        return set_err(ctx, TM_E_LIMIT, "time span t_max - t_min must be below 2^32 - 1");
    uint32_t m = (uint32_t)m1;
    // ---- compact to (t', src, dst)
    uint32_t *T0 = (uint32_t *)salloc(ctx, (size_t)(m ? m : 1) * 4);
    uint32_t *S0 = (uint32_t *)salloc(ctx, (size_t)(m ? m : 1) * 4);
    uint32_t *D0 = (uint32_t *)salloc(ctx, (size_t)(m ? m : 1) * 4);
    if (!T0 || !S0 || !D0) return TM_E_NOMEM;
    int vbits = bits_for(n ? n - 1 : 0);
    int tbits = bits_for((unsigned long long)tmax - (unsigned long long)tmin);
    const DigitPlan Dt = digit_plan(tbits), Dv = digit_plan(vbits);
    // cleared together: digit counts of t', src, dst; the pair kernel's ticket
    // (16 words) and tile words
    uint32_t *hist = (uint32_t *)salloc(ctx, (3 * OS_HIST + 16) * 4 + ((size_t)m + 2047) / 2048 * 8 + 64);
    if (!hist) return TM_E_NOMEM;
    unsigned long long *pair_state = (unsigned long long *)(hist + 3 * OS_HIST + 16);
    cudaMemsetAsync(hist, 0, (3 * OS_HIST + 16) * 4 + ((size_t)m + 2047) / 2048 * 8 + 64, st);
    const unsigned cblk = (unsigned)std::min<uint64_t>(blocks_for((m0 + kElemItems - 1) / kElemItems, TB),
                                                       (uint64_t)ctx->num_sms * 8);
    if (hs.nself) {
        uint32_t *keep = (uint32_t *)salloc(ctx, m0 * 4), *pos = (uint32_t *)salloc(ctx, m0 * 4);
        if (!keep || !pos) return TM_E_NOMEM;
        launch(ctx, k_keep_nonself, blocks_for(m0, TB), TB, ctx->in_src, ctx->in_dst, m0, keep);
        rc = exclusive_scan_u32(ctx, keep, pos, m0, nullptr);
        if (rc) return rc;
        launch(ctx, k_compact_input, cblk, TB, ctx->in_src, ctx->in_dst, ctx->in_t, m0, keep, pos, tmin, T0, S0, D0,
               Dt, Dv, hist);
    } else if (m) {
        launch(ctx, k_compact_input, cblk, TB, ctx->in_src, ctx->in_dst, ctx->in_t, m0, nullptr, nullptr, tmin, T0,
               S0, D0, Dt, Dv, hist);
    }
    // every m- and n-sized array of the graph in one block, sized before the
    // duplicates are known (they are rare; their slots stay unused)
    {
        const size_t mf = (size_t)m, a_m = align256((mf ? mf : 1) * 4), a_n = align256(((size_t)n + 1) * 4);
        const size_t a_b = align256((mf / 32 + 1) * 4);
        // (the pair tables are sized by m too: the pair count is read only at the end)
        if (!gblock_open(ctx, gb, 20 * a_m + 256 + 3 * a_n + 3 * a_b)) return TM_E_NOMEM;
    }
    g.g_t = gtake(gb, m); g.g_src = gtake(gb, m); g.g_dst = gtake(gb, m);
    if (!g.g_t || !g.g_src || !g.g_dst) return TM_E_NOMEM;
    // ---- GLOBAL order (t', src, dst): LSD by t' straight into the graph's
    // arrays, then each run of equal t' ordered by (src, dst) in place; a run
    // longer than kBlockRunMax sends the whole array through the full LSD sort
    // by dst, src and t' instead
    sec.reset();
    sec.reset(new PhaseScope(ctx, TM_PH_CSR_GLOBAL));
    {
        RsTo ts{T0, {S0, D0}, g.g_t, {g.g_src, g.g_dst}};
        ts.hist = hist;
        rc = radix_sort_to(ctx, ts, m, tbits);
        if (rc) return rc;
    }
    // ---- duplicates (and the run check, read with the same copy)
    {
        uint32_t *keep = (uint32_t *)salloc(ctx, (size_t)(m ? m : 1) * 4);
        // [0] duplicates, [1] a run too long, [2] number of listed runs
        unsigned long long *nd = (unsigned long long *)(ctx->status + 4);
        uint2 *long_runs = (uint2 *)salloc(ctx, ((size_t)m / (kRunMax + 1) + 1) * sizeof(uint2));
        if (!keep || !long_runs) return TM_E_NOMEM;
        cudaMemsetAsync(nd, 0, 24, st);
        if (m) {
            launch(ctx, k_order_runs, blocks_for(((uint64_t)m + kElemItems - 1) / kElemItems, TB), TB,
                   (const uint32_t *)g.g_t, g.g_src, g.g_dst, m,
                   (uint32_t *)(nd + 1), long_runs, (uint32_t *)(nd + 2), nd);
            launch(ctx, k_order_long_runs, (unsigned)ctx->num_sms * 2, 256, g.g_src, g.g_dst, (const uint2 *)long_runs,
                   (const uint32_t *)(nd + 2), nd);
        }
        unsigned long long hnd[2] = {0, 0};
        copy_d2h(ctx, ctx->status_host, ctx->status, kStatusBytes);
        rc = check_cuda(ctx, cudaStreamSynchronize(st), "duplicate scan");
        if (rc || (rc = build_status(ctx))) return rc;
        memcpy(hnd, ctx->status_host + 4, 16);
        if (hnd[1]) {
            // (the work arrays hold the same tuples in input order)
            const RsTo by_dst{D0, {S0, T0}, g.g_dst, {g.g_src, g.g_t}}, by_src{g.g_src, {g.g_dst, g.g_t}, S0, {D0, T0}},
                by_t{T0, {S0, D0}, g.g_t, {g.g_src, g.g_dst}};
            rc = radix_sort_to(ctx, by_dst, m, vbits);
            if (!rc) rc = radix_sort_to(ctx, by_src, m, vbits);
            if (!rc) rc = radix_sort_to(ctx, by_t, m, tbits);
            if (rc) return rc;
            cudaMemsetAsync(nd, 0, 8, st);
            launch(ctx, k_flag_unique, blocks_for(m, TB), TB, g.g_t, g.g_src, g.g_dst, m, keep, nd);
            copy_d2h(ctx, ctx->status_host, ctx->status, kStatusBytes);
            rc = check_cuda(ctx, cudaStreamSynchronize(st), "duplicate scan");
            if (rc || (rc = build_status(ctx))) return rc;
            memcpy(hnd, ctx->status_host + 4, 8);
        }
        const unsigned long long ndup = hnd[0];
        if (ndup && !(ctx->load_flags & TM_DEDUP)) {
            return set_err(ctx, TM_E_DUP, "input repeats a (u,v,t) tuple (pass TM_DEDUP to drop repeats)");
        }
        if (ndup && !hnd[1]) {   // the run kernels only counted the repeats: flag them (same count)
            cudaMemsetAsync(nd, 0, 8, st);
            launch(ctx, k_flag_unique, blocks_for(m, TB), TB, g.g_t, g.g_src, g.g_dst, m, keep, nd);
        }
        if (ndup) {
            // compact into the work arrays, then back
            uint32_t *pos = (uint32_t *)salloc(ctx, (size_t)m * 4);
            if (!pos) return TM_E_NOMEM;
            rc = exclusive_scan_u32(ctx, keep, pos, m, nullptr);
            if (rc) return rc;
            launch(ctx, k_compact3, blocks_for(m, TB), TB, g.g_t, g.g_src, g.g_dst, m, keep, pos, T0, S0, D0);
            const size_t bytes = (size_t)(m - ndup) * 4;
            cudaMemcpyAsync(g.g_t, T0, bytes, cudaMemcpyDeviceToDevice, st);
            cudaMemcpyAsync(g.g_src, S0, bytes, cudaMemcpyDeviceToDevice, st);
            cudaMemcpyAsync(g.g_dst, D0, bytes, cudaMemcpyDeviceToDevice, st);
        }
        m = (uint32_t)(m - ndup);
        if (ndup) {   // the counts of the endpoints' digits without the repeats
            cudaMemsetAsync(hist + OS_HIST, 0, 2 * OS_HIST * 4, st);
            const unsigned hb = (unsigned)std::min<uint64_t>(((uint64_t)m + 4095) / 4096, (uint64_t)ctx->num_sms * 8);
            launch(ctx, k_rs_hist, hb, OS_THREADS, (const uint32_t *)g.g_src, m, Dv, hist + OS_HIST);
            launch(ctx, k_rs_hist, hb, OS_THREADS, (const uint32_t *)g.g_dst, m, Dv, hist + 2 * OS_HIST);
        }
    }
    g.m = m;
    g.tmin = tmin;
    g.T = (uint32_t)((unsigned long long)tmax - (unsigned long long)tmin);
    // S0/D0/T0 are reused below as work space
    // ---- OUT and IN orders: stable sorts of gid by src and by dst, run as
    // one two-array sort; the sorted keys are out_src and in_dst themselves
    sec.reset();
    sec.reset(new PhaseScope(ctx, TM_PH_CSR_OUT));
    g.out_gid = gtake(gb, m); g.out_t = gtake(gb, m); g.out_nbr = gtake(gb, m); g.out_off = gtake(gb, (size_t)n + 1);
    g.in_gid = gtake(gb, m); g.in_t = gtake(gb, m); g.in_nbr = gtake(gb, m); g.in_off = gtake(gb, (size_t)n + 1);
    g.out_src = gtake(gb, m); g.in_dst = gtake(gb, m);
    g.out_xrank = gtake(gb, m); g.in_xrank = gtake(gb, m); g.out_pos = gtake(gb, m); g.in_pos = gtake(gb, m);
    if (!g.out_gid || !g.out_t || !g.out_nbr || !g.out_off || !g.in_gid || !g.in_t || !g.in_nbr || !g.in_off ||
        !g.out_src || !g.in_dst || !g.out_xrank || !g.in_xrank || !g.out_pos || !g.in_pos)
        return TM_E_NOMEM;
    g.in_to_out = gtake(gb, m);
    if (!g.in_to_out) return TM_E_NOMEM;
    if (m) {
        // payloads: the input index (gid), t' and the other endpoint, so every
        // list array comes out of the sort (no gathers); the last pass also
        // writes each edge's list position by gid (the inverse permutation).
        // The in-list sort then carries each edge's out-list position (read in
        // GLOBAL order), which gives the in -> out map directly.
        RsTo os{g.g_src, {nullptr, g.g_t, g.g_dst}, g.out_src, {g.out_gid, g.out_t, g.out_nbr}};
        os.inv = g.out_pos; os.hist = hist + OS_HIST;
        rc = radix_sort_to(ctx, os, m, vbits);
        if (rc) return rc;
        RsTo is{g.g_dst, {nullptr, g.g_t, g.g_src, g.out_pos}, g.in_dst, {g.in_gid, g.in_t, g.in_nbr, g.in_to_out}};
        is.inv = g.in_pos; is.hist = hist + 2 * OS_HIST;
        rc = radix_sort_to(ctx, is, m, vbits);
        if (rc) return rc;
    }
    sec.reset();
    sec.reset(new PhaseScope(ctx, TM_PH_CSR_IN));
    g.own_out = gtake(gb, (size_t)m / 32 + 1); g.own_in = gtake(gb, (size_t)m / 32 + 1);
    g.own_multi = gtake(gb, (size_t)m / 32 + 1);
    if (!g.own_out || !g.own_in || !g.own_multi) return TM_E_NOMEM;
    const uint32_t words = m / 32 + 1;
    launch(ctx, k_owners, blocks_for(((uint64_t)words * 32 + kElemItems - 1) / kElemItems, TB), TB, g.out_src, g.in_dst,
           m, n, words, g.out_off, g.in_off, g.own_out, g.own_in, ctx->status);
    uint32_t *key = S0, *tmp = D0;
    // ---- multi-edge order: stable re-sort of the IN order by source
    sec.reset();
    sec.reset(new PhaseScope(ctx, TM_PH_CSR_MULTI));
    g.multi_t = gtake(gb, m);
    g.multi_to_out = gtake(gb, m);
    g.vpair_off = gtake(gb, (size_t)n + 1);
    if (!g.multi_t || !g.vpair_off || !g.multi_to_out) return TM_E_NOMEM;
    uint32_t np = 0;
    if (m) {
        {
            // payloads: t', the destination and each entry's out-list
            // position, straight into the multi-edge arrays
            RsTo ms{g.in_nbr, {g.in_t, g.in_dst, g.in_to_out}, key, {g.multi_t, tmp, g.multi_to_out}};
            ms.hist = hist + OS_HIST;   // the sources again
            rc = radix_sort_to(ctx, ms, m, vbits);
            if (rc) return rc;
        }
        // key = pair src, tmp = pair dst per multi position; the pair tables
        // are m-sized slots of the graph block, the pair count stays on the
        // device until the closing synchronize
        g.pair_off = gtake(gb, (size_t)m + 1);
        g.pair_dst = gtake(gb, m);
        if (!g.pair_off || !g.pair_dst) return TM_E_NOMEM;
        launch(ctx, m <= kPairSmall ? k_pairs<kPairRowsSmall> : k_pairs<kPairRowsLarge>, pair_tiles(m), 256,
               (const uint32_t *)key, (const uint32_t *)tmp, m, n, pair_state, hist + 3 * OS_HIST, g.pair_off,
               g.pair_dst, g.vpair_off, g.own_multi, ctx->status + 1, ctx->status);
        // cross ranks between a vertex's out- and in-lists
        const int per = m <= kPairSmall ? 4 : 8;
        launch(ctx, per == 4 ? k_cross_rank<4> : k_cross_rank<8>, dim3(blocks_for(((uint64_t)m + per - 1) / per, TB), 2), TB,
               XR{g.out_t, g.out_src, g.in_off, g.in_t, g.out_xrank},
               XR{g.in_t, g.in_dst, g.out_off, g.out_t, g.in_xrank}, m, (const uint32_t *)ctx->status);
    } else {
        GraphBlock pbk;
        if (!gblock_open(ctx, pbk, 3 * 256)) return TM_E_NOMEM;
        g.pair_off = gtake(pbk, 1);
        g.pair_dst = gtake(pbk, 1);
        cudaMemsetAsync(g.pair_off, 0, 4, st);
        cudaMemsetAsync(g.vpair_off, 0, ((size_t)n + 1) * 4, st);
    }
    uint32_t bits = 0;
    int rc2 = read_status(ctx, &bits);   // the build's one closing synchronize
    if (rc2) return rc2;
    if (m) np = ctx->status_host[1];   // copied with the status
    g.npairs = np;
    return build_status(ctx);
}

}  // namespace timest

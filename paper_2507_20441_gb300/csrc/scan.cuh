// Device-wide scans used by the CSR builder and the weight pass.
//
// * exclusive_scan_u32: reduce-then-scan over u32 counts (recursive over the
//   tile totals), for compaction.
// * segmented_scan2_u64: inclusive prefix sums that restart at segment heads,
//   with every 64-bit addition inside a segment checked for wrap-around, in one
//   pass with a bounded look-back between tiles.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "tm_device.cuh"
#include "tm_internal.h"

namespace timest {
namespace {

constexpr int SCAN_THREADS = 256;
constexpr int SCAN_ITEMS = 8;
constexpr int SCAN_TILE = SCAN_THREADS * SCAN_ITEMS;

// ---------------------------------------------------------------- u32 ----
__global__ void k_tile_sum_u32(const uint32_t *__restrict__ in, uint64_t n, uint32_t *__restrict__ tile_sum)
{
    grid_wait();
    __shared__ uint32_t warp_sum[SCAN_THREADS / 32];
    uint64_t base = (uint64_t)blockIdx.x * SCAN_TILE;
    uint32_t s = 0;
#pragma unroll
    for (int j = 0; j < SCAN_ITEMS; ++j) {
        uint64_t i = base + (uint64_t)j * SCAN_THREADS + threadIdx.x;
        if (i < n) s += in[i];
    }
    for (int o = 16; o > 0; o >>= 1) s += __shfl_down_sync(0xffffffffu, s, o);
    if ((threadIdx.x & 31) == 0) warp_sum[threadIdx.x >> 5] = s;
    __syncthreads();
    if (threadIdx.x < 32) {
        uint32_t v = threadIdx.x < SCAN_THREADS / 32 ? warp_sum[threadIdx.x] : 0;
        for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
        if (threadIdx.x == 0) tile_sum[blockIdx.x] = v;
    }
}

// Exclusive scan of one tile with a carry-in taken from carry[blockIdx.x]
// (or 0 when carry is null); blocked layout (each thread SCAN_ITEMS
// consecutive values).  Writes the grand total to *total when it is the last
// tile and total is non-null.
// With tile_sums non-null the carry-in is instead the sum of the unscanned
// tile totals tile_sums[0 .. blockIdx.x), added up by the block itself.
__global__ void k_tile_scan_u32(const uint32_t *__restrict__ in, uint64_t n, const uint32_t *__restrict__ carry,
                                uint32_t *__restrict__ out, uint32_t *__restrict__ total,
                                const uint32_t *__restrict__ tile_sums = nullptr)
{
    grid_wait();
    __shared__ uint32_t warp_tot[SCAN_THREADS / 32];
    __shared__ uint32_t s_carry;
    if (tile_sums) {
        uint32_t c = 0;
        for (uint32_t i = threadIdx.x; i < blockIdx.x; i += SCAN_THREADS) c += tile_sums[i];
        for (int o = 16; o > 0; o >>= 1) c += __shfl_down_sync(0xffffffffu, c, o);
        if ((threadIdx.x & 31) == 0) warp_tot[threadIdx.x >> 5] = c;
        __syncthreads();
        if (threadIdx.x == 0) {
            uint32_t t = 0;
            for (int w = 0; w < SCAN_THREADS / 32; ++w) t += warp_tot[w];
            s_carry = t;
        }
        __syncthreads();
    }
    uint64_t base = (uint64_t)blockIdx.x * SCAN_TILE + (uint64_t)threadIdx.x * SCAN_ITEMS;
    uint32_t v[SCAN_ITEMS];
    uint32_t s = 0;
#pragma unroll
    for (int j = 0; j < SCAN_ITEMS; ++j) {
        uint64_t i = base + j;
        v[j] = (i < n) ? in[i] : 0;
        s += v[j];
    }
    int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    uint32_t incl = s;
    for (int o = 1; o < 32; o <<= 1) {
        uint32_t y = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += y;
    }
    if (lane == 31) warp_tot[warp] = incl;
    __syncthreads();
    if (warp == 0) {
        uint32_t w = lane < SCAN_THREADS / 32 ? warp_tot[lane] : 0;
        uint32_t wi = w;
        for (int o = 1; o < 32; o <<= 1) {
            uint32_t y = __shfl_up_sync(0xffffffffu, wi, o);
            if (lane >= o) wi += y;
        }
        if (lane < SCAN_THREADS / 32) warp_tot[lane] = wi - w;
    }
    __syncthreads();
    uint32_t run = (tile_sums ? s_carry : carry ? carry[blockIdx.x] : 0) + warp_tot[warp] + incl - s;
#pragma unroll
    for (int j = 0; j < SCAN_ITEMS; ++j) {
        uint64_t i = base + j;
        if (i < n) out[i] = run;
        run += v[j];
    }
    if (total && blockIdx.x == gridDim.x - 1 && threadIdx.x == SCAN_THREADS - 1) *total = run;
}

// Exclusive scan of n u32 values (in may equal out).  If total is non-null
// the grand total is written there (device pointer).
inline int exclusive_scan_u32(tm_ctx *ctx, const uint32_t *in, uint32_t *out, uint64_t n, uint32_t *total)
{
    if (n == 0) {
        if (total) cudaMemsetAsync(total, 0, sizeof(uint32_t), ctx->stream);
        return TM_OK;
    }
    uint64_t tiles = (n + SCAN_TILE - 1) / SCAN_TILE;
    if (tiles == 1) {
        launch(ctx, k_tile_scan_u32, 1, SCAN_THREADS, in, n, (const uint32_t *)nullptr, out, total,
               (const uint32_t *)nullptr);
        return check_cuda(ctx, cudaGetLastError(), "scan");
    }
    ScratchScope scope(ctx);
    uint32_t *ts = (uint32_t *)salloc(ctx, tiles * sizeof(uint32_t));
    if (!ts) return TM_E_NOMEM;
    launch(ctx, k_tile_sum_u32, (unsigned)tiles, SCAN_THREADS, in, n, ts);
    if (tiles <= 4096) {   // each block adds up the totals before it: two launches in all
        launch(ctx, k_tile_scan_u32, (unsigned)tiles, SCAN_THREADS, in, n, (const uint32_t *)nullptr, out, total,
               (const uint32_t *)ts);
        return check_cuda(ctx, cudaGetLastError(), "scan");
    }
    int rc = exclusive_scan_u32(ctx, ts, ts, tiles, nullptr);
    if (rc == TM_OK) {
        launch(ctx, k_tile_scan_u32, (unsigned)tiles, SCAN_THREADS, in, n, (const uint32_t *)ts, out, total,
               (const uint32_t *)nullptr);
        rc = check_cuda(ctx, cudaGetLastError(), "scan");
    }
    return rc;
}

// ------------------------------------------ segmented u64, two layers ----
// Inclusive prefix sums that restart at segment heads, with every 64-bit
// addition inside a segment checked for wrap-around, over pairs (layer 0,
// layer 1) that share their positions (one gather of a 16-byte pair serves
// both layers).  A segment of layer p starts where the window of layer p
// changes or, in both layers, where a new owner starts.  Functor interface: w
// (the pairs), perm (position -> place in w; null: the same), nz (null, or a bit
// set of the non-zero pairs by place in w), tarr (position -> t'), wv (the
// window divider) and owner_word(w) -> the owner-start bits of positions 32 w ..
// 32 w + 31.  A pair behind a map is a random sector of memory and most are
// zero, which the bit set, small enough for L2, tells first.
struct SegAgg2 {
    uint64_t v0, v1;
    uint32_t f;     // bit p: the range contains a head of layer p
    uint32_t pad;
};

__device__ __forceinline__ SegAgg2 seg_combine2(SegAgg2 a, SegAgg2 b, bool &ovf)
{
    SegAgg2 r;
    r.f = a.f | b.f;
    r.v0 = (b.f & 1u) ? b.v0 : add_chk(a.v0, b.v0, ovf);
    r.v1 = (b.f & 2u) ? b.v1 : add_chk(a.v1, b.v1, ovf);
    r.pad = 0;
    return r;
}

// ---- one pass with decoupled look-back -------------------------------
// (Merrill and Garland, "Single-pass Parallel Prefix Scan with Decoupled
// Look-back", NVIDIA NVR-2016-002, 2016)
// Each block takes the next tile from a counter (so every tile before it has
// been started), scans it, publishes its aggregate, then its first warp walks
// back over the tiles before it, 32 at a time, combining their aggregates
// until it meets a published inclusive prefix or both layers have met a
// segment head (a head cuts the sums off), and publishes its own inclusive
// prefix.  Waits are bounded: a tile that does not publish within the limit
// latches ST_TIMEOUT.
// A tile's words: the halves of both layers' sums, first of its aggregate, then
// of its inclusive prefix.  The upper half of a word holds which of the two it
// is (1, 2; 0: not written) and the head bits, so a word carries its own
// validity: nothing is fenced, and a reader makes one trip to memory, over one
// sector, instead of two (status, then values).  Words of both kinds, read
// while the prefix replaces the aggregate, are read again.  (With fenced values
// and a status word of their own the scan of a node took 266 us on 1e7 edges
// and 570 us on 5e7; so 237 and 496.)
struct alignas(32) SegTile {
    unsigned long long w[4];
};

// Polls before a look-back gives up (ST_TIMEOUT), with __nanosleep(64) between
// them, or (32) in the radix passes, the pair tables and the windows.  The sleep
// is a hint with an upper bound of twice its argument and no lower one, so this
// bounds the number of polls alone.
constexpr int kLookbackPolls = 1 << 22;

__device__ __forceinline__ void seg_publish(SegTile *t, const SegAgg2 &v, uint32_t st)   // st 1: aggregate, 2: prefix
{
    const unsigned long long tag = (unsigned long long)((st << 2) | v.f) << 32;
    asm volatile("st.volatile.global.v2.u64 [%0], {%1, %2};" ::"l"(t->w), "l"(tag | (uint32_t)v.v0), "l"(tag | (v.v0 >> 32)) : "memory");
    asm volatile("st.volatile.global.v2.u64 [%0], {%1, %2};" ::"l"(t->w + 2), "l"(tag | (uint32_t)v.v1), "l"(tag | (v.v1 >> 32)) : "memory");
}

// What tile t has published (v is set): 2 its prefix, 1 its aggregate; 0: nothing yet.
__device__ __forceinline__ uint32_t seg_read(const SegTile *t, SegAgg2 &v)
{
    unsigned long long a, b, c, d;
    asm volatile("ld.volatile.global.v2.u64 {%0, %1}, [%2];" : "=l"(a), "=l"(b) : "l"(t->w) : "memory");
    asm volatile("ld.volatile.global.v2.u64 {%0, %1}, [%2];" : "=l"(c), "=l"(d) : "l"(t->w + 2) : "memory");
    const uint32_t h = (uint32_t)(a >> 32);
    v.v0 = (uint32_t)a | (b << 32);
    v.v1 = (uint32_t)c | (d << 32);
    v.f = h & 3u;
    return (uint32_t)(b >> 32) == h && (uint32_t)(c >> 32) == h && (uint32_t)(d >> 32) == h ? h >> 2 : 0u;
}

// A warp takes kScanRows rows of 32 consecutive positions, a lane one position
// of each, so that every load and store but a gather is coalesced, an owner
// word serves a row as it is, and a row is scanned with four shuffles a step (a
// lane knows from the head bits how far back its segment reaches).  With eight
// consecutive positions per thread instead, 16-byte accesses at a stride of 128
// bytes kept the L1 busiest (62 % of its throughput) and the two scans of a
// node took 356 us on 1e7 edges.
constexpr int kScanRows = 8;   // (4 and 6 rows at more blocks per SM measured 2 - 6 % slower)
constexpr int kScan2Tile = SCAN_THREADS * kScanRows;
#ifndef TM_SCAN_MINB
#define TM_SCAN_MINB 4   // 64 registers, four blocks per SM
#endif
template <class F>
__global__ void __launch_bounds__(SCAN_THREADS, TM_SCAN_MINB) k_segscan2_onepass(F f, uint64_t n, SegTile *__restrict__ tiles,
                                                                   uint32_t *__restrict__ counter,
                                                                   uint64_t *__restrict__ out0,
                                                                   uint64_t *__restrict__ out1,
                                                                   ulonglong2 *__restrict__ outp, uint32_t *status)
{
    grid_wait();
    __shared__ SegAgg2 warp_agg[SCAN_THREADS / 32];
    __shared__ uint32_t s_tile;
    if (threadIdx.x == 0) s_tile = atomicAdd(counter, 1u);
    __syncthreads();
    const uint32_t tile = s_tile;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const uint64_t base = (uint64_t)tile * kScan2Tile + (uint64_t)warp * (32 * kScanRows);   // the warp's first position
    const uint32_t le = 0xffffffffu >> (31 - lane);                                         // lanes up to this one
    bool ovf = false;
    ulonglong2 v[kScanRows];
    uint32_t t[kScanRows];
#pragma unroll
    for (int r = 0; r < kScanRows; ++r) {
        const uint64_t i = base + r * 32 + lane;
        t[r] = i < n ? __ldg(f.tarr + i) : 0u;
    }
    uint32_t tb = base > 0 && base < n ? __ldg(f.tarr + base - 1) : 0u;   // the time before the warp's first
    {
        uint32_t x[kScanRows];
#pragma unroll
        for (int r = 0; r < kScanRows; ++r) {
            const uint64_t i = base + r * 32 + lane;
            x[r] = i < n ? (f.perm ? __ldg(f.perm + i) : (uint32_t)i) : 0u;
        }
        uint32_t on = 0xffffffffu;   // bit r: row r's pair is read
        if (f.perm && f.nz) {
            on = 0;
#pragma unroll
            for (int r = 0; r < kScanRows; ++r) on |= ((__ldg(f.nz + (x[r] >> 5)) >> (x[r] & 31)) & 1u) << r;
        }
#pragma unroll
        for (int r = 0; r < kScanRows; ++r) {
            const uint64_t i = base + r * 32 + lane;
            v[r] = i < n && ((on >> r) & 1u) ? __ldg(f.w + x[r]) : make_ulonglong2(0, 0);
        }
    }
    uint32_t qb = f.wv.quot(tb);    // the quotient before the row's first
    uint32_t need0 = 0, need1 = 0;  // bit r: no head of the layer in the chunk up to row r's position
    bool seen0 = false, seen1 = false;
    uint64_t c0 = 0, c1 = 0;        // the sums at the row before's last position
#pragma unroll
    for (int r = 0; r < kScanRows; ++r) {
        const uint64_t row = base + r * 32;
        const uint32_t q = f.wv.quot(t[r]);
        uint32_t qp = __shfl_up_sync(0xffffffffu, q, 1);
        if (lane == 0) qp = qb;
        qb = __shfl_sync(0xffffffffu, q, 31);
        const bool in = row + lane < n;
        // the window of layer p is that of q with parity p: q / 2 and (q + 1) / 2 tell it
        uint32_t h0 = __ballot_sync(0xffffffffu, in && (q >> 1) != (qp >> 1));
        uint32_t h1 = __ballot_sync(0xffffffffu, in && ((q + 1) >> 1) != ((qp + 1) >> 1));
        uint32_t own = row < n ? f.owner_word(row >> 5) : 0u;
        if (row == 0) own |= 1u;
        h0 |= own;
        h1 |= own;
        const uint32_t b0 = h0 & le, b1 = h1 & le;
        const int reach0 = b0 ? lane - (31 - __clz((int)b0)) : lane, reach1 = b1 ? lane - (31 - __clz((int)b1)) : lane;
        uint64_t x0 = v[r].x, x1 = v[r].y;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint64_t y0 = __shfl_up_sync(0xffffffffu, x0, o), y1 = __shfl_up_sync(0xffffffffu, x1, o);
            if (o <= reach0) x0 = add_chk(y0, x0, ovf);
            if (o <= reach1) x1 = add_chk(y1, x1, ovf);
        }
        if (!b0) { x0 = add_chk(c0, x0, ovf); need0 |= seen0 ? 0u : 1u << r; }
        if (!b1) { x1 = add_chk(c1, x1, ovf); need1 |= seen1 ? 0u : 1u << r; }
        c0 = __shfl_sync(0xffffffffu, x0, 31);
        c1 = __shfl_sync(0xffffffffu, x1, 31);
        seen0 |= h0 != 0;
        seen1 |= h1 != 0;
        v[r] = make_ulonglong2(x0, x1);
    }
    if (lane == 0) warp_agg[warp] = SegAgg2{c0, c1, (seen0 ? 1u : 0u) | (seen1 ? 2u : 0u), 0};
    __syncthreads();
    if (warp == 0) {
        // the tile's aggregate (every lane of warp 0 folds the warp totals)
        SegAgg2 T = warp_agg[0];
        for (int w = 1; w < SCAN_THREADS / 32; ++w) T = seg_combine2(T, warp_agg[w], ovf);
        SegAgg2 ex{0, 0, 0, 0};
        if (tile == 0) {
            if (lane == 0) seg_publish(tiles, T, 2);
        } else {
            if (lane == 0) seg_publish(tiles + tile, T, 1);
            // look back 32 tiles at a time, lane i at tile (base - i): a tile
            // ends the walk when it holds an inclusive prefix, when the heads
            // met so far (from the closest tile outward) cover both layers, or
            // before tile 0
            for (int64_t jb = (int64_t)tile - 1;; jb -= 32) {
                const int64_t j = jb - lane;
                SegAgg2 v{0, 0, 0, 0};
                uint32_t st = 2;
                if (j >= 0) {
                    st = seg_read(tiles + j, v);
                    for (int it = 0; st == 0 && it < kLookbackPolls; ++it) {
                        __nanosleep(64);
                        st = seg_read(tiles + j, v);
                    }
                    if (st == 0) { latch(status, ST_TIMEOUT); v = SegAgg2{0, 0, 0, 0}; }
                }
                // heads met from the closest tile (lane 0) up to this lane
                uint32_t cf = v.f;
                for (int o = 1; o < 32; o <<= 1) {
                    const uint32_t y = __shfl_up_sync(0xffffffffu, cf, o);
                    if (lane >= o) cf |= y;
                }
                const bool term = j < 0 || st != 1 || (cf & 3u) == 3u;
                const unsigned tb = __ballot_sync(0xffffffffu, term);
                const int L = tb ? __ffs((int)tb) - 1 : 31;   // the last lane to take
                if (lane > L) v = SegAgg2{0, 0, 0, 0};
                // fold lanes L .. 0 in tile order (earlier tiles first)
                for (int o = 1; o < 32; o <<= 1) {
                    const SegAgg2 y{__shfl_down_sync(0xffffffffu, v.v0, o), __shfl_down_sync(0xffffffffu, v.v1, o),
                                    __shfl_down_sync(0xffffffffu, v.f, o), 0};
                    if (lane + o < 32) v = seg_combine2(y, v, ovf);
                }
                v = SegAgg2{__shfl_sync(0xffffffffu, v.v0, 0), __shfl_sync(0xffffffffu, v.v1, 0),
                            __shfl_sync(0xffffffffu, v.f, 0), 0};
                ex = seg_combine2(v, ex, ovf);
                if (tb) break;
            }
            if (lane == 0) seg_publish(tiles + tile, seg_combine2(ex, T, ovf), 2);
        }
        if (lane == 0) {
            SegAgg2 run = ex;
            for (int w = 0; w < SCAN_THREADS / 32; ++w) {
                const SegAgg2 c = warp_agg[w];
                warp_agg[w] = run;
                run = seg_combine2(run, c, ovf);
            }
        }
    }
    __syncthreads();
    // (storing what needs no carry before the look-back measured 5 - 10 % slower)
    const SegAgg2 pre = warp_agg[warp];
#pragma unroll
    for (int r = 0; r < kScanRows; ++r) {
        const uint64_t i = base + r * 32 + lane;
        if (i < n) {
            uint64_t r0 = v[r].x, r1 = v[r].y;
            if ((need0 >> r) & 1u) r0 = add_chk(pre.v0, r0, ovf);
            if ((need1 >> r) & 1u) r1 = add_chk(pre.v1, r1, ovf);
            if (outp) {
                outp[i] = make_ulonglong2(r0, r1);
            } else {
                out0[i] = r0;
                out1[i] = r1;
            }
        }
    }
    if (ovf) latch(status, ST_OVERFLOW);
}

// Scratch of one scan (tile words and a ticket), to be cleared before it.
inline size_t scan_state_bytes(uint64_t n)
{
    return ((n + kScan2Tile - 1) / kScan2Tile * sizeof(SegTile) + 64 + 255) / 256 * 256;
}

// Outputs: out0 / out1 (one array per layer), or outp (the (layer 0,
// layer 1) pairs interleaved) when it is non-null.
template <class F>
int segmented_scan2_u64(tm_ctx *ctx, const F &f, uint64_t n, char *state, uint64_t *out0, uint64_t *out1,
                        ulonglong2 *outp = nullptr)
{
    if (n == 0) return TM_OK;
    const uint64_t tiles = (n + kScan2Tile - 1) / kScan2Tile;
    if (tiles >= 0xFFFFFFFFull) return set_err(ctx, TM_E_LIMIT, "scan of more than 2^32 tiles");
    launch(ctx, k_segscan2_onepass<F>, (unsigned)tiles, SCAN_THREADS, f, n, (SegTile *)(state + 64), (uint32_t *)state,
           out0, out1, outp, ctx->status);
    return check_cuda(ctx, cudaGetLastError(), "segmented scan");
}

}  // namespace
}  // namespace timest

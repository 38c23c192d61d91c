// Stable radix sort of a batch's lookups by (table, row) for batches whose tables are too large for the cluster sort
// (or on request): the lookups arrive table-major, so every table is sorted by itself, by the row number within the
// table, and all tables move through the same launches.  Digits are at most ten bits wide and as few as the largest
// table needs: a million rows take two passes.  Measured on B200, 8.5 M lookups of 26 tables of a million rows, with the kernels
// that number the segments behind it: 204 us (228 before the first pass ranked by masks); one sort over the arena rows of all
// tables, with a kernel of its own that expanded the bags and three passes of nine bits, took 490.
//
//   rs_setup     one block: where each table begins, which table each tile of TILE lookups belongs to
//   per pass     rs_hist     digit counts of every tile (the first pass reads the indices themselves)
//                rs_scan     running counts over a table's tiles, totals per table and digit
//                rs_scatter  ranks its tile (stable), orders it by digit in shared memory so that a digit's entries leave
//                            as one run (a warp's 32 single pairs would touch 32 sectors), and writes it out; the first
//                            pass finds each lookup's bag on the way, the last one leaves keys and payloads apart
// No block waits for another.
#pragma once
#include "common.cuh"

namespace rsort {

constexpr int THREADS = 256;
constexpr int WARPS = THREADS / 32;
constexpr int ITEMS = 16;
constexpr int TILE = THREADS * ITEMS;
constexpr int MAX_DIGIT_BITS = 10;
constexpr int SCAN_DIGITS = 64, SCAN_GROUPS = 16;      // a block of rs_scan: digits x shares of the table's tiles

struct Args {
    const int32_t *indices, *offsets;
    const int64_t *row_off;
    int T, B;
    int64_t L, G;
    u32 *tb, *tile0, *tile_table;   // [T+1] first lookup of a table, [T+1] its first tile, [tiles] the tile's table
    u32 *tilehist;                  // [tiles][nb]
    u32 *totals;                    // [T][nb]
    int dbits;
    int payload_position;           // 0: payload = row of grad_out [B][T][D]; 1: payload = position of the lookup
    int *status;
};

inline int64_t max_tiles(int T, int64_t L) { return (L + TILE - 1) / TILE + T; }
inline size_t setup_smem(int T) { return (size_t)(T + 1) * 2 * sizeof(u32); }
inline size_t scatter_smem(int nb) { return (size_t)TILE * sizeof(uint2) + (size_t)nb * sizeof(u32) + (size_t)WARPS * nb * sizeof(unsigned short); }

__global__ void __launch_bounds__(1024)
rs_setup_kernel(const Args a)
{
    dq_wait_before();
    extern __shared__ __align__(16) u32 s_tb[];                      // [T+1]
    u32 *s_t0 = s_tb + (a.T + 1);                      // [T+1]
    const int lane = threadIdx.x & 31;
    if (threadIdx.x < 32) {
        // the tables' boundaries; unusable ones are reported and made to ascend, so that every lookup has a table
        u32 top = 0;
        for (int t0 = 0; t0 <= a.T; t0 += 32) {
            const int t = t0 + lane;
            int64_t o = t <= a.T ? (int64_t)__ldg(a.offsets + (int64_t)t * a.B) : a.L;
            const int64_t want = o;
            if (t == 0) o = 0;
            if (t >= a.T) o = a.L;
            u32 v = (u32)min(max(o, (int64_t)0), a.L);
            v = max(v, top);
#pragma unroll
            for (int s = 1; s < 32; s <<= 1) {
                const u32 x = __shfl_up_sync(0xffffffffu, v, s);
                if (lane >= s) v = max(v, x);
            }
            if (t <= a.T && (int64_t)v != want) dq_report(a.status, DQRM_ERR_INDEX_RANGE);
            if (t <= a.T) s_tb[t] = v;
            top = __shfl_sync(0xffffffffu, v, 31);
        }
        __syncwarp();
        u32 run = 0;
        for (int t0 = 0; t0 < a.T; t0 += 32) {
            const int t = t0 + lane;
            const u32 cnt = t < a.T ? (s_tb[t + 1] - s_tb[t] + TILE - 1) / TILE : 0u;
            u32 incl = cnt;
#pragma unroll
            for (int s = 1; s < 32; s <<= 1) {
                const u32 x = __shfl_up_sync(0xffffffffu, incl, s);
                if (lane >= s) incl += x;
            }
            if (t < a.T) s_t0[t] = run + incl - cnt;
            run += __shfl_sync(0xffffffffu, incl, 31);
        }
        if (lane == 0) s_t0[a.T] = run;
    }
    __syncthreads();
    for (int t = threadIdx.x; t <= a.T; t += blockDim.x) { a.tb[t] = s_tb[t]; a.tile0[t] = s_t0[t]; }
    const u32 tiles = s_t0[a.T];
    for (u32 i = threadIdx.x; i < tiles; i += blockDim.x) {
        int lo = 0, hi = a.T;                          // largest t with s_t0[t] <= i (empty tables share a start: the last)
        while (hi - lo > 1) {
            const int mid = (lo + hi) >> 1;
            if (s_t0[mid] <= i) lo = mid; else hi = mid;
        }
        a.tile_table[i] = (u32)lo;
    }
}

struct Tile { int t, len; u32 start; };

// (block-uniform; false for the launches' spare blocks)
__device__ __forceinline__ bool tile_of(const Args &a, Tile &x)
{
    if (blockIdx.x >= __ldg(a.tile0 + a.T)) return false;
    x.t = (int)__ldg(a.tile_table + blockIdx.x);
    x.start = __ldg(a.tb + x.t) + (blockIdx.x - __ldg(a.tile0 + x.t)) * TILE;
    x.len = (int)min((u32)TILE, __ldg(a.tb + x.t + 1) - x.start);
    return true;
}

// row within the table of the lookup at position i, kept inside the table
__device__ __forceinline__ u32 row_at(const Args &a, int64_t i, int32_t nrows, bool &bad)
{
    const int32_t idx = __ldg(a.indices + i);
    bad |= (idx < 0) | (idx >= nrows);
    return (u32)min(max(idx, 0), nrows - 1);
}

template <bool FIRST>
__global__ void __launch_bounds__(THREADS)
rs_hist_kernel(const Args a, const uint2 *__restrict__ pairs, int shift)
{
    dq_wait_before();
    __shared__ u32 cnt[1 << MAX_DIGIT_BITS];
    Tile x;
    if (!tile_of(a, x)) return;
    const int nb = 1 << a.dbits;
    const u32 mask = (u32)nb - 1u;
    for (int i = threadIdx.x; i < nb; i += THREADS) cnt[i] = 0u;
    bool bad = false;
    const int32_t nrows = FIRST ? (int32_t)(__ldg(a.row_off + x.t + 1) - __ldg(a.row_off + x.t)) : 0;
    u32 key[ITEMS];
#pragma unroll
    for (int k = 0; k < ITEMS; ++k) {
        const int i = k * THREADS + threadIdx.x;
        key[k] = 0u;
        if (i < x.len) key[k] = FIRST ? row_at(a, (int64_t)x.start + i, nrows, bad) : __ldg(&pairs[x.start + i].x);
    }
    if (FIRST) {                                       // offsets must not decrease: every block looks at some of them
        const int64_t step = (int64_t)__ldg(a.tile0 + a.T) * THREADS;
        for (int64_t g = (int64_t)blockIdx.x * THREADS + threadIdx.x; g < a.G; g += step)
            bad |= __ldg(a.offsets + g) > __ldg(a.offsets + g + 1);
        if (bad) dq_report(a.status, DQRM_ERR_INDEX_RANGE);
    }
    __syncthreads();
#pragma unroll
    for (int k = 0; k < ITEMS; ++k)
        if (k * THREADS + (int)threadIdx.x < x.len) atomicAdd(&cnt[(key[k] >> shift) & mask], 1u);
    __syncthreads();
    for (int i = threadIdx.x; i < nb; i += THREADS) a.tilehist[(size_t)blockIdx.x * nb + i] = cnt[i];
}

// blockIdx.y = table, blockIdx.x = 64 digits: counts become running counts over the table's tiles
__global__ void __launch_bounds__(SCAN_DIGITS * SCAN_GROUPS)
rs_scan_kernel(const Args a)
{
    dq_wait_before();
    __shared__ u32 part[SCAN_GROUPS][SCAN_DIGITS];
    const int nb = 1 << a.dbits;
    const int dl = threadIdx.x % SCAN_DIGITS, g = threadIdx.x / SCAN_DIGITS, d = blockIdx.x * SCAN_DIGITS + dl;
    const int t = blockIdx.y;
    const u32 first = __ldg(a.tile0 + t), n = __ldg(a.tile0 + t + 1) - first;
    const u32 per = (n + SCAN_GROUPS - 1) / SCAN_GROUPS, b0 = min(n, g * per), b1 = min(n, b0 + per);
    u32 *h = a.tilehist + (size_t)first * nb + d;
    u32 sum = 0;
    if (d < nb)
        for (u32 b = b0; b < b1; b += 8) {
#pragma unroll
            for (int k = 0; k < 8; ++k) sum += b + k < b1 ? h[(size_t)(b + k) * nb] : 0u;
        }
    part[g][dl] = sum;
    __syncthreads();
    u32 run = 0, all = 0;
#pragma unroll
    for (int k = 0; k < SCAN_GROUPS; ++k) {
        const u32 v = part[k][dl];
        if (k < g) run += v;
        all += v;
    }
    if (d >= nb) return;
    if (g == 0) a.totals[(size_t)t * nb + d] = all;
    for (u32 b = b0; b < b1; b += 8) {
        u32 c[8];
#pragma unroll
        for (int k = 0; k < 8; ++k) c[k] = b + k < b1 ? h[(size_t)(b + k) * nb] : 0u;
#pragma unroll
        for (int k = 0; k < 8; ++k)
            if (b + k < b1) { h[(size_t)(b + k) * nb] = run; run += c[k]; }
    }
}

// exclusive sum over the block of one value per thread
__device__ __forceinline__ u32 block_exclusive(u32 v, u32 *s_warp)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    u32 incl = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const u32 x = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += x;
    }
    if (lane == 31) s_warp[warp] = incl;
    __syncthreads();
    u32 before = incl - v;
#pragma unroll
    for (int w = 0; w < WARPS; ++w)
        if (w < warp) before += s_warp[w];
    __syncthreads();
    return before;
}

template <bool FIRST, bool LAST>
__global__ void __launch_bounds__(THREADS, 3)
rs_scatter_kernel(const Args a, const uint2 *__restrict__ pairs_in, uint2 *__restrict__ pairs_out,
                  u32 *__restrict__ keys_out, u32 *__restrict__ vals_out, int shift)
{
    dq_wait_before();
    extern __shared__ __align__(16) uint2 s_pair[];                  // [TILE]
    const int nb = 1 << a.dbits;
    u32 *s_delta = reinterpret_cast<u32 *>(s_pair + TILE);                               // [nb]
    unsigned short *s_cnt = reinterpret_cast<unsigned short *>(s_delta + nb);            // [WARPS][nb]
    __shared__ u32 s_warp[WARPS];
    Tile x;
    if (!tile_of(a, x)) return;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const u32 mask = (u32)nb - 1u, lt = (1u << lane) - 1u;
    const int w0 = warp * (TILE / WARPS) + lane;       // a warp holds 512 consecutive entries, 32 at a time
    const int64_t r0 = __ldg(a.row_off + x.t);
    u32 key[ITEMS], val[ITEMS], rank[ITEMS / 2];       // ranks: two 16-bit halves per word
    for (int i = threadIdx.x; i < WARPS * nb / 2; i += THREADS) reinterpret_cast<u32 *>(s_cnt)[i] = 0u;
    if (FIRST) {
        const int32_t nrows = (int32_t)(__ldg(a.row_off + x.t + 1) - r0);
        bool bad = false;
#pragma unroll
        for (int k = 0; k < ITEMS; ++k) {
            const int i = w0 + k * 32;
            key[k] = i < x.len ? row_at(a, (int64_t)x.start + i, nrows, bad) : 0u;       // (rs_hist has reported it)
        }
        if (a.payload_position) {
#pragma unroll
            for (int k = 0; k < ITEMS; ++k) val[k] = x.start + w0 + k * 32;
        } else {
            // the lookups' bags: the tile's first bag by a search with all threads, then every bag marks its first
            // lookup and every other lookup takes the mark before it (of bags that begin at the same lookup the last
            // counts: the others are empty).  A vote finds the mark inside the warp's 32 entries; a running maximum by
            // shuffles in its place took twice as long as the whole rest of the pass
            const int32_t *off = a.offsets + (int64_t)x.t * a.B;
            const int64_t end = (int64_t)x.start + x.len;
            int lo = 0, size = a.B;                    // invariant: the bag is in [lo, lo + size)
            while (size > 1) {
                const int step = (size + THREADS - 1) / THREADS;
                const int at = lo + (int)threadIdx.x * step;
                const int c = __syncthreads_count((int)threadIdx.x * step < size && (int64_t)__ldg(off + at) <= (int64_t)x.start);
                const int skip = max(c - 1, 0) * step;
                lo += skip;
                size = min(step, size - skip);
            }
            u32 *mark = reinterpret_cast<u32 *>(s_pair);
            for (int i = threadIdx.x; i < TILE; i += THREADS) mark[i] = 0u;
            __syncthreads();
            for (int g = lo + (int)threadIdx.x; g < a.B; g += THREADS) {
                const int64_t o = __ldg(off + g);
                if (o >= end) break;
                if (o >= (int64_t)x.start) atomicMax(&mark[o - x.start], (u32)(g - lo) + 1u);
            }
            __syncthreads();
            u32 top = 0;
#pragma unroll
            for (int k = 0; k < ITEMS; ++k) {
                const u32 v = mark[w0 + k * 32];
                const u32 marked = __ballot_sync(0xffffffffu, v != 0u);
                const u32 upto = marked & (lt | (1u << lane));
                const u32 y = __shfl_sync(0xffffffffu, v, upto ? 31 - __clz(upto) : 0);
                val[k] = upto ? y : top;
                const u32 last = __shfl_sync(0xffffffffu, v, marked ? 31 - __clz(marked) : 0);
                top = marked ? last : top;
            }
            if (lane == 0) s_warp[warp] = top;
            __syncthreads();
            u32 before = 1;                            // (the tile's first bag)
#pragma unroll
            for (int w = 0; w < WARPS; ++w)
                if (w < warp && s_warp[w]) before = s_warp[w];
#pragma unroll
            for (int k = 0; k < ITEMS; ++k) val[k] = (u32)(lo + (val[k] ? val[k] : before) - 1) * (u32)a.T + (u32)x.t;
        }
    } else {
#pragma unroll
        for (int k = 0; k < ITEMS; ++k) {
            const int i = w0 + k * 32;
            const uint2 pr = i < x.len ? __ldcs(pairs_in + x.start + i) : make_uint2(0u, 0u);
            key[k] = pr.x;
            val[k] = pr.y;
        }
    }
    __syncthreads();
    // ---- rank within (warp, digit), counting on the way.  The first pass finds the lanes with the same digit by an OR into shared
    // memory, where the pairs will stand (by match.any, which takes the longer the more digits differ, 16 K of a tile's 38 K clocks);
    // in the later ones equal rows already stand together, and a match of few digits is the faster.  With what the digits' places
    // below save: the two scatters of 8.5 M lookups 156 -> 131 us
    u32 *my_mask = reinterpret_cast<u32 *>(s_pair) + warp * nb;
    static_assert(sizeof(uint2) * TILE >= (sizeof(u32) * WARPS << MAX_DIGIT_BITS), "");
    if (FIRST) {
        for (int i = lane; i < nb; i += 32) my_mask[i] = 0u;
        __syncwarp();
    }
    unsigned short *my_cnt = s_cnt + warp * nb;
#pragma unroll
    for (int k = 0; k < ITEMS; ++k) {
        const bool valid = w0 + k * 32 < x.len;
        const u32 d = (key[k] >> shift) & mask;
        const u32 peers = FIRST ? dq_same_digit_lanes(my_mask, d, valid) : __match_any_sync(0xffffffffu, valid ? d : (u32)nb);
        u32 r = 0;
        if (valid) r = my_cnt[d] + __popc(peers & lt);
        __syncwarp();
        if (valid && (peers & lt) == 0u) my_cnt[d] = (unsigned short)(r + __popc(peers));       // (the first of the peers)
        __syncwarp();
        if (k & 1) rank[k / 2] |= r << 16; else rank[k / 2] = r;
    }
    // the digits of this thread (four consecutive ones): how many entries the table has, and the tiles before this one
    const int d0 = (int)threadIdx.x * 4;
    uint4 all = make_uint4(0u, 0u, 0u, 0u), earlier = all;
    if (d0 < nb) {
        all = __ldg(reinterpret_cast<const uint4 *>(a.totals + (size_t)x.t * nb + d0));
        earlier = __ldg(reinterpret_cast<const uint4 *>(a.tilehist + (size_t)blockIdx.x * nb + d0));
    }
    __syncthreads();
    // ---- per digit: the warps' counts become places in the tile's order, and what leads from there to the output.  Two
    // digits a word: a tile's counts fit 16 bits
    {
        uint2 before[WARPS], tot = make_uint2(0u, 0u);
        uint2 *c4 = reinterpret_cast<uint2 *>(s_cnt) + threadIdx.x;
        if (d0 < nb) {
#pragma unroll
            for (int w = 0; w < WARPS; ++w) before[w] = c4[w * (nb / 4)];
#pragma unroll
            for (int w = 0; w < WARPS; ++w) {
                const uint2 c = before[w];
                before[w] = tot;
                tot.x += c.x;
                tot.y += c.y;
            }
        }
        const u32 n0 = tot.x & 0xffffu, n1 = tot.x >> 16, n2 = tot.y & 0xffffu, n3 = tot.y >> 16;
        const u32 place = block_exclusive(n0 + n1 + n2 + n3, s_warp);
        const u32 base = block_exclusive(all.x + all.y + all.z + all.w, s_warp) + __ldg(a.tb + x.t);
        if (d0 < nb) {
            const u32 p1 = place + n0, p2 = p1 + n1, p3 = p2 + n2, b1 = base + all.x, b2 = b1 + all.y, b3 = b2 + all.z;
            *reinterpret_cast<uint4 *>(s_delta + d0) = make_uint4(base + earlier.x - place, b1 + earlier.y - p1, b2 + earlier.z - p2, b3 + earlier.w - p3);
            const uint2 p = make_uint2(place | p1 << 16, p2 | p3 << 16);
#pragma unroll
            for (int w = 0; w < WARPS; ++w) c4[w * (nb / 4)] = make_uint2(p.x + before[w].x, p.y + before[w].y);
        }
    }
    __syncthreads();
#pragma unroll
    for (int k = 0; k < ITEMS; ++k) {
        if (w0 + k * 32 < x.len) {
            const u32 d = (key[k] >> shift) & mask;
            s_pair[my_cnt[d] + ((k & 1) ? rank[k / 2] >> 16 : rank[k / 2] & 0xffffu)] = make_uint2(key[k], val[k]);
        }
    }
    __syncthreads();
#pragma unroll 4
    for (int i = threadIdx.x; i < x.len; i += THREADS) {
        const uint2 pr = s_pair[i];
        const u32 at = s_delta[(pr.x >> shift) & mask] + (u32)i;
        if (LAST) {
            keys_out[at] = (u32)r0 + pr.x;
            vals_out[at] = pr.y;
        } else {
            pairs_out[at] = pr;
        }
    }
}

}  // namespace rsort

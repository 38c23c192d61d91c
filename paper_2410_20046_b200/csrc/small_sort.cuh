// Per-table stable sort of a small batch's lookups by row: one block per table.  At up to two thousand lookups a table the
// sort of cluster_sort.cuh is all fixed cost (cluster barriers, three passes through other blocks' memory for large tables).
//
// Up to 256 lookups: a bitonic network over (row, position) held in registers: log2(n) (log2(n) + 1) / 2 steps whatever the row
// count; most of them stay inside a warp, and unrolled they cost about 0.15 us each (with the steps in a loop, 1.5 times
// that).  Every thread holds one entry: steps across less than 32 entries are shuffles, wider ones go through shared memory (two
// buffers in turn, one barrier a step).  Row and position
// make every key distinct, so the order is that of a stable sort.  Beyond that: the radix sort of sort_parts.cuh.
//
// A table with more lookups than the block holds is sorted by its cluster where the batch has clusters standing by
// (csort::sort_by_cluster with EPT > 0).  By the block in global memory, with 8-bit digits, at 7 ns a lookup against 2 in a cluster
// (12.8 K lookups), only in the one-launch step, which takes no batch in which that is the longer way, and in batches with as many
// lookups as bags that are uneven all the same, of up to 1024 lookups a table or of more tables than have room for clusters.
// The lists that it leaves are those of the cluster sort's lists_by_table.
//
// Kernels take their arguments as grid constants: the functions that stay out of line get a pointer to them, and without that
// every thread would first copy them to its stack (128 lookups a table 4.0 -> 3.6 us).
#pragma once
#include "cluster_sort.cuh"

namespace ssort {

typedef unsigned long long u64;

inline size_t smem_bytes(int threads)
{
    const size_t net = (size_t)threads * 2 * sizeof(u64);
    const size_t digits = (size_t)(threads / 32) * csort::BINS * sizeof(u32);
    return net > digits ? net : digits;
}

__host__ __device__ constexpr int log2c(int x) { return x <= 1 ? 0 : 1 + log2c(x / 2); }

__device__ __forceinline__ u64 shfl_xor64(u64 v, int mask)
{
    return __shfl_xor_sync(0xffffffffu, v, mask);
}

// (row within the table, payload) of the lookup at position p of table t
__device__ __forceinline__ uint2 lookup(const csort::Args &a, int t, int64_t tb0, int64_t n, int64_t nrows, int64_t p, bool &bad)
{
    const int32_t *off_t = a.offsets + (int64_t)t * a.B;
    int32_t idx = __ldg(a.indices + tb0 + p);
    bool single = false;
    if (n == a.B) {
        const int64_t o0 = __ldg(off_t + p), o1 = __ldg(off_t + p + 1);
        single = o0 == tb0 + p && o1 == tb0 + p + 1;
        bad |= o0 > o1;
    }
    bad |= (idx < 0) | (idx >= nrows);
    idx = (int32_t)min((int64_t)max(idx, 0), nrows - 1);
    int64_t bag = p;
    if (!single) {                                 // largest bag b with offsets[t*B + b] <= tb0 + p
        int lo = 0, hi = a.B;
        while (hi - lo > 1) {
            const int mid = (lo + hi) >> 1;
            if ((int64_t)__ldg(off_t + mid) <= tb0 + p) lo = mid; else hi = mid;
        }
        bag = lo;
    }
    return make_uint2((u32)idx, a.payload_position ? (u32)(tb0 + p) : (u32)(bag * a.T + t));
}

// The block's table in global memory, 8 bits a pass; returns the buffer that holds the result
template <int THREADS>
__device__ __noinline__ const uint2 *sort_in_memory(const csort::Args &a, int t, int64_t tb0, int64_t n, int64_t nrows, u32 *s_cnt)
{
    constexpr int WARPS = THREADS / 32, BINS = csort::BINS;
    __shared__ u32 s_scan[BINS / 32];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    bool bad = false;
    for (int64_t p = threadIdx.x; p < n; p += THREADS) a.gp[0][tb0 + p] = lookup(a, t, tb0, n, nrows, p, bad);
    if (bad) dq_report(a.status, DQRM_ERR_INDEX_RANGE);
    __syncthreads();
    const int64_t part = ((n + WARPS - 1) / WARPS + 31) / 32 * 32;
    const int64_t w0 = min(n, (int64_t)warp * part), w1 = min(n, w0 + part);
    int s = 0;
    for (int shift = 0; ((int64_t)1 << shift) < nrows; shift += 8) {
        const uint2 *src = a.gp[s] + tb0;
        uint2 *dst = a.gp[s ^ 1] + tb0;
        for (int i = threadIdx.x; i < WARPS * BINS; i += THREADS) s_cnt[i] = 0u;
        __syncthreads();
        for (int64_t i = w0 + lane; i < w1; i += 32) atomicAdd(&s_cnt[warp * BINS + ((src[i].x >> shift) & 255u)], 1u);
        __syncthreads();
        u32 tot = 0, incl = 0;
        if (threadIdx.x < BINS) {
            for (int w = 0; w < WARPS; ++w) tot += s_cnt[w * BINS + threadIdx.x];
            incl = tot;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const u32 v = __shfl_up_sync(0xffffffffu, incl, o);
                if (lane >= o) incl += v;
            }
            if (lane == 31) s_scan[warp] = incl;
        }
        __syncthreads();
        if (threadIdx.x < BINS) {
            u32 run = incl - tot;
            for (int w = 0; w < warp; ++w) run += s_scan[w];
            for (int w = 0; w < WARPS; ++w) {
                const u32 c = s_cnt[w * BINS + threadIdx.x];
                s_cnt[w * BINS + threadIdx.x] = run;
                run += c;
            }
        }
        __syncthreads();
        for (int64_t i0 = w0; i0 < w1; i0 += 32) {
            const bool valid = i0 + lane < w1;
            const uint2 pr = valid ? src[i0 + lane] : make_uint2(0u, 0u);
            const u32 d = (pr.x >> shift) & 255u;
            const u32 peers = __match_any_sync(0xffffffffu, valid ? d : 256u + lane);       // (slow, but without room of its own)
            const int leader = __ffs(peers) - 1;
            u32 base = 0;
            if (valid && lane == leader) { base = s_cnt[warp * BINS + d]; s_cnt[warp * BINS + d] = base + __popc(peers); }
            base = __shfl_sync(0xffffffffu, base, leader & 31);
            __syncwarp();
            if (valid) dst[base + __popc(peers & ((1u << lane) - 1u))] = pr;
        }
        __syncthreads();
        s ^= 1;
    }
    return a.gp[s] + tb0;
}

// The block's table (n <= THREADS lookups) into s_net[0 .. n): row << 32 | payload; s_net has 2 * THREADS places
template <int THREADS>
__device__ __forceinline__ void sort_in_block(const csort::Args &a, int t, int64_t tb0, int64_t n, int64_t nrows, u64 *s_net, bool &bad)
{
    const int tid = threadIdx.x;
    u64 e = ~0ull;                                 // row << 32 | position, later row << 32 | payload
    u32 pay = 0u;
    if (tid < n) {
        const uint2 pr = lookup(a, t, tb0, n, nrows, tid, bad);
        e = (u64)pr.x << 32 | (u32)tid;
        pay = pr.y;
    }
    int top = 1;                               // entries that the network covers: a power of two from 32 on
    while ((1 << top) < n) ++top;
    const bool live = (tid & ~31) < (1 << top);       // (warps of places beyond only keep the barriers)
    u64 *buf = s_net;
    constexpr int TOP = log2c(THREADS);
#pragma unroll
    for (int p = 1; p <= TOP; ++p) {
        if (p > top) break;                    // (block-uniform)
#pragma unroll
        for (int s = p - 1; s >= 0; --s) {
            const int stride = 1 << s;
            if (stride >= 32) {
                buf[tid] = e;
                __syncthreads();
                const bool up = ((tid >> p) & 1) == 0, low = (tid & stride) == 0;      // (before the barrier they cost it 0.07 us)
                const u64 o = buf[tid ^ stride];
                e = (up == low) == (e < o) ? e : o;
                buf = buf == s_net ? s_net + THREADS : s_net;
            } else {
                const bool up = ((tid >> p) & 1) == 0, low = (tid & stride) == 0;
                if (live) {
                    const u64 o = shfl_xor64(e, stride);
                    e = (up == low) == (e < o) ? e : o;
                }
            }
        }
    }
    // the payloads come back by position
    __syncthreads();
    u32 *s_pay = reinterpret_cast<u32 *>(s_net);
    s_pay[tid] = pay;
    __syncthreads();
    if (tid < n) e = (e & 0xffffffff00000000ull) | s_pay[(u32)e];
    __syncthreads();
    s_net[tid] = e;
    __syncthreads();
}

// The sorted keys and payloads of the block's table, and where its segments stand: THREADS consecutive entries at a time, out
// of the network's places or of memory
template <int THREADS>
__device__ __forceinline__ void write_table(const csort::Args &a, int t, int64_t tb0, int64_t tb1, const u64 *s_net, const uint2 *mem)
{
    constexpr int WARPS = THREADS / 32;
    __shared__ u32 s_warp[WARPS];
    __shared__ u32 s_total;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int64_t n = tb1 - tb0, r0 = __ldg(a.row_off + t);
    u32 *segs = a.seg_start + tb0 + t;
    const u32 ck_mask = (1u << a.ck_shift) - 1u;
    u32 base = 0;                                  // segments that begin before these entries
    for (int64_t c0 = 0; c0 < n; c0 += THREADS) {
        const int64_t i = c0 + tid, j = tb0 + i;
        bool head = false;
        if (i < n) {
            u32 row, pay, prev;
            if (mem) {
                row = mem[i].x;
                pay = mem[i].y;
                prev = i > 0 ? mem[i - 1].x : ~row;
            } else {
                row = (u32)(s_net[i] >> 32);
                pay = (u32)s_net[i];
                prev = i > 0 ? (u32)(s_net[i - 1] >> 32) : ~row;
            }
            a.keys_out[j] = (u32)(r0 + row);
            a.vals_out[j] = pay;
            head = row != prev;
        }
        const u32 m = __ballot_sync(0xffffffffu, head);
        if (lane == 0) s_warp[warp] = __popc(m);
        __syncthreads();
        if (warp == 0) {
            const u32 v = lane < WARPS ? s_warp[lane] : 0u;
            u32 incl = v;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const u32 x = __shfl_up_sync(0xffffffffu, incl, o);
                if (lane >= o) incl += x;
            }
            if (lane < WARPS) s_warp[lane] = incl - v;
            if (lane == 31) s_total = incl;
        }
        __syncthreads();
        if (i < n) {
            const u32 upto = base + s_warp[warp] + __popc(m & (0xffffffffu >> (31 - lane)));      // segment starts in [0, i]
            if (head) segs[upto - 1] = (u32)j;
            if (((u32)j & ck_mask) == 0u) {
                a.chunk_first[j >> a.ck_shift] = upto - 1;
                a.tile_done[j >> a.ck_shift] = make_uint2(0u, 0u);
            }
        }
        base += s_total;
        __syncthreads();
    }
    if (tid == 0) {
        a.table_cnt[t] = base;
        segs[base] = (u32)tb1;                     // the slot behind the last segment holds the table's end
    }
}

// offsets must not decrease inside the table
template <int THREADS>
__device__ __forceinline__ bool offsets_fall(const csort::Args &a, int t)
{
    bool bad = false;
    for (int i = threadIdx.x; i < a.B; i += THREADS) bad |= __ldg(a.offsets + (int64_t)t * a.B + i) > __ldg(a.offsets + (int64_t)t * a.B + i + 1);
    return bad;
}

// A block's table by the network
template <int THREADS>
__device__ __forceinline__ void sort_by_network(const csort::Args &a)
{
    extern __shared__ __align__(16) u64 s_net[];                 // [2][THREADS]
    const int t = blockIdx.x, tid = threadIdx.x;
    const int64_t tb0 = __ldg(a.offsets + (int64_t)t * a.B), tb1 = __ldg(a.offsets + (int64_t)(t + 1) * a.B);
    if (tb0 < 0 || tb1 < tb0 || tb1 > a.L || (t == 0 && tb0 != 0) || (t == a.T - 1 && tb1 != a.L)) {
        if (tid == 0) {
            dq_report(a.status, DQRM_ERR_INDEX_RANGE);
            a.table_cnt[t] = a.cnt_broken;         // nothing is summed; the quantiser behind finds an empty gradient
            a.absmax[t] = 0u;
        }
        return;
    }
    const int64_t n = tb1 - tb0;
    if (tid == 0) {
        a.tb[t] = (u32)tb0;
        if (t == a.T - 1) a.tb[a.T] = (u32)tb1;
        a.absmax[t] = 0u;
        if (n == 0) a.table_cnt[t] = 0u;
    }
    if (n <= THREADS) {
        const int64_t nrows = __ldg(a.row_off + t + 1) - __ldg(a.row_off + t);
        bool bad = n != a.B && offsets_fall<THREADS>(a, t);       // (otherwise every lookup looks at its own bag's offsets)
        if (n > 0) sort_in_block<THREADS>(a, t, tb0, n, nrows, s_net, bad);
        if (bad) dq_report(a.status, DQRM_ERR_INDEX_RANGE);
        if (n > 0) write_table<THREADS>(a, t, tb0, tb1, s_net, nullptr);
    } else {                                       // (a one-index batch that is none)
        if (offsets_fall<THREADS>(a, t)) dq_report(a.status, DQRM_ERR_INDEX_RANGE);
        const int64_t nrows = __ldg(a.row_off + t + 1) - __ldg(a.row_off + t);
        const uint2 *mem = sort_in_memory<THREADS>(a, t, tb0, n, nrows, reinterpret_cast<u32 *>(s_net));
        write_table<THREADS>(a, t, tb0, tb1, nullptr, mem);
    }
}

// ... of up to 512 * E lookups by the radix sort of sort_parts.cuh
template <int E>
__device__ __forceinline__ void sort_by_block(const csort::Args &a)
{
    extern __shared__ __align__(16) uint2 s_pair[];              // [THREADS * E]
    __shared__ __align__(16) u32 s_cnt[csort::WARPS * csort::BINS];
    const int t = blockIdx.x;
    const int64_t tb0 = __ldg(a.offsets + (int64_t)t * a.B), tb1 = __ldg(a.offsets + (int64_t)(t + 1) * a.B);
    if (csort::broken_table(a, t, t, tb0, tb1, threadIdx.x == 0)) return;
    if (threadIdx.x == 0) csort::open_table(a, t, tb0, tb1);
    const int64_t n = tb1 - tb0;
    if (n <= csort::THREADS * E) {
        csort::sort_alone<E>(a, t, (u32)tb0, (u32)tb1, s_cnt, s_pair);
    } else {                                       // (a one-index batch that is none)
        if (offsets_fall<csort::THREADS>(a, t)) dq_report(a.status, DQRM_ERR_INDEX_RANGE);
        const int64_t nrows = __ldg(a.row_off + t + 1) - __ldg(a.row_off + t);
        const uint2 *mem = sort_in_memory<csort::THREADS>(a, t, tb0, n, nrows, s_cnt);
        csort::write_sorted(a, t, (u32)tb0, (u32)tb1, mem);
    }
}

// 256 threads: the network.  512 threads: the radix sort; CL > 1: a cluster of blocks stands by for every table and sorts one that
// is larger.  (No minimum of blocks without clusters: with a minimum of one the radix sort takes 94 registers instead of 64, 8.2 us
// instead of 8.5 alone, and leaves a third less of its SM to what runs beside it)
template <int THREADS, int E, int CL>
__global__ void __launch_bounds__(THREADS, CL > 1 ? csort::resident(CL) : 0)
small_sort_kernel(const __grid_constant__ csort::Args a)
{
    dq_wait_before();
    if constexpr (CL > 1) csort::sort_by_cluster<CL, E, false>(a);
    else if constexpr (THREADS == csort::THREADS) sort_by_block<E>(a);
    else sort_by_network<THREADS>(a);
}

}  // namespace ssort

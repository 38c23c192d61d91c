// Arguments of the two sorts that a table's own blocks do (small_sort.cuh: one block, cluster_sort.cuh: a cluster of blocks), and
// how one block sorts a table alone, which both use: loading of lookups, a stable radix sort in registers, the write-out with the
// segment lists.
//
// Entries are (row within the table, payload).  A block holds them warp-striped: warp w has `rounds` consecutive groups of 32
// entries, the group's entry l in lane l.  Places beyond the last entry hold the row ~0, which sorts behind every other.
#pragma once
#include <cooperative_groups.h>
#include "common.cuh"

namespace csort {

namespace cg = cooperative_groups;

constexpr int THREADS = 512;
constexpr int WARPS = THREADS / 32;
constexpr int BINS = 256;
constexpr int SORT_ROOM = WARPS * BINS / 2;      // entries that take the place of a word for every warp and digit

struct Args {
    const int32_t *indices;
    const int32_t *offsets;
    const int64_t *row_off;
    int T, B;
    int64_t L;
    u32 *keys_out, *vals_out;       // [L] sorted result
    uint2 *gp[2];                   // [L] global staging of pairs (tables too large for shared memory)
    int cap;                        // pairs per block that fit in each of the two buffers in shared memory
    int payload_position;           // 0: payload = row of grad_out [B][T][D]; 1: payload = position of the lookup in indices
    int *status;
    u32 *tile_heads;                // [ceil(L / 2048)] zeroed by the caller: segment heads per tile of the sorted order
    // lists_by_table: instead of the per-tile head counts (from which a later kernel numbers the segments over the
    // whole batch), every cluster numbers its own table's segments from 0 and leaves
    //   seg_start[tb0 + t + u] = sorted position where the table's segment u begins, [.. + count] = the table's end
    //   chunk_first[c]         = the table's segment that holds sorted entry c << ck_shift (for c inside the table)
    //   table_cnt[t], tb[t]    = segments and first sorted position of table t (tb[T] = L)
    //                            (cnt_broken instead when boundary offsets are unusable)
    // and zeroes what the kernel behind it counts in (tile_done[c], absmax[t]); that kernel, which sums the segments,
    // adds the tables' bases
    int lists_by_table;
    int parts;                      // (cluster sort with the lists only) clusters of a table, each with its own share of the rows and its own
                                    // lists, numbered table by table; a power of two
    u32 *seg_start, *chunk_first, *table_cnt, *tb, *absmax;
    uint2 *tile_done;
    int ck_shift;
    u32 cnt_broken;
};

// a table whose boundary offsets cannot be used is reported and left out (the same answer in every thread)
__device__ __forceinline__ bool broken_table(const Args &a, int t, int list, int64_t tb0, int64_t tb1, bool reports)
{
    if (tb0 >= 0 && tb1 >= tb0 && tb1 <= a.L && !(a.lists_by_table && ((t == 0 && tb0 != 0) || (t == a.T - 1 && tb1 != a.L))))
        return false;
    if (reports) {
        dq_report(a.status, DQRM_ERR_INDEX_RANGE);
        if (a.lists_by_table) {                    // nothing is summed; the quantiser behind finds an empty gradient
            a.table_cnt[list] = a.cnt_broken;
            a.absmax[t] = 0u;
        }
    }
    return true;
}

// what a table leaves whatever its lookups are (one thread of the table)
__device__ __forceinline__ void open_table(const Args &a, int t, int64_t tb0, int64_t tb1)
{
    a.tb[t] = (u32)tb0;
    if (t == a.T - 1) a.tb[a.T] = (u32)tb1;
    a.absmax[t] = 0u;
    if (tb1 == tb0) a.table_cnt[t] = 0u;
}

// The rows of grad_out of table t's n lookups, into s_pay; whether an offset was found to fall.  Apart from
// load_lookups: batches with an index a bag do not come here
__device__ __noinline__ bool find_bags(const Args &a, int t, u32 tb0, int n, u32 *s_pay)
{
    __shared__ u32 s_last[WARPS];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int32_t *off_t = a.offsets + (int64_t)t * a.B;
    bool bad = false;
    for (int i = tid; i < a.B; i += THREADS) bad |= __ldg(off_t + i) > __ldg(off_t + i + 1);      // (they must not decrease)
    if (a.payload_position) {
        for (int i = tid; i < n; i += THREADS) s_pay[i] = tb0 + i;
        __syncthreads();
        return bad;
    }
    int lo = 0, size = a.B;                        // the first lookup's bag is in [lo, lo + size)
    while (size > 1) {
        const int step = (size + THREADS - 1) / THREADS;
        const int c = __syncthreads_count(tid * step < size && __ldg(off_t + lo + tid * step) <= (int32_t)tb0);
        const int skip = max(c - 1, 0) * step;
        lo += skip;
        size = min(step, size - skip);
    }
    for (int i = tid; i < n; i += THREADS) s_pay[i] = 0u;
    __syncthreads();
    for (int g = lo + tid; g < a.B; g += THREADS) {
        const int64_t o = (int64_t)__ldg(off_t + g) - tb0;
        if (o >= n) break;
        if (o >= 0) atomicMax(&s_pay[o], (u32)(g - lo) + 1u);
    }
    __syncthreads();
    const int share = ((n + WARPS - 1) / WARPS + 31) / 32 * 32, w0 = min(n, warp * share), w1 = min(n, w0 + share);
    u32 last = 0;                                  // of the warp's lookups the last mark
    for (int i0 = w0; i0 < w1; i0 += 32) {
        const u32 v = i0 + lane < w1 ? s_pay[i0 + lane] : 0u, marked = __ballot_sync(0xffffffffu, v != 0u);
        const u32 x = __shfl_sync(0xffffffffu, v, marked ? 31 - __clz(marked) : 0);
        if (marked) last = x;
    }
    if (lane == 0) s_last[warp] = last;
    __syncthreads();
    u32 top = 1;                                   // (the first lookup's bag)
    for (int w = 0; w < warp; ++w)
        if (s_last[w]) top = s_last[w];
    for (int i0 = w0; i0 < w1; i0 += 32) {
        const int i = i0 + lane;
        const u32 v = i < w1 ? s_pay[i] : 0u, marked = __ballot_sync(0xffffffffu, v != 0u), upto = marked & (0xffffffffu >> (31 - lane));
        const u32 x = __shfl_sync(0xffffffffu, v, upto ? 31 - __clz(upto) : 0), y = __shfl_sync(0xffffffffu, v, marked ? 31 - __clz(marked) : 0);
        if (i < w1) s_pay[i] = (u32)((lo + (int)(upto ? x : top) - 1) * a.T + t);
        if (marked) top = y;
    }
    __syncthreads();
    return bad;
}

// Table t's n lookups into registers; every thread of the block calls this.  s_mark: a word for each of them.
//
// In a table of one-index bags in order (n == B, offsets = identity: the Criteo-shaped case) the bag of lookup p is bag p, which
// every lookup checks from the two offsets around it, loaded beside the index.  Otherwise the first lookup's bag is found by a
// search with all threads, every bag marks its first lookup, and the other lookups take the mark before theirs (of bags that
// begin at the same lookup the last counts: the others are empty).  A search for every lookup by itself is a chain of a
// dozen loads.
template <int E>
__device__ __forceinline__ void load_lookups(const Args &a, int t, u32 tb0, int n, u32 nrows, int rounds, u32 (&row)[E], u32 (&pay)[E],
                                             u32 *s_mark, bool &bad)
{
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int w0 = warp * rounds * 32 + lane;
    const int32_t *off_t = a.offsets + (int64_t)t * a.B;
    bool single = n == a.B && !a.payload_position;
    {
        int32_t idx[E];
#pragma unroll
        for (int e = 0; e < E; ++e)
            if (e < rounds) idx[e] = __ldg(a.indices + tb0 + min(w0 + e * 32, n - 1));
        if (n == a.B) {
#pragma unroll
            for (int e = 0; e < E; ++e) {
                if (e < rounds) {
                    const u32 p = min(w0 + e * 32, n - 1);
                    single &= ((u32)__ldg(off_t + p) == tb0 + p) & ((u32)__ldg(off_t + p + 1) == tb0 + p + 1);
                }
            }
        }
#pragma unroll
        for (int e = 0; e < E; ++e) {
            row[e] = 0xffffffffu;
            pay[e] = 0u;
            const int i = w0 + e * 32;
            if (e < rounds && i < n) {
                bad |= (u32)idx[e] >= nrows;
                row[e] = min((u32)max(idx[e], 0), nrows - 1u);
                pay[e] = i * a.T + t;
            }
        }
    }
    if (__syncthreads_and(single)) return;
    bad |= find_bags(a, t, tb0, n, s_mark);
#pragma unroll
    for (int e = 0; e < E; ++e) {
        const int i = w0 + e * 32;
        if (e < rounds && i < n) pay[e] = s_mark[i];
    }
    __syncthreads();                               // (s_mark may be written again)
}

// Places of a warp's entries among those of the warp with the same digit, in order, and how many it has of every digit, in
// mine[] (zero before).  mask: as above, for the warp
template <int E>
__device__ __forceinline__ void rank_digits(const u32 (&key)[E], u32 (&rank)[E], int rounds, int shift, u32 digits, unsigned short *mine, u32 *mask)
{
    const u32 lt = (1u << (threadIdx.x & 31)) - 1u;
#pragma unroll
    for (int e = 0; e < E; ++e) {
        if (e < rounds) {
            const u32 d = (key[e] >> shift) & digits, peers = dq_same_digit_lanes(mask, d, true);
            const u32 before = mine[d];
            __syncwarp();
            if ((peers & lt) == 0u) mine[d] = (unsigned short)(before + __popc(peers));
            rank[e] = before + __popc(peers & lt);
        }
    }
}

// Running sums of the warps' counts of digits 2 tid and 2 tid + 1, two in a word, for threads below BINS / 2: pre[w] = those of
// the warps before w; returns the block's
__device__ __forceinline__ u32 sum_warps(const u32 *cnt, u32 (&pre)[WARPS])
{
    u32 tot = 0;
#pragma unroll
    for (int w = 0; w < WARPS; ++w) pre[w] = cnt[w * (BINS / 2) + threadIdx.x];
#pragma unroll
    for (int w = 0; w < WARPS; ++w) { const u32 c = pre[w]; pre[w] = tot; tot += c; }
    return tot;
}

// Exclusive sum over the threads below BINS / 2, which call it together
__device__ __forceinline__ u32 sum_digits(u32 v, u32 *s_scan)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    u32 incl = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const u32 x = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += x;
    }
    if (lane == 31) s_scan[warp] = incl;
    asm volatile("bar.sync 1, 128;" ::: "memory");
    static_assert(BINS / 2 == 128, "");
    u32 base = incl - v;
#pragma unroll
    for (int w = 0; w < 4; ++w)
        if (w < warp) base += s_scan[w];
    return base;
}

// Stable radix sort of the block's entries by row, rows below 2^bits: digits of at most eight bits, as few passes as that
// allows.  cnt: [WARPS][BINS] 16-bit counters; the result lies in out[0, count), which has room for SORT_ROOM entries at least.
// Per pass: each warp counts and ranks its own entries, 128 threads turn the counts into places, and the entries move once,
// through shared memory, whose bandwidth bounds it: about 25 clocks for 32 entries and 600 a pass beside that (2048 entries, three
// passes: 7.1 K clocks; a sorting network takes 66 steps of 280).
template <int E>
__device__ __forceinline__ void sort_block(u32 (&key)[E], u32 (&pay)[E], int rounds, int count, int bits, u32 *cnt, uint2 *out)
{
    __shared__ u32 s_scan[4];
    const int tid = threadIdx.x, warp = tid >> 5;
    const int i0 = warp * rounds * 32 + (tid & 31);
    const int passes = (bits + 7) / 8;
    if (passes == 0) {
#pragma unroll
        for (int e = 0; e < E; ++e)
            if (e < rounds && i0 + e * 32 < count) out[i0 + e * 32] = make_uint2(key[e], pay[e]);
        __syncthreads();
        return;
    }
    const int dbits = (bits + passes - 1) / passes;
    const u32 digits = (1u << dbits) - 1u;
    unsigned short *mine = reinterpret_cast<unsigned short *>(cnt) + warp * BINS;
    u32 *mask = reinterpret_cast<u32 *>(out) + warp * BINS;
#pragma unroll 1
    for (int pass = 0;; ++pass) {
        const int shift = pass * dbits;
        reinterpret_cast<uint4 *>(cnt)[tid] = make_uint4(0u, 0u, 0u, 0u);
        static_assert(WARPS * BINS * 2 == THREADS * 16, "");
#pragma unroll
        for (int k = 0; k < 2; ++k) reinterpret_cast<uint4 *>(out)[tid + k * THREADS] = make_uint4(0u, 0u, 0u, 0u);
        __syncthreads();
        u32 rank[E];
        rank_digits<E>(key, rank, rounds, shift, digits, mine, mask);
        __syncthreads();
        if (tid < BINS / 2) {
            u32 pre[WARPS];
            const u32 tot = sum_warps(cnt, pre), low = tot & 0xffffu;
            u32 base = sum_digits(low + (tot >> 16), s_scan);
            base |= (base + low) << 16;
#pragma unroll
            for (int w = 0; w < WARPS; ++w) cnt[w * (BINS / 2) + tid] = base + pre[w];
        }
        __syncthreads();
#pragma unroll
        for (int e = 0; e < E; ++e)
            if (e < rounds) {
                const u32 to = mine[(key[e] >> shift) & digits] + rank[e];
                if (to < (u32)count) out[to] = make_uint2(key[e], pay[e]);
            }
        __syncthreads();
        if (pass + 1 == passes) return;
#pragma unroll
        for (int e = 0; e < E; ++e) {
            if (e < rounds) {
                const int i = i0 + e * 32;
                const uint2 pr = i < count ? out[i] : make_uint2(0xffffffffu, 0u);
                key[e] = pr.x;
                pay[e] = pr.y;
            }
        }
        __syncthreads();
    }
}

// Writes sorted table t, entries fin[0, n): arena row keys, payloads, and the lists (lists_by_table)
__device__ __forceinline__ void write_sorted(const Args &a, int t, u32 tb0, u32 tb1, const uint2 *fin)
{
    __shared__ u32 s_wheads[WARPS];                // segment starts in each warp's share, then before it
    __shared__ u32 s_total;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, n = (int)(tb1 - tb0);
    const u32 first_key = (u32)__ldg(a.row_off + t);
    // every warp takes a contiguous share [w0, w1), so that the segment starts before an entry are those of the warps before and a
    // count the warp carries along (of up to 32 rounds lane k keeps the k-th one's head bits, so that the second walk need not
    // read the entries again)
    const int share = ((n + WARPS - 1) / WARPS + 31) / 32 * 32, w0 = min(n, warp * share), w1 = min(n, w0 + share);
    u32 mine = 0, kept = 0;
#pragma unroll 2
    for (int i0 = w0, it = 0; i0 < w1; i0 += 32, ++it) {
        const int i = i0 + lane;
        bool head = false;
        if (i < w1) {
            const uint2 pr = fin[i];
            a.keys_out[tb0 + i] = first_key + pr.x;
            a.vals_out[tb0 + i] = pr.y;
            head = pr.x != (i > 0 ? fin[i - 1].x : 0xffffffffu);
        }
        const u32 bits = __ballot_sync(0xffffffffu, head);
        if (lane == it) kept = bits;
        mine += __popc(bits);
    }
    if (lane == 0) s_wheads[warp] = mine;
    __syncthreads();
    if (warp == 0) {
        const u32 v = lane < WARPS ? s_wheads[lane] : 0u;
        u32 incl = v;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const u32 x = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += x;
        }
        if (lane < WARPS) s_wheads[lane] = incl - v;
        if (lane == WARPS - 1) s_total = incl;
    }
    __syncthreads();
    u32 *segs = a.seg_start + tb0 + t;
    if (tid == 0) {
        a.table_cnt[t] = s_total;
        segs[s_total] = tb1;                       // the slot behind the last segment holds the table's end
    }
    const u32 ck_mask = (1u << a.ck_shift) - 1u, upto_me = 0xffffffffu >> (31 - lane);
    u32 seg = s_wheads[warp] - 1u;
#pragma unroll 2
    for (int i0 = w0, it = 0; i0 < w1; i0 += 32, ++it) {
        const int i = i0 + lane;
        const u32 j = tb0 + i;
        const u32 bits = share <= 1024 ? __shfl_sync(0xffffffffu, kept, it & 31)
                                       : __ballot_sync(0xffffffffu, i < w1 && fin[i].x != (i > 0 ? fin[i - 1].x : 0xffffffffu));
        if (i < w1) {
            const u32 u = seg + __popc(bits & upto_me);            // the entry's segment
            if ((bits >> lane) & 1u) segs[u] = j;
            if ((j & ck_mask) == 0u) {
                a.chunk_first[j >> a.ck_shift] = u;
                a.tile_done[j >> a.ck_shift] = make_uint2(0u, 0u);
            }
        }
        seg += __popc(bits);
    }
}

// bits of a row below `rows`
__device__ __forceinline__ int row_bits(u32 rows) { return rows > 1u ? 32 - __clz(rows - 1u) : 0; }

// a table of up to THREADS * E lookups, by one block; room in shared memory for as many pairs, and SORT_ROOM at least
template <int E>
__device__ __forceinline__ void sort_alone(const Args &a, int t, u32 tb0, u32 tb1, u32 *cnt, uint2 *s_pair)
{
    const int n = (int)(tb1 - tb0), rounds = (n + THREADS - 1) / THREADS;
    const u32 nrows = (u32)(__ldg(a.row_off + t + 1) - __ldg(a.row_off + t));
    bool bad = false;
    if (n == 0) {                                  // (its empty lists have been written)
        const int32_t *off_t = a.offsets + (int64_t)t * a.B;
        for (int i = threadIdx.x; i < a.B; i += THREADS) bad |= __ldg(off_t + i) > __ldg(off_t + i + 1);
        if (bad) dq_report(a.status, DQRM_ERR_INDEX_RANGE);
        return;
    }
    u32 row[E], pay[E];
    load_lookups<E>(a, t, tb0, n, nrows, rounds, row, pay, reinterpret_cast<u32 *>(s_pair), bad);
    if (bad) dq_report(a.status, DQRM_ERR_INDEX_RANGE);
    sort_block<E>(row, pay, rounds, n, row_bits(nrows), cnt, s_pair);
    write_sorted(a, t, tb0, tb1, s_pair);
}

}  // namespace csort

// Per-table stable sort of a batch's lookups by row, one thread-block cluster per table.
//
// The lookups of a batch arrive table-major, so sorting them by arena row is T independent
// sorts of a few thousand to a few tens of thousands of keys each.  A cluster of eight
// blocks owns one table: every block holds one eighth of the table's (row, payload) pairs
// in shared memory, and a least-significant-digit radix sort (8-bit digits, only as many
// passes as the table's row count needs) moves the pairs between the blocks' shared
// memories with distributed-shared-memory stores.  Per pass: per-warp digit counts over
// the block's slice (shared-memory atomics), the eight per-block histograms are exchanged
// through DSMEM, every block derives its scatter offsets, ranks its slice in order (warp ballots, stable)
// and scatters.  Cluster barriers separate the phases; no block waits on anything else.
// Tables whose lookups do not fit the shared-memory slices use the same algorithm on
// global staging buffers.  The result - keys (arena rows) ascending, payloads (rows of
// grad_out) in the original order within equal keys - is written table-major, which is
// the globally sorted order the segmented reduction expects.  On the way out the cluster
// also finds where every row's run begins: either it numbers its table's segments itself
// (the kernel that sums them adds the tables' bases), or it counts the segment starts per
// 2048-entry tile for a kernel that numbers them over the whole batch.
#pragma once
#include "sort_parts.cuh"

namespace csort {

constexpr int CLUSTER = 8;            // blocks per table
constexpr int CLUSTER_HALF = 4;       // ... of which so many work where there are many tables of few lookups
constexpr int CLUSTER_WIDE = 16;      // ... when the batch has so few tables that eight blocks each would leave most SMs idle
constexpr int MAX_PARTS = 4;           // ... of such clusters for a table alone, which would leave more of them idle still

__device__ __forceinline__ u32 *remote(cg::cluster_group &cluster, u32 *p, unsigned rank)
{
    return cluster.map_shared_rank(p, rank);
}

// lanes of the warp that hold the same 8-bit digit as this lane (one call by all lanes; a lane without an
// entry matches nobody).  Slow, but hidden behind the stores into the other blocks' shared memory
__device__ __forceinline__ u32 same_digit_lanes(u32 d, bool valid)
{
    const u32 peers = __match_any_sync(0xffffffffu, valid ? d : 256u + (threadIdx.x & 31));
    return valid ? peers : 0u;
}

// Rows [row0, row1) of a table alone that list `list` of MAX_PARTS takes; the same shares in every block, whose s_room takes
// SAMPLE * (1 + THREADS / SAMPLE) words and a few.  Called by the block together.
constexpr int SAMPLE = 128;
__device__ __forceinline__ void share_rows(const Args &a, int64_t n, int64_t nrows, u32 *s_room, u32 list, int64_t &row0, int64_t &row1)
{
    constexpr int RANKERS = THREADS / SAMPLE;      // threads that rank a lookup of the sample, each against a part of it
    static_assert(MAX_PARTS == 4 && SAMPLE % (4 * RANKERS) == 0, "");
    u32 *s_rank = s_room + SAMPLE, *s_share = s_rank + THREADS, *s_cut = s_share + SAMPLE / 32 * 4;
    const u32 tid = threadIdx.x, i = tid % SAMPLE, rows = (u32)nrows;
    auto even = [&](u32 q) { return (u32)((uint64_t)rows * q >> 2); };
    auto passes = [](u32 x) { return x <= 1 ? 0 : (39 - __clz(x - 1u)) / 8; };
    row0 = even(list);
    row1 = even(list + 1);
    // (a quarter that takes a pass less than the table makes up for lookups that fall unevenly: 10,000 of 120 K rows that are numbered by
    // how often they come 20.2 us a backward, at the quantiles 22.3, by one cluster 21.3; 65,536 29.4, 27.7, 32.4)
    if (n < 32768 && passes((rows + 3) / 4) < passes(rows)) return;
    u32 mine = 0;
    if (tid < SAMPLE) {
        mine = min((u32)max(__ldg(a.indices + tid * n / SAMPLE), 0), rows - 1u);
        s_room[tid] = mine;
        const u32 q = (mine >= even(1)) + (mine >= even(2)) + (mine >= even(3));
        u32 share = 0;
#pragma unroll
        for (u32 k = 0; k < 4; ++k) {
            const u32 in = __ballot_sync(0xffffffffu, q == k);
            if ((tid & 31) == k) share = __popc(in);
        }
        if ((tid & 31) < 4) s_share[tid / 32 * 4 + (tid & 31)] = share;
    }
    __syncthreads();
    u32 most = 0;
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        u32 share = 0;
#pragma unroll
        for (int w = 0; w < SAMPLE / 32; ++w) share += s_share[w * 4 + q];
        most = max(most, share);
    }
    // (a share of two fifths is sorted no later than the whole table by one cluster, and even shares often take a pass less)
    if (most * 5 <= SAMPLE * 2) return;
    const u32 me = s_room[i], j0 = tid / SAMPLE * (SAMPLE / RANKERS);
    u32 rank = 0;
#pragma unroll
    for (u32 j = j0; j < j0 + SAMPLE / RANKERS; j += 4) {
        const uint4 x = *reinterpret_cast<const uint4 *>(s_room + j);
        rank += (x.x < me + (j < i)) + (x.y < me + (j + 1 < i)) + (x.z < me + (j + 2 < i)) + (x.w < me + (j + 3 < i));
    }
    s_rank[tid] = rank;
    __syncthreads();
    if (tid < SAMPLE) {
#pragma unroll
        for (int k = 1; k < RANKERS; ++k) rank += s_rank[k * SAMPLE + tid];
        if (rank % (SAMPLE / 4) == 0) s_cut[rank / (SAMPLE / 4)] = mine;
    }
    __syncthreads();
    u32 cut = 0;                                   // where share q begins: behind the one before, which has a row at least
#pragma unroll
    for (u32 q = 0; q < 4; ++q) {
        if (q == list) row0 = cut;
        cut = q < 3 ? min(rows, max(s_cut[q + 1], cut + 1u)) : rows;
        if (q == list) row1 = cut;
    }
    __syncthreads();                               // (s_room is used again)
}

// What every block of the cluster does.  EPT > 0: for small batches whose tables may be uneven.  A table of up to THREADS * EPT
// lookups, which is nearly all of them, is sorted by one of the cluster's blocks alone (sort_parts.cuh), and only a larger one by
// the cluster.  Which block that is goes round the tables: from the sixteenth on clusters share their SMs with earlier ones, and two
// working blocks on one SM take half as long again (26 tables of 2000 lookups: 11.5 us with the first block working in every
// cluster, 8.2 this way, 8.5 without clusters; from 33 tables on 11.5, a third cluster waiting for its SMs).
//
// PARTS: a table alone, for which one cluster would leave most SMs idle.  a.parts clusters take it, each a share of its rows: every one
// reads all lookups and keeps those of its rows, so nothing passes between the clusters; where its lookups stand behind those
// of the rows before it counts itself, and its segments have lists of their own.  Rows are shared out evenly where a sample of the
// lookups falls evenly, and otherwise at the sample's quantiles: rows may be numbered by how often they come (65,536 lookups all in
// the first quarter of 4 M rows 36.4 us a backward with even shares, 27.7), and padding that is most of a batch becomes a share of one row.
// All pairs fit the blocks' shared memory (the launch sees to that).
//
// OF: blocks launched for every cluster, of which CL call this, from block `from` on; the others have left.
template <int CL, int EPT, bool PARTS, int OF = CL>
__device__ __forceinline__ void sort_by_cluster(const Args &a, unsigned from = 0)
{
    extern __shared__ __align__(16) uint2 s_dyn[];               // pair buffers [2][cap]: (row within table, payload)
    __shared__ __align__(16) u32 s_cnt[WARPS][BINS];
    __shared__ u32 s_hist[BINS];
    __shared__ u32 s_scan[BINS / 32];
    __shared__ u32 s_wheads[WARPS];                // write-out: segment starts in each warp's part of the slice
    __shared__ u32 s_totals[16];                   // ... and in every block's slice (each block sends its own)
    __shared__ u32 s_cbase, s_ctotal;              // ... in the blocks before this one, and in the whole table
    __shared__ u32 s_kept[2], s_below[PARTS ? WARPS : 1];      // PARTS: the block's lookups in the cluster's rows and in rows before them
    __shared__ u32 s_sum[2];                       // ... the cluster's

    cg::cluster_group cluster = cg::this_cluster();
    const unsigned rank0 = OF > CL ? from : 0u, c = cluster.block_rank() - rank0;
    const int list = blockIdx.x / OF, t = PARTS ? 0 : list;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const u32 lt = (1u << lane) - 1u;

    const int64_t tb0 = __ldg(a.offsets + (int64_t)t * a.B), tb1 = __ldg(a.offsets + (int64_t)(t + 1) * a.B);
    const int64_t r0 = __ldg(a.row_off + t), nrows = __ldg(a.row_off + t + 1) - r0;
    if (broken_table(a, t, list, tb0, tb1, c == 0 && threadIdx.x == 0)) return;   // uniform over the cluster
    const int64_t n = tb1 - tb0;
    if (PARTS) {
        if (c == 0 && threadIdx.x == 0) {
            if (list == 0) a.absmax[0] = 0u;
            if (list + 1 == MAX_PARTS) a.tb[MAX_PARTS] = (u32)tb1;
        }
    } else if (a.lists_by_table && c == 0 && threadIdx.x == 0) open_table(a, t, tb0, tb1);
    if constexpr (EPT > 0) {
        if (n <= THREADS * EPT) {
            if (c == (unsigned)(t / 3) % CL) sort_alone<EPT>(a, t, (u32)tb0, (u32)tb1, &s_cnt[0][0], s_dyn);
            return;
        }
    }
    if (n == 0) return;
    int npc = (int)(((n + CL - 1) / CL + 31) / 32 * 32);            // pairs per block
    const bool in_smem = PARTS || npc <= a.cap;
    int my_n = (int)max((int64_t)0, min((int64_t)npc, n - (int64_t)c * npc));
    // the scatter divides every destination by npc: a float reciprocal gives the quotient (a block number,
    // since pos < n <= CL * npc) to within one, and one correction step settles it
    float npc_inv = 1.0f / (float)npc;
    // the cluster's rows, its lookups and their place among the sorted ones (PARTS: known further on)
    int64_t row0 = 0, row1 = nrows, m = n, first = tb0;

    // buffers of this block for stage s (shared memory slices, or this block's part of the global staging)
    // a pair travels as one 8-byte store: distributed-shared-memory traffic is bound by the number of stores
    uint2 *pb0, *pb1;
    if (in_smem) {
        pb0 = s_dyn; pb1 = s_dyn + a.cap;
    } else {
        pb0 = a.gp[0] + tb0 + (int64_t)c * npc; pb1 = a.gp[1] + tb0 + (int64_t)c * npc;
    }
    // ---- load this block's slice: key = row within the table, payload = row of grad_out ----
    // In a table of one-index bags in order (n == B and offsets = identity, the Criteo-shaped case) the bag of
    // the lookup at position p is bag p.  That is checked per lookup from the two offsets around it, which are
    // loaded together with the index, so nothing here waits on another block.  Any other lookup finds its
    // bag by a search of the offsets, which must not decrease inside the table.
    const int32_t *off_t = a.offsets + (int64_t)t * a.B;
    if (n != a.B) {
        bool dec = false;
        const int per = (a.B + CL - 1) / CL;
        const int b0 = c * per, b1 = min(a.B, b0 + per);
        for (int i = b0 + threadIdx.x; i < b1; i += THREADS) dec |= __ldg(off_t + i) > __ldg(off_t + i + 1);
        if (dec) dq_report(a.status, DQRM_ERR_INDEX_RANGE);
    }
    if (blockIdx.x == 0 && threadIdx.x == 0 &&
        (__ldg(a.offsets) != 0 || (int64_t)__ldg(a.offsets + (int64_t)a.T * a.B) != a.L))
        dq_report(a.status, DQRM_ERR_INDEX_RANGE);
    bool bad = false;
    if constexpr (PARTS) {
        // each warp has a contiguous part of the slice: it counts its lookups that are kept, then puts them behind those of the warps before
        const int wsz = ((my_n + WARPS - 1) / WARPS + 31) / 32 * 32, w0 = min(my_n, warp * wsz), w1 = min(my_n, w0 + wsz);
        const int32_t *idx_c = a.indices + tb0 + (int64_t)c * npc;
        int32_t idx[8];
        auto fetch = [&](int i0) {
#pragma unroll
            for (int k = 0; k < 8; ++k) idx[k] = __ldg(idx_c + min(i0 + k * 32 + lane, my_n - 1));
        };
        if (w0 < w1) fetch(w0);                    // (on their way while the sample is looked at)
        share_rows(a, n, nrows, &s_cnt[0][0], (u32)list, row0, row1);
        u32 kept = 0, below = 0;
        for (int i0 = w0; i0 < w1; i0 += 8 * 32) {
            if (i0 != w0) fetch(i0);
#pragma unroll
            for (int k = 0; k < 8; ++k) {
                const bool valid = i0 + k * 32 + lane < w1;
                const int64_t row = min((int64_t)max(idx[k], 0), nrows - 1);
                kept += __popc(__ballot_sync(0xffffffffu, valid && row >= row0 && row < row1));
                below += __popc(__ballot_sync(0xffffffffu, valid && row < row0));
            }
        }
        if (lane == 0) { s_wheads[warp] = kept; s_below[warp] = below; }
        __syncthreads();
        u32 at = 0, all = 0, all_below = 0;
#pragma unroll
        for (int w = 0; w < WARPS; ++w) {
            if (w < warp) at += s_wheads[w];
            all += s_wheads[w];
            all_below += s_below[w];
        }
        if (threadIdx.x == 0) { s_kept[0] = all; s_kept[1] = all_below; }
        for (int i0 = w0; i0 < w1; i0 += 4 * 32) {
            int32_t idx[4], o0[4], o1[4];
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                const int i = min(i0 + k * 32 + lane, my_n - 1);
                idx[k] = __ldg(idx_c + i);
                o0[k] = n == a.B ? __ldg(off_t + (int64_t)c * npc + i) : 1;
                o1[k] = n == a.B ? __ldg(off_t + (int64_t)c * npc + i + 1) : 1;
            }
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                const bool valid = i0 + k * 32 + lane < w1;
                const int64_t p = (int64_t)c * npc + i0 + k * 32 + lane, row = min((int64_t)max(idx[k], 0), nrows - 1);
                const bool single = o0[k] == tb0 + p && o1[k] == tb0 + p + 1, in = valid && row >= row0 && row < row1;
                bad |= valid && ((o0[k] > o1[k]) | (idx[k] < 0) | (idx[k] >= nrows));
                const u32 in_mask = __ballot_sync(0xffffffffu, in), to = at + __popc(in_mask & lt);
                at += __popc(in_mask);
                if (in) {
                    int64_t bag = p;
                    if (!single || n != a.B) {     // (as below)
                        int lo = 0, hi = a.B;
                        while (hi - lo > 1) {
                            const int mid = (lo + hi) >> 1;
                            if ((int64_t)__ldg(off_t + mid) <= tb0 + p) lo = mid; else hi = mid;
                        }
                        bag = lo;
                    }
                    pb0[to] = make_uint2((u32)(row - row0), (u32)bag);
                }
            }
        }
        my_n = (int)all;
    } else {
        for (int i0 = threadIdx.x; i0 < my_n; i0 += 4 * THREADS) {
            int32_t idx[4], o0[4], o1[4];              // (four lookups in flight: one at a time, 34 us instead of 32 for 26 tables of 16 K)
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                const int64_t p = (int64_t)c * npc + min(i0 + k * THREADS, my_n - 1);      // position within the table's lookups
                idx[k] = __ldg(a.indices + tb0 + p);
                o0[k] = n == a.B ? __ldg(off_t + p) : 1;
                o1[k] = n == a.B ? __ldg(off_t + p + 1) : 1;
            }
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                const int i = i0 + k * THREADS;
                if (i >= my_n) break;
                const int64_t p = (int64_t)c * npc + i;
                const bool single = o0[k] == tb0 + p && o1[k] == tb0 + p + 1;
                bad |= (o0[k] > o1[k]) | (idx[k] < 0) | (idx[k] >= nrows);
                int64_t bag = p;
                if (!single || n != a.B) {             // largest bag b with offsets[t*B + b] <= tb0 + p
                    int lo = 0, hi = a.B;
                    while (hi - lo > 1) {
                        const int mid = (lo + hi) >> 1;
                        if ((int64_t)__ldg(off_t + mid) <= tb0 + p) lo = mid; else hi = mid;
                    }
                    bag = lo;
                }
                pb0[i] = make_uint2((u32)min((int64_t)max(idx[k], 0), nrows - 1), a.payload_position ? (u32)(tb0 + p) : (u32)(bag * a.T + t));
            }
        }
    }
    if (bad) dq_report(a.status, DQRM_ERR_INDEX_RANGE);

    int bits = 0;
    while (((int64_t)1 << bits) < row1 - row0) ++bits;
    const int passes = PARTS ? max(1, (bits + 7) / 8) : (bits + 7) / 8;      // (PARTS: the first pass also shares the lookups out over the blocks)
    // the slice of this block is cut into WARPS contiguous parts, walked 32 entries at a time
    int wsz = ((my_n + WARPS - 1) / WARPS + 31) / 32 * 32;
    int w0 = min(my_n, warp * wsz), w1 = min(my_n, w0 + wsz);

    int s = 0;
    __syncthreads();
    // a one-row table takes no pass, so no cluster barrier separates the loads above from the
    // neighbour's read of this slice's last pair in the write-out below
    if (passes == 0) cluster.sync();
    for (int pass = 0; pass < passes; ++pass) {
        const int shift = 8 * pass;
        const uint2 *src = s ? pb1 : pb0;                           // this pass reads stage s ...
        uint2 *dst = s ? pb0 : pb1;                                 // ... and fills the other one
        uint2 *gdst = s ? a.gp[0] : a.gp[1];
        for (int i = threadIdx.x; i < WARPS * BINS; i += THREADS) (&s_cnt[0][0])[i] = 0u;
        __syncthreads();
        // phase 1: digit counts of this warp's part
        for (int i = w0 + lane; i < w1; i += 32) atomicAdd(&s_cnt[warp][(src[i].x >> shift) & 255u], 1u);
        __syncthreads();
        if (threadIdx.x < BINS) {
            u32 h = 0;
#pragma unroll 8
            for (int w = 0; w < WARPS; ++w) h += s_cnt[w][threadIdx.x];
            s_hist[threadIdx.x] = h;
        }
        cluster.sync();
        if (PARTS && pass == 0) {
            if (warp == WARPS - 1) {
                u32 kept = lane < CL ? *remote(cluster, &s_kept[0], lane % CL) : 0u, below = lane < CL ? *remote(cluster, &s_kept[1], lane % CL) : 0u;
                kept = __reduce_add_sync(0xffffffffu, kept);
                below = __reduce_add_sync(0xffffffffu, below);
                if (lane == 0) { s_sum[0] = kept; s_sum[1] = below; }
            }
            __syncthreads();
            m = s_sum[0];
            first = tb0 + s_sum[1];
            npc = (int)(((m + CL - 1) / CL + 31) / 32 * 32);
            npc_inv = 1.0f / (float)npc;
            if (c == 0 && threadIdx.x == 0) a.tb[list] = (u32)first;
            if (m == 0) {                          // (uniform over the cluster)
                if (c == 0 && threadIdx.x == 0) a.table_cnt[list] = 0u;
                cluster.sync();                    // nobody leaves while its shared memory is read
                return;
            }
        }
        // offsets: digits first, then blocks of the cluster, then warps of this block
        u32 tot = 0, pre = 0, incl = 0;
        if (threadIdx.x < BINS) {                  // one thread per digit (the first BINS / 32 warps)
            u32 h[CL];
#pragma unroll
            for (unsigned cc = 0; cc < CL; ++cc) h[cc] = *remote(cluster, &s_hist[threadIdx.x], rank0 + cc);
#pragma unroll
            for (unsigned cc = 0; cc < CL; ++cc) { if (cc < c) pre += h[cc]; tot += h[cc]; }
            incl = tot;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                u32 v = __shfl_up_sync(0xffffffffu, incl, o);
                if (lane >= o) incl += v;
            }
            if (lane == 31) s_scan[warp] = incl;
        }
        __syncthreads();
        if (threadIdx.x < BINS) {
            u32 woff = 0;
            for (int w = 0; w < warp; ++w) woff += s_scan[w];
            u32 run = woff + incl - tot + pre;      // first destination of (digit, this block)
#pragma unroll 8
            for (int w = 0; w < WARPS; ++w) {
                const u32 cnt = s_cnt[w][threadIdx.x];
                s_cnt[w][threadIdx.x] = run;
                run += cnt;
            }
        }
        __syncthreads();
        // phase 2: rank again and scatter into the owners' buffers of the other stage
        for (int i0 = w0; i0 < w1; i0 += 32) {
            const int i = i0 + lane;
            const bool valid = i < w1;
            const uint2 pr = valid ? src[i] : make_uint2(0u, 0u);
            const u32 key = pr.x;
            const u32 d = (key >> shift) & 255u;
            const u32 peers = same_digit_lanes(d, valid);
            const int leader = __ffs(peers) - 1;
            u32 base = 0;
            if (valid && lane == leader) { base = s_cnt[warp][d]; s_cnt[warp][d] = base + __popc(peers); }
            base = __shfl_sync(0xffffffffu, base, leader);
            __syncwarp();
            if (valid) {
                const u32 pos = base + __popc(peers & lt);      // position within the table, < n
                if ((int64_t)pos < m) {
                    if (in_smem) {
                        unsigned owner = (unsigned)((float)pos * npc_inv);       // within one of pos / npc
                        if (owner * (u32)npc > pos) --owner;
                        else if ((owner + 1u) * (u32)npc <= pos) ++owner;
                        const u32 j = pos - owner * npc;
                        cluster.map_shared_rank(dst, rank0 + owner)[j] = pr;
                    } else {
                        gdst[tb0 + pos] = pr;
                    }
                }
            }
        }
        cluster.sync();
        s ^= 1;
        if (PARTS && pass == 0) {
            my_n = (int)max((int64_t)0, min((int64_t)npc, m - (int64_t)c * npc));
            wsz = ((my_n + WARPS - 1) / WARPS + 31) / 32 * 32;
            w0 = min(my_n, warp * wsz);
            w1 = min(my_n, w0 + wsz);
        }
    }
    // ---- write the sorted slice: arena row keys ----
    // and either count, per 2048-entry tile of the sorted order, the entries that start a new row, or number the
    // table's segments right here
    {
        const uint2 *fin = s ? pb1 : pb0;
        u32 prev_last = 0xFFFFFFFFu;               // last row of the previous block's slice (full by construction)
        if (c > 0) {
            const uint2 *pf = in_smem ? cluster.map_shared_rank(s ? pb1 : pb0, rank0 + c - 1)
                                      : (s ? a.gp[1] : a.gp[0]) + tb0 + (int64_t)(c - 1) * npc;
            prev_last = pf[npc - 1].x;
        }
        if (!a.lists_by_table) {
            for (int i0 = warp * 32; i0 < my_n; i0 += THREADS) {
                const int i = i0 + lane;
                const bool valid = i < my_n;
                const int64_t j = tb0 + (int64_t)c * npc + i;
                bool head = false;
                if (valid) {
                    const uint2 pr = fin[i];
                    a.keys_out[j] = (u32)(r0 + pr.x);
                    a.vals_out[j] = pr.y;
                    const u32 before = i > 0 ? fin[i - 1].x : prev_last;
                    head = (c == 0 && i == 0) || before != pr.x;
                }
                const int64_t tile = j >> 11;
                const int64_t tile0 = __shfl_sync(0xffffffffu, tile, 0);
                const u32 m0 = __ballot_sync(0xffffffffu, head && tile == tile0);
                const u32 m1 = __ballot_sync(0xffffffffu, head && tile != tile0);
                if (lane == 0) {
                    if (m0) atomicAdd(&a.tile_heads[tile0], __popc(m0));
                    if (m1) atomicAdd(&a.tile_heads[tile0 + 1], __popc(m1));
                }
            }
        } else {
            // every warp takes a contiguous part [w0, w1) of the slice, so that the segment starts before an entry
            // are those of the blocks before, of the warps before, and a count the warp carries along
            // (a part of up to 1024 entries: lane k keeps the 32 head bits of the part's k-th round, so that the
            // second walk need not read the pairs again)
            const bool few = wsz <= 1024;
            u32 mine = 0, kept = 0;
            for (int i0 = w0, it = 0; i0 < w1; i0 += 32, ++it) {
                const int i = i0 + lane;
                bool head = false;
                if (i < w1) {
                    const int64_t j = first + (int64_t)c * npc + i;
                    const uint2 pr = fin[i];
                    a.keys_out[j] = (u32)(r0 + row0 + pr.x);
                    a.vals_out[j] = pr.y;
                    const u32 before = i > 0 ? fin[i - 1].x : prev_last;
                    head = (c == 0 && i == 0) || before != pr.x;
                }
                const u32 m = __ballot_sync(0xffffffffu, head);
                if (lane == it) kept = m;
                mine += __popc(m);
            }
            if (lane == 0) s_wheads[warp] = mine;
            __syncthreads();
            if (warp == 0) {                       // the warps' bases within the block, and the block's total
                const u32 v = lane < WARPS ? s_wheads[lane] : 0u;
                u32 incl = v;
#pragma unroll
                for (int o = 1; o < 32; o <<= 1) {
                    const u32 x = __shfl_up_sync(0xffffffffu, incl, o);
                    if (lane >= o) incl += x;
                }
                if (lane < WARPS) s_wheads[lane] = incl - v;
                // the block's total goes into every block's shared memory, under cover of the barrier below
                // (sending or fetching made no measurable difference, here or for the passes' digit counts)
                const u32 mine_all = __shfl_sync(0xffffffffu, incl, WARPS - 1);
                if (lane < CL) *cluster.map_shared_rank(&s_totals[c], rank0 + lane) = mine_all;
            }
            cluster.sync();                        // every block's total has arrived (and the warps' bases are here)
            if (warp == 0) {
                const u32 v = lane < CL ? s_totals[lane] : 0u;
                u32 before = lane < (int)c ? v : 0u, all = v;
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) {
                    before += __shfl_xor_sync(0xffffffffu, before, o);
                    all += __shfl_xor_sync(0xffffffffu, all, o);
                }
                if (lane == 0) { s_cbase = before; s_ctotal = all; }
            }
            __syncthreads();
            const u32 base = s_cbase, total = s_ctotal;
            u32 *segs = a.seg_start + first + list;
            if (c == 0 && threadIdx.x == 0) {
                a.table_cnt[list] = total;
                segs[total] = (u32)(first + m);    // the slot behind the last segment holds the table's end
            }
            const u32 ck_mask = (1u << a.ck_shift) - 1u;
            u32 before_me = base + s_wheads[warp];
            for (int i0 = w0, it = 0; i0 < w1; i0 += 32, ++it) {
                const int i = i0 + lane;
                const int64_t j = first + (int64_t)c * npc + i;
                u32 m;
                if (few) {
                    m = __shfl_sync(0xffffffffu, kept, it);
                } else {
                    bool again = false;
                    if (i < w1) {
                        const u32 before = i > 0 ? fin[i - 1].x : prev_last;
                        again = (c == 0 && i == 0) || before != fin[i].x;
                    }
                    m = __ballot_sync(0xffffffffu, again);
                }
                const bool head = (m >> lane) & 1u;
                if (i < w1) {
                    const u32 upto = before_me + __popc(m & (lt | (1u << lane)));     // segment starts in [0, i]
                    if (head) segs[upto - 1] = (u32)j;
                    if (((u32)j & ck_mask) == 0u) {
                        a.chunk_first[j >> a.ck_shift] = upto - 1;
                        a.tile_done[j >> a.ck_shift] = make_uint2(0u, 0u);
                    }
                }
                before_me += __popc(m);
            }
        }
    }
    // nobody leaves while its shared memory may still be read or written (with the lists, the last remote access came before
    // the barrier behind the totals)
    if (!a.lists_by_table) cluster.sync();
}

// Two blocks resident for clusters of eight, so that the clusters of all tables run at once: without the bound the
// kernel takes 95 registers and 26 tables of 16 K lookups 40 us instead of 32, with three 37.  Clusters of sixteen are
// launched for a few tables only and have their SMs to themselves: 36.6 us without the bound, 42.2 with it, for one table
// of 64 K lookups
__host__ __device__ constexpr int resident(int CL) { return CL <= CLUSTER ? 2 : 1; }

template <int CL, int EPT, bool PARTS = false>
__global__ void __launch_bounds__(THREADS, resident(CL))
cluster_sort_kernel(const __grid_constant__ Args a)
{
    dq_wait_before();
    sort_by_cluster<CL, EPT, PARTS>(a);
}

// Clusters of eight of which four blocks sort the table where it fits into their shared memory, and all eight where it does not: how
// large a table is shows on the device alone.  The four that leave make room for the clusters that wait; which four they are alternates
// from table to table, so that clusters that share SMs work on different ones (64 tables of 4000 lookups 46.3 -> 43.2 us a backward).
__global__ void __launch_bounds__(THREADS, resident(CLUSTER))
cluster_sort_half_kernel(const __grid_constant__ Args a)
{
    dq_wait_before();
    const unsigned t = blockIdx.x / CLUSTER, from = t % 2 * CLUSTER_HALF;
    const int64_t n = (int64_t)__ldg(a.offsets + (int64_t)(t + 1) * a.B) - __ldg(a.offsets + (int64_t)t * a.B);
    if (n > (int64_t)CLUSTER_HALF * a.cap) sort_by_cluster<CLUSTER, 0, false>(a);
    else if (blockIdx.x % CLUSTER / CLUSTER_HALF == t % 2) sort_by_cluster<CLUSTER_HALF, 0, false, CLUSTER>(a, from);
}

inline size_t smem_bytes(int cap) { return (size_t)2 * cap * sizeof(uint2); }

// the same for the clusters of which only the first block works in nearly every table: room for the batch in one of them, up
// to what leaves two blocks resident
inline int shared_cap(int64_t L) { return (int)((L < 8 * 5600 ? L / 8 : 5600) + 32) / 32 * 32; }

// pairs per block to provision in shared memory for an expected n per table sorted by `cluster` blocks
inline int choose_cap(int64_t expect_n, int cluster)
{
    int64_t npc = ((expect_n + cluster - 1) / cluster + 31) / 32 * 32;
    int64_t cap = (npc + npc / 4 + 31) / 32 * 32;         // 25 % head room for uneven tables
    if (cap < 256) cap = 256;
    if (cap > 12288) cap = 12288;                         // 192 KB of the 227 KB a block may use
    return (int)cap;
}

}  // namespace csort

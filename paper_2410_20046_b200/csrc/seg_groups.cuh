// Segmented sum of the upstream gradient over the sorted lookups for rows of up to 48 features (wider ones: seg_reduce.cuh, whose
// inputs, arguments and results these are).
//
// A row takes LPR lanes with four features each; a warp has 32 / LPR such lane groups, and every group walks a contiguous
// range of the sorted order by itself, BATCH entries at a time: keys and payloads are one 128-bit load each, read two
// batches ahead, the rows of the next batch are requested before the present one is summed, and rows AHEAD batches further on
// are asked into L2 (by a lane each: with one or two lanes for a row, of 4 and 8 features, only that many of a batch's four rows).  An entry whose key differs from the one before it ends a run and begins the
// next: the number of the group's first segment comes from chunk_first, so that groups need nothing from one another until
// the end.  There a segmented scan over the warp's groups (shuffles) joins the runs that cross them, and
// only a run cut by the edge of a warp's range leaves a partial
// in global memory; the warp that brings a run's last partial adds all of them, in order, as in seg_reduce.cuh.  All sums are
// FP64 and have a shape fixed by the entry positions and the launch, so results are reproducible.  The per-table
// abs-max of the rounded sums is collected on the way: every lane keeps that of its group's present table.
//
// Bound by its chain of latencies: tables' lists, keys, payloads, rows, partials.  Counters at 426 K rows of 64 bytes (cold caches):
// issue slots 26 %, warps 20 % of the SM's, DRAM 19 %, conversions 16 % of their pipe; at 64 K rows of 144 bytes 28, 17, 2 and 13 %.  A
// warp issues 80 instructions an entry of its groups (their runs end at different entries, so that both sides of the branch are
// taken).  Measured on B200 (graph replay, us) against seg_reduce.cuh's way with several groups a warp, which scanned over the groups
// for every tile of 64 entries, looked up the table of every row where a tile held several and had fences around its arrivals: 3.3 K
// rows of 64 bytes in 26 tables 8.8 -> 7.2, 53 K 9.9 -> 8.2, 426 K 18.8 -> 15.5, 5.4 M in bags of 18 100.8 -> 82.4; 426 K rows of 16
// bytes 14.6 -> 10.0, of 32 15.6 -> 12.0, of 80 26.2 -> 23.4, of 128 24.0 -> 21.4; with two groups a warp, 64 K rows of 144 bytes
// 15.5 -> 11.6, 20 K of 192 12.9 -> 9.5, 426 K of 192 39.5 -> 35.0.
// Rows of 52 features and more are better off with a warp each, whose branches are uniform: this way 100 K of 240 bytes took 18.8
// instead of 17.1 us, 53 K of 256 14.7 instead of 11.5, 8.5 M in bags of 20 387 instead of 319, 82 K of 384 25.9 instead of 19.0
// (but 852 K of 256 56.6 instead of 60.3, 13 K of 512 10.8 instead of 12.7; none of it shows beside a forward and a sort).  Integer
// conversions into a scaled range instead of those by the conversion unit: 16.7 -> 18.2.
#pragma once
#include <type_traits>
#include "seg_reduce.cuh"

namespace segred {

constexpr int BATCH = 4;                     // entries that a lane group takes at a time
constexpr int AHEAD = 4;                     // batches between a row's request into L2 and its use
// Twenty warps an SM: with 24 some values are spilled (360 K rows of 80 bytes 25.3 us, 21.5 this way), with 16 long runs wait for
// their rows (5.4 M rows of 64 bytes 90.2, 81.9)
constexpr int GROUPS_THREADS = 128, GROUPS_BLOCKS = 5;
constexpr int CHUNK_SHIFT = 3;               // a group's range begins at a multiple of eight entries
static_assert((1 << CHUNK_SHIFT) % (2 * BATCH) == 0, "the walk takes two batches a round and has no rest of one");

// the rows that come here, and lanes for one of them
__host__ __device__ constexpr bool takes_groups(int D) { return D <= 48; }
__host__ __device__ constexpr int lanes_per_row(int D) { return D <= 4 ? 1 : D <= 8 ? 2 : D <= 16 ? 4 : D <= 32 ? 8 : 16; }

// One range a warp; blocks of two warps at least.  EXACT: every lane holds features.  VEC: features of one access to the rows,
// fewer than four where a caller's rows do not begin on 16 bytes
__host__ __device__ constexpr int unaligned_vec(int LPR) { return LPR == 1 ? 1 : 2; }

template <int LPR, bool EXACT, int VEC = 4>
__global__ void __launch_bounds__(GROUPS_THREADS, GROUPS_BLOCKS)
seg_groups_kernel(const __grid_constant__ Args a)
{
    dq_wait_before();
    constexpr int GP = 32 / LPR;                  // lane groups of the warp
    extern __shared__ __align__(16) u32 s_uoff[];                                                      // [T+1]
    u32 *s_tb = s_uoff + (a.T + 1);                                                      // [T+1] (by table)
    u32 *s_row = s_tb + (a.T + 1);                                                       // [T+1] (by table)
    __shared__ u32 s_broken;
    __shared__ double s_lead[4][GROUPS_THREADS];         // sum of the run that enters a group's range

    const int T = a.T, D = EXACT ? LPR * 4 : a.D, dv = D / 4;
    const int wl = threadIdx.x & 31, lane = wl % LPR, grp = wl / LPR;
    const int threads = (int)blockDim.x;
    const u32 range = (blockIdx.x * threads + threadIdx.x) >> 5;
    const bool on = EXACT || lane < dv;
    const u32 L = (u32)a.L, G = (u32)a.G;
    const u32 per_warp = GP * a.span;             // entries of a warp's range
    const u32 w0 = range < a.ranges ? range * per_warp : L, w1 = w0 + min(L - w0, per_warp);
    const u32 e0 = w0 + min(w1 - w0, grp * a.span), e1 = e0 + min(w1 - e0, a.span);      // of this group's

    // ---- the first two batches' keys and payloads (arrays end on a multiple of 256 bytes)
    auto load4 = [&](const u32 *p, u32 e) { return e < e1 ? __ldg(reinterpret_cast<const uint4 *>(p + e)) : make_uint4(0u, 0u, 0u, 0u); };
    auto payloads = [&](u32 e) {                  // (0 past the end)
        uint4 x = load4(a.vals, e);
        if (e + BATCH > e1) { if (e + 1u >= e1) x.y = 0u; if (e + 2u >= e1) x.z = 0u; x.w = 0u; }
        return x;
    };
    uint4 key = load4(a.keys, e0), val = payloads(e0), key1 = load4(a.keys, e0 + BATCH), val1 = payloads(e0 + BATCH);
    // asks L2 for the rows of the batch at e: a line of a row per lane (rows that do not begin on a line's start: half a line)
    constexpr int LINES = EXACT ? (LPR + 7) / 8 : (LPR + 3) / 4, STEP = EXACT ? 128 : 64;      // lanes for a row
    const int ahead_row = lane / LINES, ahead_byte = (lane % LINES) * STEP;
    auto payload_ahead = [&](u32 e) { return ahead_row < BATCH && e + ahead_row < e1 ? __ldg(a.vals + e + ahead_row) : G; };
    auto ask = [&](u32 row) {
        if (row < G && (EXACT || ahead_byte < D * 4)) dq_prefetch_l2(reinterpret_cast<const char *>(a.grad_out) + (int64_t)row * D * 4 + ahead_byte);
    };
    u32 far[AHEAD - 1];
#pragma unroll
    for (int b = 2; b <= AHEAD; ++b) far[b - 2] = payload_ahead(e0 + b * BATCH);
    // the runs that may be cut: lane 0 has the one that enters the range, lane 1 the one that leaves it
    u32 cut_u = 0u;                               // segment of the entry at the edge, later of the run
    bool cut = false;
    const u32 edge = wl == 0 ? w0 : w1;
    if (wl < 2 && w0 < w1 && edge > 0u && edge < L) {
        cut_u = __ldg(a.chunk_first + (edge >> CHUNK_SHIFT));
        cut = __ldg(a.keys + edge) == __ldg(a.keys + edge - 1u);
    }
    u32 prev = e0 < e1 && e0 > 0u ? __ldg(a.keys + e0 - 1u) : ~key.x;
    u32 u = e0 < e1 ? __ldg(a.chunk_first + (e0 >> CHUNK_SHIFT)) : 0u;
    // ---- the tables' first segments, positions and rows; the counts' running sum is one warp's work
    if (a.by_table) {
        if (threadIdx.x < 32) {
            u32 run = 0;
            bool broken = false;
            for (int t0 = 0; t0 < T; t0 += 32) {
                const int t = t0 + wl;
                const u32 cnt = t < T ? __ldg(a.table_cnt + t) : 0u;
                broken |= cnt == CNT_BROKEN;
                u32 incl = cnt;
#pragma unroll
                for (int o = 1; o < 32; o <<= 1) {
                    const u32 v = __shfl_up_sync(0xffffffffu, incl, o);
                    if (wl >= o) incl += v;
                }
                if (t < T) s_uoff[t] = run + incl - cnt;
                run += __shfl_sync(0xffffffffu, incl, 31);
            }
            broken = __any_sync(0xffffffffu, broken);
            if (wl == 0) { s_uoff[T] = run; s_broken = broken; }
        } else {
            for (int t = threadIdx.x - 32; t <= T; t += threads - 32) { s_tb[t] = __ldg(a.tb + t); s_row[t] = (u32)__ldg(a.row_off + (t >> a.parts_log)); }
        }
    } else {
        for (int t = threadIdx.x; t <= T; t += threads) s_uoff[t] = (u32)__ldg(a.uniq_off + t);
        if (threadIdx.x == 0) s_broken = 0u;
    }
    __syncthreads();
    if (a.by_table && blockIdx.x == 0)
        for (int t = threadIdx.x; t <= T >> a.parts_log; t += threads) a.uniq_off[t] = s_broken ? 0 : (int32_t)s_uoff[t << a.parts_log];
    if (s_broken || w0 >= w1) return;             // (warp-uniform; no block barrier below)

    // a one-index batch reads every upstream-gradient row once, a pooled one as often as the bag has indices
    const uint64_t keep = dq_policy_evict_last();
    const uint64_t pol = L <= G ? dq_policy_evict_first() : dq_policy_evict_normal();
    const float4 *go = reinterpret_cast<const float4 *>(a.grad_out) + (on ? lane : 0);
    auto load_row = [&](u32 row) {
        const float4 *p = go + (int64_t)row * dv;
        if constexpr (VEC == 4) {
            return dq_ld_nc(p, pol);
        } else if constexpr (VEC == 2) {
            const float2 *q = reinterpret_cast<const float2 *>(p), x = ld_row(q, pol), y = ld_row(q + 1, pol);
            return make_float4(x.x, x.y, y.x, y.y);
        } else {
            const float *q = reinterpret_cast<const float *>(p);
            return make_float4(__ldg(q), __ldg(q + 1), __ldg(q + 2), __ldg(q + 3));
        }
    };
    auto checked = [&](u32 row) {
        if (row >= G) { dq_report(a.status, DQRM_ERR_INDEX_RANGE); row = 0u; }
        return row;
    };
    // the rows of a batch, all at once (any row for entries past the end, and a vector of the row for lanes past its end:
    // nothing is done with either)
    auto request = [&](const uint4 &v, float4 (&r)[BATCH]) {
        r[0] = load_row(checked(v.x));
        r[1] = load_row(checked(v.y));
        r[2] = load_row(checked(v.z));
        r[3] = load_row(checked(v.w));
    };
    float4 v[2][BATCH];
    request(val, v[0]);
#pragma unroll
    for (int b = 2; b < AHEAD; ++b) ask(far[b - 2]);
    u32 soon = far[AHEAD - 2];                    // payload of the batch that is asked for next

    int t = a.by_table ? last_not_above(s_tb, 0, T, e0) : last_not_above(s_uoff, 0, T, u);
    if (a.by_table) u += s_uoff[t];
    // of a run that is cut: where it begins and ends, and so in which ranges its pieces are
    u32 first_range = 0, last_range = 0, t_run = 0;
    if (cut) {
        t_run = (u32)(a.by_table ? last_not_above(s_tb, 0, T, edge) : last_not_above(s_uoff, 0, T, cut_u));
        const u32 *start = a.seg_start + (a.by_table ? s_tb[t_run] + t_run + cut_u : cut_u);
        first_range = __ldg(start) / per_warp;
        last_range = (__ldg(start + 1) - 1u) / per_warp;
        if (a.by_table) cut_u += s_uoff[t_run];
    }
    const bool head0 = key.x != prev;             // (true for a group without entries, too)
    u -= head0;                                   // the run that is open when the group begins
    const u32 u_in = u;
    u32 t_end = s_uoff[t + 1], t_row = a.by_table ? s_row[t] : 0u;
    float m = 0.f;                                // abs-max of the rows of table t that this lane has rounded
    auto note = [&](int tt, float x) { if (x > 0.f) atomicMax(a.absmax + (tt >> a.parts_log), __float_as_uint(x)); };
    auto store_row = [&](u32 uu, const double (&acc)[4]) {
        float x = 0.f;
        if (on) {
            const float4 r = rounded(acc, x);
            float *p = reinterpret_cast<float *>(reinterpret_cast<float4 *>(a.grad_rows + (int64_t)uu * D) + lane);
            if constexpr (VEC == 4) {
                dq_st_keep(reinterpret_cast<float4 *>(p), r, keep);      // quantise+update reads it next
            } else if constexpr (VEC == 2) {
                st_row(reinterpret_cast<float2 *>(p), make_float2(r.x, r.y), keep);
                st_row(reinterpret_cast<float2 *>(p) + 1, make_float2(r.z, r.w), keep);
            } else {
                p[0] = r.x; p[1] = r.y; p[2] = r.z; p[3] = r.w;
            }
        }
        return x;
    };
    double acc[4] = {0.0, 0.0, 0.0, 0.0};         // the open run
    bool seen = false;                            // a segment has begun in the range
    auto entry = [&](u32 k, const float4 &x) {
        if (k != prev) {
            prev = k;
            if (seen) {
                m = fmaxf(m, store_row(u, acc));
            } else {
#pragma unroll
                for (int q = 0; q < 4; ++q) s_lead[q][threadIdx.x] = acc[q];
                seen = true;
            }
            ++u;
            if (u >= t_end) {
                note(t, m);
                m = 0.f;
#pragma unroll 1
                do { ++t; t_end = s_uoff[t + 1]; } while (u >= t_end);
                if (a.by_table) t_row = s_row[t];
            }
            if (a.by_table && lane == 0) a.unique_rows[u] = (int32_t)(k - t_row);
#pragma unroll
            for (int q = 0; q < 4; ++q) acc[q] = 0.0;
        }
        add(acc, x);
    };
    // (every group of the warp makes as many rounds as the first, whose range is the longest)
    const u32 n0 = min(w1 - w0, a.span);
    auto walk = [&](auto whole) {                 // whole: every group of the warp has all its entries
#pragma unroll 1
        for (u32 b = 0; b < n0; b += 2 * BATCH) {
            const u32 e = e0 + b;
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const uint4 k = key;
                request(val1, v[h ^ 1]);
                key = key1;
                key1 = load4(a.keys, e + (h + 2) * BATCH);
                val1 = payloads(e + (h + 2) * BATCH);
                ask(soon);
                soon = payload_ahead(e + (h + AHEAD + 1) * BATCH);
                const u32 left = decltype(whole)::value ? BATCH : e1 - min(e1, e + h * BATCH);
                if (left > 0u) entry(k.x, v[h][0]);
                if (left > 1u) entry(k.y, v[h][1]);
                if (left > 2u) entry(k.z, v[h][2]);
                if (left > 3u) entry(k.w, v[h][3]);
            }
        }
    };
    if (w1 - w0 == per_warp) walk(std::true_type()); else walk(std::false_type());
    __syncwarp();

    // ---- the runs that cross the groups: a scan makes of acc the run that is open behind each group
    const bool had = e0 < e1;
    bool any = seen;
#pragma unroll
    for (int o = 1; o < GP; o <<= 1) {
        const bool any_o = __shfl_up_sync(0xffffffffu, any, o * LPR);
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const double x = __shfl_up_sync(0xffffffffu, acc[q], o * LPR);
            if (grp >= o && !any) acc[q] = x + acc[q];
        }
        if (grp >= o) any |= any_o;
    }
    const bool any_before = GP > 1 && __shfl_up_sync(0xffffffffu, any, LPR) && grp > 0;
    const int t_before = __shfl_up_sync(0xffffffffu, t, LPR < 32 ? LPR : 0);
    {
        double in[4];                             // the run that was open when the group began
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const double x = __shfl_up_sync(0xffffffffu, acc[q], LPR < 32 ? LPR : 0);
            in[q] = (grp > 0 ? x : 0.0) + (seen ? s_lead[q][threadIdx.x] : 0.0);
        }
        if (seen) {
            if (any_before) {
                const float x = store_row(u_in, in);
                if (t_before == t) m = fmaxf(m, x); else note(t_before, x);
            } else if (!(grp == 0 && head0)) {    // it comes from the range before
                if (on) {
#pragma unroll
                    for (int q = 0; q < 4; ++q) a.partials[(size_t)range * 2 * D + lane * 4 + q] = in[q];
                }
            }
        }
    }
    __syncwarp();
    // ---- the run that is open at the end of the range, in the last group that has entries
    const int last_grp = (int)(31 - __clz(__ballot_sync(0xffffffffu, had))) / LPR;
    const bool any_all = __shfl_sync(0xffffffffu, any, last_grp * LPR);
    const u32 cuts = __ballot_sync(0xffffffffu, cut);
    const bool cut_trail = any_all && (cuts & 2u);
    if (grp == last_grp) {
        if (!any_all || cut_trail) {
            if (on) {
#pragma unroll
                for (int q = 0; q < 4; ++q) a.partials[((size_t)range * 2 + (any_all ? 1 : 0)) * D + lane * 4 + q] = acc[q];
            }
        } else {
            m = fmaxf(m, store_row(u, acc));
        }
    }
    __syncwarp();
    {   // the maxima: one atomic where the whole warp is in one table
        const int t_first = __shfl_sync(0xffffffffu, t, 0);
        if (__all_sync(0xffffffffu, t == t_first)) {
            const u32 mb = __reduce_max_sync(0xffffffffu, __float_as_uint(m));
            if (wl == 0 && mb) atomicMax(a.absmax + (t_first >> a.parts_log), mb);
        } else {
            note(t, m);
        }
    }

    // ---- the warp that brings a cut run's last piece adds the pieces
    if (!any_all) cut = cut && wl == 0;           // (one run all along: a single piece)
    if (cuts == 0u) return;
    const u32 group = range / FOLD_GROUP;
    u32 last = 0, groups = 0;                     // pieces to add here; the run's groups, when it has many pieces
    if (cut) {
        const u32 g0 = first_range / FOLD_GROUP;
        u32 pieces = last_range - first_range + 1;
        u32 *arrived = &a.range_done[first_range].x;
        if (pieces > FOLD_GROUP) {
            groups = last_range / FOLD_GROUP - g0 + 1;
            pieces = min(last_range, group * FOLD_GROUP + FOLD_GROUP - 1) - max(first_range, group * FOLD_GROUP) + 1;
            arrived = &a.range_done[2 * group + (group == g0 ? 1 : 0)].y;
        }
        last = arrive(arrived) == pieces - 1u ? pieces : 0u;
    }
    __syncwarp();
    // adds np partials of D features each (`at(p)` = where piece p lies), this lane's features
    auto fold = [&](int np, double (&sum)[4], auto at) {
#pragma unroll
        for (int x = 0; x < 4; ++x) sum[x] = 0.0;
#pragma unroll 1
        for (int p0 = grp; on && p0 < np; p0 += 4 * GP) {
            double x[4][4];
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const int p = p0 + j * GP;
                const double *src = at(min(p, np - 1)) + lane * 4;
#pragma unroll
                for (int q = 0; q < 4; ++q) x[j][q] = p < np ? __ldcg(src + q) : 0.0;
            }
#pragma unroll
            for (int j = 0; j < 4; ++j)
#pragma unroll
                for (int q = 0; q < 4; ++q) sum[q] += x[j][q];
        }
        __syncwarp();
#pragma unroll
        for (int o = LPR; o < 32; o <<= 1)
#pragma unroll
            for (int x = 0; x < 4; ++x) sum[x] += __shfl_xor_sync(0xffffffffu, sum[x], o);
    };
#pragma unroll 1
    for (int q = 0; q < 2; ++q) {
        const int np = (int)__shfl_sync(0xffffffffu, last, q);
        if (np == 0) continue;
        const u32 ur = __shfl_sync(0xffffffffu, cut_u, q), tr = __shfl_sync(0xffffffffu, t_run, q), f = __shfl_sync(0xffffffffu, first_range, q);
        const u32 ng = __shfl_sync(0xffffffffu, groups, q), g0 = f / FOLD_GROUP;
        const u32 p_first = ng ? max(f, group * FOLD_GROUP) : f;
        double sum[4];
        fold(np, sum, [&](int p) { return a.partials + ((size_t)(p_first + p) * 2 + (p_first + p == f ? 1 : 0)) * D; });
        if (ng) {
            if (grp == 0 && on) {
#pragma unroll
                for (int x = 0; x < 4; ++x) a.group_partials[((size_t)group * 2 + (group == g0 ? 1 : 0)) * D + lane * 4 + x] = sum[x];
            }
            __syncwarp();
            bool final = false;
            if (wl == 0) final = arrive(&a.range_done[f].x) == ng - 1u;
            __syncwarp();                         // (what lane 0 has acquired, the warp loads)
            if (!__shfl_sync(0xffffffffu, final, 0)) continue;
            fold((int)ng, sum, [&](int p) { return a.group_partials + ((size_t)(g0 + p) * 2 + (p == 0 ? 1 : 0)) * D; });
        }
        if (grp == 0) note((int)tr, store_row(ur, sum));
        __syncwarp();
    }
}

}  // namespace segred

// Segmented sum of the upstream gradient over the sorted lookups (second half of the backward; paper
// Section 4.3 / Appendix B.1: duplicates of a row are coalesced).
//
// Input: keys[L] (arena rows, ascending), vals[L] (row of grad_out for each lookup, in stable order),
// chunk_first[c] = index of the segment that holds sorted entry c << log2_of(I), seg_start[] = sorted position where
// every segment begins; the segments are numbered over the whole batch, or per table (Args::by_table), and
// in the second case this kernel also writes unique_rows and uniq_off.
//
// A warp walks a contiguous range of the sorted order by itself (no block barrier inside the walk), a tile of I
// entries at a time.  The sum is bound by the latency of the chain index -> payload -> row: indices are fetched a
// tile ahead, the rows of the next tile are asked into L2 as soon as its payloads are there (without that the kernel
// took 89 instead of 71 us on 852 K rows of 256 bytes, 541 instead of 318 us on 8.5 M), and the next batch of rows is
// requested before the present one is summed.  A row takes the whole warp, VEC features a lane (rows of up to 48 features go
// to seg_groups.cuh): every branch on a run's end is then uniform and a run that goes on is simply carried in
// registers.  Only a run cut by the edge of a warp's range leaves a partial
// in global memory; the warp that brings a run's last partial adds all of them, in order (nobody waits; the pieces of a
// long run are first added by groups of 32 ranges, or one warp's chain over hundreds of them is what the kernel waits
// for).  All sums are
// FP64 and have a shape fixed by the entry positions and the launch, so results are reproducible.  The per-table
// abs-max of the rounded sums is collected on the way.
//
// Measured on B200 (cold L2, alone) against a kernel that walked 32-entry chunks per lane group and left
// a partial per chunk for a second launch: 852 K rows of 256 bytes
// 69.9 + 12.9 -> 70.9 us, 8.5 M lookups of 256-byte rows 330 + 63 -> 318 us.
#pragma once
#include "common.cuh"

namespace segred {

constexpr int THREADS = 256;
constexpr int WARPS = THREADS / 32;
constexpr u32 FOLD_GROUP = 32;               // ranges whose pieces of one run are added before the groups' sums are
constexpr u32 CNT_BROKEN = 0xFFFFFFFFu;      // table_cnt[t]: the table's boundary offsets were unusable (reported)

// features per lane for feature size D (D > 128: 128 features per warp)
__host__ __device__ constexpr int floats_per_lane(int D) { return D <= 64 ? 2 : 4; }
__host__ __device__ constexpr int column_blocks(int D) { return (D + 127) / 128; }
// rows of a batch, of which one is in flight while the other is summed.  With two features a lane four of them leave room for a fourth
// resident block: 852 K rows of 256 bytes 58.4 -> 56.5 us, 1.3 M in bags of twenty 97.9 -> 89.7 (eight rows and three blocks
// before; five blocks 65 and more: values are spilled).  With four features a lane a fourth block spills, 984 K rows of 512 bytes 82 -> 119
constexpr int BATCH_ROWS = 4;
__host__ __device__ constexpr int log2_of(int tile) { return tile == 8 ? 3 : tile == 16 ? 4 : 5; }
// ... but where that gives a warp less than 18 entries, registers count for more than warps: 53 K rows of 208 bytes 17.6 us a backward with
// four blocks, 17.2 with three (Zipf 1.1 19.1 and 18.6), 80 K 28.8 and 28.1 (28.9 and 28.2); 112 K 30.1 and 31.3
inline int sum_blocks(int D, int64_t L, int num_sms) { return floats_per_lane(D) == 2 && L >= 18LL * num_sms * 4 * WARPS ? 4 : 3; }
// Entries of a tile: 8, 16 or (64 features alone) 32.  A warp that has one tile takes its batches of rows one after the other, 4 to 8 us
// for 32 rows, so a batch that would give every resident warp few tiles is cut finely; a tile's heads and keys cost the same whatever it
// holds.  Measured on B200 (us a backward; 128 features, tiles of 8 / of 16, uniform indices and Zipf 1.1: 26 K rows 13.4 / 17.1 and 15.7 / 17.3,
// 213 K 56.2 / 60.5 and 47.0 / 49.3; 16 / 32: 416 K 118 / 124 and 80.1 / 88.6, 855 K in bags of two 263 / 276 and 166 / 183; 96 features, 16 /
// 32: 416 K 93.9 / 104 and 73.5 / 91.5, 901 K in bags of nine 189 / 202 and 149 / 175).  Rows whose lanes stand idle part from tiles of 8
// sooner (52 features, 8 / 16: 53 K 17.5 / 16.8 and 18.9 / 18.1, 156 K 38.7 / 35.9 and 36.1 / 33.5, but in bags of six 94 K 31.1 / 33.0).
// 64 features, an index a bag: 8 / 16 213 K 42.0 / 43.9 and 38.3 / 37.0, 416 K 66.7 / 70.4 and 57.6 / 56.2, 16 / 32 624 K 101 / 107 and
// 75.2 / 78.9, 900 K 157 / 170 and 114 / 117; in bags 8 / 16 416 K 69.8 / 69.9 and 56.9 / 56.4, 400 K in bags of twenty 80.5 / 77.6 and 63.1 /
// 61.0, but with bags of more than four 16 / 32 901 K 150 / 152 and 122 / 119, 2 M 226 / 227 and 162 / 158, 8.5 M 710 / 692 and 497 / 475
inline int tile_entries(int D, int64_t L, int num_sms, int64_t bags)
{
    const int64_t warps = (int64_t)num_sms * (floats_per_lane(D) == 2 ? 4 : 3) / column_blocks(D) * WARPS;
    if (L < (D < 64 ? 24 : D == 64 && L > bags ? 72 : 96) * warps) return 8;
    return D == 64 && L > 4 * bags ? 32 : 16;
}
// Where a warp would get far more than 512 entries its range has fewer, and there are more blocks than the GPU holds at once: they pass over
// the tables one after the other, each table's share of grad_out stays in L2 while it is read from all sides, and warps with many short
// runs hold up fewer others.  Measured on B200 (us a backward, one range for every resident warp / of 256 entries, Zipf 1.1): 64 features,
// 8.5 M rows in bags of twenty 546 / 512, 5.1 M in bags of twelve 363 / 346, 3.6 M 261 / 253, 2 M 167 / 172; of 52 features, one range / 256
// entries / 384: 8.5 M 643 / 678 / 656, 3.6 M 304 / 317 / 311 (uniform 384 / 373 / 372), 3.3 M in bags of two 390 / 358 / 363, 2.6 M in
// bags of twelve 248 / 268 / 277.  A loop over the ranges in each warp, instead of more blocks, costs registers (356 against 276 us a sum).
// With four features a lane it does not help: 1.6 M rows of 512 bytes 116 -> 122
constexpr int RANGE_ENTRIES = 256;
inline int range_tiles(int D, int64_t tiles, int64_t warps, int tile)
{
    const int64_t even = (tiles + warps - 1) / warps;
    if (tile == 8 || floats_per_lane(D) != 2 || even <= (tile == 32 ? 16 : 36)) return (int)even;
    return (D == 64 || even < 48 ? RANGE_ENTRIES : RANGE_ENTRIES + RANGE_ENTRIES / 2) / tile;
}
// of such ranges, for L lookups (rows of 48 features and fewer have ranges of their own, seg_groups.cuh)
inline int64_t max_ranges(int D, int64_t L) { return D > 48 && floats_per_lane(D) == 2 ? L / RANGE_ENTRIES + 1 : 0; }

struct Args {
    const u32 *keys, *vals, *seg_start, *chunk_first;
    // zero: .x [range] partials that have arrived for the run that begins in a range, .y [group][2] for a run of many
    // pieces, those of its pieces that lie in a group of 32 ranges (the run that comes into the group, the one that begins
    // in it)
    uint2 *range_done;
    // by_table: the cluster sort numbered each table's segments from 0: table t's starts sit at
    // seg_start[tb[t] + t + .] (tb[t] = first sorted position of the table, one slot more than it has segments: the
    // last holds the table's end), chunk_first[c] counts within the table that holds entry c << log2_of(I), table_cnt[t] says
    // how many segments the table has (CNT_BROKEN: nothing is summed, no row is updated); unique_rows and uniq_off
    // are then written here, with the tables' bases added
    int by_table;
    int parts_log;
    const u32 *table_cnt, *tb;
    const int64_t *row_off;
    int32_t *unique_rows, *uniq_off;
    const float *grad_out;
    float *grad_rows;
    double *partials;           // [ranges][2][D]: run that enters the range, run that leaves it
    double *group_partials;     // [ranges / 32 + 1][2][D]: the same for groups of 32 ranges
    u32 *absmax;                // [T] zero
    int T, D;                   // T: lists, 2^parts_log for every table (by_table; one otherwise)
    int64_t L, G;
    int64_t num_tiles;          // rows that take a warp: tiles, tiles of a warp's range, blocks of 128 features
    int range_tiles, columns;
    u32 span, ranges;           // rows that take a lane group: entries of a group's range, a multiple of eight, and ranges of warps
    int *status;
};

inline size_t smem_bytes(int T) { return (size_t)(T + 1) * 3 * sizeof(u32); }

// Counts an arrival behind what the warp has stored before it (__syncwarp between), and ahead of what it loads afterwards when
// it is the last.  One instruction that releases and acquires; an atomic between two fences of __threadfence took
// up to two thousand clocks more at the end of the kernel (53 K rows of 256 bytes 11.5 us that way, 10.4 this way; 3.3 K of 64 7.5 and
// 6.8, 426 K of 64 16.8 and 15.9)
__device__ __forceinline__ u32 arrive(u32 *count)
{
    u32 before;
    asm volatile("atom.acq_rel.gpu.global.add.u32 %0, [%1], 1;" : "=r"(before) : "l"(count) : "memory");
    return before;
}

// largest t in [lo, T) with list[t] <= x (list ascends; of tables that share a start, the last)
__device__ __forceinline__ int last_not_above(const u32 *list, int lo, int T, u32 x)
{
    int hi = T;
    while (hi - lo > 1) {
        const int mid = (lo + hi) >> 1;
        if (list[mid] <= x) lo = mid; else hi = mid;
    }
    return lo;
}

// VEC consecutive floats (2 or 4)
template <int VEC> struct Vec;
template <> struct Vec<2> { typedef float2 type; };
template <> struct Vec<4> { typedef float4 type; };

__device__ __forceinline__ float2 ld_row(const float2 *p, uint64_t pol)
{
    float2 v;
    asm volatile("ld.global.nc.L2::cache_hint.v2.f32 {%0, %1}, [%2], %3;\n" : "=f"(v.x), "=f"(v.y) : "l"(p), "l"(pol));
    return v;
}
__device__ __forceinline__ float4 ld_row(const float4 *p, uint64_t pol) { return dq_ld_nc(p, pol); }
__device__ __forceinline__ void st_row(float2 *p, const float2 &v, uint64_t pol)
{
    asm volatile("st.global.L2::cache_hint.v2.f32 [%0], {%1, %2}, %3;\n" ::"l"(p), "f"(v.x), "f"(v.y), "l"(pol) : "memory");
}
__device__ __forceinline__ void st_row(float4 *p, const float4 &v, uint64_t pol) { dq_st_keep(p, v, pol); }

__device__ __forceinline__ void add(double (&acc)[2], const float2 &v) { acc[0] += (double)v.x; acc[1] += (double)v.y; }
__device__ __forceinline__ void add(double (&acc)[4], const float4 &v)
{
    acc[0] += (double)v.x; acc[1] += (double)v.y; acc[2] += (double)v.z; acc[3] += (double)v.w;
}
// rounds a finished sum
__device__ __forceinline__ float2 rounded(const double (&a)[2], float &mx)
{
    const float2 r = make_float2((float)a[0], (float)a[1]);
    mx = fmaxf(fabsf(r.x), fabsf(r.y));
    return r;
}
__device__ __forceinline__ float4 rounded(const double (&a)[4], float &mx)
{
    const float4 r = make_float4((float)a[0], (float)a[1], (float)a[2], (float)a[3]);
    mx = fmaxf(fmaxf(fabsf(r.x), fabsf(r.y)), fmaxf(fabsf(r.z), fabsf(r.w)));
    return r;
}

// abs-max of a row where the tile holds rows of several tables (rare in large batches: kept out of the unrolled code).
// Called by the warp together.
__device__ __noinline__ void note_max(u32 *absmax, const u32 *s_uoff, int t_first, int T, int parts_log, u32 u, float x)
{
    const u32 m = __reduce_max_sync(0xffffffffu, __float_as_uint(x));
    if ((threadIdx.x & 31) == 0 && m) atomicMax(absmax + (last_not_above(s_uoff, t_first, T, u) >> parts_log), m);
}

// I: entries of a tile.  blockIdx.x * WARPS + warp: range of tiles and block of 128 features (COLS: D > 128, there are several).  EXACT: every lane
// holds features.  Rows of 3 KB and more are not asked into L2 ahead: their blocks of features ask for whole rows already
// (65 K rows of 4080 bytes 138 us, 154 with the request; of 2064 bytes 87 and 85)
template <int VEC, bool EXACT, int I, bool COLS, int BLOCKS>
__global__ void __launch_bounds__(THREADS, BLOCKS)
seg_sum_kernel(const Args a)
{
    dq_wait_before();
    constexpr int C = BATCH_ROWS;
    constexpr int NB = I / C;                     // batches per tile
    static_assert(NB % 2 == 0 && I <= 32, "");
    typedef typename Vec<VEC>::type vec_t;
    extern __shared__ __align__(16) u32 s_uoff[];                                                      // [T+1]
    u32 *s_tb = s_uoff + (a.T + 1);                                                      // [T+1] (by table)
    u32 *s_row = s_tb + (a.T + 1);                                                       // [T+1] (by table)
    __shared__ u32 s_broken;

    const int T = a.T, D = EXACT && !COLS ? 32 * VEC : a.D, dv = D / VEC;
    const int wl = threadIdx.x & 31;
    // the blocks of features of a range are neighbouring warps: a row's pieces are asked for at about the same time
    const u32 cols = COLS ? (u32)a.columns : 1u, slot = blockIdx.x * WARPS + (threadIdx.x >> 5);
    const u32 col = COLS ? slot % cols : 0u, range = COLS ? slot / cols : slot;
    const int cv = (int)col * 32 + wl;         // this lane's vector of the row
    const bool on = EXACT || cv < dv;
    const bool first_col = col == 0u;
    const u32 tile0 = min((u32)a.num_tiles, range * (u32)a.range_tiles);
    const u32 tile1 = min((u32)a.num_tiles, tile0 + (u32)a.range_tiles);

    // ---- indices of a tile, one entry per lane.  An entry starts a segment when its key differs from the key
    // before it
    u32 kn, vn, kp;
    auto fetch = [&](u32 tile) {
        const int64_t i = (int64_t)tile * I + wl;
        kn = vn = kp = 0u;
        if (i < a.L && (I == 32 || wl < I)) {
            kn = __ldg(a.keys + i);
            vn = __ldg(a.vals + i);
            kp = i > 0 ? __ldg(a.keys + i - 1) : ~kn;
        }
    };
    u32 kc, vc, heads;                            // the present tile's keys, payloads and head bits
    auto take = [&]() {
        heads = __ballot_sync(0xffffffffu, kn != kp);         // (equal past the end)
        kc = kn;
        vc = vn;
        if ((int64_t)vc >= a.G) { dq_report(a.status, DQRM_ERR_INDEX_RANGE); vc = 0u; }
    };
    fetch(tile0);
    u32 u_base = tile0 < tile1 ? a.chunk_first[(int64_t)tile0 * I >> log2_of(I)] : 0u;
    // the runs that may be cut: lane 0 has the one that enters the range, lane 1 the one that leaves it.  Where rows take several
    // warps what is to be known of them is asked for now (243 K rows of 1200 bytes 111 -> 109 us; narrower rows, whose loop wants the
    // registers, 78.6 -> 79.5 at 520 K of 512 bytes, and small batches are better without)
    constexpr bool EARLY = COLS && I > 8;
    u32 cut_u = 0u;                               // segment of the entry at the edge
    bool cut = false;
    const u32 edge = (wl == 0 ? tile0 : tile1) * I;
    if (EARLY && wl < 2 && tile0 < tile1 && edge > 0u && edge < (u32)a.L) {
        cut_u = __ldg(a.chunk_first + (edge >> log2_of(I)));
        cut = __ldg(a.keys + edge) == __ldg(a.keys + edge - 1u);
    }
    if (a.by_table) {
        if (threadIdx.x < 32) {                   // the tables' first segments: a running sum over their counts
            u32 run = 0;
            bool broken = false;
            for (int t0 = 0; t0 < T; t0 += 32) {
                const int t = t0 + wl;
                const u32 cnt = t < T ? a.table_cnt[t] : 0u;
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
            for (int t = threadIdx.x - 32; t <= T; t += THREADS - 32) { s_tb[t] = a.tb[t]; s_row[t] = (u32)a.row_off[t >> a.parts_log]; }
        }
    } else {
        for (int t = threadIdx.x; t <= T; t += THREADS) s_uoff[t] = (u32)a.uniq_off[t];
        if (threadIdx.x == 0) s_broken = 0u;
    }
    __syncthreads();
    if (a.by_table && blockIdx.x == 0)
        for (int t = threadIdx.x; t <= T >> a.parts_log; t += THREADS) a.uniq_off[t] = s_broken ? 0 : (int32_t)s_uoff[t << a.parts_log];
    if (s_broken || tile0 >= tile1) return;       // (warp-uniform; no block barrier below)

    // a one-index batch reads every upstream-gradient row once, a pooled one as often as the bag has indices
    const uint64_t keep = dq_policy_evict_last();
    const uint64_t pol = a.L <= a.G ? dq_policy_evict_first() : dq_policy_evict_normal();
    const vec_t *go = reinterpret_cast<const vec_t *>(a.grad_out) + (on ? cv : 0);
    vec_t v[2][C];                                // two batches in turn when the warp takes one row at a time
    // the rows of batch b of the present tile, all at once (row 0 for entries past the end, and a vector of the row for
    // lanes past its end: nothing is done with either)
    auto request = [&](int b, vec_t (&r)[C]) {
#pragma unroll
        for (int k = 0; k < C; ++k)
            r[k] = ld_row(go + (int64_t)__shfl_sync(0xffffffffu, vc, b * C + k) * dv, pol);       // (no condition: a branch per row would expose every shuffle)
    };
    // asks L2 for the rows of the tile whose indices have just arrived: a row per lane
    auto prefetch = [&]() {
        const int c0 = (int)col * 32 * VEC;
        const int bytes = (EXACT ? 32 * VEC : min(D - c0, 32 * VEC)) * (int)sizeof(float);
        if (I < 32 && wl >= I) return;
        const char *row = reinterpret_cast<const char *>(a.grad_out + (int64_t)((int64_t)vn < a.G ? vn : 0u) * D + c0);
#pragma unroll
        for (int b = 0; b < 32 * VEC * 4; b += 128)
            if (EXACT || b < bytes) dq_prefetch_l2(row + b);
        if (!EXACT) dq_prefetch_l2(row + bytes - 4);          // (rows that do not begin on a line's start)
    };
    take();
    request(0, v[0]);
    fetch(tile0 + 1);

    u32 first_range = 0, last_range = 0;          // of a run that is cut: in which ranges its pieces are
    auto find_pieces = [&](int t, int64_t at) {
        const u32 R = (u32)a.range_tiles * I;
        const u32 *start = a.seg_start + (a.by_table ? (int64_t)s_tb[t] + t + at : at);
        first_range = __ldg(start) / R;
        last_range = (__ldg(start + 1) - 1u) / R;
    };
    if (EARLY && cut) find_pieces(last_not_above(a.by_table ? s_tb : s_uoff, 0, T, a.by_table ? edge : cut_u), cut_u);
    const u32 cuts = EARLY ? __ballot_sync(0xffffffffu, cut) : 0u;
    const bool head0 = heads & 1u;
    int t_first = a.by_table ? last_not_above(s_tb, 0, T, tile0 * I) : last_not_above(s_uoff, 0, T, u_base);
    if (a.by_table) u_base += s_uoff[t_first];
    const u32 u_lead = u_base;                    // the run that enters the range, if one does
    u_base -= head0;                              // segment of entry e of the tile = u_base + heads in [0, e]
    bool open_lead = !head0;                      // no segment has begun in the range yet
    bool one_table = false;                       // everything that the present tile closes belongs to table t_first
    int t_max = t_first;
    float m = 0.f;                                // abs-max of the rows of table t_max that this thread has rounded
    auto push_max = [&]() {
        const u32 mb = __reduce_max_sync(0xffffffffu, __float_as_uint(m));
        if (wl == 0 && mb) atomicMax(a.absmax + (t_max >> a.parts_log), mb);
        m = 0.f;
    };
    // rounds a finished sum and writes it; leaves a piece of a cut run (called by all lanes of a group)
    auto store_row = [&](u32 u, const double (&acc)[VEC]) {
        float x = 0.f;
        if (on) st_row(reinterpret_cast<vec_t *>(a.grad_rows + (int64_t)u * D) + cv, rounded(acc, x), keep);  // quantise+update reads it next
        if (one_table) m = fmaxf(m, x);
        else note_max(a.absmax, s_uoff, t_first, T, a.parts_log, u, x);
    };
    auto store_piece = [&](int slot, const double (&acc)[VEC]) {
        if (on) {
            double *p = a.partials + ((size_t)range * 2 + slot) * D + cv * VEC;
#pragma unroll
            for (int q = 0; q < VEC; ++q) p[q] = acc[q];
        }
    };
    double acc[VEC];                              // the open run
#pragma unroll
    for (int q = 0; q < VEC; ++q) acc[q] = 0.0;

    for (u32 tile = tile0; tile < tile1; ++tile) {
        const int n = (int)min((int64_t)I, a.L - (int64_t)tile * I);
        const u32 n_heads = __popc(heads);
        // the table of the run that is open when the tile begins (of the first entry's when none is)
        const bool fresh = tile == tile0 && head0;
        while (t_first < T - 1 && u_base + fresh >= s_uoff[t_first + 1]) ++t_first;
        one_table = u_base + n_heads < s_uoff[t_first + 1];
        if (one_table && t_first != t_max) { push_max(); t_max = t_first; }
        if (a.by_table && first_col && wl < n && ((heads >> wl) & 1u)) {      // every entry that starts a segment names the segment's row
            const u32 u = u_base + __popc(heads & (0xffffffffu >> (31 - wl)));
            const int t = one_table ? t_first : last_not_above(s_uoff, t_first, T, u);
            a.unique_rows[u] = (int32_t)(kc - s_row[t]);
        }
        if (tile + 1 < tile1 && (!COLS || D < 768)) prefetch();
        u32 u = u_base;
        const u32 now = heads;
#pragma unroll
        for (int b = 0; b < NB; ++b) {
            if (b + 1 < NB) {
                request(b + 1, v[(b + 1) & 1]);
            } else if (tile + 1 < tile1) {
                take();
                request(0, v[0]);
                fetch(tile + 2);
            }
            const u32 bits = (now >> (b * C)) & ((1u << C) - 1u);
            if (bits == 0u && n >= (b + 1) * C) {             // inside a run
#pragma unroll
                for (int k = 0; k < C; ++k) add(acc, v[b & 1][k]);
            } else {
#pragma unroll
                for (int k = 0; k < C; ++k) {
                    if ((bits >> k) & 1u) {                   // (warp-uniform)
                        if (open_lead) { store_piece(0, acc); open_lead = false; }
                        else if (!(fresh && b * C + k == 0)) store_row(u, acc);
                        ++u;
#pragma unroll
                        for (int q = 0; q < VEC; ++q) acc[q] = 0.0;
                    }
                    if (b * C + k < n) add(acc, v[b & 1][k]);
                }
            }
        }
        u_base = u;
    }
    // ---- the run that is open at the end of the range
    const int64_t i1 = min((int64_t)tile1 * I, a.L);
    const bool ends = EARLY ? !(cuts & 2u) : i1 == a.L || __ldg(a.keys + i1) != __ldg(a.keys + i1 - 1);
    const bool cut_lead = !head0, cut_trail = !open_lead && !ends;
    if (open_lead || cut_trail) store_piece(open_lead ? 0 : 1, acc);
    else store_row(u_base, acc);
    __syncwarp();
    push_max();

    // ---- the warp that brings a cut run's last piece adds the pieces
    if (!(cut_lead || cut_trail)) return;
    const u32 group = range / FOLD_GROUP;
    u32 last = 0, groups = 0;                     // pieces to add here; the run's groups, when it has many pieces
    if (wl == 0 ? cut_lead : (wl == 1 && cut_trail)) {
        if (!EARLY) {
            const u32 u = wl == 0 ? u_lead : u_base;
            const int t = last_not_above(s_uoff, 0, T, u);
            find_pieces(t, a.by_table ? u - s_uoff[t] : u);
        }
        const u32 g0 = first_range / FOLD_GROUP;
        u32 pieces = last_range - first_range + 1;
        u32 *arrived = &a.range_done[first_range].x;
        if (pieces > FOLD_GROUP) {
            groups = last_range / FOLD_GROUP - g0 + 1;
            pieces = min(last_range, group * FOLD_GROUP + FOLD_GROUP - 1) - max(first_range, group * FOLD_GROUP) + 1;
            arrived = &a.range_done[2 * group + (group == g0 ? 1 : 0)].y;
        }
        last = arrive(arrived) == pieces * cols - 1u ? pieces : 0u;
    }
    __syncwarp();
    // adds np partials of D features each (`at(p)` = where piece p lies), this lane's features of columns cc
    auto fold = [&](int np, int cc, double (&sum)[VEC], auto at) {
#pragma unroll
        for (int x = 0; x < VEC; ++x) sum[x] = 0.0;
        for (int p0 = 0; (EXACT || cc < dv) && p0 < np; p0 += 8) {
            double x[8][VEC];
#pragma unroll
            for (int j = 0; j < 8; ++j) {
                const int p = p0 + j;
                const double *src = at(min(p, np - 1)) + cc * VEC;
#pragma unroll
                for (int q = 0; q < VEC; ++q) x[j][q] = p < np ? __ldcg(src + q) : 0.0;
            }
#pragma unroll
            for (int j = 0; j < 8; ++j)
#pragma unroll
                for (int q = 0; q < VEC; ++q) sum[q] += x[j][q];
        }
    };
    auto store_total = [&](u32 u, int cc, const double (&sum)[VEC]) {
        float x = 0.f;
        if (EXACT || cc < dv) st_row(reinterpret_cast<vec_t *>(a.grad_rows + (int64_t)u * D) + cc, rounded(sum, x), keep);
        note_max(a.absmax, s_uoff, 0, T, a.parts_log, u, x);
    };
#pragma unroll 1
    for (int q = 0; q < 2; ++q) {                 // (columns: all of them, the blocks of the others are done too)
        const int np = (int)__shfl_sync(0xffffffffu, last, q);
        if (np == 0) continue;
        const u32 u = q ? u_base : u_lead, f = __shfl_sync(0xffffffffu, first_range, q);
        const u32 ng = __shfl_sync(0xffffffffu, groups, q), g0 = f / FOLD_GROUP;
        const u32 p_first = ng ? max(f, group * FOLD_GROUP) : f;
        for (int cc = wl; cc - wl < (COLS ? dv : 1); cc += 32) {
            double sum[VEC];
            fold(np, cc, sum, [&](int p) { return a.partials + ((size_t)(p_first + p) * 2 + (p_first + p == f ? 1 : 0)) * D; });
            if (ng == 0) {
                store_total(u, cc, sum);
            } else if (EXACT || cc < dv) {
#pragma unroll
                for (int x = 0; x < VEC; ++x) a.group_partials[((size_t)group * 2 + (group == g0 ? 1 : 0)) * D + cc * VEC + x] = sum[x];
            }
        }
        if (ng) {
            __syncwarp();
            bool final = false;
            if (wl == 0) final = arrive(&a.range_done[f].x) == ng - 1u;
            __syncwarp();                         // (what lane 0 has acquired, the warp loads)
            if (!__shfl_sync(0xffffffffu, final, 0)) continue;
            for (int cc = wl; cc - wl < (COLS ? dv : 1); cc += 32) {
                double sum[VEC];
                fold((int)ng, cc, sum, [&](int p) { return a.group_partials + ((size_t)(g0 + p) * 2 + (p == 0 ? 1 : 0)) * D; });
                store_total(u, cc, sum);
            }
        }
    }
}

}  // namespace segred

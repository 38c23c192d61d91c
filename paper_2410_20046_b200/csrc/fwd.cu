// Forward of the quantisation-aware embedding lookup (paper Section 3.1, Figure 2(b)):
// gather the rows a batch uses from the FP32 master table, fake-quantise each gathered
// row with the table's stored scale, and sum-pool over the bag.  No low-precision copy
// of the table exists; only the gathered rows are ever quantised.
//
// HBM-bound random row gather.  Measured on B200, a bare gather of this access pattern
// runs fastest with many resident warps and only two to four independent 128-bit loads
// per lane, so the kernels are kept lean (46 to 64 registers, a few of the one-index
// kernel's values spilled for its fifth block) rather than deeply unrolled.  A block works for one table, which makes scale, bit width and row base block
// constants.  A group of LPR lanes owns one row: a feature-16 row is one 64-byte request
// of four lanes, a feature-64 row one 256-byte request of sixteen.
//   * fwd_onehot_kernel (launched when L == T*B and no codes are asked for, the Criteo-shaped
//     training case): a warp owns 32 consecutive bags, does their bookkeeping one bag per
//     lane, then fetches the rows 32/LPR per step with NB steps in flight; the pooled value
//     is the fake-quantised row itself.  A bag that turns out not to hold exactly one index
//     is pooled by a plain loop.
//   * fwd_bags_kernel (any other batch): a lane group walks one bag at a time, NB of its
//     rows per batch, and sums them in bag order in FP64, rounded once, so the result
//     does not depend on the launch shape.
//   * fwd_long_bags_kernel: the same for long bags of rows of 36 to 64 features, a warp a bag.
#include <algorithm>
#include <type_traits>
#include "common.cuh"

namespace {

constexpr int FW_THREADS = 256;
// independent rows in flight per lane group.  Measured on B200: four for rows of up to 128
// bytes, two for 256- and 512-byte rows (more resident warps beat deeper unrolling), one
// when a lane already holds several 128-bit pieces of every row
template <int LPR, int CH>
struct NBOf { static constexpr int v = CH >= 2 ? 1 : 4; };

struct FwdArgs {
    const float *tables;
    const int64_t *row_off;
    const int32_t *indices;
    const int32_t *offsets;
    const float *scales;
    const int32_t *bits;
    float *out;
    int8_t *codes_out;
    int T, D, B;
    int64_t L;
    int *status;
    int per_warp;                // one-index batches: bags of a warp, up to 32 (before the launch: the fewest that it may take)
    int let_next;                // the kernel behind this one may begin (it waits itself where it has to)
};

// Waits for the kernels before this one and only then lets the next one begin.  The order is what the one-launch step
// (small_step.cuh) stands on: it reads the batch and writes the workspace, unique_rows and grad_rows before its own wait, so
// everything before this kernel must be over by then.  The other way round it would race with all of that.
__device__ __forceinline__ void before_and_next(const FwdArgs &a)
{
    dq_wait_before();
    if (a.let_next) dq_let_next();
}

__device__ __forceinline__ void store_codes(int8_t *codes_out, int64_t j, int D, int c4, const float4 &c)
{
    char4 cc = make_char4((signed char)(int)c.x, (signed char)(int)c.y, (signed char)(int)c.z, (signed char)(int)c.w);
    *reinterpret_cast<char4 *>(codes_out + j * D + 4 * c4) = cc;
}

// clamps an index into [0, nrows) and remembers that it had to
__device__ __forceinline__ int32_t clamp_index(int32_t idx, int32_t nrows, bool &bad)
{
    bad |= (idx < 0) | (idx >= nrows);
    return min(max(idx, 0), nrows - 1);
}

// Per-table constants of a block
struct TableCtx {
    QuantScale qs;
    const float *tbl;
    int32_t nrows;
    int64_t g0;
};

__device__ __forceinline__ TableCtx table_ctx(const FwdArgs &a, int t, int D)
{
    TableCtx c;
    c.qs = dq_make_scale(__ldg(a.scales + t), __ldg(a.bits + t));
    const int64_t r0 = __ldg(a.row_off + t);
    c.nrows = (int32_t)(__ldg(a.row_off + t + 1) - r0);
    c.tbl = a.tables + r0 * D;
    c.g0 = (int64_t)t * a.B;
    return c;
}

// plain pooling of one bag (one row at a time): used for the rare bags of a one-index batch
template <int LPR, int CH>
__device__ __forceinline__ void pool_bag_plain(const FwdArgs &a, const TableCtx &tc, int D, int d4, int32_t lo,
                                               int32_t hi, float *out_row, int lane, bool &bad)
{
    if (lo < 0 || hi < lo || (int64_t)hi > a.L) { bad = true; hi = lo = 0; }
#pragma unroll 1
    for (int c = 0; c < CH; ++c) {
        const int c4 = c * LPR + lane;
        if (c4 >= d4) continue;
        double a0 = 0, a1 = 0, a2 = 0, a3 = 0;
#pragma unroll 1
        for (int32_t j = lo; j < hi; ++j) {
            const int32_t idx = clamp_index(__ldg(a.indices + j), tc.nrows, bad);
            float4 cd, f;
            dq_fq4(__ldg(reinterpret_cast<const float4 *>(tc.tbl + (int64_t)idx * D) + c4), tc.qs, cd, f);
            a0 += (double)f.x; a1 += (double)f.y; a2 += (double)f.z; a3 += (double)f.w;
            if (a.codes_out) store_codes(a.codes_out, j, D, c4, cd);
        }
        reinterpret_cast<float4 *>(out_row)[c4] = make_float4((float)a0, (float)a1, (float)a2, (float)a3);
    }
}

// A warp takes 32 consecutive bags of its table.  The bookkeeping of a bag (its offsets, its index,
// the range checks) is done once, by the one lane that owns the bag; the rows are then fetched
// 32/LPR at a time by all lanes, each step reading its bag's index from the owner lane by shuffle.
// Measured on B200 the kernel is bound by instruction issue, not by HBM, at 256-byte rows, which
// is why the per-bag work is kept off the per-row path.
//
// FEW: a warp takes a.per_warp bags instead of 32 (launch2).  An instance of its own: as a value at run time the number of bags cost the
// others registers, and values were spilled (200 K rows of 800 bytes 65.2 -> 69.4 us, 65 K 17.6 -> 19.7, 426 K of 80 15.1 -> 15.4).
template <int LPR, int CH, bool EXACT, bool FEW>
__global__ void __launch_bounds__(FW_THREADS, 5)
fwd_onehot_kernel(const FwdArgs a)
{
    before_and_next(a);
    constexpr int NB = NBOf<LPR, CH>::v;      // row steps in flight
    constexpr int RPW = 32 / LPR;             // rows one warp instruction covers
    constexpr int WPB = FW_THREADS / 32;
    const int D = EXACT ? 4 * LPR * CH : a.D;
    const int d4 = D >> 2;
    const int t = blockIdx.x;
    const int wlane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int lane = wlane % LPR, grp = wlane / LPR;
    const int64_t g0 = (int64_t)t * a.B;
    const int per = FEW ? a.per_warp : 32;
    const unsigned all = 0xffffffffu >> (32 - per);
    // a bag's offsets and its index, the right one when the offsets are the identity (L == T*B): on their way before the
    // table's constants are waited for (426 K rows of 64 bytes 8.9 -> 8.4 us, 852 K packed ones of 32 40.6 -> 39.5; not where the
    // rows take the whole warp, which would spill more: 65 K of 512 bytes 12.8, 13.0)
    int32_t lo = 0, hi = 0, idx = 0;
    auto load = [&](int i) {
        if (i < a.B && wlane < per) {
            lo = __ldg(a.offsets + g0 + i);
            hi = __ldg(a.offsets + g0 + i + 1);
            idx = __ldg(a.indices + g0 + i);
        }
    };
    const int stride = gridDim.y * (WPB * per);
    const int start = (blockIdx.y * WPB + warp) * per;
    if (LPR < 32) load(start + wlane);
    const TableCtx tc = table_ctx(a, t, D);
    const float4 *tbl_lane = reinterpret_cast<const float4 *>(tc.tbl) + lane;
    const int TD4 = a.T * d4;                 // 128-bit vectors between the output rows of bags i and i+1
    bool bad = false;
    const uint64_t keep = dq_policy_evict_last();

    for (int i0 = start; i0 < a.B; i0 += stride) {
        if (LPR == 32 || i0 != start) load(i0 + wlane);
        // ---- lane-per-bag bookkeeping
        const int i = i0 + wlane;
        const bool mine = i < a.B && wlane < per;
        bool single = false;
        if (mine) {
            single = (hi - lo == 1) & (lo >= 0) & ((int64_t)hi <= a.L);
            if (single) {
                if ((int64_t)lo != tc.g0 + i) idx = __ldg(a.indices + lo);
                idx = clamp_index(idx, tc.nrows, bad);
            }
        }
        const unsigned one = __ballot_sync(0xffffffffu, single);
        unsigned rare = __ballot_sync(0xffffffffu, mine && !single);
        float4 *out_lane = reinterpret_cast<float4 *>(a.out) + ((int64_t)i0 * a.T + t) * d4 + lane;

        // ---- rows, RPW per step, NB steps in flight
        // (nearly always: no checks; but rows of more than 1 KB whose last lanes stand idle are better without their loads: 65 K
        // of 2064 bytes 112 us, 120 with)
        if ((EXACT || CH <= 2) && one == all) {
#pragma unroll 1
            for (int k0 = 0; k0 < per; k0 += RPW * NB) {
                int32_t ib[NB];
#pragma unroll
                for (int b = 0; b < NB; ++b) ib[b] = __shfl_sync(0xffffffffu, idx, (k0 + b * RPW + grp) & 31);
#pragma unroll
                for (int c = 0; c < CH; ++c) {
                    const bool on = EXACT || c * LPR + lane < d4;
                    float4 v[NB];
#pragma unroll
                    for (int b = 0; b < NB; ++b)           // the update reads the row again
                        v[b] = dq_ld_nc(tbl_lane + (int64_t)ib[b] * d4 + (on ? c * LPR : -lane), keep);
#pragma unroll
                    for (int b = 0; b < NB; ++b) {
                        const int bag = k0 + b * RPW + grp;
                        float4 cd, f;
                        dq_fq4(v[b], tc.qs, cd, f);
                        if (on && (RPW * NB <= 32 || bag < 32))
                            __stcs(out_lane + (int64_t)bag * TD4 + c * LPR, f);     // written once, read by nobody here
                    }
                }
            }
            continue;
        }
#pragma unroll 1
        for (int k0 = 0; k0 < per; k0 += RPW * NB) {
            if ((one >> k0) == 0u) break;
            int32_t ib[NB];
#pragma unroll
            for (int b = 0; b < NB; ++b) ib[b] = __shfl_sync(0xffffffffu, idx, (k0 + b * RPW + grp) & 31);
#pragma unroll
            for (int c = 0; c < CH; ++c) {
                const int c4 = c * LPR + lane;
                float4 v[NB];
#pragma unroll
                for (int b = 0; b < NB; ++b) {
                    const int bag = k0 + b * RPW + grp;
                    if (bag < 32 && ((one >> bag) & 1u) && (EXACT || c4 < d4))
                        v[b] = dq_ld_nc(tbl_lane + (int64_t)ib[b] * d4 + c * LPR, keep);   // the update reads the row again
                }
#pragma unroll
                for (int b = 0; b < NB; ++b) {
                    const int bag = k0 + b * RPW + grp;
                    if (bag < 32 && ((one >> bag) & 1u) && (EXACT || c4 < d4)) {
                        float4 cd, f;
                        dq_fq4(v[b], tc.qs, cd, f);
                        __stcs(out_lane + (int64_t)bag * TD4 + c * LPR, f);   // written once, read by nobody here
                    }
                }
            }
        }
        // ---- bags that do not hold exactly one index: pooled by the first lane group, one at a time
        while (rare) {
            const int bag = __ffs(rare) - 1;
            rare &= rare - 1;
            const int ii = i0 + bag;
            if (grp == 0) {
                const int32_t l = __ldg(a.offsets + tc.g0 + ii), h = __ldg(a.offsets + tc.g0 + ii + 1);
                pool_bag_plain<LPR, CH>(a, tc, D, d4, l, h, a.out + ((int64_t)ii * a.T + t) * D, lane, bad);
            }
        }
    }
    if (bad) dq_report(a.status, DQRM_ERR_INDEX_RANGE);
}

// Resident blocks asked for.  The gather wants warps more than registers: left to itself the compiler takes 76 and up, and
// 426 K rows of 256 bytes, two a bag, take 70 us with three blocks and 54 with four; 65 K rows of 1 KB 33 with four and 28
// with five; of 2 KB, which then spill nothing either, 72 us without a bound and 56 with four
__host__ __device__ constexpr int bags_blocks(int CH) { return CH == 2 ? 5 : CH == 8 ? 1 : 4; }

// A lane group walks one bag at a time, its rows NB at a time in bag order.  Every lane loads the bag's indices itself:
// loaded one per lane and handed round by shuffle they cost a round trip more per bag, and lane groups whose bags differ
// in length wait for one another on the way (measured on
// B200, random rows of 26 tables: 640 K rows of 64 bytes in bags of three on average 29 us this way, 42 by shuffle; of 256
// bytes 67 and 88).
// MIXED: the grid is (tables, blocks of a table), else (blocks of a table, tables)
template <int LPR, int CH, bool EXACT, bool CODES, bool MIXED>
__global__ void __launch_bounds__(FW_THREADS, bags_blocks(CH))
fwd_bags_kernel(const FwdArgs a)
{
    before_and_next(a);
    constexpr int NB = NBOf<LPR, CH>::v;
    constexpr int GPB = FW_THREADS / LPR;
    const int D = EXACT ? 4 * LPR * CH : a.D;
    const int d4 = D >> 2;
    const int t = MIXED ? blockIdx.x : blockIdx.y;
    const int lane = threadIdx.x % LPR;
    const int grp = threadIdx.x / LPR;
    const TableCtx tc = table_ctx(a, t, D);
    bool bad = false;

    for (int i = (MIXED ? blockIdx.y : blockIdx.x) * GPB + grp; i < a.B; i += (MIXED ? gridDim.y : gridDim.x) * GPB) {
        int32_t lo = __ldg(a.offsets + tc.g0 + i), hi = __ldg(a.offsets + tc.g0 + i + 1);
        if (lo < 0 || hi < lo || (int64_t)hi > a.L) { bad = true; hi = lo = 0; }
        double acc[CH][4];
#pragma unroll
        for (int c = 0; c < CH; ++c) acc[c][0] = acc[c][1] = acc[c][2] = acc[c][3] = 0.0;
        for (int32_t j0 = lo; j0 < hi; j0 += NB) {
            int32_t idx[NB];
#pragma unroll
            for (int b = 0; b < NB; ++b) idx[b] = (j0 + b < hi) ? clamp_index(__ldg(a.indices + j0 + b), tc.nrows, bad) : 0;
#pragma unroll
            for (int c = 0; c < CH; ++c) {
                const int c4 = c * LPR + lane;
                float4 v[NB];
#pragma unroll
                for (int b = 0; b < NB; ++b)
                    if (j0 + b < hi && (EXACT || c4 < d4))
                        v[b] = __ldg(reinterpret_cast<const float4 *>(tc.tbl + (int64_t)idx[b] * D) + c4);
#pragma unroll
                for (int b = 0; b < NB; ++b) {
                    if (j0 + b < hi && (EXACT || c4 < d4)) {
                        const float x[4] = {v[b].x, v[b].y, v[b].z, v[b].w};
                        float f[4];
                        if constexpr (CODES)
                            *reinterpret_cast<u32 *>(a.codes_out + (int64_t)(j0 + b) * D + 4 * c4) = dq_fq4_bytes(x, tc.qs, f);
                        else
                            dq_fq_many<4>(x, tc.qs, f);
#pragma unroll
                        for (int q = 0; q < 4; ++q) acc[c][q] += (double)f[q];
                    }
                }
            }
        }
        float4 *o = reinterpret_cast<float4 *>(a.out + ((int64_t)i * a.T + t) * D);
#pragma unroll
        for (int c = 0; c < CH; ++c) {
            const int c4 = c * LPR + lane;
            if (EXACT || c4 < d4)
                o[c4] = make_float4((float)acc[c][0], (float)acc[c][1], (float)acc[c][2], (float)acc[c][3]);
        }
    }
    if (bad) dq_report(a.status, DQRM_ERR_INDEX_RANGE);
}

// Long bags of rows of 36 to 64 features: a warp per bag, two features a lane.  Every lane of a warp is then in the same
// bag, so the indices are loaded 32 at a time, one per lane, and checked once; the rows are fetched eight at a time, their
// numbers handed round by shuffle, and summed in bag order (measured
// on B200, 26 x 16384 bags of 20 on average, Zipf 1.2: 316 us, 351 with four rows at a time and 352 by lane groups).
template <bool EXACT>
__global__ void __launch_bounds__(FW_THREADS, 4)
fwd_long_bags_kernel(const FwdArgs a)
{
    before_and_next(a);
    constexpr int WPB = FW_THREADS / 32;
    const int D = EXACT ? 64 : a.D;
    const int t = blockIdx.y, lane = threadIdx.x & 31;
    const bool on = EXACT || 2 * lane < D;
    const TableCtx tc = table_ctx(a, t, D);
    const float2 *tbl = reinterpret_cast<const float2 *>(tc.tbl) + (on ? lane : 0);
    bool bad = false;

    for (int i = blockIdx.x * WPB + (threadIdx.x >> 5); i < a.B; i += gridDim.x * WPB) {
        int32_t lo = __ldg(a.offsets + tc.g0 + i), hi = __ldg(a.offsets + tc.g0 + i + 1);
        if (lo < 0 || hi < lo || (int64_t)hi > a.L) { bad = true; hi = lo = 0; }
        double acc[2] = {0.0, 0.0};
        int32_t mine = lo + lane < hi ? __ldg(a.indices + lo + lane) : 0;
        for (int32_t j0 = lo; j0 < hi; j0 += 32) {
            const int32_t row = clamp_index(mine, tc.nrows, bad);      // (lanes past the bag's end hold row 0)
            mine = j0 + 32 + lane < hi ? __ldg(a.indices + j0 + 32 + lane) : 0;
            const int cnt = min(32, hi - j0);
            // rows b0 .. b0 + NB, of which `n` count
            auto rows = [&](int b0, int n, auto nb_tag) {
                constexpr int NB = decltype(nb_tag)::value;
                float x[2 * NB], f[2 * NB];
#pragma unroll
                for (int b = 0; b < NB; ++b) {
                    const int32_t r = __shfl_sync(0xffffffffu, row, (b0 + b) & 31);
                    const float2 v = __ldg(tbl + (int64_t)r * (D / 2));
                    x[2 * b] = v.x;
                    x[2 * b + 1] = v.y;
                }
                dq_fq_many<2 * NB>(x, tc.qs, f);
#pragma unroll
                for (int b = 0; b < NB; ++b)
                    if (b < n) {
                        acc[0] += (double)f[2 * b];
                        acc[1] += (double)f[2 * b + 1];
                    }
            };
            int b0 = 0;
            for (; b0 + 8 <= cnt; b0 += 8) rows(b0, 8, std::integral_constant<int, 8>{});
            for (; b0 < cnt; b0 += 4) rows(b0, cnt - b0, std::integral_constant<int, 4>{});
        }
        if (on) reinterpret_cast<float2 *>(a.out + ((int64_t)i * a.T + t) * D)[lane] = make_float2((float)acc[0], (float)acc[1]);
    }
    if (bad) dq_report(a.status, DQRM_ERR_INDEX_RANGE);
}

// From 18 indices a bag on average: at 16 of equal length, where no lane group waits for another, the two are even in large
// batches (26 x 8192 bags of 256-byte rows 159 us both) and lane groups ahead in small ones (4 x 2048 bags 9.2 against 10.3
// us); at 24 it is 212 against 223 us, and with bags of uneven length the warps are ahead from 12 on
constexpr int LONG_BAG = 18;
inline bool long_bags(const int8_t *codes_out, int T, int B, int64_t L) { return !codes_out && L >= LONG_BAG * (int64_t)T * B; }
inline bool warp_per_bag(const FwdArgs &a, int lpr) { return lpr == 16 && long_bags(a.codes_out, a.T, a.B, a.L); }

// Warps an SM below which a one-index batch's warps take fewer bags, down to one step of their rows: a warp's steps are a chain, and a
// small batch has too few warps to hide it.  Measured on B200 (us; 32 bags a warp / so many that there are twelve warps an SM
// at least): 26 tables of 2048 bags of 64 features (11 warps an SM) 5.25 / 4.45, one of 5000 of 128 6.51 / 2.82, four of 9000 of 32
// 3.35 / 2.94.  Not in a step that runs it beside a sort, which needs the room: five tables of 10,000 bags of 128 features in one call
// 40.8, 42.6 with fewer bags a warp, eight pipelined steps of three of 8000 of 64 206 and 210; but in a step that keeps to one stream
// (eight steps of five of 10,000 of 128 274 / 262) and in the host-fed one (train_step_host).  The line was drawn while steps were
// under the rule, too; a forward alone gains beyond it (one table of 65,536 of 128, 14 warps an SM, 12.6 / 10.6)
constexpr int FEW_WARPS = 12;
constexpr int MIXED_TABLES = 8;
// Order of the blocks.  All tables' blocks for the same bags side by side: the pooled rows of a bag lie next to one another in the
// output, and DRAM takes them better together (one index a bag, 852 K rows of 256 bytes 49.0 -> 46.9 us, 426 K of 64 bytes 9.1 -> 8.9).
// Table by table: the rows that a bag shares with others are found again in L2, or a warp's in L1.  Which of the two counts for
// more goes by the width of the rows and the length of the bags.  Measured on B200 for pooled bags, 26 tables of 8192 bags, side by
// side / table by table (uniform indices over 30 K to 1.5 M rows a table, and Zipf 1.2): 4 to 16 features 0.97 to 1.02 for bags of
// two, 1.0 to 1.14 for twelve, 1.0 to 1.51 for thirty; 32 features 0.96 to 0.98 up to eight indices a bag, 0.96 to 1.00 for twelve, 1.03
// for 17 where every row comes several times; 64 features 0.94 to 0.98 for two to four, 0.97 to 1.02 for six, 1.08 for twelve; 128
// features 0.94 to 0.97 for two, 0.98 to 1.03 for four, up to 1.08 for six; 256 features 0.99 and 1.07 for two, 1.18 for twelve.  Five
// tables: 0.99 to 1.02.  Long bags, a warp each: 8.5 M rows of 256 bytes 324 us side by side, 314 table by table
__host__ __device__ constexpr int mixed_upto(int LPR, int CH) { return CH > 1 ? 0 : LPR == 8 ? 16 : LPR == 16 ? 5 : LPR == 32 ? 3 : 0; }
template <int LPR, int CH>
inline bool bags_mixed(const FwdArgs &a) { return a.T >= MIXED_TABLES && a.L < mixed_upto(LPR, CH) * (int64_t)a.T * a.B; }

template <int LPR, int CH, bool EXACT>
cudaError_t launch_bags(const FwdArgs &a, dim3 grid, cudaStream_t st)
{
    if (LPR == 16 && warp_per_bag(a, LPR)) return dq_launch(fwd_long_bags_kernel<EXACT>, grid, dim3(FW_THREADS), 0, st, a);
    constexpr bool MAY = mixed_upto(LPR, CH) > 0;
    if (MAY && bags_mixed<LPR, CH>(a)) {
        if (a.codes_out) return dq_launch(fwd_bags_kernel<LPR, CH, EXACT, true, MAY>, grid, dim3(FW_THREADS), 0, st, a);
        return dq_launch(fwd_bags_kernel<LPR, CH, EXACT, false, MAY>, grid, dim3(FW_THREADS), 0, st, a);
    }
    if (a.codes_out) return dq_launch(fwd_bags_kernel<LPR, CH, EXACT, true, false>, grid, dim3(FW_THREADS), 0, st, a);
    return dq_launch(fwd_bags_kernel<LPR, CH, EXACT, false, false>, grid, dim3(FW_THREADS), 0, st, a);
}

template <int LPR, int CH, bool EXACT>
int launch2(dqrm_ctx *ctx, FwdArgs a, cudaStream_t st)
{
    constexpr int GPB = FW_THREADS / LPR;
    // the one-index kernel does not emit codes; a caller that asks for them gets the general kernel
    const bool onehot = a.L == (int64_t)a.T * a.B && a.codes_out == nullptr;
    const int fewest = std::max(a.per_warp, 32 / LPR * NBOf<LPR, CH>::v);
    a.per_warp = 32;
    if (onehot) {
        while (a.per_warp / 2 >= fewest && (int64_t)a.T * ((a.B + a.per_warp - 1) / a.per_warp) < (int64_t)ctx->num_sms * FEW_WARPS) a.per_warp /= 2;
    }
    const int per_block = onehot ? FW_THREADS / 32 * a.per_warp : warp_per_bag(a, LPR) ? GPB / 2 : GPB;
    int bx = (a.B + per_block - 1) / per_block;
    const int cap = (ctx->num_sms * 32 + ctx->T - 1) / ctx->T;     // a few waves over all tables
    if (bx > cap) bx = cap;
    if (bx < 1) bx = 1;
    const bool mixed = onehot || bags_mixed<LPR, CH>(a);
    const dim3 grid((unsigned)(mixed ? ctx->T : bx), (unsigned)(mixed ? bx : ctx->T));
    constexpr bool MAY = 32 / LPR * NBOf<LPR, CH>::v < 32;
    DQRM_CUDA_TRY(ctx, (!onehot                 ? launch_bags<LPR, CH, EXACT>(a, grid, st)
                        : MAY && a.per_warp < 32 ? dq_launch(fwd_onehot_kernel<LPR, CH, EXACT, MAY>, grid, dim3(FW_THREADS), 0, st, a)
                                                 : dq_launch(fwd_onehot_kernel<LPR, CH, EXACT, false>, grid, dim3(FW_THREADS), 0, st, a)));
    dq_mark(ctx, st, DQ_K_FWD);
    return DQRM_OK;
}

template <int LPR, int CH>
int launch(dqrm_ctx *ctx, const FwdArgs &a, cudaStream_t st)
{
    if (a.D == 4 * LPR * CH) return launch2<LPR, CH, true>(ctx, a, st);
    return launch2<LPR, CH, false>(ctx, a, st);
}

}  // namespace

size_t dq_fwd_align(const dqrm_ctx *ctx, const int8_t *codes_out, int B, int64_t L)
{
    return ctx->D > 32 && ctx->D <= 64 && long_bags(codes_out, ctx->T, B, L) ? sizeof(float2) : sizeof(float4);
}

int dq_launch_fwd(dqrm_ctx *ctx, const float *tables, const int32_t *indices, const int32_t *offsets,
                  const float *scales, const int32_t *bits, float *out, int8_t *codes_out,
                  int B, int64_t L, cudaStream_t st, bool let_next, bool beside)
{
    FwdArgs a{tables, ctx->d_row_off, indices, offsets, scales, bits, out, codes_out, ctx->T, ctx->D, B, L,
              ctx->d_status, beside ? 32 : 1, let_next ? 1 : 0};
    const int d4 = ctx->D / 4;
    if (d4 <= 1) return launch<1, 1>(ctx, a, st);
    if (d4 <= 2) return launch<2, 1>(ctx, a, st);
    if (d4 <= 4) return launch<4, 1>(ctx, a, st);
    if (d4 <= 8) return launch<8, 1>(ctx, a, st);
    if (d4 <= 16) return launch<16, 1>(ctx, a, st);
    if (d4 <= 32) return launch<32, 1>(ctx, a, st);
    if (d4 <= 64) return launch<32, 2>(ctx, a, st);
    if (d4 <= 128) return launch<32, 4>(ctx, a, st);
    return launch<32, 8>(ctx, a, st);
}

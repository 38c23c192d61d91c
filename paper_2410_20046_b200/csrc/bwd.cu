// Backward of the embedding lookup (paper Section 4.3 and Appendix B.1): the gradient of
// an embedding table is a sparse (indices, values) tensor over the rows the batch
// touched; lookups that hit the same row are coalesced.  Sum pooling and the
// straight-through quantiser hand every lookup its bag's upstream gradient unchanged.
//
// Pipeline (all on one stream; no block waits for another outside its cluster):
//   sort         one block per table (small_sort.cuh), one cluster of blocks per table
//                (cluster_sort.cuh), or a radix sort of all tables at once (radix_sort.cuh); the
//                first two can also number the segments
//   seg_count / seg_emit  head flags of the sorted keys -> unique_rows, uniq_off,
//                         segment starts, first segment of every tile of the sum
//   seg_sum      every warp walks a range of the sorted order: gathers the upstream gradient rows,
//                sums runs in FP64, rounds and writes them; of a run that spans ranges every
//                range leaves an FP64 partial and the last to arrive adds them
// The sort is stable and every sum has a fixed shape, so results are reproducible bit
// for bit.  The per-table abs-max of the summed gradient (needed by the INT8 gradient
// quantiser) is folded into the last kernel.
#include <algorithm>
#include "common.cuh"
#include "seg_reduce.cuh"
#include "seg_groups.cuh"
#include "cluster_sort.cuh"
#include "radix_sort.cuh"
#include "small_sort.cuh"
#include "small_step.cuh"

namespace {

constexpr int ST_THREADS = 256;
constexpr int ST_ITEMS = 8;
constexpr int ST_TILE = ST_THREADS * ST_ITEMS;   // 2048 entries per tile
constexpr int ST_WARPS = ST_THREADS / 32;

struct Layout {
    int passes, digit_bits;                    // radix sort: digits of the row number within a table
    int64_t radix_tiles, num_tiles;
    // the summing kernel: log2 of the entries between two of chunk_first; rows of more than 48 features: entries of a tile, tiles, tiles of
    // a warp's range; narrower ones: entries of a lane group's range, ranges of warps
    int sum_shift, sum_tile;
    int64_t sum_tiles, sum_ranges;
    int range_tiles, sum_span;
    size_t absmax, tile_heads, tile0, tile_table, totals, tilehist;
    size_t keys_a, vals_a, pairs_a, pairs_b, seg_start, chunk_first, tile_done, partials, group_partials, table_cnt, tb;
    size_t total;
};

// bags: of the batch, which how it is summed depends on, but not where the parts lie
Layout make_layout(const dqrm_ctx *ctx, int64_t L, int64_t bags = 0)
{
    Layout y;
    y.passes = (ctx->row_bits + rsort::MAX_DIGIT_BITS - 1) / rsort::MAX_DIGIT_BITS;
    y.digit_bits = (ctx->row_bits + y.passes - 1) / y.passes;
    if (y.digit_bits < 2) y.digit_bits = 2;        // (the scatter takes four digits a thread)
    int64_t Lc = L < 1 ? 1 : L;
    y.num_tiles = (Lc + ST_TILE - 1) / ST_TILE;
    y.radix_tiles = rsort::max_tiles(ctx->T, Lc);
    // the sum: every warp that the GPU holds at once walks one range (long batches: segred::range_tiles)
    int64_t warps = segred::takes_groups(ctx->D) ? (int64_t)ctx->num_sms * segred::GROUPS_BLOCKS * segred::GROUPS_THREADS / 32
                                                 : (int64_t)ctx->num_sms * segred::sum_blocks(ctx->D, Lc, ctx->num_sms) /
                                                       segred::column_blocks(ctx->D) * segred::WARPS;
    if (warps < 1) warps = 1;
    y.sum_tile = segred::tile_entries(ctx->D, Lc, ctx->num_sms, bags);
    y.sum_shift = segred::takes_groups(ctx->D) ? segred::CHUNK_SHIFT : segred::log2_of(y.sum_tile);
    y.sum_tiles = (Lc + y.sum_tile - 1) / y.sum_tile;
    y.range_tiles = segred::range_tiles(ctx->D, y.sum_tiles, warps, y.sum_tile);
    const int64_t groups = 32 / segred::lanes_per_row(ctx->D), chunk = (int64_t)1 << segred::CHUNK_SHIFT;
    y.sum_span = (int)(((Lc + warps * groups - 1) / (warps * groups) + chunk - 1) / chunk * chunk);
    y.sum_ranges = (Lc + y.sum_span * groups - 1) / (y.sum_span * groups);
    size_t o = 0;
    auto take = [&](size_t bytes) { size_t at = o; o = align_up(o + bytes, 256); return at; };
    y.absmax = take(sizeof(u32) * ctx->T);
    y.tile_heads = take(sizeof(u32) * y.num_tiles);
    y.tile0 = take(sizeof(u32) * (ctx->T + 1));
    y.tile_table = take(sizeof(u32) * y.radix_tiles);
    y.totals = take((sizeof(u32) * ctx->T) << y.digit_bits);
    y.tilehist = take((sizeof(u32) * y.radix_tiles) << y.digit_bits);
    y.keys_a = take(sizeof(u32) * Lc);
    y.vals_a = take(sizeof(u32) * Lc);
    y.pairs_a = take(sizeof(uint2) * Lc);
    y.pairs_b = take(sizeof(uint2) * Lc);
    const int64_t lists = (int64_t)ctx->T * csort::MAX_PARTS;
    y.seg_start = take(sizeof(u32) * (Lc + lists + 1));      // (lists by table: one slot more per list)
    y.table_cnt = take(sizeof(u32) * lists);
    y.tb = take(sizeof(u32) * (lists + 1));
    y.chunk_first = take(sizeof(u32) * (Lc / 8 + 1));      // (the most that any L up to this one may need)
    y.tile_done = take(sizeof(uint2) * (Lc / 8 + 1));
    const int64_t ranges = std::max(std::min(Lc / 8 + 1, warps), segred::max_ranges(ctx->D, Lc));      // (the most that any L up to this one may need)
    y.partials = take(sizeof(double) * ranges * 2 * ctx->D);
    y.group_partials = take(sizeof(double) * (ranges / segred::FOLD_GROUP + 1) * 2 * ctx->D);
    y.total = o;
    return y;
}

// ---------------------------------------------------------------------------------
// heads of the sorted key array
__device__ __forceinline__ void load_tile_keys(const u32 *__restrict__ keys, int64_t L, int64_t i0,
                                               u32 (&k)[ST_ITEMS], u32 &prev, int &n)
{
    n = (int)max((int64_t)0, min((int64_t)ST_ITEMS, L - i0));
    prev = (i0 > 0 && i0 <= L) ? keys[i0 - 1] : 0xFFFFFFFFu;
    static_assert(ST_ITEMS == 8, "");
    if (n == ST_ITEMS) {                // (eight loads of a word by every thread: 16 us for 8.5 M keys)
        const uint4 x = __ldg(reinterpret_cast<const uint4 *>(keys + i0)), y = __ldg(reinterpret_cast<const uint4 *>(keys + i0) + 1);
        k[0] = x.x; k[1] = x.y; k[2] = x.z; k[3] = x.w;
        k[4] = y.x; k[5] = y.y; k[6] = y.z; k[7] = y.w;
        return;
    }
#pragma unroll
    for (int e = 0; e < ST_ITEMS; ++e) k[e] = (e < n) ? keys[i0 + e] : 0u;
}

__global__ void __launch_bounds__(ST_THREADS)
seg_count_kernel(const u32 *__restrict__ keys, int64_t L, u32 *__restrict__ tile_heads)
{
    dq_wait_before();
    __shared__ u32 wsum[ST_WARPS];
    const int64_t i0 = (int64_t)blockIdx.x * ST_TILE + (int64_t)threadIdx.x * ST_ITEMS;
    u32 k[ST_ITEMS], prev; int n;
    load_tile_keys(keys, L, i0, k, prev, n);
    u32 c = 0;
#pragma unroll
    for (int e = 0; e < ST_ITEMS; ++e) {
        if (e < n) c += (i0 + e == 0 || k[e] != prev) ? 1u : 0u;
        prev = k[e];
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) c += __shfl_xor_sync(0xffffffffu, c, o);
    if ((threadIdx.x & 31) == 0) wsum[threadIdx.x >> 5] = c;
    __syncthreads();
    if (threadIdx.x == 0) {
        u32 s = 0;
        for (int w = 0; w < ST_WARPS; ++w) s += wsum[w];
        tile_heads[blockIdx.x] = s;
    }
}

__global__ void __launch_bounds__(ST_THREADS)
seg_emit_kernel(const u32 *__restrict__ keys, int64_t L, const u32 *__restrict__ tile_heads,
                const int64_t *__restrict__ row_off, int T,
                u32 *__restrict__ seg_start, u32 *__restrict__ chunk_first,
                int32_t *__restrict__ unique_rows, int32_t *__restrict__ uniq_off, uint2 *__restrict__ tile_done,
                u32 *__restrict__ absmax, int ck_shift)
{
    dq_wait_before();
    extern __shared__ __align__(16) unsigned char smem_raw[];
    int64_t *s_off = reinterpret_cast<int64_t *>(smem_raw);   // [T+1]
    __shared__ u32 wsum[ST_WARPS];
    __shared__ u32 s_prefix;
    // this thread's keys first: they depend on nothing, so they fly beside the loads of the prefix below
    const int64_t i0 = (int64_t)blockIdx.x * ST_TILE + (int64_t)threadIdx.x * ST_ITEMS;
    const int ck = 1 << ck_shift;
    u32 k[ST_ITEMS], prev0; int n;
    load_tile_keys(keys, L, i0, k, prev0, n);
    if (blockIdx.x == 0)
        for (int t = threadIdx.x; t < T; t += ST_THREADS) absmax[t] = 0u;
    for (int t = threadIdx.x; t <= T; t += ST_THREADS) s_off[t] = row_off[t];
    // heads in all earlier tiles
    u32 p = 0;
    for (int64_t i = threadIdx.x; i < blockIdx.x; i += ST_THREADS) p += tile_heads[i];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) p += __shfl_xor_sync(0xffffffffu, p, o);
    if ((threadIdx.x & 31) == 0) wsum[threadIdx.x >> 5] = p;
    __syncthreads();
    if (threadIdx.x == 0) {
        u32 s = 0;
        for (int w = 0; w < ST_WARPS; ++w) s += wsum[w];
        s_prefix = s;
    }
    __syncthreads();
    const u32 tile_prefix = s_prefix;
    __syncthreads();

    u32 c = 0;
    {
        u32 prev = prev0;
#pragma unroll
        for (int e = 0; e < ST_ITEMS; ++e) {
            if (e < n) c += (i0 + e == 0 || k[e] != prev) ? 1u : 0u;
            prev = k[e];
        }
    }
    // block exclusive scan of c
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    u32 incl = c;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        u32 v = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += v;
    }
    if (lane == 31) wsum[warp] = incl;
    __syncthreads();
    u32 woff = 0;
    for (int w = 0; w < warp; ++w) woff += wsum[w];
    u32 heads_before = tile_prefix + woff + incl - c;   // heads strictly before entry i0

    // only the entries that start a segment are looked at (the walk over all eight with a test each took 35 us for
    // 8.5 M entries).  Tables of the keys: found once for the key before this thread's entries, then only advanced
    // (keys ascend), so a head costs a comparison instead of two searches
    u32 heads = 0;
    {
        u32 prev = prev0;
#pragma unroll
        for (int e = 0; e < ST_ITEMS; ++e) {
            if (e < n && (i0 + e == 0 || k[e] != prev)) heads |= 1u << e;
            prev = k[e];
        }
    }
    if (n <= 0) return;
    int t_prev = -1, t = 0;
    if (heads || i0 + n == L) {
        if (i0 > 0) t_prev = dq_table_of(s_off, T, (int64_t)prev0);
        t = t_prev < 0 ? 0 : t_prev;
    }
    for (u32 h = heads, u = heads_before; h; h &= h - 1u, ++u) {
        const int e = __ffs(h) - 1;
        const int64_t i = i0 + e;
        seg_start[u] = (u32)i;
        u32 ke = k[0];
#pragma unroll
        for (int x = 1; x < ST_ITEMS; ++x) if (e == x) ke = k[x];
        // a sort that refused a table leaves that table's keys undefined: keep them inside the arena and
        // the walk inside the offset list, whatever they hold
        const int64_t key = min((int64_t)ke, s_off[T] - 1);
        while (t < T - 1 && key >= s_off[t + 1]) ++t;
        unique_rows[u] = (int32_t)max((int64_t)0, key - s_off[t]);
        for (int tt = t_prev + 1; tt <= t; ++tt) uniq_off[tt] = (int32_t)u;
        t_prev = t;
    }
    // the chunks that begin among this thread's entries (a chunk is a power of two, at least eight entries)
    if ((i0 & (int64_t)(ck - 1)) == 0) {
        chunk_first[i0 >> ck_shift] = heads_before + (heads & 1u) - 1u;
        tile_done[i0 >> ck_shift] = make_uint2(0u, 0u);
    }
    if (i0 + n == L) {
        const u32 U = heads_before + __popc(heads);
        seg_start[U] = (u32)L;
        for (int tt = t_prev + 1; tt <= T; ++tt) uniq_off[tt] = (int32_t)U;
    }
}

// ---------------------------------------------------------------------------------
template <int VEC>
int launch_sum(dqrm_ctx *ctx, const segred::Args &a, int tile, cudaStream_t st)
{
    using namespace segred;
    const size_t smem = smem_bytes(a.T);
    const int64_t ranges = (a.num_tiles + a.range_tiles - 1) / a.range_tiles;
    const dim3 grid((unsigned)((ranges * a.columns + WARPS - 1) / WARPS));
    const bool exact = ctx->D % (32 * VEC) == 0;
    constexpr bool wide = VEC == 4;                          // (only those rows may have several blocks of features)
    constexpr int MOST = VEC == 2 ? 4 : 3;                   // blocks an SM
#define DQ_SUM(EXACT, I, COLS, BLOCKS) \
    DQRM_CUDA_TRY(ctx, (dq_launch(seg_sum_kernel<VEC, EXACT, I, COLS, BLOCKS>, grid, dim3(THREADS), smem, st, a)))
#define DQ_SUM2(I, BLOCKS)                                                          \
    do {                                                                            \
        if (a.columns > 1 && exact) DQ_SUM(true, I, wide, BLOCKS);                  \
        else if (a.columns > 1) DQ_SUM(false, I, wide, BLOCKS);                     \
        else if (exact) DQ_SUM(true, I, false, BLOCKS);                             \
        else DQ_SUM(false, I, false, BLOCKS);                                       \
    } while (0)
    if (tile == 8 && sum_blocks(ctx->D, a.L, ctx->num_sms) == 3) DQ_SUM2(8, 3);
    else if (tile == 8) DQ_SUM2(8, MOST);
    else if (tile == 16) DQ_SUM2(16, MOST);
    else if constexpr (VEC == 2) DQ_SUM(true, 32, false, MOST);        // (64 features)
#undef DQ_SUM2
#undef DQ_SUM
    dq_mark(ctx, st, DQ_K_SEG_SUM);
    return DQRM_OK;
}

template <int LPR>
int launch_sum_groups(dqrm_ctx *ctx, const segred::Args &a, cudaStream_t st)
{
    using namespace segred;
    // (small batches: smaller blocks, on more SMs)
    unsigned warps = GROUPS_THREADS / 32;
    while (warps > 2 && a.ranges < warps * (unsigned)ctx->num_sms) warps /= 2;
    const dim3 grid((a.ranges + warps - 1) / warps), block(warps * 32);
    if (!dq_aligned(a.grad_out, sizeof(float4)) || !dq_aligned(a.grad_rows, sizeof(float4)))
        DQRM_CUDA_TRY(ctx, (dq_launch(seg_groups_kernel<LPR, false, unaligned_vec(LPR)>, grid, block, smem_bytes(a.T), st, a)));
    else if (takes_groups(LPR * 4) && ctx->D == LPR * 4)
        DQRM_CUDA_TRY(ctx, (dq_launch(seg_groups_kernel<LPR, takes_groups(LPR * 4)>, grid, block, smem_bytes(a.T), st, a)));
    else DQRM_CUDA_TRY(ctx, (dq_launch(seg_groups_kernel<LPR, false>, grid, block, smem_bytes(a.T), st, a)));
    dq_mark(ctx, st, DQ_K_SEG_GROUPS);
    return DQRM_OK;
}

template <bool FIRST, bool LAST>
int launch_radix_pass(dqrm_ctx *ctx, const rsort::Args &a, const uint2 *in, uint2 *out, u32 *keys, u32 *vals, int shift,
                      cudaStream_t st)
{
    const unsigned tiles = (unsigned)rsort::max_tiles(a.T, a.L);
    const int nb = 1 << a.dbits;
    DQRM_CUDA_TRY(ctx, dq_launch(rsort::rs_hist_kernel<FIRST>, dim3(tiles), dim3(rsort::THREADS), 0, st, a, in, shift));
    dq_mark(ctx, st, DQ_K_SORT_HIST);
    DQRM_CUDA_TRY(ctx, dq_launch(rsort::rs_scan_kernel, dim3((unsigned)((nb + rsort::SCAN_DIGITS - 1) / rsort::SCAN_DIGITS), (unsigned)a.T),
                                 dim3(rsort::SCAN_DIGITS * rsort::SCAN_GROUPS), 0, st, a));
    dq_mark(ctx, st, DQ_K_SORT_SCAN);
    bool &raised = ctx->smem_raised[(FIRST ? 1 : 0) + (LAST ? 2 : 0)];
    if (!raised)
        DQRM_CUDA_TRY(ctx, cudaFuncSetAttribute(rsort::rs_scatter_kernel<FIRST, LAST>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                                (int)rsort::scatter_smem(1 << rsort::MAX_DIGIT_BITS)));
    raised = true;
    DQRM_CUDA_TRY(ctx, (dq_launch(rsort::rs_scatter_kernel<FIRST, LAST>, dim3(tiles), dim3(rsort::THREADS), rsort::scatter_smem(nb),
                                  st, a, in, out, keys, vals, shift)));
    dq_mark(ctx, st, DQ_K_SORT_SCATTER);
    return DQRM_OK;
}

int launch_radix_sort(dqrm_ctx *ctx, const rsort::Args &a, int passes, uint2 *const (&pairs)[2], u32 *keys, u32 *vals,
                      cudaStream_t st)
{
    DQRM_CUDA_TRY(ctx, dq_launch(rsort::rs_setup_kernel, dim3(1), dim3(1024), rsort::setup_smem(a.T), st, a));
    dq_mark(ctx, st, DQ_K_SORT_SETUP);
    for (int p = 0; p < passes; ++p) {
        const uint2 *in = pairs[(p + 1) & 1];          // (the first pass reads the indices)
        uint2 *out = pairs[p & 1];
        const int shift = p * a.dbits;
        int rc;
        if (p == 0) rc = passes == 1 ? launch_radix_pass<true, true>(ctx, a, in, out, keys, vals, shift, st)
                                     : launch_radix_pass<true, false>(ctx, a, in, out, keys, vals, shift, st);
        else rc = p + 1 == passes ? launch_radix_pass<false, true>(ctx, a, in, out, keys, vals, shift, st)
                                  : launch_radix_pass<false, false>(ctx, a, in, out, keys, vals, shift, st);
        if (rc != DQRM_OK) return rc;
    }
    return DQRM_OK;
}

// (slot: of smem_raised, one for each kernel)
template <int CL>
cudaError_t launch_clusters(dqrm_ctx *ctx, void (*kernel)(csort::Args), int slot, const csort::Args &ca, size_t smem, cudaStream_t st)
{
    bool &raised = ctx->smem_raised[DQ_SMEM_SLOT_CSORT + slot];
    cudaError_t e = cudaSuccess;
    if (!raised) {
        e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)csort::smem_bytes(12288));
        if (e == cudaSuccess && CL > 8)       // more than eight blocks in a cluster is an opt-in
            e = cudaFuncSetAttribute(kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
        raised = (e == cudaSuccess);
    }
    if (e == cudaSuccess) {
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3((unsigned)(ca.T * ca.parts * CL));
        cfg.blockDim = dim3(csort::THREADS);
        cfg.dynamicSmemBytes = smem;
        cfg.stream = st;
        cudaLaunchAttribute attr[2];
        attr[0].id = cudaLaunchAttributeClusterDimension;
        attr[0].val.clusterDim.x = CL; attr[0].val.clusterDim.y = 1; attr[0].val.clusterDim.z = 1;
        attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
        attr[1].val.programmaticStreamSerializationAllowed = 1;
        cfg.attrs = attr; cfg.numAttrs = 2;
        e = cudaLaunchKernelEx(&cfg, kernel, ca);
    }
    if (e != cudaSuccess) (void)cudaGetLastError();
    return e;
}

template <int CL, bool PARTS = false>
cudaError_t launch_cluster_sort(dqrm_ctx *ctx, csort::Args ca, int cap, cudaStream_t st)
{
    ca.cap = cap;
    return launch_clusters<CL>(ctx, csort::cluster_sort_kernel<CL, 0, PARTS>, PARTS ? 6 : CL == csort::CLUSTER_HALF ? 8 : CL == csort::CLUSTER ? 0 : 3, ca, csort::smem_bytes(cap), st);
}

cudaError_t launch_half_clusters(dqrm_ctx *ctx, csort::Args ca, int cap, cudaStream_t st)
{
    ca.cap = cap;
    return launch_clusters<csort::CLUSTER>(ctx, csort::cluster_sort_half_kernel, 7, ca, csort::smem_bytes(cap), st);
}

// Clusters of sixteen blocks for few tables of 16 K lookups and more, and of 5 K (a table alone: 8 K) where the rows take three passes and no
// training step runs beside, from which they would take twice the room.  Measured on B200 (us; sixteen blocks / eight): sort of 2 tables of
// 12,000 lookups of 1.5 M rows 15.2 / 16.8, 3 of 8000 13.4 / 14.3, 4 of 5000 13.0 / 13.3, of one (in its parts, see below) of 15,000 15.5 / 19.7,
// of 10,000 14.6 / 15.2, of 8000 of 30 K rows 12.0 / 11.3; steps of 4 tables of 4100 29.2 / 28.9, of one of 4500 28.8 / 28.1; eight
// pipelined steps of one table of 10,000 182 / 142, of 4 of 5000 172 / 142
bool wide_clusters(const dqrm_ctx *ctx, int64_t per_table, bool beside)
{
    const int64_t least = ctx->row_bits <= 16 || beside ? 1024 : ctx->T > 1 ? 320 : 512;       // lookups for a block
    return ctx->T * csort::CLUSTER_WIDE * 2 <= ctx->num_sms && per_table >= csort::CLUSTER_WIDE * least;
}

// A table alone is shared by four clusters of sixteen blocks where as many as eight would fit (eight do not find room at the same
// moment: 34 us), from 16 K lookups on; of tables whose rows take two passes from 48 K, of those whose quarters take a pass less than
// they do from 8 K.  Measured on B200 (us a backward; four clusters / one): 65,536 lookups of 4 M rows 26.5 / 35.3, Zipf 1.2 28.1 / 32.0, all in
// the first quarter 27.7 / 34.2, nine tenths in one row 26.7 / 33.2, all in one 21.8 / 27.8; 25,000 21.1 / 23.2, 23.4 / 24.1, 23.4 /
// 24.4, 23.8 / 24.5, 18.6 / 22.5; 17,000 20.4 / 21.5, but rows numbered by how often they come 23.4 / 22.8 (eight pipelined steps
// around them 160 / 180); of 260 K rows 10,000 18.4 / 20.7; of 3000 rows 50,000 22.1 / 24.9, nine tenths in one row 22.5 / 23.2, 32,000 20.0 /
// 21.1 but 21.1 / 20.0.  Two tables by two clusters each: 65,536 of 2 M rows 18.1 / 18.6 the sort, 30,000 of 1500 13.9 / 13.2, so they
// have one each.  Clusters of eight as parts: 28.9 (four), 40.3 (sixteen)
int table_parts(const dqrm_ctx *ctx, int64_t per_table)
{
    if (ctx->T > 1 || per_table < csort::CLUSTER_WIDE * (ctx->row_bits <= 16 ? 3072 : ctx->row_bits <= 18 ? 512 : 1024)) return 1;
    return 2 * csort::CLUSTER_WIDE * csort::MAX_PARTS <= ctx->num_sms ? csort::MAX_PARTS : 1;
}

// Batches of an index a bag, whose tables are all alike: clusters of four blocks.  Where clusters of eight for all tables do not fit at
// once (two blocks an SM: from 34 tables on) the last of them wait for the first: 40 tables of 4000 lookups 37.5 -> 26.7 us a backward, of
// 10,000 55.9 -> 43.7, 64 of 4000 42.7 -> 30.3, eight pipelined steps around them (40 of 3000 of 16 features, of 16,000 of 8) 313 -> 213 and
// 530 -> 426; the sort of 20,000 36.1 -> 40.5, four blocks have too much to do.  Where they fit, but share SMs (from 19 tables on): 26 tables of
// 2500 lookups 21.2 -> 19.5 a backward, of 8000 29.7 -> 28.0, the sort of 9000 18.1 -> 18.4.  Beside a training step (dqrm_sort_batch) four
// blocks leave it more room and take longer themselves, so that count the step's rows: 26 tables of 8000 lookups of 48 features 487 -> 452 us
// for eight steps, of 16 282 -> 287, of 8 250 -> 266, of 2500 of 16 189 -> 160; they are taken there for rows of 32 features and
// more, and for small tables.  (A batch that has as many lookups as bags without one in each, and most of them in one table, pays for it:
// 26 tables of 8000 with nine tenths in one 240 -> 430.  All that is known at the launch are the two numbers.)
bool narrow_clusters(const dqrm_ctx *ctx, int64_t per_table, bool beside)
{
    if (ctx->T * csort::CLUSTER > 2 * ctx->num_sms) return per_table <= 16384;
    return ctx->T * csort::CLUSTER > ctx->num_sms && per_table <= (!beside || ctx->D >= 32 ? 8192 : 2560);
}

// Other batches, of which one table may hold most, and the merge of ranks' gradients: clusters of eight of which half works unless a table
// is large (cluster_sort_half_kernel).  33 clusters of eight run at once; blocks that leave at once let those beyond in.  Measured on B200
// (us a backward; eight blocks / half of them): 34 tables of 2100 lookups 30.5 / 22.7, 40 of 4000 37.5 / 27.9, of 10,000 55.9 / 45.7, 46 of
// 16,000 70.3 / 59.9, 58 of 12,000 63.5 / 54.0, 64 of 2100 35.3 / 34.6, of 8000 54.7 / 56.2, of 12,000 66.5 / 74.1 (two full rounds of clusters
// of eight), 70 of 16,000 100.2 / 98.3, 148 of 6000 109.1 / 84.5; 33 of 6000 27.3 / 30.0; 36 of 12,000 52.8 / 53.3.  With nine tenths
// of the lookups in one table as before: 40 of 4000 194 / 194, 64 of 4000 287 / 288 (clusters of four in every table 344 and 524).
// Beside a training step of rows of 32 features and more the room counts from 19 tables on: eight pipelined steps of 26 tables of 2500
// lookups of 32 features 225 / 205, of 8000 of 48 487 / 455; of 2500 of 16 189 / 195
bool half_clusters(const dqrm_ctx *ctx, int64_t per_table, bool beside)
{
    constexpr int AT_ONCE = 33;
    if (ctx->T > AT_ONCE) {
        if (ctx->T > 2 * AT_ONCE - 8 && ctx->T <= 2 * AT_ONCE) return per_table <= 4096;
        return per_table <= (ctx->T > AT_ONCE + 4 ? 16384 : 8192);
    }
    return beside && ctx->D >= 32 && ctx->T * csort::CLUSTER > ctx->num_sms && per_table <= 8192;
}

// clusters that stand by for tables beyond what their first block takes
template <int EPT>
cudaError_t launch_standby_sort(dqrm_ctx *ctx, csort::Args ca, bool even, cudaStream_t st)
{
    constexpr int CL = csort::CLUSTER;
    ca.cap = even ? csort::SORT_ROOM / 2 : csort::shared_cap(ca.L);
    const size_t smem = std::max(csort::smem_bytes(ca.cap), sizeof(uint2) * csort::SORT_ROOM);
    if constexpr (EPT == 4)
        if (even) return launch_clusters<CL>(ctx, ssort::small_sort_kernel<csort::THREADS, EPT, CL>, 5, ca, smem, st);
    return launch_clusters<CL>(ctx, csort::cluster_sort_kernel<CL, EPT>, EPT, ca, smem, st);
}

// The block sort; false where the batch is too large for it.  `per_table` lookups a table on average, with room for a
// quarter more where bags are uneven.  Up to 256 the network, beyond it the radix sort.  Measured on B200 (graph replay, 26
// tables of up to 6 M rows, us per batch; radix sort / network / cluster): 64 lookups a table 4.9 / 3.2, 256 4.9 / 4.1, 500
// 4.7 / 6.2, 1000 5.8 / 8.2 / 12.6, 2000 8.2 / - / 13.3, one table of 3000 11.5 / - / 11.1.  Unless the batch has an index a
// bag, one table may hold most of it: a cluster of blocks then stands by for every table (a table of
// 12.8 K lookups beside 25 of 128: 22.8 us, 99 by one block in global memory, 34.8 in a cluster of whole batches; bags of
// five everywhere 9.9, 9.2 by the network without the clusters standing by).  Even batches (as many lookups as bags, which
// need not be one in each) have them from 1024 lookups a table on, where there is room for the clusters: 26 tables of 2048 with 90 %
// of the lookups in one 66 us, 390 without, and none the slower where they are not needed; pairs beyond 8192 in a table go through
// global memory, since more shared memory would be held by every block.
bool launch_small_sort(dqrm_ctx *ctx, const csort::Args &ca, int64_t per_table, bool even, cudaStream_t st, cudaError_t &e)
{
    const int64_t want = even ? per_table : per_table + per_table / 4;
    if (want > 2048) return false;
    const dim3 grid((unsigned)ctx->T), block(csort::THREADS);
    constexpr size_t room = sizeof(uint2) * csort::SORT_ROOM;
    static_assert(csort::SORT_ROOM >= 4 * csort::THREADS, "");
    if (!even || (want > 1024 && ctx->T * csort::CLUSTER <= 2 * ctx->num_sms)) {
        e = want <= 512    ? launch_standby_sort<1>(ctx, ca, even, st)
            : want <= 1024 ? launch_standby_sort<2>(ctx, ca, even, st)
                           : launch_standby_sort<4>(ctx, ca, even, st);
    } else if (want <= 256) e = dq_launch(ssort::small_sort_kernel<256, 1, 1>, grid, dim3(256), ssort::smem_bytes(256), st, ca);
    else if (want <= 512) e = dq_launch(ssort::small_sort_kernel<csort::THREADS, 1, 1>, grid, block, room, st, ca);
    else if (want <= 1024) e = dq_launch(ssort::small_sort_kernel<csort::THREADS, 2, 1>, grid, block, room, st, ca);
    else e = dq_launch(ssort::small_sort_kernel<csort::THREADS, 4, 1>, grid, block, room, st, ca);
    return true;
}

}  // namespace

void dq_bwd_ws_views(const dqrm_ctx *ctx, int64_t L, char *ws, const u32 **sorted_vals, const u32 **seg_start)
{
    const Layout y = make_layout(ctx, L);
    *sorted_vals = reinterpret_cast<const u32 *>(ws + y.vals_a);
    *seg_start = reinterpret_cast<const u32 *>(ws + y.seg_start);
}

const u32 *dq_bwd_absmax_bits(const dqrm_ctx *ctx, int64_t L, const void *ws)
{
    return reinterpret_cast<const u32 *>(reinterpret_cast<const char *>(ws) + make_layout(ctx, L).absmax);
}

size_t dq_bwd_ws_bytes(const dqrm_ctx *ctx, int64_t L, int64_t G)
{
    (void)G;
    return make_layout(ctx, L).total;
}

size_t dq_sum_align(const dqrm_ctx *ctx)
{
    if (segred::takes_groups(ctx->D)) return sizeof(float) * segred::unaligned_vec(segred::lanes_per_row(ctx->D));
    return sizeof(float) * segred::floats_per_lane(ctx->D);
}

// first half of the backward: everything that depends only on the indices (sort, unique rows,
// segment starts).  It needs no upstream gradient, so a training step runs it beside the forward.
int dq_launch_bwd_sort(dqrm_ctx *ctx, const int32_t *indices, const int32_t *offsets,
                       int32_t *unique_rows, int32_t *uniq_off, int B, int64_t L,
                       void *ws_, size_t ws_bytes, cudaStream_t st, int *lists, bool beside)
{
    const bool lists_by_table = lists != nullptr;
    const int64_t G = (int64_t)ctx->T * B;
    const Layout y = make_layout(ctx, L, G);
    if (ws_bytes < y.total) return DQRM_ERR_WORKSPACE;
    char *ws = reinterpret_cast<char *>(ws_);
    if (lists) *lists = 0;
    const bool fits_cluster = (L + ctx->T - 1) / ctx->T <= (int64_t)csort::CLUSTER * 12288;   // (a table beyond its
    // blocks' shared memory still sorts, through global staging, but slowly)
    const bool try_cluster = ctx->sort_path != 1 && fits_cluster;
    if (L == 0) {
        DQRM_CUDA_TRY(ctx, cudaMemsetAsync(ws + y.absmax, 0, sizeof(u32) * ctx->T, st));
        DQRM_CUDA_TRY(ctx, cudaMemsetAsync(uniq_off, 0, sizeof(int32_t) * (ctx->T + 1), st));
        return DQRM_OK;
    }
    u32 *keys[1] = {reinterpret_cast<u32 *>(ws + y.keys_a)};
    u32 *vals[1] = {reinterpret_cast<u32 *>(ws + y.vals_a)};
    uint2 *pairs[2] = {reinterpret_cast<uint2 *>(ws + y.pairs_a), reinterpret_cast<uint2 *>(ws + y.pairs_b)};
    const u32 *skeys = nullptr;      // sorted keys; the sorted payloads sit beside them in vals[0]
    bool sorted = false;
    int parts = 1;                   // clusters, and so lists, of a table
    // (tables far beyond the shared-memory slices sort faster with the global radix sort)
    if (try_cluster) {
        if (!lists_by_table) {
            DQRM_CUDA_TRY(ctx, cudaMemsetAsync(ws + y.tile_heads, 0, sizeof(u32) * y.num_tiles, st));
            dq_mark(ctx, st, DQ_K_MEMSET);
        }
        // one cluster of eight blocks per table (sixteen when so few tables would leave most SMs idle); falls
        // through to clusters of eight, then to the global radix sort, if a launch is refused
        csort::Args ca;
        ca.indices = indices; ca.offsets = offsets; ca.row_off = ctx->d_row_off;
        ca.T = ctx->T; ca.B = B; ca.L = L;
        ca.keys_out = keys[0]; ca.vals_out = vals[0];
        // global staging of (row, payload) pairs, used only by tables too large for shared memory
        ca.gp[0] = reinterpret_cast<uint2 *>(ws + y.pairs_a); ca.gp[1] = reinterpret_cast<uint2 *>(ws + y.pairs_b);
        ca.status = ctx->d_status;
        ca.payload_position = ctx->payload_position;
        ca.tile_heads = reinterpret_cast<u32 *>(ws + y.tile_heads);
        // when dq_launch_bwd_sum follows, the clusters number their own tables' segments and seg_emit is not run
        ca.lists_by_table = lists_by_table ? 1 : 0;
        ca.seg_start = reinterpret_cast<u32 *>(ws + y.seg_start);
        ca.chunk_first = reinterpret_cast<u32 *>(ws + y.chunk_first);
        ca.table_cnt = reinterpret_cast<u32 *>(ws + y.table_cnt);
        ca.tb = reinterpret_cast<u32 *>(ws + y.tb);
        ca.tile_done = reinterpret_cast<uint2 *>(ws + y.tile_done);
        ca.absmax = reinterpret_cast<u32 *>(ws + y.absmax);
        ca.ck_shift = y.sum_shift;
        ca.cnt_broken = segred::CNT_BROKEN;
        ca.parts = 1;
        const int64_t per_table = (L + ctx->T - 1) / ctx->T;
        cudaError_t e = cudaErrorUnknown;
        if (lists_by_table && launch_small_sort(ctx, ca, per_table, L == G, st, e)) {
            if (e == cudaSuccess) {
                dq_mark(ctx, st, L == G ? DQ_K_SMALL_SORT : DQ_K_CLUSTER_SORT);
                *lists = 1;
                return DQRM_OK;
            }
            ctx->last_cuda_error = (int)e;         // (taken off the runtime, so that nobody finds it behind the sort that follows)
            (void)cudaGetLastError();
        }
        const bool wide = wide_clusters(ctx, per_table, beside);
        e = cudaErrorUnknown;
        if (wide && lists_by_table) {
            ca.parts = table_parts(ctx, per_table);
            if (ca.parts > 1) e = launch_cluster_sort<csort::CLUSTER_WIDE, true>(ctx, ca, csort::choose_cap(per_table, csort::CLUSTER_WIDE), st);
            if (e != cudaSuccess) ca.parts = 1;
        }
        if (wide && e != cudaSuccess) e = launch_cluster_sort<csort::CLUSTER_WIDE>(ctx, ca, csort::choose_cap(per_table, csort::CLUSTER_WIDE), st);
        if (e != cudaSuccess && L == G && lists_by_table && narrow_clusters(ctx, per_table, beside))
            e = launch_cluster_sort<csort::CLUSTER_HALF>(ctx, ca, csort::choose_cap(per_table, csort::CLUSTER_HALF), st);
        else if (e != cudaSuccess && half_clusters(ctx, per_table, beside))
            e = launch_half_clusters(ctx, ca, csort::choose_cap(per_table, csort::CLUSTER_HALF), st);
        if (e != cudaSuccess) e = launch_cluster_sort<csort::CLUSTER>(ctx, ca, csort::choose_cap(per_table, csort::CLUSTER), st);
        if (e == cudaSuccess) {
            dq_mark(ctx, st, DQ_K_CLUSTER_SORT);
            skeys = keys[0];
            sorted = true;
            parts = ca.parts;
        } else {
            ctx->last_cuda_error = (int)e;
        }
    }
    if (!sorted) {
        rsort::Args ra;
        ra.indices = indices; ra.offsets = offsets; ra.row_off = ctx->d_row_off;
        ra.T = ctx->T; ra.B = B; ra.L = L; ra.G = G;
        ra.tb = reinterpret_cast<u32 *>(ws + y.tb);
        ra.tile0 = reinterpret_cast<u32 *>(ws + y.tile0);
        ra.tile_table = reinterpret_cast<u32 *>(ws + y.tile_table);
        ra.tilehist = reinterpret_cast<u32 *>(ws + y.tilehist);
        ra.totals = reinterpret_cast<u32 *>(ws + y.totals);
        ra.dbits = y.digit_bits;
        ra.payload_position = ctx->payload_position;
        ra.status = ctx->d_status;
        const int rc = launch_radix_sort(ctx, ra, y.passes, pairs, keys[0], vals[0], st);
        if (rc != DQRM_OK) return rc;
        skeys = keys[0];
    }
    if (sorted && lists_by_table) {                    // the lists are there; unique_rows and uniq_off come with the sums
        *lists = parts;
        return DQRM_OK;
    }
    if (!sorted) {        // (a cluster sort that did not number the segments itself has counted the segment heads of every tile)
        DQRM_CUDA_TRY(ctx, dq_launch(seg_count_kernel, dim3((unsigned)y.num_tiles), dim3(ST_THREADS), 0, st, skeys, L,
                                     reinterpret_cast<u32 *>(ws + y.tile_heads)));
        dq_mark(ctx, st, DQ_K_SEG_COUNT);
    }
    DQRM_CUDA_TRY(ctx, dq_launch(seg_emit_kernel, dim3((unsigned)y.num_tiles), dim3(ST_THREADS),
        (size_t)(ctx->T + 1) * sizeof(int64_t), st, skeys, L, reinterpret_cast<const u32 *>(ws + y.tile_heads), ctx->d_row_off, ctx->T,
        reinterpret_cast<u32 *>(ws + y.seg_start), reinterpret_cast<u32 *>(ws + y.chunk_first), unique_rows, uniq_off,
        reinterpret_cast<uint2 *>(ws + y.tile_done), reinterpret_cast<u32 *>(ws + y.absmax), y.sum_shift));
    dq_mark(ctx, st, DQ_K_SEG_EMIT);
    return DQRM_OK;
}

// second half: segmented sum of the upstream gradient over the sorted lookups
int dq_launch_bwd_sum(dqrm_ctx *ctx, const float *grad_out, int32_t *unique_rows, int32_t *uniq_off, float *grad_rows,
                      int B, int64_t L, int lists, void *ws_, size_t ws_bytes, cudaStream_t st)
{
    const Layout y = make_layout(ctx, L, (int64_t)ctx->T * B);
    if (ws_bytes < y.total) return DQRM_ERR_WORKSPACE;
    if (L == 0) return DQRM_OK;
    char *ws = reinterpret_cast<char *>(ws_);
    segred::Args a = {};
    const int D = ctx->D;
    // both sort paths leave the sorted pairs in the first key / payload buffers
    a.keys = reinterpret_cast<const u32 *>(ws + y.keys_a);
    a.vals = reinterpret_cast<const u32 *>(ws + y.vals_a);
    a.seg_start = reinterpret_cast<const u32 *>(ws + y.seg_start);
    a.chunk_first = reinterpret_cast<const u32 *>(ws + y.chunk_first);
    a.range_done = reinterpret_cast<uint2 *>(ws + y.tile_done);
    a.by_table = lists > 0;
    while ((1 << a.parts_log) < lists) ++a.parts_log;
    a.table_cnt = reinterpret_cast<const u32 *>(ws + y.table_cnt);
    a.tb = reinterpret_cast<const u32 *>(ws + y.tb);
    a.row_off = ctx->d_row_off;
    a.unique_rows = unique_rows; a.uniq_off = uniq_off;
    a.grad_out = grad_out; a.grad_rows = grad_rows;
    a.partials = reinterpret_cast<double *>(ws + y.partials);
    a.group_partials = reinterpret_cast<double *>(ws + y.group_partials);
    a.absmax = reinterpret_cast<u32 *>(ws + y.absmax);
    a.T = ctx->T << a.parts_log; a.D = ctx->D;
    a.L = L; a.G = (int64_t)ctx->T * B;
    a.num_tiles = y.sum_tiles;
    a.range_tiles = y.range_tiles;
    a.columns = segred::column_blocks(D);
    a.span = (u32)y.sum_span;
    a.ranges = (u32)y.sum_ranges;
    a.status = ctx->d_status;
    if (!segred::takes_groups(D)) return D <= 64 ? launch_sum<2>(ctx, a, y.sum_tile, st) : launch_sum<4>(ctx, a, y.sum_tile, st);
    switch (segred::lanes_per_row(D)) {
    case 1: return launch_sum_groups<1>(ctx, a, st);
    case 2: return launch_sum_groups<2>(ctx, a, st);
    case 4: return launch_sum_groups<4>(ctx, a, st);
    case 8: return launch_sum_groups<8>(ctx, a, st);
    default: return launch_sum_groups<16>(ctx, a, st);
    }
}

// The one-launch step takes tables of up to 512 lookups and 16 K gathered values, up to 4096 lookups in all (what a block
// counts in front of its own).  Measured on B200 (us a step with the forward, this way / in four launches, in graph replay and
// launched one by one): 4 tables of 128 lookups of 16 features 8.1 / 14.6, 9.2 / 14.6; 512 of 16 12.2 / 18.8, 11.9 / 18.4; 256 of 64
// 13.4 / 18.0, 12.9 / 17.1; 128 of 128 13.3 / 19.1, 12.6 / 18.1; 26 tables of 128 of 16 12.4 / 18.5, 12.4 / 17.7, of 64
// 13.8 / 19.6, 13.2 / 18.9.  At the line the two ways of launching part: 26 tables of 128 of 128 16.4 / 15.4 but 15.9 / 18.7, 16 of 256
// of 64 17.6 / 15.4 but 17.0 / 18.7; beyond it (when the line was drawn) 4 tables of 1024 of 16 22.3 / 21.0, 512 of 64 24.8 / 22.0.
// (With a row summary attached, or the sort chosen by the caller, the launches stay apart.)
static bool small_bwd_takes(const dqrm_ctx *ctx, int B, int64_t L)
{
    const int64_t per_table = (L + ctx->T - 1) / ctx->T, want = L == (int64_t)ctx->T * B ? per_table : per_table + per_table / 4;
    // unless the batch has an index a bag, all of it may lie in one table, whose block then does everything: 1536 lookups of 16
    // features 29.8 us, 32.2 in separate launches; 2048 38 / 29, 1024 of 32 features 29 / 27, of 64 42 / 27
    if (L != (int64_t)ctx->T * B && (L > 1536 || L * ctx->D > 32768)) return false;
    return L > 0 && L <= sstep::MAX_LOOKUPS && want <= sstep::THREADS && want * ctx->D <= 16384 && ctx->D <= 128 &&
           ctx->T <= ctx->num_sms && ctx->sort_path != 1 && !ctx->payload_position;
}

bool dq_small_step_takes(const dqrm_ctx *ctx, int B, int64_t L) { return !ctx->row_summary && small_bwd_takes(ctx, B, L); }

template <bool STEP>
static int launch_small(dqrm_ctx *ctx, float *tables, const int32_t *indices, const int32_t *offsets, const float *grad_out,
                         int32_t *unique_rows, int32_t *uniq_off, float *grad_rows, int8_t *codes, float *grad_scales, float lr,
                         int B, int64_t L, void *ws_, size_t ws_bytes, cudaStream_t st)
{
    const Layout y = make_layout(ctx, L);
    if (ws_bytes < y.total) return DQRM_ERR_WORKSPACE;
    char *ws = reinterpret_cast<char *>(ws_);
    sstep::Args x = {};
    x.s.indices = indices; x.s.offsets = offsets; x.s.row_off = ctx->d_row_off;
    x.s.T = ctx->T; x.s.B = B; x.s.L = L;
    x.s.gp[0] = reinterpret_cast<uint2 *>(ws + y.pairs_a); x.s.gp[1] = reinterpret_cast<uint2 *>(ws + y.pairs_b);
    x.s.status = ctx->d_status;
    x.grad_out = grad_out; x.tables = tables; x.grad_rows = grad_rows;
    x.unique_rows = unique_rows; x.uniq_off = uniq_off; x.codes = codes; x.grad_scales = grad_scales;
    x.lr = lr; x.D = ctx->D;
    while ((4 << x.lpr_log) < ctx->D) ++x.lpr_log;
    const size_t smem = sstep::smem_bytes(ctx->T);
    bool &raised = ctx->smem_raised[DQ_SMEM_SLOT_STEP + (STEP ? 0 : 1)];
    // (the limit belongs to the function on the device, not to this context: every context sets the same, that of the most
    // tables that dq_small_step_takes lets through, or one with few tables would lower it for one with many)
    if (!raised)
        DQRM_CUDA_TRY(ctx, cudaFuncSetAttribute(sstep::small_step_kernel<STEP>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                                (int)sstep::smem_bytes(ctx->num_sms)));
    raised = true;
    DQRM_CUDA_TRY(ctx, dq_launch(sstep::small_step_kernel<STEP>, dim3((unsigned)ctx->T), dim3(sstep::THREADS), smem, st, x));
    dq_mark(ctx, st, DQ_K_SMALL_STEP);
    return DQRM_OK;
}

int dq_launch_small_step(dqrm_ctx *ctx, float *tables, const int32_t *indices, const int32_t *offsets, const float *grad_out,
                         int32_t *unique_rows, int32_t *uniq_off, float *grad_rows, int8_t *codes, float *grad_scales, float lr,
                         int B, int64_t L, void *ws, size_t ws_bytes, cudaStream_t st)
{
    return launch_small<true>(ctx, tables, indices, offsets, grad_out, unique_rows, uniq_off, grad_rows, codes, grad_scales, lr, B, L, ws,
                              ws_bytes, st);
}

// A backward that stands alone (behind it a step would read the workspace's maxima) in one launch instead of two: up to 3600 lookups of
// an index a bag, fewer of rows of less than 16 features, 64 K gathered values, unless they are many tables of up to 64.  Measured on
// B200 (us a backward in graph replay; two launches / one): 4 tables of 128 lookups of 16 features 9.5 / 7.2, of 512 11.6 / 10.4, 16 of
// 200 10.9 / 10.2, of 128 of 32 features 10.4 / 9.1, 2 of 100 of 128 10.0 / 8.1; around it the four calls of 16 tables of 200 22.0 / 20.0, of
// 26 of 64 19.0 / 18.2, of 26 of 90 22.0 / 20.0, of 26 of 128 20.2 / 19.8 (all of 100 K rows 20.1 / 20.9), of 13 of 256 21.7 / 20.3, of 40 of
// 90 22.5 / 22.1, but of 48 of 64 19.8 / 21.2, of 8 of 512 21.1 / 21.5 to 22.1, of 10 of 400 19.7 / 21.0 where tables have three rows, and of 26 of 128 of 8 features 19.2 / 20.6.  (The block counts the
// lookups in front of its own by their rows; all in one row they wait for one another: 8 tables of 256 of one row each 20.5 / 22.9.)
// Other batches may lie in one table, whose block then does everything: up to 1100 lookups and 32 K values.  13 tables of 40 bags of two
// 13.4 / 7.5, with nine tenths of the lookups in one 16.1 / 14.5; 4 of 90 bags of four 11.3 / 8.8, but 15.5 / 20.2; 4 of 64 bags of four of
// 16 features 13.4 / 8.2 and 15.7 / 15.6; 10 of 25 of 32 features 13.6 / 7.5 and 15.5 / 17.5.
static bool small_bwd_takes_alone(const dqrm_ctx *ctx, int B, int64_t L)
{
    if (L == (int64_t)ctx->T * B) {
        if (L > (ctx->D < 16 ? 192 * ctx->D : 3600) || L * ctx->D > 65536 || (L > 2048 && B <= 64)) return false;
    } else if (L > 1100 || L * 4 * segred::lanes_per_row(ctx->D) > 32768) {        // (with the features that idle lanes stand for)
        return false;
    }
    return small_bwd_takes(ctx, B, L);
}

int dq_launch_bwd(dqrm_ctx *ctx, const float *grad_out, const int32_t *indices, const int32_t *offsets,
                  int32_t *unique_rows, int32_t *uniq_off, float *grad_rows, int B, int64_t L,
                  void *ws, size_t ws_bytes, cudaStream_t st, bool alone)
{
    if (alone && small_bwd_takes_alone(ctx, B, L) && dq_aligned(grad_out, sizeof(float4)) && dq_aligned(grad_rows, sizeof(float4)))
        return launch_small<false>(ctx, nullptr, indices, offsets, grad_out, unique_rows, uniq_off, grad_rows, nullptr, nullptr, 0.f, B, L, ws,
                                   ws_bytes, st);
    int lists = 0;
    int rc = dq_launch_bwd_sort(ctx, indices, offsets, unique_rows, uniq_off, B, L, ws, ws_bytes, st, &lists);
    if (rc != DQRM_OK) return rc;
    return dq_launch_bwd_sum(ctx, grad_out, unique_rows, uniq_off, grad_rows, B, L, lists, ws, ws_bytes, st);
}

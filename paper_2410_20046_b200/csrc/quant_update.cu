// INT8 gradient quantiser and touched-row SGD update (paper Appendix B.1): the values of
// the sparse embedding gradient are quantised to INT8 with one scale per table, fixed
// by the bit width and the tensor's own abs-max, and the local step is taken with the
// dequantised gradient on the FP32 master rows (Section 3.1).
//
// Three variants of one row-streaming kernel share the addressing: quantise only,
// update only (from stored codes), and quantise + update fused (the training step).
// A group of LPR lanes owns a contiguous range of unique rows and keeps a few of them in flight;
// rows are distinct, so the read-modify-write of the master rows needs no atomics.  All
// streams are 128-bit per lane.
#include <algorithm>
#include <cooperative_groups.h>
#include <mutex>
#include "common.cuh"
#include "row_stream.cuh"

namespace {

using namespace rowstream;

__global__ void __launch_bounds__(QU_THREADS)
absmax_kernel(const float *__restrict__ grad_rows, const int32_t *__restrict__ uniq_off, int T, int D,
              u32 *__restrict__ absmax)
{
    dq_wait_before();
    extern __shared__ __align__(16) unsigned char smem_raw[];
    int32_t *s_uoff = reinterpret_cast<int32_t *>(smem_raw);      // [T+1]
    u32 *s_max = reinterpret_cast<u32 *>(s_uoff + (T + 1));       // [T]
    for (int t = threadIdx.x; t <= T; t += QU_THREADS) s_uoff[t] = uniq_off[t];
    for (int t = threadIdx.x; t < T; t += QU_THREADS) s_max[t] = 0u;
    __syncthreads();
    const int d4 = D >> 2;
    const int64_t n4 = (int64_t)s_uoff[T] * d4;
    const float4 *g4 = reinterpret_cast<const float4 *>(grad_rows);
    int cur_t = -1;
    int64_t cur_end4 = -1;
    float m = 0.f;
    for (int64_t base = (int64_t)blockIdx.x * QU_THREADS; base < n4; base += (int64_t)gridDim.x * QU_THREADS) {
        int64_t i = base + threadIdx.x;
        bool ok = i < n4;
        float v = 0.f;
        int t = cur_t;
        if (ok) {
            float4 x = __ldg(g4 + i);
            v = fmaxf(fmaxf(fabsf(x.x), fabsf(x.y)), fmaxf(fabsf(x.z), fabsf(x.w)));
            if (i >= cur_end4) {
                t = table_of_row(s_uoff, T, i / d4);
                cur_end4 = (int64_t)s_uoff[t + 1] * d4;
            }
        }
        if (t != cur_t) {
            if (cur_t >= 0 && m > 0.f) atomicMax(&s_max[cur_t], __float_as_uint(m));
            cur_t = t;
            m = 0.f;
        }
        m = fmaxf(m, v);
    }
    if (cur_t >= 0 && m > 0.f) atomicMax(&s_max[cur_t], __float_as_uint(m));
    __syncthreads();
    for (int t = threadIdx.x; t < T; t += QU_THREADS)
        if (s_max[t]) atomicMax(&absmax[t], s_max[t]);
}

__global__ void __launch_bounds__(QU_THREADS)
zero_kernel(u32 *__restrict__ p, int n)
{
    dq_wait_before();
    for (int i = threadIdx.x; i < n; i += QU_THREADS) p[i] = 0u;
}

// per-table maxima of |grad_rows|: cleared by a kernel and not by a memset, behind which the next kernel could not be
// set up early (four calls of a small batch, before one launch took these: 29.9 us with the memset, 26.7 with the kernel)
int launch_absmax(dqrm_ctx *ctx, const float *grad_rows, const int32_t *uniq_off, u32 *absmax, cudaStream_t st)
{
    const size_t smem = (size_t)(ctx->T + 1) * sizeof(int32_t) + (size_t)ctx->T * sizeof(u32);
    DQRM_CUDA_TRY(ctx, dq_launch(zero_kernel, dim3(1), dim3(QU_THREADS), 0, st, absmax, ctx->T));
    dq_mark(ctx, st, DQ_K_ZERO);
    DQRM_CUDA_TRY(ctx, dq_launch(absmax_kernel, dim3(ctx->num_sms * 8), dim3(QU_THREADS), smem, st, grad_rows, uniq_off, ctx->T,
                                 ctx->D, absmax));
    dq_mark(ctx, st, DQ_K_ABSMAX);
    return DQRM_OK;
}

// Quantiser in one launch: a cluster of up to eight blocks takes a table, finds its abs-max (over shared memory of the
// cluster) and quantises what it still holds in registers; what does not fit in them is read again.  Three launches that
// clear the maxima, find them and quantise are bound by the launches' own latency until the values fill the memory system.
// Measured on B200 (us, graph replay; one launch / three), 26 tables: 8 K values a table 3.2 / 6.5, 64 K 4.4 / 9.4,
// 128 K 5.9 / 13.8, 512 K 19 / 33; one table: 8 K 2.7 / 5.2, 128 K 4.1 / 5.8, 256 K 5.6 / 5.9, 320 K 6.6 / 5.9 (eight
// blocks are too few for what they do not hold); seven tables of 512 K 10.2 / 13.2.  256 threads a block while that
// holds a table (40 tables of 64 K values take 5.2 us with 256 and 8.4 with 512: a second wave), 512 then, and 1024
// where the tables are few and do not fill the chip with 512 (seven of 256 K: 5.8 us, 8.0 with 512).
//
// How the values spread over the tables is not known before the launch, and one table may hold nearly all of them.  A
// table beyond `limit` vectors, twice what its cluster holds, is therefore left by its cluster to all: its abs-max is found
// by every block that is there (one partial a block), and a second launch, made only when max_values allows such a table,
// quantises it with the whole chip.  Measured on B200 (us; this way / its cluster alone / three launches), 26 tables of which
// one has 61 K rows of 64 values and the others 1024: 18.5 / 103 / 18.6; 2048 rows of 64 in every table 7.4 / 6.0 / 18.3, the
// second launch having nothing to do; all rows, 4096 of 64, in one of 26 tables 12.3 / 14.8 / 10.4.
constexpr int QC_VEC = 8;             // vectors of four that a thread holds
constexpr int QC_CLUSTER = 8;
constexpr int QH_THREADS = 512;

struct Heavy {
    int64_t limit;                    // vectors of a table that its cluster takes itself
    u32 *partial;                     // [T][blocks] abs-max that a block found in a table beyond it; null: there can be none
    int blocks;                       // blocks that look for it
};

__device__ __forceinline__ int64_t table_vectors(const int32_t *uniq_off, int t, int d4)
{
    return max((int64_t)__ldg(uniq_off + t + 1) - __ldg(uniq_off + t), (int64_t)0) * d4;
}

// whether a table is beyond the limit (the same answer in every thread of the block)
__device__ __forceinline__ bool any_heavy(const int32_t *uniq_off, int T, int d4, int64_t limit)
{
    bool any = false;
    for (int t = threadIdx.x; t < T; t += blockDim.x) any |= table_vectors(uniq_off, t, d4) > limit;
    return __syncthreads_or(any);
}

__device__ __forceinline__ float abs_max4(const float4 &v)
{
    return fmaxf(fmaxf(fabsf(v.x), fabsf(v.y)), fmaxf(fabsf(v.z), fabsf(v.w)));
}

// abs-max over the block, in thread 0 (non-negative floats order as their bits)
template <int THREADS>
__device__ __forceinline__ float block_max(float m, float *s_warp)
{
    const u32 wm = __reduce_max_sync(0xffffffffu, __float_as_uint(m));
    __syncthreads();                                   // (s_warp may still be read)
    if (threadIdx.x % 32 == 0) s_warp[threadIdx.x / 32] = __uint_as_float(wm);
    __syncthreads();
    float b = 0.f;
    if (threadIdx.x == 0)
        for (int w = 0; w < THREADS / 32; ++w) b = fmaxf(b, s_warp[w]);
    return b;
}

__device__ __forceinline__ void put_codes(char4 *c, const float4 &v, const QuantScale &qs)
{
    float4 q, unused;
    dq_fq4(v, qs, q, unused);
    __stcs(c, make_char4((signed char)(int)q.x, (signed char)(int)q.y, (signed char)(int)q.z, (signed char)(int)q.w));
}

template <int QC_THREADS>
__global__ void __launch_bounds__(QC_THREADS, 1024 / QC_THREADS)
quant_table_kernel(const float4 *__restrict__ grad_rows, const int32_t *__restrict__ uniq_off, int T, int d4,
                   char4 *__restrict__ codes, float *__restrict__ grad_scales, const Heavy heavy)
{
    namespace cg = cooperative_groups;
    cg::cluster_group cluster = cg::this_cluster();
    __shared__ float s_warp[QC_THREADS / 32], s_block[QC_CLUSTER];
    const int rank = (int)cluster.block_rank(), blocks = (int)cluster.num_blocks(), t = (int)blockIdx.x / blocks;
    auto started = cluster.barrier_arrive();           // (shared memory of a block that has not begun is out of reach)
    dq_wait_before();
    const int64_t n = t < T ? table_vectors(uniq_off, t, d4) : 0;
    if (t < T && n <= heavy.limit) {                   // (the same in the whole cluster)
        const int64_t first = __ldg(uniq_off + t), stride = (int64_t)blocks * QC_THREADS;
        const float4 *g = grad_rows + first * d4;
        char4 *c = codes + first * d4;
        const int64_t i0 = (int64_t)rank * QC_THREADS + threadIdx.x;
        float4 x[QC_VEC];
        float m = 0.f;
#pragma unroll
        for (int k = 0; k < QC_VEC; ++k) {
            x[k] = make_float4(0.f, 0.f, 0.f, 0.f);
            if (i0 + k * stride < n) x[k] = __ldg(g + i0 + k * stride);
        }
#pragma unroll
        for (int k = 0; k < QC_VEC; ++k) m = fmaxf(m, abs_max4(x[k]));
        for (int64_t i = i0 + QC_VEC * stride; i < n; i += stride) m = fmaxf(m, abs_max4(__ldg(g + i)));
        const u32 wm = __reduce_max_sync(0xffffffffu, __float_as_uint(m));
        if (threadIdx.x % 32 == 0) s_warp[threadIdx.x / 32] = __uint_as_float(wm);
        __syncthreads();
        cluster.barrier_wait(std::move(started));
        if (threadIdx.x < (unsigned)blocks) {
            float b = 0.f;
#pragma unroll
            for (int w = 0; w < QC_THREADS / 32; ++w) b = fmaxf(b, s_warp[w]);
            cluster.map_shared_rank(s_block, threadIdx.x)[rank] = b;
        }
        cluster.sync();
        m = 0.f;
        for (int b = 0; b < blocks; ++b) m = fmaxf(m, s_block[b]);
        const float s = dq_scale_from_absmax(m, 8);
        if (rank == 0 && threadIdx.x == 0) grad_scales[t] = s;
        const QuantScale qs = dq_make_scale(s, 8);
#pragma unroll
        for (int k = 0; k < QC_VEC; ++k)
            if (i0 + k * stride < n) put_codes(c + i0 + k * stride, x[k], qs);
        for (int64_t i = i0 + QC_VEC * stride; i < n; i += stride) put_codes(c + i, __ldg(g + i), qs);
    } else {
        cluster.barrier_wait(std::move(started));
    }
    if (heavy.partial == nullptr || (int)blockIdx.x >= heavy.blocks || !any_heavy(uniq_off, T, d4, heavy.limit)) return;
    for (int h = 0; h < T; ++h) {
        const int64_t nh = table_vectors(uniq_off, h, d4), stride = (int64_t)heavy.blocks * QC_THREADS;
        if (nh <= heavy.limit) continue;
        const float4 *g = grad_rows + (int64_t)__ldg(uniq_off + h) * d4;
        float m = 0.f;
        for (int64_t i = (int64_t)blockIdx.x * QC_THREADS + threadIdx.x; i < nh; i += 4 * stride) {
            float4 x[4];
#pragma unroll
            for (int k = 0; k < 4; ++k) x[k] = __ldg(g + min(i + k * stride, nh - 1));
#pragma unroll
            for (int k = 0; k < 4; ++k) m = fmaxf(m, abs_max4(x[k]));
        }
        m = block_max<QC_THREADS>(m, s_warp);
        if (threadIdx.x == 0) heavy.partial[(size_t)h * heavy.blocks + blockIdx.x] = __float_as_uint(m);
    }
}

// the tables that the kernel above has left, by the whole grid
__global__ void __launch_bounds__(QH_THREADS)
quant_heavy_kernel(const float4 *__restrict__ grad_rows, const int32_t *__restrict__ uniq_off, int T, int d4,
                   char4 *__restrict__ codes, float *__restrict__ grad_scales, const Heavy heavy)
{
    dq_wait_before();
    __shared__ u32 s_max;
    if (!any_heavy(uniq_off, T, d4, heavy.limit)) return;
    for (int h = 0; h < T; ++h) {
        const int64_t nh = table_vectors(uniq_off, h, d4), stride = (int64_t)gridDim.x * QH_THREADS;
        if (nh <= heavy.limit) continue;
        __syncthreads();                               // (the maximum of the table before has been read)
        if (threadIdx.x == 0) s_max = 0u;
        __syncthreads();
        u32 m = 0u;
        for (int b = threadIdx.x; b < heavy.blocks; b += QH_THREADS) m = max(m, heavy.partial[(size_t)h * heavy.blocks + b]);
        m = __reduce_max_sync(0xffffffffu, m);
        if (threadIdx.x % 32 == 0 && m) atomicMax(&s_max, m);
        __syncthreads();
        const float s = dq_scale_from_absmax(__uint_as_float(s_max), 8);
        if (blockIdx.x == 0 && threadIdx.x == 0) grad_scales[h] = s;
        const QuantScale qs = dq_make_scale(s, 8);
        const int64_t first = (int64_t)__ldg(uniq_off + h) * d4;
        for (int64_t i = (int64_t)blockIdx.x * QH_THREADS + threadIdx.x; i < nh; i += 4 * stride) {
            float4 x[4];
#pragma unroll
            for (int k = 0; k < 4; ++k) x[k] = __ldg(grad_rows + first + min(i + k * stride, nh - 1));
#pragma unroll
            for (int k = 0; k < 4; ++k)
                if (i + k * stride < nh) put_codes(codes + first + i + k * stride, x[k], qs);
        }
    }
}

constexpr int64_t cluster_holds(int threads) { return (int64_t)QC_CLUSTER * threads * QC_VEC; }

// whether a batch of up to max_vectors goes through the kernels above.  With few tables up to what the cluster of one holds:
// beyond it three launches are faster for that one (three tables, one of 128 K vectors: 11.8 us here)
inline bool quant_by_table(const dqrm_ctx *ctx, int64_t max_vectors)
{
    return max_vectors <= (ctx->T >= 6 ? 2 * ctx->T * cluster_holds(1024) : cluster_holds(1024));
}

template <int QC_THREADS>
int launch_quant_table(dqrm_ctx *ctx, const float *grad_rows, const int32_t *uniq_off, int8_t *codes, float *grad_scales,
                       int64_t max_vectors, u32 *ws, size_t ws_bytes, cudaStream_t st, bool &taken)
{
    const int64_t per_table = (max_vectors + ctx->T - 1) / ctx->T;
    unsigned blocks = 1;
    while (blocks < (unsigned)QC_CLUSTER && per_table > (int64_t)blocks * QC_THREADS * 2) blocks *= 2;
    // more blocks where no table can then be beyond them: a second launch costs more than they do
    const int64_t held = (int64_t)QC_THREADS * QC_VEC;
    if (max_vectors <= 2 * QC_CLUSTER * held)
        while (max_vectors > 2 * blocks * held) blocks *= 2;
    Heavy heavy = {2 * blocks * held, nullptr, 0};
    unsigned clusters = (unsigned)ctx->T;
    if (max_vectors > heavy.limit) {
        heavy.blocks = 4 * ctx->num_sms;
        clusters = std::max(clusters, ((unsigned)ctx->num_sms + blocks - 1) / blocks);
        heavy.blocks = std::min(heavy.blocks, (int)(clusters * blocks));
        taken = ws_bytes >= sizeof(u32) * ctx->T * heavy.blocks;
        if (!taken) return DQRM_OK;
        heavy.partial = ws;
    } else {
        heavy.limit = INT64_MAX;       // (the bound may be wrong; the result must not be)
        taken = true;
    }
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(clusters * blocks);
    cfg.blockDim = dim3(QC_THREADS);
    cfg.stream = st;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = blocks; attr[0].val.clusterDim.y = 1; attr[0].val.clusterDim.z = 1;
    attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 2;
    const float4 *g = reinterpret_cast<const float4 *>(grad_rows);
    char4 *c = reinterpret_cast<char4 *>(codes);
    DQRM_CUDA_TRY(ctx, cudaLaunchKernelEx(&cfg, quant_table_kernel<QC_THREADS>, g, uniq_off, ctx->T, ctx->D / 4, c, grad_scales, heavy));
    dq_mark(ctx, st, DQ_K_QUANT_TABLE);
    if (heavy.partial == nullptr) return DQRM_OK;
    DQRM_CUDA_TRY(ctx, dq_launch(quant_heavy_kernel, dim3(ctx->num_sms), dim3(QH_THREADS), 0, st, g, uniq_off, ctx->T, ctx->D / 4, c,
                                 grad_scales, heavy));
    dq_mark(ctx, st, DQ_K_QUANT_HEAVY);
    return DQRM_OK;
}

// Blocks resident (with the rows' (min, max) stored the compiler would take registers that cost a block: 190 K rows of 64
// features 38.9 us with four, 48.7 without the bound; 108 K rows of 16 features 15.7 with three; quantise and update of
// rows of up to 32 features would take 85 registers and a block fewer: 131 K rows of 16 features 15.9 us with three, 16.6
// with two, eight pipelined steps around it 376 and 387.  The others are best with what a minimum of one gives: without any
// the update alone of 426 K rows of 128 features takes 88 us instead of 85)
constexpr int stream_blocks(int mode, int lpr, int ch, bool track)
{
    if (ch > 1) return 1;
    if (track) return lpr >= 16 ? 4 : 3;
    return mode == MODE_FUSED && lpr < 16 ? 3 : 1;
}

template <int MODE, int LPR, int CH, bool EXACT, bool TRACK = false>
__global__ void __launch_bounds__(QU_THREADS, stream_blocks(MODE, LPR, CH, TRACK))
row_stream_kernel(float *__restrict__ tables, const int64_t *__restrict__ row_off,
                  const int32_t *__restrict__ unique_rows, const int32_t *__restrict__ uniq_off,
                  const float *__restrict__ grad_rows, const u32 *__restrict__ absmax,
                  int8_t *__restrict__ codes, float *__restrict__ grad_scales, float lr, int T, int D_any,
                  int *__restrict__ status, float2 *__restrict__ row_summary)
{
    dq_wait_before();
    extern __shared__ __align__(16) unsigned char smem_raw[];
    row_stream_body<MODE, LPR, CH, EXACT, TRACK>(smem_raw, tables, row_off, unique_rows, uniq_off, grad_rows, absmax,
                                                 codes, grad_scales, lr, T, D_any, status, row_summary);
}

template <int MODE, int LPR, int CH>
int launch_rows(dqrm_ctx *ctx, float *tables, const int32_t *unique_rows, const int32_t *uniq_off,
                const float *grad_rows, const u32 *absmax, int8_t *codes, float *grad_scales, float lr,
                cudaStream_t st)
{
    const size_t smem = (size_t)(ctx->T + 1) * sizeof(int32_t) + (size_t)ctx->T * sizeof(float);
    int grid = ctx->num_sms * 8;      // U lives on the device: a fixed grid splits the rows evenly
    // with a row summary attached, every kernel that writes master rows keeps the rows' (min, max) current
    float2 *summary = MODE == MODE_QUANT ? nullptr : ctx->row_summary;
#define DQ_ROW_STREAM(EXACT, TRACK)                                                                               \
    DQRM_CUDA_TRY(ctx, (dq_launch(row_stream_kernel<MODE, LPR, CH, EXACT, TRACK>, dim3(grid), dim3(QU_THREADS), smem, st, \
        tables, ctx->d_row_off, unique_rows, uniq_off, grad_rows, absmax, codes, grad_scales, lr, ctx->T, ctx->D, \
        ctx->d_status, summary)))
    if (ctx->D == 4 * LPR * CH) {
        if (summary) DQ_ROW_STREAM(true, (MODE != MODE_QUANT));
        else DQ_ROW_STREAM(true, false);
    } else {
        if (summary) DQ_ROW_STREAM(false, (MODE != MODE_QUANT));
        else DQ_ROW_STREAM(false, false);
    }
#undef DQ_ROW_STREAM
    dq_mark(ctx, st, MODE == MODE_QUANT ? DQ_K_QUANT : (MODE == MODE_UPDATE ? DQ_K_UPDATE : DQ_K_QUANT_UPDATE));
    return DQRM_OK;
}

template <int MODE>
int dispatch(dqrm_ctx *ctx, float *tables, const int32_t *unique_rows, const int32_t *uniq_off,
             const float *grad_rows, const u32 *absmax, int8_t *codes, float *grad_scales, float lr,
             cudaStream_t st)
{
    const int d4 = ctx->D / 4;
#define DQ_ROWS(LPR, CH) \
    return launch_rows<MODE, LPR, CH>(ctx, tables, unique_rows, uniq_off, grad_rows, absmax, codes, grad_scales, lr, st)
    if (d4 <= 1) DQ_ROWS(1, 1);
    if (d4 <= 2) DQ_ROWS(2, 1);
    if (d4 <= 4) DQ_ROWS(4, 1);
    if (d4 <= 8) DQ_ROWS(8, 1);
    if (d4 <= 16) DQ_ROWS(16, 1);
    if (d4 <= 32) DQ_ROWS(32, 1);
    if (d4 <= 64) DQ_ROWS(32, 2);
    if (d4 <= 128) DQ_ROWS(32, 4);
    DQ_ROWS(32, 8);
#undef DQ_ROWS
}

}  // namespace

size_t dq_quant_ws_bytes(const dqrm_ctx *ctx) { return align_up(sizeof(u32) * ctx->T, 256); }

int dq_launch_grad_quant(dqrm_ctx *ctx, const float *grad_rows, const int32_t *uniq_off, int8_t *codes,
                         float *grad_scales, int64_t max_values, void *ws, size_t ws_bytes, cudaStream_t st)
{
    if (ws_bytes < dq_quant_ws_bytes(ctx)) return DQRM_ERR_WORKSPACE;
    if (quant_by_table(ctx, max_values / 4)) {
        const int64_t most = max_values / 4, per_table = (most + ctx->T - 1) / ctx->T;
        // threads a block: as many as the tables' mean needs; more where one table may then hold everything without being
        // beyond its cluster, and the clusters still run at once (53 K vectors over 26 tables: 4.1 us with 512
        // threads, 4.8 with 256 and the second launch)
        int threads = per_table <= cluster_holds(256) ? 256
                      : per_table > cluster_holds(512) && ctx->T * QC_CLUSTER < ctx->num_sms ? 1024 : 512;
        for (int more = threads; more <= 1024 && ctx->T * QC_CLUSTER * more <= ctx->num_sms * 1024; more *= 2)
            if (most <= 2 * cluster_holds(more)) { threads = more; break; }
        u32 *w = reinterpret_cast<u32 *>(ws);
        bool taken = false;            // (not with a workspace that has no room for the partial maxima)
        const int rc = threads == 256    ? launch_quant_table<256>(ctx, grad_rows, uniq_off, codes, grad_scales, most, w, ws_bytes, st, taken)
                       : threads == 512 ? launch_quant_table<512>(ctx, grad_rows, uniq_off, codes, grad_scales, most, w, ws_bytes, st, taken)
                                        : launch_quant_table<1024>(ctx, grad_rows, uniq_off, codes, grad_scales, most, w, ws_bytes, st, taken);
        if (rc != DQRM_OK || taken) return rc;
    }
    u32 *absmax = reinterpret_cast<u32 *>(ws);
    const int rc = launch_absmax(ctx, grad_rows, uniq_off, absmax, st);
    if (rc != DQRM_OK) return rc;
    return dispatch<MODE_QUANT>(ctx, nullptr, nullptr, uniq_off, grad_rows, absmax, codes, grad_scales, 0.f, st);
}

// per-table max |grad_rows| as floats (the bit pattern of a non-negative float orders like the uint the kernel maximises)
int dq_launch_grad_absmax(dqrm_ctx *ctx, const float *grad_rows, const int32_t *uniq_off, float *absmax,
                          cudaStream_t st)
{
    return launch_absmax(ctx, grad_rows, uniq_off, reinterpret_cast<u32 *>(absmax), st);
}

// quantise with scales derived from abs-max values that were unified across ranks
int dq_launch_grad_quant_unified(dqrm_ctx *ctx, const float *grad_rows, const int32_t *uniq_off,
                                 const float *unified_absmax, int8_t *codes, float *grad_scales, cudaStream_t st)
{
    return dispatch<MODE_QUANT>(ctx, nullptr, nullptr, uniq_off, grad_rows, reinterpret_cast<const u32 *>(unified_absmax),
                                codes, grad_scales, 0.f, st);
}

int dq_launch_row_update(dqrm_ctx *ctx, float *tables, const int32_t *unique_rows, const int32_t *uniq_off,
                         const int8_t *codes, const float *grad_scales, float lr, cudaStream_t st)
{
    return dispatch<MODE_UPDATE>(ctx, tables, unique_rows, uniq_off, nullptr, nullptr, const_cast<int8_t *>(codes),
                                 const_cast<float *>(grad_scales), lr, st);
}

int dq_launch_quant_update(dqrm_ctx *ctx, float *tables, const int32_t *unique_rows, const int32_t *uniq_off,
                           const float *grad_rows, const u32 *absmax_bits, int8_t *codes, float *grad_scales,
                           float lr, cudaStream_t st)
{
    return dispatch<MODE_FUSED>(ctx, tables, unique_rows, uniq_off, grad_rows, absmax_bits, codes, grad_scales, lr, st);
}

// ---------------------------------------------------------------------------------
// Allocation-free variant of the INT8 gradient quantiser.
//
// Some users of this library may not allocate device memory at the point where they
// quantise gradients: a plug-in that runs inside another framework's step after that
// framework has reserved the whole HBM for its own pool (a cudaMalloc there fails or
// fragments the pool), or a latency-critical loop in which the implicit device-wide
// synchronisation of cudaMalloc/cudaFree would stall every other stream.  Such callers
// have no way to provide the per-table abs-max scratch word that dqrm_grad_quant_int8
// takes from its workspace, and they cannot create a context either (dqrm_create
// allocates).  For them the scratch lives in the array below, which is part of the
// loaded module: every GPU that loads the library holds these 4 KB until the process
// exits.  The name `g_static_absmax` is only a handle in host code; the device address
// is looked up once per device with cudaGetSymbolAddress and cached.
// ---------------------------------------------------------------------------------
static __device__ __align__(256) u32 g_static_absmax[DQRM_STATIC_MAX_TABLES];

namespace {

constexpr int STATIC_MAX_DEVICES = 64;
struct StaticSlot {
    u32 *absmax = nullptr;   // device address of g_static_absmax on this device
    int num_sms = 0;
    bool ready = false;
};
StaticSlot g_static_slots[STATIC_MAX_DEVICES];
std::mutex g_static_mutex;        // host threads may make a device's first call at the same time

}  // namespace

extern "C" int dqrm_grad_quant_int8_static(int T, int D, const float *grad_rows, const int32_t *uniq_off,
                                           int8_t *codes, float *grad_scales, void *stream)
{
    if (T <= 0 || D < 4 || D > 1024 || (D % 4) != 0 || !grad_rows || !uniq_off || !codes || !grad_scales ||
        !dq_aligned(grad_rows, sizeof(float4)) || !dq_aligned(codes, sizeof(char4)))
        return DQRM_ERR_INVALID_ARG;
    if (T > DQRM_STATIC_MAX_TABLES) return DQRM_ERR_STATIC_LIMIT;
    int dev = -1;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= STATIC_MAX_DEVICES) {
        (void)cudaGetLastError();
        return DQRM_ERR_CUDA;
    }
    StaticSlot slot;
    {
        std::lock_guard<std::mutex> lock(g_static_mutex);
        StaticSlot &shared = g_static_slots[dev];
        if (!shared.ready) {
            // first call on this device: resolve the array's device address (with this device current)
            u32 *p = nullptr;
            if (cudaGetSymbolAddress(reinterpret_cast<void **>(&p), g_static_absmax) != cudaSuccess || !p ||
                cudaDeviceGetAttribute(&shared.num_sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) {
                (void)cudaGetLastError();
                return DQRM_ERR_CUDA;
            }
            shared.absmax = p;
            shared.ready = true;
        }
        slot = shared;
    }
    // a stack context carries the shape to the shared launch helpers; nothing is allocated
    dqrm_ctx tmp;
    tmp.T = T;
    tmp.D = D;
    tmp.device = dev;
    tmp.num_sms = slot.num_sms;
    cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
    // the array keeps the previous call's maxima: the entries this call uses are cleared first
    const int rc = launch_absmax(&tmp, grad_rows, uniq_off, slot.absmax, st);
    if (rc != DQRM_OK) return rc;
    return dispatch<MODE_QUANT>(&tmp, nullptr, nullptr, uniq_off, grad_rows, slot.absmax, codes, grad_scales, 0.f, st);
}

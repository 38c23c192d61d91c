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
    extern __shared__ unsigned char smem_raw[];
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
constexpr int QC_VEC = 8;             // vectors of four that a thread holds
constexpr int QC_CLUSTER = 8;

template <int QC_THREADS>
__global__ void __launch_bounds__(QC_THREADS, 1024 / QC_THREADS)
quant_table_kernel(const float4 *__restrict__ grad_rows, const int32_t *__restrict__ uniq_off, int d4,
                   char4 *__restrict__ codes, float *__restrict__ grad_scales)
{
    namespace cg = cooperative_groups;
    cg::cluster_group cluster = cg::this_cluster();
    __shared__ float s_warp[QC_THREADS / 32], s_block[QC_CLUSTER];
    const int rank = (int)cluster.block_rank(), blocks = (int)cluster.num_blocks(), t = (int)blockIdx.x / blocks;
    auto started = cluster.barrier_arrive();           // (shared memory of a block that has not begun is out of reach)
    dq_wait_before();
    const int64_t first = __ldg(uniq_off + t), rows = max((int64_t)__ldg(uniq_off + t + 1) - first, (int64_t)0);
    const int64_t n = rows * d4, stride = (int64_t)blocks * QC_THREADS;
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
    for (int k = 0; k < QC_VEC; ++k)
        m = fmaxf(m, fmaxf(fmaxf(fabsf(x[k].x), fabsf(x[k].y)), fmaxf(fabsf(x[k].z), fabsf(x[k].w))));
    for (int64_t i = i0 + QC_VEC * stride; i < n; i += stride) {
        const float4 y = __ldg(g + i);
        m = fmaxf(m, fmaxf(fmaxf(fabsf(y.x), fabsf(y.y)), fmaxf(fabsf(y.z), fabsf(y.w))));
    }
    const u32 wm = __reduce_max_sync(0xffffffffu, __float_as_uint(m));      // (non-negative floats order as their bits)
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
    auto put = [&](int64_t i, const float4 &v) {
        float4 q, unused;
        dq_fq4(v, qs, q, unused);
        __stcs(c + i, make_char4((signed char)(int)q.x, (signed char)(int)q.y, (signed char)(int)q.z, (signed char)(int)q.w));
    };
#pragma unroll
    for (int k = 0; k < QC_VEC; ++k)
        if (i0 + k * stride < n) put(i0 + k * stride, x[k]);
    for (int64_t i = i0 + QC_VEC * stride; i < n; i += stride) put(i, __ldg(g + i));
}

// whether a batch of up to max_vectors goes through the kernel above
inline bool quant_by_table(const dqrm_ctx *ctx, int64_t max_vectors)
{
    const int64_t held = (int64_t)ctx->T * QC_CLUSTER * 1024 * QC_VEC;
    return max_vectors <= (ctx->T >= 6 ? 2 * held : held);
}

template <int QC_THREADS>
int launch_quant_table(dqrm_ctx *ctx, const float *grad_rows, const int32_t *uniq_off, int8_t *codes, float *grad_scales,
                       int64_t per_table, cudaStream_t st)
{
    unsigned blocks = 1;
    while (blocks < (unsigned)QC_CLUSTER && per_table > (int64_t)blocks * QC_THREADS * 2) blocks *= 2;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)ctx->T * blocks);
    cfg.blockDim = dim3(QC_THREADS);
    cfg.stream = st;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = blocks; attr[0].val.clusterDim.y = 1; attr[0].val.clusterDim.z = 1;
    attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 2;
    DQRM_CUDA_TRY(ctx, cudaLaunchKernelEx(&cfg, quant_table_kernel<QC_THREADS>, reinterpret_cast<const float4 *>(grad_rows), uniq_off,
                                          ctx->D / 4, reinterpret_cast<char4 *>(codes), grad_scales));
    dq_mark(ctx, st, DQ_K_QUANT);
    return DQRM_OK;
}

// (with the rows' (min, max) stored the compiler would take registers that cost a resident block: 190 K rows of 64 features
// 38.9 us with four blocks, 48.7 without the bound; 108 K rows of 16 features 15.7 with three)
template <int MODE, int LPR, int CH, bool EXACT, bool TRACK = false>
__global__ void __launch_bounds__(QU_THREADS, TRACK && CH == 1 ? (LPR >= 16 ? 4 : 3) : 1)
row_stream_kernel(float *__restrict__ tables, const int64_t *__restrict__ row_off,
                  const int32_t *__restrict__ unique_rows, const int32_t *__restrict__ uniq_off,
                  const float *__restrict__ grad_rows, const u32 *__restrict__ absmax,
                  int8_t *__restrict__ codes, float *__restrict__ grad_scales, float lr, int T, int D_any,
                  int *__restrict__ status, float2 *__restrict__ row_summary)
{
    dq_wait_before();
    extern __shared__ unsigned char smem_raw[];
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
        const int64_t per_table = (max_values / 4 + ctx->T - 1) / ctx->T;
        if (per_table <= (int64_t)QC_CLUSTER * 256 * QC_VEC)
            return launch_quant_table<256>(ctx, grad_rows, uniq_off, codes, grad_scales, per_table, st);
        if (per_table > (int64_t)QC_CLUSTER * 512 * QC_VEC && ctx->T * QC_CLUSTER < ctx->num_sms)
            return launch_quant_table<1024>(ctx, grad_rows, uniq_off, codes, grad_scales, per_table, st);
        return launch_quant_table<512>(ctx, grad_rows, uniq_off, codes, grad_scales, per_table, st);
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
    if (T <= 0 || D < 4 || D > 1024 || (D % 4) != 0 || !grad_rows || !uniq_off || !codes || !grad_scales)
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

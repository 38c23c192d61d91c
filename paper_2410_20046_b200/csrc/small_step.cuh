// Everything of a training step behind the forward for a small batch, in one launch: one block per table sorts the
// table's lookups (the network of small_sort.cuh), sums the gradient rows of each distinct row, finds the abs-max,
// quantises and updates the master rows.  Sort, sum and update by themselves are three launches of 3 to 5 us each that
// are bound by their own latency.
//
// A table's rows stand behind those of the tables before it in unique_rows and grad_rows, so a block has to know how
// many distinct rows these have.  It counts them itself, in a hash table over the lookups in front of its own (at
// most MAX_LOOKUPS of them): cheaper than a launch more, and no block waits for another.
//
// The kernel begins while the forward runs: up to the update it touches neither tables nor pooled output, and only
// there waits for the forward to end.  What it reads before that (offsets, indices, upstream gradient) and writes
// (unique_rows, grad_rows, the workspace) may belong to kernels before the forward: it is launched behind a forward that
// waits for them before it lets this kernel begin (before_and_next in fwd.cu), and must not be launched behind anything else.
//
// Sums are FP64, in order of the entries inside a lane group's share and then over the shares: results are
// reproducible.
//
// Bound by its chain of latencies (two loads, the network, a gather, a row).  Measured on B200 (graph replay): a step of 4
// tables of 128 lookups of 16 features 8.1 us (14.6 in four launches), 26 tables of 128 12.4 (13.9 before the counted lookups
// were all asked for at once; 18.5 in four).
#pragma once
#include "small_sort.cuh"

namespace sstep {

using ssort::u64;

constexpr int THREADS = 512;
constexpr int WARPS = THREADS / 32;
constexpr int MAX_LOOKUPS = 4096;
constexpr int HASH_BITS = 14;                      // at most a quarter full (half: 15.1 instead of 13.9 us at 26 tables of 128)
constexpr int WORDS = MAX_LOOKUPS / 32;

struct Args {
    csort::Args s;                  // (of its lists only gp is used)
    const float *grad_out;
    float *tables, *grad_rows;
    int32_t *unique_rows, *uniq_off;
    int8_t *codes;
    float *grad_scales;
    float lr;
    int D, lpr_log;                 // lanes per row, four features a lane: a power of two from D / 4 on
};

// network | hash table, digit counts or shares' sums, whichever is in use | tables' boundaries
constexpr size_t MID_WORDS = (size_t)1 << HASH_BITS;
static_assert(MID_WORDS >= (size_t)WARPS * csort::BINS && MID_WORDS >= (size_t)THREADS * 8, "");
inline size_t smem_bytes(int T) { return (size_t)THREADS * 2 * sizeof(u64) + (MID_WORDS + 3 * T + 1) * sizeof(u32); }

// STEP: the whole step behind the forward; otherwise the backward alone (unique_rows, uniq_off, grad_rows), an ordinary kernel that
// may be launched behind anything
template <bool STEP>
__global__ void __launch_bounds__(THREADS)
small_step_kernel(const __grid_constant__ Args x)
{
    if (!STEP) dq_wait_before();
    extern __shared__ __align__(16) u64 s_net[];                 // [2][THREADS]
    u32 *s_mid = reinterpret_cast<u32 *>(s_net + 2 * THREADS);
    u32 *s_tb = s_mid + MID_WORDS;                 // [T+1]
    u32 *s_first = s_tb + x.s.T + 1, *s_rows = s_first + x.s.T;        // [T] arena row where a table begins, and its rows
    __shared__ u32 s_head[WORDS], s_pre[WORDS + 1], s_base, s_max;
    const csort::Args &a = x.s;
    const int t = blockIdx.x, T = a.T, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;

    // ---- the tables' boundaries
    static_assert(THREADS > 148, "a thread has one table's boundary");
    u32 bound = 0, first = 0, rows = 0;
    if (tid <= T) bound = (u32)__ldg(a.offsets + (int64_t)tid * a.B);
    if (tid < T) { first = (u32)__ldg(a.row_off + tid); rows = (u32)__ldg(a.row_off + tid + 1) - first; }
    for (int i = tid; i < (1 << HASH_BITS) / 4; i += THREADS)
        reinterpret_cast<uint4 *>(s_mid)[i] = make_uint4(0xffffffffu, 0xffffffffu, 0xffffffffu, 0xffffffffu);
    if (tid <= T) s_tb[tid] = bound;
    if (tid < T) { s_first[tid] = first; s_rows[tid] = rows; }
    if (tid == 0) s_base = s_max = 0u;
    __syncthreads();
    bool broken = false;
    for (int i = tid; i <= T; i += THREADS)
        broken |= (int64_t)s_tb[i] > a.L || (i == 0 ? s_tb[0] != 0u : s_tb[i] < s_tb[i - 1]) || (i == T && (int64_t)s_tb[i] != a.L);
    if (__syncthreads_or(broken)) {                // nothing is summed, no row is updated
        if (STEP) dq_wait_before();
        if (tid == 0) {
            dq_report(a.status, DQRM_ERR_INDEX_RANGE);
            if (STEP) x.grad_scales[t] = dq_scale_from_absmax(0.f, 8);
            x.uniq_off[t] = 0;
            if (t == T - 1) x.uniq_off[T] = 0;
        }
        return;
    }
    const int tb0 = (int)s_tb[t], n = (int)s_tb[t + 1] - tb0;
    const int64_t r0 = s_first[t], nrows = s_rows[t];
    bool bad = false;

    // ---- distinct rows of the tables before this one
    {
        u32 fresh = 0;
        constexpr int EACH = MAX_LOOKUPS / THREADS;
        int32_t idx[EACH];                         // (all of a thread's at once: in turn they were 8.4 K clocks for 3.2 K lookups)
#pragma unroll
        for (int k = 0; k < EACH; ++k) idx[k] = k * THREADS + tid < tb0 ? __ldg(a.indices + k * THREADS + tid) : 0;
#pragma unroll 1
        for (int k = 0; k * THREADS < tb0; ++k) {
            const int p = k * THREADS + tid;
            if (p >= tb0) break;
            int32_t row = idx[0];
#pragma unroll
            for (int j = 1; j < EACH; ++j) if (k == j) row = idx[j];
            int lo = 0, hi = t;
            while (hi - lo > 1) {
                const int mid = (lo + hi) >> 1;
                if ((int)s_tb[mid] <= p) lo = mid; else hi = mid;
            }
            const u32 key = s_first[lo] + min((u32)max(row, 0), s_rows[lo] - 1u);
            u32 h = (key * 2654435761u) >> (32 - HASH_BITS);
            for (int tries = 0; tries < (1 << HASH_BITS); ++tries) {
                const u32 seen = reinterpret_cast<volatile u32 *>(s_mid)[h];
                if (seen == key) break;
                if (seen == 0xffffffffu) {
                    const u32 was = atomicCAS(s_mid + h, 0xffffffffu, key);
                    if (was == key) break;
                    if (was == 0xffffffffu) { ++fresh; break; }
                }
                h = (h + 1) & ((1u << HASH_BITS) - 1u);
            }
        }
        fresh = __reduce_add_sync(0xffffffffu, fresh);
        if (lane == 0 && fresh) atomicAdd(&s_base, fresh);
    }
    if (n != a.B)                                  // (otherwise every lookup looks at its own bag's offsets)
        for (int i = tid; i < a.B; i += THREADS) bad |= __ldg(a.offsets + (int64_t)t * a.B + i) > __ldg(a.offsets + (int64_t)t * a.B + i + 1);
    __syncthreads();
    const u32 base = s_base;

    // ---- sorted (row, row of grad_out); where the segments begin
    const uint2 *mem = nullptr;                    // (an uneven batch: a table that does not fit the block)
    if (n > THREADS) mem = ssort::sort_in_memory<THREADS>(a, t, tb0, n, nrows, s_mid);
    else if (n > 0) ssort::sort_in_block<THREADS>(a, t, tb0, n, nrows, s_net, bad);
    if (bad) dq_report(a.status, DQRM_ERR_INDEX_RANGE);
    auto row_at = [&](int i) { return mem ? mem[i].x : (u32)(s_net[i] >> 32); };
    const int words = (n + 31) / 32;
    for (int c0 = 0; c0 < n; c0 += THREADS) {
        const int i = c0 + tid;
        const u32 row = i < n ? row_at(i) : 0u;
        const bool head = i < n && (i == 0 || row_at(i - 1) != row);
        if (STEP && head)                          // the update needs the row soon
            for (int o = 0; o < x.D; o += 32) dq_prefetch_l2(x.tables + (r0 + row) * x.D + o);
        const u32 m = __ballot_sync(0xffffffffu, head);
        if (lane == 0 && c0 + warp * 32 < n) s_head[(c0 >> 5) + warp] = m;
    }
    __syncthreads();
    if (warp == 0) {
        u32 run = 0;
        for (int w0 = 0; w0 < words; w0 += 32) {
            const u32 v = w0 + lane < words ? __popc(s_head[w0 + lane]) : 0u;
            u32 incl = v;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const u32 y = __shfl_up_sync(0xffffffffu, incl, o);
                if (lane >= o) incl += y;
            }
            if (w0 + lane < words) s_pre[w0 + lane] = run + incl - v;
            run += __shfl_sync(0xffffffffu, incl, 31);
        }
        if (lane == 0) s_pre[words] = run;
    }
    __syncthreads();
    const int U = (int)s_pre[words];
    auto is_head = [&](int i) { return (s_head[i >> 5] >> (i & 31)) & 1u; };
    auto segment = [&](int i) { return (int)(s_pre[i >> 5] + __popc(s_head[i >> 5] & (0xffffffffu >> (31 - (i & 31))))) - 1; };
    for (int i = tid; i < n; i += THREADS)
        if (is_head(i)) x.unique_rows[base + segment(i)] = (int32_t)row_at(i);

    // ---- sums: every lane group takes a share of the entries; a run that goes on into the next share is finished by
    //      the group in whose share it begins
    const int lpr = 1 << x.lpr_log, col = tid & (lpr - 1), grp = tid >> x.lpr_log, groups = THREADS >> x.lpr_log;
    const bool act = 4 * col < x.D;
    double *s_sum = reinterpret_cast<double *>(s_mid);           // [THREADS][4] sum of the run that comes into the share
    float4 *out_rows = reinterpret_cast<float4 *>(x.grad_rows) + (size_t)base * (x.D >> 2) + col;
    const int per = max(1, (n + groups - 1) / groups), b0 = min(n, grp * per), b1 = min(n, b0 + per);
    const int d4 = x.D >> 2;
    float mx = 0.f;
    double acc[4] = {0., 0., 0., 0.};
    auto put = [&](int seg) {
        const float4 r = make_float4((float)acc[0], (float)acc[1], (float)acc[2], (float)acc[3]);
        mx = fmaxf(mx, fmaxf(fmaxf(fabsf(r.x), fabsf(r.y)), fmaxf(fabsf(r.z), fabsf(r.w))));
        if (act) out_rows[(size_t)seg * d4] = r;
    };
    bool came = false, leaves = false;
    int seg = 0;
    if (b0 < b1) {
        seg = segment(b0);
        came = !is_head(b0);
        for (int i0 = b0; i0 < b1; i0 += 4) {
            float4 v[4];
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                v[k] = make_float4(0.f, 0.f, 0.f, 0.f);
                if (i0 + k < b1 && act) {
                    const u32 from = mem ? mem[i0 + k].y : (u32)s_net[i0 + k];
                    v[k] = __ldg(reinterpret_cast<const float4 *>(x.grad_out) + (size_t)from * d4 + col);
                }
            }
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                const int i = i0 + k;
                if (i < b1) {
                    if (i > b0 && is_head(i)) {
                        if (came) {
#pragma unroll
                            for (int j = 0; j < 4; ++j) s_sum[4 * tid + j] = acc[j];
                        } else put(seg);
                        came = false;
                        ++seg;
#pragma unroll
                        for (int j = 0; j < 4; ++j) acc[j] = 0.;
                    }
                    acc[0] += (double)v[k].x; acc[1] += (double)v[k].y; acc[2] += (double)v[k].z; acc[3] += (double)v[k].w;
                }
            }
        }
        leaves = b1 < n && !is_head(b1);
        if (came) {
#pragma unroll
            for (int j = 0; j < 4; ++j) s_sum[4 * tid + j] = acc[j];
        } else if (!leaves) put(seg);
    }
    __syncthreads();
    if (b0 < b1 && leaves && !came) {
        int w = b1 >> 5;
        u32 m = s_head[w] & (0xffffffffu << (b1 & 31));
        while (m == 0u && ++w < words) m = s_head[w];
        const int end = m ? w * 32 + __ffs(m) - 1 : n;
        for (int g = grp + 1; g * per < end; ++g)
#pragma unroll
            for (int j = 0; j < 4; ++j) acc[j] += s_sum[4 * ((g << x.lpr_log) + col) + j];
        put(seg);
    }
    if (!STEP) {
        if (tid == 0) {
            x.uniq_off[t] = (int32_t)base;
            if (t == T - 1) x.uniq_off[T] = (int32_t)base + U;
        }
        return;
    }
    const u32 wm = __reduce_max_sync(0xffffffffu, __float_as_uint(mx));
    if (lane == 0 && wm) atomicMax(&s_max, wm);
    __syncthreads();                               // (also: the block's writes to grad_rows and unique_rows are seen by it)
    const float s = dq_scale_from_absmax(__uint_as_float(s_max), 8);
    const QuantScale qs = dq_make_scale(s, 8);

    // ---- quantise and update
    dq_wait_before();
    if (tid == 0) {
        x.grad_scales[t] = s;
        x.uniq_off[t] = (int32_t)base;
        if (t == T - 1) x.uniq_off[T] = (int32_t)base + U;
    }
    if (!act) return;
    for (int u0 = grp; u0 < U; u0 += 4 * groups) {
        float4 g[4], w[4];
        float4 *row[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const int u = u0 + k * groups;
            if (u < U) {
                row[k] = reinterpret_cast<float4 *>(x.tables) + (r0 + x.unique_rows[base + u]) * d4 + col;
                g[k] = out_rows[(size_t)u * d4];
                w[k] = *row[k];
            }
        }
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const int u = u0 + k * groups;
            if (u < U) {
                float4 q, unused;
                dq_fq4(g[k], qs, q, unused);
                reinterpret_cast<char4 *>(x.codes)[(size_t)(base + u) * d4 + col] =
                    make_char4((signed char)(int)q.x, (signed char)(int)q.y, (signed char)(int)q.z, (signed char)(int)q.w);
                w[k].x = __fsub_rn(w[k].x, __fmul_rn(x.lr, __fmul_rn(q.x, s)));
                w[k].y = __fsub_rn(w[k].y, __fmul_rn(x.lr, __fmul_rn(q.y, s)));
                w[k].z = __fsub_rn(w[k].z, __fmul_rn(x.lr, __fmul_rn(q.z, s)));
                w[k].w = __fsub_rn(w[k].w, __fmul_rn(x.lr, __fmul_rn(q.w, s)));
                *row[k] = w[k];
            }
        }
    }
}

}  // namespace sstep

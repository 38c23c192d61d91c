// The C ABI over a stand-in for the CUDA runtime that counts launches: which pointers a call takes, by their alignment, and what its
// grids are.  Nothing runs on a device and no pointer is followed.  One scenario per run, named by argv[1]; 0 when what it asserts holds.
#include <cstdint>
#include <cstdio>
#include <cstring>
#include "dqrm.h"
#include "launch_host.h"

namespace {

constexpr int T = 4;
alignas(256) char workspace[64 << 20];
const uintptr_t BASE = 1 << 20;                    // (of pointers that are only looked at)
template <typename P> P at(int by) { return reinterpret_cast<P>(BASE + by); }
float *f(int by) { return at<float *>(by); }
int32_t *i32() { return at<int32_t *>(0); }
int8_t *c(int by) { return at<int8_t *>(by); }
uint8_t *u8(int by) { return at<uint8_t *>(by); }

struct Ctx {
    dqrm_ctx *h = nullptr;
    explicit Ctx(int D, int tables = T)
    {
        int64_t off[16];
        for (int t = 0; t <= tables; ++t) off[t] = 100 * t;
        if (dqrm_create(&h, tables, D, off) != DQRM_OK) h = nullptr;
    }
    ~Ctx() { dqrm_destroy(h); }
};

int failed = 0;
// a call that is taken launches something, one that is refused nothing
void want(bool taken, int rc, const char *what, int D, int by)
{
    const bool launched = fake::launches > 0;
    fake::launches = 0;
    if (rc == (taken ? DQRM_OK : DQRM_ERR_INVALID_ARG) && launched == taken) return;
    std::printf("%s, D = %d, pointer %d bytes off: status %d, %s\n", what, D, by, rc, launched ? "launched" : "nothing launched");
    failed = 1;
}
#define WANT(TAKEN, CALL) want(TAKEN, CALL, #CALL, D, by)

int bwd(dqrm_ctx *h, int go, int gr, int B = 500) { return dqrm_emb_bwd(h, f(go), i32(), i32(), i32(), i32(), f(gr), B, (int64_t)T * B, workspace, sizeof(workspace), nullptr); }
int fwd(dqrm_ctx *h, int tb, int out, int codes, int bag)
{
    return dqrm_emb_fwd(h, f(tb), i32(), i32(), f(0), i32(), f(out), codes < 0 ? nullptr : c(codes), 64, (int64_t)T * 64 * bag, nullptr);
}
int step(dqrm_ctx *h, int tb, int go, int out, int gr, int codes, int B)
{
    return dqrm_train_step(h, f(tb), i32(), i32(), f(go), f(0), i32(), f(out), i32(), i32(), f(gr), c(codes), f(0), 0.1f, B, (int64_t)T * B,
                           workspace, sizeof(workspace), nullptr);
}
int sorted_step(dqrm_ctx *h, int tb, int go, int out, int gr, int codes)
{
    const int B = 500;
    if (dqrm_sort_batch(h, i32(), i32(), i32(), i32(), B, T * B, workspace, sizeof(workspace), nullptr) != DQRM_OK) return -100;
    fake::launches = 0;
    return dqrm_train_step_sorted(h, f(tb), i32(), i32(), f(go), f(0), i32(), f(out), i32(), i32(), f(gr), c(codes), f(0), 0.1f, B, T * B,
                                  workspace, sizeof(workspace), nullptr);
}

// the summed gradient takes what a row's lanes take
int sum()
{
    for (const int D : {4, 8, 12, 32, 36, 48, 52, 64, 68, 128, 1024}) {
        Ctx x(D);
        const int need = D == 4 ? 4 : D <= 64 ? 8 : 16;
        for (const int by : {0, 4, 8, 16}) {
            WANT(by % need == 0, bwd(x.h, by, 0));
            WANT(by % need == 0, bwd(x.h, 0, by));
            WANT(by % need == 0, step(x.h, 0, by, 0, 0, 0, 4000));
            WANT(by % need == 0, step(x.h, 0, by, 0, 0, 0, 16));           // (small enough for the one-launch step)
            WANT(by % need == 0, sorted_step(x.h, 0, by, 0, 0, 0));
            for (const int B : {16, 4000}) {
                WANT(by % 16 == 0, step(x.h, by, 0, 0, 0, 0, B));
                WANT(by % 16 == 0, step(x.h, 0, 0, by, 0, 0, B));
                WANT(by % 16 == 0, step(x.h, 0, 0, 0, by, 0, B));
            }
            WANT(by % 16 == 0, sorted_step(x.h, by, 0, 0, 0, 0));
            WANT(by % 16 == 0, sorted_step(x.h, 0, 0, by, 0, 0));
            WANT(by % 16 == 0, sorted_step(x.h, 0, 0, 0, by, 0));
        }
        for (const int by : {0, 2, 4}) {
            WANT(by % 4 == 0, step(x.h, 0, 0, 0, 0, by, 16));
            WANT(by % 4 == 0, sorted_step(x.h, 0, 0, 0, 0, by));
        }
    }
    return failed;
}

int forward()
{
    for (const int D : {4, 36, 64, 128}) {
        Ctx x(D);
        for (const int by : {0, 4, 8, 16})
            for (const int bag : {1, 3, 18}) {
                const int need = bag == 18 && (D == 36 || D == 64) ? 8 : 16;
                WANT(by % need == 0, fwd(x.h, by, 0, -1, bag));
                WANT(by % need == 0, fwd(x.h, 0, by, -1, bag));
                WANT(by % 16 == 0, fwd(x.h, 0, by, 0, bag));
            }
        for (const int by : {0, 1, 4}) WANT(by % 4 == 0, fwd(x.h, 0, 0, by, 1));
        for (const int bits : {2, 4, 8})
            for (const int by : {0, 1, 2, 4, 8}) {
                WANT(by % (bits / 2) == 0, dqrm_pack_tables(x.h, f(0), f(0), bits, u8(by), nullptr));
                WANT(by % (bits / 2) == 0, dqrm_emb_fwd_codes(x.h, f(0), i32(), i32(), f(0), bits, u8(by), 64, T * 64, nullptr));
                WANT(by % (bits / 2) == 0, dqrm_decode_payload(x.h, u8(by), f(0), bits, f(0), 64, T, T, 0, nullptr));
                WANT(by % (bits / 2) == 0, dqrm_packed_fwd(x.h, u8(by), i32(), i32(), f(0), bits, f(0), 64, T * 64, nullptr));
                const int pooled = D % 8 == 0 ? bits : bits / 2;
                WANT(by % pooled == 0, dqrm_packed_fwd(x.h, u8(by), i32(), i32(), f(0), bits, f(0), 64, T * 64 * 2, nullptr));
            }
        for (const int by : {0, 8, 16}) {
            WANT(by % 16 == 0, dqrm_pack_tables(x.h, f(by), f(0), 4, u8(0), nullptr));
            WANT(by % 16 == 0, dqrm_emb_fwd_codes(x.h, f(by), i32(), i32(), f(0), 4, u8(0), 64, T * 64, nullptr));
            WANT(by % 16 == 0, dqrm_decode_payload(x.h, u8(0), f(0), 4, f(by), 64, T, T, 0, nullptr));
            WANT(by % 16 == 0, dqrm_packed_fwd(x.h, u8(0), i32(), i32(), f(0), 4, f(by), 64, T * 64, nullptr));
        }
    }
    return failed;
}

int rows()
{
    const int D = 16;
    Ctx x(D);
    for (const int by : {0, 8, 16}) {
        WANT(by % 16 == 0, dqrm_scale_refresh(x.h, f(by), i32(), f(0), nullptr, workspace, sizeof(workspace), nullptr));
        WANT(by % 16 == 0, dqrm_grad_quant_int8(x.h, f(by), i32(), c(0), f(0), workspace, sizeof(workspace), nullptr));
        WANT(by % 16 == 0, dqrm_grad_quant_int8_static(T, D, f(by), i32(), c(0), f(0), nullptr));
        WANT(by % 16 == 0, dqrm_grad_quant_int8_unified(x.h, f(by), i32(), f(0), c(0), f(0), nullptr));
        WANT(by % 16 == 0, dqrm_grad_absmax(x.h, f(by), i32(), f(0), nullptr));
        WANT(by % 16 == 0, dqrm_row_update(x.h, f(by), i32(), i32(), c(0), f(0), 0.1f, nullptr));
        WANT(by % 16 == 0, dqrm_train_step_host(x.h, f(by), i32(), i32(), f(0), f(0), i32(), f(0), 0.1f, 16, T * 16, workspace, sizeof(workspace), nullptr));
        WANT(by % 16 == 0, dqrm_dp_merge_update(x.h, f(by), 1, 64, i32(), i32(), c(0), f(0), 0.1f, 64, 64, i32(), i32(), i32(), workspace, sizeof(workspace), nullptr));
        WANT(by % 16 == 0, dqrm_dp_merge_update(x.h, f(0), 1, 64, i32(), i32(), c(0), f(0), 0.1f, 64, 64, i32(), i32(), at<int32_t *>(by), workspace, sizeof(workspace), nullptr));
    }
    for (const int by : {0, 1, 4}) {
        WANT(by % 4 == 0, dqrm_grad_quant_int8(x.h, f(0), i32(), c(by), f(0), workspace, sizeof(workspace), nullptr));
        WANT(by % 4 == 0, dqrm_grad_quant_int8_static(T, D, f(0), i32(), c(by), f(0), nullptr));
        WANT(by % 4 == 0, dqrm_grad_quant_int8_unified(x.h, f(0), i32(), f(0), c(by), f(0), nullptr));
        WANT(by % 4 == 0, dqrm_row_update(x.h, f(0), i32(), i32(), c(by), f(0), 0.1f, nullptr));
        WANT(by % 4 == 0, dqrm_dp_merge_update(x.h, f(0), 1, 64, i32(), i32(), c(by), f(0), 0.1f, 64, 64, i32(), i32(), nullptr, workspace, sizeof(workspace), nullptr));
    }
    for (const int by : {0, 8, 16}) WANT(by % 16 == 0, dqrm_row_summary_attach(x.h, f(by), f(0), 1 << 20, nullptr));
    return failed;
}

// an empty batch follows no pointer to rows
int empty()
{
    const int D = 16, by = 4;
    Ctx x(D);
    WANT(true, dqrm_emb_fwd(x.h, f(by), nullptr, i32(), f(0), i32(), f(0), nullptr, 64, 0, nullptr));
    const int rc = dqrm_emb_bwd(x.h, f(by), nullptr, i32(), nullptr, i32(), f(by), 64, 0, workspace, sizeof(workspace), nullptr);
    if (rc != DQRM_OK) { std::printf("empty backward: status %d\n", rc); failed = 1; }
    return failed;
}

// the blocks of short bags of wide rows stand side by side for all tables, those of long bags and narrow rows table by table
int order()
{
    const int B = 3000;
    for (const int T : {7, 8}) {
        for (const int D : {4, 8, 16, 20, 32, 36, 48, 64, 68, 128, 132, 256, 1024}) {
            Ctx x(D, T);
            const int upto = T < 8 || D <= 16 ? 0 : D <= 32 ? 16 : D <= 64 ? 5 : D <= 128 ? 3 : 0;
            for (const int bag : {1, 2, 3, 4, 5, 12, 16, 30}) {
                const int64_t L = (int64_t)T * B * bag;
                auto mixed = [=] { return fake::grid_x == (unsigned)T && fake::grid_y > (unsigned)T; };
                if (dqrm_emb_fwd(x.h, f(0), i32(), i32(), f(0), i32(), f(0), nullptr, B, L, nullptr) != DQRM_OK || mixed() != (bag == 1 || bag < upto))
                    failed = 1, std::printf("forward, D = %d, bags of %d: grid %u, %u\n", D, bag, fake::grid_x, fake::grid_y);
                if (dqrm_packed_fwd(x.h, u8(0), i32(), i32(), f(0), 4, f(0), B, L, nullptr) != DQRM_OK || mixed() != (bag == 1 || (D > 32 && T >= 8)))
                    failed = 1, std::printf("packed lookup, D = %d, bags of %d: grid %u, %u\n", D, bag, fake::grid_x, fake::grid_y);
            }
        }
    }
    return failed;
}

}  // namespace

int main(int argc, char **argv)
{
    const char *name = argc > 1 ? argv[1] : "";
    if (!strcmp(name, "sum")) return sum();
    if (!strcmp(name, "forward")) return forward();
    if (!strcmp(name, "rows")) return rows();
    if (!strcmp(name, "empty")) return empty();
    if (!strcmp(name, "order")) return order();
    std::printf("no scenario %s\n", name);
    return 2;
}

// The launch code of the backward over a stand-in for the CUDA runtime: launches are counted, refused and checked against
// the functions' shared-memory limits on the host, and nothing runs on a device.  One scenario per run, named by argv[1];
// 0 when what it asserts holds.
#include "../paper_2410_20046_b200/csrc/bwd.cu"
#include <cstdio>
#include <cstring>
#include "launch_host.h"

namespace {

#define WANT(X)                                                                                          \
    do {                                                                                                 \
        if (!(X)) { std::printf("line %d: not so: %s\n", __LINE__, #X); return 1; }                      \
    } while (0)

char workspace[16 << 20];
int32_t dummy[4];

struct Ctx {
    dqrm_ctx c;
    Ctx(int T, int D)
    {
        c.T = T;
        c.D = D;
        c.num_sms = 148;
        c.row_bits = 10;
        c.total_rows = (int64_t)1000 * T;
    }
    int sort(int B, int64_t L, bool *by_table)
    {
        int lists = -1;
        const int rc = dq_launch_bwd_sort(&c, dummy, dummy, dummy, dummy, B, L, workspace, sizeof(workspace), nullptr, &lists);
        *by_table = lists > 0;
        return rc;
    }
    int small_step(int B, int64_t L)
    {
        return dq_launch_small_step(&c, nullptr, dummy, dummy, nullptr, dummy, dummy, nullptr, nullptr, nullptr, 0.1f, B, L,
                                    workspace, sizeof(workspace), nullptr);
    }
};

// contexts of many and of few tables take small steps in turn
int contexts_in_turn()
{
    Ctx many(26, 16), few(4, 16), most(148, 16);
    for (int k = 0; k < 2; ++k) {
        WANT(many.small_step(8, 26 * 8) == DQRM_OK);
        WANT(few.small_step(128, 4 * 128) == DQRM_OK);
    }
    for (int k = 0; k < 2; ++k) {
        WANT(most.small_step(8, 148 * 8) == DQRM_OK);
        WANT(few.small_step(128, 4 * 128) == DQRM_OK);
    }
    return 0;
}

// each sort that is refused leaves the next one to run, and no error for whoever asks next
int refused_sorts()
{
    for (const int refused : {0, 1, 2}) {          // block sort, cluster sort, radix sort
        fake::launches = 0;
        fake::refuse.clear();
        for (int k = 0; k < refused; ++k) fake::refuse.insert(k);
        Ctx x(4, 16);
        bool by_table = false;
        WANT(x.sort(128, 4 * 128, &by_table) == DQRM_OK);
        WANT(by_table == (refused < 2));
        WANT(x.c.last_cuda_error == (refused ? (int)cudaErrorInvalidValue : 0));
        WANT(cudaGetLastError() == cudaSuccess);
    }
    return 0;
}

// a batch with as many lookups as bags may hold most of them in one table: beyond a thousand a table a cluster stands by for it,
// while the clusters of all tables have room
int clusters_stand_by()
{
    bool by_table = false;
    for (const int T : {1, 2, 26, 37, 38, 100})
        for (const int B : {300, 1024, 1025, 1500, 2048, 2049}) {
            Ctx x(T, 16);
            WANT(x.sort(B, (int64_t)T * B, &by_table) == DQRM_OK && by_table);
            WANT((fake::cluster > 1) == (B > 2048 || (B > 1024 && T <= 37)));
        }
    return 0;
}

// a batch's mean does not say how large its largest table is: unless the batch has an index a bag, clusters of eight stand ready for every table
int eight_blocks_a_table()
{
    bool by_table = false;
    for (const int T : {10, 19, 26, 33, 34, 38, 64, 100})
        for (const int B : {2100, 2600, 8000, 12000}) {
            if ((int64_t)T * B > 260000) continue;
            Ctx x(T, 16);
            WANT(x.sort(B, (int64_t)T * B, &by_table) == DQRM_OK && by_table);
            const unsigned blocks = T >= 38 || (T >= 19 && B <= 8192) ? 4 : 8;
            WANT(fake::cluster == blocks && fake::grid_x == blocks * T);
            WANT(x.sort(B, (int64_t)T * B + 1, &by_table) == DQRM_OK && by_table);
            WANT(fake::cluster == 8 && fake::grid_x == 8u * T);
        }
    return 0;
}

// tiles of 8, 16 and 32 entries on both sides of the lines, and ranges of a few of them, of which there are no more than the workspace
// has room for
int tiles_of_the_sum()
{
    auto cut = [](int64_t n, int64_t by) { return (n + by - 1) / by; };
    for (const int D : {52, 64, 96, 128})
        for (const int64_t L : {60000LL, 85200LL, 85300LL, 113600LL, 113700LL, 340000LL, 342000LL, 454600LL, 454700LL, 852000LL, 2000000LL, 2800000LL, 3700000LL, 8500000LL})
            for (const int bag : {1, 4, 5}) {
                Ctx x(4, D);
                const int64_t full = 148 * (D <= 64 ? 4 : 3) * 8, warps = D <= 64 && L < 18 * full ? full / 4 * 3 : full, B = L / 4 / bag;
                const int64_t tile = L < (D < 64 ? 24 : D == 64 && bag > 1 ? 72 : 96) * full ? 8 : D == 64 && bag > 4 ? 32 : 16;
                const int64_t tiles = cut(L, tile), even = cut(tiles, warps);
                int64_t range = even;
                if (D <= 64 && tile > 8 && even > (tile == 32 ? 16 : 36)) range = (D == 64 || even < 48 ? 256 : 384) / tile;
                WANT(dq_launch_bwd_sum(&x.c, nullptr, dummy, dummy, nullptr, (int)B, L / bag / 4 * 4 * bag, 1, workspace, (size_t)1 << 40, nullptr) == DQRM_OK);
                WANT((int64_t)fake::grid_x == cut(cut(cut(L / bag / 4 * 4 * bag, tile), range), 8));
                WANT(cut(tiles, range) <= std::max(warps, L / 256 + 1));
            }
    return 0;
}

}  // namespace

int main(int argc, char **argv)
{
    const char *name = argc > 1 ? argv[1] : "";
    if (!strcmp(name, "contexts_in_turn")) return contexts_in_turn();
    if (!strcmp(name, "refused_sorts")) return refused_sorts();
    if (!strcmp(name, "clusters_stand_by")) return clusters_stand_by();
    if (!strcmp(name, "eight_blocks_a_table")) return eight_blocks_a_table();
    if (!strcmp(name, "tiles_of_the_sum")) return tiles_of_the_sum();
    std::printf("no scenario %s\n", name);
    return 2;
}

// Host checks of the tiled sweep's plans (tile_plan.cpp), linked against the library and run by
// test_tile_plan_cpu.py.  Usage: tile_plan_check alloc depth mesh [mesh ...]
//   mesh: file with int32 nv, nt, then double V[nv][3], int32 F[nt][3]; several meshes form a batch
//   alloc: while a plan is built, one host allocation fails, each in turn (sampled); the failure has to
//          come back as std::bad_alloc, whichever thread met it
#include <atomic>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <new>
#include <string>

#include "tile_plan.h"

using namespace lbmg;

static std::atomic<long> g_allocs{0}, g_fail_at{-1};
static void *get(size_t n) {
    const long k = g_allocs.fetch_add(1);
    return k == g_fail_at.load() ? nullptr : std::malloc(n ? n : 1);
}
void *operator new(size_t n) {
    if (void *p = get(n)) return p;
    throw std::bad_alloc();
}
void *operator new[](size_t n) { return operator new(n); }
void *operator new(size_t n, const std::nothrow_t &) noexcept { return get(n); }
void operator delete(void *p) noexcept { std::free(p); }
void operator delete[](void *p) noexcept { std::free(p); }
void operator delete(void *p, size_t) noexcept { std::free(p); }
void operator delete[](void *p, size_t) noexcept { std::free(p); }
void operator delete(void *p, const std::nothrow_t &) noexcept { std::free(p); }

static const int kDown[8] = {0, 1, 2, 3, 4, 5, 6, 7};

// the host work of a level's tiles, as the upload does it
static bool plan_of(const HostLevel &L, int ntile, TilePlan &plan, TileCut &cut) {
    cut_tiles(L, ntile, cut);
    if (!build_tile_plan(L, cut, kDown, 8, true, plan)) return false;
    rebalance_tiles(plan, cut);
    split_tiles(plan, 64, cut);
    return build_tile_plan(L, cut, kDown, 8, true, plan);
}

static int check_alloc(const HostLevel &L) {
    long failed = 0, total = 0;
    {
        TilePlan plan;
        TileCut cut;
        g_allocs = 0;
        if (!plan_of(L, 13, plan, cut)) return std::printf("no plan\n"), 1;
        total = g_allocs;
    }
    for (long k = 0; k < total; k += 1 + total / 300) {
        TilePlan plan;
        TileCut cut;
        g_allocs = 0;
        g_fail_at = k;
        try {
            plan_of(L, 13, plan, cut);
        } catch (const std::bad_alloc &) {
            failed++;
        }
        g_fail_at = -1;
    }
    std::printf("%ld allocations, %ld failures came back\n", total, failed);
    return failed > 0 ? 0 : 1;
}

int main(int argc, char **argv) {
    if (argc < 4) return 2;
    std::vector<HostHierarchy> parts(argc - 3);
    HostHierarchy H;
    std::string err;
    for (int m = 0; m < argc - 3; m++) {
        FILE *f = std::fopen(argv[m + 3], "rb");
        int n[2];
        if (!f || std::fread(n, 4, 2, f) != 2) return 2;
        std::vector<double> V(3 * (size_t)n[0]);
        std::vector<int> F(3 * (size_t)n[1]);
        if (std::fread(V.data(), 8, V.size(), f) != V.size() || std::fread(F.data(), 4, F.size(), f) != F.size()) return 2;
        std::fclose(f);
        if (build_host_hierarchy(V.data(), n[0], F.data(), n[1], std::atoi(argv[2]), -1, 160, 1, 0, parts[m], err, false,
                                 false))
            return std::printf("%s\n", err.c_str()), 2;
    }
    if (combine_batch(parts, H, err)) return std::printf("%s\n", err.c_str()), 2;
    for (int d = H.d0 + 1; d <= H.D; d++)
        if (H.lev[d].ns > 0 && !std::strcmp(argv[1], "alloc") && check_alloc(H.lev[d])) return 1;
    return 0;
}

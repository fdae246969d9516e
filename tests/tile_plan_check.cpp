// Host checks of the tiled sweep's plans (tile_plan.cpp), linked against the library and run by
// test_tile_plan_cpu.py.  Usage: tile_plan_check plan|alloc depth mesh [mesh ...]
//   mesh: file with int32 nv, nt, then double V[nv][3], int32 F[nt][3]; several meshes form a batch
//   plan:  every tile, walked on its own from the level's vector, has to give its rows the values and the
//          residuals of the sweep over the whole level, bit for bit, and nothing may lie outside the plan's
//          tables; each direction, whole sweeps and halves, one tile and many, as cut, rebalanced and split
//   alloc: while a plan is built, one host allocation fails, each in turn (sampled); the failure has to
//          come back as std::bad_alloc, whichever thread met it
#include <atomic>
#include <cmath>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <new>
#include <random>
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

static const int kUp[8] = {7, 6, 5, 4, 3, 2, 1, 0};

struct System {
    std::vector<double> A, x, b, d;
    explicit System(const HostLevel &L) : A(L.rp[L.ndof]), x(L.ndof), b(L.ndof), d(L.ndof) {
        std::mt19937 rng(1);
        std::uniform_real_distribution<double> u(-1, 1);
        for (double &v : A) v = u(rng);
        for (int i = 0; i < L.ndof; i++) { x[i] = u(rng); b[i] = u(rng); d[i] = 0.05 * u(rng); }
    }
};

// one launch: the steps seq[0..nsteps) and, when asked, the residual; the plan's tiles against the whole level
static const char *check_launch(const HostLevel &L, const System &S, const TileCut &cut, const int *seq, int nsteps,
                                bool residual) {
    TilePlan P;
    if (!build_tile_plan(L, cut, seq, nsteps, residual, P)) return "no plan";
    std::vector<double> y = S.x, r(L.ndof, 0.0), xo(L.ndof, NAN), ro(L.ndof, NAN);
    auto row_sum = [&](int i) {
        double acc = 0;
        for (int k = L.rp[i]; k < L.rp[i + 1]; k++) acc = std::fma(S.A[k], y[L.ci[k]], acc);
        return acc;
    };
    for (int s = 0; s < nsteps; s++)
        for (int i = L.colour_start[seq[s]]; i < L.colour_start[seq[s] + 1]; i++) y[i] += (S.b[i] - row_sum(i)) * S.d[i];
    for (int i = 0; i < L.ns; i++) r[i] = S.b[i] - row_sum(i);
    for (int t = 0; t < P.ntile; t++) {
        const int32_t *f = &P.info[(size_t)t * kTileInfo], *cum = &P.cum[(size_t)t * (P.maxgrp + 1)];
        const int32_t *loc = &P.loc[(size_t)t * P.maxloc];
        if (f[0] > P.maxloc || f[1] > P.maxcomp || f[2] > f[1] || f[1] > f[0] || f[5 + nsteps] > P.maxgrp) return "sizes";
        std::vector<double> sx(f[0]);
        for (int q = 0; q < f[0]; q++) sx[q] = S.x[loc[q]];
        for (int s = 0, g = 0; s <= nsteps; s++) {
            if (s == nsteps && nsteps > 0)
                for (int q = 0; q < f[2]; q++) {
                    if (!std::isnan(xo[loc[q]])) return "row of two tiles";
                    xo[loc[q]] = sx[q];
                }
            if (s == nsteps && !residual) break;
            for (; g < f[5 + s]; g++) {
                const size_t G = (size_t)f[3] + g, q0 = (size_t)f[4] + cum[g];
                const int K = cum[g + 1] - cum[g];
                if (K > P.maxquads) return "quads";
                for (int k = 0; k < K; k++)
                    if (P.qgroup[q0 + k] != (int)G) return "group of a quad";
                for (int l = 0; l < kTileRows; l++) {
                    const int slot = P.slot[kTileRows * G + l], row = P.row[kTileRows * G + l];
                    if (slot == kTileNoRow) {
                        if (row != -1) return "row without a slot";
                        continue;
                    }
                    if (slot >= f[1] || loc[slot] != row) return "slot";
                    double acc = 0;
                    for (int k = 0; k < 4 * K; k++) {
                        const size_t p = 32 * (q0 + (k >> 2)) + 4 * l + (k & 3);
                        if (P.col[p] >= f[0]) return "column";
                        acc = std::fma(P.map[p] >= 0 ? S.A[P.map[p]] : 0.0, sx[P.col[p]], acc);
                    }
                    if (s < nsteps) sx[slot] += (S.b[row] - acc) * S.d[row];
                    else ro[row] = S.b[row] - acc;
                }
            }
        }
    }
    for (int i = 0; i < L.ns; i++) {
        bool mine = false;
        for (int s = 0; s < nsteps; s++) mine |= i >= L.colour_start[seq[s]] && i < L.colour_start[seq[s] + 1];
        if (mine ? xo[i] != y[i] : !std::isnan(xo[i])) return "value";
        if (residual && ro[i] != r[i]) return "residual";
    }
    return nullptr;
}

static int check_plans(const HostLevel &L) {
    const System S(L);
    for (int ntile : {1, 2, 13, 152}) {
        TileCut cut;
        cut_tiles(L, ntile, cut);
        for (int stage = 0; stage < (ntile > 1 ? 3 : 1); stage++) {   // as cut, rebalanced, split
            TilePlan P;
            if (stage > 0 && !build_tile_plan(L, cut, kDown, 8, true, P)) return std::printf("no plan\n"), 1;
            if (stage == 1) rebalance_tiles(P, cut);
            if (stage == 2) split_tiles(P, (int)(L.ns / ntile) + 16, cut);
            struct { const int *seq; int nsteps; bool residual; } job[] = {
                {kDown, 8, true}, {kDown, 8, false}, {kUp, 8, false}, {kDown, 4, false}, {kDown + 4, 4, false},
                {kUp, 4, false},  {kUp + 4, 4, false}, {kDown, 0, true}};
            for (const auto &j : job)
                if (const char *what = check_launch(L, S, cut, j.seq, j.nsteps, j.residual))
                    return std::printf("rows %d tiles %d stage %d steps %d: %s\n", L.ns, ntile, stage, j.nsteps, what), 1;
        }
    }
    return 0;
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
        if (H.lev[d].ns > 0 && (!std::strcmp(argv[1], "alloc") ? check_alloc(H.lev[d]) : check_plans(H.lev[d]))) return 1;
    return 0;
}

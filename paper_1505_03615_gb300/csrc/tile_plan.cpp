// tile_plan.cpp -- host side of the tiled Gauss-Seidel sweep (tile.cu): cuts a level's rows into
// tiles and finds, for a sequence of colour steps, the rows each tile has to update itself.
//
// A tile owns the rows of some blocks of 2x2x2 corners (all eight colours).  To produce their values
// after the whole sequence without hearing from other tiles, it also updates, step by step, the rows
// of other tiles that its own rows read in the meantime.  Going backwards through the steps, the set
// of needed rows of colour c only grows: at a step of colour c all rows of colour c needed so far are
// updated, and their neighbours join the needed rows of their colours.  Rows needed at the start are
// read from the level's vector.  With colours by corner parity a sweep reaches at most 7, 3 and 1
// corners along the axes, so on surfaces the overlap is a thin rim of the tile.
#include <algorithm>
#include <atomic>
#include <cstring>
#include <new>
#include <numeric>

#include "tile_plan.h"

namespace lbmg {

namespace {

using Block = TileCut::Block;

// A host allocation that fails inside a parallel region or a task: remembered there (an exception that leaves
// one ends the process) and thrown by the caller's thread behind it.
struct AllocFailure {
    std::atomic<bool> failed{false};
    template <class F>
    void guard(F &&work) {
        if (failed) return;
        try {
            work();
        } catch (...) {
            failed = true;
        }
    }
    void rethrow() const {
        if (failed) throw std::bad_alloc();
    }
};

// The steps reach over at most 7 (x), 3 (y) and 1 (z) corners, the residual and the rim's own reads over
// one or two more: tiles are cut across the axis along which they measure the most reaches.
constexpr int kReach[3] = {8, 4, 2};

// blocks [b0, b1) into ntile tiles from t0 on, by recursive bisection at equal shares of entries
void bisect(std::vector<Block> &blk, int64_t b0, int64_t b1, int t0, int ntile, std::vector<int64_t> &start,
            AllocFailure &alloc) {
    if (ntile <= 1) {
        start[t0] = b0;
        return;
    }
    const int tl = ntile / 2;
    int64_t m = b0;
    auto cut = [&]() {
        int lo[3], hi[3], il = blk[b0].inst, ih = il;
        for (int a = 0; a < 3; a++) lo[a] = hi[a] = blk[b0].at[a];
        double w = 0;
        for (int64_t q = b0; q < b1; q++) {
            const Block &B = blk[q];
            for (int a = 0; a < 3; a++) { lo[a] = std::min(lo[a], B.at[a]); hi[a] = std::max(hi[a], B.at[a]); }
            il = std::min(il, B.inst); ih = std::max(ih, B.inst);
            w += B.weight;
        }
        int ax = 0;
        for (int a = 1; a < 3; a++)
            if ((int64_t)(hi[a] - lo[a] + 1) * kReach[ax] > (int64_t)(hi[ax] - lo[ax] + 1) * kReach[a]) ax = a;
        auto key = [&](const Block &B) { return ih > il ? B.inst : B.at[ax]; };   // meshes of a batch first
        const int k0 = ih > il ? il : lo[ax], nk = (ih > il ? ih : hi[ax]) - k0 + 1;
        std::vector<double> hist(nk, 0.0);
        for (int64_t q = b0; q < b1; q++) hist[key(blk[q]) - k0] += blk[q].weight;
        // the plane in which the left share ends: planes before it go left, of its own blocks as many as needed
        double left = w * tl / ntile, acc = 0;
        int k = 0;
        while (k + 1 < nk && acc + hist[k] <= left) acc += hist[k++];
        auto mid = std::stable_partition(blk.begin() + b0, blk.begin() + b1, [&](const Block &B) { return key(B) - k0 < k; });
        auto end = std::stable_partition(mid, blk.begin() + b1, [&](const Block &B) { return key(B) - k0 == k; });
        m = mid - blk.begin();
        // within the plane along the next most extended axis (a batch: the mesh's own cut follows below)
        const int ay = ax == 0 ? ((int64_t)(hi[1] - lo[1] + 1) * kReach[2] >= (int64_t)(hi[2] - lo[2] + 1) * kReach[1] ? 1 : 2) : 0;
        std::stable_sort(mid, end, [&](const Block &A, const Block &B) { return A.at[ay] < B.at[ay]; });
        for (; m < end - blk.begin() && acc + blk[m].weight <= left; m++) acc += blk[m].weight;
    };
    if (b1 > b0) alloc.guard(cut);
    const int64_t mm = m;
#pragma omp task shared(blk, start, alloc) if (b1 - b0 > 4096)
    bisect(blk, b0, mm, t0, tl, start, alloc);
#pragma omp task shared(blk, start, alloc) if (b1 - b0 > 4096)
    bisect(blk, mm, b1, t0 + tl, ntile - tl, start, alloc);
#pragma omp taskwait
}

void bisect_all(TileCut &cut, int ntile) {
    cut.start.assign(ntile + 1, (int64_t)cut.blocks.size());
    AllocFailure alloc;
#pragma omp parallel
#pragma omp single
    bisect(cut.blocks, 0, (int64_t)cut.blocks.size(), 0, ntile, cut.start, alloc);
    alloc.rethrow();
}

struct TileOut {
    std::vector<int32_t> loc, gk, row, map;
    std::vector<uint16_t> slot, col;
    int32_t step_end[kTileSteps + 1] = {0};
    int ncomp = 0, nown = 0, quads = 0;
    bool ok = true;
};

}  // namespace

void cut_tiles(const HostLevel &L, int ntile, TileCut &cut) {
    std::vector<Block> &blk = cut.blocks;
    auto key = [&](int i) {
        return std::make_pair(L.inst.empty() ? 0 : L.inst[i],
                              morton(L.corner[3 * (size_t)i], L.corner[3 * (size_t)i + 1], L.corner[3 * (size_t)i + 2]) >> 3);
    };
    // a colour's rows come by mesh and Morton key: merge the eight colours
    int at[8], end[8];
    std::pair<int32_t, uint64_t> k[8];
    for (int c = 0; c < 8; c++) {
        at[c] = L.colour_start[c]; end[c] = L.colour_start[c + 1];
        if (at[c] < end[c]) k[c] = key(at[c]);
    }
    blk.clear();
    for (;;) {
        int b = -1;
        for (int c = 0; c < 8; c++)
            if (at[c] < end[c] && (b < 0 || k[c] < k[b])) b = c;
        if (b < 0) break;
        const auto kb = k[b];
        Block B;
        for (int a = 0; a < 3; a++) B.at[a] = L.corner[3 * (size_t)at[b] + a] >> 1;
        B.inst = kb.first;
        B.weight = 0;
        for (int c = 0; c < 8; c++) {
            B.first[c] = at[c];
            while (at[c] < end[c] && k[c] == kb) {
                B.weight += L.rp[at[c] + 1] - L.rp[at[c]];
                if (++at[c] < end[c]) k[c] = key(at[c]);
            }
            B.rows[c] = at[c] - B.first[c];
        }
        blk.push_back(B);
    }
    bisect_all(cut, ntile);
}

void rebalance_tiles(const TilePlan &plan, TileCut &cut) {
    for (int t = 0; t < plan.ntile; t++) {
        const int32_t *f = &plan.info[(size_t)t * kTileInfo], *cum = &plan.cum[(size_t)t * (plan.maxgrp + 1)];
        const double proc = 32.0 * cum[plan.nsteps > 0 ? f[5 + plan.nsteps - 1] : 0];
        double own = 0;
        for (int64_t q = cut.start[t]; q < cut.start[t + 1]; q++) own += cut.blocks[q].weight;
        if (own > 0 && proc > 0)
            for (int64_t q = cut.start[t]; q < cut.start[t + 1]; q++) cut.blocks[q].weight *= proc / own;
    }
    bisect_all(cut, plan.ntile);
}

bool split_tiles(const TilePlan &plan, int maxloc, TileCut &cut) {
    std::vector<int64_t> start, half(3);
    bool any = false;
    for (int t = 0; t < plan.ntile; t++) {
        start.push_back(cut.start[t]);
        if (plan.info[(size_t)t * kTileInfo] <= maxloc || cut.start[t + 1] - cut.start[t] < 2) continue;
        AllocFailure alloc;
        bisect(cut.blocks, cut.start[t], cut.start[t + 1], 0, 2, half, alloc);
        alloc.rethrow();
        if (half[1] > cut.start[t] && half[1] < cut.start[t + 1]) { start.push_back(half[1]); any = true; }
    }
    start.push_back(cut.start[plan.ntile]);
    cut.start = start;
    return any;
}

bool build_tile_plan(const HostLevel &L, const TileCut &cut, const int *seq, int nsteps, bool residual, TilePlan &out) {
    const int ntile = (int)cut.start.size() - 1;
    const std::vector<Block> &blk = cut.blocks;
    const std::vector<int64_t> &start = cut.start;
    out = TilePlan();
    if (L.ns <= 0 || ntile < 1 || nsteps < 0 || nsteps > kTileSteps) return false;
    std::vector<TileOut> tiles(ntile);
    bool steps_colour[8] = {false};
    for (int s = 0; s < nsteps; s++) steps_colour[seq[s]] = true;
    std::vector<uint8_t> colour(L.ns);
    for (int c = 0; c < 8; c++) std::fill(colour.begin() + L.colour_start[c], colour.begin() + L.colour_start[c + 1], (uint8_t)c);
    AllocFailure alloc;
#pragma omp parallel
    {
        std::vector<int32_t> mark, slot_of, list[8], order;
        alloc.guard([&]() {
            mark.assign(L.ndof, -1);
            slot_of.assign(L.ndof, 0);
        });
        auto one = [&](int t) {
            TileOut &T = tiles[t];
            size_t own[8], cnt[kTileSteps], comp[8] = {0};   // needed rows at each step, computed rows of each colour
            for (int c = 0; c < 8; c++) {
                list[c].clear();
                for (int64_t q = start[t]; q < start[t + 1]; q++)
                    for (int i = blk[q].first[c]; i < blk[q].first[c] + blk[q].rows[c]; i++) {
                        list[c].push_back(i);
                        mark[i] = t;
                    }
                std::sort(list[c].begin(), list[c].end());
                own[c] = list[c].size();
            }
            auto add_neighbours = [&](int i) {
                for (int k = L.rp[i]; k < L.rp[i + 1]; k++) {
                    const int j = L.ci[k];
                    if (j >= L.ns) { T.ok = false; continue; }   // smoothed rows couple with smoothed rows only
                    if (mark[j] != t) { mark[j] = t; list[colour[j]].push_back(j); }
                }
            };
            if (residual)
                for (int c = 0; c < 8; c++)
                    for (size_t q = 0; q < own[c]; q++) add_neighbours(list[c][q]);
            for (int s = nsteps - 1; s >= 0; s--) {
                const int c = seq[s];
                cnt[s] = list[c].size();
                // (rows of a later step of this colour have their neighbours listed already)
                for (size_t q = comp[c]; q < cnt[s]; q++) add_neighbours(list[c][q]);
                comp[c] = cnt[s];
            }
            // local slots: the rows to compute first, own rows ahead, then those that are only read
            T.loc.clear();
            for (int c = 0; c < 8; c++)
                if (steps_colour[c] || (residual && nsteps == 0))
                    T.loc.insert(T.loc.end(), list[c].begin(), list[c].begin() + own[c]);
            T.nown = (int)T.loc.size();
            for (int c = 0; c < 8; c++)
                if (comp[c] > own[c]) {
                    order.assign(list[c].begin() + own[c], list[c].begin() + comp[c]);
                    std::sort(order.begin(), order.end());
                    T.loc.insert(T.loc.end(), order.begin(), order.end());
                }
            T.ncomp = (int)T.loc.size();
            for (int c = 0; c < 8; c++) {
                const size_t from = steps_colour[c] ? std::max(comp[c], own[c]) : (residual && nsteps == 0 ? own[c] : 0);
                order.assign(list[c].begin() + from, list[c].end());
                std::sort(order.begin(), order.end());
                T.loc.insert(T.loc.end(), order.begin(), order.end());
            }
            if (T.loc.size() > 65534) { T.ok = false; return; }
            for (size_t q = 0; q < T.loc.size(); q++) slot_of[T.loc[q]] = (int32_t)q;
            // groups of kTileRows rows, longest rows first, so that a group's rows are about equally long
            auto len = [&](int i) { return L.rp[i + 1] - L.rp[i]; };
            auto groups = [&](std::vector<int32_t> &rows) {
                std::sort(rows.begin(), rows.end(),
                          [&](int a, int b) { return len(a) != len(b) ? len(a) > len(b) : a < b; });
                for (size_t r0 = 0; r0 < rows.size(); r0 += kTileRows) {
                    const int m = (int)std::min<size_t>(kTileRows, rows.size() - r0);
                    const int K = (len(rows[r0]) + 3) / 4;
                    T.gk.push_back(K);
                    T.quads += K;
                    const size_t base = T.col.size(), s0 = T.slot.size();
                    T.slot.resize(s0 + kTileRows, kTileNoRow);
                    T.row.resize(s0 + kTileRows, -1);
                    T.col.resize(base + 32 * (size_t)K, 0);
                    T.map.resize(base + 32 * (size_t)K, -1);
                    for (int l = 0; l < m; l++) {
                        const int i = rows[r0 + l], n = len(i), k0 = L.rp[i];
                        T.slot[s0 + l] = (uint16_t)slot_of[i];
                        T.row[s0 + l] = i;
                        for (int k = 0; k < 4 * K; k++) {
                            const size_t p = base + 32 * (size_t)(k >> 2) + 4 * l + (k & 3);
                            // pads: the row's own slot with a zero value
                            T.col[p] = (uint16_t)(k < n ? slot_of[L.ci[k0 + k]] : slot_of[i]);
                            T.map[p] = k < n ? k0 + k : -1;
                        }
                    }
                }
            };
            for (int s = 0; s < nsteps; s++) {
                order.assign(list[seq[s]].begin(), list[seq[s]].begin() + cnt[s]);
                groups(order);
                T.step_end[s] = (int32_t)T.gk.size();
            }
            if (residual) {
                order.clear();
                for (int c = 0; c < 8; c++) order.insert(order.end(), list[c].begin(), list[c].begin() + own[c]);
                groups(order);
            }
            T.step_end[nsteps] = (int32_t)T.gk.size();
        };
#pragma omp for schedule(dynamic, 1)
        for (int t = 0; t < ntile; t++) alloc.guard([&]() { one(t); });
    }
    alloc.rethrow();
    for (const TileOut &T : tiles)
        if (!T.ok) return false;
    std::vector<int64_t> g0(ntile + 1, 0), q0(ntile + 1, 0);
    for (int t = 0; t < ntile; t++) {
        const TileOut &T = tiles[t];
        g0[t + 1] = g0[t] + (int64_t)T.gk.size();
        q0[t + 1] = q0[t] + T.quads;
        out.maxloc = std::max(out.maxloc, (int)T.loc.size());
        out.maxcomp = std::max(out.maxcomp, T.ncomp);
        out.maxgrp = std::max(out.maxgrp, (int)T.gk.size());
        for (int32_t k : T.gk) out.maxquads = std::max(out.maxquads, (int)k);
    }
    if (q0[ntile] > INT32_MAX || g0[ntile] > INT32_MAX / kTileRows) return false;
    out.ntile = ntile;
    out.nsteps = nsteps;
    out.groups = g0[ntile];
    out.quads = q0[ntile];
    out.info.assign((size_t)ntile * kTileInfo, 0);
    out.loc.assign((size_t)ntile * out.maxloc, -1);
    out.cum.assign((size_t)ntile * (out.maxgrp + 1), 0);
    out.row.resize(kTileRows * (size_t)out.groups);
    out.slot.resize(kTileRows * (size_t)out.groups);
    out.qgroup.resize((size_t)out.quads);
    out.col.resize(32 * (size_t)out.quads);
    out.map.resize(32 * (size_t)out.quads);
#pragma omp parallel for schedule(dynamic, 1)
    for (int t = 0; t < ntile; t++) {
        const TileOut &T = tiles[t];
        int32_t *f = &out.info[(size_t)t * kTileInfo];
        f[0] = (int32_t)T.loc.size();
        f[1] = T.ncomp;
        f[2] = T.nown;
        f[3] = (int32_t)g0[t];
        f[4] = (int32_t)q0[t];
        for (int s = 0; s <= nsteps; s++) f[5 + s] = T.step_end[s];
        std::copy(T.loc.begin(), T.loc.end(), out.loc.begin() + (size_t)t * out.maxloc);
        int32_t *cum = &out.cum[(size_t)t * (out.maxgrp + 1)];
        int64_t q = 0;
        for (size_t g = 0; g < T.gk.size(); g++) {
            cum[g] = (int32_t)q;
            for (int k = 0; k < T.gk[g]; k++) out.qgroup[(size_t)(q0[t] + q + k)] = (int32_t)(g0[t] + (int64_t)g);
            q += T.gk[g];
        }
        for (size_t g = T.gk.size(); g <= (size_t)out.maxgrp; g++) cum[g] = (int32_t)q;
        std::copy(T.row.begin(), T.row.end(), out.row.begin() + kTileRows * g0[t]);
        std::copy(T.slot.begin(), T.slot.end(), out.slot.begin() + kTileRows * g0[t]);
        std::copy(T.col.begin(), T.col.end(), out.col.begin() + 32 * q0[t]);
        std::copy(T.map.begin(), T.map.end(), out.map.begin() + 32 * q0[t]);
    }
    return true;
}

void tile_shape(int rows, int sms, int *parts, int *ntile) {
    if (rows <= sms * kTileOneRound) {
        *ntile = std::max(1, std::min(sms, rows / kTileMinRows));
    } else {
        const int per = (rows + 2 * sms - 1) / (2 * sms);
        *ntile = 2 * sms * ((per + kTileMaxRows - 1) / kTileMaxRows);
    }
    *parts = rows >= kTileTwoParts ? 2 : 1;
}

}  // namespace lbmg

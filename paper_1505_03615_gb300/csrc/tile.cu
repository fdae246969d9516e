// tile.cu -- tiled Gauss-Seidel sweep: all eight colour steps of a sweep (Sections 4.3 and 5.2), the
// prolongation in front of it and the residual behind it, in one launch.
//
// Launched colour by colour, a sweep is eight dependent kernels, each of which waits for the last one
// to drain, fetches its rows and gathers x from L2: 2.2 us each in FP32 on small levels, about 5 us in
// FP64, whatever the level's size.  Here a block takes a tile of rows (tile_plan.cpp) and walks the eight
// steps on its own: x of the tile and its rim lives in shared memory, a block barrier separates the steps,
// and the rim rows that other tiles own are updated here again, from the same values by the same
// arithmetic, so no block waits for another.  x is read from one vector and written to another, since
// other tiles still read the old values.  A launch then takes 5 to 6 us in FP32 (a wait of 1 us for x, 0.3
// to 0.4 us a step) and 12 us in FP64 (its pipe, which a tile's few rows keep busy 1.2 us a step): V(2,2)
// cycles of the 200k-triangle knot at depth 8 went from 394 to 285 us mixed and from 1225 to 840 us FP64.
//
// Where the line lies (kTileLevel32, kTileLevel64): the rim costs work, about 3.5 times the own entries at
// 64 rows a tile, 1.5 to 2 at 250 rows in two launches per sweep of four colours each, and every plan has a
// copy of the entries, which on larger levels pushes the other levels' data out of L2.  Measured per FP32
// sweep of torus-knot levels, colour launches / tiles: 18 / 5.5 us at 5,000 rows, 18 / 7.5 at 19,000, 18 / 11
// at 78,000, 28 / 27 at 232,000, 76 / 71-79 at 927,000.  It depends on the components and on what else has to
// stay in L2: a cycle of the 1M-triangle sheets with their 91,202 rows tiled / not took 852 / 860 us at one
// right-hand side, 1007 / 1011 at two, 1246 / 1239 at three, with the next level of 359,326 rows tiled too
// 895, 1068 and 1244; between 77,584 and 91,202 rows nothing was measured, and 80,000 is a coarse line.  FP64 at
// three right-hand sides: 42 / 14 us, 42 / 30, 42 / 37, 60 / 70, 290 / 310, with colour launches that summed the
// padding lane too; without it the line still holds (a cycle of the 200k knot 608 us with it at 60,000 rows, 632
// with it at 15,000).  Plans for FP64 exist up to kTileLevel32: the tuner takes them at 77,584 rows for one and
// two right-hand sides.
//
// Four lanes share a row, as in packed.cu, so that a row's gathers are few per lane and all in flight
// together (a step is one chain of shared-memory latencies); the lanes' sums are added so that lane c ends
// with component c, which it updates.  A group is one run of bytes (slots,
// inverse diagonals, then per quad 16-bit local columns and values), which the warp that will process it
// pulls into its own ring in shared memory with TMA bulk copies, several groups ahead: the entries are
// static, so they arrive while the warp waits at the step barriers, and on small levels the whole tile is
// under way before the launch has to wait for its predecessor.
#include <algorithm>

#include "lbmg_internal.h"

namespace lbmg {

namespace {

constexpr int kTileWarps = 8, kTileThreads = 32 * kTileWarps;
constexpr int kTileRing = 16;                                 // groups in flight per warp at most
// a copy or a step's barrier is given up after one second; after 10 ms where arrivals are missing on purpose
constexpr unsigned kTileWaitNs = 1000000000u, kTilePhantomWaitNs = 10000000u;

template <int N> struct Int { static constexpr int value = N; };
template <class T> struct TileCfg;
template <> struct TileCfg<float> { using T2 = float2; };
template <> struct TileCfg<double> { using T2 = double2; };

// bytes of a group's head (slots, inverse diagonals) and of one quad of its rows (columns, values)
template <class T> constexpr int kHead = kTileRows * (2 + (int)sizeof(T));
template <class T> constexpr int kQuad = 32 * (2 + (int)sizeof(T));

template <class T>
struct TileArgs {
    const int *info, *loc, *cum;
    const unsigned char *stream;
    int nsteps, maxloc, maxcomp, maxgrp, gbytes, ring;
    bool residual;
    const T *b;
    // rows of part q (from bound[q - 1] to bound[q]) are read from buf[bit q of cur], as zero when bit q of
    // zero is set, plus the prolonged coarse correction xc when bit q of prolong is set
    const T *buf[2];
    int bound[kTileParts - 1];
    unsigned cur, zero, prolong;
    T *xout;
    const T *xc;
    const int *par;
    const int8_t *npl2;
    T *r;
    int *status;               // set to 1 when a copy or a warp did not arrive in time
    int arrivals;              // of a step's barrier: the warps, and in a test more that never come
    unsigned wait_ns;          // bound of every wait
};

// a row of R components, in one or two vector accesses
template <class T, int R>
__device__ __forceinline__ void ld_row(const T *p, T (&v)[R]) {
    if constexpr (sizeof(T) * R == 16 && R == 4) {
        const float4 q = *reinterpret_cast<const float4 *>(p);
        v[0] = q.x; v[1] = q.y; v[2] = q.z; v[3] = q.w;
    } else if constexpr (R == 1) {
        v[0] = p[0];
    } else {
        using T2 = typename TileCfg<T>::T2;
#pragma unroll
        for (int c = 0; c < R; c += 2) {
            const T2 q = reinterpret_cast<const T2 *>(p)[c >> 1];
            v[c] = q.x; v[c + 1] = q.y;
        }
    }
}
template <class T, int R>
__device__ __forceinline__ void st_row(T *p, const T (&v)[R]) {
    if constexpr (sizeof(T) * R == 16 && R == 4) {
        *reinterpret_cast<float4 *>(p) = make_float4(v[0], v[1], v[2], v[3]);
    } else if constexpr (R == 1) {
        p[0] = v[0];
    } else {
        using T2 = typename TileCfg<T>::T2;
#pragma unroll
        for (int c = 0; c < R; c += 2) reinterpret_cast<T2 *>(p)[c >> 1] = T2{v[c], v[c + 1]};
    }
}

// asynchronous copies of 4, 8 or 16 bytes into shared memory
template <int N>
__device__ __forceinline__ void copy_async(void *dst, const void *src) {
    const uint32_t d = (uint32_t)__cvta_generic_to_shared(dst);
    if constexpr (N == 16) asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(d), "l"(src) : "memory");
    else asm volatile("cp.async.ca.shared.global [%0], [%1], %2;" ::"r"(d), "l"(src), "n"(N) : "memory");
}
__device__ __forceinline__ void copies_done() { asm volatile("cp.async.wait_all;" ::: "memory"); }

template <class T, int R>
__device__ __forceinline__ void copy_row_async(T *dst, const T *src) {
    constexpr int kBytes = R * (int)sizeof(T);
    if constexpr (kBytes <= 16) {
        copy_async<kBytes>(dst, src);
    } else {
#pragma unroll
        for (int k = 0; k < kBytes / 16; k++) copy_async<16>(dst + k * (16 / sizeof(T)), src + k * (16 / sizeof(T)));
    }
}

__device__ __forceinline__ unsigned tile_now() {   // (differences of up to four seconds)
    unsigned t;
    asm volatile("mov.u32 %0, %%globaltimer_lo;" : "=r"(t));
    return t;
}

// waits for the barrier's phase, at most wait_ns by the lane's own clock: lanes may disagree, so no control
// flow that the lanes of a warp take together may follow from one lane's answer
__device__ __forceinline__ bool tile_wait(uint32_t mbar, uint32_t parity, unsigned wait_ns) {
    unsigned t0 = 0;
    bool first = true;
    for (;;) {
        uint32_t done;
        asm volatile(
            "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}"
            : "=r"(done)
            : "r"(mbar), "r"(parity)
            : "memory");
        if (done) return true;
        const unsigned t = tile_now();
        if (first) { t0 = t; first = false; }
        if (t - t0 >= wait_ns) return false;
    }
}

// NC of the R components are live (three right-hand sides are padded to four; the pad stays zero)
template <class T, int R, int NC>
__global__ void __launch_bounds__(kTileThreads, sizeof(T) == 4 ? 3 : 2) tile_kernel(const TileArgs<T> a) {
    extern __shared__ __align__(128) unsigned char sm[];
    __shared__ int s_info[kTileInfo];
    __shared__ __align__(8) unsigned long long s_bar[kTileWarps * kTileRing], s_step;
    unsigned char *ring = sm;
    T *sx = reinterpret_cast<T *>(sm + (size_t)kTileWarps * a.ring * a.gbytes);
    T *sb = sx + (size_t)a.maxloc * R;
    int *srow = reinterpret_cast<int *>(sb + (size_t)a.maxcomp * R);
    int *scum = srow + a.maxloc;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    if (tid < kTileInfo) s_info[tid] = __ldg(a.info + (size_t)blockIdx.x * kTileInfo + tid);
    if (tid == 0)
        asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"((uint32_t)__cvta_generic_to_shared(&s_step)),
                     "r"(a.arrivals)
                     : "memory");
    if (tid < kTileWarps * a.ring) {
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"((uint32_t)__cvta_generic_to_shared(s_bar + tid))
                     : "memory");
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    // (their strides and lengths are multiples of four)
    for (int i = 4 * tid; i < a.maxloc; i += 4 * kTileThreads) copy_async<16>(srow + i, a.loc + (size_t)blockIdx.x * a.maxloc + i);
    for (int i = 4 * tid; i < a.maxgrp; i += 4 * kTileThreads) copy_async<16>(scum + i, a.cum + (size_t)blockIdx.x * a.maxgrp + i);
    copies_done();
    __syncthreads();
    const int nloc = s_info[0], ncomp = s_info[1], nown = s_info[2];
    const int gend = a.residual ? s_info[5 + a.nsteps] : (a.nsteps > 0 ? s_info[5 + a.nsteps - 1] : 0);
    const unsigned char *src = a.stream + (size_t)s_info[3] * kHead<T> + (size_t)s_info[4] * kQuad<T>;
    // lane 0 fetches the warp's group g into its ring's place `at`
    auto fetch = [&](int g, int at) {
        const int q0 = scum[g], q1 = scum[g + 1];
        const unsigned bytes = (unsigned)(kHead<T> + (q1 - q0) * kQuad<T>);
        const uint32_t mb = (uint32_t)__cvta_generic_to_shared(s_bar + warp * a.ring + at);
        const uint32_t dst = (uint32_t)__cvta_generic_to_shared(ring + (size_t)(warp * a.ring + at) * a.gbytes);
        asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(mb), "r"(bytes) : "memory");
        asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(dst),
                     "l"(src + (size_t)g * kHead<T> + (size_t)q0 * kQuad<T>), "r"(bytes), "r"(mb)
                     : "memory");
    };
    if (lane == 0)
        for (int k = 0; k < a.ring; k++)
            if (warp + k * kTileWarps < gend) fetch(warp + k * kTileWarps, k);
    grid_dep_wait();
    grid_dep_launch();
    auto part_of = [&](int row) {
        int part = 0;
#pragma unroll
        for (int q = 0; q < kTileParts - 1; q++) part += row >= a.bound[q];
        return part;
    };
    for (int i = tid; i < nloc; i += kTileThreads) {
        const int row = srow[i], part = part_of(row);
        if (!((a.zero >> part) & 1u)) {
            copy_row_async<T, R>(sx + (size_t)i * R, (((a.cur >> part) & 1u) ? a.buf[1] : a.buf[0]) + (size_t)row * R);
        } else {
            T v[R];
#pragma unroll
            for (int c = 0; c < R; c++) v[c] = T(0);
            st_row<T, R>(sx + (size_t)i * R, v);
        }
        if (i < ncomp) copy_row_async<T, R>(sb + (size_t)i * R, a.b + (size_t)row * R);
    }
    if (a.prolong)
        for (int i = tid; i < nloc; i += kTileThreads) {   // (the thread's own rows of the loop above)
            const int row = srow[i];
            if (!((a.prolong >> part_of(row)) & 1u)) continue;
            const int np = 1 << __ldg(a.npl2 + row);
            const int4 p0 = __ldg(reinterpret_cast<const int4 *>(a.par + 8 * (size_t)row));
            const int4 p1 = __ldg(reinterpret_cast<const int4 *>(a.par + 8 * (size_t)row) + 1);
            const int q[8] = {p0.x, p0.y, p0.z, p0.w, p1.x, p1.y, p1.z, p1.w};
            T acc[R], v[R];
#pragma unroll
            for (int c = 0; c < R; c++) acc[c] = T(0);
#pragma unroll
            for (int k = 0; k < 8; k++)
                if (k < np) {
                    T e[R];
                    ld_row<T, R>(a.xc + (size_t)q[k] * R, e);
#pragma unroll
                    for (int c = 0; c < R; c++) acc[c] += e[c];
                }
            const T w = T(1) / T(np);
            copies_done();
            ld_row<T, R>(sx + (size_t)i * R, v);
#pragma unroll
            for (int c = 0; c < R; c++) v[c] += w * acc[c];
            st_row<T, R>(sx + (size_t)i * R, v);
        }
    // The warp's next group: everything that does not depend on x is read while the warp waits for the
    // others at the barrier in front of its step, so that behind it only the gathers of x, the sums and the
    // update remain.
    constexpr int KP = 8;
    constexpr unsigned kFull = 0xffffffffu;
    const int comp = lane & 3;
    int g = warp, at = 0, K = 0, slot = kTileNoRow;
    unsigned phase = 0, j[KP];
    T d = T(0), bv = T(0), v[KP];
    bool ok = true, stale = false;
    auto place = [&]() { return ring + (size_t)(warp * a.ring + at) * a.gbytes; };
    auto arrived = [&]() { return tile_wait((uint32_t)__cvta_generic_to_shared(s_bar + warp * a.ring + at), phase, a.wait_ns); };
    auto read_ahead = [&]() {
        stale = false;
        if (g >= gend || !ok) return;
        K = scum[g + 1] - scum[g];
        if (!__all_sync(kFull, arrived())) {
            ok = false;
            if (lane == 0) atomicExch(a.status, 1);
            return;
        }
        const unsigned char *p = place(), *e = p + kHead<T>;
        slot = reinterpret_cast<const uint16_t *>(p)[lane >> 2];
        d = reinterpret_cast<const T *>(p + 2 * kTileRows)[lane >> 2];
        const unsigned own = slot == kTileNoRow ? 0u : (unsigned)slot;
#pragma unroll
        for (int k = 0; k < KP; k++) {   // (absent entries: the row's own value times zero, like the pads)
            j[k] = own;
            v[k] = T(0);
            if (k < K) {
                j[k] = reinterpret_cast<const uint16_t *>(e + k * kQuad<T>)[lane];
                v[k] = reinterpret_cast<const T *>(e + k * kQuad<T> + 64)[lane];
            }
        }
    };
    auto rhs = [&]() { bv = slot != kTileNoRow && comp < NC ? sb[slot * R + comp] : T(0); };
    // lane c < NC of a row returns component c of b - A x
    auto row_sum = [&]() -> T {
        T ac[R];
#pragma unroll
        for (int c = 0; c < R; c++) ac[c] = T(0);
        auto some = [&](auto from, auto count) {
            constexpr int k0 = decltype(from)::value, n = decltype(count)::value;
            T x[n][R];
#pragma unroll
            for (int k = 0; k < n; k++) ld_row<T, R>(sx + j[k0 + k] * R, x[k]);
#pragma unroll
            for (int k = 0; k < n; k++)
#pragma unroll
                for (int c = 0; c < NC; c++) ac[c] = fma(v[k0 + k], x[k][c], ac[c]);
        };
        if constexpr (sizeof(T) == 4) {
            if (K > 4) some(Int<0>(), Int<8>());
            else some(Int<0>(), Int<4>());
        } else {   // the FP64 pipe is the bound: no absent entries
            some(Int<0>(), Int<1>());
            if (K > 1) some(Int<1>(), Int<1>());
            if (K > 2) some(Int<2>(), Int<1>());
            if (K > 3) some(Int<3>(), Int<1>());
            if (K > 4) some(Int<4>(), Int<1>());
            if (K > 5) some(Int<5>(), Int<1>());
            if (K > 6) some(Int<6>(), Int<1>());
            if (K > 7) some(Int<7>(), Int<1>());
        }
        const unsigned char *e = place() + kHead<T> + KP * kQuad<T>;
        for (int k = KP; k < K; k++, e += kQuad<T>) {   // rows of more than 32 entries
            T x[R];
            ld_row<T, R>(sx + reinterpret_cast<const uint16_t *>(e)[lane] * R, x);
            const T ev = reinterpret_cast<const T *>(e + 64)[lane];
#pragma unroll
            for (int c = 0; c < NC; c++) ac[c] = fma(ev, x[c], ac[c]);
        }
        T sum;
        if constexpr (R == 4) {
            const bool hi = comp & 2, odd = comp & 1;
            T k0 = hi ? ac[2] : ac[0], k1 = hi ? ac[3] : ac[1];
            const T g0s = hi ? ac[0] : ac[2], g1s = hi ? ac[1] : ac[3];
            k0 += __shfl_xor_sync(kFull, g0s, 2);
            k1 += __shfl_xor_sync(kFull, g1s, 2);
            const T give = odd ? k0 : k1;
            sum = (odd ? k1 : k0) + __shfl_xor_sync(kFull, give, 1);
        } else if constexpr (R == 2) {
            const bool odd = comp & 1;
            const T give = odd ? ac[0] : ac[1];
            sum = (odd ? ac[1] : ac[0]) + __shfl_xor_sync(kFull, give, 1);
            sum += __shfl_xor_sync(kFull, sum, 2);
        } else {
            sum = ac[0] + __shfl_xor_sync(kFull, ac[0], 1);
            sum += __shfl_xor_sync(kFull, sum, 2);
        }
        return bv - sum;
    };
    auto next = [&](int e) {   // the group's place is free: refill it, and go on to the warp's next group
        __syncwarp();
        if (lane == 0 && g + a.ring * kTileWarps < gend) fetch(g + a.ring * kTileWarps, at);
        g += kTileWarps;
        if (++at == a.ring) { at = 0; phase ^= 1u; }
        stale = true;
        if (g < e) { read_ahead(); rhs(); }
    };
    const uint32_t sbar = (uint32_t)__cvta_generic_to_shared(&s_step);
    unsigned step_ns = a.wait_ns;
    read_ahead();
    copies_done();
    __syncthreads();
    rhs();
    int e = s_info[5];
    for (int s = 0; s < a.nsteps; s++) {
        while (g < e && ok) {
            T *xp = sx + (slot != kTileNoRow ? slot * R : 0) + comp;
            const T xo = comp < R ? *xp : T(0);
            const T res = row_sum();
            if (slot != kTileNoRow && comp < NC) *xp = xo + res * d;
            next(e);
        }
        __syncwarp();
        if (lane == 0) asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(sbar) : "memory");
        e = s_info[5 + s + 1];
        if (stale) { read_ahead(); rhs(); }
        // A lane whose wait expires goes on with the others (the loops above take the lanes of a warp together):
        // what it reads is invalid but in place, and it does not wait at the steps that are left.
        if (!tile_wait(sbar, s & 1, step_ns)) {
            step_ns = 0;
            atomicExch(a.status, 1);
        }
    }
    if (a.nsteps > 0)
        for (int i = tid; i < nown; i += kTileThreads) {
            T w[R];
            ld_row<T, R>(sx + (size_t)i * R, w);
            st_row<T, R>(a.xout + (size_t)srow[i] * R, w);
        }
    while (g < gend && ok) {   // the residual of the own rows
        const T res = row_sum();
        if (slot != kTileNoRow && comp < NC) {
            T *r = a.r + (size_t)srow[slot] * R + comp;
            *r = res;
            if (NC < R && comp == NC - 1) r[1] = T(0);   // the pad
        }
        next(gend);
    }
    if (!ok)   // what is still on its way gets one more bounded wait before the block leaves
        for (int k = 0; k < a.ring && g < gend; k++) {
            arrived();
            g += kTileWarps;
            if (++at == a.ring) { at = 0; phase ^= 1u; }
        }
}

// the static part of a plan's stream, once: slots and columns (one thread per entry, then per row)
template <class T>
__global__ void tile_layout_kernel(int64_t quads, int64_t groups, const int *__restrict__ qgroup,
                                   const uint16_t *__restrict__ col, const uint16_t *__restrict__ slot,
                                   const int64_t *__restrict__ gquad, unsigned char *__restrict__ out) {
    const int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (k < 32 * quads) {
        const int64_t q = k >> 5;
        const size_t at = (size_t)(__ldg(qgroup + q) + 1) * kHead<T> + (size_t)q * kQuad<T>;
        reinterpret_cast<uint16_t *>(out + at)[k & 31] = col[k];
    }
    if (k < kTileRows * groups) {
        const int64_t g = k / kTileRows;
        const size_t at = (size_t)g * kHead<T> + (size_t)gquad[g] * kQuad<T>;
        reinterpret_cast<uint16_t *>(out + at)[k % kTileRows] = slot[k];
    }
}

// matrix values and inverse diagonals of both precisions into the streams
__global__ void tile_fill_kernel(int64_t quads, int64_t groups, const int *__restrict__ qgroup,
                                 const int64_t *__restrict__ gquad, const int *__restrict__ map,
                                 const int *__restrict__ row, const float *__restrict__ A32,
                                 const double *__restrict__ A64, const float *__restrict__ d32,
                                 const double *__restrict__ d64, unsigned char *__restrict__ s32,
                                 unsigned char *__restrict__ s64) {
    const int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (k < 32 * quads) {
        const int64_t q = k >> 5;
        const int src = __ldg(map + k);
        const size_t g = (size_t)(__ldg(qgroup + q) + 1);
        reinterpret_cast<float *>(s32 + g * kHead<float> + (size_t)q * kQuad<float> + 64)[k & 31] =
            src >= 0 ? __ldg(A32 + src) : 0.f;
        reinterpret_cast<double *>(s64 + g * kHead<double> + (size_t)q * kQuad<double> + 64)[k & 31] =
            src >= 0 ? __ldg(A64 + src) : 0.0;
    }
    if (k < kTileRows * groups) {
        const int64_t g = k / kTileRows;
        const int i = __ldg(row + k), l = (int)(k % kTileRows);
        const size_t q = (size_t)__ldg(gquad + g);
        reinterpret_cast<float *>(s32 + g * kHead<float> + q * kQuad<float> + 2 * kTileRows)[l] = i >= 0 ? d32[i] : 0.f;
        reinterpret_cast<double *>(s64 + g * kHead<double> + q * kQuad<double> + 2 * kTileRows)[l] = i >= 0 ? d64[i] : 0.0;
    }
}

template <class T> const unsigned char *tile_stream(const TileDev &t);
template <> const unsigned char *tile_stream<float>(const TileDev &t) { return t.s32; }
template <> const unsigned char *tile_stream<double>(const TileDev &t) { return t.s64; }

// shared memory of a block: x and b rows, row and quad tables, and `ring` groups per warp
template <class T>
size_t tile_smem(const TileDev &t, int R, int ring) {
    return (size_t)kTileWarps * ring * (kHead<T> + t.maxquads * kQuad<T>) + (size_t)(t.maxloc + t.maxcomp) * R * sizeof(T) +
           (size_t)(t.maxloc + t.maxgrp) * sizeof(int);
}

constexpr int kTileStatic = 3072;   // upper bound of the kernel's static shared memory and the system's share

// Groups in flight per warp.  A group takes about a microsecond to arrive, longer than a step on a small
// level, so a tile is fetched whole where that leaves room for the blocks the launch has per SM; on large
// levels three or two blocks share an SM, each with at least two groups per warp on their way.
template <class T>
int tile_ring(const TileDev &t, int R, int sms, int sm_bytes, int block_bytes, bool &at_once) {
    const int whole = std::min(kTileRing, (t.maxgrp + kTileWarps - 1) / kTileWarps);
    auto fits = [&](int ring, int blocks) {
        const size_t need = tile_smem<T>(t, R, ring);
        return (need + kTileStatic) * blocks <= (size_t)sm_bytes && need + kTileStatic <= (size_t)block_bytes;
    };
    const int want = std::max(1, std::min(3, (t.ntile + sms - 1) / sms));
    for (int blocks = want; blocks >= 1; blocks--)
        for (int ring = whole; ring >= (blocks == 1 ? 1 : std::min(whole, 2)); ring--)
            if (fits(ring, blocks)) { at_once = blocks == want; return ring; }
    return 0;
}

template <class T, int R, int NC>
bool allow_smem(int bytes) {
    return cudaFuncSetAttribute(tile_kernel<T, R, NC>, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes) == cudaSuccess;
}

struct SmemLimits { int sm = 0, block = 0, sms = 0; };
bool smem_limits(SmemLimits &l) {
    int dev = 0;
    return cudaGetDevice(&dev) == cudaSuccess &&
           cudaDeviceGetAttribute(&l.sms, cudaDevAttrMultiProcessorCount, dev) == cudaSuccess &&
           cudaDeviceGetAttribute(&l.sm, cudaDevAttrMaxSharedMemoryPerMultiprocessor, dev) == cudaSuccess &&
           cudaDeviceGetAttribute(&l.block, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev) == cudaSuccess;
}

}  // namespace

// The kernels' dynamic shared-memory limit is set to what the device offers a block, always the same
// value, so handles and threads cannot take it away from one another.
bool tile_setup() {
    SmemLimits l;
    if (!smem_limits(l)) { cudaGetLastError(); return false; }
    const int bytes = l.block - kTileStatic;
    if (!allow_smem<float, 1, 1>(bytes) || !allow_smem<float, 2, 2>(bytes) || !allow_smem<float, 4, 3>(bytes) ||
        !allow_smem<float, 4, 4>(bytes) || !allow_smem<double, 1, 1>(bytes) || !allow_smem<double, 2, 2>(bytes) ||
        !allow_smem<double, 4, 3>(bytes) || !allow_smem<double, 4, 4>(bytes)) {
        cudaGetLastError();
        return false;
    }
    return true;
}

// the plan's sizes as launches will see them, and whether every kind of launch fits a block
bool tile_fits(const TilePlan &p, TileDev &t) {
    t.ntile = p.ntile; t.nsteps = p.nsteps;
    t.maxloc = (p.maxloc + 3) / 4 * 4; t.maxcomp = (p.maxcomp + 3) / 4 * 4;
    t.maxgrp = (p.maxgrp + 1 + 3) / 4 * 4;   // quads before each group, and of all
    t.maxquads = p.maxquads;
    t.groups = p.groups; t.quads = p.quads;
    SmemLimits l;
    if (!smem_limits(l)) { cudaGetLastError(); return false; }
    const int rs[3] = {1, 2, 4};
    for (int q = 0; q < 3; q++) {
        t.ring[0][q] = tile_ring<float>(t, rs[q], l.sms, l.sm, l.block, t.at_once[0][q]);
        t.ring[1][q] = tile_ring<double>(t, rs[q], l.sms, l.sm, l.block, t.at_once[1][q]);
        if (t.ring[0][q] < 1 || t.ring[1][q] < 1) return false;
    }
    return true;
}

cudaError_t launch_tile_layout(const TileDev &t, const uint16_t *col, const uint16_t *slot, cudaStream_t s) {
    const int64_t n = std::max(32 * t.quads, kTileRows * t.groups);
    if (n == 0) return cudaSuccess;
    const unsigned blocks = (unsigned)((n + 255) / 256);
    tile_layout_kernel<float><<<blocks, 256, 0, s>>>(t.quads, t.groups, t.qgroup, col, slot, t.gquad, t.s32);
    tile_layout_kernel<double><<<blocks, 256, 0, s>>>(t.quads, t.groups, t.qgroup, col, slot, t.gquad, t.s64);
    return cudaGetLastError();
}

size_t tile_stream_bytes(const TileDev &t, bool fp64) {
    return fp64 ? (size_t)t.groups * kHead<double> + (size_t)t.quads * kQuad<double>
                : (size_t)t.groups * kHead<float> + (size_t)t.quads * kQuad<float>;
}

static void fill(const DevLevel &L, const TileDev &t, cudaStream_t s) {
    const int64_t n = std::max(32 * t.quads, kTileRows * t.groups);
    if (n)
        tile_fill_kernel<<<(unsigned)((n + 255) / 256), 256, 0, s>>>(t.quads, t.groups, t.qgroup, t.gquad, t.map, t.row,
                                                                     L.A32, L.A64, L.dinv32, L.dinv64, t.s32, t.s64);
}

void launch_tile_fill(const DevLevel &L, cudaStream_t s) {
    for (int q = 0; q < 2; q++)
        for (int p = 0; p < L.tparts; p++) fill(L, L.tile[q][p], s);
    if (L.tparts > 0 && !L.tfused) fill(L, L.tres, s);
}

template <class T>
static void launch_tile(const DevLevel &L, const TileDev &t, int part, const TileVec<T> &v, const T *b, T *r, int R,
                        const Ctx &c, cudaStream_t s, Chain *ch) {
    TileArgs<T> a;
    a.info = t.info; a.loc = t.loc; a.cum = t.cum; a.stream = tile_stream<T>(t);
    a.nsteps = t.nsteps; a.maxloc = t.maxloc; a.maxcomp = t.maxcomp; a.maxgrp = t.maxgrp;
    a.gbytes = kHead<T> + t.maxquads * kQuad<T>;
    a.ring = t.ring[sizeof(T) == 8][R >> 1];
    a.residual = r != nullptr;
    a.b = b;
    a.buf[0] = v.x; a.buf[1] = v.y;
    a.cur = v.cur; a.zero = v.zero; a.prolong = v.xc ? v.prolong : 0u;
    const int per = 8 / L.tparts;
    for (int q = 0; q + 1 < kTileParts; q++) a.bound[q] = q + 1 < L.tparts ? L.cs[(q + 1) * per] : L.n;
    a.xout = ((v.cur >> part) & 1u) ? v.x : v.y;
    a.xc = v.xc; a.par = L.par; a.npl2 = L.npl2; a.r = r;
    a.status = c.narrow.status;
    a.arrivals = kTileWarps + std::min(c.barrier_phantoms, 1024);   // (a barrier counts to 2^20)
    a.wait_ns = c.barrier_phantoms > 0 ? kTilePhantomWaitNs : kTileWaitNs;
    auto k = R == 1 ? tile_kernel<T, 1, 1> : R == 2 ? tile_kernel<T, 2, 2>
             : c.lanes == 3 ? tile_kernel<T, 4, 3> : tile_kernel<T, 4, 4>;
    klaunch(k, (unsigned)t.ntile, (unsigned)kTileThreads, tile_smem<T>(t, R, a.ring), s, ch, a);
}

template <class T>
void launch_tile_sweep(const Ctx &c, const DevLevel &L, bool forward, TileVec<T> &v, const T *b, T *r, int R,
                       cudaStream_t s, Chain *ch) {
    const int dir = forward ? 0 : 1;
    for (int q = 0; q < L.tparts; q++) {
        const int part = forward ? q : L.tparts - 1 - q;
        launch_tile<T>(L, L.tile[dir][part], part, v, b, L.tfused ? r : (T *)nullptr, R, c, s, ch);
        v.cur ^= 1u << part;
        v.zero &= ~(1u << part);
        v.prolong &= ~(1u << part);
    }
    if (r && !L.tfused) launch_tile<T>(L, L.tres, 0, v, b, r, R, c, s, ch);
}

template void launch_tile_sweep<float>(const Ctx &, const DevLevel &, bool, TileVec<float> &, const float *, float *, int,
                                       cudaStream_t, Chain *);
template void launch_tile_sweep<double>(const Ctx &, const DevLevel &, bool, TileVec<double> &, const double *, double *,
                                        int, cudaStream_t, Chain *);

}  // namespace lbmg

// relax.cu -- multigrid kernels of the V-cycle (Chuang & Kazhdan, Sections 4.3
// and 5.2): coloured Gauss-Seidel and weighted-Jacobi relaxation, residual,
// restriction P^T r, prolongation x += P e, the coarsest-level dense solve, and
// small vector kernels.  Vectors are row-major [n][R], R in {1, 2, 4}.
//
// Rows of one colour (one corner parity class) never couple, because supports
// of equal-parity corners are disjoint and the components of one corner are
// disjoint, so a colour is relaxed in parallel with exact Gauss-Seidel updates.
// A group of G threads shares one matrix row.
#include <algorithm>

#include "lbmg_internal.h"

namespace lbmg {

template <class T, int R>
__device__ __forceinline__ void load_vec(const T *__restrict__ p, T (&v)[R]) {
#pragma unroll
    for (int r = 0; r < R; r++) v[r] = p[r];
}
template <>
__device__ __forceinline__ void load_vec<float, 4>(const float *__restrict__ p, float (&v)[4]) {
    const float4 q = __ldg(reinterpret_cast<const float4 *>(p));
    v[0] = q.x; v[1] = q.y; v[2] = q.z; v[3] = q.w;
}
template <>
__device__ __forceinline__ void load_vec<double, 2>(const double *__restrict__ p, double (&v)[2]) {
    const double2 q = __ldg(reinterpret_cast<const double2 *>(p));
    v[0] = q.x; v[1] = q.y;
}
template <>
__device__ __forceinline__ void load_vec<double, 4>(const double *__restrict__ p, double (&v)[4]) {
    const double2 q0 = __ldg(reinterpret_cast<const double2 *>(p));
    const double2 q1 = __ldg(reinterpret_cast<const double2 *>(p) + 1);
    v[0] = q0.x; v[1] = q0.y; v[2] = q1.x; v[3] = q1.y;
}

// x may be written by other rows of the same launch only at rows of the same
// colour, which this row never reads, so plain (non-__ldg) loads are not needed
// for correctness; __ldg is avoided anyway for x because the GS kernel writes it.
template <class T, int R>
__device__ __forceinline__ void load_x(const T *p, T (&v)[R]) {
#pragma unroll
    for (int r = 0; r < R; r++) v[r] = p[r];
}

template <>
__device__ __forceinline__ void load_x<float, 4>(const float *p, float (&v)[4]) {
    const float4 q = *reinterpret_cast<const float4 *>(p);
    v[0] = q.x; v[1] = q.y; v[2] = q.z; v[3] = q.w;
}
template <>
__device__ __forceinline__ void load_x<double, 2>(const double *p, double (&v)[2]) {
    const double2 q = *reinterpret_cast<const double2 *>(p);
    v[0] = q.x; v[1] = q.y;
}
template <>
__device__ __forceinline__ void load_x<double, 4>(const double *p, double (&v)[4]) {
    const double2 q0 = reinterpret_cast<const double2 *>(p)[0], q1 = reinterpret_cast<const double2 *>(p)[1];
    v[0] = q0.x; v[1] = q0.y; v[2] = q1.x; v[3] = q1.y;
}

// The static part of a matrix row (pattern and values) is loaded before the
// kernel waits for its predecessor: each of the G threads of a row keeps its first
// P entries in registers, so after the wait only the x gathers remain.
template <class T, int G>
struct RowPrefetch {
    static constexpr int P = 32 / G;
    int k = 0, k1 = 0;
    int j[P];
    T a[P];
    __device__ __forceinline__ void load(int row, bool active, int lane, const int *__restrict__ rp,
                                         const int *__restrict__ ci, const T *__restrict__ A) {
        if (active) { k = __ldg(rp + row) + lane; k1 = __ldg(rp + row + 1); }
#pragma unroll
        for (int q = 0; q < P; q++) {
            const int kk = k + q * G;
            if (kk < k1) { j[q] = __ldg(ci + kk); a[q] = __ldg(A + kk); }
            else { j[q] = -1; a[q] = T(0); }
        }
    }
    template <int R>
    __device__ __forceinline__ void dot(const int *__restrict__ ci, const T *__restrict__ A, const T *x,
                                        T (&acc)[R]) const {
#pragma unroll
        for (int r = 0; r < R; r++) acc[r] = T(0);
#pragma unroll
        for (int q = 0; q < P; q++) {
            if (j[q] >= 0) {
                T xv[R];
                load_x<T, R>(x + (size_t)j[q] * R, xv);
#pragma unroll
                for (int r = 0; r < R; r++) acc[r] = fma(a[q], xv[r], acc[r]);
            }
        }
        for (int kk = k + P * G; kk < k1; kk += G) {
            const int jj = __ldg(ci + kk);
            const T aa = __ldg(A + kk);
            T xv[R];
            load_x<T, R>(x + (size_t)jj * R, xv);
#pragma unroll
            for (int r = 0; r < R; r++) acc[r] = fma(aa, xv[r], acc[r]);
        }
    }
};

template <class T, int R, int G>
__device__ __forceinline__ void group_sum(T (&acc)[R]) {
#pragma unroll
    for (int o = G / 2; o > 0; o >>= 1)
#pragma unroll
        for (int r = 0; r < R; r++) acc[r] += __shfl_xor_sync(0xffffffffu, acc[r], o, G);
}

// sums of the components over a warp, halved across its lanes so that an FP64 sum takes 6 additions of 4
// components instead of 20 (an SM's FP64 pipe takes a warp instruction in 16 cycles): one lane per component
// returns its sum and the component in comp, the others -1
template <class T, int R>
__device__ __forceinline__ T warp_sum(const T (&a)[R], int lane, int &comp) {
    constexpr unsigned kFull = 0xffffffffu;
    T v;
    int from;   // first of the butterfly steps left
    if constexpr (R == 4) {
        const bool hi = lane & 16, odd = lane & 8;
        T a0 = hi ? a[2] : a[0], a1 = hi ? a[3] : a[1];
        const T g0 = hi ? a[0] : a[2], g1 = hi ? a[1] : a[3];
        a0 += __shfl_xor_sync(kFull, g0, 16);
        a1 += __shfl_xor_sync(kFull, g1, 16);
        const T give = odd ? a0 : a1;
        v = (odd ? a1 : a0) + __shfl_xor_sync(kFull, give, 8);
        from = 4;
        comp = (lane & 7) == 0 ? lane >> 3 : -1;
    } else if constexpr (R == 2) {
        const bool hi = lane & 16;
        const T give = hi ? a[0] : a[1];
        v = (hi ? a[1] : a[0]) + __shfl_xor_sync(kFull, give, 16);
        from = 8;
        comp = (lane & 15) == 0 ? lane >> 4 : -1;
    } else {
        v = a[0];
        from = 16;
        comp = lane == 0 ? 0 : -1;
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1)
        if (o <= from) v += __shfl_xor_sync(kFull, v, o);
    return v;
}

template <class T, int R, int G>
__global__ void __launch_bounds__(512) smooth_colour_kernel(int r0, int r1, const int *__restrict__ rp,
                                                            const int *__restrict__ ci, const T *__restrict__ A,
                                                            const T *__restrict__ dinv, const T *__restrict__ b, T *x) {
    const int tid = blockIdx.x * blockDim.x + threadIdx.x;
    const int row = r0 + tid / G, lane = tid % G;
    const bool active = row < r1;
    RowPrefetch<T, G> pf;
    pf.load(row, active, lane, rp, ci, A);
    const T d = (active && lane == 0) ? __ldg(dinv + row) : T(0);
    grid_dep_wait();
    grid_dep_launch();
    T acc[R];
    pf.template dot<R>(ci, A, x, acc);
    group_sum<T, R, G>(acc);
    if (active && lane == 0) {
#pragma unroll
        for (int r = 0; r < R; r++) x[(size_t)row * R + r] += (b[(size_t)row * R + r] - acc[r]) * d;
    }
}

template <class T, int R, int G>
__global__ void __launch_bounds__(512) residual_kernel(int n, const int *__restrict__ rp, const int *__restrict__ ci,
                                                       const T *__restrict__ A, const T *__restrict__ b,
                                                       const T *x, T *__restrict__ r) {
    const int tid = blockIdx.x * blockDim.x + threadIdx.x;
    const int row = tid / G, lane = tid % G;
    const bool active = row < n;
    RowPrefetch<T, G> pf;
    pf.load(row, active, lane, rp, ci, A);
    grid_dep_wait();
    grid_dep_launch();
    T acc[R];
    pf.template dot<R>(ci, A, x, acc);
    group_sum<T, R, G>(acc);
    if (active && lane == 0) {
#pragma unroll
        for (int q = 0; q < R; q++) r[(size_t)row * R + q] = b[(size_t)row * R + q] - acc[q];
    }
}

// kernel instance for (R, threads per row); nullptr for an unsupported pair
template <class T>
using SmoothFn = void (*)(int, int, const int *, const int *, const T *, const T *, const T *, T *);
template <class T>
using ResidualFn = void (*)(int, const int *, const int *, const T *, const T *, const T *, T *);

template <class T, int R>
SmoothFn<T> smooth_fn(int tpr) {
    switch (tpr) {
        case 4: return smooth_colour_kernel<T, R, 4>;
        case 8: return smooth_colour_kernel<T, R, 8>;
        case 16: return smooth_colour_kernel<T, R, 16>;
        default: return nullptr;
    }
}
template <class T, int R>
ResidualFn<T> residual_fn(int tpr) {
    switch (tpr) {
        case 4: return residual_kernel<T, R, 4>;
        case 8: return residual_kernel<T, R, 8>;
        case 16: return residual_kernel<T, R, 16>;
        default: return nullptr;
    }
}

template <class T>
void launch_sweeps(const Ctx &c, const DevLevel &L, int sweeps, bool forward, const T *A, const T *dinv, const T *b,
                   T *x, int R, cudaStream_t s, Chain *ch, int skip, bool from_zero) {
    if (sweeps <= 0) return;
    skip = std::max(0, std::min(skip, 8));
    const LaunchShape &sh = L.shape[sizeof(T) == 8][kShapeSmooth];
    if (sizeof(T) == 4 && sh.tpb == kSweepShapeTpb && 8 * sweeps <= 32 && c.sweep_bar && A == (const T *)L.A32) {
        int seq[32];
        for (int q = skip; q < 8 * sweeps; q++) seq[q - skip] = forward ? q % 8 : 7 - q % 8;
        const int blocks = sh.grid > 0 && sh.grid < c.sweep_blocks[R] ? sh.grid : c.sweep_blocks[R];
        if (ch) ch->cut();   // a cooperative launch takes no programmatic serialisation
        if (launch_packed_sweep(L, seq, 8 * sweeps - skip, (const float *)dinv, (const float *)b, (float *)x, R,
                                c.sweep_bar, c.narrow.status, blocks, s))
            return;
        cudaGetLastError();   // refused: the per-colour launches below
    }
    for (int sw = 0; sw < sweeps; sw++)
        for (int q = sw == 0 ? skip : 0; q < 8; q++) {
            const int colour = forward ? q : 7 - q;
            // the colour that follows on this level: the next of this sweep, or the first of the next sweep
            const int nq = q < 7 ? q + 1 : (sw + 1 < sweeps ? 0 : -1);
            const int next = nq < 0 ? -1 : (forward ? nq : 7 - nq);
            if (from_zero && sw == 0 && forward) {
                const int tpb = sh.tpb;
                if (L.cs[colour + 1] > L.cs[colour])
                    launch_packed_smooth<T>(L, colour, A, dinv, b, x, R, tpb, s, ch, next, L.cs[colour], c.lanes);
            } else {
                launch_smooth_colour<T>(L, colour, A, dinv, b, x, R, s, ch, next, c.lanes);
            }
        }
}

template <class T>
bool sweeps_from_zero(const DevLevel &L) {
    const LaunchShape &sh = L.shape[sizeof(T) == 8][kShapeSmooth];
    return L.pk_map && sh.tpr == 4 && sh.tpb != kSweepShapeTpb;
}

template <class T>
void launch_smooth_colour(const DevLevel &L, int colour, const T *A, const T *dinv, const T *b, T *x, int R,
                          cudaStream_t s, Chain *ch, int next, int lanes) {
    const int r0 = L.cs[colour], r1 = L.cs[colour + 1];
    if (r1 <= r0) return;
    const LaunchShape &sh = L.shape[sizeof(T) == 8][kShapeSmooth];
    // four threads per row: the packed copy of the matrix (one 256-byte load per warp and quad)
    const int tpb = sh.tpb == kSweepShapeTpb ? 256 : sh.tpb;   // one colour of a whole-sweep level
    if (sh.tpr == 4 && launch_packed_smooth<T>(L, colour, A, dinv, b, x, R, tpb, s, ch, next, INT32_MAX, lanes)) return;
    const unsigned blocks = (unsigned)(((int64_t)(r1 - r0) * sh.tpr + tpb - 1) / tpb);
    const SmoothFn<T> k = R == 1 ? smooth_fn<T, 1>(sh.tpr) : R == 2 ? smooth_fn<T, 2>(sh.tpr) : smooth_fn<T, 4>(sh.tpr);
    klaunch(k, blocks, (unsigned)tpb, 0, s, ch, r0, r1, L.rp, L.ci, A, dinv, b, x);
}

template <class T>
void launch_residual(const DevLevel &L, const T *A, const T *b, const T *x, T *r, int R, cudaStream_t s, int nrows,
                     Chain *ch, int lanes) {
    const int n = nrows < 0 ? L.n : nrows;
    if (n == 0) return;
    const LaunchShape &sh = L.shape[sizeof(T) == 8][kShapeResidual];
    if (sh.tpr == 4 && launch_packed_residual<T>(L, A, b, x, r, R, n, sh.tpb, s, ch, lanes)) return;
    const unsigned blocks = (unsigned)(((int64_t)n * sh.tpr + sh.tpb - 1) / sh.tpb);
    const ResidualFn<T> k =
        R == 1 ? residual_fn<T, 1>(sh.tpr) : R == 2 ? residual_fn<T, 2>(sh.tpr) : residual_fn<T, 4>(sh.tpr);
    klaunch(k, blocks, (unsigned)sh.tpb, 0, s, ch, n, L.rp, L.ci, A, b, x, r);
}

template <class T>
__global__ void jacobi_update_kernel(int n, int R, const T *__restrict__ dinv, const T *__restrict__ r, T *x, T omega) {
    const int64_t q = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (q >= (int64_t)n * R) return;
    x[q] += omega * dinv[q / R] * r[q];
}

template <class T>
void launch_jacobi_update(const DevLevel &L, const T *dinv, const T *r, T *x, T omega, int R, cudaStream_t s) {
    const int64_t m = (int64_t)L.ns * R;
    if (m == 0) return;
    jacobi_update_kernel<T><<<(unsigned)((m + 255) / 256), 256, 0, s>>>(L.ns, R, dinv, r, x, omega);
}

// b_c[J] = sum over fine children i of J of r_f[i] / #parents(i); x_c[J] = 0 when x_c is given.
// Eight lanes share a coarse row (14 children on average, up to 60 or so): neighbouring lanes read
// neighbouring list entries, and a row's gathers are three per lane and all in flight together.  One thread
// per row read the lists a row apart and chained its gathers: 46 us from 927k to 232k rows (four FP32
// components) and 8 to 11 us on levels of some thousand rows, where the chain was the time.  Each lane's
// first kPreChildren entries are loaded before the grid-dependency wait.  The components' sums are halved
// across the lanes: lane 4 h + 2 o of a row ends with component 2 h + o.
constexpr int kPreChildren = 3;

template <class T, int R>
__global__ void __launch_bounds__(256) restrict_kernel(int nc, const int *__restrict__ crp,
                                                       const uint32_t *__restrict__ cch, const T *__restrict__ rf,
                                                       T *__restrict__ bc, T *__restrict__ xc,
                                                       const T *__restrict__ dinv, int c1) {
    const int tid = blockIdx.x * blockDim.x + threadIdx.x;
    const int J = tid >> 3, l = tid & 7;
    const bool active = J < nc;
    int k0 = 0, k1 = 0;
    uint32_t e[kPreChildren];
    if (active) { k0 = __ldg(crp + J) + l; k1 = __ldg(crp + J + 1); }
    // colour 0 (rows [0, c1)) of the first sweep, fused: its inverse diagonal
    const T d = (active && dinv && J < c1) ? __ldg(dinv + J) : T(0);
#pragma unroll
    for (int u = 0; u < kPreChildren; u++) e[u] = k0 + 8 * u < k1 ? __ldg(cch + k0 + 8 * u) : 0u;
    grid_dep_wait();
    grid_dep_launch();
    T acc[R];
#pragma unroll
    for (int r = 0; r < R; r++) acc[r] = T(0);
    auto child = [&](uint32_t ek) {
        const T w = T(1) / T(1u << (ek >> kPackShift));
        T v[R];
        load_x<T, R>(rf + (size_t)(ek & kPackMask) * R, v);
#pragma unroll
        for (int r = 0; r < R; r++) acc[r] = fma(w, v[r], acc[r]);
    };
#pragma unroll
    for (int u = 0; u < kPreChildren; u++)
        if (k0 + 8 * u < k1) child(e[u]);
    for (int k = k0 + 8 * kPreChildren; k < k1; k += 8) child(__ldg(cch + k));
    constexpr unsigned kFull = 0xffffffffu;
    T v;
    int comp;
    bool writes;
    if constexpr (R == 4) {
        const bool hi = l & 4, odd = l & 2;
        T a0 = hi ? acc[2] : acc[0], a1 = hi ? acc[3] : acc[1];
        const T g0 = hi ? acc[0] : acc[2], g1 = hi ? acc[1] : acc[3];
        a0 += __shfl_xor_sync(kFull, g0, 4);
        a1 += __shfl_xor_sync(kFull, g1, 4);
        const T give = odd ? a0 : a1;
        v = (odd ? a1 : a0) + __shfl_xor_sync(kFull, give, 2);
        comp = l >> 1;
        writes = (l & 1) == 0;
    } else if constexpr (R == 2) {
        const bool hi = l & 4;
        const T give = hi ? acc[0] : acc[1];
        v = (hi ? acc[1] : acc[0]) + __shfl_xor_sync(kFull, give, 4);
        v += __shfl_xor_sync(kFull, v, 2);
        comp = l >> 2;
        writes = (l & 3) == 0;
    } else {
        v = acc[0] + __shfl_xor_sync(kFull, acc[0], 4);
        v += __shfl_xor_sync(kFull, v, 2);
        comp = 0;
        writes = l == 0;
    }
    v += __shfl_xor_sync(kFull, v, 1);
    if (!active || !writes) return;
    bc[(size_t)J * R + comp] = v;
    // the colour kernels' step x = x + (b - A x) / a_ii with x = 0 (so A x = +0): 0 + b d
    if (xc) xc[(size_t)J * R + comp] = dinv && J < c1 ? T(0) + (v - T(0)) * d : T(0);
}

template <class T>
void launch_restrict(const DevLevel &Lc, const T *rf, T *bc, int R, cudaStream_t s, T *xc, Chain *ch,
                     bool first_colour) {
    if (Lc.n == 0) return;
    const unsigned blocks = (unsigned)(((int64_t)Lc.n * 8 + 255) / 256);
    auto k = R == 1 ? restrict_kernel<T, 1> : R == 2 ? restrict_kernel<T, 2> : restrict_kernel<T, 4>;
    const T *dinv = first_colour && xc ? (sizeof(T) == 4 ? (const T *)Lc.dinv32 : (const T *)Lc.dinv64) : nullptr;
    klaunch(k, blocks, 256u, 0, s, ch, Lc.n, Lc.crp, Lc.cch, rf, bc, xc, dinv, dinv ? Lc.cs[1] : 0);
}

// x_f[i] += (sum of parent values) / #parents(i)
template <class T, int R>
__global__ void prolong_add_kernel(int nf, const int *__restrict__ par, const int8_t *__restrict__ npl2,
                                   const T *__restrict__ xc, T *__restrict__ xf) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    const bool active = i < nf;
    int np = 0, p[8];
    if (active) {
        np = 1 << __ldg(npl2 + i);
        const int4 p0 = __ldg(reinterpret_cast<const int4 *>(par + 8 * (size_t)i));
        const int4 p1 = __ldg(reinterpret_cast<const int4 *>(par + 8 * (size_t)i) + 1);   // the same 32 bytes
        p[0] = p0.x; p[1] = p0.y; p[2] = p0.z; p[3] = p0.w;
        p[4] = p1.x; p[5] = p1.y; p[6] = p1.z; p[7] = p1.w;
    }
    grid_dep_wait();
    grid_dep_launch();
    if (!active) return;
    T acc[R];
#pragma unroll
    for (int r = 0; r < R; r++) acc[r] = T(0);
#pragma unroll
    for (int q = 0; q < 8; q++) {
        if (q < np) {
            T v[R];
            load_x<T, R>(xc + (size_t)p[q] * R, v);
#pragma unroll
            for (int r = 0; r < R; r++) acc[r] += v[r];
        }
    }
    const T w = T(1) / T(np);
#pragma unroll
    for (int r = 0; r < R; r++) xf[(size_t)i * R + r] += w * acc[r];
}

template <class T>
void launch_prolong_add(const DevLevel &Lf, const T *xc, T *xf, int R, cudaStream_t s, Chain *ch) {
    if (Lf.ns == 0) return;   // only smoothed rows have a coarser level
    const unsigned blocks = (unsigned)((Lf.ns + 255) / 256);
    auto k = R == 1 ? prolong_add_kernel<T, 1> : R == 2 ? prolong_add_kernel<T, 2> : prolong_add_kernel<T, 4>;
    klaunch(k, blocks, 256u, 0, s, ch, Lf.ns, Lf.par, Lf.npl2, xc, xf);
}

// x = inv * b on every coarsest block of a level (one per mesh), one warp per row, kCoarseRows rows per
// thread block, so that the rows spread over the SMs: in one thread block the FP64 product of 124 rows kept
// one SM's FP64 pipe busy for 73 us of a cycle.  The row of the inverse, static during a solve, is loaded
// before the grid-dependency wait (its first 32 kCoarsePre entries).
constexpr int kCoarseRows = 4, kCoarsePre = 5;

template <class T, int R>
__global__ void __launch_bounds__(32 * kCoarseRows) coarse_apply_kernel(const int *__restrict__ cblk, int chunks,
                                                                        const T *__restrict__ inv,
                                                                        const T *__restrict__ b, T *__restrict__ x) {
    const int *cb = cblk + 5 * (blockIdx.x / chunks);
    const int row0 = cb[2], n = cb[3];
    const int lane = threadIdx.x & 31, row = (int)(blockIdx.x % chunks) * kCoarseRows + (int)(threadIdx.x >> 5);
    const T *M = inv + cb[4] + (size_t)row * n;
    T a[kCoarsePre];
#pragma unroll
    for (int u = 0; u < kCoarsePre; u++) a[u] = row < n && lane + 32 * u < n ? __ldg(M + lane + 32 * u) : T(0);
    grid_dep_wait();
    grid_dep_launch();
    if (row >= n) return;
    T acc[R];
#pragma unroll
    for (int r = 0; r < R; r++) acc[r] = T(0);
    auto term = [&](int j, T av) {
        T v[R];
        load_x<T, R>(b + (size_t)(row0 + j) * R, v);
#pragma unroll
        for (int r = 0; r < R; r++) acc[r] = fma(av, v[r], acc[r]);
    };
#pragma unroll
    for (int u = 0; u < kCoarsePre; u++)
        if (lane + 32 * u < n) term(lane + 32 * u, a[u]);
    for (int j = lane + 32 * kCoarsePre; j < n; j += 32) term(j, __ldg(M + j));
    int comp;
    const T v = warp_sum<T, R>(acc, lane, comp);
    if (comp >= 0) x[(size_t)(row0 + row) * R + comp] = v;
}

template <class T>
void launch_coarse_apply(const Ctx &c, const DevLevel &L, const T *inv, const T *b, T *x, int R, cudaStream_t s,
                         Chain *ch) {
    if (L.ncb == 0) return;
    const int *cb = c.cblk + 5 * L.cb0;
    int n = 1;
    for (int k = L.cb0; k < L.cb0 + L.ncb; k++) n = std::max(n, c.cblk_host[5 * (size_t)k + 3]);
    const int chunks = (n + kCoarseRows - 1) / kCoarseRows;
    auto k = R == 1 ? coarse_apply_kernel<T, 1> : R == 2 ? coarse_apply_kernel<T, 2> : coarse_apply_kernel<T, 4>;
    klaunch(k, (unsigned)(L.ncb * chunks), 32u * kCoarseRows, 0, s, ch, cb, chunks, inv, b, x);
}

// ---- coarsest-level dense FP64 Cholesky of A + eps Id, eps = 1e-12 mean diag ----
// dense copy of each coarsest block (rows and columns row0..row0+n-1 of its level)
__global__ void dense_from_csr_kernel(const int *__restrict__ cblk, const int *const *__restrict__ rps,
                                      const int *const *__restrict__ cis, const double *const *__restrict__ As,
                                      double *__restrict__ D) {
    const int *cb = cblk + 5 * blockIdx.y;
    const int lev = cb[0], row0 = cb[2], n = cb[3];
    double *Dk = D + cb[4];
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const int *rp = rps[lev], *ci = cis[lev];
    const double *A = As[lev];
    for (int j = 0; j < n; j++) Dk[(size_t)i * n + j] = 0.0;
    for (int k = rp[row0 + i]; k < rp[row0 + i + 1]; k++) {
        const int j = ci[k] - row0;
        if (j >= 0 && j < n) Dk[(size_t)i * n + j] = A[k];
    }
}

__global__ void __launch_bounds__(1024) cholesky_kernel(const int *__restrict__ cblk, double *D, int *flag) {
    __shared__ double s_val;
    const int *cb = cblk + 5 * blockIdx.x;
    const int n = cb[3];
    double *Dk = D + cb[4];
    const int tid = threadIdx.x, nthr = blockDim.x, warp = tid >> 5, lane = tid & 31, nw = nthr >> 5;
    if (tid == 0) {
        double tr = 0.0;
        for (int i = 0; i < n; i++) tr += Dk[(size_t)i * n + i];
        s_val = 1e-12 * tr / (double)(n > 0 ? n : 1);
    }
    __syncthreads();
    const double eps = s_val;
    for (int i = tid; i < n; i += nthr) Dk[(size_t)i * n + i] += eps;
    for (int j = 0; j < n; j++) {
        __syncthreads();
        if (tid == 0) {
            double d = Dk[(size_t)j * n + j];
            if (!(d > 0.0)) { atomicExch(flag, 1); d = 1.0; }
            s_val = sqrt(d);
            Dk[(size_t)j * n + j] = s_val;
        }
        __syncthreads();
        const double piv = s_val;
        for (int i = j + 1 + tid; i < n; i += nthr) Dk[(size_t)i * n + j] /= piv;
        __syncthreads();
        for (int i = j + 1 + warp; i < n; i += nw) {
            const double lij = Dk[(size_t)i * n + j];
            for (int k = j + 1 + lane; k <= i; k += 32) Dk[(size_t)i * n + k] -= lij * Dk[(size_t)k * n + j];
        }
    }
}

// column c of (L L^T)^{-1} of every block: forward then backward substitution on e_c
__global__ void __launch_bounds__(256) cholesky_inverse_kernel(const int *__restrict__ cblk, const double *__restrict__ D,
                                                               double *__restrict__ inv64, float *__restrict__ inv32) {
    extern __shared__ double y[];
    const int *cb = cblk + 5 * blockIdx.y;
    const int n = cb[3];
    const int c = blockIdx.x;
    if (c >= n) return;
    const double *Lf = D + cb[4];
    const int tid = threadIdx.x, nthr = blockDim.x;
    for (int i = tid; i < n; i += nthr) y[i] = (i == c) ? 1.0 : 0.0;
    for (int k = 0; k < n; k++) {
        __syncthreads();
        if (tid == 0) y[k] /= Lf[(size_t)k * n + k];
        __syncthreads();
        const double yk = y[k];
        for (int i = k + 1 + tid; i < n; i += nthr) y[i] -= Lf[(size_t)i * n + k] * yk;
    }
    for (int k = n - 1; k >= 0; k--) {
        __syncthreads();
        if (tid == 0) y[k] /= Lf[(size_t)k * n + k];
        __syncthreads();
        const double yk = y[k];
        for (int i = tid; i < k; i += nthr) y[i] -= Lf[(size_t)k * n + i] * yk;
    }
    __syncthreads();
    for (int i = tid; i < n; i += nthr) {
        inv64[cb[4] + (size_t)i * n + c] = y[i];
        inv32[cb[4] + (size_t)i * n + c] = (float)y[i];
    }
}

void launch_coarse_factor(const Ctx &c, const int *const *rps, const int *const *cis, const double *const *As,
                          cudaStream_t s) {
    if (c.ncblk == 0) return;
    dense_from_csr_kernel<<<dim3((c.n0max + 127) / 128, c.ncblk), 128, 0, s>>>(c.cblk, rps, cis, As, c.cdense);
    cholesky_kernel<<<c.ncblk, 1024, 0, s>>>(c.cblk, c.cdense, c.flag);
    cholesky_inverse_kernel<<<dim3(c.n0max, c.ncblk), 256, c.n0max * sizeof(double), s>>>(c.cblk, c.cdense, c.cinv64,
                                                                                         c.cinv32);
}

// ---- per-right-hand-side sums of squares, two passes (deterministic) ----
// the block's sum of each component: per warp, then over the warps; thread c < R returns component c.
// rest, when given: FP32 sums of each component to be added with the weight w
template <int R>
__device__ __forceinline__ double block_sum(const double (&acc)[R], const float (*rest)[R] = nullptr, double w = 0.0) {
    __shared__ double sh[8][4];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    int comp;
    double v = warp_sum<double, R>(acc, lane, comp);
    if (rest) v = fma((double)warp_sum<float, R>(*rest, lane, comp), w, v);
    if (comp >= 0) sh[warp][comp] = v;
    __syncthreads();
    double t = 0.0;
    if (threadIdx.x < R)
        for (int w = 0; w < 8; w++) t += sh[w][threadIdx.x];
    return t;
}

// One round of blocks over the GPU, a row's components in one or two vector loads.  (256 blocks and scalar
// loads took 38 us for 927k rows of four components, 30 MB.)
template <int R>
__global__ void __launch_bounds__(256) norm_partial_kernel(const double *__restrict__ v, int n, double *__restrict__ part) {
    grid_dep_wait();
    grid_dep_launch();
    double acc[R];
#pragma unroll
    for (int r = 0; r < R; r++) acc[r] = 0.0;
#pragma unroll 4
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
        double x[R];
        load_x<double, R>(v + (size_t)i * R, x);
#pragma unroll
        for (int r = 0; r < R; r++) acc[r] = fma(x[r], x[r], acc[r]);
    }
    const double t = block_sum<R>(acc);
    if (threadIdx.x < R) part[blockIdx.x * 4 + threadIdx.x] = t;
}

// The same for a vector of FP32 pairs: (hi + lo)^2 = hi^2 + (2 hi + lo) lo, hi^2 in FP64 and the rest, mostly below
// 2^-23 of it, in FP32 sums, scaled by 2^64 against underflow.  The FP64 pipe's instructions are the time (6 us each for
// 927k rows of four components; all in FP64, four of them, it took 32.5 us), so hi is widened by moving its bits.
// Pairs for which the FP32 range might not hold (hi below 2^-85 or from 2^20 on, but for zero; lo above hi, as
// cancellation at rounding level can leave it) take the FP64 way.
constexpr float kPairScale = 1.8446744073709552e19f;   // 2^64

__device__ __forceinline__ double pair_sum(float hi, float lo) {   // (volatile: not before its branch is taken)
    double h, l;
    asm volatile("cvt.f64.f32 %0, %1;" : "=d"(h) : "f"(hi));
    asm volatile("cvt.f64.f32 %0, %1;" : "=d"(l) : "f"(lo));
    return h + l;
}

template <int R>
__global__ void __launch_bounds__(256) norm_pair_partial_kernel(const float *__restrict__ hi, const float *__restrict__ lo,
                                                                int n, double *__restrict__ part) {
    grid_dep_wait();
    grid_dep_launch();
    if ((int)(blockIdx.x * blockDim.x) >= n) {   // no rows (the sums alone take some FP64 time)
        if (threadIdx.x < R) part[blockIdx.x * 4 + threadIdx.x] = 0.0;
        return;
    }
    constexpr int U = R == 4 ? 2 : 4;   // rows in flight
    double acc[R];
    float rest[R];
#pragma unroll
    for (int r = 0; r < R; r++) { acc[r] = 0.0; rest[r] = 0.f; }
    const int step = gridDim.x * blockDim.x;
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += U * step) {
        float h[U][R], l[U][R];
        bool usual = true;
#pragma unroll
        for (int u = 0; u < U; u++) {
            if (u == 0 || i + u * (int64_t)step < n) {
                load_x<float, R>(hi + (size_t)(i + u * (int64_t)step) * R, h[u]);
                load_x<float, R>(lo + (size_t)(i + u * (int64_t)step) * R, l[u]);
            } else {
#pragma unroll
                for (int r = 0; r < R; r++) h[u][r] = l[u][r] = 0.f;
            }
        }
#pragma unroll
        for (int u = 0; u < U; u++)
#pragma unroll
            for (int r = 0; r < R; r++) {
                const unsigned a = __float_as_uint(h[u][r]) & 0x7fffffffu, al = __float_as_uint(l[u][r]) & 0x7fffffffu;
                usual = usual && (a - 0x15000000u < 0x34800000u || a == 0u) && al <= a;
            }
        if (usual) {
#pragma unroll
            for (int u = 0; u < U; u++)
#pragma unroll
                for (int r = 0; r < R; r++) {
                    const unsigned a = __float_as_uint(h[u][r]) & 0x7fffffffu;
                    const double d = __hiloint2double(a ? (int)((a >> 3) + 0x38000000u) : 0, (int)(a << 29));
                    acc[r] = fma(d, d, acc[r]);
                    rest[r] = fmaf(fmaf(2.f, h[u][r], l[u][r]), l[u][r] * kPairScale, rest[r]);
                }
        } else {
#pragma unroll
            for (int u = 0; u < U; u++)
#pragma unroll
                for (int r = 0; r < R; r++) {
                    const double d = pair_sum(h[u][r], l[u][r]);
                    acc[r] = fma(d, d, acc[r]);
                }
        }
    }
    const double t = block_sum<R>(acc, &rest, 1.0 / (double)kPairScale);
    if (threadIdx.x < R) part[blockIdx.x * 4 + threadIdx.x] = t;
}

// sum of the blocks' partials of component c, by warp c
__device__ __forceinline__ double partials_sum(const double *__restrict__ part, int nblocks, int c, int lane) {
    double acc[1] = {0.0};
    for (int b = lane; b < nblocks; b += 32) acc[0] += part[b * 4 + c];
    int comp;
    return warp_sum<double, 1>(acc, lane, comp);
}

__global__ void __launch_bounds__(128) norm_final_kernel(const double *__restrict__ part, int nblocks, int R,
                                                         double *__restrict__ out) {
    grid_dep_wait();
    grid_dep_launch();
    const int c = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const double v = c < R ? partials_sum(part, nblocks, c, lane) : 0.0;
    if (lane == 0) out[c] = v;
}

// ---- conjugate gradients preconditioned by the V-cycle (per right-hand side lane) ----
// An iteration's vector work is four passes, each doing all that its operands allow: z from the cycle with
// r.z of the old and the new z; p (and its FP32 pairs for the product); p.q; x, r, the next cycle's right-hand
// side and r.r.  An iteration on 927k rows took 1007 us (mixed, 3 components) with them apart, 983 us so.
//
// Rows are taken in rounds over the GPU (one mesh, kNormBlocks blocks), or, for a batch, as work items: ranges
// of kDotRows rows of one mesh and colour, a warp each, whose sums are added mesh by mesh.  (With items of 2048
// rows, added by one thread per mesh and component, an iteration of twelve meshes of 727k rows took 749 us, of
// 512 rows 691, of 256 678, of 128 680.)
struct RowRange { int i, end, step; };
__device__ __forceinline__ RowRange rows_of(const int *items, int nitems, int n) {
    if (!items) return {(int)(blockIdx.x * blockDim.x + threadIdx.x), n, (int)(gridDim.x * blockDim.x)};
    const int it = (int)(blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5));
    if (it >= nitems) return {0, 0, 32};
    return {__ldg(items + 3 * it + 1) + (int)(threadIdx.x & 31), __ldg(items + 3 * it + 2), 32};
}

// component sums of a block (one mesh: part[block][8], from `at` on) or of a warp's item (part[item][8])
template <int R>
__device__ __forceinline__ void put_sums(const double (&acc)[R], const int *items, int nitems, int at, double *part) {
    if (items) {
        const int it = (int)(blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5));
        int comp;
        const double v = warp_sum<double, R>(acc, threadIdx.x & 31, comp);
        if (it < nitems && comp >= 0) part[8 * (size_t)it + at + comp] = v;
    } else {
        const double v = block_sum<R>(acc);
        if (threadIdx.x < R) part[8 * (size_t)blockIdx.x + at + threadIdx.x] = v;
        __syncthreads();   // its scratch is used again
    }
}

template <int R>
__device__ __forceinline__ void st_vec(double *p, const double (&v)[R]) {
    if constexpr (R == 1) p[0] = v[0];
    else
#pragma unroll
        for (int c = 0; c < R; c += 2) reinterpret_cast<double2 *>(p)[c >> 1] = make_double2(v[c], v[c + 1]);
}

// z_old.r and z.r, z = the cycle's result; z_old <- z
template <class T, int R>
__global__ void __launch_bounds__(256) pcg_z_kernel(const int *__restrict__ items, int nitems, int n,
                                                    const double *__restrict__ r, const T *__restrict__ znew, double *z,
                                                    double *__restrict__ part) {
    grid_dep_wait();
    grid_dep_launch();
    const RowRange q = rows_of(items, nitems, n);
    double a0[R], a1[R];
#pragma unroll
    for (int c = 0; c < R; c++) a0[c] = a1[c] = 0.0;
#pragma unroll 2
    for (int i = q.i; i < q.end; i += q.step) {
        double rv[R], zo[R], zd[R];
        T zn[R];
        load_x<double, R>(r + (size_t)i * R, rv);
        load_x<double, R>(z + (size_t)i * R, zo);
        load_x<T, R>(znew + (size_t)i * R, zn);
#pragma unroll
        for (int c = 0; c < R; c++) {
            zd[c] = (double)zn[c];
            a0[c] = fma(rv[c], zo[c], a0[c]);
            a1[c] = fma(rv[c], zd[c], a1[c]);
        }
        st_vec<R>(z + (size_t)i * R, zd);
    }
    put_sums<R>(a0, items, nitems, 0, part);
    put_sums<R>(a1, items, nitems, 4, part);
}

// a.b (components 0..3) and, when c is given, c.d (4..7)
template <int R>
__global__ void __launch_bounds__(256) dot_kernel(const int *__restrict__ items, int nitems, int n,
                                                  const double *__restrict__ a, const double *__restrict__ b,
                                                  const double *__restrict__ cv, const double *__restrict__ dv,
                                                  double *__restrict__ part) {
    grid_dep_wait();
    grid_dep_launch();
    const RowRange q = rows_of(items, nitems, n);
    double a0[R], a1[R];
#pragma unroll
    for (int c = 0; c < R; c++) a0[c] = a1[c] = 0.0;
#pragma unroll 4
    for (int i = q.i; i < q.end; i += q.step) {
        double x[R], y[R];
        load_x<double, R>(a + (size_t)i * R, x);
        load_x<double, R>(b + (size_t)i * R, y);
#pragma unroll
        for (int c = 0; c < R; c++) a0[c] = fma(x[c], y[c], a0[c]);
        if (cv) {
            load_x<double, R>(cv + (size_t)i * R, x);
            load_x<double, R>(dv + (size_t)i * R, y);
#pragma unroll
            for (int c = 0; c < R; c++) a1[c] = fma(x[c], y[c], a1[c]);
        }
    }
    put_sums<R>(a0, items, nitems, 0, part);
    if (cv) put_sums<R>(a1, items, nitems, 4, part);
}

// one scalar step of lane r on the reduced value v (scalars sc, see pcg_scalar_kernel)
// (done: the lane already meets its tolerance and takes no further steps)
__device__ __forceinline__ void pcg_scalar_step(double *sc, int r, double v, int mode, bool done = false) {
    double *rz = sc + kPcgRz, *s1 = sc + kPcgS1, *s2 = sc + kPcgS2, *al = sc + kPcgAlpha, *be = sc + kPcgBeta,
           *rz0 = sc + kPcgRz0;
    if (mode == 0) {
        s2[r] = v;
    } else if (mode == 1) {
        if (rz[r] == 0.0 && rz0[r] == 0.0) rz0[r] = v;   // the first step
        const bool live = !done && v > kPcgStop * rz0[r];   // false at rounding level, for 0 and NaN
        s1[r] = live ? v : 0.0;
        be[r] = (live && rz[r] > 0.0) ? (v - s2[r]) / rz[r] : 0.0;
        rz[r] = live ? v : 0.0;
    } else {
        const double pap = -v;
        al[r] = (pap > 0.0 && s1[r] > 0.0) ? s1[r] / pap : 0.0;
    }
}

// sum over the items [i0, i1) of component q, by a warp
__device__ __forceinline__ double items_sum(const double *__restrict__ part, int i0, int i1, int q) {
    const int lane = threadIdx.x & 31;
    double acc[1] = {0.0};
#pragma unroll 4
    for (int it = i0 + lane; it < i1; it += 32) acc[0] += __ldg(part + 8 * (size_t)it + q);
    int comp;
    return warp_sum<double, 1>(acc, lane, comp);
}

// block m: the scalar steps of mesh m, component r by warp r, from the partials [istart[m], istart[m + 1])
// (one mesh: all kNormBlocks)
//   mode 1: s2 = v0 (r . z of the previous z), then s1 = v1; beta = (s1 - s2) / rz, rz = s1  (Polak-Ribiere; 0 on
//           the first step, rz = 0; a lane at rounding level, v <= kPcgStop * its first v, keeps beta = alpha = 0)
//   mode 2: alpha = s1 / (p . A p), with v0 = p . q and q = -A p
//   norms (batch): [ninst][16] per-mesh squared norms of r (0..3) and b (4..7) after the last step; tol: the
//   solve's tolerance.  A mesh lane that meets it takes no further steps: the other meshes keep iterating, and a
//   converged lane's FP32-preconditioned recurrence would otherwise run on rounding noise.
__global__ void __launch_bounds__(128) pcg_scalar_kernel(const int *__restrict__ istart, int R,
                                                         const double *__restrict__ part, double *__restrict__ sc,
                                                         int mode, const double *__restrict__ norms,
                                                         const double *__restrict__ tol) {
    grid_dep_wait();
    grid_dep_launch();
    const int m = blockIdx.x, r = threadIdx.x >> 5;
    if (r >= R) return;
    const int i0 = istart ? __ldg(istart + m) : 0, i1 = istart ? __ldg(istart + m + 1) : kNormBlocks;
    const double v0 = items_sum(part, i0, i1, r);
    const double v1 = mode == 1 ? items_sum(part, i0, i1, 4 + r) : 0.0;
    if ((threadIdx.x & 31) != 0) return;
    double *s = sc + (size_t)m * kPcgScalars;
    bool done = false;
    if (norms) {
        const double t = *tol;
        done = norms[16 * (size_t)m + r] <= t * t * norms[16 * (size_t)m + 4 + r];
    }
    if (mode == 1) {
        pcg_scalar_step(s, r, v0, 0, done);
        pcg_scalar_step(s, r, v1, 1, done);
    } else {
        pcg_scalar_step(s, r, v0, mode, done);
    }
}

// per mesh m (a block) and component q < count (a warp each): out[m * ostride + q] = sum of its items' partials
// (0 for the lanes q & 3 >= R, which have none)
__global__ void __launch_bounds__(256) inst_sum_kernel(const int *__restrict__ istart, const double *__restrict__ part,
                                                       double *__restrict__ out, int ostride, int count, int R) {
    grid_dep_wait();
    grid_dep_launch();
    const int m = blockIdx.x, q = threadIdx.x >> 5;
    if (q >= count) return;
    double v = 0.0;
    if ((q & 3) < R)
        v = items_sum(part, istart ? __ldg(istart + m) : 0, istart ? __ldg(istart + m + 1) : kNormBlocks, q);
    if ((threadIdx.x & 31) == 0) out[(size_t)m * ostride + q] = v;
}

// p = z + beta p, and its FP32 pairs when given; row_inst: the mesh of a row (null: one mesh)
template <int R>
__global__ void __launch_bounds__(256) pcg_direction_kernel(const double *__restrict__ z, double *p,
                                                            const double *__restrict__ sc, const int *__restrict__ row_inst,
                                                            float *__restrict__ pair, int n) {
    grid_dep_wait();
    grid_dep_launch();
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const double *s = sc + (row_inst ? (size_t)__ldg(row_inst + i) * kPcgScalars : 0) + kPcgBeta;
    double zv[R], pv[R];
    load_x<double, R>(z + (size_t)i * R, zv);
    load_x<double, R>(p + (size_t)i * R, pv);
#pragma unroll
    for (int c = 0; c < R; c++) pv[c] = fma(s[c], pv[c], zv[c]);
    st_vec<R>(p + (size_t)i * R, pv);
    if (pair) {
        float h[R], l[R];
#pragma unroll
        for (int c = 0; c < R; c++) {
            h[c] = (float)pv[c];
            l[c] = (float)(pv[c] - (double)h[c]);
        }
        float *q = pair + (size_t)i * (2 * R);
#pragma unroll
        for (int c = 0; c < R; c++) { q[c] = h[c]; q[R + c] = l[c]; }
    }
}

// x += alpha p, r += alpha q (q = -A p), the next cycle's right-hand side in its type, and r.r
template <class T, int R>
__global__ void __launch_bounds__(256) pcg_update_kernel(const int *__restrict__ items, int nitems, int n, double *x,
                                                         double *r, const double *__restrict__ p,
                                                         const double *__restrict__ qv, const double *__restrict__ sc,
                                                         const int *__restrict__ row_inst, T *__restrict__ b,
                                                         double *__restrict__ part) {
    grid_dep_wait();
    grid_dep_launch();
    const RowRange w = rows_of(items, nitems, n);
    double acc[R];
#pragma unroll
    for (int c = 0; c < R; c++) acc[c] = 0.0;
#pragma unroll 2
    for (int i = w.i; i < w.end; i += w.step) {
        const double *s = sc + (row_inst ? (size_t)__ldg(row_inst + i) * kPcgScalars : 0) + kPcgAlpha;
        double xv[R], rv[R], pv[R], qq[R];
        load_x<double, R>(x + (size_t)i * R, xv);
        load_x<double, R>(r + (size_t)i * R, rv);
        load_x<double, R>(p + (size_t)i * R, pv);
        load_x<double, R>(qv + (size_t)i * R, qq);
#pragma unroll
        for (int c = 0; c < R; c++) {
            xv[c] = fma(s[c], pv[c], xv[c]);
            rv[c] = fma(s[c], qq[c], rv[c]);
            acc[c] = fma(rv[c], rv[c], acc[c]);
        }
        st_vec<R>(x + (size_t)i * R, xv);
        st_vec<R>(r + (size_t)i * R, rv);
#pragma unroll
        for (int c = 0; c < R; c++) b[(size_t)i * R + c] = (T)rv[c];
    }
    put_sums<R>(acc, items, nitems, 0, part);
}

static unsigned pcg_blocks(const PcgRows &w) { return w.items ? (unsigned)((w.nitems + 7) / 8) : (unsigned)kNormBlocks; }

template <class T>
void launch_pcg_z(const PcgRows &w, const double *r, const T *znew, double *z, int R, double *part, cudaStream_t s,
                  Chain *ch) {
    auto k = R == 1 ? pcg_z_kernel<T, 1> : R == 2 ? pcg_z_kernel<T, 2> : pcg_z_kernel<T, 4>;
    klaunch(k, pcg_blocks(w), 256u, 0, s, ch, w.items, w.nitems, w.n, r, znew, z, part);
}
template void launch_pcg_z<float>(const PcgRows &, const double *, const float *, double *, int, double *, cudaStream_t, Chain *);
template void launch_pcg_z<double>(const PcgRows &, const double *, const double *, double *, int, double *, cudaStream_t, Chain *);

void launch_pcg_dot(const PcgRows &w, const double *a, const double *b, const double *c, const double *d, int R,
                    double *part, cudaStream_t s, Chain *ch) {
    auto k = R == 1 ? dot_kernel<1> : R == 2 ? dot_kernel<2> : dot_kernel<4>;
    klaunch(k, pcg_blocks(w), 256u, 0, s, ch, w.items, w.nitems, w.n, a, b, c, d, part);
}
void launch_pcg_scalar(const PcgRows &w, int R, const double *part, double *sc, int mode, const double *norms,
                       const double *tol, cudaStream_t s, Chain *ch) {
    klaunch(pcg_scalar_kernel, (unsigned)w.ninst, 128u, 0, s, ch, w.istart, R, part, sc, mode, norms, tol);
}
void launch_pcg_sum(const PcgRows &w, const double *part, double *out, int ostride, int count, int R, cudaStream_t s,
                    Chain *ch) {
    klaunch(inst_sum_kernel, (unsigned)w.ninst, 256u, 0, s, ch, w.istart, part, out, ostride, count, R);
}
void launch_pcg_direction(const PcgRows &w, const double *z, double *p, const double *sc, float *pair, int R,
                          cudaStream_t s, Chain *ch) {
    auto k = R == 1 ? pcg_direction_kernel<1> : R == 2 ? pcg_direction_kernel<2> : pcg_direction_kernel<4>;
    if (w.n) klaunch(k, (unsigned)((w.n + 255) / 256), 256u, 0, s, ch, z, p, sc, w.row_inst, pair, w.n);
}
template <class T>
void launch_pcg_update(const PcgRows &w, double *x, double *r, const double *p, const double *q, const double *sc, T *b,
                       int R, double *part, cudaStream_t s, Chain *ch) {
    auto k = R == 1 ? pcg_update_kernel<T, 1> : R == 2 ? pcg_update_kernel<T, 2> : pcg_update_kernel<T, 4>;
    klaunch(k, pcg_blocks(w), 256u, 0, s, ch, w.items, w.nitems, w.n, x, r, p, q, sc, w.row_inst, b, part);
}
template void launch_pcg_update<float>(const PcgRows &, double *, double *, const double *, const double *,
                                       const double *, float *, int, double *, cudaStream_t, Chain *);
template void launch_pcg_update<double>(const PcgRows &, double *, double *, const double *, const double *,
                                        const double *, double *, int, double *, cudaStream_t, Chain *);

void launch_norms(const double *v, int n, int R, double *part, double *out, cudaStream_t s, Chain *ch) {
    auto k = R == 1 ? norm_partial_kernel<1> : R == 2 ? norm_partial_kernel<2> : norm_partial_kernel<4>;
    klaunch(k, (unsigned)kNormBlocks, 256u, 0, s, ch, v, n, part);
    klaunch(norm_final_kernel, 1u, 128u, 0, s, ch, (const double *)part, (int)kNormBlocks, R, out);
}
void launch_norms_pair(const float *hi, const float *lo, int n, int R, double *part, double *out, cudaStream_t s,
                       Chain *ch) {
    auto k = R == 1 ? norm_pair_partial_kernel<1> : R == 2 ? norm_pair_partial_kernel<2> : norm_pair_partial_kernel<4>;
    klaunch(k, (unsigned)kNormBlocks, 256u, 0, s, ch, hi, lo, n, part);
    klaunch(norm_final_kernel, 1u, 128u, 0, s, ch, (const double *)part, (int)kNormBlocks, R, out);
}

// ---- layout and elementwise kernels ----
// user row u of [n][nrhs] <-> internal row perm[u] of [n][R] (perm = null: identity)
__global__ void pack_kernel(const double *__restrict__ u, int n, int nrhs, int R, const int *__restrict__ perm,
                            double *__restrict__ v) {
    const int64_t q = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (q >= (int64_t)n * R) return;
    const int64_t i = q / R;
    const int r = (int)(q % R);
    const int64_t row = perm ? perm[i] : i;
    v[row * R + r] = r < nrhs ? u[i * nrhs + r] : 0.0;
}
__global__ void unpack_kernel(const double *__restrict__ v, int n, int nrhs, int R, const int *__restrict__ perm,
                              double *__restrict__ u) {
    const int64_t q = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (q >= (int64_t)n * nrhs) return;
    const int64_t i = q / nrhs;
    const int r = (int)(q % nrhs);
    const int64_t row = perm ? perm[i] : i;
    u[q] = v[row * R + r];
}
__global__ void to_float_kernel(const double *__restrict__ a, float *__restrict__ b, int64_t n,
                                float *__restrict__ zero) {
    const int64_t q = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    grid_dep_wait();
    grid_dep_launch();
    if (q < n) {
        b[q] = (float)a[q];
        if (zero) zero[q] = 0.f;
    }
}
__global__ void add_float_kernel(double *__restrict__ x, const float *__restrict__ e, int64_t n) {
    const int64_t q = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    grid_dep_wait();
    grid_dep_launch();
    if (q < n) x[q] += (double)e[q];
}
__global__ void add_double_kernel(double *__restrict__ x, const double *__restrict__ e, int64_t n) {
    const int64_t q = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (q < n) x[q] += e[q];
}

void launch_pack(const double *user, int n, int nrhs, int R, double *v, cudaStream_t s, const int *perm) {
    const int64_t m = (int64_t)n * R;
    if (m) pack_kernel<<<(unsigned)((m + 255) / 256), 256, 0, s>>>(user, n, nrhs, R, perm, v);
}
void launch_unpack(const double *v, int n, int nrhs, int R, double *user, cudaStream_t s, const int *perm) {
    const int64_t m = (int64_t)n * nrhs;
    if (m) unpack_kernel<<<(unsigned)((m + 255) / 256), 256, 0, s>>>(v, n, nrhs, R, perm, user);
}
void launch_to_float(const double *a, float *b, int64_t n, cudaStream_t s, float *zero, Chain *ch) {
    if (n) klaunch(to_float_kernel, (unsigned)((n + 255) / 256), 256u, 0, s, ch, a, b, n, zero);
}
void launch_add_float(double *x, const float *e, int64_t n, cudaStream_t s, Chain *ch) {
    if (n) klaunch(add_float_kernel, (unsigned)((n + 255) / 256), 256u, 0, s, ch, x, e, n);
}
void launch_add_double(double *x, const double *e, int64_t n, cudaStream_t s) {
    if (n) add_double_kernel<<<(unsigned)((n + 255) / 256), 256, 0, s>>>(x, e, n);
}

// explicit instantiations
#define LBMG_INST(T)                                                                                           \
    template void launch_sweeps<T>(const Ctx &, const DevLevel &, int, bool, const T *, const T *, const T *, T *, \
                                   int, cudaStream_t, Chain *, int, bool);                                    \
    template bool sweeps_from_zero<T>(const DevLevel &);                                                       \
    template void launch_smooth_colour<T>(const DevLevel &, int, const T *, const T *, const T *, T *, int,   \
                                          cudaStream_t, Chain *, int, int);                                    \
    template void launch_residual<T>(const DevLevel &, const T *, const T *, const T *, T *, int, cudaStream_t, int, \
                                     Chain *, int);                                                            \
    template void launch_jacobi_update<T>(const DevLevel &, const T *, const T *, T *, T, int, cudaStream_t);   \
    template void launch_restrict<T>(const DevLevel &, const T *, T *, int, cudaStream_t, T *, Chain *, bool); \
    template void launch_prolong_add<T>(const DevLevel &, const T *, T *, int, cudaStream_t, Chain *);         \
    template void launch_coarse_apply<T>(const Ctx &, const DevLevel &, const T *, const T *, T *, int, cudaStream_t, \
                                         Chain *);
LBMG_INST(float)
LBMG_INST(double)

}  // namespace lbmg

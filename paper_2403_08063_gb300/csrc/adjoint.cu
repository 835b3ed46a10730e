// Adjoint of the octree-block multigrid solve: the transposed operator, the exact transpose of the forward V-cycle, the
// adjoint solve by defect correction, and dL/dk.  The paper has no adjoint; every step here is the transpose of a forward
// step that cites its passage.
//
// A = S E: E fills ghosts from interiors (reflection, copy, C2F extrapolation of Sec. 3.3.2, F2C mean of Sec. 3.3.1
// or the conservative flux ghost), S is the 7-point stencil; A^T = E^T S^T.  At the domain boundary, and between blocks of one
// level that hold the same coefficient of their common face, E and S transpose into themselves, so there A^T y is the
// forward stencil on y with the forward's ghosts.  (A merged level under face averaging can hold two coefficients of a face,
// each its own side's mean of finer faces: the neighbour's coefficient then belongs to its value, and the difference times
// that value goes to the right-hand side, k_adj_uneven.)  At a refinement interface, with a_j the adjoint of fine ghost j,
// T~ = T / h^2 and y_C the coarse cell behind it:
//     conservative: the fine ghost reads y_C / 8 and the coarse one y_C (the rows of u_j and u_C in the coarse ghost
//                   G = u_C - sum_j T_j / (2 T_C) (g_j - u_j)), and a_j = -T~_j (y_j - y_C / 8);
//     ghost-only:   both read 0, a_j = -T~_j y_j, and each of the eight fine cells of the coarse ghost's mean gets
//                   -T~_C y_C / 8;
//     either way (A^T y) gets a_j times the quadratic weights at the coarse cells ghost j was extrapolated from.
// That last part is the only one that is not a 7-point stencil.  It moves to the right-hand side: with f' = f - (the
// interface part of A^T y) and the ghosts above, f - A^T y = f' - (stencil of y), so the transposed cycle runs on the
// forward's kernels, layouts and launch shapes, and one small kernel per exchange (k_adj_iface) keeps ghosts and f' current
// by adding what changed since the last one.
//
// The forward V-cycle is a linear map M of its right-hand side; M^T runs its steps backwards, each transposed.  The
// transpose of a half-sweep u += Pi_c D^-1 (f - A u) in terms of the accumulated result y is y += Pi_c D^-1 (f - A^T y): the
// same half-sweep on A^T, with the colours in reverse order.  Prolongation and restriction transpose into the gather
// k_prolong_T and the injection k_inject.  So lambda += M^T (g - A^T lambda) converges at the forward cycle's rate.
//
// What bounds it: HBM, in the half-sweeps (10 B per updated cell) and the FP64 residual's FP64 rate.  The transposed cycle
// step by step on natural-layout arrays of its own (the correction, its stencil with ghost adjoints, their scatter by
// atomics over every face, two vector updates per half-sweep: ~70 B per cell and half-sweep) made set-up, forward solve and
// adjoint on 448 + 512 blocks of 32^3 (31.5M cells) take 174 to 183 ms, depending on the inputs; this form, with the later
// steps' kernels, 65 ms.
#include <cmath>

#include "forest_state.h"

namespace octmg {
namespace {

__device__ inline void decode_cell(int64_t t, int lg, int &x, int &y, int &z, int64_t &b) {
    const int n = 1 << lg;
    x = static_cast<int>(t & (n - 1));
    y = static_cast<int>((t >> lg) & (n - 1));
    z = static_cast<int>((t >> (2 * lg)) & (n - 1));
    b = t >> (3 * lg);
}

#define GRID_STRIDE(total) \
    for (int64_t t = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x; t < (total); \
         t += static_cast<int64_t>(gridDim.x) * blockDim.x)

// Scaled face coefficient T / h^2 of the face between depth 0 (g0) and depth 1 (g1) of a block face (axis, side).
template <typename T, int MODE>
__device__ __forceinline__ T scaled_face(const Coef &cf, const T *ih2, int64_t b, int64_t g0, int64_t g1, int axis,
                                         int side) {
    if constexpr (MODE == 0) return ih2[b];
    const T t = face_coef<T, MODE>(cf, side ? g0 : g1, side ? g1 : g0, axis);
    return MODE == 1 ? t : t * ih2[b];
}

// Shared memory of the transposed quadratic C2F rule of one strip of an item: the adjoints of its 2 rows x n ghosts, their
// sums after the first tangential step, 2 rows of the w1 <= n/2 + 2 coarse cells, and the tangential weights [case][a][base].
__host__ __device__ inline size_t scatter_values(int n) {
    const size_t lines = n / iface_strips(n);
    return lines * n + lines * (n / 2 + 2) + 18;
}
template <typename T>
struct ScatterMem {
    T *D, *S, *W;
    __device__ ScatterMem(unsigned char *raw, const IfaceStrip &Q)
        : D(reinterpret_cast<T *>(raw)), S(D + 2 * Q.rows * Q.n), W(S + 2 * Q.rows * (Q.h + 2)) {
        if (threadIdx.x < 18) W[threadIdx.x] = w_tang<T>(0, threadIdx.x / 6, threadIdx.x / 3 % 2, threadIdx.x % 3);
    }
};

// One tangential step of the transpose: the sum over the fine positions of coarse cells c0 .. c0 + count - 1 (values at
// v[0], v[stride], ..) of the weight with which the ghost there reads coarse cell y.
template <typename T>
__device__ __forceinline__ T gather_tangential(const T *v, int stride, const T *W, int y, int c0, int count, int n) {
    T s = T(0);
    for (int c = max(y - 2, c0); c <= min(y + 2, c0 + count - 1); ++c) {
        const int cs = tang_case(c, n), k = y - c - tang_first(cs);
        if (k < 0 || k > 2) continue;
        const int i = 2 * (c - c0);
        s = fma(W[cs * 6 + k], v[i * stride], s);
        s = fma(W[cs * 6 + 3 + k], v[(i + 1) * stride], s);
    }
    return s;
}

// The transposed quadratic C2F rule on a strip of item F: the ghosts' adjoints in m.D[line n + i1] (written by the CTA's
// threads just before) times sgn to the coarse cells the ghosts were extrapolated from, through add(b, X, Y, Z, v).  One
// tangential direction after the other, then the three coarse layers behind the face: about 6 + 6 + 3 operations per value,
// as gathers (sums by floating-point atomics in shared memory, which are compare-and-swap loops, took 34 us on 384 faces of
// 32 x 32 cells; this 19 us).
template <typename T, class Add>
__device__ __forceinline__ void scatter_c2f(const ScatterMem<T> &m, const IfaceStrip &Q, const FaceItem &F, T sgn, Add &&add) {
    __syncthreads();
    for (int q = threadIdx.x; q < 2 * Q.rows * Q.w1; q += blockDim.x) {
        const int y = q % Q.w1, line = q / Q.w1;
        m.S[q] = gather_tangential<T>(m.D + line * Q.n, 1, m.W, Q.lo1 + y, F.seg1 * Q.h, Q.h, Q.n);
    }
    __syncthreads();
    for (int q = threadIdx.x; q < Q.w1 * Q.w2; q += blockDim.x) {
        const int y = q % Q.w1, z = Q.lo2 + q / Q.w1;
        const T v = sgn * gather_tangential<T>(m.S + y, Q.w1, m.W, z, F.seg2 * Q.h + Q.c0, Q.rows, Q.n);
#pragma unroll
        for (int d = 0; d < 3; ++d) {
            int X, Y, Z;
            face_xyz(F.axis, 1 - F.side, 1 + d, Q.lo1 + y, z, Q.n, X, Y, Z);
            add(F.nbr, X, Y, Z, w_normal<T>(0, d) * v);
        }
    }
}

// Where an interface kernel adds: a padded pool, or (user != null) a field in the caller's layout.
template <typename T>
struct Target {
    T *pool;
    double *user;
    const int64_t *off;  // start of every leaf in the caller's array, or null
};
template <typename T>
__device__ __forceinline__ void add_to(const Target<T> &t, const LevelGeom &g, int64_t b, int X, int Y, int Z, T v) {
    if (t.pool) {
        atomicAdd(&t.pool[Lay<T>::at(g, b, X, Y, Z)], v);
    } else {
        const int64_t at = t.off ? t.off[b] : b << (3 * g.lg);
        atomicAdd(&t.user[at + ((static_cast<int64_t>(Z - 1) * g.n + (Y - 1)) * g.n + (X - 1))], static_cast<double>(v));
    }
}

// One strip of an interface item per CTA, one lane per fine ghost (a coarse cell's four next to each other): the transposed
// ghosts of y on both sides (GHOSTS), and sgn times the part of A^T y that is no 7-point stencil added to `to`.  old (may be
// null: 0) keeps the ghost adjoints that `to` already holds, n^2 per item, and with the ghost-only variant old_c the coarse
// ones, (n/2)^2 per item; what is added is the change.  Where strips meet, atomics order the sums.
template <typename T, int MODE, bool FLUX, bool GHOSTS>
__global__ void __launch_bounds__(kThreads)
    k_adj_iface(T *__restrict__ y, Coef cf, const T *__restrict__ ih2, const FaceItem *__restrict__ items, LevelGeom g,
                T *__restrict__ old, T *__restrict__ old_c, Target<T> to, T sgn) {
    pdl_enter(y, old, old_c, to.pool, to.user);
    extern __shared__ __align__(16) unsigned char adj_smem[];
    const int strips = iface_strips(g.n), item = blockIdx.x / strips;
    const FaceItem F = items[item];
    const IfaceStrip Q(F, g.n, blockIdx.x % strips);
    const int n = Q.n, h = Q.h;
    const bool adds = to.pool || to.user;
    const ScatterMem<T> m(adj_smem, Q);
    const auto add = [&](int64_t b, int X, int Y, int Z, T v) { add_to(to, g, b, X, Y, Z, v); };
    for (int q = threadIdx.x; q < 4 * Q.rows * h; q += blockDim.x) {
        const int a1 = q & 1, a2 = (q >> 1) & 1, ycl = (q >> 2) & (h - 1), zcl = Q.c0 + (q >> (g.lg + 1));
        const int i1 = 2 * ycl + a1, i2 = 2 * zcl + a2, yc = F.seg1 * h + ycl, zc = F.seg2 * h + zcl;
        const int64_t gC = fidx<T>(g, F.nbr, F.axis, 1 - F.side, 1, yc, zc);
        const int64_t g0c = fidx<T>(g, F.nbr, F.axis, 1 - F.side, 0, yc, zc);
        const int64_t g0 = fidx<T>(g, F.blk, F.axis, F.side, 0, i1, i2);
        const int64_t g1 = fidx<T>(g, F.blk, F.axis, F.side, 1, i1, i2);
        const T yC = y[gC], through = FLUX ? T(0.125) * yC : T(0);
        if (GHOSTS) {
            y[g0] = through;
            if ((q & 3) == 0) y[g0c] = FLUX ? yC : T(0);
        }
        if (!adds) continue;
        T a = -scaled_face<T, MODE>(cf, ih2, F.blk, g0, g1, F.axis, F.side) * (y[g1] - through);
        if (old) {
            T *keep = old + (static_cast<int64_t>(item) * n + i2) * n + i1;
            const T before = *keep;
            *keep = a;
            a -= before;
        }
        m.D[(i2 - 2 * Q.c0) * n + i1] = a;
        if (!FLUX && (q & 3) == 0) {
            T v = -scaled_face<T, MODE>(cf, ih2, F.nbr, g0c, gC, F.axis, 1 - F.side) * yC;
            if (old_c) {
                T *keep = old_c + (static_cast<int64_t>(item) * h + zcl) * h + ycl;
                const T before = *keep;
                *keep = v;
                v -= before;
            }
            for (int e = 0; e < 8; ++e) {
                int X, Y, Z;
                face_xyz(F.axis, F.side, 1 + (e >> 2), 2 * ycl + (e & 1), 2 * zcl + ((e >> 1) & 1), n, X, Y, Z);
                add(F.blk, X, Y, Z, sgn * T(0.125) * v);
            }
        }
    }
    if (adds) scatter_c2f<T>(m, Q, F, sgn, add);
}

// Same-level faces with a coefficient on either side: row i of A^T has the neighbour's one, T_B, where the stencil has the
// block's own, T_A, so f' takes (T_B - T_A) / h^2 times what changed of the value on the other side (old: what f' holds).
// One thread per face cell of every item; the cells at a block's edges belong to several.  A launch of 3.7 us like the level's
// others: 240 of them are 0.9 of 65 ms in a gradient on 448 + 512 blocks of 32^3 (31.5M cells).
template <typename T, int MODE>
__global__ void __launch_bounds__(kThreads)
    k_adj_uneven(const T *__restrict__ y, Coef cf, const T *__restrict__ ih2, const FaceItem *__restrict__ items, int nitems,
                 LevelGeom g, T *__restrict__ old, T *__restrict__ f) {
    pdl_enter(y, old, f);
    const int n = g.n, lg = g.lg;
    const int64_t total = static_cast<int64_t>(nitems) << (2 * lg);
    GRID_STRIDE(total) {
        const FaceItem F = items[t >> (2 * lg)];
        if (F.kind != FK_SAME) continue;
        const int r = static_cast<int>(t) & ((1 << (2 * lg)) - 1), i1 = r & (n - 1), i2 = r >> lg;
        const auto at = [&](int64_t b, int side, int depth) { return fidx<T>(g, b, F.axis, side, depth, i1, i2); };
        const int64_t own = at(F.blk, F.side, 1), other = at(F.nbr, 1 - F.side, 1);
        const T Ta = scaled_face<T, MODE>(cf, ih2, F.blk, at(F.blk, F.side, 0), own, F.axis, F.side);
        const T Tb = scaled_face<T, MODE>(cf, ih2, F.nbr, at(F.nbr, 1 - F.side, 0), other, F.axis, 1 - F.side);
        const T now = y[other], before = old[t];
        old[t] = now;
        if (Ta != Tb) atomicAdd(&f[own], (Tb - Ta) * (now - before));
    }
}

// fe = g again at the cells that k_adj_iface adds to, one strip of an item per CTA.
template <bool FLUX>
__global__ void __launch_bounds__(kThreads)
    k_adj_restore(double *__restrict__ fe, const double *__restrict__ gv, const FaceItem *__restrict__ items, LevelGeom g) {
    const int strips = iface_strips(g.n);
    const FaceItem F = items[blockIdx.x / strips];
    const IfaceStrip Q(F, g.n, blockIdx.x % strips);
    for (int q = threadIdx.x; q < Q.w1 * Q.w2; q += blockDim.x)
        for (int d = 1; d <= 3; ++d) {
            const int64_t i = fidx<double>(g, F.nbr, F.axis, 1 - F.side, d, Q.lo1 + q % Q.w1, Q.lo2 + q / Q.w1);
            fe[i] = gv[i];
        }
    if (!FLUX)
        for (int q = threadIdx.x; q < 2 * Q.rows * Q.n; q += blockDim.x)
            for (int d = 1; d <= 2; ++d) {
                const int64_t i = fidx<double>(g, F.blk, F.axis, F.side, d, q % Q.n, 2 * Q.c0 + q / Q.n);
                fe[i] = gv[i];
            }
}

// r = f - (stencil of y) over the interior, written through to the ghosts that mirror it (same level) or reflect it
// (boundary); interface ghosts of r stay 0.  With part (FP64) per-CTA partials of h^3 r^2.
template <typename T, int MODE>
__global__ void k_adj_residual(const T *__restrict__ y, const T *f, Coef cf, const T *__restrict__ ih2, LevelGeom g,
                               const int32_t *__restrict__ nbr6, T *r, const double *__restrict__ vol,
                               double *__restrict__ part) {
    pdl_enter(y, f, r);
    const int n = g.n;
    const int64_t total = static_cast<int64_t>(g.nb) << (3 * g.lg);
    double acc = 0.0;
    GRID_STRIDE(total) {
        int x, yy, z;
        int64_t b;
        decode_cell(t, g.lg, x, yy, z, b);
        T v;
        if constexpr (sizeof(T) == 4)
            v = residual_xyz<T, MODE>(y, f, cf, g, b, x + 1, yy + 1, z + 1, ih2[b]);
        else
            v = residual_at<T, MODE>(y, f, cf, b * g.bs + off3(x + 1, yy + 1, z + 1, g.P), g.P, MODE == 1 ? T(0) : ih2[b]);
        r[Lay<T>::at(g, b, x + 1, yy + 1, z + 1)] = v;
        if (part) acc = fma(vol[b] * static_cast<double>(v), static_cast<double>(v), acc);
        if (nbr6 && (x == 0 || x == n - 1 || yy == 0 || yy == n - 1 || z == 0 || z == n - 1)) {
            const int c[3] = {x, yy, z};
#pragma unroll
            for (int axis = 0; axis < 3; ++axis)
#pragma unroll
                for (int side = 0; side < 2; ++side) {
                    if (c[axis] != (side ? n - 1 : 0)) continue;
                    const int nb = nbr6[b * 6 + 2 * axis + side];
                    const int i1 = axis == 0 ? yy : x, i2 = axis == 2 ? yy : z;
                    if (nb >= 0) r[fidx<T>(g, nb, axis, 1 - side, 0, i1, i2)] = v;
                    else if (nb == -1) r[fidx<T>(g, b, axis, side, 0, i1, i2)] = -v;
                }
        }
    }
    if (!part) return;
    __shared__ double sm[kThreads / 32];
    for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
    if ((threadIdx.x & 31) == 0) sm[threadIdx.x >> 5] = acc;
    __syncthreads();
    if (threadIdx.x == 0) {
        double s = 0.0;
        for (int w = 0; w < kThreads / 32; ++w) s += sm[w];
        part[blockIdx.x] = s;
    }
}

// The same in FP32 on colour-split blocks of edge 2^LG, one thread per pair of cells x = 2j, 2j + 1 of a row: they and their
// neighbours are 12 values of y (and of 1/k), at immediate offsets from one position of either half, and share a face.  The
// generic form above computes every address in 64 bits and loads 14 values per cell: 533 us on 31.5M cells; this 190 us.
template <int MODE, int LG>
__global__ void __launch_bounds__(kThreads)
    k_adj_residual32(const float *__restrict__ y, const float *__restrict__ f, Coef cf, const float *__restrict__ ih2,
                     int64_t bs, int64_t pairs, const int32_t *__restrict__ nbr6, float *__restrict__ r) {
    pdl_enter(y, f, r);
    constexpr int n = 1 << LG, NH = n / 2, P = n + 2, H = half_row(P), PL = P * H, HALF = P * PL;
    const int64_t t = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x;
    if (t >= pairs) return;
    const int j = static_cast<int>(t) & (NH - 1), yy = static_cast<int>(t >> (LG - 1)) & (n - 1);
    const int z = static_cast<int>(t >> (2 * LG - 1)) & (n - 1);
    const int64_t b = t >> (3 * LG - 1), base = b * bs;
    // cell A (padded X = 2j + 1) at q of half s, cell B (X = 2j + 2) at q + 1 of the other half
    const int s = (yy + z + 1) & 1, q = ((z + 1) * P + yy + 1) * H + j;
    const int hs = s * HALF, ho = (s ^ 1) * HALF;
    const float *us = y + base + hs + q, *uo = y + base + ho + q;
    const float A = us[0], B = uo[1];
    const float nA[6] = {uo[0], B, uo[-H], uo[H], uo[-PL], uo[PL]};
    const float nB[6] = {A, us[1], us[1 - H], us[1 + H], us[1 - PL], us[1 + PL]};
    const float fA = __ldg(f + base + hs + q), fB = __ldg(f + base + ho + q + 1);
    const float ih = __ldg(ih2 + b);
    float rA, rB;
    if constexpr (MODE == 0) {
        const float SA = ((nA[0] + nA[1]) + (nA[2] + nA[3])) + (nA[4] + nA[5]);
        const float SB = ((nB[0] + nB[1]) + (nB[2] + nB[3])) + (nB[4] + nB[5]);
        rA = fmaf(fmaf(-6.0f, A, SA), ih, fA);
        rB = fmaf(fmaf(-6.0f, B, SB), ih, fB);
    } else {
        float cA[6], cB[6];
        if constexpr (MODE == 2) {
            const float *ks = cf.kap + base + hs + q, *ko = cf.kap + base + ho + q;
            const float kA = __ldg(ks), kB = __ldg(ko + 1);
            cA[0] = frcp(kA + __ldg(ko));
            cA[1] = frcp(kA + kB);
            cA[2] = frcp(kA + __ldg(ko - H));
            cA[3] = frcp(kA + __ldg(ko + H));
            cA[4] = frcp(kA + __ldg(ko - PL));
            cA[5] = frcp(kA + __ldg(ko + PL));
            cB[0] = cA[1];
            cB[1] = frcp(kB + __ldg(ks + 1));
            cB[2] = frcp(kB + __ldg(ks + 1 - H));
            cB[3] = frcp(kB + __ldg(ks + 1 + H));
            cB[4] = frcp(kB + __ldg(ks + 1 - PL));
            cB[5] = frcp(kB + __ldg(ks + 1 + PL));
        } else {  // a cell's lower faces at the cell, its upper ones at the upper neighbour
            const int64_t is = base + hs + q, io = base + ho + q;
            cA[0] = __ldg(cf.ax + is);
            cA[1] = __ldg(cf.ax + io + 1);
            cA[2] = __ldg(cf.ay + is);
            cA[3] = __ldg(cf.ay + io + H);
            cA[4] = __ldg(cf.az + is);
            cA[5] = __ldg(cf.az + io + PL);
            cB[0] = cA[1];
            cB[1] = __ldg(cf.ax + is + 1);
            cB[2] = __ldg(cf.ay + io + 1);
            cB[3] = __ldg(cf.ay + is + 1 + H);
            cB[4] = __ldg(cf.az + io + 1);
            cB[5] = __ldg(cf.az + is + 1 + PL);
        }
        float SA = 0.0f, DA = 0.0f, SB = 0.0f, DB = 0.0f;
#pragma unroll
        for (int i = 0; i < 6; ++i) {
            SA = fmaf(cA[i], nA[i], SA);
            DA += cA[i];
            SB = fmaf(cB[i], nB[i], SB);
            DB += cB[i];
        }
        rA = fmaf(2.0f * fmaf(-DA, A, SA), ih, fA);
        rB = fmaf(2.0f * fmaf(-DB, B, SB), ih, fB);
    }
    float *rs = r + base + hs + q, *ro = r + base + ho + q;
    rs[0] = rA;
    ro[1] = rB;
    // write-through, as in smooth32_column: the mirroring ghost at the same place of its half n cells along the axis, the
    // reflected one at the neighbour position of the other half
    if (j == 0) {
        const int nb = nbr6[b * 6];
        if (nb >= 0) r[nb * bs + hs + q + NH] = rA;
        else if (nb == -1) ro[0] = -rA;
    }
    if (j == NH - 1) {
        const int nb = nbr6[b * 6 + 1];
        if (nb >= 0) r[nb * bs + ho + q + 1 - NH] = rB;
        else if (nb == -1) rs[1] = -rB;
    }
#pragma unroll
    for (int axis = 1; axis < 3; ++axis) {
        const int c = axis == 1 ? yy : z, D = axis == 1 ? n * H : n * PL, E = axis == 1 ? H : PL;
        if (c != 0 && c != n - 1) continue;
        const int side = c ? 1 : 0, nb = nbr6[b * 6 + 2 * axis + side];
        if (nb >= 0) {
            r[nb * bs + hs + q + (side ? -D : D)] = rA;
            r[nb * bs + ho + q + 1 + (side ? -D : D)] = rB;
        } else if (nb == -1) {
            ro[side ? E : -E] = -rA;
            rs[1 + (side ? E : -E)] = -rB;
        }
    }
}

// Transposed prolongation of a level whose blocks all halve, as a gather: e_C enters its eight children and, as the
// neighbour on their side, the four cells across each of its six faces, every time with weight 1/4 (u_f += 1/4 (e_C +
// e_{C+sx} + e_{C+sy} + e_{C+sz})); the reflected boundary ghost of r carries the reflected e.  Writes the coarse
// right-hand side and zeroes the coarse result with its face ghosts.
template <typename T>
__global__ void k_prolong_T(const T *__restrict__ r, LevelGeom gf, T *__restrict__ fc, T *__restrict__ yc,
                            const XferItem *__restrict__ xf, LevelGeom gc) {
    pdl_enter(r, fc, yc);
    const int nc = gc.n;
    const int64_t total = static_cast<int64_t>(gc.nb) << (3 * gc.lg);
    GRID_STRIDE(total) {
        int X, Y, Z;
        int64_t B;
        decode_cell(t, gc.lg, X, Y, Z, B);
        const int64_t b = xf[B].src[0];
        T s = T(0);
#pragma unroll
        for (int k = 0; k < 4; ++k)
#pragma unroll
            for (int j = 0; j < 4; ++j)
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    const int out = (i == 0 || i == 3) + (j == 0 || j == 3) + (k == 0 || k == 3);
                    if (out <= 1) s += r[Lay<T>::at(gf, b, 2 * X + i, 2 * Y + j, 2 * Z + k)];
                }
        const int64_t gi = Lay<T>::at(gc, B, X + 1, Y + 1, Z + 1);
        fc[gi] = T(0.25) * s;
        yc[gi] = T(0);
        if (X == 0) yc[Lay<T>::at(gc, B, 0, Y + 1, Z + 1)] = T(0);
        if (X == nc - 1) yc[Lay<T>::at(gc, B, nc + 1, Y + 1, Z + 1)] = T(0);
        if (Y == 0) yc[Lay<T>::at(gc, B, X + 1, 0, Z + 1)] = T(0);
        if (Y == nc - 1) yc[Lay<T>::at(gc, B, X + 1, nc + 1, Z + 1)] = T(0);
        if (Z == 0) yc[Lay<T>::at(gc, B, X + 1, Y + 1, 0)] = T(0);
        if (Z == nc - 1) yc[Lay<T>::at(gc, B, X + 1, Y + 1, nc + 1)] = T(0);
    }
}

// The same in FP32 for fine edges 2^LG, with the box at immediate offsets (Box32).
template <int LG>
__global__ void __launch_bounds__(kThreads)
    k_prolong_T32(const float *__restrict__ r, int64_t bsf, float *__restrict__ fc, float *__restrict__ yc,
                  const XferItem *__restrict__ xf, int64_t total, int64_t bsc) {
    pdl_enter(r, fc, yc);
    using Bx = Box32<LG>;
    constexpr int nc = (1 << LG) / 2, LC = LG - 1;
    const int64_t t = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x;
    if (t >= total) return;
    const int q = static_cast<int>(t) & ((1 << (3 * LC)) - 1);
    const int64_t B = t >> (3 * LC);
    const int X = q & (nc - 1), Y = (q >> LC) & (nc - 1), Z = q >> (2 * LC);
    const float *rb = r + xf[B].src[0] * bsf + (2 * Z * Bx::P + 2 * Y) * Bx::HP + X;
    float s = 0.0f;
#pragma unroll
    for (int k = 0; k < 4; ++k)
#pragma unroll
        for (int j = 0; j < 4; ++j)
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const int out = (i == 0 || i == 3) + (j == 0 || j == 3) + (k == 0 || k == 3);
                if (out <= 1) s += rb[Bx::off(i, j, k)];
            }
    rr32_store<LG>(fc, yc, B, bsc, X, Y, Z, 2.0f * s);  // stores 1/8 of it: a quarter of the sum
}

// The same for a level with merged octets or carried-over blocks: scattered into the coarse padded right-hand side
// (ghost positions included; k_et_faces and k_et_iface follow).
template <typename T>
__global__ void k_prolong_T_scatter(const T *__restrict__ r, LevelGeom gf, T *__restrict__ Ec,
                                    const XferItem *__restrict__ xf, LevelGeom gc) {
    pdl_enter(r, Ec);
    const int nc = gc.n;
    const int64_t total = static_cast<int64_t>(gc.nb) << (3 * gc.lg);
    GRID_STRIDE(total) {
        int X, Y, Z;
        int64_t B;
        decode_cell(t, gc.lg, X, Y, Z, B);
        const XferItem xi = xf[B];
        if (xi.kind == XF_COPY) {
            atomicAdd(&Ec[Lay<T>::at(gc, B, X + 1, Y + 1, Z + 1)], r[Lay<T>::at(gf, xi.src[0], X + 1, Y + 1, Z + 1)]);
            continue;
        }
        int64_t b = xi.src[0];
        int x0 = 2 * X, y0 = 2 * Y, z0 = 2 * Z;
        if (xi.kind == XF_MERGE) {
            const int hc = nc >> 1, ox = X >= hc, oy = Y >= hc, oz = Z >= hc;
            b = xi.src[ox + 2 * oy + 4 * oz];
            x0 -= ox * nc;
            y0 -= oy * nc;
            z0 -= oz * nc;
        }
        T all = T(0), sx[2] = {T(0), T(0)}, sy[2] = {T(0), T(0)}, sz[2] = {T(0), T(0)};
        for (int c = 0; c < 2; ++c)
            for (int bb = 0; bb < 2; ++bb)
                for (int a = 0; a < 2; ++a) {
                    const T v = T(0.25) * r[Lay<T>::at(gf, b, x0 + a + 1, y0 + bb + 1, z0 + c + 1)];
                    all += v;
                    sx[a] += v;
                    sy[bb] += v;
                    sz[c] += v;
                }
        atomicAdd(&Ec[Lay<T>::at(gc, B, X + 1, Y + 1, Z + 1)], all);
        for (int s = 0; s < 2; ++s) {
            atomicAdd(&Ec[Lay<T>::at(gc, B, X + 2 * s, Y + 1, Z + 1)], sx[s]);
            atomicAdd(&Ec[Lay<T>::at(gc, B, X + 1, Y + 2 * s, Z + 1)], sy[s]);
            atomicAdd(&Ec[Lay<T>::at(gc, B, X + 1, Y + 1, Z + 2 * s)], sz[s]);
        }
    }
}

// E^T of the faces filled from one source block: reflection (ghost = -u_i) and copy from the neighbour.
template <typename T>
__global__ void k_et_faces(T *__restrict__ G, const FaceItem *__restrict__ items, int nitems, LevelGeom g) {
    pdl_enter(G);
    const int n = g.n, lg = g.lg;
    const int64_t total = static_cast<int64_t>(nitems) << (2 * lg);
    GRID_STRIDE(total) {
        const FaceItem F = items[t >> (2 * lg)];
        const int r = static_cast<int>(t) & ((1 << (2 * lg)) - 1);
        const int i1 = r & (n - 1), i2 = r >> lg;
        const T a = G[fidx<T>(g, F.blk, F.axis, F.side, 0, i1, i2)];
        if (F.kind == FK_BND) atomicAdd(&G[fidx<T>(g, F.blk, F.axis, F.side, 1, i1, i2)], -a);
        else atomicAdd(&G[fidx<T>(g, F.nbr, F.axis, 1 - F.side, 1, i1, i2)], a);
    }
}

// E^T of a level's interface ghosts, one strip of an item per CTA and one lane per fine ghost, added to the interior of fc.
// The ghost adjoints are those of the transposed prolongation: GATHER: a quarter of the four finer cells next to the ghost
// (the level's blocks are halved blocks, r the finer level's residual); else they stand in fc's own ghosts
// (k_prolong_T_scatter).
template <typename T, int MODE, bool FLUX, bool GATHER>
__global__ void __launch_bounds__(kThreads)
    k_et_iface(T *__restrict__ fc, Coef cf, const FaceItem *__restrict__ items, LevelGeom g, const T *__restrict__ r,
               LevelGeom gf, const XferItem *__restrict__ xf) {
    pdl_enter(fc, r);
    extern __shared__ __align__(16) unsigned char adj_smem[];
    const int strips = iface_strips(g.n), item = blockIdx.x / strips;
    const FaceItem F = items[item];
    const IfaceStrip Q(F, g.n, blockIdx.x % strips);
    const int n = Q.n, h = Q.h;
    const ScatterMem<T> m(adj_smem, Q);
    const int64_t bf = GATHER ? xf[F.blk].src[0] : 0, bc = GATHER ? xf[F.nbr].src[0] : 0;
    const auto add = [&](int64_t b, int X, int Y, int Z, T v) { atomicAdd(&fc[Lay<T>::at(g, b, X, Y, Z)], v); };
    const auto ghost = [&](int64_t blk, int64_t fine, int side, int i1, int i2) {
        if constexpr (!GATHER) return fc[fidx<T>(g, blk, F.axis, side, 0, i1, i2)];
        T s = T(0);
#pragma unroll
        for (int e = 0; e < 4; ++e) s += r[fidx<T>(gf, fine, F.axis, side, 1, 2 * i1 + (e & 1), 2 * i2 + (e >> 1))];
        return T(0.25) * s;
    };
    for (int q = threadIdx.x; q < 4 * Q.rows * h; q += blockDim.x) {
        const int a1 = q & 1, a2 = (q >> 1) & 1, ycl = (q >> 2) & (h - 1), zcl = Q.c0 + (q >> (g.lg + 1));
        const int i1 = 2 * ycl + a1, i2 = 2 * zcl + a2, yc = F.seg1 * h + ycl, zc = F.seg2 * h + zcl;
        T a = ghost(F.blk, bf, F.side, i1, i2);
        const T aG = ghost(F.nbr, bc, 1 - F.side, yc, zc);
        if constexpr (FLUX) {  // G = u_C - sum_j c (g_j - u_j), c = T_j / (2 T_C) (MODE 1: T~_j / (8 T~_C))
            const int64_t gC = fidx<T>(g, F.nbr, F.axis, 1 - F.side, 1, yc, zc);
            const int64_t g0c = fidx<T>(g, F.nbr, F.axis, 1 - F.side, 0, yc, zc);
            const int64_t g0 = fidx<T>(g, F.blk, F.axis, F.side, 0, i1, i2);
            const int64_t g1 = fidx<T>(g, F.blk, F.axis, F.side, 1, i1, i2);
            const T Tc = face_coef<T, MODE>(cf, F.side ? gC : g0c, F.side ? g0c : gC, F.axis);
            const T Tj = face_coef<T, MODE>(cf, F.side ? g0 : g1, F.side ? g1 : g0, F.axis);
            const T v = Tj / (T(MODE == 1 ? 8 : 2) * Tc) * aG;
            a -= v;
            atomicAdd(&fc[g1], v);
            if ((q & 3) == 0) atomicAdd(&fc[gC], aG);
        } else if ((q & 3) == 0) {
            for (int e = 0; e < 8; ++e) {
                int X, Y, Z;
                face_xyz(F.axis, F.side, 1 + (e >> 2), 2 * ycl + (e & 1), 2 * zcl + ((e >> 1) & 1), n, X, Y, Z);
                add(F.blk, X, Y, Z, T(0.125) * aG);
            }
        }
        m.D[(i2 - 2 * Q.c0) * n + i1] = a;
    }
    scatter_c2f<T>(m, Q, F, T(1), add);
}

// Transposed restriction and correction, y_f += R^T e_c: every fine cell receives 1/8 of its parent's value (carried-over
// blocks all of it).  Interior only: the ghosts of y_f need an exchange.
template <typename T>
__global__ void k_inject(T *__restrict__ yf, LevelGeom gf, const T *__restrict__ ec, const XferItem *__restrict__ xf,
                         LevelGeom gc) {
    pdl_enter(yf, ec);
    const int nc = gc.n;
    const int64_t total = static_cast<int64_t>(gc.nb) << (3 * gc.lg);
    GRID_STRIDE(total) {
        int X, Y, Z;
        int64_t B;
        decode_cell(t, gc.lg, X, Y, Z, B);
        const XferItem xi = xf[B];
        const T v = ec[Lay<T>::at(gc, B, X + 1, Y + 1, Z + 1)];
        if (xi.kind == XF_COPY) {
            yf[Lay<T>::at(gf, xi.src[0], X + 1, Y + 1, Z + 1)] += v;
            continue;
        }
        int64_t b = xi.src[0];
        int x0 = 2 * X, y0 = 2 * Y, z0 = 2 * Z;
        if (xi.kind == XF_MERGE) {
            const int hc = nc >> 1, ox = X >= hc, oy = Y >= hc, oz = Z >= hc;
            b = xi.src[ox + 2 * oy + 4 * oz];
            x0 -= ox * nc;
            y0 -= oy * nc;
            z0 -= oz * nc;
        }
#pragma unroll
        for (int c = 0; c < 2; ++c)
#pragma unroll
            for (int bb = 0; bb < 2; ++bb)
#pragma unroll
                for (int a = 0; a < 2; ++a) yf[Lay<T>::at(gf, b, x0 + a + 1, y0 + bb + 1, z0 + c + 1)] += T(0.125) * v;
    }
}

// y += x over the interior, FP64.
__global__ void k_add(double *__restrict__ y, const double *__restrict__ x, LevelGeom g) {
    const int64_t total = static_cast<int64_t>(g.nb) << (3 * g.lg);
    GRID_STRIDE(total) {
        int xx, yy, zz;
        int64_t b;
        decode_cell(t, g.lg, xx, yy, zz, b);
        const int64_t gi = b * g.bs + off3(xx + 1, yy + 1, zz + 1, g.P);
        y[gi] += x[gi];
    }
}

// dL/dk = -lambda^T (dA/dk) u, written in the caller's layout.  A face between cells i and f with T = 2 k_i k_f / (k_i +
// k_f) enters rows i and f with (1/h^2) T (u_i - u_f) and its negative, and dT/dk_i = 2 k_f^2 / (k_i + k_f)^2 =
// T^2 / (2 k_i^2), so with T~ = T / h^2
//     dL/dk_i = -h^2 / 2 sum_f (T~_f / k_i)^2 (lambda_i - lambda_f) (u_i - u_f),
// where T~_f / k_i <= 2 / h^2 whatever the scale of k (T~_f^2 would overflow from k / h^2 = 2^512 on):
// one division per cell (six in the form with (k_i + k_f)^2, and the other cell's share by atomics: 5.5 ms on 31.5M cells;
// this one 2.5 ms, its 51 FP64 operations per cell at the measured FP64 rate; ncu: FP64 pipe 86 % active).  Ghosts of u and lambda: copies and
// reflections (at the boundary T = k_i, dT/dk_i = 1: the reflected pair gives the same).  Refinement interfaces are left to
// k_gradk_iface.
__global__ void k_gradk(const double *__restrict__ u, const double *__restrict__ lam, const double *__restrict__ k,
                        Coef cf, const double *__restrict__ h2, const int32_t *__restrict__ nbr6, LevelGeom g,
                        double *__restrict__ out, const int64_t *__restrict__ off) {
    const int n = g.n, P = g.P;
    const int64_t PP = static_cast<int64_t>(P) * P;
    const int64_t total = static_cast<int64_t>(g.nb) << (3 * g.lg);
    GRID_STRIDE(total) {
        int x, y, z;
        int64_t b;
        decode_cell(t, g.lg, x, y, z, b);
        const int64_t gi = b * g.bs + off3(x + 1, y + 1, z + 1, P);
        const double ui = u[gi], li = lam[gi], ki = k[gi];
        const double T[6] = {cf.tx[gi], cf.tx[gi + 1], cf.ty[gi], cf.ty[gi + P], cf.tz[gi], cf.tz[gi + PP]};
        const int64_t nb[6] = {gi - 1, gi + 1, gi - P, gi + P, gi - PP, gi + PP};
        const bool edge[6] = {x == 0, x == n - 1, y == 0, y == n - 1, z == 0, z == n - 1};
        const double rk = 1.0 / ki;
        double s = 0.0;
#pragma unroll
        for (int f = 0; f < 6; ++f) {
            if (edge[f] && nbr6[b * 6 + f] == -2) continue;
            const double w = T[f] * rk;
            s = fma((w * w) * (li - lam[nb[f]]), ui - u[nb[f]], s);
        }
        const int64_t at = off ? off[b] + (t & ((int64_t(1) << (3 * g.lg)) - 1)) : t;
        out[at] = -0.5 * h2[b] * s;
    }
}

// The interface faces' part of dL/dk, one thread per coarse cell of a quarter.  Fine face j (coefficient T_j of k_j and the
// injected coarse k_C) stands in the fine row with (1/h^2) T_j (u_j - g_j) and, conservative variant, with half of
// (1/h_C^2) T_j (g_j - u_j) in the coarse row; in the ghost-only variant the coarse row has its own face, of k_C and the mean
// of the eight fine k.
template <bool FLUX>
__global__ void k_gradk_iface(const double *__restrict__ u, const double *__restrict__ lam, const double *__restrict__ k,
                              Coef cf, const double *__restrict__ h2, const double *__restrict__ ih2,
                              const FaceItem *__restrict__ items, int nitems, LevelGeom g, Target<double> to) {
    const int n = g.n, lgh = g.lg - 1, h = n >> 1;
    const int64_t total = static_cast<int64_t>(nitems) << (2 * lgh);
    GRID_STRIDE(total) {
        const FaceItem F = items[t >> (2 * lgh)];
        const int q = static_cast<int>(t) & ((1 << (2 * lgh)) - 1), ycl = q & (h - 1), zcl = q >> lgh;
        const int yc = F.seg1 * h + ycl, zc = F.seg2 * h + zcl;
        int X, Y, Z;
        face_xyz(F.axis, 1 - F.side, 1, yc, zc, n, X, Y, Z);
        const int64_t gC = Lay<double>::at(g, F.nbr, X, Y, Z);
        const int64_t g0c = fidx<double>(g, F.nbr, F.axis, 1 - F.side, 0, yc, zc);
        const double lC = lam[gC], kC = k[gC], hf = h2[F.blk];
        const auto add_fine = [&](int d, int e, double v) {
            int x, y, z;
            face_xyz(F.axis, F.side, d, 2 * ycl + (e & 1), 2 * zcl + (e >> 1), n, x, y, z);
            add_to(to, g, F.blk, x, y, z, v);
        };
        double toC = 0.0;
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            const int64_t g0 = fidx<double>(g, F.blk, F.axis, F.side, 0, 2 * ycl + (e & 1), 2 * zcl + (e >> 1));
            const int64_t g1 = fidx<double>(g, F.blk, F.axis, F.side, 1, 2 * ycl + (e & 1), 2 * zcl + (e >> 1));
            const double T = face_coef<double, 1>(cf, F.side ? g0 : g1, F.side ? g1 : g0, F.axis) * hf;
            double w = -lam[g1] * ih2[F.blk];
            if (FLUX) w = fma(0.5 * lC, ih2[F.nbr], w);
            const double v = 0.5 * T * T * w * (u[g1] - u[g0]), kj = k[g1];
            add_fine(1, e, v / (kj * kj));
            toC += v / (kC * kC);
        }
        if (!FLUX) {
            const double T = face_coef<double, 1>(cf, F.side ? gC : g0c, F.side ? g0c : gC, F.axis) * h2[F.nbr];
            const double v = -0.5 * T * T * lC * ih2[F.nbr] * (u[gC] - u[g0c]), kG = k[g0c];
            toC += v / (kC * kC);
            for (int d = 1; d <= 2; ++d)
                for (int e = 0; e < 4; ++e) add_fine(d, e, 0.125 * v / (kG * kG));
        }
        add_to(to, g, F.nbr, X, Y, Z, toC);
    }
}

// ---------------------------------------------------------------------------------------------------------------
// Host side
// ---------------------------------------------------------------------------------------------------------------
// The transposed cycle's pools in its working precision: result, right-hand side, residual, interface adjoints.  FP32
// cycles run on the forward cycle's pools (dead between solves); FP64 ones too, but level 0's right-hand side is the
// forward solve's and has a pool of its own.
template <typename T>
struct APools {
    T *y, *f, *r, *old, *old_c;
};
template <typename T> APools<T> apools(mg_forest *F, int l);
template <> APools<double> apools<double>(mg_forest *F, int l) {
    DevLevel &d = F->L[l];
    return {d.u64, l == 0 ? F->a_fe : d.f64, static_cast<double *>(d.a_r), static_cast<double *>(d.a_old),
            static_cast<double *>(d.a_old_c)};
}
template <> APools<float> apools<float>(mg_forest *F, int l) {
    DevLevel &d = F->L[l];
    return {d.u32, d.f32, static_cast<float *>(d.a_r), static_cast<float *>(d.a_old), static_cast<float *>(d.a_old_c)};
}
template <typename T> const T *aih2(const DevLevel &d);
template <> const double *aih2<double>(const DevLevel &d) { return d.ih2_64; }
template <> const float *aih2<float>(const DevLevel &d) { return d.ih2_32; }
template <typename T> Coef acoef(const DevLevel &d);
template <> Coef acoef<double>(const DevLevel &d) { return d.c64(); }
template <> Coef acoef<float>(const DevLevel &d) { return d.c32(); }

// Calls fn(integral constant) with the coefficient mode of a level in precision T.
template <typename T, class Fn>
void with_mode(const mg_forest *F, const DevLevel &d, Fn &&fn) {
    if (!F->cfg.coeff) fn(std::integral_constant<int, 0>{});
    else if constexpr (sizeof(T) == 8) fn(std::integral_constant<int, 1>{});
    else if (d.face32) fn(std::integral_constant<int, 3>{});
    else fn(std::integral_constant<int, 2>{});
}

// Launch of an interface kernel, one CTA per strip of every item.
template <typename T, class Fn, class... Args>
void launch_iface(mg_forest *F, const DevLevel &d, Fn fn, Args... args) {
    const int n = d.g.n;
    launch_pdl(F->st, !F->batch_member, fn, d.nifaces * iface_strips(n), iface_threads(n),
               scatter_values(n) * sizeof(T), args...);
}

// Transposed interface ghosts of y (ghosts) and sgn times the interface part of A^T y into `to` (see k_adj_iface).
template <typename T>
void adj_iface(mg_forest *F, DevLevel &d, T *y, bool ghosts, T *old, T *old_c, Target<T> to, T sgn) {
    if (!d.nifaces) return;
    Prof p(F, P_ADJ, 1);
    with_mode<T>(F, d, [&](auto m) {
        constexpr int M = decltype(m)::value;
        auto *fn = F->cfg.interface_flux ? (ghosts ? k_adj_iface<T, M, true, true> : k_adj_iface<T, M, true, false>)
                                         : (ghosts ? k_adj_iface<T, M, false, true> : k_adj_iface<T, M, false, false>);
        launch_iface<T>(F, d, fn, y, acoef<T>(d), aih2<T>(d), d.ifaces, d.g, old, old_c, to, sgn);
    });
}

// What of A^T y on a level is no 7-point stencil with the block's own coefficients, brought up to date in y's ghosts and in f.
template <typename T>
void adj_update(mg_forest *F, DevLevel &d, const APools<T> &a) {
    adj_iface<T>(F, d, a.y, true, a.old, a.old_c, {a.f, nullptr, nullptr}, T(-1));
    if (!d.a_old_s) return;
    Prof p(F, P_ADJ, 1);
    constexpr int M = sizeof(T) == 8 ? 1 : 3;  // face-averaged coarse levels only
    launch_pdl(F->st, !F->batch_member, k_adj_uneven<T, M>,
               grid_for(static_cast<int64_t>(d.nsfaces) << (2 * d.g.lg)), kThreads, 0, a.y, acoef<T>(d), aih2<T>(d),
               d.sfaces, d.nsfaces, d.g, static_cast<T *>(d.a_old_s), a.f);
}

// E^T of level c's interface ghosts, from the finer level d's residual r (gather) or from fc's own ghosts.
template <typename T>
void et_iface(mg_forest *F, DevLevel &d, DevLevel &c, T *fc, const T *r, bool gather) {
    if (!c.nifaces) return;
    Prof p(F, P_ADJ, 1);
    with_mode<T>(F, c, [&](auto m) {
        constexpr int M = decltype(m)::value;
        auto *fn = F->cfg.interface_flux ? (gather ? k_et_iface<T, M, true, true> : k_et_iface<T, M, true, false>)
                                         : (gather ? k_et_iface<T, M, false, true> : k_et_iface<T, M, false, false>);
        launch_iface<T>(F, c, fn, fc, acoef<T>(c), c.ifaces, c.g, r, d.g, d.xfer);
    });
}

// Ghosts of y filled from one source block (same level, boundary).
template <typename T>
void exchange_same(mg_forest *F, DevLevel &d, T *y) {
    if (!d.nsfaces) return;
    Prof p(F, P_ADJ, 1);
    launch_pdl(F->st, !F->batch_member, k_exchange_faces<T, false>,
               grid_for(static_cast<int64_t>(d.nsfaces) << (2 * d.g.lg)), kThreads, 0, y, d.sfaces, d.nsfaces, d.g,
               Skip{}, 0, nullptr);
}

// Red-black iterations on A^T with the colours in reverse order.  `stale`: y changed since the last interface exchange.
template <typename T>
void smooth_T(mg_forest *F, int l, int iters, bool &stale) {
    DevLevel &d = F->L[l];
    const APools<T> a = apools<T>(F, l);
    for (int i = 0; i < iters; ++i)
        for (int colour = 1; colour >= 0; --colour) {
            if (stale) adj_update<T>(F, d, a);
            if constexpr (sizeof(T) == 4) {
                smooth_level32(F, d, colour);
            } else {
                Prof p(F, P_ADJ, 1);
                auto *fn = F->cfg.coeff ? k_smooth<double, 1> : k_smooth<double, 0>;
                launch_pdl(F->st, !F->batch_member, fn, grid_for(d.cells() / 2), kThreads, 0, a.y, a.f, d.c64(),
                           d.h2_64, d.g, colour, d.nbr6, Skip{}, nullptr);
            }
            stale = true;
        }
}

// The FP32 residual of a level with block edge 4 .. 128 on its own pools into r.
void launch_residual32(mg_forest *F, DevLevel &d, float *r) {
    with_mode<float>(F, d, [&](auto m) {
        constexpr int M = decltype(m)::value;
        static constexpr decltype(&k_adj_residual32<M, 2>) fns[6] = {
            k_adj_residual32<M, 2>, k_adj_residual32<M, 3>, k_adj_residual32<M, 4>,
            k_adj_residual32<M, 5>, k_adj_residual32<M, 6>, k_adj_residual32<M, 7>};
        const int64_t pairs = d.cells() / 2;
        launch_pdl(F->st, !F->batch_member, fns[d.g.lg - 2], static_cast<unsigned>((pairs + kThreads - 1) / kThreads),
                   kThreads, 0, d.u32, d.f32, d.c32(), d.ih2_32, d.g.bs, pairs, d.nbr6, r);
    });
}

// y = M_l^T f (level l's pools), in precision T, from y = 0 with zero ghosts; the coarsest level's dense inverse is FP64.
template <typename T>
void vcycle_T(mg_forest *F, int l) {
    DevLevel &d = F->L[l];
    const APools<T> a = apools<T>(F, l);
    const int last = static_cast<int>(F->L.size()) - 1;
    if (l == last) {
        Prof p(F, P_ADJ, 1);
        launch_pdl(F->st, !F->batch_member, k_coarse_solve<T>, (F->Nc * 32 + kThreads - 1) / kThreads, kThreads, 0, a.y,
                   a.f, F->AinvT, sizeof(T) == 4 ? F->cmap32 : F->cmap, F->uprob, F->ustart, F->moff, F->Nc, nullptr);
        return;
    }
    const int64_t n2 = static_cast<int64_t>(d.g.n) * d.g.n;
    if (d.nifaces) {
        cudaMemsetAsync(a.old, 0, d.nifaces * n2 * sizeof(T), F->st);
        if (a.old_c) cudaMemsetAsync(a.old_c, 0, d.nifaces * n2 / 4 * sizeof(T), F->st);
    }
    if (d.a_old_s) cudaMemsetAsync(d.a_old_s, 0, d.nsfaces * n2 * sizeof(T), F->st);
    bool stale = false;
    smooth_T<T>(F, l, F->cfg.nu2, stale);
    if (stale) adj_update<T>(F, d, a);
    DevLevel &c = F->L[l + 1];
    const APools<T> ac = apools<T>(F, l + 1);
    {
        Prof p(F, P_ADJ, 1);
        if (sizeof(T) == 4 && smooth32_specialised(d))
            launch_residual32(F, d, reinterpret_cast<float *>(a.r));
        else
            with_mode<T>(F, d, [&](auto m) {
                launch_pdl(F->st, !F->batch_member, k_adj_residual<T, decltype(m)::value>, grid_for(d.cells()),
                           kThreads, 0, a.y, a.f, acoef<T>(d), aih2<T>(d), d.g, d.nbr6, a.r, nullptr, nullptr);
            });
    }
    const bool gather = d.all_halve;
    if (sizeof(T) == 4 && transfer_specialised(d)) {
        Prof p(F, P_ADJ, 1);
        static constexpr decltype(&k_prolong_T32<3>) fns[5] = {k_prolong_T32<3>, k_prolong_T32<4>, k_prolong_T32<5>,
                                                               k_prolong_T32<6>, k_prolong_T32<7>};
        launch_pdl(F->st, !F->batch_member, fns[d.g.lg - 3],
                   static_cast<unsigned>((c.cells() + kThreads - 1) / kThreads), kThreads, 0,
                   reinterpret_cast<float *>(a.r), d.g.bs, c.f32, c.u32, d.xfer, c.cells(), c.g.bs);
    } else if (gather) {
        Prof p(F, P_ADJ, 1);
        launch_pdl(F->st, !F->batch_member, k_prolong_T<T>, grid_for(c.cells()), kThreads, 0, a.r, d.g, ac.f, ac.y,
                   d.xfer, c.g);
    } else {
        Prof p(F, P_ADJ, 2);
        cudaMemsetAsync(ac.f, 0, c.pool_elems() * sizeof(T), F->st);
        cudaMemsetAsync(ac.y, 0, c.pool_elems() * sizeof(T), F->st);
        launch_pdl(F->st, !F->batch_member, k_prolong_T_scatter<T>, grid_for(c.cells()), kThreads, 0, a.r, d.g, ac.f,
                   d.xfer, c.g);
        if (c.nsfaces)
            launch_pdl(F->st, !F->batch_member, k_et_faces<T>,
                       grid_for(static_cast<int64_t>(c.nsfaces) << (2 * c.g.lg)), kThreads, 0, ac.f, c.sfaces,
                       c.nsfaces, c.g);
    }
    et_iface<T>(F, d, c, ac.f, a.r, gather);
    vcycle_T<T>(F, l + 1);
    bool through = false;  // the injection wrote same-level and boundary ghosts
    {
        Prof p(F, P_ADJ, 1);
        if constexpr (sizeof(T) == 4) through = inject32(F, d, c);
        if (!through)
            launch_pdl(F->st, !F->batch_member, k_inject<T>, grid_for(c.cells()), kThreads, 0, a.y, d.g, ac.y, d.xfer,
                       c.g);
    }
    if (!through) exchange_same<T>(F, d, a.y);
    stale = true;
    smooth_T<T>(F, l, F->cfg.nu1, stale);
}

mg_status ensure_adjoint_pools(mg_forest *F) {
    MG_TRY(ensure_fp64_coefficients(F));
    if (F->a_g) return MG_OK;
    const bool fp32 = F->cfg.precision == 1;
    const int64_t tb = fp32 ? sizeof(float) : sizeof(double);
    const int64_t bytes0 = F->L[0].pool_elems() * static_cast<int64_t>(sizeof(double));
    void *p;
    bool uneven = false;  // faces with two coefficients: from where a merge took away an interface, under face averaging
    for (size_t l = 0; l < F->L.size(); ++l) {
        DevLevel &d = F->L[l];
        const int64_t n2 = static_cast<int64_t>(d.g.n) * d.g.n, adj = d.nifaces * n2 * tb;
        if (l > 0 && F->cfg.coeff && F->cfg.coarse_coef == 1 && !F->L[l - 1].all_halve) uneven |= F->L[l - 1].nifaces > 0;
        if (uneven && d.nsfaces && l + 1 < F->L.size()) MG_TRY(forest_alloc(F, &d.a_old_s, d.nsfaces * n2 * tb));
        MG_TRY(forest_alloc(F, &d.a_r, d.pool_elems() * tb));
        if (adj) MG_TRY(forest_alloc(F, &d.a_old, adj));
        if (adj && !F->cfg.interface_flux) MG_TRY(forest_alloc(F, &d.a_old_c, adj / 4));
    }
    MG_TRY(forest_alloc(F, &p, bytes0));
    F->a_lam = static_cast<double *>(p);
    MG_TRY(forest_alloc(F, &p, bytes0));
    F->a_fe = static_cast<double *>(p);
    MG_TRY(forest_alloc(F, &p, bytes0));
    F->a_g = static_cast<double *>(p);
    return MG_OK;
}

mg_status read_sum(mg_forest *F, int grid, double *out) {
    k_sum_partials<<<1, kThreads, 0, F->st>>>(F->partial, grid, F->sums);
    MG_CUDA(cudaMemcpyAsync(F->pinned, F->sums, sizeof(double), cudaMemcpyDeviceToHost, F->st));
    MG_CUDA(cudaStreamSynchronize(F->st));
    *out = F->pinned[0];
    return MG_OK;
}

// The transposed operator and cycle are written for the quadratic coarse-to-fine scheme, red-black Gauss-Seidel, the
// dense coarsest solve and homogeneous boundary data (the k-gradient of a boundary term would need g).
mg_status adjoint_supported(const mg_forest *F) {
    if (F->cfg.c2f_variant != 0 || F->cfg.smoother != 0 || F->cfg.coarse_iters != 0 || F->cfg.prolongation != 0) {
        set_error("the adjoint needs c2f_variant 0, the Gauss-Seidel smoother, the dense coarsest solve and the "
                  "face-neighbour linear prolongation");
        return MG_ERR_INVALID_ARG;
    }
    if (F->gb) {
        set_error("the adjoint needs homogeneous boundary data (mg_set_boundary(forest, NULL))");
        return MG_ERR_STATE;
    }
    return MG_OK;
}

// Half a defect-correction step: r = g - A^T lambda (r = g while lambda is 0).  FP32 cycles: r scaled by `mult` into the
// level-0 FP32 right-hand side, its result zeroed; FP64 cycles: r into the level-0 right-hand side a_fe, u64 zeroed.
// rr: the volume-weighted ||g||^2 over all problems on entry, ||r||^2 on exit, in FP64 like the test it is for.
template <int MODE>
mg_status adjoint_residual(mg_forest *F, bool zero, double mult, double *rr) {
    DevLevel &d = F->L[0];
    const double *f = F->a_g;
    if (!zero) {
        if (F->cfg.precision == 0) exchange_same<double>(F, d, F->a_lam);  // else k_update_mixed wrote these ghosts
        if (d.nifaces) {
            // FP32 cycles leave a_fe alone, so it differs from g only where the last step added to it
            if (F->cfg.precision == 1) {
                auto *fn = F->cfg.interface_flux ? k_adj_restore<true> : k_adj_restore<false>;
                fn<<<d.nifaces * iface_strips(d.g.n), iface_threads(d.g.n), 0, F->st>>>(F->a_fe, F->a_g, d.ifaces, d.g);
            } else {
                MG_CUDA(cudaMemcpyAsync(F->a_fe, F->a_g, d.pool_elems() * sizeof(double), cudaMemcpyDeviceToDevice, F->st));
            }
            adj_iface<double>(F, d, F->a_lam, true, nullptr, nullptr, {F->a_fe, nullptr, nullptr}, -1.0);
            f = F->a_fe;
        }
    }
    if (F->cfg.precision == 1) {
        const std::vector<double> m(F->np, mult);
        set_scales_host(F, m);
        MG_TRY(enqueue_scales(F));
        const int cpb = F->bsum_cpb;
        Prof p(F, P_ADJ, 1);
        MG_CUDA(cudaMemsetAsync(F->bsum, 0, static_cast<size_t>(d.g.nb) * cpb * sizeof(double), F->st));
        if (zero) {
            MG_CUDA(cudaMemsetAsync(d.u32, 0, d.pool_elems() * sizeof(float), F->st));
            k_scaled_rhs<<<d.g.nb * cpb, kThreads, 0, F->st>>>(f, d.vol_32, d.g, cpb, d.f32, F->pscale, d.bprob, F->bsum,
                                                               Skip{});
            MG_CUDA(cudaStreamSynchronize(F->st));  // the scales' host copies may change again
            return MG_OK;
        }
        k_residual_norm<MODE, true><<<d.g.nb * cpb, kThreads, 0, F->st>>>(F->a_lam, f, d.c64(), d.ih2_64, d.vol_32, d.g,
                                                                          cpb, d.f32, F->pscale, d.bprob, F->bsum, d.u32,
                                                                          Skip{}, d.vol_64);
        MG_TRY(enqueue_problem_sums(F));
        MG_CUDA(cudaStreamSynchronize(F->st));
        *rr = 0.0;
        for (int p2 = 0; p2 < F->np; ++p2) *rr += F->psum_h[p2];
        return MG_OK;
    }
    const int grid = grid_for(d.cells());
    {
        Prof p(F, P_ADJ, 1);
        k_adj_residual<double, MODE><<<grid, kThreads, 0, F->st>>>(F->a_lam, f, d.c64(), d.ih2_64, d.g, nullptr, F->a_fe,
                                                                   d.vol_64, F->partial);
    }
    MG_CUDA(cudaMemsetAsync(d.u64, 0, d.pool_elems() * sizeof(double), F->st));
    return read_sum(F, grid, rr);
}

template <int MODE>
mg_status adjoint_solve(mg_forest *F, const double *u_dev, const double *dLdu_dev, double *lambda_dev,
                        double *dLdk_dev, double rtol, int max_cycles) {
    MG_TRY(ensure_adjoint_pools(F));
    DevLevel &d = F->L[0];
    const int grid = grid_for(d.cells());
    MG_CUDA(cudaMemsetAsync(F->a_lam, 0, d.pool_elems() * sizeof(double), F->st));
    k_pack<double><<<grid, kThreads, 0, F->st>>>(F->a_g, dLdu_dev, d.g, F->leaf_off);
    if (d.nifaces) k_pack<double><<<grid, kThreads, 0, F->st>>>(F->a_fe, dLdu_dev, d.g, F->leaf_off);
    k_norm64<<<grid, kThreads, 0, F->st>>>(F->a_g, d.vol_64, d.g, F->partial);
    double gg = 0.0;
    MG_TRY(read_sum(F, grid, &gg));
    const double gn = std::sqrt(gg);
    double rel = gn > 0.0 ? 1.0 : 0.0, mult = pow2_near(1.0 / gn);
    int it = 0;
    // Defect correction lambda += M^T (g - A^T lambda): the residual and the update in FP64; the transposed cycle
    // M^T in FP64, or, on forests with FP32 forward cycles, in FP32 on the residual scaled by a power of two near
    // 1 / ||r|| of the step before (the forward solve's mixed precision, transposed)
    for (; gn > 0.0; ++it) {
        double rr = gg;
        MG_TRY(adjoint_residual<MODE>(F, it == 0, mult, &rr));
        rel = std::sqrt(rr) / gn;
        if (!std::isfinite(rel) || rel <= rtol || it >= max_cycles) break;
        if (F->cfg.precision == 1) {
            MG_TRY(replay(F, F->vT_rec, [&] { vcycle_T<float>(F, 0); }));
            Prof p(F, P_ADJ, 1);
            k_update_mixed<false><<<update_grid(d), kThreads, 0, F->st>>>(F->a_lam, d.u32, F->pinv, d.bprob, d.g, d.nbr6,
                                                                        nullptr, Skip{});
        } else {
            MG_TRY(replay(F, F->vT_rec, [&] { vcycle_T<double>(F, 0); }));
            Prof p(F, P_ADJ, 1);
            k_add<<<grid, kThreads, 0, F->st>>>(F->a_lam, d.u64, d.g);
        }
        mult = pow2_near(1.0 / std::sqrt(rr));
    }
    k_unpack<double><<<grid, kThreads, 0, F->st>>>(lambda_dev, F->a_lam, d.g, F->leaf_off);
    MG_CUDA(cudaGetLastError());
    if (dLdk_dev && F->cfg.coeff) {
        // forward ghosts of u; lambda's were filled by the last residual (and are 0 while lambda is)
        MG_TRY(ensure_scratch64(F));
        k_pack<double><<<grid, kThreads, 0, F->st>>>(F->s64a, u_dev, d.g, F->leaf_off);
        exchange_any64(F, d, F->s64a);
        Prof p(F, P_ADJ, 1 + (d.nifaces > 0));
        k_gradk<<<grid, kThreads, 0, F->st>>>(F->s64a, F->a_lam, d.k64, d.c64(), d.h2_64, d.nbr6, d.g, dLdk_dev,
                                              F->leaf_off);
        if (d.nifaces) {
            auto *fn = F->cfg.interface_flux ? k_gradk_iface<true> : k_gradk_iface<false>;
            fn<<<grid_for(static_cast<int64_t>(d.nifaces) << (2 * (d.g.lg - 1))), kThreads, 0, F->st>>>(
                F->s64a, F->a_lam, d.k64, d.c64(), d.h2_64, d.ih2_64, d.ifaces, d.nifaces, d.g,
                Target<double>{nullptr, dLdk_dev, F->leaf_off});
        }
    }
    MG_CUDA(cudaStreamSynchronize(F->st));
    if (F->cfg.precision == 1) MG_TRY(check_kernel_waits(F));
    if (!std::isfinite(rel) || rel > rtol) {
        set_error("adjoint: relative residual " + fmt_e(rel) + " above rtol after " + std::to_string(it) +
                  " cycles");
        return MG_ERR_NOT_CONVERGED;
    }
    return MG_OK;
}

}  // namespace
}  // namespace octmg

using namespace octmg;

extern "C" mg_status mg_apply_transpose(mg_forest *F, const double *y_dev, double *ATy_dev) {
    if (!F || !y_dev || !ATy_dev) {
        set_error("null argument");
        return MG_ERR_INVALID_ARG;
    }
    if (F->cfg.coeff && !F->rhs_set) {
        set_error("mg_set_rhs (k) has not been called");
        return MG_ERR_STATE;
    }
    MG_TRY(adjoint_supported(F));
    MG_TRY(ensure_fp64_coefficients(F));
    MG_TRY(ensure_scratch64(F));
    DevLevel &d = F->L[0];
    // the stencil on y with the transposed ghosts, then the interface part added to the caller's field
    k_pack<double><<<grid_for(d.cells()), kThreads, 0, F->st>>>(F->s64a, y_dev, d.g, F->leaf_off);
    exchange_same<double>(F, d, F->s64a);
    adj_iface<double>(F, d, F->s64a, true, nullptr, nullptr, {nullptr, nullptr, nullptr}, 1.0);
    apply64(F, d, F->s64a, ATy_dev, true);
    adj_iface<double>(F, d, F->s64a, false, nullptr, nullptr, {nullptr, ATy_dev, F->leaf_off}, 1.0);
    MG_CUDA(cudaStreamSynchronize(F->st));
    return MG_OK;
}

extern "C" mg_status mg_adjoint_solve(mg_forest *F, const double *u_dev, const double *dLdu_dev, double *lambda_dev,
                                      double *dLdk_dev, double rtol, int32_t max_cycles) {
    if (!F || !dLdu_dev || !lambda_dev || (dLdk_dev && !u_dev) || max_cycles < 0 || !(rtol >= 0.0)) {
        set_error("bad argument");
        return MG_ERR_INVALID_ARG;
    }
    MG_TRY(check_ready(F));
    MG_TRY(adjoint_supported(F));
    if (F->cfg.coeff) return adjoint_solve<1>(F, u_dev, dLdu_dev, lambda_dev, dLdk_dev, rtol, max_cycles);
    return adjoint_solve<0>(F, u_dev, dLdu_dev, lambda_dev, dLdk_dev, rtol, max_cycles);
}

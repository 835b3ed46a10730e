// Inversion of the coarsest-level operators (this library's direct coarsest solver), every problem's dense block at once:
// in-place Gauss-Jordan elimination with partial pivoting, W columns (a panel) per step.
//
// One step on panel columns J = [c0, c0 + W): eliminating them one after another inside the panel alone leaves in it the
// columns J of the product M of the W elementary transformations (in-place elimination stores exactly those; the other
// columns of M are the identity's).  So the panel is eliminated first, by one thread-block cluster per problem that holds
// it in distributed shared memory (k_gj_panel), and the W transformations then reach the rest of the matrix as one
// product of rank W over the whole GPU (k_gj_update):
//     Y[r, j] = (r in J ? 0 : X[src r, j]) + sum_w M[r, J_w] X[src J_w, j]   (j not in J),   Y[:, J] = M[:, J],
// with src the row exchanges of the panel.  After all panels the matrix holds (P A)^-1 = A^-1 P^T for the exchanges P,
// and org[r] the row of A that ended in row r, so A^-1[:, org r] is column r.
//
// What bounds it: the chain of N pivot searches (2.3 us each with 512 unknowns, 2.9 us with 1728: one cluster barrier, one
// block barrier, a division, and the panel's update on the 2 FP64 FMA per clock of each of the cluster's SMs), then the
// FP64 rate in the update.  Elimination of one column per step with two launches per column (every element rewritten each
// time) took 4.85 ms for 512 unknowns and 58 ms for 1728 (three root blocks per axis); this takes 1.5 ms and 10.1 ms.
// Operators without interfaces take their pivots on the diagonal (k_gj_panel_diag), symmetric ones half of the updates:
// 0.65 ms and 4.4 ms.
#include <cooperative_groups.h>

#include "forest_state.h"

namespace octmg {
namespace {
namespace cg = cooperative_groups;

constexpr int kGjCluster = 8;  // CTAs that share a panel's rows (the portable cluster size)
constexpr int kGjThreads = 256;
constexpr int kGjTile = 32;    // the update's output tile edge

// One candidate pivot row of a panel column, as each CTA of the cluster receives it.
template <int W>
struct GjCand {
    uint64_t key;   // magnitude bits + 1 (0: none): non-negative binary64 values order as their bits
    double rcp;     // 1 / pivot
    double row[W];  // the row's panel entries
    int32_t r, id;  // its row and the row of the matrix it came from
};
template <int W>
struct GjRow {
    double row[W];
    int32_t id;
};

// Rows of a problem held by one CTA (r % cluster size == rank), and its dynamic shared memory: rows x W doubles (rounded up
// to whole passes of the CTA) and the rows' origins.
__host__ __device__ constexpr int gj_rows(int N) { return (N + kGjCluster - 1) / kGjCluster; }
__host__ __device__ constexpr int64_t gj_panel_elems(int N, int W) {
    return (static_cast<int64_t>(gj_rows(N)) * W + kGjThreads - 1) / kGjThreads * kGjThreads;
}
constexpr int64_t gj_smem(int N, int W) { return gj_panel_elems(N, W) * 8 + static_cast<int64_t>(gj_rows(N)) * 4; }

// The key of a pivot candidate: its magnitude bits + 1, or 0 for NaN.
__device__ __forceinline__ uint64_t a_key(const double *a, int i) {
    const uint64_t bits = static_cast<uint64_t>(__double_as_longlong(a[i])) & ~(1ull << 63);
    return bits <= 0x7ff0000000000000ull ? bits + 1 : 0;
}

// Whether `pivot` can be a diagonal pivot of a problem with N unknowns whose matrix had `before` there.  Elimination of a
// diagonally dominant matrix leaves a positive pivot; the roundings of up to N updates of this entry, each at most eps / 2 of
// it, move it by less than N eps times what it was, so a pivot above that has its sign and some digits, and one below may be
// noise (cells coupled to each other by more than 1 / (N eps) times what couples them to the rest).
__device__ __forceinline__ bool dominant_pivot(double pivot, double before, int N) {
    return pivot > N * 2.220446049250313e-16 * before && pivot <= 1.7976931348623157e308;
}

// Eliminates panel columns c0 .. c0 + W - 1 of every problem with more than c0 unknowns, one cluster per problem, row r in
// CTA r % 8.  Per column one cluster barrier: before it each CTA sends the others its best pivot
// candidate with the whole panel row and the reciprocal, and the owner of the diagonal row sends that one; after it every
// CTA picks the same winner (largest magnitude, lowest row on ties) and updates its rows.  Messages alternate between two
// buffers: a CTA that writes a buffer again has passed a barrier that every reader of it reached afterwards.  A thread
// keeps one column of the panel (W divides the CTA); the W threads of a row share a warp, so the multiplier comes by
// shuffle.  A zero or non-finite pivot sets *bad and the elimination goes on with the diagonal row.  In a problem of kind
// GJ_DOMINANT the diagonal row is the only candidate, and one that is no dominant_pivot sets *bad too (dg: the diagonal before
// the elimination, kept by the first panel).
template <int W>
__global__ void __cluster_dims__(kGjCluster, 1, 1) __launch_bounds__(kGjThreads)
    k_gj_panel(const double *__restrict__ A, const int64_t *__restrict__ moff, const int64_t *__restrict__ ustart, int c0,
               double *__restrict__ panel, int32_t *__restrict__ src, const int8_t *__restrict__ kind,
               double *__restrict__ dg, int *__restrict__ bad) {
    extern __shared__ __align__(16) unsigned char gj_raw[];
    __shared__ GjCand<W> cand[2][kGjCluster];
    __shared__ GjRow<W> diag[2];
    __shared__ int act;
    const cg::cluster_group cluster = cg::this_cluster();
    const int p = blockIdx.x / kGjCluster, rank = static_cast<int>(cluster.block_rank());
    const bool diagonal = kind && kind[p];
    const int N = static_cast<int>(ustart[p + 1] - ustart[p]);
    if (c0 >= N) return;  // uniform over the cluster, before any barrier
    const int wn = min(W, N - c0), nr = (N - rank + kGjCluster - 1) / kGjCluster;  // row i of this CTA: rank + 8 i
    const auto row_of = [&](int i) { return rank + i * kGjCluster; };
    double *a = reinterpret_cast<double *>(gj_raw);
    int32_t *id = reinterpret_cast<int32_t *>(a + gj_panel_elems(N, W));
    const int tid = threadIdx.x, lane = tid & 31, col = tid & (W - 1);
    const double *Ap = A + moff[p];
    for (int e = tid; e < gj_panel_elems(N, W); e += kGjThreads) {
        const int row = e / W;
        a[e] = row < nr && col < wn ? Ap[static_cast<int64_t>(row_of(row)) * N + c0 + col] : 0.0;
    }
    for (int i = tid; i < nr; i += kGjThreads) {
        id[i] = row_of(i);
        if (diagonal && c0 == 0) dg[ustart[p] + row_of(i)] = Ap[static_cast<int64_t>(row_of(i)) * N + row_of(i)];
    }
    // rows of zeros stay as they are (a zero multiplier, never a pivot): the panel ends at the last other row, or at its own
    // rows, which receive the pivot rows
    if (tid == 0) act = 0;
    __syncthreads();
    int last = (min(c0 + W, N) - 1 - rank + kGjCluster) / kGjCluster;  // local rows up to row c0 + wn - 1
    for (int e = tid; e < nr * W; e += kGjThreads)
        if (a[e] != 0.0) last = max(last, e / W + 1);
    atomicMax(&act, last);
    cluster.sync();
    const int na = act;
    for (int cc = 0; cc < wn; ++cc) {
        const int c = c0 + cc, buf = cc & 1;
        const bool checks = diagonal && rank == 0 && tid == 0;
        const double before = !checks ? 0.0 : (c0 == 0 ? Ap[static_cast<int64_t>(c) * N + c] : dg[ustart[p] + c]);
        if (tid < 32) {
            uint64_t best = 0;
            int at = -1;
            for (int i = (max(0, c - rank) + kGjCluster - 1) / kGjCluster + lane; i < na; i += 32) {
                const uint64_t key = !diagonal || row_of(i) == c ? a_key(a, i * W + cc) : 0;
                if (key > best) {
                    best = key;
                    at = i;
                }
            }
            // the warp's largest, its upper word first, then the lower one, then the lowest row
            const uint32_t hi = static_cast<uint32_t>(best >> 32), top = __reduce_max_sync(0xffffffffu, hi);
            const uint32_t lo = __reduce_max_sync(0xffffffffu, hi == top ? static_cast<uint32_t>(best) : 0u);
            best = static_cast<uint64_t>(top) << 32 | lo;
            at = static_cast<int>(__reduce_min_sync(
                0xffffffffu, hi == top && at >= 0 && a_key(a, at * W + cc) == best ? static_cast<uint32_t>(at) : 0x7fffffffu));
            const double rcp = best ? 1.0 / a[at * W + cc] : 0.0;
            for (int to = 0; to < kGjCluster; ++to) {
                GjCand<W> *m = cluster.map_shared_rank(&cand[buf][rank], to);
                if (best && lane < W) m->row[lane] = a[at * W + lane];
                if (lane == 0) {
                    m->key = best;
                    m->rcp = rcp;
                    m->r = best ? row_of(at) : N;
                    m->id = best ? id[at] : -1;
                }
            }
        } else if (tid < 64 && c % kGjCluster == rank) {
            for (int to = 0; to < kGjCluster; ++to) {
                GjRow<W> *m = cluster.map_shared_rank(&diag[buf], to);
                if (lane < W) m->row[lane] = a[c / kGjCluster * W + lane];
                if (lane == 0) m->id = id[c / kGjCluster];
            }
        }
        cluster.sync();
        int win = 0;
#pragma unroll
        for (int i = 1; i < kGjCluster; ++i) {
            const GjCand<W> &x = cand[buf][i], &y = cand[buf][win];
            if (x.key > y.key || (x.key == y.key && x.r < y.r)) win = i;
        }
        const GjCand<W> &w = cand[buf][win];
        // usable: found, not zero (key 1) and not infinite
        const bool ok = w.key > 1 && w.key < 0x7ff0000000000001ull;
        if (rank == 0 && tid == 0 && (!ok || (checks && !dominant_pivot(w.row[cc], before, N)))) atomicOr(bad, 1);
        const int q = ok ? w.r : c;
        const double *prow = ok ? w.row : diag[buf].row;
        const double v = ok ? w.rcp : 1.0 / diag[buf].row[cc];
        const double pv = col == cc ? v : prow[col] * v;  // row c of the eliminated panel
        const double dc = diag[buf].row[col];
#pragma unroll 4
        for (int base = 0; base < na * W; base += kGjThreads) {
            const int e = base + tid, r = row_of(e / W);
            const double x = r == q ? dc : a[e];  // row q now holds the former row c
            const double fr = W == 1 ? x : __shfl_sync(0xffffffffu, x, (lane & ~(W - 1)) | cc);
            const double out = fma(-fr, pv, col == cc ? 0.0 : x);
            if (e < na * W) a[e] = r == c ? pv : out;
        }
        if (tid == 0) {  // q == c: the second store keeps the row's own origin
            if (q % kGjCluster == rank) id[q / kGjCluster] = diag[buf].id;
            if (c % kGjCluster == rank) id[c / kGjCluster] = ok ? w.id : diag[buf].id;
        }
        __syncthreads();
    }
    for (int e = tid; e < nr * W; e += kGjThreads) panel[(ustart[p] + row_of(e / W)) * W + col] = a[e];
    for (int i = tid; i < nr; i += kGjThreads) src[ustart[p] + row_of(i)] = id[i];
    cluster.sync();  // no CTA leaves while another may still write to its shared memory
}

// The panel's transformations on the whole matrix, X -> Y (see the top), and the composed row origins org_in -> org_out
// (c0 = 0: from the identity).  One CTA per 32 x 32 output tile, its 32 x W and W x 32 factors in shared memory; a tile with
// a factor of zeros is copied, which the unknowns' order makes frequent: with the unknowns sorted by position a row of the
// operator reaches no further than a plane of cells, so before column c only the first c + plane rows and columns are touched
// (1728 unknowns: 2.15e9 of 5.16e9 FMA, 5.1 instead of 9.0 ms).  Problems with c0 unknowns or fewer are copied through.
// GJ_SYMMETRIC: the problem's matrix is symmetric and eliminated without row exchanges.  It then stays symmetric up to a
// sign, Y[j, r] = Y[r, j] where both or neither of r and j are eliminated and -Y[r, j] otherwise, and the tiles above the
// diagonal are written from those below: with 1728 unknowns 30 us per update instead of 47, and a gradient on 48^3 cells 8.2
// instead of 9.8 ms.
template <int W>
__global__ void __launch_bounds__(kGjThreads)
    k_gj_update(const double *__restrict__ X, double *__restrict__ Y, const int64_t *__restrict__ moff,
                const int64_t *__restrict__ ustart, int c0, const double *__restrict__ panel,
                const int32_t *__restrict__ src, const int32_t *__restrict__ org_in, int32_t *__restrict__ org_out,
                const int8_t *__restrict__ kind) {
    constexpr int T = kGjTile, ROWS = kGjThreads / T;  // rows of the tile per pass
    __shared__ double M[T][W], B[W][T];
    __shared__ int32_t from[T];
    __shared__ double low[T][T + 1];
    const int p = blockIdx.z;
    const bool sym = kind && (kind[p] & GJ_SYMMETRIC);
    if (sym && blockIdx.x > blockIdx.y) return;
    const int64_t u0 = ustart[p];
    const int N = static_cast<int>(ustart[p + 1] - u0);
    const int j0 = blockIdx.x * T, i0 = blockIdx.y * T;
    if (j0 >= N || i0 >= N) return;
    const double *x = X + moff[p];
    double *y = Y + moff[p];
    const int tx = threadIdx.x % T, ty = threadIdx.x / T, j = j0 + tx;
    const bool done = c0 >= N;
    bool m_any = false, b_any = false;
    if (threadIdx.x < T) {
        const int r = i0 + threadIdx.x;
        const int s = r < N && !done ? src[u0 + r] : r;
        from[threadIdx.x] = s;
        if (blockIdx.x == 0 && r < N) org_out[u0 + r] = c0 == 0 ? s : org_in[u0 + s];
    }
    if (!done) {
        for (int e = threadIdx.x; e < T * W; e += kGjThreads) {
            const int r = i0 + e / W;
            const double v = r < N ? panel[(u0 + r) * W + e % W] : 0.0;
            M[e / W][e % W] = v;
            m_any = m_any || v != 0.0;
        }
        for (int e = threadIdx.x; e < T * W; e += kGjThreads) {
            const int w = e / T, jj = j0 + e % T;
            const double v = c0 + w < N && jj < N ? x[static_cast<int64_t>(src[u0 + c0 + w]) * N + jj] : 0.0;
            B[w][e % T] = v;
            b_any = b_any || v != 0.0;
        }
    }
    const bool product = __syncthreads_or(m_any) && __syncthreads_or(b_any);
#pragma unroll
    for (int k = 0; k < T / ROWS; ++k) {
        const int i = ty + k * ROWS, r = i0 + i;
        if (r >= N || j >= N) continue;
        const bool in_j = !done && r >= c0 && r < c0 + W;
        double s = in_j ? 0.0 : x[static_cast<int64_t>(from[i]) * N + j];
        if (!done) {
            if (j >= c0 && j < c0 + W) {
                s = M[i][j - c0];
            } else if (product) {
#pragma unroll
                for (int w = 0; w < W; ++w) s = fma(M[i][w], B[w][tx], s);
            }
        }
        y[static_cast<int64_t>(r) * N + j] = s;
        if (sym) low[i][tx] = s;
    }
    if (!sym || i0 == j0) return;  // uniform over the CTA
    __syncthreads();
    const int r = i0 + tx;  // now along the rows of the tile above the diagonal
    if (r >= N) return;
#pragma unroll
    for (int k = 0; k < T / ROWS; ++k) {
        const int jj = j0 + ty + k * ROWS;  // < N: j0 < i0 < N and both are multiples of T
        const double s = low[tx][ty + k * ROWS];
        y[static_cast<int64_t>(jj) * N + r] = (r < c0 + W) == (jj < c0 + W) ? s : -s;
    }
}

// A^-1 from the eliminated matrix R, its columns put back: X[:, org r] = R[:, r].
__global__ void k_gj_unpermute(const double *__restrict__ R, double *__restrict__ X, const int64_t *__restrict__ moff,
                               const int64_t *__restrict__ ustart, const int32_t *__restrict__ org) {
    const int p = blockIdx.y;
    const int N = static_cast<int>(ustart[p + 1] - ustart[p]);
    const int64_t NN = static_cast<int64_t>(N) * N;
    for (int64_t e = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x; e < NN;
         e += static_cast<int64_t>(gridDim.x) * blockDim.x) {
        const int r = static_cast<int>(e / N), k = static_cast<int>(e - static_cast<int64_t>(r) * N);
        X[moff[p] + static_cast<int64_t>(r) * N + org[ustart[p] + k]] = R[moff[p] + e];
    }
}
__global__ void k_gj_transpose(const double *__restrict__ X, double *__restrict__ T, const int64_t *__restrict__ moff,
                               const int64_t *__restrict__ ustart) {
    const int p = blockIdx.y;
    const int N = static_cast<int>(ustart[p + 1] - ustart[p]);
    const int64_t NN = static_cast<int64_t>(N) * N;
    for (int64_t e = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x; e < NN;
         e += static_cast<int64_t>(gridDim.x) * blockDim.x) {
        const int r = static_cast<int>(e / N), k = static_cast<int>(e - static_cast<int64_t>(r) * N);
        T[moff[p] + static_cast<int64_t>(k) * N + r] = X[moff[p] + e];
    }
}

// The panel when no problem needs row exchanges (GJ_DIAGONAL): the pivot rows are then the panel's own W = 16 rows,
// so each CTA eliminates these and kGjRows others by itself and nothing passes between CTAs.  A thread keeps one entry of
// the pivot rows and one of its CTA's rows in registers; the W threads of a row share a warp, and the pivot row of a step
// goes through one of two shared buffers (who writes a buffer again has passed the barrier after its last read).  The
// operations and their order are those of k_gj_panel for a problem of kind GJ_DOMINANT.  Bound by the chain of a
// shuffle, a reciprocal, a barrier and an update per column: 9.5 us per panel, where the cluster's search takes 37 us with
// 512 unknowns and 46 us with 1728 (new coefficients and a solve on 128^3 cells 3.79 -> 2.94 ms, a gradient on 48^3 cells
// with 1728 coarsest unknowns 13.8 -> 9.8 ms).
constexpr int kGjRows = 16;
__global__ void __launch_bounds__(kGjThreads)
    k_gj_panel_diag(const double *__restrict__ A, const int64_t *__restrict__ moff, const int64_t *__restrict__ ustart, int c0,
                    double *__restrict__ panel, int32_t *__restrict__ src, double *__restrict__ dg, int *__restrict__ bad) {
    constexpr int W = 16;
    static_assert(kGjRows == W && kGjThreads == W * W, "one entry of each half per thread");
    __shared__ double prow[2][W];
    const int p = blockIdx.y;
    const int64_t u0 = ustart[p];
    const int N = static_cast<int>(ustart[p + 1] - u0), r0 = blockIdx.x * kGjRows;
    if (c0 >= N || r0 >= N) return;  // uniform over the CTA
    const int i = threadIdx.x / W, col = threadIdx.x % W, lane = threadIdx.x & 31, wn = min(W, N - c0);
    const int r = r0 + i;
    const double *a = A + moff[p];
    double d = i < wn && col < wn ? a[static_cast<int64_t>(c0 + i) * N + c0 + col] : 0.0;
    double x = r < N && col < wn ? a[static_cast<int64_t>(r) * N + c0 + col] : 0.0;
    // the diagonal before the elimination, kept by the first panel; the pivot rows' own CTA (c0 is a multiple of W) checks
    const bool own = r0 == c0;
    double before = 0.0;
    if (c0 == 0 && r < N) {
        before = a[static_cast<int64_t>(r) * N + r];
        if (col == 0) dg[u0 + r] = before;
    } else if (own && r < N) {
        before = dg[u0 + r];
    }
    bool lost = false;
    for (int cc = 0; cc < wn; ++cc) {
        const int from = (lane & ~(W - 1)) | cc;
        const double fd = __shfl_sync(0xffffffffu, d, from), fx = __shfl_sync(0xffffffffu, x, from);
        double *row = prow[cc & 1];
        if (i == cc) {
            lost = lost || !dominant_pivot(fd, before, N);
            const double v = 1.0 / fd;
            row[col] = col == cc ? v : d * v;
        }
        __syncthreads();
        const double pv = row[col];
        d = i == cc ? pv : fma(-fd, pv, col == cc ? 0.0 : d);
        x = fma(-fx, pv, col == cc ? 0.0 : x);
    }
    if (own) {
        x = d;
        if (lost) atomicOr(bad, 1);
    }
    if (r >= N) return;
    panel[(u0 + r) * W + col] = x;
    if (col == 0) src[u0 + r] = r;
}

constexpr int64_t kGjMaxSmem = 200 * 1024;

template <int W>
void invert(mg_forest *F, int maxN, GjPivots pivots) {
    const int8_t *kind = pivots == GJ_SEARCH_ALL ? nullptr : F->gj_kind;
    if (pivots != GJ_DIAGONAL) cudaFuncSetAttribute(k_gj_panel<W>, cudaFuncAttributeMaxDynamicSharedMemorySize, kGjMaxSmem);
    const unsigned tiles = static_cast<unsigned>((maxN + kGjTile - 1) / kGjTile);
    const int steps = (maxN + W - 1) / W;
    double *X = steps % 2 ? F->Ainv : F->AinvT, *Y = steps % 2 ? F->AinvT : F->Ainv;
    int32_t *in = F->gj_org, *out = F->gj_org + F->Nc;
    for (int c0 = 0; c0 < maxN; c0 += W) {
        if (pivots == GJ_DIAGONAL)
            k_gj_panel_diag<<<dim3(static_cast<unsigned>((maxN + kGjRows - 1) / kGjRows), F->np), kGjThreads, 0, F->st>>>(
                X, F->moff, F->ustart, c0, F->gj_panel, F->gj_src, F->gj_diag, F->flag);
        else
            k_gj_panel<W><<<F->np * kGjCluster, kGjThreads, gj_smem(maxN, W), F->st>>>(
                X, F->moff, F->ustart, c0, F->gj_panel, F->gj_src, kind, F->gj_diag, F->flag);
        k_gj_update<W><<<dim3(tiles, tiles, F->np), kGjThreads, 0, F->st>>>(X, Y, F->moff, F->ustart, c0, F->gj_panel,
                                                                            F->gj_src, in, out, kind);
        std::swap(X, Y);
        std::swap(in, out);
    }
    const dim3 grid(static_cast<unsigned>(std::min<int64_t>(1024, (static_cast<int64_t>(maxN) * maxN + 255) / 256)),
                    static_cast<unsigned>(F->np));
    k_gj_unpermute<<<grid, 256, 0, F->st>>>(F->AinvT, F->Ainv, F->moff, F->ustart, in);
    k_gj_transpose<<<grid, 256, 0, F->st>>>(F->Ainv, F->AinvT, F->moff, F->ustart);
}

}  // namespace

// Panel width: 16 columns where the pivots are on the diagonal, and while a panel's rows fit the cluster's shared memory
// (12,800 unknowns in 8 x 200 KB); narrower panels above.  Wider ones would make the panel's own FP64 work the longer part.
int gj_width(int maxN, GjPivots pivots) {
    return pivots == GJ_DIAGONAL || gj_smem(maxN, 16) <= kGjMaxSmem ? 16 : (gj_smem(maxN, 4) <= kGjMaxSmem ? 4 : 1);
}

// The buffer the caller fills with the operators before enqueue_gauss_jordan (the eliminated matrix ends in AinvT).
double *gj_input(mg_forest *F, int maxN, GjPivots pivots) {
    const int w = gj_width(maxN, pivots);
    return (maxN + w - 1) / w % 2 ? F->Ainv : F->AinvT;
}

// Ainv and AinvT (the transposes) from the operators in gj_input; a singular one sets *F->flag (cleared by the caller).
// A problem without interfaces on this level (GJ_DOMINANT) has 7-point rows, diagonally dominant by rows.  Elimination on the
// diagonal keeps that of what is left, so a scaled pivot row's other entries sum to at most 1 and no row's sum of magnitudes
// grows: nothing is gained by a search for pivots, which is left out when all problems are of this kind (GJ_DIAGONAL).
// Where coefficients differ by more than binary64 resolves, rounding can cancel a pivot all the same or leave noise in its
// place (dominant_pivot): the flag says so, and the caller comes again with GJ_SEARCH_ALL.
void enqueue_gauss_jordan(mg_forest *F, int maxN, GjPivots pivots) {
    switch (gj_width(maxN, pivots)) {
        case 16: invert<16>(F, maxN, pivots); break;
        case 4: invert<4>(F, maxN, pivots); break;
        default: invert<1>(F, maxN, pivots); break;
    }
}

}  // namespace octmg

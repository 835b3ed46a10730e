// The paper's coarsest solver (Sec. 5: 256 damped Jacobi sweeps) in one launch.  The coarsest level is a few blocks of 4^3
// cells, so a sweep launched as an exchange and an update is two launches of about 2 us each for a microsecond of work:
// 1.0 ms per cycle for 8 blocks (512 unknowns).  Here one cluster of eight CTAs keeps the blocks in shared memory, CTA c
// those with b % 8 == c, and a sweep is: ghosts of the own blocks from the neighbours' interiors (distributed shared
// memory), a CTA barrier, the update into the second buffer, a cluster barrier.  323 us per cycle (1.26 us per sweep), bound by
// these two barriers and the chain of eight FP64 operations between them.
#include <cooperative_groups.h>

#include "forest_state.h"

namespace octmg {
namespace {
namespace cg = cooperative_groups;

constexpr int kCjCluster = 8, kCjThreads = 256;
constexpr int kCjN = 4, kCjP = kCjN + 2, kCjBlock = kCjP * kCjP * kCjP;  // every coarsest level has 4^3 blocks
constexpr int kCjArrays = 7;  // u (two buffers), f and, with variable coefficients, tx, ty, tz, 1 / diagonal

// The same operations in the same order as k_exchange_faces (boundary and same-level faces) and k_jacobi64.
template <int MODE>
__global__ void __cluster_dims__(kCjCluster, 1, 1) __launch_bounds__(kCjThreads)
    k_coarse_jacobi(double *__restrict__ u, const double *__restrict__ f, Coef cf, const double *__restrict__ h2,
                    const int32_t *__restrict__ nbr6, LevelGeom g, double omega, int iters, Skip skip) {
    pdl_enter(u, f);
    extern __shared__ __align__(16) unsigned char cj_raw[];
    double *sm = reinterpret_cast<double *>(cj_raw);
    const cg::cluster_group cluster = cg::this_cluster();
    const int rank = static_cast<int>(cluster.block_rank()), per = (g.nb + kCjCluster - 1) / kCjCluster;
    const int mine = g.nb > rank ? (g.nb - rank + kCjCluster - 1) / kCjCluster : 0;  // blocks rank, rank + 8, ..
    const int stride = per * kCjBlock;
    const double *src[kCjArrays] = {u, u, f, cf.tx, cf.ty, cf.tz, cf.dinv};
    for (int a = 0; a < (MODE == 1 ? 7 : 3); ++a)
        for (int i = threadIdx.x; i < mine * kCjBlock; i += kCjThreads)
            sm[a * stride + i] = src[a][(rank + i / kCjBlock * kCjCluster) * g.bs + i % kCjBlock];
    cluster.sync();
    const double *sf = sm + 2 * stride;
    const Coef sc{sm + 3 * stride, sm + 4 * stride, sm + 5 * stride, nullptr, sm + 6 * stride,
                  nullptr,         nullptr,         nullptr,         nullptr};
    for (int it = 0; it < iters; ++it) {
        double *cur = sm + (it & 1) * stride, *nxt = sm + ((it + 1) & 1) * stride;
        for (int i = threadIdx.x; i < mine * 6 * kCjN * kCjN; i += kCjThreads) {
            const int lb = i / (6 * kCjN * kCjN), r = i % (6 * kCjN * kCjN), face = r / (kCjN * kCjN);
            const int axis = face >> 1, side = face & 1, i1 = r % kCjN, i2 = r / kCjN % kCjN;
            const int nb = nbr6[(rank + lb * kCjCluster) * 6 + face];
            double v;
            if (nb >= 0) {
                const double *there = cluster.map_shared_rank(cur, nb % kCjCluster);
                v = there[nb / kCjCluster * kCjBlock + face_off(axis, 1 - side, 1, i1, i2, kCjN, kCjP)];
            } else {
                v = -cur[lb * kCjBlock + face_off(axis, side, 1, i1, i2, kCjN, kCjP)];
            }
            cur[lb * kCjBlock + face_off(axis, side, 0, i1, i2, kCjN, kCjP)] = v;
        }
        __syncthreads();
        for (int i = threadIdx.x; i < mine * kCjN * kCjN * kCjN; i += kCjThreads) {
            const int lb = i >> 6, x = i & 3, y = (i >> 2) & 3, z = (i >> 4) & 3, b = rank + lb * kCjCluster;
            const int64_t gi = lb * kCjBlock + off3(x + 1, y + 1, z + 1, kCjP);
            double nw = cur[gi];
            if (!skip(b)) {
                if constexpr (MODE == 1)
                    nw = sten1(cur, sc, gi, kCjP, sf[gi]) * sc.dinv[gi];
                else
                    nw = fma(h2[b], sf[gi], sten0<double>(cur, gi, kCjP)) * (1.0 / 6.0);
                nw = fma(omega, nw - cur[gi], cur[gi]);
            }
            nxt[gi] = nw;
        }
        cluster.sync();
    }
    const double *res = sm + (iters & 1) * stride;
    for (int i = threadIdx.x; i < mine * kCjN * kCjN * kCjN; i += kCjThreads) {
        const int64_t c = off3((i & 3) + 1, ((i >> 2) & 3) + 1, ((i >> 4) & 3) + 1, kCjP);
        u[(rank + (i >> 6) * kCjCluster) * g.bs + c] = res[(i >> 6) * kCjBlock + c];
    }
}

}  // namespace

static size_t smem_bytes(const mg_forest *F, const DevLevel &d) {
    const int arrays = F->cfg.coeff ? kCjArrays : 3, per = (d.g.nb + kCjCluster - 1) / kCjCluster;
    return static_cast<size_t>(arrays) * per * kCjBlock * sizeof(double);
}

// Whether the one-launch form applies to coarsest level d: no refinement interface (its ghosts depend on several blocks), no
// boundary data (level 0 of a one-level forest), blocks that fit the cluster's shared memory (128 with variable coefficients).
bool coarse_jacobi_fits(const mg_forest *F, const DevLevel &d) {
    return d.g.n == kCjN && !d.nifaces && !(&d == &F->L[0] && F->gb) && smem_bytes(F, d) <= 200 * 1024;
}

// `iters` sweeps from the level's u64, which receives the result (interior only).
void launch_coarse_jacobi(mg_forest *F, DevLevel &d, int iters) {
    auto *fn = F->cfg.coeff ? k_coarse_jacobi<1> : k_coarse_jacobi<0>;
    cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024);
    launch_pdl(F->st, false, fn, kCjCluster, kCjThreads, smem_bytes(F, d), d.u64, d.f64, d.c64(), d.h2_64, d.nbr6, d.g,
               F->omega, iters, Skip{d.bprob, done_mask(F)});
}

}  // namespace octmg

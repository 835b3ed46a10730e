// Forest state shared by the solver translation units: device level structures and the opaque mg_forest.
#pragma once
#include <algorithm>
#include <cstdio>
#include <string>
#include <utility>
#include <array>
#include <vector>

#include <cuda_runtime.h>

#include "kernels.cuh"
#include "octmg_internal.h"

namespace octmg {

#define MG_CUDA(call)                                                                          \
    do {                                                                                       \
        cudaError_t e_ = (call);                                                               \
        if (e_ != cudaSuccess) {                                                               \
            set_error(std::string(#call) + ": " + cudaGetErrorString(e_));                     \
            return MG_ERR_CUDA;                                                                \
        }                                                                                      \
    } while (0)

#define MG_TRY(expr)                      \
    do {                                  \
        mg_status s_ = (expr);            \
        if (s_ != MG_OK) return s_;       \
    } while (0)

// A kernel that begins with pdl_enter, launched so that its start-up overlaps the end of the kernel before it in the stream
// (programmatic dependent launch; captured as such in the recorded cycles).
template <class... P, class... A>
void launch_pdl(cudaStream_t st, bool overlap, void (*fn)(P...), unsigned grid, unsigned threads, size_t smem, A &&...args) {
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cfg.attrs = attr;
    cfg.numAttrs = overlap && grid <= kPdlGrid ? 1 : 0;
    cudaLaunchKernelEx(&cfg, fn, static_cast<P>(args)...);
}

constexpr int kMaxGrid = 152 * 32;  // grid-stride loops: at most 32 CTAs of 256 threads per SM

inline int grid_for(int64_t total) {
    int64_t g = (total + kThreads - 1) / kThreads;
    return static_cast<int>(std::max<int64_t>(1, std::min<int64_t>(g, kMaxGrid)));
}

struct DevLevel {
    LevelGeom g{};
    FaceItem *faces = nullptr;
    int nfaces = 0;
    SegItem *segs = nullptr;
    int nsegs = 0;
    XferItem *xfer = nullptr;  // from this level to the next (per block of the next level)
    double *h2_64 = nullptr, *ih2_64 = nullptr, *vol_64 = nullptr;  // per block h^2, 1/h^2, h^3
    float *h2_32 = nullptr, *ih2_32 = nullptr, *vol_32 = nullptr;
    double *u64 = nullptr, *f64 = nullptr;
    double *u64b = nullptr;  // second FP64 iterate pool (damped Jacobi)
    float *u32 = nullptr, *f32 = nullptr;
    double *k64 = nullptr, *tx = nullptr, *ty = nullptr, *tz = nullptr, *dg = nullptr, *dinv = nullptr;
    float *kap = nullptr;
    int32_t *bprob = nullptr;  // problem of each block
    int32_t *nbr6 = nullptr;   // per block face: same-level neighbour, -1 boundary, -2 refinement interface
    FaceItem *ifaces = nullptr;  // the C2F faces alone: each with the coarse quarter face it covers, an interface item
    int nifaces = 0;
    FaceItem *sfaces = nullptr;  // the other faces: boundary and same level
    int nsfaces = 0;
    bool all_halve = false;  // every block of the next level is a halved block of this one
    // FP32 smoother launch shape (kind, parameters): {1, ZC, threads, 0, 0} k_smooth32, {2, TY, TZ, D, R}
    // k_smooth32t; kind 0 = not chosen yet
    std::array<int32_t, 5> s32{0, 0, 0, 0, 0};
    // transposed cycles (allocated by the first adjoint call, in the cycles' precision): residual pool, and per interface
    // item the ghost adjoints that the right-hand side already holds
    void *a_r = nullptr, *a_old = nullptr, *a_old_c = nullptr;
    // same-level faces whose two blocks hold different coefficients (a merged level under face averaging): per face cell the
    // value on the other side that the right-hand side already holds (null: the level has none)
    void *a_old_s = nullptr;
    // FP32 cycles on a face-averaged coarse level: its halved face coefficients (colour-split) and mode 3
    float *ax32 = nullptr, *ay32 = nullptr, *az32 = nullptr;
    bool face32 = false;
    DiagItem *edges = nullptr, *corners = nullptr;  // trilinear prolongation: edge / corner items of every block
    int nedges = 0, ncorners = 0;
    Coef c64() const { return Coef{tx, ty, tz, dg, dinv, nullptr, nullptr, nullptr, nullptr}; }
    Coef c32() const { return Coef{nullptr, nullptr, nullptr, nullptr, nullptr, kap, ax32, ay32, az32}; }
    int64_t pool_elems() const { return static_cast<int64_t>(g.nb) * g.bs; }
    int64_t cells() const { return static_cast<int64_t>(g.nb) << (3 * g.lg); }
};

// CTAs of k_update_mixed: one thread per pair of cells in kUpdatePlanes planes.
inline unsigned update_grid(const DevLevel &d) {
    return static_cast<unsigned>((d.cells() / (2 * kUpdatePlanes) + kThreads - 1) / kThreads);
}

// One FP32 level as the persistent tail kernel sees it.
struct TailLevel {
    LevelGeom g;
    float *u, *f;
    const float *kap, *h2, *ih2;
    const FaceItem *sfaces, *ifaces;
    const XferItem *xfer;  // to the next level
    const int32_t *nbr6, *bprob;
    int nsfaces, nifaces;
    int fast;  // the transfers to the next level use the specialised kernels (every block halves, edge 8..128)
    const float *ax, *ay, *az;  // halved face coefficients of a face-averaged coarse level (mode 3)
    int face32;                 // 1: this level's smoothing, ghosts and restriction use them
};

// One step of the tail's V-cycle; every step is followed by a grid barrier.
enum TailOp : int32_t {
    T_SMOOTH0 = 0, T_SMOOTH1, T_EXCH_IFACE, T_EXCH_FULL, T_RESTRICT, T_PROLONG, T_COARSE
};
struct TailPhase {
    int32_t op, level;
};

// Everything the tail kernel reads of one forest (its level descriptors, phase list, coarsest inverse, done-mask and
// the barrier and error words of its launch).
struct TailArgs {
    const TailLevel *L;
    const TailPhase *ph;
    int nph;
    int flux;  // conservative F2C ghosts
    const double *Ainv;
    const int64_t *cmap32;
    const int32_t *uprob;
    const int64_t *ustart, *moff;
    int Nc;
    const uint8_t *done;
    unsigned *bar;  // arrivals
    int *err;
};

// One entry of a batch's joint tail: phase P of group `group`'s recorded tail; a grid barrier follows the entry when
// `last` is set (the entries between two barriers belong to different groups and are independent).
struct BatchEntry {
    int32_t group, last;
    TailPhase P;
};

// A launch sequence that depends only on the forest, recorded as a CUDA graph and replayed (see replay below).
struct Replay {
    cudaGraphExec_t exec = nullptr;
    int runs = 0;
    bool off = false;  // the recording failed or cannot be replayed: launched directly
    int64_t nlaunch[32] = {};  // its launches per kernel family, counted at every replay
    // What it records has changed: the next run is a first one again, and a recording that failed is tried again.
    void drop() {
        if (exec) cudaGraphExecDestroy(exec);
        exec = nullptr;
        runs = 0;
        off = false;
    }
};

}  // namespace octmg

struct mg_forest {
    mg_config cfg{};
    cudaStream_t st = nullptr;
    octmg::HostHierarchy H;
    std::vector<octmg::DevLevel> L;
    std::vector<void *> allocs;
    double *Ainv = nullptr;
    int64_t *cmap = nullptr;    // coarsest unknowns' offsets in the FP64 pools (natural layout)
    int64_t *cmap32 = nullptr;  // ... and in the colour-split FP32 pools
    int Nc = 0;
    double *partial = nullptr;  // 2 * kMaxGrid
    double *sums = nullptr;     // 2 doubles on the device
    double *pinned = nullptr;   // 2 doubles, host pinned
    double *s64a = nullptr;     // level-0 FP64 scratch pool
    double *coarse_r = nullptr;               // coarsest-level scratch pool (operator assembly)
    int *flag = nullptr;                      // input-check flag
    double *gb = nullptr;                     // 2 g on the finest level's boundary faces (mg_set_boundary), or null
    double *gb_pool = nullptr;                // its storage (kept when g is reset to 0)
    double omega = 0.8;                       // damping of the Jacobi smoother
    int *kerr = nullptr;                      // set by a device wait that gave up (staged smoother)
    double *AinvT = nullptr;                  // transpose of the coarsest inverses (adjoint cycles)
    double *gj_panel = nullptr;                // device Gauss-Jordan: the eliminated panel, its row exchanges
    int32_t *gj_src = nullptr, *gj_org = nullptr;  // and the composed row origins (two buffers)
    double *gj_diag = nullptr;  // the operators' diagonals before the elimination
    int8_t *gj_kind = nullptr;  // per problem: GJ_DOMINANT, GJ_SYMMETRIC (assemble_coarse)
    cudaStream_t cap_st = nullptr;             // private stream: graph recording, host-input copies
    // recorded sequences: coarsest-level probe + inversion (assemble_coarse), FP64 V-cycle, FP32 V-cycle, transposed V-cycle
    octmg::Replay coarse_rec, v64_rec, v32_rec, vT_rec;
    double *hst_f = nullptr, *hst_k = nullptr, *hst_u = nullptr;  // mg_solve_host staging buffers (user layout)
    cudaEvent_t hst_ev = nullptr;              // orders the staging copies against the forest's stream
    int32_t *pnbu = nullptr;                   // interface-free coarsest level: the unknowns of each 7-point row (-1: outside)
    // several independent problems: per-problem reductions, scales, block-diagonal coarsest inverse
    int np = 1;
    int32_t *pstart = nullptr, *pblk = nullptr;  // level-0 blocks of problem p: pblk[pstart[p] .. pstart[p+1])
    double *bsum = nullptr;                      // per-CTA partial sums of h^3 x^2 over level 0, bsum_cpb per block
    int bsum_cpb = 1;
    uint8_t *guess_zero = nullptr;               // per chunk of level 0: the initial guess is 0 there (k_pack_nonzero)
    double *psum = nullptr, *psum_h = nullptr;   // per-problem sums (device, pinned host)
    float *pscale = nullptr, *pscale_h = nullptr;  // per-problem power-of-two residual scale (device, pinned host)
    double *pinv = nullptr, *pinv_h = nullptr;     // its inverse in FP64
    uint8_t *pdone = nullptr, *pdone_h = nullptr;  // per problem: met rtol in the running solve (device, pinned host)
    int32_t *uprob = nullptr;                    // coarsest unknown -> problem
    int64_t *ustart = nullptr, *moff = nullptr;  // coarsest unknowns / inverse offsets per problem
    std::vector<int64_t> ustart_h, moff_h;
    std::vector<double> fnorm_p;                 // ||f|| per problem
    int64_t *leaf_off = nullptr;                 // optional: start of every leaf in the user arrays (elements)
    bool batch_member = false;                   // inputs are checked by the owning batch
    // adjoint right-hand side, solution, and right-hand side with the interface part moved to it (level 0)
    double *a_g = nullptr, *a_lam = nullptr, *a_fe = nullptr;
    bool rhs_set = false;
    double fnorm = 0.0;
    // per-kernel-family launch counters (always on) and CUDA-event timing (mg_profile)
    bool prof = false;
    int64_t nlaunch[32] = {};
    std::vector<cudaEvent_t> ev_pool;
    size_t ev_used = 0;
    std::vector<std::pair<int, size_t>> recs;  // (family, index of the start event; stop = +1)
    // persistent tail: the FP32 V-cycle from level tail_level down is one cooperative launch (tail_level < 0: off)
    int tail_level = -1;
    bool tail_tuned = false;
    octmg::TailLevel *tail_L = nullptr;  // device copy of the level descriptors
    octmg::TailPhase *tail_ph = nullptr;  // device phase list
    int tail_nph = 0, tail_for = -2;      // phases recorded, and for which tail level
    unsigned *tail_bar = nullptr;          // grid-barrier arrivals
    std::vector<octmg::TailPhase> tail_ph_host;  // host copy of the phase list (merged into a batch's joint tail)
};


namespace octmg {
// Kernel families for launch counting and timing.
enum ProfCat {
    P_EXCH64 = 0, P_EXCH32, P_SMOOTH64, P_SMOOTH32, P_RESTR64, P_RESTR32, P_PROL64, P_PROL32, P_COARSE64,
    P_COARSE32, P_RESID64, P_UPDATE, P_LAYOUT, P_ADJ, P_SMOOTH64_L0, P_SMOOTH32_L0, P_TAIL32, P_NCAT
};
template <typename T> constexpr int cat_of(int cat64) { return sizeof(T) == 8 ? cat64 : cat64 + 1; }

cudaEvent_t next_event(mg_forest *F);

// The done-mask of the forest's problems.  A problem that is solved alone needs none: its solve ends when it is done, and
// without a mask a kernel starts two dependent loads earlier (0.5 us of a launch of 3).  In a batch it does, also as the
// only one of its block size: the others go on.
inline uint8_t *done_mask(const mg_forest *F) { return F->np > 1 || F->batch_member ? F->pdone : nullptr; }

// RAII scope around the launches of one kernel family (a negative family: no accounting).
struct Prof {
    mg_forest *F;
    int cat;
    size_t start = 0;
    bool on = false;
    Prof(mg_forest *f, int c, int launches) : F(f), cat(c) {  // c < 0: inside another family's scope, not counted
        if (c < 0) return;
        F->nlaunch[c] += launches;
        if (F->prof) {
            cudaEvent_t a = next_event(F), b = next_event(F);
            if (a && b) {
                start = F->ev_used - 2;
                cudaEventRecord(a, F->st);
                on = true;
            }
        }
    }
    ~Prof() {
        if (on) {
            cudaEventRecord(F->ev_pool[start + 1], F->st);
            F->recs.emplace_back(cat, start);
        }
    }
};

inline std::string fmt_e(double v) {
    char b[32];
    std::snprintf(b, sizeof(b), "%.3e", v);
    return b;
}

// Runs `body` (launches on F->st that depend only on the forest) as a recorded CUDA graph: directly the first time (it loads
// the kernels, which a capture does not allow), recorded at the second on the private stream (the forest's may be the legacy
// default stream, which cannot be captured), replayed on the forest's stream from then on.  One launch per step costs the
// host about 5 us each, more than most of the coarse levels' kernels last.  Directly also while profiling (per-family
// events), while the caller's stream is being captured, and when the recording fails or `recorded()`, called after it,
// says that it cannot be replayed.
template <class Body, class Ok>
mg_status replay(mg_forest *F, Replay &r, Body &&body, Ok &&recorded) {
    cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
    MG_CUDA(cudaStreamIsCapturing(F->st, &cap));
    if (F->prof || r.off || cap != cudaStreamCaptureStatusNone || r.runs++ == 0) {
        body();
        MG_CUDA(cudaGetLastError());
        return MG_OK;
    }
    if (!r.exec) {
        cudaGraph_t graph = nullptr;
        cudaError_t e = F->cap_st ? cudaSuccess : cudaStreamCreateWithFlags(&F->cap_st, cudaStreamNonBlocking);
        if (e == cudaSuccess) e = cudaStreamBeginCapture(F->cap_st, cudaStreamCaptureModeThreadLocal);
        bool ok = false;
        if (e == cudaSuccess) {
            int64_t before[32];
            std::copy(F->nlaunch, F->nlaunch + 32, before);
            cudaStream_t own = F->st;
            F->st = F->cap_st;
            body();
            F->st = own;
            e = cudaStreamEndCapture(F->cap_st, &graph);
            const cudaError_t launch = cudaGetLastError();  // of one that failed without ending the capture
            if (e == cudaSuccess) e = launch;
            ok = recorded();
            for (int c = 0; c < 32; ++c) {
                r.nlaunch[c] = F->nlaunch[c] - before[c];
                F->nlaunch[c] = before[c];
            }
        }
        if (e == cudaSuccess && graph && ok) e = cudaGraphInstantiate(&r.exec, graph, 0);
        if (graph) cudaGraphDestroy(graph);
        if (e != cudaSuccess || !ok || !r.exec) {
            r.exec = nullptr;
            r.off = true;
            cudaGetLastError();
            body();
            MG_CUDA(cudaGetLastError());
            return MG_OK;
        }
    }
    MG_CUDA(cudaGraphLaunch(r.exec, F->st));
    for (int c = 0; c < 32; ++c) F->nlaunch[c] += r.nlaunch[c];
    return MG_OK;
}
template <class Body>
mg_status replay(mg_forest *F, Replay &r, Body &&body) {
    return replay(F, r, body, [] { return true; });
}

// FP64 operator application A u on a level (ghosts of u already exchanged) into a padded pool, or into a field in the
// caller's layout (user, level 0), defined in solver.cu.
void apply64(mg_forest *F, DevLevel &d, const double *u, double *out, bool user = false);

// FP64 ghost exchange of one level on a pool laid out like the level's pools (defined in solver.cu).
void exchange_any64(mg_forest *F, DevLevel &d, double *u);
// Device allocation owned by the forest (freed by mg_forest_destroy), zero-filled (defined in solver.cu).
mg_status forest_alloc(mg_forest *F, void **p, int64_t bytes);
mg_status check_ready(mg_forest *F);
mg_status check_kernel_waits(mg_forest *F);
mg_status launch_tail32(mg_forest *F);  // tail.cu
octmg::TailArgs tail_args(mg_forest *F);  // tail.cu: the forest's recorded tail as the kernel reads it
// tail.cu: a batch's joint tail, one cooperative launch on groups[0]'s stream walking `ne` entries (device) over the
// groups' tail arguments (device), with a grid of at most `need` CTAs
mg_status launch_batch_tail32(mg_forest *const *groups, const octmg::TailArgs *args, const octmg::BatchEntry *entries,
                              int ne, unsigned *bar, int64_t need);
// coarse_jacobi.cu: the coarsest level's Jacobi sweeps in one launch, where it applies
bool coarse_jacobi_fits(const mg_forest *F, const DevLevel &d);
void launch_coarse_jacobi(mg_forest *F, DevLevel &d, int iters);
// gauss_jordan.cu: inverses of the coarsest operators (input buffer, panel width, launches)
// How the coarsest elimination finds its pivots: on the diagonal in all problems; by search, on the diagonal in those of kind
// GJ_DOMINANT; by search in all (gauss_jordan.cu, enqueue_gauss_jordan).
enum GjPivots { GJ_DIAGONAL, GJ_SEARCH, GJ_SEARCH_ALL };
enum GjKind : int8_t { GJ_DOMINANT = 1, GJ_SYMMETRIC = 2 };
double *gj_input(mg_forest *F, int maxN, GjPivots pivots);
int gj_width(int maxN, GjPivots pivots);
void enqueue_gauss_jordan(mg_forest *F, int maxN, GjPivots pivots);
int64_t tail_ctas(mg_forest *F);  // tail.cu: CTAs the largest phase of F's tail can use
// solver.cu: one FP32 V-cycle in two parts around a joint tail: part 1 the steps down to the tail level's entry,
// part 2 the steps after the tail (0: the whole cycle, its tail launched as usual)
void vcycle32_part(mg_forest *F, int part);
// solver.cu: u64 += e32 / scale_p (set: u64 = e32 / scale_p), same-level and boundary ghosts written
mg_status enqueue_update_mixed(mg_forest *F, bool set = false);
mg_status set_tail_level(mg_forest *F, int l);  // solver.cu
mg_status drop_cycles32(mg_forest *F);          // solver.cu
mg_status launch_selftest_wait(mg_forest *F, int which);  // tail.cu (F->tail_bar allocated)
void reset_done(mg_forest *F);
mg_status enqueue_done(mg_forest *F);
mg_status reference_norms(mg_forest *F);
mg_status ensure_scratch64(mg_forest *F);
mg_status create(const mg_config *cfg, mg_forest **out);
mg_status set_rhs(mg_forest *F, const double *f_dev, const double *k_dev);
double pow2_near(double x);
void set_scales_host(mg_forest *F, const std::vector<double> &mult);
mg_status enqueue_scales(mg_forest *F);
// FP64 residual -> FP32 scaled rhs, zeroed correction, per-block sums (zero_u: u is zero, r = f; current: u's same-level and
// boundary ghosts are)
mg_status enqueue_residual(mg_forest *F, bool zero_u, bool current);
mg_status pack_initial_guess(mg_forest *F, const double *u_dev, bool *zero, bool keep_zero);
mg_status enqueue_problem_sums(mg_forest *F);  // per-problem sums -> pinned psum_h (no synchronisation)
mg_status enqueue_fp32_step(mg_forest *F, int cycles);  // `cycles` FP32 V-cycles and the FP64 update

mg_status ensure_fp64_coefficients(mg_forest *F);
// solver.cu, for the transposed cycles: one FP32 half-sweep on a level's own pools, and the injection y_f += R^T e_c with
// its write-through (false: not for this level's transfer)
bool smooth32_specialised(const DevLevel &d);
bool transfer_specialised(const DevLevel &d);
void smooth_level32(mg_forest *F, DevLevel &d, int colour);
bool inject32(mg_forest *F, DevLevel &d, DevLevel &c);
}  // namespace octmg

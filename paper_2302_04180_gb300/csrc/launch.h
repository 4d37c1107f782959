// Host-side interface between the C ABI (capi.cu) and the kernel translation
// units. Plain C++; no kernel code here.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include <map>
#include <mutex>
#include <utility>

#include "rbs.h"

namespace rbs {

struct DotScratch;
struct SolverState;

struct CSRArgs {
    int64_t n, nnz;
    const int64_t *rowptr;
    const int32_t *col;
    const double *val;
};

// A matrix of few diagonals as the solvers' set-up lays it out (kernels.cuh):
// per row a word whose bit j says that the row has an entry at column
// row + off[j] (off ascending, m of them; with at most 7, bits 8 and up hold the
// row's first value within its 32 rows), and per 32 rows the first nonzero.
constexpr int SPMV_DIAGS = 32;
struct DiagArgs {
    const uint32_t *mask;
    const int64_t *base;
    int32_t m, pad;
    int32_t off[SPMV_DIAGS];
};

// SpMV row schedules (Cfg::mode): one thread per row, warp-staged chunks of
// up to SPMV_CAP_SHORT or SPMV_CAP_LONG nonzeros, rows of up to 7 or 32
// diagonals.
// Bit SPMV_TEST_STALL above the schedule bits selects the staged SpMV's test
// mode of its bounded wait (kernels.cuh).
enum : int { SPMV_MODE_ROW = 1, SPMV_MODE_SHORT = 2, SPMV_MODE_LONG = 3, SPMV_MODE_DIAG7 = 4, SPMV_MODE_DIAG32 = 5,
             SPMV_MODE_MASK = 0xff, SPMV_TEST_STALL = 0x100 };
// Most percent of the L1/shared storage for the kernels that stage short rows:
// what their three blocks per SM take (48 to 50 KB each). More would only shrink
// the L1 that the x gathers live on: 500000 ragged random rows 35.0 us at 75 %,
// 31.1 at this (K1 36.7, 35.1); Poisson 128^3 is as fast at either.
constexpr int SPMV_SHORT_CARVEOUT = 64;
// Launch `kern`, which calls chain_wait() (common.cuh), so that it may be set up and
// clear its shared memory while the kernel before it in the stream, whosever it
// is, ends. Without it the GPU idles 2 us between two kernels, as long as a dot of
// a million elements takes from HBM: SpMV of Poisson 128^3 42.2 -> 39.8 us, of 500000
// ragged rows 29.6 -> 27.5, dots of 2^24 55.4 -> 52.9, five of 2^21 32.9 -> 30.5,
// and 0.5 to 1 us less per iteration of a solver (40^3 rows, 20 iterations: 768 ->
// 748 us; 64^3 1014 -> 996). The blocks start once the earlier kernel's have all left.
// Letting them in before (griddepcontrol.launch_dependents) costs more than it
// hides: at the start of a solver's kernels 40^3 865 us and 160^3 6 % more, before
// their flush between the two.
template <class... P, class... A>
cudaError_t launch_chained(void (*kern)(P...), dim3 grid, int block, cudaStream_t s, A &&...args) {
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute at;
    at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at.val.programmaticStreamSerializationAllowed = 1;
    cfg.gridDim = grid;
    cfg.blockDim = dim3((unsigned)block);
    cfg.stream = s;
    cfg.attrs = &at;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kern, std::forward<A>(args)...);
}
// Long rows run register-staged in blocks of SPMV_REG_WARPS warps: the
// standalone SpMV, and the classic loop's fused K1/K3.
constexpr int SPMV_REG_WARPS = 4;

struct Cfg {
    int grid = 0;
    int block = 256;
    int mode = 2;       // SpMV row schedule (SPMV_MODE_*)
    int carveout = -1;  // shared-memory carveout percent, -1 = driver default
};

// A launch-shape query's answer per device and key, asked once (the runtime's
// occupancy queries take a microsecond or two each, which every short call would
// pay). query() runs under the lock.
template <class Key>
class QueryCache {
    std::mutex mu;
    std::map<std::pair<int, Key>, int> known;

public:
    template <class F>
    int get(const Key &key, F &&query) {
        int dev = 0;
        if (cudaGetDevice(&dev) != cudaSuccess) {
            cudaGetLastError();
            dev = -1;
        }
        std::lock_guard<std::mutex> lk(mu);
        const auto at = known.find({dev, key});
        if (at != known.end()) return at->second;
        return known[{dev, key}] = query();
    }
};

// Set the calling thread's rbs_last_error() message and return `code`.
int set_error(int code, const char *msg);
// Free the workspace of stream `s` on the current device (before the stream is destroyed).
void release_stream_workspace(cudaStream_t s);

// ---- standalone kernels (kernels_dot.cu: exact dots, limbs, FPE-8;
// kernels_spmv.cu: SpMV, Jacobi, CSR check) ----
// k dots in one launch: cfg.grid blocks each.
cudaError_t launch_exdot(int k, const double *const *xs, const double *const *ys, int64_t n,
                         DotScratch *g, double *out, int window, Cfg cfg, cudaStream_t s);
cudaError_t launch_exdot_partial(const double *x, const double *y, int64_t n, DotScratch *g,
                                 int64_t *limbs, int32_t *flags, Cfg cfg, cudaStream_t s);
cudaError_t launch_fpe_dot(const double *x, const double *y, int64_t n, DotScratch *g, double *out,
                           unsigned *lost, Cfg cfg, cudaStream_t s);
// Resident blocks per SM of the exact-dot kernel (window size knob) at this block
// size: the persistent grid is a whole number of waves of it.
int exdot_blocks_per_sm(int window, int block);
int fpe_blocks_per_sm(int block);
cudaError_t launch_round_limbs(const int64_t *limbs, const int32_t *flags, double *out, cudaStream_t s);
// y = A x. Without a solver state every index is checked (ERR_INDEX on a bad
// one); with one, the solver has validated the structure and the kernel skips
// the checks (and does nothing once the solver has stopped).
cudaError_t launch_spmv(const CSRArgs &A, const double *x, double *y, const SolverState *st,
                        unsigned *err, Cfg cfg, cudaStream_t s);
// The same product of a solver on a matrix laid out by its diagonals.
cudaError_t launch_spmv_diag(const CSRArgs &A, const DiagArgs &D, const double *x, double *y, const SolverState *st,
                             unsigned *err, Cfg cfg, cudaStream_t s);
cudaError_t launch_jacobi_invd(const CSRArgs &A, const double *diag, double *invd, unsigned *err,
                               Cfg cfg, cudaStream_t s);
cudaError_t launch_jacobi_apply(int64_t n, const double *invd, const double *p, double *phat, Cfg cfg,
                                cudaStream_t s);
cudaError_t launch_csr_check(const CSRArgs &A, unsigned *err, Cfg cfg, cudaStream_t s);
// The structure check, the Jacobi inverse and the diagonal layout in one pass
// over the rows. *diags (device): the diagonals of a sample of rows, m = 0 if
// they are too many; mask and base are written for them, and a row that does
// not fit them sets ERR_DIAGS in err (it is no error of the matrix).
constexpr unsigned ERR_DIAGS = 16u;
// A row of more than LONG_ROW nonzeros sets ERR_LONG, is not looked into and has no
// layout: launch_csr_check and launch_jacobi_invd then do the whole set-up, the
// check with the nonzeros spread over the grid. (One thread took 13.8 ms for one
// dense row of 200000, they take 0.09.)
constexpr unsigned ERR_LONG = 32u;
constexpr int LONG_ROW = 256;
cudaError_t launch_prepare(const CSRArgs &A, const double *diag, double *invd, DiagArgs *diags, uint32_t *mask,
                           int64_t *base, unsigned *err, Cfg cfg, cudaStream_t s);

// ---- solver kernels (kernels_solver.cu) ----
struct SolverVecs {
    double *x, *r, *r0, *p, *ph, *s, *q, *qh, *y, *invd;  // classic (x, r, r0, q, qh, y, invd shared)
    double *rh, *w, *wh, *t, *sh, *z, *zh, *v;            // pipelined
};

struct SolverArgs {
    CSRArgs A;
    DiagArgs D;  // with the SPMV_MODE_DIAG* schedules
    SolverVecs v;
    const double *b, *x0;
    SolverState *st;
    DotScratch *g;
    double *hist;
    unsigned *err;
    int dot_mode;
    int carveout;  // shared-memory carveout percent for staging kernels, -1 = driver default
    Cfg vec, spmv;
    Cfg p3;  // the pipelined P3 kernel, sized from its own occupancy
    Cfg k3;  // the classic K3 kernel (SpMV + two dots), sized from its own occupancy
};

// Kernel kinds for profiling (rbs_prof.kinds).
enum ProfKind { PK_K1 = 0, PK_VEC = 1, PK_SETUP = 2, PK_SPMV = 3, PK_VEC_DOT = 4, PK_K3 = 5, PK_K4 = 6 };

struct KernelTimer {
    virtual void before(int kind) = 0;
    virtual void after(int kind) = 0;
    virtual void gap() {}  // other work was enqueued since the last after()
    virtual ~KernelTimer() {}
};

cudaError_t solver_setup(const SolverArgs &a, int variant, cudaStream_t s, KernelTimer *t);
cudaError_t solver_iteration(const SolverArgs &a, int variant, cudaStream_t s, KernelTimer *t);

// Last node of the graph loop body: keeps the WHILE loop going while the stop
// flag is clear, and at most maxit + 1 bodies in any case (maxit up to 2^31 - 1).
cudaError_t launch_set_cond(cudaGraphConditionalHandle h, SolverState *st, cudaStream_t s);

// ---- batched solver (kernels_batch.cu) ----
struct BatchSys {
    CSRArgs A;
    const double *b, *x0, *diag;
    double *x;       // solution (device)
    double *work;    // 17 vector slots of `stride` doubles (9 for classic)
    int64_t stride;  // elements per slot
    double tol;
    int32_t maxit, variant;
    double *hist;    // device history records (hist_cap of them), may be null
    int32_t hist_cap, pad;
};
struct BatchOut {
    int32_t iters, converged, status;
    unsigned err;  // bit 0 invalid CSR, bit 1 zero/NaN/missing diagonal
    double tau0, tau_final, rho0, tau_max, alpha0, mu0;
};
cudaError_t launch_batch_prepare(const BatchSys *d_sys, int nsys, BatchOut *d_out, cudaStream_t s);
// Schedule of one batched launch: `clusters` clusters of `cluster` CTAs; a
// queued system with at least `split` unknowns is solved by a whole cluster,
// smaller ones by one CTA each.
struct BatchSchedule {
    int cluster, clusters;
    int64_t split;
};
cudaError_t launch_batch(const BatchSys *d_sys, const int32_t *d_order, const int64_t *d_sizes, int nsys,
                         unsigned *d_queue, BatchOut *d_out, BatchSchedule sched, cudaStream_t s);
// Clusters of `csize` CTAs that fit on the device at once (0 if none).
int batch_max_clusters(int csize);

// ---- one small system in one cluster (kernels_small.cu) ----
constexpr int SMALL_CTAS = 16;
// Whether this device can run such a solve and the system fits, its nonzeros
// spread evenly over the rows. A solve whose rows do not fit after all sets
// bit 8 in d_out->err and leaves x alone.
bool small_fits(int64_t n, int64_t nnz, int variant);
constexpr unsigned SMALL_NO_ROOM = 8u;
// Structure check, Jacobi (diag or the first stored (i, i)), set-up and loop;
// *d_out zero before.
cudaError_t launch_small(const CSRArgs &A, const double *b, const double *x0, const double *diag, double *x, double tol,
                         int32_t maxit, int variant, double *hist, int32_t hist_cap, BatchOut *d_out, cudaStream_t s);

// ---- per-step kernels of the serving engine (kernels_step.cu) ----
// One block of a per-step launch: rows [lo, hi) of the system in slot `sys`
// (lo even), which has nblk blocks in the launch.
struct StepTask {
    int32_t sys, nblk;
    int64_t lo, hi;
};
// Size of the device-side view of one system, and that view written to `out`
// (host memory, step_ctx_bytes() bytes): matrix, vectors (v.x is the caller's
// solution buffer, 16-byte aligned), right-hand side, optional x0 and Jacobi
// diagonal, the system's own state and dot scratch (zero at rest), and its
// device history records (nullable; state->hist_cap of them).
size_t step_ctx_bytes();
// mask, base (nullable): room for the system's layout by diagonals, one word per
// row rounded up to 32 and one int64 per 32 rows.
void step_ctx_make(void *out, const CSRArgs &A, const SolverVecs &v, const double *b, const double *x0,
                   const double *diag, SolverState *st, DotScratch *g, double *hist, uint32_t *mask = nullptr,
                   int64_t *base = nullptr);
// Whether such room is worth giving: the steps know layouts of up to 7 diagonals.
bool step_wants_layout(const CSRArgs &A);
// Where in the device-side view the number of the system's diagonals stands after
// its admission (int32; 0: not laid out).
size_t step_ctx_diags_offset();
// Admission of new systems (all of one variant): structure check and Jacobi,
// then the set-up of Fig. 2 or Fig. 4; a system that fails its checks ends with
// status RBS_EINVAL and its error bits in its scratch's err word. layouts: whether
// any of them has room for a layout by diagonals.
cudaError_t step_admit(void *ctxs, const StepTask *tasks, int ntasks, int variant, bool layouts, cudaStream_t s);
// One iteration of every listed system, all of one variant: first the `laid` tasks
// of systems laid out by their diagonals, whose products have launches of their
// own, then `rest` tasks of others. Stopped systems skip it.
cudaError_t step_iteration(const void *ctxs, const StepTask *tasks, int laid, int rest, int variant, cudaStream_t s);

// occupancy-derived persistent grid for the kernels of one kind: which = 0 the
// SpMV kernels (classic K1, pipelined S10/S18), 1 the vector kernels, 2 the
// pipelined P3 kernel, 3 the classic K3 kernel
int solver_blocks_per_sm(int variant, int dot_mode, int which, int block, int carveout, int spmv_mode);
// Resident blocks per SM of the standalone SpMV kernel at this block size and
// shared-memory carveout (applies the carveout first).
int spmv_blocks_per_sm(int block, int carveout, int mode);

}  // namespace rbs

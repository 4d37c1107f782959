// Per-step kernels of the serving engine: one launch runs one phase of one
// iteration (Fig. 2 classic K1..K5, Fig. 4 pipelined P1..P4) for every system
// that is in flight at once. A launch is a list of tasks, one per block: a
// system (its Ctx in device memory) and a segment of its rows. Each block runs
// the same per-element functions as the per-solve kernels (solver_elem.cuh)
// over its segment; the exact dots of a system are reduced over that system's
// blocks only (its own scratch and ticket, nblk arrivals), and the system's
// last block runs the scalar tail on the system's own device state. Every
// system therefore gets the bits a solve of it alone gives, whatever else
// shares the launch, and a system that has stopped skips every later phase.
#include <cstddef>
#include <cstring>
#include <mutex>
#include <type_traits>

#include "kernels.cuh"
#include "launch.h"
#include "solver_elem.cuh"
#include "tails.cuh"

namespace rbs {

namespace {

// The rows of a segment [lo, hi) as element pairs (2j, 2j+1) with 16-byte
// accesses (lo is even), then an odd last element in thread 0.
template <class F>
__device__ __forceinline__ void seg_pairs(int64_t lo, int64_t hi, F &&f) {
    for (int64_t i = lo + 2 * (int64_t)threadIdx.x; i + 1 < hi; i += 2 * (int64_t)blockDim.x) f(i, true);
    if (((hi - lo) & 1) && threadIdx.x == 0) f(hi - 1, false);
}

// The odd last element of a segment (lo is even) in the thread that takes it.
__device__ __forceinline__ int64_t seg_odd(const StepTask &t) {
    return (t.hi & 1) && threadIdx.x == 0 ? t.hi - 1 : -1;
}

// y = A x over the block's segment with the warp-staged SpMV (structure
// validated at admission), epilogue fn(row, y_row, z_row).
template <class F>
__device__ __forceinline__ void seg_spmv(const Ctx &c, const StepTask &t, const double *x, const double *z,
                                         unsigned &err, F &&fn) {
    spmv_rows<false, SPMV_CAP_SHORT, false>(c.A, t.lo, t.hi, threadIdx.x >> 5, blockDim.x >> 5, x, z, true, false,
                                            err, fn);
}

constexpr int SCR = SpmvLayout<SPMV_CAP_SHORT>::SCRATCH;

// The same for a system laid out by its diagonals (segments start at multiples of
// 64 rows). Every thread of the block calls it.
constexpr int STEP_DIAGS = 7;
template <class F>
__device__ __forceinline__ void seg_spmv_diag(const Ctx &c, const int32_t *off, const StepTask &t, const double *x,
                                              const double *z, unsigned &err, F &&fn) {
    __shared__ int s_off[STEP_DIAGS];
    if (threadIdx.x < STEP_DIAGS) s_off[threadIdx.x] = off[threadIdx.x];
    __syncthreads();
    spmv_rows_diag<STEP_DIAGS>(
        c.A, c.D.mask, c.D.base, c.D.m, [&](int j) { return s_off[j]; }, (int)(t.lo >> 5), (int)((t.hi + 31) >> 5),
        (int)t.hi, 0, 1, x, z, false, err, fn);
}
template <bool DIAG, class F>
__device__ __forceinline__ void step_spmv(const Ctx *ctxs, const Ctx &c, const StepTask &t, const double *x,
                                          const double *z, unsigned &err, F &&fn) {
    if constexpr (DIAG) seg_spmv_diag(c, ctxs[t.sys].D.off, t, x, z, err, fn);
    else seg_spmv(c, t, x, z, err, fn);
}
// K dots beside either product: windows in shared memory where the staging leaves
// it, as in the per-solve kernels.
template <int K, bool DIAG>
using StepDot = typename std::conditional<DIAG, ExactRows<K, 12, false>, ExactR<K, SQ>>::type;
template <int K>
__device__ __forceinline__ bool finish_step(ExactR<K, SQ> &red, DotScratch *g, double *vals, unsigned nblk, bool coop) {
    return red.template finish<SCR>(g, vals, nblk, coop);
}
template <int K, int W>
__device__ __forceinline__ bool finish_step(ExactRows<K, W, false> &red, DotScratch *g, double *vals, unsigned nblk, bool) {
    return red.finish(g, vals, nblk);
}

// ---- admission ------------------------------------------------------------------

// The diagonals of every system that has room for a layout by them (its first
// task's block).
__global__ void __launch_bounds__(256) k_step_sample(Ctx *ctxs, const StepTask *tasks) {
    const StepTask t = tasks[blockIdx.x];
    Ctx &c = ctxs[t.sys];
    if (t.lo != 0 || !c.D.mask) return;
    const int m = sample_diags(c.A, STEP_DIAGS, c.D.off);
    if (threadIdx.x == 0) c.D.m = m;
}

// Structure check, Jacobi set-up and layout by diagonals of the segment's rows
// (check_row; the checks of the per-solve path). Segments start at multiples of
// 64 rows.
__global__ void __launch_bounds__(256) k_step_prepare(const Ctx *ctxs, const StepTask *tasks) {
    __shared__ int s_off[STEP_DIAGS + 1];
    const StepTask t = tasks[blockIdx.x];
    const Ctx &c = ctxs[t.sys];
    const CSRView A = c.A;
    const int m = c.D.mask ? c.D.m : 0;
    if (threadIdx.x <= STEP_DIAGS) s_off[threadIdx.x] = (int)threadIdx.x < m ? c.D.off[threadIdx.x] : 0x7fffffff;
    __syncthreads();
    unsigned eb = 0u;
    if (threadIdx.x == 0 && t.lo == 0 && A.rowptr[0] != 0) eb |= 1u;
    if (threadIdx.x == 0 && t.hi == A.n && A.rowptr[A.n] != A.nnz) eb |= 1u;
    uint32_t *mask = const_cast<uint32_t *>(c.D.mask);
    int64_t *base = const_cast<int64_t *>(c.D.base);
    const int64_t end = t.hi == A.n ? (A.n + 31) / 32 * 32 : t.hi;
    for (int64_t i = t.lo + threadIdx.x; i < end; i += blockDim.x) {
        uint32_t word = 0u;
        if (i < A.n) {
            const RowSetup r = check_row(A, i, c.diag, s_off, m);
            eb |= m > 0 ? r.err : r.err & ~ERR_DIAGS;
            c.invd[i] = r.inv;
            if (m > 0 && (i & 31) == 0) base[i >> 5] = r.first;
            word = r.word | (uint32_t)(r.first - A.rowptr[i & ~31LL]) << 8;
        }
        if (m > 0) mask[i] = word;
    }
    eb = __reduce_or_sync(__activemask(), eb);
    if (eb && (*(volatile unsigned *)c.err & eb) != eb) atomicOr(c.err, eb);
}

// A system that failed its checks stops before its set-up, one whose rows do not
// lie on its sampled diagonals has no layout (one thread per system: the one of
// its first task).
__global__ void k_step_validate(Ctx *ctxs, const StepTask *tasks, int ntasks) {
    const int j = blockIdx.x * blockDim.x + threadIdx.x;
    if (j >= ntasks || tasks[j].lo != 0) return;
    Ctx &c = ctxs[tasks[j].sys];
    if (!c.D.mask || (*c.err & ERR_DIAGS)) c.D.m = 0;
    *c.err &= ~ERR_DIAGS;
    if (*c.err) {
        c.st->status = RBS_EINVAL;
        c.st->done = 1;
    }
}

// ---- classic (Fig. 2) -----------------------------------------------------------

template <class R>
__global__ void __launch_bounds__(256) k_step_cls_setup(const Ctx *ctxs, const StepTask *tasks) {
    const StepTask t = tasks[blockIdx.x];
    const Ctx c = ctxs[t.sys];
    StateCopy sc;
    sc.load(c.st);
    R red;
    red.init();  // ends in a barrier
    if (sc.copy->done) return;
    bool bad = false;
    for (int64_t i = t.lo + threadIdx.x; i < t.hi; i += blockDim.x) red.add_sq(0, cls_setup_elem(c, i, bad));
    if (bad) atomicOr(c.err, 1u);
    __shared__ double vals[R::K];
    if (red.finish(c.g, vals, t.nblk)) sc.tail([&](SolverState *st) { tail_cls_setup(st, vals); });
}

template <bool DIAG>
__device__ __forceinline__ void step_k1(const Ctx *ctxs, const StepTask *tasks) {
    StepDot<1, DIAG> red;
    red.init();
    chain_wait();
    const StepTask t = tasks[blockIdx.x];
    const Ctx c = ctxs[t.sys];
    StateCopy sc;
    sc.load(c.st);
    __syncthreads();
    if (sc.copy->done) return;
    unsigned eb = 0u;
    step_spmv<DIAG>(ctxs, c, t, c.ph, c.r0, eb, [&](int64_t i, double si, double r0) {
        c.s[i] = si;
        red.add(0, r0, si);
    });
    if (eb) atomicOr(c.err, eb);
    __shared__ double vals[1];
    if (finish_step(red, c.g, vals, t.nblk, !(eb & ERR_TIMEOUT)))
        sc.tail([&](SolverState *st) { tail_cls_alpha(st, vals); });
}
__global__ void __launch_bounds__(256, 3) k_step_cls_k1(const Ctx *ctxs, const StepTask *tasks) { step_k1<false>(ctxs, tasks); }
// (systems laid out by their diagonals)
__global__ void __launch_bounds__(256, 3) k_step_diag_k1(const Ctx *ctxs, const StepTask *tasks) { step_k1<true>(ctxs, tasks); }

__global__ void __launch_bounds__(256) k_step_cls_k2(const Ctx *ctxs, const StepTask *tasks) {
    chain_wait();
    const StepTask t = tasks[blockIdx.x];
    const Ctx c = ctxs[t.sys];
    if (c.st->done) return;
    const double na = -c.st->alpha;
    seg_pairs(t.lo, t.hi, [&](int64_t i, bool pair) {
        if (pair) {
            const double2 s = ld2(c.s, i), r = ld2(c.r, i), d = ld2(c.invd, i);
            const VPair u0 = cls_k2(na, s.x, r.x, d.x), u1 = cls_k2(na, s.y, r.y, d.y);
            st2(c.q, i, make_double2(u0.a, u1.a));
            st2(c.qh, i, make_double2(u0.b, u1.b));
        } else {
            const VPair u = cls_k2(na, c.s[i], c.r[i], c.invd[i]);
            c.q[i] = u.a;
            c.qh[i] = u.b;
        }
    });
}

template <bool DIAG>
__device__ __forceinline__ void step_k3(const Ctx *ctxs, const StepTask *tasks) {
    StepDot<2, DIAG> red;
    red.init();
    chain_wait();
    const StepTask t = tasks[blockIdx.x];
    const Ctx c = ctxs[t.sys];
    StateCopy sc;
    sc.load(c.st);
    __syncthreads();
    if (sc.copy->done) return;
    unsigned eb = 0u;
    step_spmv<DIAG>(ctxs, c, t, c.qh, c.q, eb, [&](int64_t i, double yi, double qi) {
        c.y[i] = yi;
        red.add(0, qi, yi);
        red.add_sq(1, yi);
    });
    if (eb) atomicOr(c.err, eb);
    __shared__ double vals[2];
    if (finish_step(red, c.g, vals, t.nblk, !(eb & ERR_TIMEOUT)))
        sc.tail([&](SolverState *st) { tail_cls_omega(st, vals); });
}
__global__ void __launch_bounds__(256, 3) k_step_cls_k3(const Ctx *ctxs, const StepTask *tasks) { step_k3<false>(ctxs, tasks); }
// (systems laid out by their diagonals)
__global__ void __launch_bounds__(256, 3) k_step_diag_k3(const Ctx *ctxs, const StepTask *tasks) { step_k3<true>(ctxs, tasks); }

template <class R>
__global__ void __launch_bounds__(256, 4) k_step_cls_k4(const Ctx *ctxs, const StepTask *tasks) {
    R red;
    red.init();
    chain_wait();
    const StepTask t = tasks[blockIdx.x];
    const Ctx c = ctxs[t.sys];
    StateCopy sc;
    sc.load(c.st);
    __syncthreads();
    if (sc.copy->done) return;
    cls_k4_pairs(c, red, sc.copy->alpha, sc.copy->omega, (t.lo >> 1) + threadIdx.x, t.hi >> 1, blockDim.x, seg_odd(t));
    __shared__ double vals[R::K];
    if (red.finish(c.g, vals, t.nblk)) sc.tail([&](SolverState *st) { tail_cls_beta(st, vals, c.hist); });
}

__global__ void __launch_bounds__(256) k_step_cls_k5(const Ctx *ctxs, const StepTask *tasks) {
    chain_wait();
    const StepTask t = tasks[blockIdx.x];
    const Ctx c = ctxs[t.sys];
    if (c.st->done) return;
    const double be = c.st->beta, nom = -c.st->omega;
    seg_pairs(t.lo, t.hi, [&](int64_t i, bool pair) {
        if (pair) {
            const double2 s = ld2(c.s, i), r = ld2(c.r, i), d = ld2(c.invd, i), p = ld2(c.p, i);
            const VPair u0 = cls_k5(be, nom, s.x, p.x, r.x, d.x), u1 = cls_k5(be, nom, s.y, p.y, r.y, d.y);
            st2(c.p, i, make_double2(u0.a, u1.a));
            st2(c.ph, i, make_double2(u0.b, u1.b));
        } else {
            const VPair u = cls_k5(be, nom, c.s[i], c.p[i], c.r[i], c.invd[i]);
            c.p[i] = u.a;
            c.ph[i] = u.b;
        }
    });
}

// ---- pipelined (Fig. 4) ---------------------------------------------------------

__global__ void __launch_bounds__(256) k_step_pipe_setup1(const Ctx *ctxs, const StepTask *tasks) {
    const StepTask t = tasks[blockIdx.x];
    const Ctx c = ctxs[t.sys];
    if (c.st->done) return;
    bool bad = false;
    for (int64_t i = t.lo + threadIdx.x; i < t.hi; i += blockDim.x) pipe_setup1_elem(c, i, bad);
    if (bad) atomicOr(c.err, 1u);
}

template <class R>
__global__ void __launch_bounds__(256, 3) k_step_pipe_setup2(const Ctx *ctxs, const StepTask *tasks) {
    const StepTask t = tasks[blockIdx.x];
    const Ctx c = ctxs[t.sys];
    StateCopy sc;
    sc.load(c.st);
    R red;
    red.init();  // ends in a barrier
    if (sc.copy->done) return;
    unsigned eb = 0u;
    seg_spmv(c, t, c.rh, c.r0, eb, [&](int64_t i, double wi, double r0) {
        c.w[i] = wi;
        c.wh[i] = __dmul_rn(wi, c.invd[i]);
        red.add_sq(0, r0);  // r = r0 at set-up
        red.add(1, r0, wi);
    });
    if (eb) atomicOr(c.err, eb);
    __shared__ double vals[R::K];
    if (red.template finish<SCR>(c.g, vals, t.nblk, !(eb & ERR_TIMEOUT)))
        sc.tail([&](SolverState *st) { tail_pipe_setup(st, vals); });
}

// y = A x without a dot: the pipelined S10 (v = A zhat) and S18 / set-up (t = A what)
template <bool TO_V, bool DIAG>
__global__ void __launch_bounds__(256, 3) k_step_spmv(const Ctx *ctxs, const StepTask *tasks) {
    chain_wait();
    const StepTask t = tasks[blockIdx.x];
    const Ctx c = ctxs[t.sys];
    if (c.st->done) return;
    unsigned eb = 0u;
    double *y = TO_V ? c.v : c.t;
    step_spmv<DIAG>(ctxs, c, t, TO_V ? c.zh : c.wh, nullptr, eb, [&](int64_t i, double yi, double) { y[i] = yi; });
    if (eb) atomicOr(c.err, eb);
}

template <class R>
__global__ void __launch_bounds__(256, 3) k_step_pipe_p1(const Ctx *ctxs, const StepTask *tasks) {
    R red;
    red.init();
    chain_wait();
    const StepTask t = tasks[blockIdx.x];
    const Ctx c = ctxs[t.sys];
    StateCopy sc;
    sc.load(c.st);
    __syncthreads();
    if (sc.copy->done) return;
    pipe_p1_pairs(c, red, sc.copy->iter == 0, -sc.copy->alpha, sc.copy->beta, -sc.copy->omega,
                  (t.lo >> 1) + threadIdx.x, t.hi >> 1, blockDim.x, seg_odd(t));
    __shared__ double vals[R::K];
    if (red.finish(c.g, vals, t.nblk)) sc.tail([&](SolverState *st) { tail_pipe_omega(st, vals); });
}

template <class R>
__global__ void __launch_bounds__(256, 2) k_step_pipe_p3(const Ctx *ctxs, const StepTask *tasks) {
    R red;
    red.init();
    chain_wait();
    const StepTask t = tasks[blockIdx.x];
    const Ctx c = ctxs[t.sys];
    StateCopy sc;
    sc.load(c.st);
    __syncthreads();
    if (sc.copy->done) return;
    pipe_p3_pairs(c, red, sc.copy->alpha, sc.copy->omega, (t.lo >> 1) + threadIdx.x, t.hi >> 1, blockDim.x, seg_odd(t));
    __shared__ double vals[R::K];
    if (red.finish(c.g, vals, t.nblk)) sc.tail([&](SolverState *st) { tail_pipe_beta(st, vals, c.hist); });
}

using R1 = ExactR<1, SQ>;
using R2 = ExactR<2, SQ>;

void step_carveout() {
    static std::once_flag once;
    std::call_once(once, [] {
        const int c = 75;  // as the per-solve staging kernels: three blocks per SM, L1 left for the gathers
        const auto set = [&](auto kern) {
            cudaFuncSetAttribute(kern, cudaFuncAttributePreferredSharedMemoryCarveout, c);
        };
        set(k_step_cls_k1);
        set(k_step_diag_k1);
        set(k_step_cls_k3);
        set(k_step_diag_k3);
        set(k_step_pipe_setup2<R2>);
        set(k_step_spmv<true, false>);
        set(k_step_spmv<true, true>);
        set(k_step_spmv<false, false>);
        set(k_step_spmv<false, true>);
        cudaGetLastError();
    });
}

}  // namespace

void step_ctx_make(void *out, const CSRArgs &A, const SolverVecs &v, const double *b, const double *x0,
                   const double *diag, SolverState *st, DotScratch *g, double *hist, uint32_t *mask, int64_t *base) {
    Ctx c;
    memset(&c, 0, sizeof c);
    c.A = CSRView{A.n, A.nnz, A.rowptr, A.col, A.val};
    c.n = A.n;
    c.x = v.x; c.r = v.r; c.r0 = v.r0; c.p = v.p; c.ph = v.ph; c.s = v.s; c.q = v.q; c.qh = v.qh;
    c.y = v.y; c.invd = v.invd; c.rh = v.rh; c.w = v.w; c.wh = v.wh; c.t = v.t; c.sh = v.sh;
    c.z = v.z; c.zh = v.zh; c.v = v.v;
    c.b = b;
    c.x0 = x0;
    c.diag = diag;
    c.st = st;
    c.g = g;
    c.hist = hist;
    c.err = &g->err;
    c.spmv_mode = SPMV_MODE_SHORT;
    c.D.mask = mask;
    c.D.base = base;
    memcpy(out, &c, sizeof c);
}

size_t step_ctx_bytes() { return sizeof(Ctx); }

size_t step_ctx_diags_offset() { return offsetof(Ctx, D) + offsetof(DiagArgs, m); }

bool step_wants_layout(const CSRArgs &A) {
    return A.nnz > 0 && A.nnz <= STEP_DIAGS * A.n && ((uintptr_t)A.val & 15) == 0;
}

cudaError_t step_admit(void *ctxs, const StepTask *tasks, int ntasks, int variant, bool layouts, cudaStream_t s) {
    if (ntasks <= 0) return cudaSuccess;
    step_carveout();
    Ctx *c = static_cast<Ctx *>(ctxs);
    if (layouts) k_step_sample<<<ntasks, 256, 0, s>>>(c, tasks);
    k_step_prepare<<<ntasks, 256, 0, s>>>(c, tasks);
    k_step_validate<<<(ntasks + 255) / 256, 256, 0, s>>>(c, tasks, ntasks);
    if (variant == RBS_CLASSIC) {
        k_step_cls_setup<R1><<<ntasks, 256, 0, s>>>(c, tasks);
    } else {
        k_step_pipe_setup1<<<ntasks, 256, 0, s>>>(c, tasks);
        k_step_pipe_setup2<R2><<<ntasks, 256, 0, s>>>(c, tasks);
        k_step_spmv<false, false><<<ntasks, 256, 0, s>>>(c, tasks);
    }
    return cudaGetLastError();
}

// Chained launches: 20 iterations of 12 systems 2.16 -> 1.88 ms, of 60 systems 6.05
// -> 5.72; 512 systems take as long either way.
cudaError_t step_iteration(const void *ctxs, const StepTask *tasks, int laid, int rest, int variant, cudaStream_t s) {
    if (laid + rest <= 0) return cudaSuccess;
    step_carveout();
    const Ctx *c = static_cast<const Ctx *>(ctxs);
    const auto go = [&](auto kern, const StepTask *t, int n) {
        if (n > 0) launch_chained(kern, dim3((unsigned)n), 256, s, c, t);
    };
    // (a vector step is the same for both kinds: one launch)
    const auto all = [&](auto kern) { go(kern, tasks, laid + rest); };
    const auto product = [&](auto diag, auto general) {
        go(diag, tasks, laid);
        go(general, tasks + laid, rest);
    };
    if (variant == RBS_CLASSIC) {
        product(k_step_diag_k1, k_step_cls_k1);
        all(k_step_cls_k2);
        product(k_step_diag_k3, k_step_cls_k3);
        all(k_step_cls_k4<RowsR2>);
        all(k_step_cls_k5);
    } else {
        all(k_step_pipe_p1<RowsR2>);
        product(k_step_spmv<true, true>, k_step_spmv<true, false>);
        all(k_step_pipe_p3<RowsR5>);
        product(k_step_spmv<false, true>, k_step_spmv<false, false>);
    }
    return cudaGetLastError();
}

}  // namespace rbs

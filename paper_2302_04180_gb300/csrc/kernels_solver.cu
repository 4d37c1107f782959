// Fused kernels of the classic (Fig. 2) and pipelined (Fig. 4) PBiCGStab
// loops, with device-resident scalars. Every dot rides in the epilogue of the
// kernel that produces its operands, and the block that finishes a reduction
// last computes the scalar recurrence (alpha, omega, beta, tau, stop test) in
// place, so the host never sits between two steps.
//
// Classic iteration (5 launches):
//   K1  s = A phat, <r0,s>                      -> alpha          (S2, S3)
//   K2  q = fma(-alpha, s, r), qhat = q*invd                        (S4, S5)
//   K3  y = A qhat, <q,y>, <y,y>                -> omega          (S6, S7)
//   K4  x = fma(omega, qhat, fma(alpha, phat, x)), r = fma(-omega, y, q),
//       <r0,r>, <r,r>                           -> tau, stop, beta (S8-S11, S10)
//   K5  p = fma(beta, fma(-omega, s, p), r), phat = p*invd        (S12, S1)
// Pipelined iteration (4 launches):
//   P1  S1-S7 and S9 element-wise, <q,y>, <y,y>  -> omega          (S1-S9, S11)
//   P2  v = A zhat                                                  (S10)
//   P3  S12-S15 and S17 element-wise, <r0,r>, <r0,w>, <r0,s>, <r0,z>, <r,r>
//                                                -> tau, stop, beta, alpha (S16, S19)
//   P4  t = A what                                                  (S18)
// Once the stop flag is set, every later kernel returns at once.
#include <mutex>
#include <tuple>
#include <type_traits>

#include "kernels.cuh"

#include "launch.h"
#include "solver_elem.cuh"
#include "tails.cuh"

namespace rbs {

// ---- classic kernels -------------------------------------------------------------

// set-up: r = b - A x0 (or b), x = x0 (or +0), r0 = p = r, phat = r*invd, <r0,r0>
template <class R>
__global__ void __launch_bounds__(256) k_cls_setup(Ctx c) {
    StateCopy sc;
    sc.load(c.st);
    R red;
    red.init();  // ends in a barrier
    bool bad = false;
    for (int64_t i = gtid(); i < c.n; i += gstride()) {
        const double ri = cls_setup_elem(c, i, bad);
        red.add_sq(0, ri);
    }
    if (bad) atomicOr(c.err, 1u);
    __shared__ double vals[R::K];
    if (red.finish(c.g, vals)) sc.tail([&](SolverState *st) { tail_cls_setup(st, vals); });
}

// SpMV rows of the fused K1/K3 with epilogue fn(row, y_row, z_row), by CAP:
// matrices of few diagonals (CAP = -N, spmv_rows_diag); short rows warp-staged
// (or one thread per row, mode 1) in 256-thread blocks; long rows (CAP =
// SPMV_CAP_LONG) register-staged in blocks of SPMV_REG_WARPS warps. finish_fused
// lets the flush of register windows reuse the staging buffer.
constexpr int CAP_DIAG7 = -7, CAP_DIAG32 = -32;
template <int CAP>
struct FusedScratch {
    static constexpr bool REG = CAP > SPMV_CAP_SHORT;
    static constexpr int BYTES = REG ? SpmvLayout<CAP>::BUF : SpmvLayout<CAP>::SCRATCH;
    static constexpr int WARPS = REG ? SPMV_REG_WARPS : MAX_WARPS;
    static constexpr int THREADS = WARPS * 32;
};
template <int N>
struct FusedDiag {
    static constexpr int BYTES = DiagLayout<N>::SCRATCH;
    static constexpr int WARPS = DiagLayout<N>::WARPS;
    static constexpr int THREADS = WARPS * 32;
};
template <> struct FusedScratch<CAP_DIAG7> : FusedDiag<7> {};
template <> struct FusedScratch<CAP_DIAG32> : FusedDiag<32> {};
// The reducer R as K1, K3 and the pipelined set-up carry it: the kernels of few
// diagonals, whose smaller staging leaves the shared memory, keep the exact
// windows there (256^3, first hundred iterations: K3 320 -> 275 us, K1 249 -> 244,
// 252 and 234 since; 283 with 10 words and 314 with 8, since products below the window go to
// atomics while the vectors fall off steeply; one branch for both of K3's products
// 291).
template <class R, int CAP>
struct FusedDot {
    using type = R;
};
template <int K>
struct FusedDot<ExactR<K, SQ>, CAP_DIAG7> {
    using type = ExactRows<K, 12, false>;
};
// finish() of either; coop = false after a timed-out staged copy
template <int CAP, class R>
__device__ __forceinline__ bool finish_fused(R &red, DotScratch *g, double *vals, bool coop) {
    return red.template finish<FusedScratch<CAP>::BYTES, FusedScratch<CAP>::WARPS>(g, vals, 0u, coop);
}
template <int CAP, int K, int W>
__device__ __forceinline__ bool finish_fused(ExactRows<K, W, false> &red, DotScratch *g, double *vals, bool) {
    return red.finish(g, vals);
}

template <int CAP, class F>
__device__ __forceinline__ void fused_spmv(const Ctx &c, const double *x, const double *z, unsigned &eb, F &&fn) {
    if constexpr (CAP < 0)
        spmv_grid_diag<-CAP>(c.A, c.D, x, z, (c.spmv_mode & SPMV_TEST_STALL) != 0, eb, fn);
    else if constexpr (FusedScratch<CAP>::REG)
        spmv_rows_reg<false, CAP, false>(c.A, 0, c.A.n, (int64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5),
                                         (int64_t)gridDim.x * (blockDim.x >> 5), x, z, true,
                                         (c.spmv_mode & SPMV_TEST_STALL) != 0, eb, fn);
    else
        spmv_each<false, CAP>(c.A, x, z, c.spmv_mode, eb, fn);
}

// K1: s = A phat, <r0, s>
template <class R, int CAP>
__global__ void __launch_bounds__(FusedScratch<CAP>::THREADS, 3) k_cls_k1(Ctx c) {
    typename FusedDot<R, CAP>::type red;
    red.init();
    chain_wait();
    StateCopy sc;
    sc.load(c.st);
    __syncthreads();
    if (sc.copy->done) return;
    unsigned eb = 0u;
    fused_spmv<CAP>(c, c.ph, c.r0, eb, [&](int64_t i, double si, double r0) {
        c.s[i] = si;
        red.add(0, r0, si);
    });
    if (eb) atomicOr(c.err, eb);
    __shared__ double vals[R::K];
    if (finish_fused<CAP>(red, c.g, vals, !(eb & ERR_TIMEOUT)))
        sc.tail([&](SolverState *st) { tail_cls_alpha(st, vals); });
}

// K2: q = fma(-alpha, s, r), qhat = q * invd. Four blocks per SM, like K4, whose
// occupancy sizes the vector grid: left free, the compiler took 80 registers, three
// blocks fit and the grid ran in 1.33 waves.
__global__ void __launch_bounds__(256, 4) k_cls_k2(Ctx c) {
    chain_wait();
    if (c.st->done) return;
    const double na = -c.st->alpha;
    for_pairs(c.n, [&](int64_t i, bool pair) {
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

// K3: y = A qhat, <q, y>, <y, y>
template <class R, int CAP>
__global__ void __launch_bounds__(FusedScratch<CAP>::THREADS, 3) k_cls_k3(Ctx c) {
    typename FusedDot<R, CAP>::type red;
    red.init();
    chain_wait();
    StateCopy sc;
    sc.load(c.st);
    __syncthreads();
    if (sc.copy->done) return;
    unsigned eb = 0u;
    fused_spmv<CAP>(c, c.qh, c.q, eb, [&](int64_t i, double yi, double qi) {
        c.y[i] = yi;
        red.add(0, qi, yi);
        red.add_sq(1, yi);
    });
    if (eb) atomicOr(c.err, eb);
    __shared__ double vals[R::K];
    if (finish_fused<CAP>(red, c.g, vals, !(eb & ERR_TIMEOUT)))
        sc.tail([&](SolverState *st) { tail_cls_omega(st, vals); });
}

// K4: x = fma(omega, qhat, fma(alpha, phat, x)), r = fma(-omega, y, q), <r0,r>, <r,r>
template <class R>
__global__ void __launch_bounds__(256, 4) k_cls_k4(Ctx c) {
    R red;
    red.init();
    chain_wait();
    StateCopy sc;
    sc.load(c.st);
    __syncthreads();
    if (sc.copy->done) return;
    cls_k4_pairs(c, red, sc.copy->alpha, sc.copy->omega, gtid(), c.n >> 1, gstride(),
                 (c.n & 1) && gtid() == 0 ? c.n - 1 : -1);
    __shared__ double vals[R::K];
    if (red.finish(c.g, vals)) sc.tail([&](SolverState *st) { tail_cls_beta(st, vals, c.hist); });
}

// K5: p = fma(beta, fma(-omega, s, p), r), phat = p * invd
__global__ void __launch_bounds__(256) k_cls_k5(Ctx c) {
    chain_wait();
    if (c.st->done) return;
    const double be = c.st->beta, nom = -c.st->omega;
    for_pairs(c.n, [&](int64_t i, bool pair) {
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

// ---- pipelined kernels -------------------------------------------------------------

// set-up 1: r = b - A x0 (or b), x, r0 = r, rhat = r * invd
__global__ void __launch_bounds__(256) k_pipe_setup1(Ctx c) {
    bool bad = false;
    for (int64_t i = gtid(); i < c.n; i += gstride()) pipe_setup1_elem(c, i, bad);
    if (bad) atomicOr(c.err, 1u);
}

// set-up 2: w = A rhat, what = w * invd, <r0,r>, <r0,w> -> alpha0
template <class R, int CAP>
__global__ void __launch_bounds__(FusedScratch<CAP>::THREADS, 3) k_pipe_setup2(Ctx c) {
    StateCopy sc;
    sc.load(c.st);
    typename FusedDot<R, CAP>::type red;
    red.init();  // ends in a barrier
    unsigned eb = 0u;
    fused_spmv<CAP>(c, c.rh, c.r0, eb, [&](int64_t i, double wi, double r0) {
        c.w[i] = wi;
        c.wh[i] = __dmul_rn(wi, c.invd[i]);
        red.add_sq(0, r0);  // r = r0 at set-up
        red.add(1, r0, wi);
    });
    if (eb) atomicOr(c.err, eb);
    __shared__ double vals[R::K];
    if (finish_fused<CAP>(red, c.g, vals, !(eb & ERR_TIMEOUT)))
        sc.tail([&](SolverState *st) { tail_pipe_setup(st, vals); });
}

// Launch shape of P1 and P3 per reducer (blocks per SM that registers are kept
// for; two elements per thread with 16-byte accesses or one), the fastest measured
// on Poisson 256^3. With the exact reducer P1 runs two of its three blocks
// (P1_GRID): a third one's loads in flight overrun the L1 beside the windows
// (192^3: 196 us against 184).
constexpr int P1_GRID = 2;
template <class R> struct P1Cfg { static constexpr int blocks = 3, pairs = 1; };
template <int K> struct P1Cfg<PlainR<K>> { static constexpr int blocks = 4, pairs = 0; };

// P1: S1-S4 (copies at iteration 0), S5-S7, S9; <q,y>, <y,y> -> omega.
// Every operand of an element is loaded before its first store (the vectors are
// not restrict-qualified, so later loads could not be issued early).
template <class R>
__global__ void __launch_bounds__(256, P1Cfg<R>::blocks) k_pipe_p1(Ctx c) {
    R red;
    red.init();
    chain_wait();
    StateCopy sc;
    sc.load(c.st);
    __syncthreads();
    if (sc.copy->done) return;
    const double al = sc.copy->alpha, nal = -al, be = sc.copy->beta, nom = -sc.copy->omega;
    const bool first = sc.copy->iter == 0;
    if (P1Cfg<R>::pairs) {
        pipe_p1_pairs(c, red, first, nal, be, nom, gtid(), c.n >> 1, gstride(),
                      (c.n & 1) && gtid() == 0 ? c.n - 1 : -1);
    } else {
        for (int64_t i = gtid(); i < c.n; i += gstride())
            p1_store(c, i, p1_elem(p1_load(c, i, first), first, nal, be, nom, red));
    }
    __shared__ double vals[R::K];
    if (red.finish(c.g, vals)) sc.tail([&](SolverState *st) { tail_pipe_omega(st, vals); });
}

// (P3's launch shape: see P1Cfg.)
template <class R> struct P3Cfg { static constexpr int blocks = 2, pairs = 1; };
template <int K> struct P3Cfg<PlainR<K>> { static constexpr int blocks = 3, pairs = 0; };

// P3: S12-S15, S17; <r0,r>, <r0,w>, <r0,s>, <r0,z>, <r,r> -> tau, beta, alpha.
// Every operand of an element is loaded before its first store (the vectors are
// not restrict-qualified, so later loads could not be issued early).
template <class R>
__global__ void __launch_bounds__(256, P3Cfg<R>::blocks) k_pipe_p3(Ctx c) {
    R red;
    red.init();
    chain_wait();
    StateCopy sc;
    sc.load(c.st);
    __syncthreads();
    if (sc.copy->done) return;
    const double al = sc.copy->alpha, nal = -al, om = sc.copy->omega, nom = -om;
    if (P3Cfg<R>::pairs) {
        pipe_p3_pairs(c, red, al, om, gtid(), c.n >> 1, gstride(), (c.n & 1) && gtid() == 0 ? c.n - 1 : -1);
    } else {
        for (int64_t i = gtid(); i < c.n; i += gstride()) {
            const P3Out o = p3_elem(P3In{c.qh[i], c.y[i], c.q[i], c.ph[i], c.x[i], c.zh[i], c.wh[i], c.v[i], c.t[i],
                                         c.invd[i], c.r0[i], c.s[i], c.z[i]},
                                    al, nal, om, nom, red);
            c.x[i] = o.x;
            c.r[i] = o.r;
            c.rh[i] = o.rh;
            c.w[i] = o.w;
            c.wh[i] = o.wh;
        }
    }
    __shared__ double vals[R::K];
    if (red.finish(c.g, vals)) sc.tail([&](SolverState *st) { tail_pipe_beta(st, vals, c.hist); });
}

// ---- launch -----------------------------------------------------------------------

static Ctx make_ctx(const SolverArgs &a) {
    Ctx c;
    c.A = CSRView{a.A.n, a.A.nnz, a.A.rowptr, a.A.col, a.A.val};
    c.D = a.D;
    c.n = a.A.n;
    c.x = a.v.x; c.r = a.v.r; c.r0 = a.v.r0; c.p = a.v.p; c.ph = a.v.ph; c.s = a.v.s;
    c.q = a.v.q; c.qh = a.v.qh; c.y = a.v.y; c.invd = a.v.invd;
    c.rh = a.v.rh; c.w = a.v.w; c.wh = a.v.wh; c.t = a.v.t; c.sh = a.v.sh; c.z = a.v.z;
    c.zh = a.v.zh; c.v = a.v.v;
    c.b = a.b; c.x0 = a.x0; c.diag = nullptr; c.st = a.st; c.g = a.g; c.hist = a.hist; c.err = a.err;
    c.spmv_mode = a.spmv.mode;
    return c;
}

#define TIMED(kind, launch)             \
    do {                                \
        if (tm) tm->before(kind);       \
        launch;                         \
        if (tm) tm->after(kind);        \
    } while (0)

// The compile-time schedule of a row schedule (mode), passed to f.
template <class F>
static void with_cap(int mode, F &&f) {
    switch (mode & SPMV_MODE_MASK) {
        case SPMV_MODE_DIAG7: f(std::integral_constant<int, CAP_DIAG7>()); break;
        case SPMV_MODE_DIAG32: f(std::integral_constant<int, CAP_DIAG32>()); break;
        case SPMV_MODE_LONG: f(std::integral_constant<int, SPMV_CAP_LONG>()); break;
        default: f(std::integral_constant<int, SPMV_CAP_SHORT>()); break;
    }
}

static bool diag_mode(int mode) {
    return (mode & SPMV_MODE_MASK) == SPMV_MODE_DIAG7 || (mode & SPMV_MODE_MASK) == SPMV_MODE_DIAG32;
}

// y = A x without a dot (pipelined S10, S18 and set-up).
static cudaError_t plain_spmv(const SolverArgs &a, const double *x, double *y, cudaStream_t s) {
    if (diag_mode(a.spmv.mode)) return launch_spmv_diag(a.A, a.D, x, y, a.st, a.err, a.spmv, s);
    return launch_spmv(a.A, x, y, a.st, a.err, a.spmv, s);
}

template <class R1, class R2, class V2, class V5>
static cudaError_t setup_t(const SolverArgs &a, int variant, cudaStream_t s, KernelTimer *tm) {
    Ctx c = make_ctx(a);
    if (variant == RBS_CLASSIC) {
        TIMED(PK_SETUP, (k_cls_setup<R1><<<a.vec.grid, a.vec.block, 0, s>>>(c)));
    } else {
        TIMED(PK_SETUP, (k_pipe_setup1<<<a.vec.grid, a.vec.block, 0, s>>>(c)));
        with_cap(a.spmv.mode, [&](auto cap) {
            TIMED(PK_SETUP, (k_pipe_setup2<R2, decltype(cap)::value><<<a.spmv.grid, a.spmv.block, 0, s>>>(c)));
        });
        TIMED(PK_SETUP, (plain_spmv(a, a.v.wh, a.v.t, s)));
    }
    return cudaGetLastError();
}

template <class R1, class R2, class V2, class V5>
static cudaError_t iter_t(const SolverArgs &a, int variant, cudaStream_t s, KernelTimer *tm) {
    Ctx c = make_ctx(a);
    const auto go = [&](auto kern, Cfg g) { launch_chained(kern, dim3((unsigned)g.grid), g.block, s, c); };
    if (variant == RBS_CLASSIC) {
        with_cap(a.spmv.mode, [&](auto cap) {
            TIMED(PK_K1, (go(k_cls_k1<R1, decltype(cap)::value>, a.spmv)));
        });
        TIMED(PK_VEC, (go(k_cls_k2, a.vec)));
        with_cap(a.spmv.mode, [&](auto cap) {
            TIMED(PK_K3, (go(k_cls_k3<R2, decltype(cap)::value>, a.k3)));
        });
        TIMED(PK_K4, (go(k_cls_k4<V2>, a.vec)));
        TIMED(PK_VEC, (go(k_cls_k5, a.vec)));
    } else {
        TIMED(PK_VEC_DOT, (go(k_pipe_p1<V2>, a.vec)));
        TIMED(PK_SPMV, (plain_spmv(a, a.v.zh, a.v.v, s)));
        TIMED(PK_VEC_DOT, (go(k_pipe_p3<V5>, a.p3)));
        TIMED(PK_SPMV, (plain_spmv(a, a.v.wh, a.v.t, s)));
    }
    return cudaGetLastError();
}

// Shared-memory carveout (percent of the unified L1/shared storage, -1 = the
// driver's choice) of the kernels that stage data per warp. The x gathers of
// the SpMV live on L1 hits, so the split is a tuning knob, not a maximum: the
// kernels of short rows take no more than SPMV_SHORT_CARVEOUT of it, those of long
// rows the driver's choice, which is what their resident blocks need (rows of 2 to
// 39 random columns, 500000 rows: K1 86 us with all of it, 67 so; K3 93, 75.5; the
// product alone 83, 69. The 27-point stencil is as fast with either).
template <class R1, class R2, class V2, class V5>
static void prefer_shared(int c) {
    for (int mode : {SPMV_MODE_SHORT, SPMV_MODE_LONG, SPMV_MODE_DIAG7, SPMV_MODE_DIAG32})
        with_cap(mode, [&](auto cap) {
            constexpr int CAP = decltype(cap)::value;
            const int share = CAP == CAP_DIAG7 ? c
                              : CAP != SPMV_CAP_SHORT ? -1
                              : c > SPMV_SHORT_CARVEOUT ? SPMV_SHORT_CARVEOUT : c;
            cudaFuncSetAttribute(k_cls_k1<R1, CAP>, cudaFuncAttributePreferredSharedMemoryCarveout, share);
            cudaFuncSetAttribute(k_cls_k3<R2, CAP>, cudaFuncAttributePreferredSharedMemoryCarveout, share);
            cudaFuncSetAttribute(k_pipe_setup2<R2, CAP>, cudaFuncAttributePreferredSharedMemoryCarveout, share);
        });
    // (the vector kernels take the driver's: no more than their windows, since
    // their loads in flight need the L1)
    cudaGetLastError();
}

// Apply the carveout to this device's kernels once per value. It must come
// before any occupancy query, which depends on it.
static void apply_carveout(int dot_mode, int c) {
    static std::mutex mu;
    static int applied_exact[64], applied_plain[64];
    static bool init = false;
    std::lock_guard<std::mutex> lk(mu);
    if (!init) {
        for (int i = 0; i < 64; i++) applied_exact[i] = applied_plain[i] = -2;
        init = true;
    }
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return;
    if (dot_mode == RBS_DOT_PLAIN && applied_plain[dev] != c) {
        prefer_shared<PlainR<1>, PlainR<2>, PlainR<2>, PlainR<5>>(c);
        applied_plain[dev] = c;
    } else if (dot_mode != RBS_DOT_PLAIN && applied_exact[dev] != c) {
        prefer_shared<ExactR<1, SQ>, ExactR<2, SQ>, RowsR2, RowsR5>(c);
        applied_exact[dev] = c;
    }
}

cudaError_t solver_setup(const SolverArgs &a, int variant, cudaStream_t s, KernelTimer *t) {
    apply_carveout(a.dot_mode, a.carveout);
    if (a.dot_mode == RBS_DOT_PLAIN) return setup_t<PlainR<1>, PlainR<2>, PlainR<2>, PlainR<5>>(a, variant, s, t);
    return setup_t<ExactR<1, SQ>, ExactR<2, SQ>, RowsR2, RowsR5>(a, variant, s, t);
}

cudaError_t solver_iteration(const SolverArgs &a, int variant, cudaStream_t s, KernelTimer *t) {
    if (a.dot_mode == RBS_DOT_PLAIN) return iter_t<PlainR<1>, PlainR<2>, PlainR<2>, PlainR<5>>(a, variant, s, t);
    return iter_t<ExactR<1, SQ>, ExactR<2, SQ>, RowsR2, RowsR5>(a, variant, s, t);
}

// (a body holds one iteration or more, so maxit bodies are enough)
__global__ void k_set_cond(cudaGraphConditionalHandle h, SolverState *st) {
    const int loops = st->loops + 1;
    st->loops = loops;
    cudaGraphSetConditional(h, (!st->done && loops <= st->maxit) ? 1u : 0u);
}

cudaError_t launch_set_cond(cudaGraphConditionalHandle h, SolverState *st, cudaStream_t s) {
    k_set_cond<<<1, 1, 0, s>>>(h, st);
    return cudaGetLastError();
}

template <class R1, class R2, class V2, class V5>
static int blocks_per_sm_t(int variant, int which, int block, int spmv_mode) {
    int nb = 0;
    cudaError_t e = cudaSuccess;
    if (which == 0 || which == 3) {
        with_cap(spmv_mode, [&](auto cap) {
            constexpr int CAP = decltype(cap)::value;
            e = which == 0 ? cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, k_cls_k1<R1, CAP>, block, 0)
                           : cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, k_cls_k3<R2, CAP>, block, 0);
        });
    } else if (variant == RBS_PIPELINED) {
        e = which == 2 ? cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, k_pipe_p3<V5>, block, 0)
                       : cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, k_pipe_p1<V2>, block, 0);
        if (which != 2 && V2::WINDOWS && block == 256 && nb > P1_GRID) nb = P1_GRID;
    } else {
        e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, k_cls_k4<V2>, block, 0);
    }
    if (e != cudaSuccess || nb < 1) nb = 1;
    return nb;
}

int solver_blocks_per_sm(int variant, int dot_mode, int which, int block, int carveout, int spmv_mode) {
    if (which == 0 && variant == RBS_PIPELINED) return spmv_blocks_per_sm(block, carveout, spmv_mode);
    static QueryCache<std::tuple<int, int, int, int, int, int>> cache;
    return cache.get({variant, dot_mode, which, block, carveout, spmv_mode}, [&] {
        apply_carveout(dot_mode, carveout);
        if (dot_mode == RBS_DOT_PLAIN)
            return blocks_per_sm_t<PlainR<1>, PlainR<2>, PlainR<2>, PlainR<5>>(variant, which, block, spmv_mode);
        return blocks_per_sm_t<ExactR<1, SQ>, ExactR<2, SQ>, RowsR2, RowsR5>(variant, which, block, spmv_mode);
    });
}

}  // namespace rbs

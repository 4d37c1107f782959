// One small system in one launch: a thread-block cluster of SMALL_CTAS CTAs
// keeps the whole solve on chip. Each CTA owns a contiguous share of the rows:
// its slice of the matrix and of every vector stay in its shared memory from
// set-up to the end, the gathered vectors are read from the other CTAs' shared
// memory, and each exact dot is summed over the cluster by exchanging limbs.
//
// Why: below about 20000 unknowns an iteration of the launch-per-step loop is
// nothing but launch and reduction latency (16^3: 35 us for five kernels and the
// loop node, whatever the matrix). Here a reduction is one cluster barrier and
// an iteration five of them: 12.5 us at 16^3, and no graph to build when the
// caller's buffers change (24 iterations, whole call: 1.12 -> 0.36 ms). What
// bounds it is that latency and, as the system grows, the 16 SMs' FP64 pipes (22
// operations per row and iteration); at 24^3 it takes 18 us against 36, so the
// line lies at what fits the shared memory.
//
// Arithmetic, fma forms and tails are those of the other paths, every CTA rounds
// the same integers and takes the same decisions, so results are bitwise theirs.
#include <mutex>

#include "kernels.cuh"
#include "launch.h"
#include "solver_elem.cuh"
#include "tails.cuh"

namespace rbs {

namespace {

constexpr int SMALL_T = 512;
constexpr int MAIL = 24;  // limbs of a CTA's partial sum that travel by mail; wider ones are read where they are

// vectors of a CTA's rows, in order (classic: the first 10)
enum { VX, VR, VR0, VPH, VS, VQ, VQH, VY, VD, VP, VRH = VP, VW, VWH, VT, VSH, VZ, VZH, VV };
constexpr int NV_CLASSIC = 10, NV_PIPE = 17;

// ---- cluster primitives ------------------------------------------------------------

__device__ __forceinline__ uint32_t cluster_rank() {
    uint32_t r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}
// Every thread of every CTA: arrive (release), wait (acquire).
__device__ __forceinline__ void cluster_barrier() {
    asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;\n" ::: "memory");
}
// Address of this CTA's shared location `addr` in the CTA of rank `rank`.
__device__ __forceinline__ uint32_t map_rank(uint32_t addr, uint32_t rank) {
    uint32_t a;
    asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(a) : "r"(addr), "r"(rank));
    return a;
}
__device__ __forceinline__ double ld_cluster(uint32_t addr) {
    double v;
    asm volatile("ld.shared::cluster.f64 %0, [%1];" : "=d"(v) : "r"(addr) : "memory");
    return v;
}
__device__ __forceinline__ unsigned long long ld_cluster_u64(uint32_t addr) {
    unsigned long long v;
    asm volatile("ld.shared::cluster.u64 %0, [%1];" : "=l"(v) : "r"(addr) : "memory");
    return v;
}
__device__ __forceinline__ void st_cluster(uint32_t addr, unsigned long long v) {
    asm volatile("st.shared::cluster.u64 [%0], %1;" ::"r"(addr), "l"(v) : "memory");
}
__device__ __forceinline__ void st_cluster(uint32_t addr, uint32_t v) {
    asm volatile("st.shared::cluster.u32 [%0], %1;" ::"r"(addr), "r"(v) : "memory");
}

// ---- exact dots over the cluster -----------------------------------------------------

// KM: most dots of one reduction. Two buffers: a reduction's partial sums may
// still be read while the next one's are written (never the one after: a
// barrier lies between).
template <int KM>
struct SmallShared {
    unsigned long long acc[2][KM][NL];
    unsigned long long mail[2][KM][SMALL_CTAS][MAIL];
    uint32_t head[2][KM][SMALL_CTAS];  // lowest limb, highest << 8, flags << 16; HEAD_EMPTY
    long long red[KM][NL];
    uint32_t flags[2][KM];
    double vals[KM];
    SolverState st;
};
constexpr uint32_t HEAD_EMPTY = 255u;
template <int KM>
__device__ __forceinline__ SmallShared<KM> &small_shared() {
    __shared__ SmallShared<KM> S;
    return S;
}

// Sum the first K accumulators of buffer b over the cluster; afterwards vals
// holds them, rounded, in every CTA, and the other buffer's accumulators are
// zero. Every thread of every CTA calls it, with its windows flushed. One copy
// of the code for all reductions (an iteration's code is walked once by one warp
// per dot: inlined and unrolled, it came from beyond the instruction cache).
template <int KM>
__device__ __noinline__ void small_exchange(int K, int b, uint32_t rank) {
    constexpr unsigned FULL = 0xffffffffu;
    SmallShared<KM> &S = small_shared<KM>();
    const int lane = threadIdx.x & 31, k = threadIdx.x >> 5;
    __syncthreads();
    if (k < K) {
        // this CTA's nonzero limbs, from a multiple of 8 on, to every CTA
        int lo = NL, hi = -1;
#pragma unroll
        for (int t = 0; t < (NL + 31) / 32; t++) {
            const int j = lane + 32 * t;
            if (j < NL && S.acc[b][k][j]) {
                lo = min(lo, j);
                hi = j;
            }
        }
        lo = (int)__reduce_min_sync(FULL, (unsigned)lo) & ~7;
        hi = (int)__reduce_max_sync(FULL, (unsigned)(hi + 1)) - 1;
        const bool empty = hi < 0;
        const uint32_t head = (empty ? HEAD_EMPTY : (uint32_t)lo | (uint32_t)hi << 8) | S.flags[b][k] << 16;
        const unsigned long long v = !empty && lane < MAIL && lo + lane < NL ? S.acc[b][k][lo + lane] : 0ull;
        const uint32_t at = smem_u32(&S.mail[b][k][rank][lane < MAIL ? lane : 0]);
        if (lane < MAIL) {
#pragma unroll
            for (uint32_t r = 0; r < SMALL_CTAS; r++) st_cluster(map_rank(at, r), v);
        }
        if (lane < SMALL_CTAS) st_cluster(map_rank(smem_u32(&S.head[b][k][rank]), (uint32_t)lane), head);
    }
    cluster_barrier();
    // the other buffer's partial sums have been read by everybody
    for (int j = threadIdx.x; j < KM * NL; j += SMALL_T) (&S.acc[b ^ 1][0][0])[j] = 0ull;
    if (threadIdx.x < KM) S.flags[b ^ 1][threadIdx.x] = 0u;
    if (k < K) {
        const uint32_t head = lane < SMALL_CTAS ? S.head[b][k][lane] : HEAD_EMPTY;
        const bool empty = (head & 255u) == HEAD_EMPTY;
        const uint32_t flags = __reduce_or_sync(FULL, head >> 16);
        const int lo = (int)__reduce_min_sync(FULL, empty ? 255u : head & 255u);
        const int hi = (int)__reduce_max_sync(FULL, empty ? 0u : ((head >> 8) & 255u) + 1u) - 1;
        double v = 0.0;
        bool done = flags == 0u && hi < 0;  // nothing but zeros
        if (!done && flags == 0u && hi - lo < MAIL && __all_sync(FULL, empty || (int)(head & 255u) == lo)) {
            // all from one limb on (the usual case): lane l sums limb lo + l
            long long sum = 0;
            if (lane < MAIL) {
#pragma unroll
                for (int r = 0; r < SMALL_CTAS; r++) sum += (long long)S.mail[b][k][r][lane];
            }
            done = round_lanes(sum, lo, v);
        }
        if (!done) {
            // (two limbs past the highest too: the rounding reads them)
            for (int L = lo + lane; L - lane <= hi + 2; L += 32) {
                long long sum = 0;
#pragma unroll 1
                for (int r = 0; r < SMALL_CTAS; r++) {
                    const uint32_t h = S.head[b][k][r];
                    const int a = (int)(h & 255u), e = (int)((h >> 8) & 255u);
                    if (a == (int)HEAD_EMPTY || L < a || L > e) continue;
                    sum += (long long)(e - a < MAIL ? S.mail[b][k][r][L - a]
                                                    : ld_cluster_u64(map_rank(smem_u32(&S.acc[b][k][L]), (uint32_t)r)));
                }
                if (L < NL) S.red[k][L] = sum;
            }
            __syncwarp();
            v = round_limbs_warp(S.red[k], flags, lo <= hi ? lo : -1, hi);
        }
        if (lane == 0) S.vals[k] = v;
    }
    __syncthreads();
}

// One thread's window into its CTA's accumulator: windows of one anchor by warp
// sums (as warp_flush), others each by its own atomics.
template <int Q>
__device__ __forceinline__ void small_flush(Win<Q> &W, unsigned long long *acc) {
    constexpr unsigned FULL = 0xffffffffu;
    const bool has = W.a >= 0;
    const int lo = (int)__reduce_min_sync(FULL, (unsigned)(has ? W.a : 0x7fffffff));
    const int hi = (int)__reduce_max_sync(FULL, (unsigned)(has ? W.a : 0));
    if (lo == 0x7fffffff) return;
    if (lo == hi) {
        warp_sum(W.w, acc, lo);
        win_clear<Q>(W);
    } else {
        win_flush<Q>(W, acc);
    }
}

// K dots over the cluster, into vals. b: the buffer, flipped here.
template <int K, int KM>
__device__ __forceinline__ void small_reduce(SmallShared<KM> &S, Win<SQ> (&win)[K], uint32_t (&fl)[K], int &b,
                                             uint32_t rank) {
#pragma unroll
    for (int j = 0; j < K; j++) {
        small_flush<SQ>(win[j], S.acc[b][j]);
        if (fl[j]) atomicOr(&S.flags[b][j], fl[j]);
        fl[j] = 0u;
    }
    small_exchange<KM>(K, b, rank);
    b ^= 1;
}

}  // namespace

struct SmallArgs {
    CSRArgs A;
    const double *b, *x0, *diag;
    double *x, *hist;
    double tol;
    BatchOut *out;  // zero
    int32_t maxit, variant, hist_cap;
    int32_t rows, cap;  // rows and nonzeros that a CTA has room for
};

namespace {

template <bool PIPE>
__global__ void __launch_bounds__(SMALL_T, 1) k_small(const __grid_constant__ SmallArgs a) {
    constexpr int KM = PIPE ? 5 : 2, NV = PIPE ? NV_PIPE : NV_CLASSIC;
    extern __shared__ __align__(16) unsigned char dyn[];
    SmallShared<KM> &S = small_shared<KM>();
    const int tid = threadIdx.x, rp = a.rows;
    const uint32_t rank = cluster_rank();
    const int n = (int)a.A.n, lo = min((int)rank * rp, n), rows = min(rp, n - lo);
    double *val = reinterpret_cast<double *>(dyn);
    double *vec = val + a.cap;  // vector v of this CTA's rows: vec + v * rp
    uint32_t *src = reinterpret_cast<uint32_t *>(vec + (size_t)NV * rp);  // where each nonzero's x entry is (of VPH)
    int *off = reinterpret_cast<int *>(src + a.cap);                      // first nonzero of each row
    auto V = [&](int v) { return vec + (size_t)v * rp; };
    for (int j = tid; j < 2 * KM * NL; j += SMALL_T) (&S.acc[0][0][0])[j] = 0ull;
    if (tid < 2 * KM) (&S.flags[0][0])[tid] = 0u;
    if (tid == 0) {
        memset(&S.st, 0, sizeof S.st);
        S.st.tol = a.tol;
        S.st.maxit = a.maxit;
        S.st.variant = a.variant;
        S.st.hist_cap = rank == 0 ? a.hist_cap : 0;
    }
    // ---- structure check, matrix slice, Jacobi ----
    const int64_t first = a.A.rowptr[lo], last = a.A.rowptr[lo + rows];
    unsigned err = 0u;
    if (rank == 0 && tid == 0 && (a.A.rowptr[0] != 0 || a.A.rowptr[n] != a.A.nnz)) err |= 1u;
    const bool sound = first >= 0 && last >= first && last <= a.A.nnz;  // the same for every thread of the CTA
    if (!sound) err |= 1u;
    else if (last - first > a.cap) err |= SMALL_NO_ROOM;
    if (sound && last - first <= a.cap) {
        const uint32_t base = smem_u32(V(VPH));
        const int count = (int)(last - first);
        for (int i = tid; i <= rows; i += SMALL_T) {
            const int64_t p = a.A.rowptr[lo + i];
            if (p < first || p > last || (i < rows && a.A.rowptr[lo + i + 1] < p)) err |= 1u;
            off[i] = (int)(p - first);
        }
        for (int k = tid; k < count; k += SMALL_T) {
            const int32_t c = a.A.col[first + k];
            const bool in = (uint32_t)c < (uint32_t)n;
            if (!in) err |= 1u;
            const uint32_t owner = in ? (uint32_t)c / (uint32_t)rp : 0u;
            src[k] = map_rank(base + (in ? (uint32_t)c - owner * (uint32_t)rp : 0u) * 8u, owner);
            val[k] = a.A.val[first + k];
        }
        const bool bad = __syncthreads_or((int)(err & 1u)) != 0;
        for (int i = tid; i < rows && !bad; i += SMALL_T) {
            const uint32_t self = map_rank(base + (uint32_t)i * 8u, rank);
            double d = 0.0;
            bool found = false;
            if (a.diag) {
                d = a.diag[lo + i];
                found = true;
            } else {
                for (int k = off[i]; k < off[i + 1]; k++)
                    if (src[k] == self) {
                        d = val[k];
                        found = true;
                        break;
                    }
            }
            if (!found || d == 0.0 || d != d) err |= 2u;
            V(VD)[i] = !found || d == 0.0 || d != d ? 0.0 : __ddiv_rn(1.0, d);
        }
    }
    if (err) atomicOr(&a.out->err, err);
    cluster_barrier();
    // (the same word for every CTA: nobody writes it after the barrier)
    if (*(volatile const unsigned *)&a.out->err != 0u) return;
    // y_i = row i times the vector that lies `shift` bytes after VPH, fma chain in
    // stored order from +0.0
    auto row = [&](int i, uint32_t shift) {
        double acc = 0.0;
        const int e = off[i + 1];
        for (int k0 = off[i]; k0 < e; k0 += 8) {
            double xv[8];
#pragma unroll
            for (int j = 0; j < 8; j++)
                if (k0 + j < e) xv[j] = ld_cluster(src[k0 + j] + shift);
#pragma unroll
            for (int j = 0; j < 8; j++)
                if (k0 + j < e) acc = fma(val[k0 + j], xv[j], acc);
        }
        return acc;
    };
    auto shift_of = [&](int v) { return (uint32_t)((v - VPH) * rp * 8); };
    auto each = [&](auto &&f) {
        for (int i = tid; i < rows; i += SMALL_T) f(i);
    };
    int b = 0;
    SolverState *st = &S.st;
    auto tail = [&](auto &&f) {
        if (tid == 0) f();
        __syncthreads();
    };
    double *x = V(VX), *r = V(VR), *r0 = V(VR0), *ph = V(VPH), *s = V(VS), *q = V(VQ), *qh = V(VQH), *y = V(VY),
           *d = V(VD);
    Win<SQ> w1[1], w2[2];
    uint32_t f1[1] = {0u}, f2[2] = {0u, 0u};
    w1[0].init();
    w2[0].init();
    w2[1].init();
    // r = b - A x0 (or b), x = x0 (or +0)
    bool bad = false;
    auto start = [&](int i) {
        double ri;
        if (a.x0) {
            const CSRView A{a.A.n, a.A.nnz, a.A.rowptr, a.A.col, a.A.val};
            ri = __dsub_rn(a.b[lo + i], spmv_row(A, lo + i, a.x0, bad));
            x[i] = a.x0[lo + i];
        } else {
            ri = a.b[lo + i];
            x[i] = 0.0;
        }
        r[i] = ri;
        r0[i] = ri;
        return ri;
    };
    if constexpr (!PIPE) {
        double *p = V(VP);
        each([&](int i) {
            const double ri = start(i);
            p[i] = ri;
            ph[i] = __dmul_rn(ri, d[i]);
            exact_add<SQ, true>(w1[0], f1[0], S.acc[b][0], ri, ri);
        });
        small_reduce<1>(S, w1, f1, b, rank);
        tail([&] { tail_cls_setup(st, S.vals); });
        for (int guard = 0; !st->done && guard <= a.maxit; guard++) {
            each([&](int i) {  // K1
                const double si = row(i, 0u);
                s[i] = si;
                exact_add<SQ>(w1[0], f1[0], S.acc[b][0], r0[i], si);
            });
            small_reduce<1>(S, w1, f1, b, rank);
            tail([&] { tail_cls_alpha(st, S.vals); });
            if (st->done) break;
            const double na = -st->alpha;
            each([&](int i) {  // K2
                const VPair u = cls_k2(na, s[i], r[i], d[i]);
                q[i] = u.a;
                qh[i] = u.b;
            });
            cluster_barrier();
            each([&](int i) {  // K3
                const double yi = row(i, shift_of(VQH));
                y[i] = yi;
                exact_add<SQ>(w2[0], f2[0], S.acc[b][0], q[i], yi);
                exact_add<SQ, true>(w2[1], f2[1], S.acc[b][1], yi, yi);
            });
            small_reduce<2>(S, w2, f2, b, rank);
            tail([&] { tail_cls_omega(st, S.vals); });
            const double al = st->alpha, om = st->omega, nom = -om;
            each([&](int i) {  // K4
                const VPair u = cls_k4(al, om, nom, qh[i], ph[i], x[i], y[i], q[i]);
                x[i] = u.a;
                r[i] = u.b;
                exact_add<SQ>(w2[0], f2[0], S.acc[b][0], r0[i], u.b);
                exact_add<SQ, true>(w2[1], f2[1], S.acc[b][1], u.b, u.b);
            });
            small_reduce<2>(S, w2, f2, b, rank);
            tail([&] { tail_cls_beta(st, S.vals, a.hist); });
            if (st->done) break;
            const double be = st->beta;
            each([&](int i) {  // K5
                const VPair u = cls_k5(be, nom, s[i], p[i], r[i], d[i]);
                p[i] = u.a;
                ph[i] = u.b;
            });
            cluster_barrier();
        }
    } else {
        double *rh = V(VRH), *w = V(VW), *wh = V(VWH), *t = V(VT), *sh = V(VSH), *z = V(VZ), *zh = V(VZH), *v = V(VV);
        Win<SQ> w5[5];
        uint32_t f5[5] = {0u, 0u, 0u, 0u, 0u};
#pragma unroll
        for (int k = 0; k < 5; k++) w5[k].init();
        each([&](int i) { rh[i] = __dmul_rn(start(i), d[i]); });
        cluster_barrier();
        each([&](int i) {
            const double wi = row(i, shift_of(VRH));
            w[i] = wi;
            wh[i] = __dmul_rn(wi, d[i]);
            exact_add<SQ, true>(w2[0], f2[0], S.acc[b][0], r0[i], r0[i]);
            exact_add<SQ>(w2[1], f2[1], S.acc[b][1], r0[i], wi);
        });
        small_reduce<2>(S, w2, f2, b, rank);  // also orders what for the gathers
        tail([&] { tail_pipe_setup(st, S.vals); });
        if (!st->done) each([&](int i) { t[i] = row(i, shift_of(VWH)); });
        struct Two {  // p1_elem's reducer
            Win<SQ> *w;
            uint32_t *f;
            unsigned long long (*acc)[NL];
            __device__ __forceinline__ void add(int k, double x, double y) { exact_add<SQ>(w[k], f[k], acc[k], x, y); }
            __device__ __forceinline__ void add_sq(int k, double x) { exact_add<SQ, true>(w[k], f[k], acc[k], x, x); }
        };
        for (int guard = 0; !st->done && guard <= a.maxit; guard++) {
            const double al = st->alpha, nal = -al, be = st->beta, nom0 = -st->omega;
            const bool first_it = st->iter == 0;
            each([&](int i) {  // P1
                P1In in{rh[i], w[i], wh[i], t[i], r[i], d[i], 0.0, 0.0, 0.0, 0.0, 0.0, 0.0};
                if (!first_it) {
                    in.ph = ph[i];
                    in.s = s[i];
                    in.sh = sh[i];
                    in.z = z[i];
                    in.zh = zh[i];
                    in.v = v[i];
                }
                Two red{w2, f2, S.acc[b]};
                const P1Out o = p1_elem(in, first_it, nal, be, nom0, red);
                ph[i] = o.ph;
                s[i] = o.s;
                sh[i] = o.sh;
                z[i] = o.z;
                q[i] = o.q;
                qh[i] = o.qh;
                y[i] = o.y;
                zh[i] = o.zh;
            });
            small_reduce<2>(S, w2, f2, b, rank);  // also orders zhat for P2's gathers
            tail([&] { tail_pipe_omega(st, S.vals); });
            each([&](int i) { v[i] = row(i, shift_of(VZH)); });  // P2
            const double om = st->omega, nom = -om;
            each([&](int i) {  // P3
                Two red{w5, f5, S.acc[b]};
                const P3Out o = p3_elem(P3In{qh[i], y[i], q[i], ph[i], x[i], zh[i], wh[i], v[i], t[i], d[i], r0[i],
                                             s[i], z[i]},
                                        al, nal, om, nom, red);
                x[i] = o.x;
                r[i] = o.r;
                rh[i] = o.rh;
                w[i] = o.w;
                wh[i] = o.wh;
            });
            small_reduce<5>(S, w5, f5, b, rank);  // also orders what for P4's gathers
            tail([&] { tail_pipe_beta(st, S.vals, a.hist); });
            if (st->done) break;
            each([&](int i) { t[i] = row(i, shift_of(VWH)); });  // P4
        }
    }
    each([&](int i) { a.x[lo + i] = x[i]; });
    if (rank == 0 && tid == 0) {
        a.out->iters = st->iter;
        a.out->status = st->status;
        a.out->converged = (st->status == RBS_OK && !(st->tau > st->tau_max)) ? 1 : 0;
        a.out->tau0 = st->tau0;
        a.out->tau_final = st->tau;
        a.out->rho0 = st->rho0;
        a.out->tau_max = st->tau_max;
        a.out->alpha0 = st->alpha0;
        a.out->mu0 = st->mu0;
    }
    cluster_barrier();  // no CTA leaves while its shared memory may be read
}

// Dynamic shared memory of a launch of this variant that this device allows; 0
// if it cannot run a cluster of SMALL_CTAS. Once per device and variant.
size_t small_room(int variant) {
    static std::mutex mu;
    static size_t room[64][2];
    static bool known[64][2];
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return 0;
    std::lock_guard<std::mutex> lk(mu);
    if (known[dev][variant]) return room[dev][variant];
    const void *fn = variant == RBS_PIPELINED ? (const void *)k_small<true> : (const void *)k_small<false>;
    size_t got = 0;
    cudaFuncAttributes at;
    int most = 0;
    if (cudaFuncGetAttributes(&at, fn) == cudaSuccess &&
        cudaDeviceGetAttribute(&most, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev) == cudaSuccess &&
        (size_t)most > at.sharedSizeBytes) {
        got = ((size_t)most - at.sharedSizeBytes) / 16 * 16;
        if (cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)got) != cudaSuccess ||
            cudaFuncSetAttribute(fn, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess)
            got = 0;
    }
    if (got) {
        cudaLaunchConfig_t cfg = {};
        cudaLaunchAttribute attr;
        cfg.gridDim = dim3(SMALL_CTAS);
        cfg.blockDim = dim3(SMALL_T);
        cfg.dynamicSmemBytes = got;
        attr.id = cudaLaunchAttributeClusterDimension;
        attr.val.clusterDim.x = SMALL_CTAS;
        attr.val.clusterDim.y = attr.val.clusterDim.z = 1;
        cfg.attrs = &attr;
        cfg.numAttrs = 1;
        int fit = 0;
        if (cudaOccupancyMaxActiveClusters(&fit, fn, &cfg) != cudaSuccess || fit < 1) got = 0;
    }
    cudaGetLastError();
    room[dev][variant] = got;
    known[dev][variant] = true;
    return got;
}

// Rows per CTA and nonzeros it then has room for.
void small_shape(int64_t n, int variant, size_t room, int *rows, int *cap) {
    *rows = (int)((n + SMALL_CTAS - 1) / SMALL_CTAS);
    const size_t vecs = (size_t)(variant == RBS_PIPELINED ? NV_PIPE : NV_CLASSIC) * (size_t)*rows * 8 +
                        ((size_t)*rows + 2) * 4;
    *cap = room > vecs ? (int)((room - vecs) / 12 / 2 * 2) : 0;
}

}  // namespace

bool small_fits(int64_t n, int64_t nnz, int variant) {
    if (n > 1 << 20) return false;
    const size_t room = small_room(variant);
    if (!room) return false;
    int rows, cap;
    small_shape(n, variant, room, &rows, &cap);
    return nnz <= (int64_t)cap * SMALL_CTAS;
}

cudaError_t launch_small(const CSRArgs &A, const double *b, const double *x0, const double *diag, double *x, double tol,
                         int32_t maxit, int variant, double *hist, int32_t hist_cap, BatchOut *d_out, cudaStream_t s) {
    const size_t room = small_room(variant);
    SmallArgs a{A, b, x0, diag, x, hist, tol, d_out, maxit, variant, hist_cap, 0, 0};
    small_shape(A.n, variant, room, &a.rows, &a.cap);
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute attr;
    cfg.gridDim = dim3(SMALL_CTAS);
    cfg.blockDim = dim3(SMALL_T);
    cfg.dynamicSmemBytes = room;
    cfg.stream = s;
    attr.id = cudaLaunchAttributeClusterDimension;
    attr.val.clusterDim.x = SMALL_CTAS;
    attr.val.clusterDim.y = attr.val.clusterDim.z = 1;
    cfg.attrs = &attr;
    cfg.numAttrs = 1;
    return variant == RBS_PIPELINED ? cudaLaunchKernelEx(&cfg, k_small<true>, a) : cudaLaunchKernelEx(&cfg, k_small<false>, a);
}

}  // namespace rbs

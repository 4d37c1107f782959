// Reducers used by every kernel that carries dot products:
//  ExactR<K, Q>  the reproducible exact dot (exact_acc.cuh), K dots at once;
//  PlainR<K>     the comparator: binary64 fma accumulation per thread, warp
//                and block trees, then atomicAdd across blocks, whose order
//                changes from run to run (the paper's non-reproducible
//                "original", Sec. 3.2 / Sec. 4.1).
// Both end with the same last-block protocol, so solver tails are shared.
#pragma once

#include "exact_acc.cuh"

namespace rbs {

template <int K_, int Q>
struct ExactR {
    static constexpr int K = K_;
    Win<Q> win[K];
    uint32_t flags[K];
    unsigned long long (*sacc)[NL];
    uint32_t *sflags;

    __device__ __forceinline__ void init() {
        __shared__ unsigned long long s_acc[K][NL];
        __shared__ uint32_t s_flags[K];
        sacc = s_acc;
        sflags = s_flags;
#pragma unroll
        for (int k = 0; k < K; k++) {
            win[k].init();
            flags[k] = 0u;
        }
        sacc_zero<K>(sacc, sflags);
    }
    __device__ __forceinline__ void add(int k, double x, double y) {
        exact_add<Q>(win[k], flags[k], sacc[k], x, y);
    }
    __device__ __forceinline__ void add_sq(int k, double x) {
        exact_add<Q, true>(win[k], flags[k], sacc[k], x, x);
    }
    // true in the last block, with vals[0..K-1] rounded (shared memory).
    // SCRATCH: the per-warp scratch size the kernel already uses, so that the
    // flush staging shares it.
    // coop = false after a timed-out staged copy (ERR_TIMEOUT): per-lane flushes
    template <int SCRATCH = FLUSH_SCRATCH, int WARPS = MAX_WARPS>
    __device__ __forceinline__ bool finish(DotScratch *g, double *vals, unsigned nblk = 0u, bool coop = true) {
        return exact_finish<K, Q, SCRATCH, WARPS>(win, flags, sacc, sflags, g, vals, false, nullptr, nullptr, nblk,
                                                  coop);
    }
};

// Exact reducer of the standalone dots: per-thread windows in shared memory, W
// 32-bit words per sign (positive and negative products kept apart, so a
// product's five words are added to five words picked by address -- no word
// selects, no two's complement) as one add-with-carry chain. A carry out of the
// chain needs the sixth word to be all ones up to the product's top few bits,
// so the ripple that continues it is a branch almost never taken. Layout
// [sign][word][thread]: a thread's words share one bank, whatever their
// placement, so every access is conflict-free.
//
// What bounds it: at the HBM rate an SM has 0.72 cycles per element pair. The
// window update used to be five 64-bit carry-save digits, whose loads and
// stores alone took 0.63 of them; 32-bit words take 0.31, and one add each
// instead of two. One branch per four products and two middle terms summed as
// 64 bits bring a product to 62 instructions from 90 (2^24 products, cond 1e48:
// 54 us from 73).
//
// The window covers W - 4 placements. All threads of a block start with one
// anchor (open()): the block's largest first product lands at placement ANCHOR,
// which leaves up to three placements (96 bits) above it. A product above the window
// flushes and re-anchors its thread's own; one below goes straight into the
// block accumulator. While a warp's anchors agree (they differ only after a
// product above the window) the flush at the end sums each word over the warp
// with one lane per word.
template <int W_>
struct ExactW {
    static constexpr int W = W_;
    static constexpr int QMAX = W - 5;             // highest placement of a product's lowest word
    // placement of the product that (re)anchors the window: up to three above it
    static constexpr int ANCHOR = QMAX - (QMAX + 2) / 4;
    static constexpr int NT = 256;                 // most threads per block (column stride)
    static_assert(2 * W <= 32, "the warp flush gives each word of each sign a lane");
    uint32_t *win;  // this thread's column: word j of sign s at win[(s * W + j) * NT]
    int a;          // anchor limb, WIN_EMPTY when there is no window yet
    unsigned long long (*sacc)[NL];
    uint32_t *sflags;
    int *amax;

    __device__ __forceinline__ void init() {
        __shared__ uint32_t s_win[(2 * W + 5) * NT];  // the last five rows take zero products
        __shared__ unsigned long long s_acc[1][NL];
        __shared__ uint32_t s_flags[1];
        __shared__ int s_amax;
        win = s_win + threadIdx.x;
        sacc = s_acc;
        sflags = s_flags;
        amax = &s_amax;
        a = WIN_EMPTY;
#pragma unroll
        for (int j = 0; j < 2 * W; j++) win[j * NT] = 0u;
        if (threadIdx.x == 0) s_amax = -1;
        sacc_zero<1>(sacc, sflags);
    }
    // The limb of x*y's lowest bit, for the common start anchor (-1: no finite nonzero normal product).
    static __device__ __forceinline__ int limb_of(double x, double y) {
        const uint32_t ex = (uint32_t)__double2hiint(x) & 0x7ff00000u, ey = (uint32_t)__double2hiint(y) & 0x7ff00000u;
        if (ex - 0x00100000u >= 0x7fe00000u || ey - 0x00100000u >= 0x7fe00000u) return -1;
        return (int)((ex + ey - (2u << 20)) >> 25);
    }
    // The common start anchor from every thread's first products (their highest
    // limb, -1 for none). All threads call it, before the first add.
    __device__ __forceinline__ void open(int limb) {
        const int m = __reduce_max_sync(0xffffffffu, limb);
        if ((threadIdx.x & 31) == 0) atomicMax(amax, m);
        __syncthreads();
        if (*amax >= 0) a = max(*amax - ANCHOR, 0);
    }
    // One thread's window (column w, anchor a) into the block
    // accumulator sk, with its own atomics; words back to zero.
    static __device__ __forceinline__ void flush_column(uint32_t *w, unsigned long long *sk, int a) {
        for (int j = 0; j < W; j++) {
            const long long d = (long long)w[j * NT] - (long long)w[(W + j) * NT];
            w[j * NT] = 0u;
            w[(W + j) * NT] = 0u;
            if (d) sacc_add(&sk[a + j], d);
        }
    }
    // +1 to word j of a sign's words p (a carry), or past the window's top into
    // the block accumulator.
    static __device__ __forceinline__ void ripple(uint32_t *p, unsigned long long *sk, int a, int j, bool neg) {
        for (; j < W; j++) {
            const uint32_t v = p[j * NT] + 1u;
            p[j * NT] = v;
            if (v) return;
        }
        if (a + W < NL) sacc_add(&sk[a + W], neg ? -1ll : 1ll);
    }
    // Products of any kind: zeros, subnormals and non-finite operands, products in
    // the window, below it (into the block accumulator) and above it (flush and
    // re-anchor). v: x and y of each in turn. Returns the thread's anchor.
    template <class... D>
    static __device__ __noinline__ int add_any(uint32_t *w, unsigned long long *sk, uint32_t *fl, int a, D... v) {
        const double xy[] = {v...};
#pragma unroll
        for (int i = 0; i < (int)sizeof...(D); i += 2) {
            uint32_t u[5], m, f = 0u;
            int L;
            if (!prod_exact(xy[i], xy[i + 1], f, u, L, m)) {
                if (f) atomicOr(fl, f);
                continue;
            }
            if (L < a) {
                smem_deposit(sk, u, L, m);
                continue;
            }
            if (L - a > QMAX) {
                if (a >= 0) flush_column(w, sk, a);
                a = L > ANCHOR ? L - ANCHOR : 0;
            }
            uint32_t *p = w + (m ? W * NT : 0);
            unsigned long long t = 0;
            for (int j = 0; j < 5; j++) {
                t += (unsigned long long)p[(L - a + j) * NT] + u[j];
                p[(L - a + j) * NT] = (uint32_t)t;
                t >>= 32;
            }
            if (t) ripple(p, sk, a, L - a + 5, m != 0u);
        }
        return a;
    }
    // The carries out of the five words of add()'s products (rare): bit i of
    // `carries` for product i, its sign at bit 16 + i, its placement in byte i
    // of qs (at most four products).
    static __device__ __noinline__ void carries_out(uint32_t *w, unsigned long long *sk, int a, uint32_t carries,
                                                    uint32_t qs) {
        for (int i = 0; i < 4; i++) {
            const int q = (int)(qs >> 8 * i) & 255;
            const bool neg = ((carries >> (16 + i)) & 1u) != 0u;
            if (((carries >> i) & 1u) && q <= QMAX) ripple(w + (neg ? W * NT : 0), sk, a, q + 5, neg);
        }
    }
    static_assert(2 * W <= 255, "placements in bytes, the zero products' included");
    // N products into the window. One branch for all of them: when every operand
    // is normal and every product lands in the window (nearly always), straight
    // code. Otherwise zero products are sent to five words that nobody reads, and
    // any other kind sends all N through add_any(). N is 1, 2 or 4.
    template <int N>
    __device__ __forceinline__ void add(const double (&x)[N], const double (&y)[N]) {
        uint32_t xh[N], yh[N], e[N], q[N], odd = 0u, far = 0u;
#pragma unroll
        for (int i = 0; i < N; i++) {
            xh[i] = (uint32_t)__double2hiint(x[i]);
            yh[i] = (uint32_t)__double2hiint(y[i]);
            const uint32_t ex = xh[i] & 0x7ff00000u, ey = yh[i] & 0x7ff00000u;
            odd = max(max(odd, ex - 0x00100000u), ey - 0x00100000u);
            e[i] = ex + ey - (2u << 20);  // bit position << 20; garbage for an odd operand
            q[i] = (e[i] >> 25) - (uint32_t)a;
            far = max(far, q[i]);
        }
        bool go = true;
        if (!(odd < 0x7fe00000u && far <= (uint32_t)QMAX)) {
            go = a >= 0;
#pragma unroll
            for (int i = 0; i < N; i++) {
                const uint32_t ex = xh[i] & 0x7ff00000u, ey = yh[i] & 0x7ff00000u;
                const uint32_t zx = (xh[i] & 0x7fffffffu) | (uint32_t)__double2loint(x[i]);
                const uint32_t zy = (yh[i] & 0x7fffffffu) | (uint32_t)__double2loint(y[i]);
                if (min(zx, zy) == 0u && max(ex, ey) < 0x7ff00000u) {
                    q[i] = (uint32_t)(2 * W);
                    xh[i] = yh[i];
                } else {
                    go = go && max(ex - 0x00100000u, ey - 0x00100000u) < 0x7fe00000u && q[i] <= (uint32_t)QMAX;
                }
            }
            if (!go) {
                if constexpr (N == 1)
                    a = add_any(win, sacc[0], sflags, a, x[0], y[0]);
                else if constexpr (N == 2)
                    a = add_any(win, sacc[0], sflags, a, x[0], y[0], x[1], y[1]);
                else
                    a = add_any(win, sacc[0], sflags, a, x[0], y[0], x[1], y[1], x[2], y[2], x[3], y[3]);
            }
        }
        if (go) {
            uint32_t carries = 0u;
#pragma unroll
            for (int i = 0; i < N; i++) {
                const uint32_t xl = (uint32_t)__double2loint(x[i]), yl = (uint32_t)__double2loint(y[i]);
                const uint32_t A1 = (xh[i] & 0xfffffu) | 0x100000u, B1 = (yh[i] & 0xfffffu) | 0x100000u;
                // 106-bit significand product: the two middle terms share one 64-bit sum (< 2^54)
                const unsigned long long lo = (unsigned long long)xl * yl, hi = (unsigned long long)A1 * B1;
                const unsigned long long mid = (unsigned long long)xl * B1 + (unsigned long long)A1 * yl;
                uint32_t p1, p2, p3, u[5], c;
                asm("add.cc.u32 %0, %3, %4;\n\t"
                    "addc.cc.u32 %1, %5, %6;\n\t"
                    "addc.u32 %2, %7, 0;"
                    : "=&r"(p1), "=&r"(p2), "=r"(p3)
                    : "r"((uint32_t)(lo >> 32)), "r"((uint32_t)mid), "r"((uint32_t)hi), "r"((uint32_t)(mid >> 32)),
                      "r"((uint32_t)(hi >> 32)));
                const uint32_t r = e[i] >> 20;  // the funnel shifts take it modulo 32
                u[0] = __funnelshift_l(0u, (uint32_t)lo, r);
                u[1] = __funnelshift_l((uint32_t)lo, p1, r);
                u[2] = __funnelshift_l(p1, p2, r);
                u[3] = __funnelshift_l(p2, p3, r);
                u[4] = __funnelshift_l(p3, 0u, r);
                uint32_t *p = win + q[i] * NT + ((xh[i] ^ yh[i]) >> 31) * (W * NT);
                uint32_t w0 = p[0], w1 = p[NT], w2 = p[2 * NT], w3 = p[3 * NT], w4 = p[4 * NT];
                asm("add.cc.u32 %0, %0, %6;\n\t"
                    "addc.cc.u32 %1, %1, %7;\n\t"
                    "addc.cc.u32 %2, %2, %8;\n\t"
                    "addc.cc.u32 %3, %3, %9;\n\t"
                    "addc.cc.u32 %4, %4, %10;\n\t"
                    "addc.u32 %5, 0, 0;"
                    : "+r"(w0), "+r"(w1), "+r"(w2), "+r"(w3), "+r"(w4), "=r"(c)
                    : "r"(u[0]), "r"(u[1]), "r"(u[2]), "r"(u[3]), "r"(u[4]));
                p[0] = w0;
                p[NT] = w1;
                p[2 * NT] = w2;
                p[3 * NT] = w3;
                p[4 * NT] = w4;
                carries += c << i;
            }
            if (carries) {
                uint32_t qs = 0u;
#pragma unroll
                for (int i = 0; i < N; i++) {
                    qs |= q[i] << 8 * i;
                    carries |= ((xh[i] ^ yh[i]) >> 31) << (16 + i);
                }
                carries_out(win, sacc[0], a, carries, qs);
            }
        }
    }
    __device__ __forceinline__ void add_one(double x, double y) {
        const double xv[1] = {x}, yv[1] = {y};
        add<1>(xv, yv);
    }
    // Flush of every lane's window at the end of the kernel (all 32 lanes call
    // it). With one anchor in the warp, lane r sums word r of the W positive and
    // W negative words over the warp's columns, each lane starting at its own
    // column (32 banks, no conflicts); else every lane flushes its own.
    __device__ __forceinline__ void flush_warp() {
        constexpr unsigned FULL = 0xffffffffu;
        const int lane = threadIdx.x & 31;
        const int a0 = __shfl_sync(FULL, a, 0);
        if (!__all_sync(FULL, a == a0)) {
            if (a >= 0) flush_column(win, sacc[0], a);
            return;
        }
        if (a0 < 0) return;
        __syncwarp();
        long long sum = 0;
        if (lane < 2 * W) {
            const uint32_t *row = win - lane + lane * NT;
#pragma unroll 8
            for (int i = 0; i < 32; i++) sum += (long long)row[(i + lane) & 31];
        }
        sum -= __shfl_down_sync(FULL, sum, W);
        if (lane < W && sum && a0 + lane < NL) sacc_add(&sacc[0][a0 + lane], sum);
    }
    // Reduction `slot` of g, over gridDim.x blocks (block_grid_finish).
    __device__ __forceinline__ bool finish(DotScratch *g, int slot, double *val, bool export_limbs = false,
                                           long long *limbs = nullptr, int32_t *fl = nullptr) {
        flush_warp();
        const uint32_t none[1] = {0u};  // add_any() has set the block's flags itself
        return block_grid_finish<1>(none, sacc, sflags, g, val, export_limbs, limbs, fl, gridDim.x, slot);
    }
};

template <int K_>
struct PlainR {
    static constexpr int K = K_;
    double s[K];

    __device__ __forceinline__ void init() {
#pragma unroll
        for (int k = 0; k < K; k++) s[k] = 0.0;
        __syncthreads();  // as the exact reducers' init
    }
    __device__ __forceinline__ void add(int k, double x, double y) { s[k] = fma(x, y, s[k]); }
    __device__ __forceinline__ void add_sq(int k, double x) { s[k] = fma(x, x, s[k]); }
    template <int SCRATCH = 0, int WARPS = MAX_WARPS>
    __device__ __forceinline__ bool finish(DotScratch *g, double *vals, unsigned nblk = 0u, bool coop = true) {
        (void)coop;  // its partials live in their own shared array
        __shared__ double s_part[K][32];
        const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
#pragma unroll
        for (int k = 0; k < K; k++) {
            double v = s[k];
            for (int o = 16; o > 0; o >>= 1) v = __dadd_rn(v, __shfl_down_sync(0xffffffffu, v, o));
            if (lane == 0) s_part[k][wid] = v;
        }
        __syncthreads();
        if (threadIdx.x < K) {
            double t = 0.0;
            for (int w = 0; w < (int)(blockDim.x >> 5); w++) t = __dadd_rn(t, s_part[threadIdx.x][w]);
            atomicAdd((double *)&g->limbs[threadIdx.x][0], t);
        }
        __threadfence();
        __syncthreads();
        __shared__ bool s_last;
        if (threadIdx.x == 0) s_last = (atomicAdd(&g->ticket[0], 1u) == (nblk ? nblk : gridDim.x) - 1);
        __syncthreads();
        if (!s_last) return false;
        __threadfence();
        if (threadIdx.x < K)
            vals[threadIdx.x] = __longlong_as_double((long long)atomicExch(&g->limbs[threadIdx.x][0], 0ull));
        if (threadIdx.x == 0) g->ticket[0] = 0u;
        __syncthreads();
        return true;
    }
};

}  // namespace rbs

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
        return exact_finish<K, Q, SCRATCH, WARPS>(win, flags, sacc, sflags, g, vals, nblk, coop);
    }
};

// Exact reducer with its per-thread windows in shared memory (the standalone dots
// and the vector kernels): per dot W 32-bit words; a product's five words are
// added to the five words at its placement, picked by address with no word
// selects, as one add-with-carry chain. Layout [dot, sign, word][thread]: a
// thread's words share one bank, whatever their placement, so every access is
// conflict-free.
//
// SPLIT: W words per sign, positive and negative products kept apart (the
// standalone dots: fewest instructions). Without it one set of words takes both,
// a negative product as its complement with 1 carried in; the words start at
// 2^31 and the flush takes that out again, so that a borrow, like a carry, leaves
// the five words only when the fifth is within the product's top few bits of its
// end: the ripple that continues it is a branch almost never taken. (Half the
// shared memory: what the vector kernels' windows take comes out of the L1 that
// their loads in flight need, and the registers that windows would take otherwise
// cost more still. K4 at 256^3: 191 us with register windows, whose products
// below the window go to atomics while the values still fall off steeply, 207
// with 47 KB of windows a block, 162 with 35; HBM alone 158.)
//
// What bounds it: at the HBM rate an SM has 0.72 cycles per element pair. The
// window update used to be five 64-bit carry-save digits, whose loads and
// stores alone took 0.63 of them; 32-bit words take 0.31, and one add each
// instead of two. One branch per four products and two middle terms summed as
// 64 bits bring a product to some 64 instructions from 90 (2^24 products, cond
// 1e48: 50 us from 73).
//
// A window covers W - 4 placements. Where a kernel has every thread's first
// products before it adds any, all threads of a block start with one anchor
// (open()): the block's largest first product lands at placement ANCHOR, which
// leaves up to three placements (96 bits) above it. Elsewhere a thread's first
// product opens its window, lanes that do so together with one anchor where their
// products all fit (a call and a divergent branch per thread: 1.5 us on a short
// dot). A product above the window flushes and re-anchors its thread's own; one
// below goes straight into the block accumulator. While a warp's anchors agree
// the flush at the end sums each word over the warp with one lane per word.
template <int K_, int W_, bool SPLIT>
struct ExactRows {
    static constexpr int K = K_;
    static constexpr int W = W_;
    static constexpr bool WINDOWS = true;  // open() before the first add
    static constexpr int QMAX = W - 5;  // highest placement of a product's lowest word
    // placement of the product that (re)anchors the window: up to three above it
    static constexpr int ANCHOR = QMAX - (QMAX + 2) / 4;
    static constexpr int NT = 256;  // most threads per block (column stride)
    static constexpr int PER = SPLIT ? 2 * W : W, ROWS = K * PER;
    static_assert(PER <= 32, "the warp flush gives each word a lane");
    static constexpr uint32_t ZERO = SPLIT ? 0u : 0x80000000u;  // a word that holds nothing
    static_assert(ROWS <= 255, "placements in bytes, the zero products' included");
    uint32_t *win;  // this thread's column: word j of sign s of dot k at win[(k * PER + s * W + j) * NT]
    // Anchor limbs. No window yet: NO_ANCHOR, with SPLIT the lowest window there is
    // (whose products, below 2^-1764, are as good as none).
    static constexpr int NO_ANCHOR = SPLIT ? 0 : WIN_EMPTY;
    int a[K];
    unsigned long long (*sacc)[NL];
    uint32_t *sflags;
    int *amax;

    __device__ __forceinline__ void init() {
        __shared__ uint32_t s_win[(ROWS + 5) * NT];  // the last five rows take zero products
        __shared__ unsigned long long s_acc[K][NL];
        __shared__ uint32_t s_flags[K];
        __shared__ int s_amax[K];
        win = s_win + threadIdx.x;
        sacc = s_acc;
        sflags = s_flags;
        amax = s_amax;
#pragma unroll
        for (int k = 0; k < K; k++) a[k] = NO_ANCHOR;
#pragma unroll
        for (int j = 0; j < ROWS; j++) win[j * NT] = ZERO;
        if (threadIdx.x < K) s_amax[threadIdx.x] = -1;
        sacc_zero<K>(sacc, sflags);
    }
    // The limb of x*y's lowest bit, for the common start anchor (-1: no finite nonzero normal product).
    static __device__ __forceinline__ int limb_of(double x, double y) {
        const uint32_t ex = (uint32_t)__double2hiint(x) & 0x7ff00000u, ey = (uint32_t)__double2hiint(y) & 0x7ff00000u;
        if (ex - 0x00100000u >= 0x7fe00000u || ey - 0x00100000u >= 0x7fe00000u) return -1;
        return (int)((ex + ey - (2u << 20)) >> 25);
    }
    // The common start anchors from every thread's first products (their highest
    // limb, -1 for none). All threads call it, before the first add.
    __device__ __forceinline__ void open(const int (&limb)[K]) {
#pragma unroll
        for (int k = 0; k < K; k++) {
            const int m = __reduce_max_sync(0xffffffffu, limb[k]);
            if ((threadIdx.x & 31) == 0) atomicMax(&amax[k], m);
        }
        __syncthreads();
#pragma unroll
        for (int k = 0; k < K; k++)
            if (amax[k] >= 0) a[k] = max(amax[k] - ANCHOR, 0);
    }
    // One thread's window (column w, anchor a) into the block accumulator sk, with
    // its own atomics; words back to nothing.
    static __device__ __forceinline__ void flush_column(uint32_t *w, unsigned long long *sk, int a) {
        for (int j = 0; j < W; j++) {
            const long long d = (long long)w[j * NT] - (SPLIT ? (long long)w[(W + j) * NT] : (long long)ZERO);
            w[j * NT] = ZERO;
            if (SPLIT) w[(W + j) * NT] = ZERO;
            if (d) sacc_add(&sk[a + j], d);
        }
    }
    // A carry (or, with down, a borrow) into word j of a set of words p, or past
    // the window's top into the block accumulator (neg: of the negative words).
    static __device__ __forceinline__ void ripple(uint32_t *p, unsigned long long *sk, int a, int j, bool down, bool neg) {
        for (; j < W; j++) {
            const uint32_t v = p[j * NT];
            p[j * NT] = down ? v - 1u : v + 1u;
            if (v != (down ? 0u : 0xffffffffu)) return;
        }
        if (a + W < NL) sacc_add(&sk[a + W], down || neg ? -1ll : 1ll);
    }
    // Products of any kind: zeros, subnormals and non-finite operands, products in
    // the window, below it (into the block accumulator) and above it (flush and
    // re-anchor). v: x and y of each in turn. Returns the thread's anchor.
    template <class... D>
    static __device__ __noinline__ int add_any(uint32_t *w, unsigned long long *sk, uint32_t *fl, int a, D... v) {
        // (SPLIT: one copy of the code, the products moving up in turn. Unrolled, the
        // call took registers that the caller's loads in flight need)
        constexpr int AHEAD = SPLIT ? 1 : 8;
        double xy[] = {v...};
#pragma unroll AHEAD
        for (int i = 0; i < (int)sizeof...(D); i += 2) {
            const double x = xy[0], y = xy[1];
#pragma unroll
            for (int k = 2; k < (int)sizeof...(D); k++) xy[k - 2] = xy[k];
            uint32_t u[5], m, f = 0u;
            int L;
            if (!prod_exact(x, y, f, u, L, m)) {
                if (f && (*(volatile uint32_t *)fl & f) != f) atomicOr(fl, f);
                continue;
            }
            if (L < a) {
                if (SPLIT) smem_deposit_ahead(sk, u, L, m);
                else smem_deposit(sk, u, L, m);
                continue;
            }
            if (L - a > QMAX) {
                int top = L;
                if (SPLIT || a >= 0) flush_column(w, sk, a);
                if (a <= 0) {
                    const int m = (int)__reduce_max_sync(__activemask(), (unsigned)L);
                    if (m - L <= ANCHOR) top = m;
                }
                a = top > ANCHOR ? top - ANCHOR : 0;
            }
            uint32_t *p = w + (SPLIT && m ? W * NT : 0);
            const uint32_t inv = SPLIT ? 0u : m;
            unsigned long long t = inv & 1u;
            for (int j = 0; j < 5; j++) {
                t += (unsigned long long)p[(L - a + j) * NT] + (u[j] ^ inv);
                p[(L - a + j) * NT] = (uint32_t)t;
                t >>= 32;
            }
            if ((uint32_t)t != (inv & 1u)) ripple(p, sk, a, L - a + 5, inv != 0u, m != 0u);
        }
        return a;
    }
    // The carries and borrows out of the five words of add()'s products (rare):
    // bit i of `out` for product i, its sign at bit 16 + i, its placement in byte
    // i of qs (at most four products).
    static __device__ __noinline__ void ripples(uint32_t *w, unsigned long long *sk, int a, uint32_t out, uint32_t qs) {
        for (int i = 0; i < 4; i++) {
            const int q = (int)(qs >> 8 * i) & 255;
            const bool neg = ((out >> (16 + i)) & 1u) != 0u;
            if (((out >> i) & 1u) && q <= QMAX) ripple(w + (SPLIT && neg ? W * NT : 0), sk, a, q + 5, !SPLIT && neg, neg);
        }
    }
    // N products into window k. One branch for all of them: when every operand
    // is normal and every product lands in the window (nearly always), straight
    // code. Otherwise zero products are sent to five words that nobody reads, and
    // any other kind sends all N through add_any(). N is 1, 2 or 4.
    // WARP: all 32 lanes call it and take the branch together if one of them has to.
    // Lanes that went out of line while the others ran the straight code cost the
    // warp both: 2^24 products of which one in a hundred lies 2^400 below the rest
    // 205 us, 98 so; exponents of -200 .. 200 331, 146.
    template <int N, bool SQ = false, bool WARP = false>
    __device__ __forceinline__ void add(int k, const double (&x)[N], const double (&y)[N]) {
        uint32_t xh[N], yh[N], e[N], q[N];
        uint32_t *wk = win + k * PER * NT;
        bool plain;  // every operand normal, every product in the window
        if constexpr (SPLIT) {
            // e: bit position above the window's lowest << 20, modulo 2^32, which holds
            // every position: one subtraction for the placement, the shift and the test
            uint32_t odd = 0u, far = 0u;
            const uint32_t base = ((uint32_t)a[k] << 25) + (2u << 20);
#pragma unroll
            for (int i = 0; i < N; i++) {
                xh[i] = (uint32_t)__double2hiint(x[i]);
                yh[i] = (uint32_t)__double2hiint(y[i]);
                const uint32_t ex = xh[i] & 0x7ff00000u, ey = yh[i] & 0x7ff00000u;
                odd = max(max(odd, ex - 0x00100000u), ey - 0x00100000u);
                e[i] = ex + ey - base;
                q[i] = e[i] >> 25;
                far = max(far, e[i]);
            }
            plain = odd < 0x7fe00000u && far < (QMAX + 1u) << 25;
        } else {
            uint32_t odd = 0u, far = 0u;
#pragma unroll
            for (int i = 0; i < N; i++) {
                xh[i] = (uint32_t)__double2hiint(x[i]);
                yh[i] = (uint32_t)__double2hiint(y[i]);
                const uint32_t ex = xh[i] & 0x7ff00000u, ey = yh[i] & 0x7ff00000u;
                odd = max(max(odd, ex - 0x00100000u), ey - 0x00100000u);
                e[i] = ex + ey - (2u << 20);  // bit position << 20; garbage for an odd operand
                q[i] = (e[i] >> 25) - (uint32_t)a[k];
                far = max(far, q[i]);
            }
            plain = odd < 0x7fe00000u && far <= (uint32_t)QMAX;
        }
        bool go = true;
        if (WARP ? __any_sync(0xffffffffu, !plain) : !plain) {
            bool some = !WARP;  // a product that is not zero
#pragma unroll
            for (int i = 0; i < N; i++) {
                const uint32_t ex = xh[i] & 0x7ff00000u, ey = yh[i] & 0x7ff00000u;
                const uint32_t zx = (xh[i] & 0x7fffffffu) | (uint32_t)__double2loint(x[i]);
                const uint32_t zy = (yh[i] & 0x7fffffffu) | (uint32_t)__double2loint(y[i]);
                if (min(zx, zy) == 0u && max(ex, ey) < 0x7ff00000u) {
                    q[i] = (uint32_t)(ROWS - k * PER);
                    xh[i] = yh[i];
                } else {
                    some = true;
                    go = go && max(ex - 0x00100000u, ey - 0x00100000u) < 0x7fe00000u && q[i] <= (uint32_t)QMAX;
                }
            }
            if (WARP) go = !__any_sync(0xffffffffu, !go);
            if (!go) {
                if constexpr (N == 1)
                    a[k] = add_any(wk, sacc[k], &sflags[k], a[k], x[0], y[0]);
                else if constexpr (N == 2)
                    a[k] = add_any(wk, sacc[k], &sflags[k], a[k], x[0], y[0], x[1], y[1]);
                else
                    a[k] = add_any(wk, sacc[k], &sflags[k], a[k], x[0], y[0], x[1], y[1], x[2], y[2], x[3], y[3]);
            } else {
                go = some;
            }
        }
        if (go) {
            uint32_t out = 0u;
#pragma unroll
            for (int i = 0; i < N; i++) {
                const uint32_t xl = (uint32_t)__double2loint(x[i]), yl = (uint32_t)__double2loint(y[i]);
                const uint32_t A1 = (xh[i] & 0xfffffu) | 0x100000u, B1 = (yh[i] & 0xfffffu) | 0x100000u;
                // 106-bit significand product: the two middle terms share one 64-bit sum (< 2^54)
                const unsigned long long lo = (unsigned long long)xl * yl, hi = (unsigned long long)A1 * B1;
                const unsigned long long mid = (unsigned long long)xl * B1 + (unsigned long long)A1 * yl;
                uint32_t p0 = (uint32_t)lo, p1, p2, p3, u[5], c;
                asm("add.cc.u32 %0, %3, %4;\n\t"
                    "addc.cc.u32 %1, %5, %6;\n\t"
                    "addc.u32 %2, %7, 0;"
                    : "=&r"(p1), "=&r"(p2), "=r"(p3)
                    : "r"((uint32_t)(lo >> 32)), "r"((uint32_t)mid), "r"((uint32_t)hi), "r"((uint32_t)(mid >> 32)),
                      "r"((uint32_t)(hi >> 32)));
                // complement of a negative product (before the shift, which fills with it)
                const uint32_t m = SPLIT || SQ ? 0u : (uint32_t)((int32_t)(xh[i] ^ yh[i]) >> 31);
                if (!SPLIT && !SQ) {
                    p0 ^= m;
                    p1 ^= m;
                    p2 ^= m;
                    p3 ^= m;
                }
                const uint32_t r = e[i] >> 20;  // the funnel shifts take it modulo 32
                u[0] = __funnelshift_l(m, p0, r);
                u[1] = __funnelshift_l(p0, p1, r);
                u[2] = __funnelshift_l(p1, p2, r);
                u[3] = __funnelshift_l(p2, p3, r);
                u[4] = __funnelshift_l(p3, m, r);
                uint32_t *p = wk + q[i] * NT + (SPLIT && !SQ ? ((xh[i] ^ yh[i]) >> 31) * (W * NT) : 0u);
                uint32_t w0 = p[0], w1 = p[NT], w2 = p[2 * NT], w3 = p[3 * NT], w4 = p[4 * NT];
                if (SPLIT || SQ) {
                    asm("add.cc.u32 %0, %0, %6;\n\t"
                        "addc.cc.u32 %1, %1, %7;\n\t"
                        "addc.cc.u32 %2, %2, %8;\n\t"
                        "addc.cc.u32 %3, %3, %9;\n\t"
                        "addc.cc.u32 %4, %4, %10;\n\t"
                        "addc.u32 %5, 0, 0;"
                        : "+r"(w0), "+r"(w1), "+r"(w2), "+r"(w3), "+r"(w4), "=r"(c)
                        : "r"(u[0]), "r"(u[1]), "r"(u[2]), "r"(u[3]), "r"(u[4]));
                } else {
                    // 1 carried in with a complement; out: 1 if a carry (positive) or a
                    // borrow (negative: no carry) leaves the five words
                    asm("{\n\t.reg .u32 t;\n\t"
                        "add.cc.u32 t, %11, %11;\n\t"
                        "addc.cc.u32 %0, %0, %6;\n\t"
                        "addc.cc.u32 %1, %1, %7;\n\t"
                        "addc.cc.u32 %2, %2, %8;\n\t"
                        "addc.cc.u32 %3, %3, %9;\n\t"
                        "addc.cc.u32 %4, %4, %10;\n\t"
                        "addc.u32 %5, %11, 0;\n\t}"
                        : "+r"(w0), "+r"(w1), "+r"(w2), "+r"(w3), "+r"(w4), "=&r"(c)
                        : "r"(u[0]), "r"(u[1]), "r"(u[2]), "r"(u[3]), "r"(u[4]), "r"(m));
                    // m + carry: 0 or 1 for a positive product, -1 (borrow) or 0 for a negative one
                    c &= 1u;
                }
                p[0] = w0;
                p[NT] = w1;
                p[2 * NT] = w2;
                p[3 * NT] = w3;
                p[4 * NT] = w4;
                out += c << i;
            }
            if (out) {
                uint32_t qs = 0u;
#pragma unroll
                for (int i = 0; i < N; i++) {
                    qs |= q[i] << 8 * i;
                    out |= (SQ ? 0u : (xh[i] ^ yh[i]) >> 31) << (16 + i);
                }
                ripples(wk, sacc[k], a[k], out, qs);
            }
        }
    }
    template <int N>
    __device__ __forceinline__ void add_sq(int k, const double (&x)[N]) {
        add<N, true>(k, x, x);
    }
    __device__ __forceinline__ void add(int k, double x, double y) {
        const double xv[1] = {x}, yv[1] = {y};
        add<1>(k, xv, yv);
    }
    __device__ __forceinline__ void add_sq(int k, double x) {
        const double xv[1] = {x};
        add_sq<1>(k, xv);
    }
    // Flush of every lane's window k at the end of the kernel (all 32 lanes call
    // it). With one anchor in the warp, lane r sums word r over the warp's
    // columns, each lane starting at its own column (32 banks, no conflicts); else
    // every lane flushes its own.
    __device__ __forceinline__ void flush_warp(int k) {
        constexpr unsigned FULL = 0xffffffffu;
        const int lane = threadIdx.x & 31;
        const int a0 = __shfl_sync(FULL, a[k], 0);
        uint32_t *wk = win + k * PER * NT;
        if (!__all_sync(FULL, a[k] == a0)) {
            if (a[k] >= 0) flush_column(wk, sacc[k], a[k]);
            return;
        }
        if (a0 < 0) return;
        __syncwarp();
        long long sum = SPLIT ? 0 : -32ll * ZERO;
        if (lane < PER) {
            const uint32_t *r = wk - lane + lane * NT;
#pragma unroll 8
            for (int i = 0; i < 32; i++) sum += (long long)r[(i + lane) & 31];
        }
        if (SPLIT) sum -= __shfl_down_sync(FULL, sum, W);
        if (lane < W && sum && a0 + lane < NL) sacc_add(&sacc[k][a0 + lane], sum);
    }
    // The K reductions from `slot` of g on, over nblk blocks (0: the grid); see
    // block_grid_finish.
    __device__ __forceinline__ bool finish(DotScratch *g, double *vals, unsigned nblk = 0u, int slot = 0,
                                           bool export_limbs = false, long long *limbs = nullptr,
                                           int32_t *fl = nullptr) {
#pragma unroll
        for (int k = 0; k < K; k++) flush_warp(k);
        const uint32_t none[K] = {};  // add_any() has set the block's flags itself
        return block_grid_finish<K>(none, sacc, sflags, g, vals, export_limbs, limbs, fl, nblk, slot);
    }
};

template <int K_>
struct PlainR {
    static constexpr int K = K_;
    static constexpr bool WINDOWS = false;
    double s[K];

    __device__ __forceinline__ void init() {
#pragma unroll
        for (int k = 0; k < K; k++) s[k] = 0.0;
        __syncthreads();  // as the exact reducers' init
    }
    __device__ __forceinline__ void add(int k, double x, double y) { s[k] = fma(x, y, s[k]); }
    __device__ __forceinline__ void add_sq(int k, double x) { s[k] = fma(x, x, s[k]); }
    template <int N>
    __device__ __forceinline__ void add(int k, const double (&x)[N], const double (&y)[N]) {
#pragma unroll
        for (int i = 0; i < N; i++) add(k, x[i], y[i]);
    }
    template <int N>
    __device__ __forceinline__ void add_sq(int k, const double (&x)[N]) {
#pragma unroll
        for (int i = 0; i < N; i++) add_sq(k, x[i]);
    }
    static __device__ __forceinline__ int limb_of(double, double) { return -1; }
    __device__ __forceinline__ void open(const int (&)[K]) {}
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

// Standalone kernels: exact dot (single and multi-output), long-accumulator
// export and rounding, the allocation-free exact dot, the FPE-8 dot.
#include <algorithm>
#include <mutex>

#include "kernels.cuh"
#include "launch.h"

namespace rbs {

struct DotArgs {
    const double *x[KMAX];
    const double *y[KMAX];
};

// Pairs of each operand that a thread loads at once, and blocks per SM to keep
// registers for. The loads in flight set the rate: two pairs at three blocks (80
// registers; one pair at four blocks, or two at four, were up to 5 % slower).
constexpr int EXDOT_PAIRS = 2, EXDOT_BLOCKS = 3;

// U pairs into the windows. WARP: every lane of the warp has them.
template <int U, bool WARP, class R>
__device__ __forceinline__ void add_pairs(R &red, const double2 (&x)[U], const double2 (&y)[U]) {
    double xv[2 * U], yv[2 * U];
#pragma unroll
    for (int u = 0; u < U; u++) {
        xv[2 * u] = x[u].x;
        xv[2 * u + 1] = x[u].y;
        yv[2 * u] = y[u].x;
        yv[2 * u + 1] = y[u].y;
    }
    red.template add<2 * U, false, WARP>(0, xv, yv);
}

// Exact dots over the same length (Sec. 2 exdot; Sec. 4.1/4.2 merged
// reductions): the blocks of row blockIdx.y take dot blockIdx.y, W the words
// per sign of their windows. Aligned operands go through 16-byte loads, the
// next pairs in flight while these are added, so that the stream does not stop
// for the products.
//
// Several dots share the launch but not their blocks: five dots' windows in one
// thread left two blocks per SM, and issue slots empty (2 million elements: 41
// us against 29 now); an operand that several dots name comes from L2 for all
// but the first of them, since their blocks walk the vectors together.
// Bound by HBM once long (2^27, cond 1: 311 us, the copy rate; 378 with 64-bit
// digits), with the integer pipe where signs and exponents mix (cond 1e16 to 1e48: 347
// us), and by the windows' set-up, flush and cross-block sum when short (2^24: 44 us,
// 39.5 of them HBM's; cond 1e48: 50 against 73).
template <int W, bool EXPORT>
__global__ void __launch_bounds__(256, EXDOT_BLOCKS)
    k_exdot(const __grid_constant__ DotArgs a, int64_t n, DotScratch *g, double *out, long long *limbs, int32_t *flags_out) {
    using R = ExactRows<1, W, true>;
    R red;
    const int slot = EXPORT ? 0 : blockIdx.y;
    const double *xp = a.x[slot], *yp = a.y[slot];
    red.init();
    chain_wait();
    const int64_t st = gstride();
    if (((reinterpret_cast<uintptr_t>(xp) | reinterpret_cast<uintptr_t>(yp)) & 15) == 0) {
        constexpr int U = EXDOT_PAIRS;
        const double2 *x2 = reinterpret_cast<const double2 *>(xp), *y2 = reinterpret_cast<const double2 *>(yp);
        const int64_t n2 = n >> 1;
        // the pair that opens the windows; a thread without one adds zeros
        double2 x0[1] = {make_double2(0.0, 0.0)}, y0[1] = {make_double2(0.0, 0.0)};
        if (gtid() < n2) {
            x0[0] = __ldcs(x2 + gtid());
            y0[0] = __ldcs(y2 + gtid());
        }
        // then `full` steps of U pairs per thread, two steps per turn of the
        // loop with the loads of each ahead of the adds of the other; the same two
        // copies of the code for the last steps (a short dot meets every copy cold:
        // with three more 2^20 took 8.1 us on the device, 7.8 so), and the pairs left
        // over at the end (taken first, values that rise along the vectors would all
        // fall below their windows). A thread has at most 2^20 products: counted in 32
        // bits, whose registers the loads in flight can use (2^27, cond 1e16: 372 -> 365
        // us; with the operands' exponents tested one by one 347).
        const int full = n2 > st ? (int)((n2 - st) / (U * st)) : 0;
        double2 xa[U], ya[U], xb[U], yb[U];
        const double2 *xq = x2 + gtid() + st, *yq = y2 + gtid() + st;
        auto load = [&](double2 (&xv)[U], double2 (&yv)[U]) {
#pragma unroll
            for (int u = 0; u < U; u++) {
                xv[u] = __ldcs(xq);
                yv[u] = __ldcs(yq);
                xq += st;
                yq += st;
            }
        };
        if (full > 0) load(xa, ya);
        red.open({max(R::limb_of(x0[0].x, y0[0].x), R::limb_of(x0[0].y, y0[0].y))});
        add_pairs<1, false>(red, x0, y0);
        for (int s = 0; s < full; s += 2) {
            if (s + 1 < full) load(xb, yb);
            add_pairs<U, true>(red, xa, ya);
            if (s + 1 >= full) break;
            if (s + 2 < full) load(xa, ya);
            add_pairs<U, true>(red, xb, yb);
        }
        for (int64_t j = gtid() + st + full * (U * st); j < n2; j += st) {
            x0[0] = __ldcs(x2 + j);
            y0[0] = __ldcs(y2 + j);
            add_pairs<1, false>(red, x0, y0);
        }
        if ((n & 1) && gtid() == 0) red.add(0, xp[n - 1], yp[n - 1]);
    } else {
        int64_t i = gtid();
        red.open({i < n ? R::limb_of(xp[i], yp[i]) : -1});
        for (; i < n; i += st) red.add(0, xp[i], yp[i]);
    }
    __shared__ double val[1];
    if (red.finish(g, val, 0u, slot, EXPORT, limbs, flags_out) && !EXPORT && threadIdx.x == 0) out[slot] = val[0];
}

// Words per sign for the "exdot.window" knob: 16 unless it asks for a small
// window (1 or 2). 12 placements hold the products from 2^-256 below to 2^96 above
// the largest of a block's first ones without re-anchoring.
template <class F>
static auto with_window(int window, F &&f) {
    if (window == 1) return f(k_exdot<6, false>);
    if (window == 2) return f(k_exdot<7, false>);
    return f(k_exdot<16, false>);
}

int exdot_blocks_per_sm(int window, int block) {
    static QueryCache<std::pair<int, int>> cache;
    return cache.get({window, block}, [&] {
        return with_window(window, [&](auto kern) {
            int v = 0;
            if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&v, kern, block, 0) != cudaSuccess || v < 1) {
                cudaGetLastError();
                v = 1;
            }
            return v;
        });
    });
}

cudaError_t launch_exdot(int k, const double *const *xs, const double *const *ys, int64_t n,
                         DotScratch *g, double *out, int window, Cfg cfg, cudaStream_t s) {
    if (k < 1 || k > KMAX) return cudaErrorInvalidValue;
    DotArgs a{};
    for (int j = 0; j < k; j++) {
        a.x[j] = xs[j];
        a.y[j] = ys[j];
    }
    return with_window(window, [&](auto kern) {
        return launch_chained(kern, dim3((unsigned)cfg.grid, (unsigned)k), cfg.block, s, a, n, g, out,
                              (long long *)nullptr, (int32_t *)nullptr);
    });
}

cudaError_t launch_exdot_partial(const double *x, const double *y, int64_t n, DotScratch *g,
                                 int64_t *limbs, int32_t *flags, Cfg cfg, cudaStream_t s) {
    DotArgs a{};
    a.x[0] = x;
    a.y[0] = y;
    return launch_chained(k_exdot<16, true>, dim3((unsigned)cfg.grid), cfg.block, s, a, n, g, (double *)nullptr,
                          (long long *)limbs, flags);
}

__global__ void k_round_limbs(const int64_t *limbs, const int32_t *flags, double *out) {
    __shared__ long long G[NL];
    for (int j = threadIdx.x; j < NL; j += blockDim.x) G[j] = (long long)limbs[j];
    __syncthreads();
    if (threadIdx.x == 0) *out = round_limbs_thread(G, (uint32_t)*flags);
}

cudaError_t launch_round_limbs(const int64_t *limbs, const int32_t *flags, double *out, cudaStream_t s) {
    k_round_limbs<<<1, 160, 0, s>>>(limbs, flags, out);
    return cudaGetLastError();
}

}  // namespace rbs

// ---- allocation-free exact dot ---------------------------------------------------
//
// rbs_exdot_noalloc runs the same exact-dot kernel as rbs_exdot_multi, but keeps
// its only scratch -- the cross-block long accumulators, flags and ticket --
// in the file-scope device array below instead of the per-stream workspace, so
// it never allocates device or pinned host memory. It serves callers that
// cannot allocate at the point of the call: code running while a CUDA graph is
// being captured (a cudaMalloc is not a capturable step), latency-critical
// loops that cannot afford the implicit device synchronisation of an
// allocation, and applications whose own memory pool owns the device memory.
//
// The array is 8 KiB and holds at most RBS_NOALLOC_MAX_DOTS accumulators.
// Every GPU that loads this library keeps the array until the process exits.
// All calls on a device share it, so calls that overlap on the GPU (for
// example on two streams at once) race and must be ordered by the caller.
namespace rbs {
namespace {

constexpr size_t NOALLOC_BYTES = 8192;
static_assert(sizeof(DotScratch) <= NOALLOC_BYTES, "scratch array too small");
static_assert(RBS_NOALLOC_MAX_DOTS == KMAX, "accumulator count");

static __device__ __align__(256) unsigned char noalloc_scratch[NOALLOC_BYTES];

constexpr int NOALLOC_MAX_DEVICES = 64;
std::mutex noalloc_mu;
void *noalloc_ptr[NOALLOC_MAX_DEVICES];
int noalloc_sms[NOALLOC_MAX_DEVICES];

// Set-up, once per device, with that device current: the array's device
// address (in host code its name is only a host-side stand-in), a one-time
// clear, and the SM count for the launch shape.
int noalloc_setup(int dev, void **ptr, int *sms) {
    std::lock_guard<std::mutex> lk(noalloc_mu);
    if (!noalloc_ptr[dev]) {
        void *p = nullptr;
        cudaError_t e = cudaGetSymbolAddress(&p, noalloc_scratch);
        if (e != cudaSuccess) return set_error(RBS_ECUDA, "cudaGetSymbolAddress of the no-alloc scratch failed");
        int n = 0;
        e = cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev);
        if (e != cudaSuccess) return set_error(RBS_ECUDA, "cudaDeviceGetAttribute failed");
        e = cudaMemset(p, 0, NOALLOC_BYTES);
        if (e == cudaSuccess) e = cudaDeviceSynchronize();
        if (e != cudaSuccess) return set_error(RBS_ECUDA, "clearing the no-alloc scratch failed");
        noalloc_sms[dev] = n;
        noalloc_ptr[dev] = p;
    }
    *ptr = noalloc_ptr[dev];
    *sms = noalloc_sms[dev];
    return RBS_OK;
}

bool device_resident(const void *p) {
    cudaPointerAttributes a;
    if (cudaPointerGetAttributes(&a, p) != cudaSuccess) {
        cudaGetLastError();
        return false;
    }
    return a.type == cudaMemoryTypeDevice || a.type == cudaMemoryTypeManaged;
}

}  // namespace
}  // namespace rbs

extern "C" int rbs_exdot_noalloc(int k, const double *const *xs, const double *const *ys, int64_t n,
                                 double *out, void *stream) {
    using namespace rbs;
    if (k < 1 || k > RBS_NOALLOC_MAX_DOTS)
        return set_error(RBS_EINVAL, "rbs_exdot_noalloc: k must be 1..RBS_NOALLOC_MAX_DOTS (6), the "
                                     "accumulators its fixed scratch array holds");
    if (n < 0 || !xs || !ys || !out) return set_error(RBS_EINVAL, "rbs_exdot_noalloc: bad argument");
    if (!device_resident(out)) return set_error(RBS_EINVAL, "rbs_exdot_noalloc: out must be device memory");
    for (int j = 0; j < k; j++)
        if (n > 0 && (!xs[j] || !ys[j] || !device_resident(xs[j]) || !device_resident(ys[j])))
            return set_error(RBS_EINVAL, "rbs_exdot_noalloc: operands must be device memory");
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= NOALLOC_MAX_DEVICES)
        return set_error(RBS_ECUDA, "rbs_exdot_noalloc: no usable current device");
    void *p = nullptr;
    int sms = 0;
    int rc = noalloc_setup(dev, &p, &sms);
    if (rc) return rc;
    cudaStream_t s = (cudaStream_t)stream;
    // the shared array keeps the last call's contents: clear it first
    if (cudaMemsetAsync(p, 0, sizeof(DotScratch), s) != cudaSuccess)
        return set_error(RBS_ECUDA, "rbs_exdot_noalloc: cudaMemsetAsync failed");
    if (n == 0) {
        if (cudaMemsetAsync(out, 0, k * sizeof(double), s) != cudaSuccess)
            return set_error(RBS_ECUDA, "rbs_exdot_noalloc: cudaMemsetAsync failed");
        return RBS_OK;
    }
    Cfg c;
    c.block = 256;
    int64_t g = (n + 2LL * c.block - 1) / (2LL * c.block);
    const int64_t cap = std::max<int64_t>((int64_t)sms * exdot_blocks_per_sm(0, c.block) / k, 1);  // whole waves
    g = g < 1 ? 1 : (g < cap ? g : cap);
    const int64_t minimum = (n + ((int64_t)c.block << 20) - 1) / ((int64_t)c.block << 20);
    if (g < minimum) g = minimum;
    c.grid = (int)(g > 0x7fffffff ? 0x7fffffff : g);
    cudaError_t e = launch_exdot(k, xs, ys, n, reinterpret_cast<DotScratch *>(p), out, 0, c, s);
    if (e != cudaSuccess) return set_error(RBS_ECUDA, "rbs_exdot_noalloc: kernel launch failed");
    return RBS_OK;
}

// ---- lightweight FPE-8 dot (Sec. 3.2) -----------------------------------------------
//
// The paper's lightweight variant: each thread keeps a floating-point
// expansion of at most eight binary64 terms. A product enters as TwoProd's
// r + s (Alg. 2) and each part is added with a cascade of TwoSums (Alg. 1)
// that stops as soon as the carried error is zero (early exit). Where the
// paper rounds the final expansion with NearSum, the terms here go into the
// exact integer accumulator and are rounded once: the same correctly rounded
// value. When a thread would need a ninth term, a TwoProd may be inexact
// (|x*y| below 2^-969, where its error can underflow) or a value is not
// finite, the kernel reports that information could be lost -- the paper's
// warning -- and the entry point falls back to the exact dot.
namespace rbs {

__device__ __forceinline__ void fpe_two_sum(double a, double b, double &r, double &s) {
    r = __dadd_rn(a, b);
    const double z = __dsub_rn(r, a);
    s = __dadd_rn(__dsub_rn(a, __dsub_rn(r, z)), __dsub_rn(b, z));
}

// c += x exactly while at most 8 terms are needed; false if a ninth is needed.
__device__ __forceinline__ bool fpe_add(double (&c)[8], double x) {
#pragma unroll
    for (int k = 0; k < 8; k++) {
        if (x == 0.0) return true;
        double r, s;
        fpe_two_sum(c[k], x, r, s);
        c[k] = r;
        x = s;
    }
    return x == 0.0;
}

__global__ void __launch_bounds__(256) k_fpe_dot(const double *__restrict__ x, const double *__restrict__ y,
                                                 int64_t n, DotScratch *g, double *out, unsigned *lost) {
    ExactR<1, 4> red;
    red.init();
    double c[8];
#pragma unroll
    for (int k = 0; k < 8; k++) c[k] = 0.0;
    bool ok = true;
    for (int64_t i = gtid(); i < n; i += gstride()) {
        const double a = x[i], b = y[i];
        const double r = __dmul_rn(a, b);
        const double s = fma(a, b, -r);
        const double ar = fabs(r);
        if (!finite_d(r) || (ar < 0x1p-969 && (r != 0.0 || (a != 0.0 && b != 0.0)))) {
            ok = false;
            continue;
        }
        ok = fpe_add(c, r) && ok;
        ok = fpe_add(c, s) && ok;
    }
#pragma unroll
    for (int k = 0; k < 8; k++) {
        if (!finite_d(c[k])) ok = false;
        else red.add(0, c[k], 1.0);
    }
    if (!ok) atomicOr(lost, 1u);
    __shared__ double vals[1];
    if (red.finish(g, vals) && threadIdx.x == 0) *out = vals[0];
}

int fpe_blocks_per_sm(int block) {
    int nb = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, k_fpe_dot, block, 0) != cudaSuccess || nb < 1) {
        cudaGetLastError();
        nb = 1;
    }
    return nb;
}

cudaError_t launch_fpe_dot(const double *x, const double *y, int64_t n, DotScratch *g, double *out,
                           unsigned *lost, Cfg cfg, cudaStream_t s) {
    k_fpe_dot<<<cfg.grid, cfg.block, 0, s>>>(x, y, n, g, out, lost);
    return cudaGetLastError();
}

}  // namespace rbs

// Standalone SpMV kernels (short rows warp-staged, long rows register-staged,
// one thread per row), Jacobi and the CSR structure check.
#include <mutex>
#include <tuple>

#include "kernels.cuh"
#include "launch.h"

namespace rbs {

// y = A x (Sec. 4.1), warp-staged short rows or, in mode 1, one thread per row
// in a grid-stride loop. CHECKED: every index is range-checked (the
// standalone product); without it the solver has validated the structure at
// set-up. With a solver state, the kernel is a no-op once the solver stopped.
template <bool CHECKED>
__global__ void __launch_bounds__(256, 3)
    k_spmv(CSRView A, const double *__restrict__ x, double *__restrict__ y, const SolverState *st, unsigned *err,
           int mode) {
    chain_wait();
    if (st && st->done) return;
    unsigned eb = 0u;
    spmv_each<CHECKED, SPMV_CAP_SHORT>(A, x, nullptr, mode, eb, [&](int64_t i, double v, double) { y[i] = v; });
    if (eb) atomicOr(err, eb);
}

// y = A x for long rows (mode 3): register-staged chunks (spmv_rows_reg) in
// 4-warp blocks, three resident per SM.
template <bool CHECKED>
__global__ void __launch_bounds__(SPMV_REG_WARPS * 32, 3)
    k_spmv_reg(CSRView A, const double *__restrict__ x, double *__restrict__ y, const SolverState *st,
               unsigned *err, int mode) {
    chain_wait();
    if (st && st->done) return;
    unsigned eb = 0u;
    spmv_rows_reg<CHECKED, SPMV_CAP_LONG, false>(
        A, 0, A.n, (int64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5), (int64_t)gridDim.x * (blockDim.x >> 5),
        x, nullptr, true, (mode & SPMV_TEST_STALL) != 0, eb, [&](int64_t i, double v, double) { y[i] = v; });
    if (eb) atomicOr(err, eb);
}

// y = A x for a matrix laid out by its diagonals (a solver's product).
template <int N>
__global__ void __launch_bounds__(DiagLayout<N>::WARPS * 32, 3)
    k_spmv_diag(CSRView A, const __grid_constant__ DiagArgs D, const double *x, double *y,
                const SolverState *st, unsigned *err, int mode) {
    chain_wait();
    if (st->done) return;
    unsigned eb = 0u;
    spmv_grid_diag<N>(A, D, x, nullptr, (mode & SPMV_TEST_STALL) != 0, eb,
                      [&](int64_t i, double v, double) { y[i] = v; });
    if (eb) atomicOr(err, eb);
}

static CSRView view(const CSRArgs &A) { return CSRView{A.n, A.nnz, A.rowptr, A.col, A.val}; }

static void spmv_carveout(int c) {
    static std::mutex mu;
    static int applied[64];
    static bool init = false;
    std::lock_guard<std::mutex> lk(mu);
    if (!init) {
        for (int i = 0; i < 64; i++) applied[i] = -2;
        init = true;
    }
    int dev = 0;
    if (cudaGetDevice(&dev) == cudaSuccess && dev >= 0 && dev < 64 && applied[dev] != c) {
        const int short_c = c > SPMV_SHORT_CARVEOUT ? SPMV_SHORT_CARVEOUT : c;
        cudaFuncSetAttribute(k_spmv<true>, cudaFuncAttributePreferredSharedMemoryCarveout, short_c);
        cudaFuncSetAttribute(k_spmv<false>, cudaFuncAttributePreferredSharedMemoryCarveout, short_c);
        cudaFuncSetAttribute(k_spmv_diag<7>, cudaFuncAttributePreferredSharedMemoryCarveout, c);
        // the kernels of long rows: what their blocks need, whatever the knob says
        cudaFuncSetAttribute(k_spmv_diag<32>, cudaFuncAttributePreferredSharedMemoryCarveout, -1);
        cudaFuncSetAttribute(k_spmv_reg<true>, cudaFuncAttributePreferredSharedMemoryCarveout, -1);
        cudaFuncSetAttribute(k_spmv_reg<false>, cudaFuncAttributePreferredSharedMemoryCarveout, -1);
        cudaGetLastError();
        applied[dev] = c;
    }
}

// Resident blocks per SM of the SpMV kernel of `mode` at this block size (the
// long-row kernel: at its own block of SPMV_REG_WARPS warps).
int spmv_blocks_per_sm(int block, int carveout, int mode) {
    static QueryCache<std::tuple<int, int, int>> cache;
    return cache.get({block, carveout, mode}, [&] {
        spmv_carveout(carveout);
        int nb = 0;
        const cudaError_t e =
            mode == SPMV_MODE_DIAG7    ? cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, k_spmv_diag<7>, block, 0)
            : mode == SPMV_MODE_DIAG32 ? cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, k_spmv_diag<32>, block, 0)
            : mode == SPMV_MODE_LONG
                ? cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, k_spmv_reg<true>, SPMV_REG_WARPS * 32, 0)
                : cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, k_spmv<true>, block, 0);
        if (e != cudaSuccess || nb < 1) {
            cudaGetLastError();
            nb = 1;
        }
        return nb;
    });
}

// The long-row kernel runs its own launch shape: blocks of SPMV_REG_WARPS
// warps, all of them resident (cfg's grid and block are not used).
static Cfg spmv_reg_cfg(int64_t n, int carveout) {
    static std::mutex mu;
    static int sms[64], bps[64];
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) dev = 0;
    int nsm, nb;
    {
        std::lock_guard<std::mutex> lk(mu);
        if (!sms[dev]) {
            int v = 0;
            if (cudaDeviceGetAttribute(&v, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || v < 1) {
                cudaGetLastError();
                v = 1;
            }
            bps[dev] = spmv_blocks_per_sm(SPMV_REG_WARPS * 32, carveout, SPMV_MODE_LONG);
            sms[dev] = v;
        }
        nsm = sms[dev];
        nb = bps[dev];
    }
    Cfg c;
    c.block = SPMV_REG_WARPS * 32;
    const int64_t need = (n + c.block - 1) / c.block, cap = (int64_t)nsm * nb;
    c.grid = (int)(need < 1 ? 1 : (need < cap ? need : cap));
    return c;
}

cudaError_t launch_spmv(const CSRArgs &A, const double *x, double *y, const SolverState *st,
                        unsigned *err, Cfg cfg, cudaStream_t s) {
    spmv_carveout(cfg.carveout);
    if ((cfg.mode & SPMV_MODE_MASK) == SPMV_MODE_LONG) {
        const Cfg r = spmv_reg_cfg(A.n, cfg.carveout);
        return launch_chained(st ? k_spmv_reg<false> : k_spmv_reg<true>, dim3((unsigned)r.grid), r.block, s, view(A), x,
                              y, st, err, cfg.mode);
    }
    return launch_chained(st ? k_spmv<false> : k_spmv<true>, dim3((unsigned)cfg.grid),
                          cfg.block, s, view(A), x, y, st, err, cfg.mode);
}

cudaError_t launch_spmv_diag(const CSRArgs &A, const DiagArgs &D, const double *x, double *y, const SolverState *st,
                             unsigned *err, Cfg cfg, cudaStream_t s) {
    spmv_carveout(cfg.carveout);
    const auto kern = (cfg.mode & SPMV_MODE_MASK) == SPMV_MODE_DIAG32 ? k_spmv_diag<32> : k_spmv_diag<7>;
    return launch_chained(kern, dim3((unsigned)cfg.grid), cfg.block, s, view(A), D, x, y, st, err, cfg.mode);
}

// invd_i = RN(1 / d_i) with d the given diagonal or the first stored (i, i)
// entry (Sec. 4, Jacobi M = diag(A)); a zero, NaN or missing entry sets err bit 2.
__global__ void __launch_bounds__(256) k_jacobi_invd(CSRView A, const double *diag, double *invd, unsigned *err) {
    bool bad = false, idx_bad = false;
    for (int64_t i = gtid(); i < A.n; i += gstride()) {
        double d = 0.0;
        bool found = false;
        if (diag) {
            d = diag[i];
            found = true;
        } else {
            const int64_t b = A.rowptr[i], e = A.rowptr[i + 1];
            if (b < 0 || e < b || e > A.nnz) {
                idx_bad = true;
            } else {
                for (int64_t k = b; k < e; k++)
                    if ((int64_t)A.col[k] == i) {
                        d = A.val[k];
                        found = true;
                        break;
                    }
            }
        }
        if (!found || d == 0.0 || d != d) {
            bad = true;
            invd[i] = 0.0;
        } else {
            invd[i] = __ddiv_rn(1.0, d);
        }
    }
    if (bad) atomicOr(err, 2u);
    if (idx_bad) atomicOr(err, 1u);
}

cudaError_t launch_jacobi_invd(const CSRArgs &A, const double *diag, double *invd, unsigned *err, Cfg cfg,
                               cudaStream_t s) {
    k_jacobi_invd<<<cfg.grid, cfg.block, 0, s>>>(view(A), diag, invd, err);
    return cudaGetLastError();
}

__global__ void __launch_bounds__(256) k_jacobi_apply(int64_t n, const double *invd, const double *p,
                                                     double *phat) {
    for (int64_t i = gtid(); i < n; i += gstride()) phat[i] = __dmul_rn(p[i], invd[i]);
}

cudaError_t launch_jacobi_apply(int64_t n, const double *invd, const double *p, double *phat, Cfg cfg,
                                cudaStream_t s) {
    k_jacobi_apply<<<cfg.grid, cfg.block, 0, s>>>(n, invd, p, phat);
    return cudaGetLastError();
}

__global__ void __launch_bounds__(256) k_diag_sample(CSRView A, DiagArgs *out) {
    const int m = sample_diags(A, SPMV_DIAGS, out->off);
    if (threadIdx.x == 0) out->m = m;
}

// One pass over the rows: the structure check of k_csr_check, the Jacobi inverse
// of k_jacobi_invd, and the diagonal layout for the sampled diagonals. Rows of
// a warp follow each other, so their column spans share cache lines. One pass
// instead of two saves 0.05 ms of the 0.69 ms set-up at 256^3, the layout
// included.
__global__ void __launch_bounds__(256) k_prepare(CSRView A, const double *diag, double *invd, const DiagArgs *diags,
                                                 uint32_t *mask, int64_t *base, unsigned *err) {
    __shared__ int s_off[SPMV_DIAGS + 1];
    const int m = diags->m;
    if (threadIdx.x <= SPMV_DIAGS) s_off[threadIdx.x] = (int)threadIdx.x < m ? diags->off[threadIdx.x] : 0x7fffffff;
    __syncthreads();
    unsigned eb = 0u;
    if (gtid() == 0 && (A.rowptr[0] != 0 || A.rowptr[A.n] != A.nnz)) eb |= 1u;
    const int64_t padded = (A.n + 31) / 32 * 32;
    for (int64_t i = gtid(); i < padded; i += gstride()) {
        uint32_t word = 0u;
        if (i < A.n) {
            const RowSetup r = check_row(A, i, diag, s_off, m, LONG_ROW);
            eb |= r.err;
            invd[i] = r.inv;
            if ((i & 31) == 0) base[i >> 5] = r.first;
            // up to 7 diagonals leave room for the row's place among its chunk's values
            word = r.word;
            if (m <= 7) word |= (uint32_t)(r.first - A.rowptr[i & ~31LL]) << 8;
        }
        if (m > 0) mask[i] = word;
    }
    // one atomic per warp and bit at most
    eb = __reduce_or_sync(__activemask(), eb);
    if (eb && (*(volatile unsigned *)err & eb) != eb) atomicOr(err, eb);
}

cudaError_t launch_prepare(const CSRArgs &A, const double *diag, double *invd, DiagArgs *diags, uint32_t *mask,
                           int64_t *base, unsigned *err, Cfg cfg, cudaStream_t s) {
    k_diag_sample<<<1, 256, 0, s>>>(view(A), diags);
    k_prepare<<<cfg.grid, cfg.block, 0, s>>>(view(A), diag, invd, diags, mask, base, err);
    return cudaGetLastError();
}

// CSR structure check: rowptr[0] == 0, non-decreasing, rowptr[n] == nnz,
// 0 <= col < n. Sets err bit 1 on any violation.
__global__ void __launch_bounds__(256) k_csr_check(CSRView A, unsigned *err) {
    bool bad = false;
    if (gtid() == 0 && (A.rowptr[0] != 0 || A.rowptr[A.n] != A.nnz)) bad = true;
    for (int64_t i = gtid(); i < A.n; i += gstride())
        if (A.rowptr[i + 1] < A.rowptr[i]) bad = true;
    for (int64_t k = gtid(); k < A.nnz; k += gstride())
        if ((uint64_t)(int64_t)A.col[k] >= (uint64_t)A.n) bad = true;
    if (bad) atomicOr(err, 1u);
}

cudaError_t launch_csr_check(const CSRArgs &A, unsigned *err, Cfg cfg, cudaStream_t s) {
    k_csr_check<<<cfg.grid, cfg.block, 0, s>>>(view(A), err);
    return cudaGetLastError();
}

}  // namespace rbs

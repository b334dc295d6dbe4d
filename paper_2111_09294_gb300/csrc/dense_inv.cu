// Batched in-place inversion of symmetric positive definite matrices in FP64
// by blocked symmetric sweeps (set-up only): the explicit inverses of the
// coarse matrix E = Z^T K Z (Section 3.2) and of the dense diagonal blocks of
// a block-Jacobi preconditioner (Section 3.4, Eqs. block_jacobi,
// block_jacobi_enr).
//
// The sweep on a pivot set P maps a symmetric A to B with
//   B_PP = -A_PP^-1,  B_QP = A_QP A_PP^-1,  B_PQ = A_PP^-1 A_PQ,
//   B_QQ = A_QQ - A_QP A_PP^-1 A_PQ,
// and after every index has been swept once the array holds -A^-1.  Pivot
// blocks of kNB indices are swept in order, all matrices at once.  Step k: the
// pivot block's own sweep (one CTA per matrix, pivots checked against a
// threshold), the column panel C = A_QP A_PP^-1, the trailing update A_QQ -= C
// A_PQ on the upper tiles (mirrored), and the write-back of the panel.  The
// trailing update carries the n^3 work as 64 x 64 x 64 FP64 tile products.
//
// The FP64 units bound it: k^3 / 2 FMA for E, 29 ms at k = 3150 by their rate
// (19 cycles per warp instruction and SM).  The pivot sweep is a chain on one
// SM (2 x 64^3 operations, 0.15 ms) that every step would wait for, so each
// step updates the tiles of the next pivot's row and column first and sweeps
// the next pivot block while the other tiles are updated: the pivot's CTA
// triggers the dependent launch of the first part of those tiles as it starts
// (and takes an SM to itself, by its shared memory, while there are few
// matrices), the panel of the second part.  k = 3150: 51.8 ms before (the
// steps' launches one after another, 0.36 ms per pivot block), 36.8 now; k =
// 426: 3.4 before, 2.3 now.
#include <algorithm>
#include <climits>

#include "cache.cuh"
#include "internal.h"
#include "pdl.cuh"

namespace xdcg {

constexpr int kNB = 64;                 // pivot block and tile edge
constexpr int kInvThreads = 256;        // 16 x 16 threads, 4 x 4 outputs each
constexpr int kLd = kNB + 1;            // padded shared-memory row

// tile index -> (matrix, tile row I, tile column J >= I) of the upper tiles
__device__ __forceinline__ int find_matrix(const int *prefix, int nMat, int t) {
    int lo = 0, hi = nMat - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (prefix[mid] <= t)
            lo = mid;
        else
            hi = mid - 1;
    }
    return lo;
}

// row-major element (i, j) of matrix m
__device__ __forceinline__ double *mat_at(const DenseBatch &B, int m, int i, int j) {
    return B.A + B.off[m] + (long long)i * B.dim[m] + j;
}

// out (64 x 16 CB, registers 4 x CB per thread) = X (64 x nb) * Y (nb x 16 CB),
// both in shared memory with row stride kLd
template <int CB>
__device__ __forceinline__ void tile_mm(const double *X, const double *Y, int nb,
                                        double (&acc)[4][CB]) {
    const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
    for (int kk = 0; kk < nb; ++kk) {
        double xa[4], yb[CB];
#pragma unroll
        for (int a = 0; a < 4; ++a) xa[a] = X[(ty + 16 * a) * kLd + kk];
#pragma unroll
        for (int b = 0; b < CB; ++b) yb[b] = Y[kk * kLd + tx + 16 * b];
#pragma unroll
        for (int a = 0; a < 4; ++a)
#pragma unroll
            for (int b = 0; b < CB; ++b) acc[a][b] = fma(xa[a], yb[b], acc[a][b]);
    }
}

// the swept pivot block and the panel of step k: two copies of each, step k + 1
// is prepared while step k's are read
__device__ __forceinline__ double *pivot_of(const DenseBatch &B, int m, int k) {
    return B.D + ((long long)(k & 1) * B.nMat + m) * kNB * kNB;
}
__device__ __forceinline__ double *panel_of(const DenseBatch &B, int m, int k) {
    return B.C + (k & 1) * B.cTotal + B.cOff[m];
}

// ---- step 0: pivot thresholds relative to each matrix's largest diagonal ----

__global__ void k_inv_thresholds(DenseBatch B, double rel) {
    const int m = blockIdx.x;
    const int n = B.dim[m];
    double mx = 0.0;
    for (int i = threadIdx.x; i < n; i += blockDim.x) mx = fmax(mx, *mat_at(B, m, i, i));
    __shared__ double red[kInvThreads];
    red[threadIdx.x] = mx;
    __syncthreads();
    for (int s = blockDim.x / 2; s > 0; s >>= 1) {
        if (threadIdx.x < s) red[threadIdx.x] = fmax(red[threadIdx.x], red[threadIdx.x + s]);
        __syncthreads();
    }
    if (threadIdx.x == 0) B.thr[m] = rel * red[0];
}

// ---- the pivot block's sweep (nb x nb) of every matrix ------------------------
//
// A thread holds 4 x 4 entries in registers.  Entry (i, l) of sweep j becomes
// S - c_i r_l / p, with c and r the pivot's column and row; the pivot's own row
// and column (r_l / p, c_i / p, and -1 / p) are the same expression with c_j =
// r_j = -1 and S = 0.  The owners of the next column and row hand them over
// through shared memory, and the next pivot's reciprocal is taken as soon as
// its entry is updated, so a sweep is its FP64 operations (2 x 64^2) and one
// barrier.
__global__ void __launch_bounds__(kInvThreads)
k_inv_pivot(DenseBatch B, int k) {
    pdl_trigger();
    const int m = blockIdx.x;
    const int n = B.dim[m], k0 = k * kNB;
    if (k0 >= n) return;
    const int nb = min(kNB, n - k0);
    __shared__ double col[2][kNB], row[2][kNB], inv[2];
    __shared__ int failed;
    const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
    const double thr = B.thr[m];
    double S[4][4];
#pragma unroll
    for (int a = 0; a < 4; ++a)
#pragma unroll
        for (int b = 0; b < 4; ++b) {
            const int i = ty + 16 * a, l = tx + 16 * b;
            S[a][b] = i < nb && l < nb ? *mat_at(B, m, k0 + i, k0 + l) : 0.0;
        }
    if (threadIdx.x == 0) failed = -1;
    __syncthreads();
    // the pivot j of the entries as they are now
    auto hand_over = [&](int j) {
        const int q = j & 1, ja = j >> 4, jt = j & 15;
        if (ty == jt && tx == jt) {
            double p = 0.0;
#pragma unroll
            for (int a = 0; a < 4; ++a)
                if (a == ja) p = S[a][a];
            // a failed pivot still sweeps (with a harmless value) so the kernel
            // finishes; the failure is reported and the result not used
            const bool ok = p > thr && isfinite(p);
            if (!ok && failed < 0) failed = k0 + j;
            inv[q] = ok ? 1.0 / p : 0.0;
        }
        if (tx == jt)
#pragma unroll
            for (int a = 0; a < 4; ++a)
#pragma unroll
                for (int b = 0; b < 4; ++b)
                    if (b == ja) col[q][ty + 16 * a] = ty + 16 * a == j ? -1.0 : S[a][b];
        if (ty == jt)
#pragma unroll
            for (int a = 0; a < 4; ++a)
#pragma unroll
                for (int b = 0; b < 4; ++b)
                    if (a == ja) row[q][tx + 16 * b] = tx + 16 * b == j ? -1.0 : S[a][b];
    };
    hand_over(0);
    __syncthreads();
    for (int j = 0; j < nb; ++j) {
        const int q = j & 1;
        const double v = inv[q];
        double c[4], r[4];
#pragma unroll
        for (int a = 0; a < 4; ++a) {
            c[a] = col[q][ty + 16 * a];
            r[a] = row[q][tx + 16 * a];
        }
#pragma unroll
        for (int a = 0; a < 4; ++a)
#pragma unroll
            for (int b = 0; b < 4; ++b) {
                const bool own = ty + 16 * a == j || tx + 16 * b == j;
                S[a][b] = __fma_rn(-__dmul_rn(c[a], r[b]), v, own ? 0.0 : S[a][b]);
            }
        if (j + 1 < nb) hand_over(j + 1);
        __syncthreads();
    }
    // the swept block, -A_PP^-1, for the panel and write-back launches
    double *D = pivot_of(B, m, k);
#pragma unroll
    for (int a = 0; a < 4; ++a)
#pragma unroll
        for (int b = 0; b < 4; ++b)
            if (ty + 16 * a < nb && tx + 16 * b < nb)
                D[(ty + 16 * a) * kNB + tx + 16 * b] = S[a][b];
    if (threadIdx.x == 0 && failed >= 0) atomicMin(B.bad, B.badByMatrix ? m : failed);
}

// ---- the column panel C = A_QP A_PP^-1 = -A_QP D ---------------------------------
//
// The previous pivot's rows of it are that step's panel, not yet written back.
__global__ void __launch_bounds__(kInvThreads)
k_inv_panel(DenseBatch B, int k) {
    pdl_trigger();
    const int t = blockIdx.x;
    const int m = find_matrix(B.rowTileOff, B.nMat, t);
    const int I = t - B.rowTileOff[m];
    const int n = B.dim[m], k0 = k * kNB;
    if (k0 >= n || I == k) return;
    const int nb = min(kNB, n - k0);
    extern __shared__ double sm[];
    double *X = sm, *Y = sm + kNB * kLd;
    const int r0 = I * kNB;
    const double *D = pivot_of(B, m, k), *Cp = panel_of(B, m, k - 1);
    for (int e = threadIdx.x; e < kNB * kNB; e += blockDim.x) {
        const int i = e / kNB, j = e - i * kNB;
        if (I + 1 == k)
            X[j * kLd + i] = i < nb ? Cp[(long long)(k0 + i) * kNB + j] : 0.0;
        else
            X[i * kLd + j] = (r0 + i < n && j < nb) ? *mat_at(B, m, r0 + i, k0 + j) : 0.0;
        Y[i * kLd + j] = (i < nb && j < nb) ? -D[i * kNB + j] : 0.0;
    }
    __syncthreads();
    double acc[4][4] = {};
    tile_mm<4>(X, Y, nb, acc);
    const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
    double *C = panel_of(B, m, k);
#pragma unroll
    for (int a = 0; a < 4; ++a)
#pragma unroll
        for (int b = 0; b < 4; ++b) {
            const int i = r0 + ty + 16 * a, j = tx + 16 * b;
            if (i < n && j < nb) C[(long long)i * kNB + j] = acc[a][b];
        }
}

// ---- A_IJ -= C_I A_kJ, J >= I, mirrored into A_JI ----------------------------------
//
// Columns [c0, c0 + 16 CB) of tile (I, J).  Everything is read from L2: the
// launches beside another kernel do not wait before they work, and it is a wait
// that would make the finished kernels' writes visible to ordinary loads.
template <int CB>
__device__ __forceinline__ void update_tile(const DenseBatch &B, int m, int k, int I, int J,
                                            int cOff) {
    constexpr int W = 16 * CB;
    const int n = B.dim[m], k0 = k * kNB;
    const int nb = min(kNB, n - k0);
    extern __shared__ double sm[];
    double *X = sm, *Y = sm + kNB * kLd;
    const int r0 = I * kNB, c0 = J * kNB + cOff;
    const double *C = panel_of(B, m, k);
    for (int e = threadIdx.x; e < kNB * kNB; e += blockDim.x) {
        const int i = e / kNB, j = e - i * kNB;
        X[i * kLd + j] =
            (r0 + i < n && j < nb) ? ld_early(C + (long long)(r0 + i) * kNB + j) : 0.0;
    }
    for (int e = threadIdx.x; e < kNB * W; e += blockDim.x) {
        const int i = e / W, j = e - i * W;
        Y[i * kLd + j] = (i < nb && c0 + j < n) ? ld_early(mat_at(B, m, k0 + i, c0 + j)) : 0.0;
    }
    __syncthreads();
    double acc[4][CB] = {};
    tile_mm<CB>(X, Y, nb, acc);
    const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
#pragma unroll
    for (int a = 0; a < 4; ++a) {
        const int i = r0 + ty + 16 * a;
        double old[CB];
#pragma unroll
        for (int b = 0; b < CB; ++b) {
            const int j = c0 + tx + 16 * b;
            old[b] = i < n && j < n ? ld_early(mat_at(B, m, i, j)) : 0.0;
        }
#pragma unroll
        for (int b = 0; b < CB; ++b) {
            const int j = c0 + tx + 16 * b;
            if (i < n && j < n) *mat_at(B, m, i, j) = old[b] - acc[a][b];
        }
    }
    if (I == J) return;
    // the mirrored tile A_JI = A_IJ^T: new values through shared memory so
    // that both stores are row-wise
    __syncthreads();
#pragma unroll
    for (int a = 0; a < 4; ++a)
#pragma unroll
        for (int b = 0; b < CB; ++b) X[(ty + 16 * a) * kLd + tx + 16 * b] = acc[a][b];
    __syncthreads();
    for (int e = threadIdx.x; e < kNB * W; e += blockDim.x) {
        const int jj = e / kNB, ii = e - jj * kNB;   // A(c0 + jj, r0 + ii) -= acc(ii, jj)
        if (c0 + jj < n && r0 + ii < n) {
            double *t = mat_at(B, m, c0 + jj, r0 + ii);
            *t = ld_early(t) - X[ii * kLd + jj];
        }
    }
}

// the tiles of the next pivot's row and column, half a tile per CTA (there are
// fewer of them than SMs)
__global__ void __launch_bounds__(kInvThreads)
k_inv_update_next(DenseBatch B, int k) {
    const int t = blockIdx.x >> 1;
    const int m = find_matrix(B.rowTileOff, B.nMat, t);
    const int I = t - B.rowTileOff[m];
    if ((k + 1) * kNB >= B.dim[m] || I == k) return;
    update_tile<2>(B, m, k, min(I, k + 1), max(I, k + 1), (blockIdx.x & 1) * (kNB / 2));
}

// the other tiles, numbers [t0, t0 + gridDim.x) of the upper tiles; launched
// beside the kernel before it (which it does not depend on): its first CTA
// waits for that kernel at its end, so that what follows both follows
__global__ void __launch_bounds__(kInvThreads)
k_inv_update_rest(DenseBatch B, int k, int t0) {
    const int t = t0 + blockIdx.x;
    const int m = find_matrix(B.tileOff, B.nMat, t);
    const int n = B.dim[m];
    if (k * kNB < n) {
        const int T = (n + kNB - 1) / kNB;
        // upper tile number u -> (I, J >= I), row by row
        int u = t - B.tileOff[m], I = 0;
        while (u >= T - I) {
            u -= T - I;
            ++I;
        }
        const int J = I + u;
        if (I != k && J != k && I != k + 1 && J != k + 1) update_tile<4>(B, m, k, I, J, 0);
    }
    if (blockIdx.x == 0) pdl_wait();
}

// ---- A_Ik = C_I, A_kI = C_I^T, A_kk = -A_kk^-1 ----------------------------------------

__global__ void __launch_bounds__(kInvThreads)
k_inv_writeback(DenseBatch B, int k) {
    const int t = blockIdx.x;
    const int m = find_matrix(B.rowTileOff, B.nMat, t);
    const int I = t - B.rowTileOff[m];
    const int n = B.dim[m], k0 = k * kNB;
    if (k0 >= n) return;
    const int nb = min(kNB, n - k0);
    const int r0 = I * kNB;
    if (I == k) {
        const double *D = pivot_of(B, m, k);
        for (int e = threadIdx.x; e < nb * nb; e += blockDim.x) {
            const int i = e / nb, j = e - i * nb;
            *mat_at(B, m, k0 + i, k0 + j) = D[i * kNB + j];
        }
        return;
    }
    const double *C = panel_of(B, m, k);
    for (int e = threadIdx.x; e < kNB * kNB; e += blockDim.x) {
        const int i = e / kNB, j = e - i * kNB;
        if (r0 + i < n && j < nb) *mat_at(B, m, r0 + i, k0 + j) = C[(long long)(r0 + i) * kNB + j];
    }
    for (int e = threadIdx.x; e < kNB * kNB; e += blockDim.x) {
        const int j = e / kNB, i = e - j * kNB;        // row k0 + j, column r0 + i
        if (r0 + i < n && j < nb) *mat_at(B, m, k0 + j, r0 + i) = C[(long long)(r0 + i) * kNB + j];
    }
}

__global__ void k_inv_negate(double *A, long long n) {
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n;
         i += (long long)gridDim.x * blockDim.x)
        A[i] = -A[i];
}

size_t dense_inv_panel_doubles(int dim) { return (size_t)dim * kNB; }
size_t dense_inv_pivot_doubles() { return (size_t)kNB * kNB; }
int dense_inv_tiles(int dim) { return (dim + kNB - 1) / kNB; }

cudaError_t launch_dense_inverse(const DenseBatch &B, int maxDim, long long nEntries, double rel,
                                 cudaStream_t st) {
    if (B.nMat == 0) return cudaSuccess;
    const int smem = 2 * kNB * kLd * (int)sizeof(double);
    // a pivot CTA that fills an SM's shared memory beside no other, while the
    // matrices leave most SMs to the tiles (measured for one matrix; the line is
    // a tenth of the SMs).  The limit is the kernel's, for every context and
    // thread, so it is always the same; only the launch's own size varies
    constexpr int kPivotSmem = 190 * 1024;
    const int pivotSmem = B.nMat <= 16 ? kPivotSmem : 0;
    for (auto k : {k_inv_panel, k_inv_update_next}) {
        const cudaError_t e =
            cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
        if (e != cudaSuccess) return e;
    }
    cudaError_t e = cudaFuncSetAttribute(k_inv_update_rest,
                                         cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    if (e != cudaSuccess) return e;
    e = cudaFuncSetAttribute(k_inv_pivot, cudaFuncAttributeMaxDynamicSharedMemorySize, kPivotSmem);
    if (e != cudaSuccess) return e;
    k_inv_thresholds<<<B.nMat, kInvThreads, 0, st>>>(B, rel);
    const int steps = (maxDim + kNB - 1) / kNB;
    // beside a pivot sweep: as many tiles as the other SMs update meanwhile (two
    // each), the rest beside the panel
    const int first = std::min(B.nTiles, 2 * device_sm_count());
    k_inv_pivot<<<B.nMat, kInvThreads, pivotSmem, st>>>(B, 0);
    k_inv_panel<<<B.nRowTiles, kInvThreads, smem, st>>>(B, 0);
    for (int k = 0; k < steps; ++k) {
        if (k + 1 == steps) {
            k_inv_update_rest<<<B.nTiles, kInvThreads, smem, st>>>(B, k, 0);
        } else {
            k_inv_update_next<<<2 * B.nRowTiles, kInvThreads, smem, st>>>(B, k);
            k_inv_pivot<<<B.nMat, kInvThreads, pivotSmem, st>>>(B, k + 1);
            if ((e = launch_pdl(k_inv_update_rest, first, kInvThreads, smem, st, B, k, 0)) !=
                cudaSuccess)
                return e;
            k_inv_panel<<<B.nRowTiles, kInvThreads, smem, st>>>(B, k + 1);
            if (B.nTiles > first &&
                (e = launch_pdl(k_inv_update_rest, B.nTiles - first, kInvThreads, smem, st, B, k,
                                first)) != cudaSuccess)
                return e;
        }
        k_inv_writeback<<<B.nRowTiles, kInvThreads, 0, st>>>(B, k);
    }
    const long long g = (nEntries + 255) / 256;
    k_inv_negate<<<(int)(g < 8LL * device_sm_count() ? (g > 0 ? g : 1) : 8LL * device_sm_count()),
                   256, 0, st>>>(B.A, nEntries);
    return cudaGetLastError();
}

}  // namespace xdcg

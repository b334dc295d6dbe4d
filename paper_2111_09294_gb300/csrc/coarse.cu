// Coarse level of the deflation (Section 3.2): W = K Z and E = Z^T K Z at
// set-up, the FP64 inverse of E, and the per-iteration coarse solve
// nu = E^-1 g that replaces the two solves of Algorithm 3 (their difference
// lambda - mu = E^-1 (Z^T r - Z^T K y)) and the two of Algorithm 2.
#include <type_traits>

#include "cache.cuh"
#include "reduce.cuh"

namespace xdcg {

// Row j of the deflation block of a node (b dofs, M = 6 or 12 columns):
// standard dof a -> R row a (and H * R row a in the enriched columns), jump
// dof a -> R row a in the enriched columns, branch dofs -> 0.
__device__ __forceinline__ void z_row(int j, int b, int menr, double X, double Y, double Z,
                                      double H, double (&o)[12]) {
#pragma unroll
    for (int c = 0; c < 12; ++c) o[c] = 0.0;
    double r[6] = {0, 0, 0, 0, 0, 0};
    const int a = (j < 3) ? j : j - 3;
    if (j < 3 || (b == 6 && menr)) {
        if (a == 0) { r[0] = 1.0; r[4] = Z; r[5] = -Y; }
        if (a == 1) { r[1] = 1.0; r[3] = -Z; r[5] = X; }
        if (a == 2) { r[2] = 1.0; r[3] = Y; r[4] = -X; }
    } else {
        return;
    }
    if (j < 3) {
#pragma unroll
        for (int c = 0; c < 6; ++c) o[c] = r[c];
        if (menr) {
#pragma unroll
            for (int c = 0; c < 6; ++c) o[6 + c] = H * r[c];
        }
    } else {
#pragma unroll
        for (int c = 0; c < 6; ++c) o[6 + c] = r[c];
    }
}

// Row j of node I's deflation block (M columns of box s): the caller's values
// in the valued form, else from the geometry.
__device__ __forceinline__ void z_row_of(const ZvalDev &Zv, int I, int j, int b, int M, int menr,
                                         double X, double Y, double Z, double H,
                                         double (&o)[12]) {
    if (Zv.v) {
        const double *r = Zv.v + Zv.off[I] + (long long)j * M;
#pragma unroll
        for (int c = 0; c < 12; ++c) o[c] = c < M ? r[c] : 0.0;
    } else {
        z_row(j, b, menr, X, Y, Z, H, o);
    }
}

// Entry (j, c) of a node's deflation block (see z_row): by value, or from the
// geometry without the rest of the row.
__device__ __forceinline__ double z_entry(const ZvalDev &Zv, int J, int j, int b, int M, int menr,
                                          const double *x, double H, int c) {
    if (Zv.v) return Zv.v[Zv.off[J] + (long long)j * M + c];
    if (j >= 3 && !(b == 6 && menr && c >= 6)) return 0.0;
    const int a = j < 3 ? j : j - 3, c6 = c < 6 ? c : c - 6;
    double r = 0.0;
    if (c6 == a) r = 1.0;
    if (a == 0) r = c6 == 4 ? x[2] : (c6 == 5 ? -x[1] : r);
    if (a == 1) r = c6 == 3 ? -x[2] : (c6 == 5 ? x[0] : r);
    if (a == 2) r = c6 == 3 ? x[1] : (c6 == 4 ? -x[0] : r);
    return j < 3 && c >= 6 ? H * r : r;
}

// W block of entry e (node I coupled to box s): W_Is = sum_{J in s} K_IJ Z_J.
// Eight threads per entry, each with three rows of one column at a time, the
// sums in registers: about 1.8 ms at 32^3 (113k entries); one thread per entry
// with its whole block in local memory took 7.3.
constexpr int kWThreads = 8;

__global__ void __launch_bounds__(128)
k_build_W(KinDev K, int nExt, const int *extBox, const int *extNode, const long long *wOff,
          const int *sub, const double *xrel, const signed char *hsign, const int *menr,
          ZvalDev Zv, double *W) {
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    const int e = t / kWThreads;
    if (e >= nExt) return;
    const int s = extBox[e], I = extNode[e], enr = menr[s];
    const int M = enr ? 12 : 6;
    const int bI = K.dofStart[I + 1] - K.dofStart[I];
    const int p0 = K.rowPtr[I], p1 = K.rowPtr[I + 1];
    double *Wb = W + wOff[e];
    for (int task = t % kWThreads; task < bI / 3 * M; task += kWThreads) {
        const int i0 = 3 * (task / M), c = task % M;
        double acc[3] = {0.0, 0.0, 0.0};
        for (int p = p0; p < p1; ++p) {
            const int J = K.col[p];
            if (sub[J] != s) continue;
            const int bJ = K.dofStart[J + 1] - K.dofStart[J];
            const double *Kb = K.val + K.valPtr[p] + (long long)i0 * bJ;
            const double x[3] = {xrel[3 * J], xrel[3 * J + 1], xrel[3 * J + 2]};
            const double H = (double)hsign[J];
            for (int j = 0; j < bJ; ++j) {
                const double z = z_entry(Zv, J, j, bJ, M, enr, x, H, c);
#pragma unroll
                for (int i = 0; i < 3; ++i) {
                    const double kij = Kb[(long long)i * bJ + j];
                    if (kij != 0.0) acc[i] = fma(kij, z, acc[i]);
                }
            }
        }
#pragma unroll
        for (int i = 0; i < 3; ++i) Wb[(i0 + i) * M + c] = acc[i];
    }
}

void launch_build_W(const KinDev &K, int nExt, const int *extBox, const int *extNode,
                    const long long *wOff, const int *sub, const double *xrel,
                    const signed char *hsign, const int *menr, const ZvalDev &Zv, double *W,
                    cudaStream_t st) {
    if (nExt == 0) return;
    const long long threads = (long long)nExt * kWThreads;
    k_build_W<<<(unsigned)((threads + 127) / 128), 128, 0, st>>>(K, nExt, extBox, extNode, wOff,
                                                                 sub, xrel, hsign, menr, Zv, W);
}

// E block (owner box t rows, box s columns) from one segment of box s's
// W entries whose nodes belong to t: sum_I Z_It^T W_Is, summed in entry order.
__global__ void k_build_E(const int *segBox, const int *segOwner, const int *segBegin,
                          const int *segEnd, const int *extNode, const long long *wOff,
                          const double *W, const int *dofStart, const double *xrel,
                          const signed char *hsign, const int *col0, const int *menr,
                          ZvalDev Zv, int k, double *E) {
    const int g = blockIdx.x;
    const int s = segBox[g], t = segOwner[g];
    const int Ms = menr[s] ? 12 : 6, Mt = menr[t] ? 12 : 6;
    const int a = threadIdx.x / 12, b = threadIdx.x % 12;
    if (a >= Mt || b >= Ms) return;
    double sum = 0.0;
    for (int e = segBegin[g]; e < segEnd[g]; ++e) {
        const int I = extNode[e];
        const int bI = dofStart[I + 1] - dofStart[I];
        const double *Wb = W + wOff[e];
        const double X = xrel[3 * I], Y = xrel[3 * I + 1], Z = xrel[3 * I + 2];
        const double H = (double)hsign[I];
        for (int i = 0; i < bI; ++i) {
            double zr[12];
            z_row_of(Zv, I, i, bI, Mt, menr[t], X, Y, Z, H, zr);
            sum += zr[a] * Wb[i * Ms + b];
        }
    }
    E[(size_t)(col0[t] + a) * k + col0[s] + b] = sum;
}

void launch_build_E(int nSeg, const int *segBox, const int *segOwner, const int *segBegin,
                    const int *segEnd, const int *extNode, const long long *wOff,
                    const double *W, const int *dofStart, const double *xrel,
                    const signed char *hsign, const int *col0, const int *menr,
                    const ZvalDev &Zv, int k, double *E, cudaStream_t st) {
    if (nSeg == 0) return;
    k_build_E<<<nSeg, 144, 0, st>>>(segBox, segOwner, segBegin, segEnd, extNode, wOff, W,
                                     dofStart, xrel, hsign, col0, menr, Zv, k, E);
}

__global__ void k_symmetrize(double *E, int k) {
    const long long idx = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    if (idx >= (long long)k * k) return;
    const int i = (int)(idx / k), j = (int)(idx % k);
    if (j <= i) return;
    const double v = 0.5 * (E[(size_t)i * k + j] + E[(size_t)j * k + i]);
    E[(size_t)i * k + j] = v;
    E[(size_t)j * k + i] = v;
}

void launch_symmetrize(double *E, int k, cudaStream_t st) {
    const long long n = (long long)k * k;
    k_symmetrize<<<(int)((n + 255) / 256), 256, 0, st>>>(E, k);
}

// ---- per-iteration coarse solve -------------------------------------------

// Scalar updates shared by the coarse kernels (modes as for k_coarse); blk
// holds the share of nu^T (Z^T r) of row block rowBlk in thread 0 (the few row
// sums gathered through shared memory: no FP64 shuffle tree in every warp).
//
// With sums.part the kernel before left its blocks' sums there (ResidualSums: the
// FP32 restriction those of ||r||^2, the FP64 update those of ||r||^2 and r^T y),
// and the launch has one more block, the first (rowBlk -1), which adds them while
// the others stream E^-1; the last block to finish makes the stopping tests (a
// stop leaves rho and beta as they are).  So those kernels need no reduction
// across their blocks (ticket, fences and FP64 trees): FP32 restriction 18.5 ->
// 15.5 us at 32^3, 16.3 -> 12.6 at 24^3, 26.5 -> 22.5 at 48^3; FP64 update 16.3 -> 13.7 at
// 8^3, 17.1 -> 14.4 at 24^3.
template <int THREADS>
__device__ __forceinline__ void coarse_scalars(double blk, int rowBlk, int mode,
                                               double *partials, const ResidualSums &sums,
                                               Scalars *sc) {
    if (rowBlk < 0) {
        if (THREADS == kThreads && sums.values == 2) {
            const double t = sum_partials<2>(sums.part, &sc->ticket[2], sums.n);
            if (threadIdx.x == 0) sc->rr = t;
            if (threadIdx.x == 1) sc->ry = t;
        } else {
            const double rr = sum_slots<THREADS>(sums.part, sums.n);
            if (threadIdx.x == 0) {
                sc->rr = rr;
                sc->ry = rr;
            }
        }
        __syncthreads();
    } else if (threadIdx.x == 0) {
        partials[rowBlk] = blk;
    }
    if (!last_block(&sc->ticket[3])) return;
    const double rr = __ldcg(&sc->rr), ry = __ldcg(&sc->ry), rho = sc->rho;
    const double tol2ff = sc->tol2ff;
    const int its = sc->its, max_it = sc->max_it;
    const double tot = sum_slots<THREADS>(partials, (int)gridDim.x - (sums.part ? 1 : 0));
    if (threadIdx.x != 0) return;
    if (sums.part) {
        if (sc->hist && its < sc->histCap) sc->hist[its] = rr;
        const int stop = rr <= tol2ff ? kConverged
                         : its >= max_it ? kMaxIter
                         : !isfinite(rr) || !isfinite(ry) ? kBreakdown : kRunning;
        if (stop != kRunning) {
            sc->done = stop;
            return;
        }
    }
    if (mode == 1) {
        sc->rho = ry + tot;
        sc->beta = 0.0;
    } else if (mode >= 2) {
        const double rho_new = ry + tot;
        const bool restart = mode == 3 && rr > 4.0 * sc->scratch[3];
        sc->beta = restart ? 0.0 : rho_new / rho;
        sc->rho = rho_new;
    }
}

// nu = E^-1 g, one warp per row, four independent FMA chains per lane and
// 16-byte loads when rows are 16-byte aligned (k even).  nu32, if given,
// receives an FP32 copy for the FP32 prolongation.  mode 0: nothing else
// (Algorithm 2); mode 1: rho = r^T y + nu^T (Z^T r), beta = 0 (start);
// mode 2: the same rho_new, beta = rho_new / rho, rho = rho_new (iteration);
// mode 3: as mode 2 after a residual replacement, except that beta = 0 (a
// restart) when the replaced residual is more than twice as long as the
// recursive one it replaced (kept in scratch[3]): the recursion had drifted
// too far from the true residual for the old direction to stay conjugate.
__global__ void __launch_bounds__(kThreads)
k_coarse(const double *__restrict__ Einv, int k, const double *g,
         const double *zr, double *nu, float *nu32, int mode, double *partials,
         ResidualSums sums, Scalars *sc) {
    pdl_wait();
    if (sc->done != kRunning) return;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int rowBlk = (int)blockIdx.x - (sums.part ? 1 : 0);
    const int i = rowBlk < 0 ? k : rowBlk * kWarps + warp;
    double part[1] = {0.0};
    if (i < k) {
        const double *row = Einv + (size_t)i * k;
        double s0 = 0.0, s1 = 0.0, s2 = 0.0, s3 = 0.0;
        if ((k & 1) == 0) {
            const double2 *r2 = reinterpret_cast<const double2 *>(row);
            const double2 *g2 = reinterpret_cast<const double2 *>(g);
            const int k2 = k >> 1;
            int j = lane;
            for (; j + 32 < k2; j += 64) {
                const double2 a = __ldg(r2 + j), b = __ldg(r2 + j + 32);
                const double2 x = ld_dep(g2 + j), y = ld_dep(g2 + j + 32);
                s0 = fma(a.x, x.x, s0);
                s1 = fma(a.y, x.y, s1);
                s2 = fma(b.x, y.x, s2);
                s3 = fma(b.y, y.y, s3);
            }
            for (; j < k2; j += 32) {
                const double2 a = __ldg(r2 + j), x = ld_dep(g2 + j);
                s0 = fma(a.x, x.x, s0);
                s1 = fma(a.y, x.y, s1);
            }
        } else {
            int j = lane;
            for (; j + 32 < k; j += 64) {
                s0 = fma(__ldg(row + j), ld_dep(g + j), s0);
                s1 = fma(__ldg(row + j + 32), ld_dep(g + j + 32), s1);
            }
            for (; j < k; j += 32) s0 = fma(__ldg(row + j), ld_dep(g + j), s0);
        }
        double s = (s0 + s1) + (s2 + s3);
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
        if (lane == 0) {
            nu[i] = s;
            if (nu32) nu32[i] = (float)s;
            if (mode != 0) part[0] = s * zr[i];
        }
    }
    __shared__ double rowPart[kWarps];
    if (lane == 0) rowPart[warp] = part[0];
    __syncthreads();
    double blk = 0.0;
    if (threadIdx.x == 0)
        for (int w = 0; w < kWarps; ++w) blk += rowPart[w];
    coarse_scalars<kThreads>(blk, rowBlk, mode, partials, sums, sc);
}

// nu = E^-1 g with E^-1 held in FP32, for the FP32 iteration of the mixed
// path.  A-DEF2 tolerates an inexact coarse solve (the coarse correction
// acts as a preconditioner, not as a projection the recurrence relies on),
// and on the test problems FP32 E^-1 changes no iteration count.
//
// A block takes four rows, its two warps one half of the columns each, added
// in that order; a lane keeps U loads per row in flight (16-byte ones when k
// is a multiple of 4, so that rows are aligned), and an entry of g (the FP32
// copy that the restriction writes, read through L1) serves the four rows.
// E^-1 is set-up data: the first loads are issued before the wait for the
// restriction.  Small blocks, because 810 of them (k = 3240) spread evenly
// over the SMs and stay resident together.
//
// k = 3240 (42 MB of E^-1, from L2): 17.9 us before (a row per two warps, g read
// for every row, few loads in flight), 14.4 now; k = 3150 (4-byte loads):
// 16.0 before, 14.5 now; k = 60: 8.6 before, 10.3 now (it now ends the iteration's
// sums as well, which the restriction did before).
constexpr int kCoarse32Rows = 4, kCoarse32Threads = 64;

template <int V>
__global__ void __launch_bounds__(kCoarse32Threads)
k_coarse32(const float *__restrict__ Einv, int k, const float *g32,
           const double *zr, double *nu, float *nu32, int mode, double *partials,
           ResidualSums sums, Scalars *sc) {
    constexpr int R = kCoarse32Rows, U = V == 4 ? 4 : 8;
    using E = typename std::conditional<V == 4, float4, float>::type;
    __shared__ float upper[R];
    const int h = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int rowBlk = (int)blockIdx.x - (sums.part ? 1 : 0);
    const int i0 = rowBlk < 0 ? k : rowBlk * R;
    const int nv = k / V, mid = (nv + 1) >> 1;
    const int j0 = (h ? mid : 0) + lane, j1 = rowBlk < 0 ? 0 : (h ? nv : mid);
    const uint64_t keep = l2_keep_policy();
    const E *row[R];
#pragma unroll
    for (int r = 0; r < R; ++r)
        row[r] = reinterpret_cast<const E *>(Einv + (size_t)min(i0 + r, k - 1) * k);
    E e[U][R];
    auto load = [&](int j) {
#pragma unroll
        for (int u = 0; u < U; ++u)
            if (j + 32 * u < j1)
#pragma unroll
                for (int r = 0; r < R; ++r) e[u][r] = ld_keep(row[r] + j + 32 * u, keep);
    };
    // a launch queued past a stop loads nothing; this early read of the flag
    // may be stale, the one after the wait decides
    const bool early = __ldcg(&sc->done) == kRunning;
    if (early) load(j0);
    pdl_wait();
    pdl_trigger();
    if (sc->done != kRunning) return;
    if (!early) load(j0);
    // the row whose sum the lane will hold (one lane of eight)
    const int r = lane >> 3, i = i0 + r;
    const bool holder = (lane & 7) == 0;
    const double zri = mode != 0 && h == 0 && holder && i < k ? zr[i] : 0.0;
    float s[R][4] = {};
    const E *gv = reinterpret_cast<const E *>(g32);
    for (int j = j0; j < j1; j += 32 * U) {
        E x[U];
#pragma unroll
        for (int u = 0; u < U; ++u)
            if (j + 32 * u < j1) x[u] = ld_dep(gv + j + 32 * u);
#pragma unroll
        for (int u = 0; u < U; ++u) {
            if (j + 32 * u < j1) {
#pragma unroll
                for (int r = 0; r < R; ++r) {
                    if constexpr (V == 4) {
                        s[r][0] = fmaf(e[u][r].x, x[u].x, s[r][0]);
                        s[r][1] = fmaf(e[u][r].y, x[u].y, s[r][1]);
                        s[r][2] = fmaf(e[u][r].z, x[u].z, s[r][2]);
                        s[r][3] = fmaf(e[u][r].w, x[u].w, s[r][3]);
                    } else {
                        s[r][0] = fmaf(e[u][r], x[u], s[r][0]);
                    }
                }
            }
        }
        load(j + 32 * U);
    }
    // the rows' sums over the lanes by halving exchanges: lane 8 r gets row r
    float v[R];
#pragma unroll
    for (int r = 0; r < R; ++r) v[r] = (s[r][0] + s[r][1]) + (s[r][2] + s[r][3]);
#pragma unroll
    for (int half = 2, o = 16; half > 0; half >>= 1, o >>= 1) {
        const bool hi = (lane & o) != 0;
#pragma unroll
        for (int i = 0; i < half; ++i) {
            const float send = hi ? v[i] : v[i + half], mine = hi ? v[i + half] : v[i];
            v[i] = mine + __shfl_xor_sync(0xffffffffu, send, o);
        }
    }
#pragma unroll
    for (int o = 4; o > 0; o >>= 1) v[0] += __shfl_xor_sync(0xffffffffu, v[0], o);
    if (h == 1 && holder) upper[r] = v[0];
    __syncthreads();
    double blk = 0.0;
    if (h == 0) {
        double part = 0.0;
        if (holder && i < k) {
            const float t = v[0] + upper[r];
            nu[i] = (double)t;
            nu32[i] = t;
            if (mode != 0) part = (double)t * zri;
        }
#pragma unroll
        for (int q = 0; q < R; ++q) blk += __shfl_sync(0xffffffffu, part, 8 * q);
    }
    coarse_scalars<kCoarse32Threads>(blk, rowBlk, mode, partials, sums, sc);
}

void launch_coarse32(const float *Einv, int k, const float *g32, const double *zr, double *nu,
                     float *nu32, int mode, double *partials, ResidualSums sums,
                     Scalars *sc, cudaStream_t st) {
    const int grid = (k + kCoarse32Rows - 1) / kCoarse32Rows;
    launch_pdl(k % 4 == 0 ? k_coarse32<4> : k_coarse32<1>, grid + (sums.part ? 1 : 0), kCoarse32Threads,
               0, st, Einv, k, g32, zr, nu, nu32, mode, partials, sums, sc);
}

void launch_coarse(const double *Einv, int k, const double *g, const double *zr, double *nu,
                   float *nu32, int mode, double *partials, ResidualSums sums,
                   Scalars *sc, cudaStream_t st) {
    const int grid = (k + kWarps - 1) / kWarps;
    launch_pdl(k_coarse, grid + (sums.part ? 1 : 0), kThreads, 0, st, Einv, k, g, zr, nu, nu32, mode,
               partials, sums, sc);
}

}  // namespace xdcg

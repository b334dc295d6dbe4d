// Node-level kernels of the A-DEF2 iteration: the update u += alpha p,
// r -= alpha q (Algorithm 1) fused with y = M^-1 r through the node-block
// Cholesky factors (Algorithm 3, first step; blocks of Eqs. block_jacobi /
// block_jacobi_enr) and the partial sums ||r||^2, r^T y; and the set-up
// factorisation of the node blocks.
#include <algorithm>

#include "reduce.cuh"

namespace xdcg {

// ---- update + block-Jacobi apply ----------------------------------------

__host__ __device__ constexpr int tri(int i, int j) { return i * (i + 1) / 2 + j; }

// The node's entries are all loaded before anything is stored (u, r and y never
// overlap p, q or the factors, but the compiler cannot know), so a thread pays
// one memory round trip instead of one per entry; the factor Lf came earlier
// still, before the wait for the previous kernel.
template <int B>
__device__ __forceinline__ void update_node(const double (&Lf)[B * (B + 1) / 2], long long d0,
                                            double *u, double *r, const double *p,
                                            const double *q, double *y, int mode,
                                            const Scalars *sc, double &rr, double &ry) {
    double w[B];
#pragma unroll
    for (int i = 0; i < B; ++i) w[i] = r[d0 + i];
    if (mode == 0) {
        double uv[B], pv[B], qv[B];
#pragma unroll
        for (int i = 0; i < B; ++i) {
            uv[i] = u[d0 + i];
            pv[i] = p[d0 + i];
            qv[i] = q[d0 + i];
        }
        const double alpha = sc->alpha;
#pragma unroll
        for (int i = 0; i < B; ++i) {
            u[d0 + i] = fma(alpha, pv[i], uv[i]);
            w[i] = fma(-alpha, qv[i], w[i]);
            r[d0 + i] = w[i];
        }
    }
    double rv[B];
#pragma unroll
    for (int i = 0; i < B; ++i) rv[i] = w[i];
    // L w = r (forward), then L^T y = w (backward); diagonal stored inverted
#pragma unroll
    for (int i = 0; i < B; ++i) {
        double s = w[i];
#pragma unroll
        for (int j = 0; j < i; ++j) s = fma(-Lf[tri(i, j)], w[j], s);
        w[i] = s * Lf[tri(i, i)];
    }
#pragma unroll
    for (int i = B - 1; i >= 0; --i) {
        double s = w[i];
#pragma unroll
        for (int j = i + 1; j < B; ++j) s = fma(-Lf[tri(j, i)], w[j], s);
        w[i] = s * Lf[tri(i, i)];
    }
#pragma unroll
    for (int i = 0; i < B; ++i) {
        y[d0 + i] = w[i];
        rr += rv[i] * rv[i];
        ry += rv[i] * w[i];
    }
}

// Branch-enriched node (15 dofs): half a warp per node, lane i of the half
// holds dof i; each solved entry of the forward and backward substitutions is
// broadcast by a shuffle, so no thread keeps the whole block in registers.
// The lane's factor row (Lr) and column (Lc) come from before the wait.  Two
// nodes share a warp because the substitutions are FP64 instructions, which
// cost the same whether 15 or 30 lanes use them.
__device__ __forceinline__ void update_tip_half(const double (&Lr)[15], const double (&Lc)[15],
                                                double dinv, bool act, int lane, long long d0,
                                                double *u, double *r, const double *p,
                                                const double *q, double *y, int mode,
                                                const Scalars *sc, double &rr, double &ry) {
    constexpr int B = 15;
    double ri = 0.0;
    if (act) {
        ri = r[d0 + lane];
        if (mode == 0) {
            const double uv = u[d0 + lane], pv = p[d0 + lane], qv = q[d0 + lane];
            const double alpha = sc->alpha;
            u[d0 + lane] = fma(alpha, pv, uv);
            ri = fma(-alpha, qv, ri);
            r[d0 + lane] = ri;
        }
    }
    double acc = 0.0, w = 0.0;
#pragma unroll
    for (int j = 0; j < B; ++j) {
        const double wj = __shfl_sync(0xffffffffu, (ri - acc) * dinv, j, 16);
        if (lane == j) w = wj;
        if (lane > j) acc = fma(Lr[j], wj, acc);
    }
    double yv = 0.0, acc2 = 0.0;
#pragma unroll
    for (int i = B - 1; i >= 0; --i) {
        const double yi = __shfl_sync(0xffffffffu, (w - acc2) * dinv, i, 16);
        if (lane == i) yv = yi;
        if (lane < i) acc2 = fma(Lc[i], yi, acc2);
    }
    if (act) {
        y[d0 + lane] = yv;
        rr += ri * ri;
        ry += ri * yv;
    }
}

// Partial sums (||r||^2, r^T y) come in units of kWarps warps' work: 256 nodes
// of 3 or 6 dofs (one block), or 8 nodes of 15 dofs (half a block, one node
// per half-warp).  Each unit's two sums are the tree over its lanes and then
// its 8 warps (or nodes); the two values share the shuffles and FP64 adds of
// a tree (they are exchanged at its first step, one half-warp keeping each),
// because FP64 instructions are what these trees cost.  The units' sums are
// added by the coarse solve (ResidualSums).
//
// Bound by FP64 issue and memory latency: everything that set-up fixed (node
// lists, factors) is loaded before the wait for the product, everything else
// in one round trip after it.  48^3 (373k dofs, 115k nodes, 1,932 of them with
// 15 dofs): 44.9 us before, 24.4 now; 8.9k dofs: 17.4 before, 14.2 now
// (event-timed in the solve, as all figures of this kernel).
__global__ void __launch_bounds__(kThreads, 3)
k_update(NodeDev<double> N, double *u, double *r, const double *p, const double *q, double *y,
         int mode, int nb3, int nb6, int nUnits, double *part, const Scalars *sc) {
    // the 15-dof nodes' blocks, whose substitutions take longest, are
    // scheduled first; their units come last in the sums
    const int nb15 = (int)gridDim.x - nb3 - nb6;
    const int bid = (int)blockIdx.x < nb15 ? nb3 + nb6 + (int)blockIdx.x : (int)blockIdx.x - nb15;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    double v[2] = {0.0, 0.0};
    __shared__ double sums[2][2 * kWarps];
    const bool tips = bid >= nb3 + nb6;
    if (!tips) {
        if (bid < nb3) {
            const int t = bid * kThreads + threadIdx.x;
            const bool act = t < N.nStd;
            long long d0 = 0;
            double Lf[6];
            if (act) {
                d0 = N.dofStart[N.stdNodes[t]];
#pragma unroll
                for (int e = 0; e < 6; ++e) Lf[e] = N.Lstd[(size_t)e * N.nStd + t];
            }
            pdl_wait();
            if (sc->done != kRunning) return;
            if (act) update_node<3>(Lf, d0, u, r, p, q, y, mode, sc, v[0], v[1]);
        } else {
            const int t = (bid - nb3) * kThreads + threadIdx.x;
            const bool act = t < N.nH;
            long long d0 = 0;
            double Lf[21];
            if (act) {
                d0 = N.dofStart[N.hNodes[t]];
#pragma unroll
                for (int e = 0; e < 21; ++e) Lf[e] = N.Lh[(size_t)e * N.nH + t];
            }
            pdl_wait();
            if (sc->done != kRunning) return;
            if (act) update_node<6>(Lf, d0, u, r, p, q, y, mode, sc, v[0], v[1]);
        }
        // lanes 0-15 keep ||r||^2, lanes 16-31 r^T y
        const bool hi = lane >= 16;
        double s = (hi ? v[1] : v[0]) + __shfl_xor_sync(0xffffffffu, hi ? v[0] : v[1], 16);
#pragma unroll
        for (int o = 8; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
        if ((lane & 15) == 0) sums[lane >> 4][warp] = s;
    } else {
        const int hl = lane & 15, hw = 2 * warp + (lane >> 4);
        const int t = (bid - nb3 - nb6) * 2 * kWarps + hw;
        const bool act = hl < 15 && t < N.nT;
        long long d0 = 0;
        double Lr[15], Lc[15], dinv = 0.0;
        if (t < N.nT) d0 = N.dofStart[N.tNodes[t]];
#pragma unroll
        for (int j = 0; j < 15; ++j) {
            Lr[j] = act && hl > j ? N.Lt[(size_t)tri(hl, j) * N.nT + t] : 0.0;
            Lc[j] = act && hl < j ? N.Lt[(size_t)tri(j, hl) * N.nT + t] : 0.0;
        }
        if (act) dinv = N.Lt[(size_t)tri(hl, hl) * N.nT + t];
        pdl_wait();
        if (sc->done != kRunning) return;
        update_tip_half(Lr, Lc, dinv, act, hl, d0, u, r, p, q, y, mode, sc, v[0], v[1]);
        // lanes 0-7 of a half-warp keep ||r||^2, lanes 8-15 r^T y
        const bool hi = (lane & 8) != 0;
        double s = (hi ? v[1] : v[0]) + __shfl_xor_sync(0xffffffffu, hi ? v[0] : v[1], 8);
#pragma unroll
        for (int o = 4; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
        if ((lane & 7) == 0) sums[(lane >> 3) & 1][hw] = s;
    }
    __syncthreads();
    if (warp == 0) {
        // lane = 16 (unit of the block) + 8 (value) + warp or node of the unit
        const int val = (lane >> 3) & 1, un = lane >> 4;
        double s = un == 0 || tips ? sums[val][8 * un + (lane & 7)] : 0.0;
#pragma unroll
        for (int o = 4; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
        const int unit = tips ? nb3 + nb6 + 2 * (bid - nb3 - nb6) + un : bid;
        if ((lane & 7) == 0 && (un == 0 || tips) && unit < nUnits)
            part[(size_t)val * nUnits + unit] = s;
    }
}

static inline int cdiv(long long a, int b) { return (int)((a + b - 1) / b); }

int update_units(const NodeDev<double> &N) {
    return std::max(cdiv(N.nStd, kThreads) + cdiv(N.nH, kThreads) + cdiv(N.nT, kWarps), 1);
}

void launch_update(const NodeDev<double> &N, double *u, double *r, const double *p,
                   const double *q, double *y, int mode, double *part, Scalars *sc,
                   cudaStream_t st) {
    const int nb3 = cdiv(N.nStd, kThreads), nb6 = cdiv(N.nH, kThreads), nu15 = cdiv(N.nT, kWarps);
    const int grid = std::max(nb3 + nb6 + (nu15 + 1) / 2, 1);
    launch_pdl(k_update, grid, kThreads, 0, st, N, u, r, p, q, y, mode, nb3, nb6, update_units(N),
               part, (const Scalars *)sc);
}

// ---- set-up: node-block Cholesky (FP64) ------------------------------------

// Node t of the list (count nodes) factored into position pos[t] of a list
// of total entries (pos == nullptr: t itself, total = count).
template <int B>
__global__ void k_block_cholesky(int count, const int *nodes, const double *__restrict__ D,
                                 double *L64, float *L32, int *bad, const int *pos, int total) {
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= count) return;
    const int w = pos ? pos[t] : t;
    double a[B * (B + 1) / 2];
    double dmax = 0.0;
#pragma unroll
    for (int i = 0; i < B; ++i) {
#pragma unroll
        for (int j = 0; j <= i; ++j) a[tri(i, j)] = D[(size_t)(i * B + j) * count + t];
        dmax = fmax(dmax, a[tri(i, i)]);
    }
    bool ok = dmax > 0.0;
#pragma unroll
    for (int j = 0; j < B; ++j) {
        double s = a[tri(j, j)];
#pragma unroll
        for (int k = 0; k < j; ++k) s -= a[tri(j, k)] * a[tri(j, k)];
        if (!(s > 1e-14 * dmax)) ok = false;
        const double ljj = sqrt(fmax(s, 1e-300));
        a[tri(j, j)] = ljj;
#pragma unroll
        for (int i = j + 1; i < B; ++i) {
            double v = a[tri(i, j)];
#pragma unroll
            for (int k = 0; k < j; ++k) v -= a[tri(i, k)] * a[tri(j, k)];
            a[tri(i, j)] = v / ljj;
        }
    }
    if (!ok) atomicMin(bad, nodes[t]);
#pragma unroll
    for (int i = 0; i < B; ++i) {
#pragma unroll
        for (int j = 0; j <= i; ++j) {
            const double v = (i == j) ? 1.0 / a[tri(i, i)] : a[tri(i, j)];
            L64[(size_t)tri(i, j) * total + w] = v;
            if (L32) L32[(size_t)tri(i, j) * total + w] = (float)v;
        }
    }
}

int launch_block_cholesky(int B, int count, const int *nodes, const double *Dsoa, double *L64,
                          float *L32, int *bad, cudaStream_t st, const int *pos, int total) {
    if (count == 0) return 0;
    if (!pos) total = count;
    const int th = 128, grid = cdiv(count, th);
    switch (B) {
        case 3:
            k_block_cholesky<3><<<grid, th, 0, st>>>(count, nodes, Dsoa, L64, L32, bad, pos, total);
            break;
        case 6:
            k_block_cholesky<6><<<grid, th, 0, st>>>(count, nodes, Dsoa, L64, L32, bad, pos, total);
            break;
        case 15:
            k_block_cholesky<15><<<grid, th, 0, st>>>(count, nodes, Dsoa, L64, L32, bad, pos, total);
            break;
        default: return -1;
    }
    return 0;
}

// Factors carried over from an earlier context: entry e of position dst[i]
// (list of total entries) = entry e of position src[i] of the earlier list
// (prevTotal entries); ents = B (B + 1) / 2 entries per node.
__global__ void k_copy_factors(int count, int ents, const int *src, const int *dst,
                               const double *prev, int prevTotal, double *L, int total) {
    const long long idx = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    if (idx >= (long long)count * ents) return;
    const int i = (int)(idx % count), e = (int)(idx / count);
    L[(size_t)e * total + dst[i]] = prev[(size_t)e * prevTotal + src[i]];
}

void launch_copy_factors(int count, int ents, const int *src, const int *dst, const double *prev,
                         int prevTotal, double *L, int total, cudaStream_t st) {
    if (count == 0) return;
    const long long n = (long long)count * ents;
    k_copy_factors<<<(int)((n + 255) / 256), 256, 0, st>>>(count, ents, src, dst, prev, prevTotal, L,
                                                          total);
}

// *differ = 1 if a and b (n doubles) differ anywhere (bitwise)
__global__ void k_differ(const double *a, const double *b, long long n, int *differ) {
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n;
         i += (long long)gridDim.x * blockDim.x)
        if (__double_as_longlong(a[i]) != __double_as_longlong(b[i])) {
            *differ = 1;
            return;
        }
}

void launch_differ(const double *a, const double *b, long long n, int *differ, cudaStream_t st) {
    if (n <= 0) return;
    const long long g = (n + 255) / 256;
    k_differ<<<(int)(g < 4LL * device_sm_count() ? g : 4LL * device_sm_count()), 256, 0, st>>>(
        a, b, n, differ);
}

__global__ void k_xrel(int n, const double *coords, const double *centre, const int *sub,
                       double *x64, float *x32) {
    const int I = blockIdx.x * blockDim.x + threadIdx.x;
    if (I >= n) return;
    const int s = sub[I];
#pragma unroll
    for (int d = 0; d < 3; ++d) {
        const double v = coords[3 * I + d] - centre[3 * s + d];
        x64[3 * I + d] = v;
        if (x32) x32[3 * I + d] = (float)v;
    }
}

void launch_xrel(int nNodes, const double *coords, const double *centre, const int *sub,
                 double *x64, float *x32, cudaStream_t st) {
    k_xrel<<<cdiv(nNodes, kThreads), kThreads, 0, st>>>(nNodes, coords, centre, sub, x64, x32);
}

}  // namespace xdcg

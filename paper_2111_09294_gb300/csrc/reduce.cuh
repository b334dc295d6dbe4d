// Deterministic warp / block / grid reductions.  Every block stores its
// partial sums; the last block to finish (ticket counter) adds them in a
// fixed order, so results do not depend on block scheduling.
//
// The accumulator type A is the kernel's own precision: FP32 kernels keep
// their per-thread, warp and block sums in FP32 (FP64 arithmetic runs at
// 1/64 of the FP32 rate on this GPU), and only the per-block partials are
// combined in FP64 by the last block.
#pragma once

#include "internal.h"
#include "pdl.cuh"

namespace xdcg {

template <typename A, int NV>
__device__ __forceinline__ void warp_sum(A (&v)[NV]) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
#pragma unroll
        for (int i = 0; i < NV; ++i) v[i] += __shfl_xor_sync(0xffffffffu, v[i], o);
    }
}

// Sum over the block; the result is valid in thread 0.
template <typename A, int NV>
__device__ __forceinline__ void block_sum(A (&v)[NV]) {
    __shared__ A sm[NV][32];
    warp_sum<A, NV>(v);
    const int w = threadIdx.x >> 5, l = threadIdx.x & 31, nw = blockDim.x >> 5;
    __syncthreads();
    if (l == 0) {
#pragma unroll
        for (int i = 0; i < NV; ++i) sm[i][w] = v[i];
    }
    __syncthreads();
    if (w == 0) {
#pragma unroll
        for (int i = 0; i < NV; ++i) v[i] = (l < nw) ? sm[i][l] : A(0);
        // eight warps or fewer: the tree's first two levels would add zeros
        if (nw <= 8) {
#pragma unroll
            for (int o = 4; o > 0; o >>= 1)
#pragma unroll
                for (int i = 0; i < NV; ++i) v[i] += __shfl_xor_sync(0xffffffffu, v[i], o);
        } else {
            warp_sum<A, NV>(v);
        }
    }
}

// Sums N <= P values over the warp by halving exchanges, P - 1 shuffles (and,
// for P = 16, one more) instead of 5 N: each value's tree is that of warp_sum
// (pairs 16, 8, 4, 2, 1 lanes apart).  Lane l gets the total of value l (P =
// 32) or l >> 1 (P = 16).
template <int P, int N>
__device__ __forceinline__ float warp_sum_scatter(const float (&in)[N]) {
    static_assert((P == 16 || P == 32) && N <= P, "");
    float v[P];
#pragma unroll
    for (int i = 0; i < P; ++i) v[i] = i < N ? in[i < N ? i : 0] : 0.0f;
    const int lane = threadIdx.x & 31;
    int o = 16;
#pragma unroll
    for (int half = P / 2; half > 0; half >>= 1) {
        const bool hi = (lane & o) != 0;
#pragma unroll
        for (int i = 0; i < half; ++i) {
            const float send = hi ? v[i] : v[i + half];
            const float keep = hi ? v[i + half] : v[i];
            v[i] = keep + __shfl_xor_sync(0xffffffffu, send, o);
        }
        o >>= 1;
    }
    if (P == 16) v[0] += __shfl_xor_sync(0xffffffffu, v[0], 1);
    return v[0];
}

// The second stage of block_sum for eight warps' sums of one value (the tree
// over 32 lanes of which eight hold a value: zeros added twice, then 4, 2, 1).
__device__ __forceinline__ float sum_of_8(const float (&x)[8]) {
    float y[8];
#pragma unroll
    for (int w = 0; w < 8; ++w) y[w] = x[w] + 0.0f;
    return ((y[0] + y[4]) + (y[2] + y[6])) + ((y[1] + y[5]) + (y[3] + y[7]));
}

// The last block's share of a grid-wide sum: value i of the nblk blocks'
// partials (partials[i * nblk + b]) added by one warp, its lanes striding
// over the blocks with four accumulators each (lane l: rounds of 128 partials
// while l + 96 is in range, the rest into the first accumulator), then across the
// lanes (a fixed order, and FP64 work spread over the warps: FP64 arithmetic is
// slow here).  Thread i < NV gets total i; thread 0 resets the ticket.
//
// This is the tail of its kernel, on one SM while the others wait: four rounds
// of loads are in flight at once (one round trip to L2 instead of one per round),
// the first partial of an accumulator is not added to a zero, and where the
// block has four warps per value each takes one accumulator.  Solves at 1e-8, this
// and what the last block reads next loaded beside the sum: 8 columns at 8^3 3.40 ->
// 3.22 ms, at 32^3 8.63 -> 8.52; one mixed one at 8^3 1.47 -> 1.42, at 32^3 3.66 ->
// 3.55; FP64 at 32^3 9.46 -> 9.32.
template <int NV>
__device__ __forceinline__ double sum_partials(const double *partials, unsigned int *ticket,
                                               int nblk) {
    __shared__ double fin[NV];
    const int w = threadIdx.x >> 5, l = threadIdx.x & 31, nw = blockDim.x >> 5;
    const int rounds = nblk > l + 96 ? (nblk - l - 96 + 127) >> 7 : 0;
    if (NV <= 2 && nw >= 4 * NV) {
        __shared__ double acc[NV <= 2 ? 4 * NV : 1][32];
        if (w < 4 * NV) {
            const int q = w & 3;
            const double *p = partials + (size_t)(w >> 2) * nblk + l;
            double x[3], s = 0.0;
#pragma unroll
            for (int t = 0; t < 3; ++t) {
                const int b = 128 * rounds + 32 * t;
                x[t] = q == 0 && l + b < nblk ? __ldcg(p + b) : 0.0;
            }
            for (int r0 = 0; r0 < rounds; r0 += 4) {
                double v[4];
#pragma unroll
                for (int u = 0; u < 4; ++u)
                    v[u] = r0 + u < rounds ? __ldcg(p + 128 * (r0 + u) + 32 * q) : 0.0;
                s = r0 == 0 ? v[0] : s + v[0];
#pragma unroll
                for (int u = 1; u < 4; ++u)
                    if (r0 + u < rounds) s += v[u];
            }
#pragma unroll
            for (int t = 0; t < 3; ++t)
                if (q == 0 && l + 128 * rounds + 32 * t < nblk) s += x[t];
            acc[w % (NV <= 2 ? 4 * NV : 1)][l] = s;
        }
        __syncthreads();
        if (w < NV) {
            const int i = NV <= 2 ? 4 * w : 0;
            double s = (acc[i][l] + acc[i + 1][l]) + (acc[i + 2][l] + acc[i + 3][l]);
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
            if (l == 0) fin[w] = s;
        }
    } else {
        for (int i = w; i < NV; i += nw) {
            const double *p = partials + (size_t)i * nblk + l;
            double x[3], s[4] = {0.0, 0.0, 0.0, 0.0};
#pragma unroll
            for (int t = 0; t < 3; ++t) {
                const int b = 128 * rounds + 32 * t;
                x[t] = l + b < nblk ? __ldcg(p + b) : 0.0;
            }
            for (int r0 = 0; r0 < rounds; r0 += 4) {
                double v[4][4];
#pragma unroll
                for (int u = 0; u < 4; ++u)
#pragma unroll
                    for (int q = 0; q < 4; ++q)
                        v[u][q] = r0 + u < rounds ? __ldcg(p + 128 * (r0 + u) + 32 * q) : 0.0;
#pragma unroll
                for (int q = 0; q < 4; ++q) s[q] = r0 == 0 ? v[0][q] : s[q] + v[0][q];
#pragma unroll
                for (int u = 1; u < 4; ++u)
                    if (r0 + u < rounds)
#pragma unroll
                        for (int q = 0; q < 4; ++q) s[q] += v[u][q];
            }
#pragma unroll
            for (int t = 0; t < 3; ++t)
                if (l + 128 * rounds + 32 * t < nblk) s[0] += x[t];
            double t = (s[0] + s[1]) + (s[2] + s[3]);
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
            if (l == 0) fin[i] = t;
        }
    }
    __syncthreads();
    if (threadIdx.x == 0) *ticket = 0u;
    return threadIdx.x < NV ? fin[threadIdx.x] : 0.0;
}

// Grid-wide sum of NV <= 32 values whose block totals lanes 0 .. NV - 1 of
// warp 0 already hold (one per lane, in v): as grid_sum without the block
// reduction, over the blocks blk = 0 .. nblk - 1 of one reduction (the launch's, or
// one system's share of a launch over several systems); in the last block to
// finish, which returns true, the totals come back to the same lanes.  Every
// thread of the block calls it.  partials: NV * nblk doubles.  loads(): run by the
// last block before the sum, for what it reads next (the latency then passes
// beside the sum).
template <int NV, typename F>
__device__ __forceinline__ bool grid_sum_lanes(double v, double *partials, unsigned int *ticket,
                                               double &tot, int blk, int nblk, F loads) {
    __shared__ bool last;
    if (threadIdx.x < 32) {
        if ((int)threadIdx.x < NV) partials[(size_t)threadIdx.x * nblk + blk] = v;
        __threadfence();
        __syncwarp();
        if (threadIdx.x == 0) last = atomicAdd(ticket, 1u) == (unsigned int)nblk - 1;
    }
    __syncthreads();
    if (!last) return false;
    __threadfence();
    loads();
    tot = sum_partials<NV>(partials, ticket, nblk);
    return true;
}

// Double-float arithmetic: a value as an unevaluated sum hi + lo of two
// floats (about 48 significant bits), added with FP32 operations only
// (Knuth's two-sum, then renormalisation).  Used where many blocks each add
// the same few hundred partial sums: FP64 runs at about 1/64 of the FP32
// rate on this part.
__device__ __forceinline__ float2 df_add(float2 a, float2 b) {
    const float s = a.x + b.x;
    const float bb = s - a.x;
    const float e = (a.x - (s - bb)) + (b.x - bb);
    const float t = (e + a.y) + b.y;
    const float hi = s + t;
    return make_float2(hi, t - (hi - s));
}
__device__ __forceinline__ float2 df_of(double v) {
    const float hi = (float)v;
    return make_float2(hi, (float)(v - (double)hi));
}

// The total of n block partials (double-float) a previous kernel stored
// (kFinDefer): every thread loads its share at once (one round trip), the
// shares are added in a fixed order within each thread, by a tree over the
// lanes and over the warps, so every block of the consuming kernel gets the
// same bits.  Valid in thread 0 (FP64 instructions cost 64 cycles each
// whatever the number of threads, and all of a block's warps would share the
// SM's FP64 units: one thread goes on alone).  A share that is not there is
// not added: a normalised pair plus zero is itself.
__device__ __forceinline__ double block_total_t0(const float2 *partials, int n) {
    __shared__ float2 wsum[32];
    const int t = threadIdx.x, nt = blockDim.x;
    const float2 none = make_float2(0.f, 0.f);
    float2 a = t < n ? __ldcg(partials + t) : none;
    float2 b = t + nt < n ? __ldcg(partials + t + nt) : none;
    if (nt < n) a = df_add(a, b);
    for (int i = t + 2 * nt; i - t < n; i += nt)
        a = df_add(a, i < n ? __ldcg(partials + i) : none);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        float2 other;
        other.x = __shfl_xor_sync(0xffffffffu, a.x, o);
        other.y = __shfl_xor_sync(0xffffffffu, a.y, o);
        a = df_add(a, other);
    }
    if ((t & 31) == 0) wsum[t >> 5] = a;
    __syncthreads();
    double total = 0.0;
    if (t == 0) {
        float2 s = wsum[0];
        for (int w = 1; w < (nt >> 5); ++w) s = df_add(s, wsum[w]);
        total = (double)s.x + (double)s.y;
    }
    return total;
}

// Grid-wide sum of one value per thread over the launch's blocks.  Returns true
// in exactly one of them (the last to finish), where thread 0 then holds the
// FP64 total in tot.  partials: one double per block; loads() as in grid_sum_lanes.
template <typename A, typename F>
__device__ __forceinline__ bool grid_sum(A v, double *partials, unsigned int *ticket,
                                         double &tot, F loads) {
    __shared__ bool last;
    A s[1] = {v};
    block_sum<A, 1>(s);
    if (threadIdx.x == 0) {
        partials[blockIdx.x] = (double)s[0];
        __threadfence();
        last = atomicAdd(ticket, 1u) == gridDim.x - 1;
    }
    __syncthreads();
    if (!last) return false;
    __threadfence();
    loads();
    tot = sum_partials<1>(partials, ticket, (int)gridDim.x);
    return true;
}

// grid_sum with the bits it has for 256 threads per block, from a launch of twice
// as many blocks of 128: groups of eight warps (two blocks), each warp's sum in
// partials (8 doubles per group), which the last block first adds within the
// groups by block_sum's tree.  Thread t of it takes groups t, t + 128, ...: in
// sum_partials' order warp q's are accumulator q's, and the last, incomplete
// round belongs to the first accumulator.
template <typename F>
__device__ __forceinline__ bool grid_sum_halves(double v, double *partials, unsigned int *ticket,
                                                double &tot, F loads) {
    __shared__ bool last;
    __shared__ double acc[4][32], rest[4][32];
    const int w = threadIdx.x >> 5, l = threadIdx.x & 31, n = (int)gridDim.x / 2;
    double s[1] = {v};
    warp_sum<double, 1>(s);
    if (l == 0) partials[blockIdx.x * 4 + w] = s[0];
    __syncthreads();
    if (threadIdx.x == 0) {
        __threadfence();
        last = atomicAdd(ticket, 1u) == gridDim.x - 1;
    }
    __syncthreads();
    if (!last) return false;
    __threadfence();
    loads();
    const int rounds = n > l + 96 ? (n - l - 96 + 127) >> 7 : 0;
    double a = 0.0, r = 0.0;
#pragma unroll 1
    for (int i = 0; i <= rounds; ++i) {
        const int g = threadIdx.x + 128 * i;
        if (g >= n) break;
        const double2 *y = reinterpret_cast<const double2 *>(partials) + 4 * g;
        const double2 y0 = __ldcg(y), y2 = __ldcg(y + 1), y4 = __ldcg(y + 2), y6 = __ldcg(y + 3);
        const double t = ((y0.x + y4.x) + (y2.x + y6.x)) + ((y0.y + y4.y) + (y2.y + y6.y));
        if (i == rounds)
            r = t;
        else
            a = i == 0 ? t : a + t;
    }
    acc[w][l] = a;
    rest[w][l] = r;
    __syncthreads();
    if (w == 0) {
#pragma unroll
        for (int q = 0; q < 3; ++q)
            if (l + 128 * rounds + 32 * q < n) a += rest[q][l];
        a = (a + acc[1][l]) + (acc[2][l] + acc[3][l]);
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) a += __shfl_xor_sync(0xffffffffu, a, o);
        if (l == 0) *ticket = 0u;
    }
    tot = a;
    return true;
}

// Sum of n block partials by one block of THREADS threads, valid in thread 0.
// The order of the sum is that of 256 threads whatever THREADS: slot t = 0 ..
// 255 adds partials t, t + 256, ..., then the tree over the 32 slots of a warp and
// the tree over the eight warps; a thread of a smaller block takes 256 / THREADS
// slots, with two rounds of loads in flight after the first.
template <int THREADS>
__device__ __forceinline__ double sum_slots(const double *p, int n) {
    constexpr int Q = kThreads / THREADS, U = 2;
    static_assert(Q == 1 || Q == 4, "");
    __shared__ double sums[kWarps];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    double s[Q];
#pragma unroll
    for (int q = 0; q < Q; ++q)
        s[q] = (int)threadIdx.x + q * THREADS < n ? __ldcg(p + threadIdx.x + q * THREADS) : 0.0;
#pragma unroll 1
    for (int b = threadIdx.x + kThreads; b < n; b += U * kThreads) {
        double v[U][Q];
#pragma unroll
        for (int u = 0; u < U; ++u)
#pragma unroll
            for (int q = 0; q < Q; ++q) {
                const int i = b + u * kThreads + q * THREADS;
                v[u][q] = i < n ? __ldcg(p + i) : 0.0;
            }
#pragma unroll
        for (int u = 0; u < U; ++u)
#pragma unroll
            for (int q = 0; q < Q; ++q)
                if (b + u * kThreads + q * THREADS < n) s[q] += v[u][q];
    }
    int o = 16;
    if (Q == 4) {   // halving exchanges: lanes 8 q .. 8 q + 7 keep the sums of slot set q
#pragma unroll
        for (int half = 2; half > 0; half >>= 1, o >>= 1) {
            const bool hi = (lane & o) != 0;
#pragma unroll
            for (int j = 0; j < half; ++j) {
                const double send = hi ? s[j] : s[(j + half) % Q];
                const double mine = hi ? s[(j + half) % Q] : s[j];
                s[j] = mine + __shfl_xor_sync(0xffffffffu, send, o);
            }
        }
    }
    for (; o > 0; o >>= 1) s[0] += __shfl_xor_sync(0xffffffffu, s[0], o);
    if (lane % (32 / Q) == 0) sums[warp + (THREADS / 32) * (lane / (32 / Q))] = s[0];
    __syncthreads();
    double t = 0.0;
    if (warp == 0) {
        t = lane < kWarps ? sums[lane] : 0.0;
#pragma unroll
        for (int l = 4; l > 0; l >>= 1) t += __shfl_xor_sync(0xffffffffu, t, l);
    }
    return t;
}

// True in the last block of the launch to get here, which may read what thread 0
// of every block wrote before.
__device__ __forceinline__ bool last_block(unsigned int *ticket) {
    __shared__ bool last;
    if (threadIdx.x == 0) {
        __threadfence();
        last = atomicAdd(ticket, 1u) == gridDim.x - 1;
        if (last) *ticket = 0u;
    }
    __syncthreads();
    if (last) __threadfence();
    return last;
}

// Reports the run's state to the host (one thread of a kernel that ends an
// iteration, after its wait; launches queued past a stop repeat the report).
__device__ __forceinline__ void report(const Scalars *sc) {
    volatile Progress *p = sc->prog;
    if (!p) return;
    const bool stopped = sc->done != kRunning;
    if (!stopped) {
        if (sc->rr == 0.0) return;   // a prolongation before the first residual
    } else {
        p->stop = (unsigned long long)(unsigned int)sc->its << 32 | (unsigned int)sc->done;
        __threadfence_system();
    }
    p->rr[sc->its % kRing] =
        report_word((unsigned long long)__double_as_longlong(sc->rr), stopped);
}

// Shared last-block actions on the scalar block.  FinLoads: what they read,
// loaded while the sum is formed (grid_sum's loads()).
struct FinLoads {
    double rho = 0.0, tol2ff = 0.0;
    int its = 0, fault = 0;
    __device__ __forceinline__ void load(const Scalars *sc) {
        if (threadIdx.x != 0) return;
        rho = sc->rho;
        tol2ff = sc->tol2ff;
        its = sc->its;
        fault = __ldcg(&sc->fault);
    }
};
__device__ __forceinline__ void finalize(Scalars *sc, int fin, int slot, double val,
                                         const FinLoads &in) {
    if (fin == kFinAlpha) {
        sc->pq = val;
        sc->its = in.its + 1;
        if (!(val > 0.0) || !isfinite(val)) {
            sc->done = kBreakdown;
        } else {
            sc->alpha = in.rho / val;
        }
    } else if (fin == kFinRR) {
        sc->rr = val;
        if (sc->hist && sc->histCap > 0) sc->hist[0] = val;
        if (val <= in.tol2ff) sc->done = kConverged;
    } else {
        sc->scratch[slot] = val;
    }
}

}  // namespace xdcg

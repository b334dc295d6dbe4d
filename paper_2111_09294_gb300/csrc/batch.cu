// Batched FP32 iteration of the mixed path: MB right-hand sides of one
// system advance together (the multi-load-case solves of a propagation step:
// the same K, several load cases).  Every kernel reads the matrix data once
// per iteration for all columns, so the bytes per right-hand side fall by up
// to MB.  Vectors are interleaved by column: entry (dof d, column j) at
// d * MB + j, so a chunk gathered by the product is one run of 3 * MB floats
// and a row of the box kernels is one run of MB floats.
//
// Columns advance independently (BatchScalars): an iteration updates the
// running columns (active and not held); a held column's residual is copied
// into the next buffer and its other vectors stay as they are, and a column
// that has left keeps zero vectors.  A replacement (open, FP64 residuals,
// judge, transforms, restriction / coarse / prolongation in their
// replacement modes, arm) touches only the columns it replaces.
//
// Every kernel body takes its block index and block count within its own
// system, so the same body runs as a launch for one system or as one launch
// over several systems (BatchSysTab): a column's result is the same bits
// either way.
#include <algorithm>
#include <climits>

#include "cache.cuh"
#include "factor.cuh"
#include "reduce.cuh"
#include "spmv_cfg.cuh"
#include "tma.cuh"

namespace xdcg {

__device__ __forceinline__ bool col_runs(const BatchScalars *bs, int j, int m) {
    return j < m && bs->active[j] && !bs->pend[j];
}

// whether a kernel of the system runs: an iteration's kernels also need the
// gate's go (a launch over several systems skips a system held for its
// replacement); the start and replacement kernels only need the run state
__device__ __forceinline__ bool batch_runs(const BatchScalars *bs, bool iteration) {
    return bs->done == kRunning && (!iteration || bs->go);
}

// the block's system in a launch over several systems: the largest s with
// off[s] <= b
__device__ __forceinline__ int sys_of(const int *__restrict__ off, int nSys, int b) {
    int lo = 0, hi = nSys - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (__ldg(off + mid) <= b)
            lo = mid;
        else
            hi = mid - 1;
    }
    return lo;
}

// ---- per-column scalar updates ----------------------------------------------

// One column per lane (the divisions of a column are a chain of FP64
// instructions of 64 cycles each, which eight lanes share); every lane of a
// warp calls it, with column j's total in lane j.
//
// fin 0 (iteration): pq_j, alpha_j for the running columns (0 for the
// others); a running column whose p^T K p is not positive is held as broken.
// The iteration counts (its, its_j) advance when a column still runs;
// otherwise the system stops until the host's next replacement.
// fin 1 (start): rr_j.
// in: the column's state, loaded while the sums are formed.
struct ColumnLoads {
    double rho = 0.0, rr = 0.0, trig = 0.0, rrRep = 0.0;
    int its = 0, fault = 0, maxIt = 0;
    bool runs = false, active = false, repl = false, broken = false;
    __device__ __forceinline__ void load(const BatchScalars *bs, int m) {
        const int j = threadIdx.x;
        if (j >= 32) return;
        fault = __ldcg(&bs->fault);
        maxIt = bs->max_it;
        if (j >= m) return;
        rho = bs->rho[j];
        rr = bs->rr[j];
        trig = bs->trig[j];
        rrRep = bs->rrRep[j];
        its = bs->itsc[j];
        active = bs->active[j] != 0;
        runs = active && !bs->pend[j];
        repl = bs->repl[j] != 0;
        broken = bs->broken[j] != 0;
    }
};
__device__ __forceinline__ void batch_finalize(BatchScalars *bs, int m, int fin, double tot,
                                               const ColumnLoads &in) {
    const int j = threadIdx.x & 31;
    if (fin != 0) {
        if (j < m) bs->rr[j] = tot;
        return;
    }
    bool any = false;
    if (j < m) {
        bs->pq[j] = tot;
        if (!in.runs) {
            bs->alpha[j] = 0.0;
        } else {
            bs->itsc[j] = in.its + 1;
            if (!(tot > 0.0) || !isfinite(tot)) {
                bs->alpha[j] = 0.0;
                bs->broken[j] = 1;
                bs->pend[j] = 1;
            } else {
                bs->alpha[j] = in.rho / tot;
                any = true;
            }
        }
    }
    any = __any_sync(0xffffffffu, any);
    if (j == 0) {
        if (any)
            bs->its += 1;
        else
            bs->done = kConverged;
    }
}

// ---- batched product Y = K~ X (+ x_j^T y_j, or ||y_j||^2 with y = b - K~ x) --
//
// A lane holds four columns, so MB = 8 gives two lanes to a slot of a step: a
// pass takes 32 / LPS slots (LPS = MB / 4 lanes each) and a step LPS passes.
// The lanes of a slot read whole 32-byte sectors of x (one lane with all eight
// columns read 16 bytes from each of 24 cache lines per load, and the L1's tag
// rate bounded the product), and the gather of the next pass is in flight
// while this one is computed.  Stages run across slice boundaries, as in the
// single product (k_spmv_lean); each row's terms are added in the order of its
// slots, partial rows by the same tree.  8 columns at 32^3 (1.1M blocks): 41.5
// us before, 29.0 now.
// The warp's copy schedule (LeanWalk of the single product, step numbers in 32
// bits: a step is 1,280 bytes).
struct BatchWalk {
    int pos, end, xPos, xEnd, isS;
    __device__ __forceinline__ bool next(int C, int &sS, int &p, int &n) {
        if (pos == end) {
            if (!isS || xPos == xEnd) return false;
            isS = 0;
            pos = xPos;
            end = xEnd;
        }
        sS = isS;
        p = pos;
        n = min(C, end - pos);
        pos += n;
        return true;
    }
};

template <int MB, bool RES>
__device__ __forceinline__ void spmm_body(const SpmmArgs &args, int blk, int nblk,
                                          unsigned char *smem) {
    constexpr int C = SpmvCfg<float, 0>::C, NS = SpmvCfg<float, 0>::NS, SB = stage_bytes<float, 0>();
    constexpr int LPS = MB / 4, SPP = 32 / LPS;   // lanes per slot, slots per pass
    const SpmvDev<float> &A = args.A;
    const int m = args.m, fin = args.fin;
    const float *x = args.x;
    const float *b = args.b;
    float *__restrict__ y = args.y;
    BatchScalars *bs = args.bs;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int sl0 = lane / LPS, qc = lane % LPS;   // the lane's slot of pass 0, its columns / 4
    unsigned char *ring = smem + (size_t)warp * NS * SB;
    uint64_t *bars = reinterpret_cast<uint64_t *>(smem + (size_t)kSpmvWarps * NS * SB) + warp * NS;
    const int nS = A.S.nSlices;
    const int gw = blk * kSpmvWarps + warp;
    const int sFirst = A.warpSlice[gw], sEnd = A.warpSlice[gw + 1];
    if (lane == 0) {
        for (int s = 0; s < NS; ++s) mbar_init(bars + s, 1);
        mbar_init_fence();
    }
    // step counts of the warp's first 32 slices, and its two parts' step runs
    __shared__ int tSteps[kSpmvWarps][32];
    if (sFirst + lane < sEnd) {
        const int g = sFirst + lane;
        const SellDev<float> &P = g < nS ? A.S : A.X;
        const int sl = g < nS ? g : g - nS;
        tSteps[warp][lane] = (int)((P.slicePtr[sl + 1] - P.slicePtr[sl]) >> 5);
    }
    const int sA = min(sEnd, nS);
    const int xa0 = max(sFirst, nS) - nS, xa1 = sEnd - nS;
    BatchWalk pw;
    pw.xPos = xa0 < xa1 ? (int)(A.X.slicePtr[xa0] >> 5) : 0;
    pw.xEnd = xa0 < xa1 ? (int)(A.X.slicePtr[xa1] >> 5) : 0;
    pw.isS = sFirst < sA;
    pw.pos = pw.isS ? (int)(A.S.slicePtr[sFirst] >> 5) : pw.xPos;
    pw.end = pw.isS ? (int)(A.S.slicePtr[sA] >> 5) : pw.xEnd;
    BatchWalk cw = pw;
    __syncwarp();
    const uint64_t stream = l2_stream_policy();
    const unsigned long long deadline = global_ns() + A.waitNs;
    int issued = 0, pslot = 0;
    bool more = true;
    auto issue = [&]() {
        int sS, n, p;
        if (!pw.next(C, sS, p, n)) {
            more = false;
            return;
        }
        if (lane == 0) {
            const SellDev<float> &P = sS ? A.S : A.X;
            unsigned char *dst = ring + pslot * SB;
            fence_proxy_async_smem();
            mbar_arrive_expect_tx(bars + pslot, (uint32_t)n * 1280u);
            bulk_g2s(dst, P.col + 32LL * p, (uint32_t)n * 128u, bars + pslot, stream);
            bulk_g2s(dst + C * 128, P.val + 288LL * p, (uint32_t)n * 1152u, bars + pslot, stream);
        }
        ++issued;
        pslot = pslot + 1 == NS ? 0 : pslot + 1;
    };
    // prologue copies before the wait unless the run has visibly stopped
    // (an L2 read that may be stale; the read after the wait decides)
    const bool early = __shfl_sync(0xffffffffu,
                                   __ldcg(&bs->done) == kRunning && (fin != 0 || __ldcg(&bs->go))
                                       ? 1 : 0, 0) != 0;
    if (early)
        while (more && issued < NS) issue();
    pdl_wait();
    if (!batch_runs(bs, fin == 0)) {
        const unsigned long long drain = global_ns() + kDrainNs;
        for (int k = 0; k < issued; ++k) mbar_wait(bars + k % NS, (uint32_t)(k / NS) & 1u, drain);
        __syncwarp();
        return;
    }
    if (!early)
        while (more && issued < NS) issue();

    float part[4] = {0.0f, 0.0f, 0.0f, 0.0f};
    int sl = sFirst - 1, remS = 0, rpw = 16;
    int row = -1;                 // the lane's chunk row, where it owns one
    float a[LPS][3][4];           // [pass][row of the block][column]
#pragma unroll
    for (int q = 0; q < LPS; ++q)
#pragma unroll
        for (int i = 0; i < 3; ++i)
#pragma unroll
            for (int j = 0; j < 4; ++j) a[q][i][j] = 0.0f;
    auto finish = [&]() {
        // slot l of the 32 is lane l % SPP of pass l / SPP: slots 1 ... SPP / 2
        // apart are LPS times as many lanes apart, slots SPP apart are passes
        for (int o = rpw; o < SPP; o <<= 1)
#pragma unroll
            for (int q = 0; q < LPS; ++q)
#pragma unroll
                for (int i = 0; i < 3; ++i)
#pragma unroll
                    for (int j = 0; j < 4; ++j)
                        a[q][i][j] += __shfl_xor_sync(0xffffffffu, a[q][i][j], o * LPS);
        if (LPS == 2)
#pragma unroll
            for (int i = 0; i < 3; ++i)
#pragma unroll
                for (int j = 0; j < 4; ++j) a[0][i][j] += a[LPS - 1][i][j];
        if (row < 0) return;
        // loads before the stores, behind which they would wait for one another
        float4 src[3];
#pragma unroll
        for (int i = 0; i < 3; ++i)
            src[i] = ld_dep(reinterpret_cast<const float4 *>(RES ? b : x) +
                            ((size_t)row * 3 + i) * LPS + qc);
#pragma unroll
        for (int i = 0; i < 3; ++i) {
            const size_t at = ((size_t)row * 3 + i) * LPS + qc;
            const float4 s4 = src[i];
            float4 o4;
            if (RES) {
                o4 = make_float4(s4.x - a[0][i][0], s4.y - a[0][i][1], s4.z - a[0][i][2],
                                 s4.w - a[0][i][3]);
                part[0] = fmaf(o4.x, o4.x, part[0]);
                part[1] = fmaf(o4.y, o4.y, part[1]);
                part[2] = fmaf(o4.z, o4.z, part[2]);
                part[3] = fmaf(o4.w, o4.w, part[3]);
            } else {
                o4 = make_float4(a[0][i][0], a[0][i][1], a[0][i][2], a[0][i][3]);
                part[0] = fmaf(s4.x, o4.x, part[0]);
                part[1] = fmaf(s4.y, o4.y, part[1]);
                part[2] = fmaf(s4.z, o4.z, part[2]);
                part[3] = fmaf(s4.w, o4.w, part[3]);
            }
            reinterpret_cast<float4 *>(y)[at] = o4;
        }
    };
    auto next_slice = [&]() {
        if (sl >= sFirst) finish();
        ++sl;
        const bool isS = sl < nS;
        rpw = isS ? 32 / kTprS : 32 / kTprX;
        const int ls = isS ? sl : sl - nS;
        const int rl = ls * rpw + sl0;
        row = sl0 < rpw && rl < (isS ? A.S.nRows : A.X.nRows)
                  ? (isS ? A.S.row[rl] : A.X.row[rl]) : -1;
#pragma unroll
        for (int q = 0; q < LPS; ++q)
#pragma unroll
            for (int i = 0; i < 3; ++i)
#pragma unroll
                for (int j = 0; j < 4; ++j) a[q][i][j] = 0.0f;
        if (sl - sFirst < 32) {
            remS = tSteps[warp][sl - sFirst];
        } else {
            const SellDev<float> &P = isS ? A.S : A.X;
            remS = (int)((P.slicePtr[ls + 1] - P.slicePtr[ls]) >> 5);
        }
    };
    // x of the lane's slot of pass q of step t of the stage in ring slot st
    auto gather = [&](int st, int t, int q, float4 (&xv)[3]) {
        const int c = reinterpret_cast<const int *>(ring + st * SB)[t * 32 + q * SPP + sl0];
        const float4 *xc = reinterpret_cast<const float4 *>(x) + (size_t)c * (3 * LPS) + qc;
#pragma unroll
        for (int jc = 0; jc < 3; ++jc) xv[jc] = ld_dep(xc + jc * LPS);
    };
    int sS, cP, curN = 0, cslot = 0, consumed = 0;
    uint32_t cpar = 0u;
    bool ok = true, have = cw.next(C, sS, cP, curN);
    float4 xn[3];
    if (have) {
        ok = __all_sync(0xffffffffu, mbar_wait(bars, 0u, deadline));
        if (ok) gather(0, 0, 0, xn);
    }
    while (ok && have) {
        int nxtN = 0;
        const bool haveN = cw.next(C, sS, cP, nxtN);
        const int nslot = cslot + 1 == NS ? 0 : cslot + 1;
        const uint32_t npar = nslot == 0 ? cpar ^ 1u : cpar;
        const float *vs = reinterpret_cast<const float *>(ring + cslot * SB + C * 128);
#pragma unroll
        for (int t = 0; t < C; ++t) {
            if (t < curN && ok) {
                if (remS == 0) next_slice();
                --remS;
#pragma unroll
                for (int q = 0; q < LPS; ++q) {
                    float4 xc[3] = {xn[0], xn[1], xn[2]};
                    // the next pass: of this step, of the next, or of the next stage
                    if (q + 1 < LPS) {
                        gather(cslot, t, q + 1, xn);
                    } else if (t + 1 < C && t + 1 < curN) {
                        gather(cslot, t + 1, 0, xn);
                    } else if (haveN) {
                        ok = __all_sync(0xffffffffu, mbar_wait_next(bars + nslot, npar, deadline));
                        if (ok) gather(nslot, 0, 0, xn);
                    }
                    const float *v = vs + t * 288 + q * SPP + sl0;
#pragma unroll
                    for (int i = 0; i < 3; ++i)
#pragma unroll
                        for (int jc = 0; jc < 3; ++jc) {
                            const float kv = v[(3 * i + jc) * 32];
                            a[q][i][0] = fmaf(kv, xc[jc].x, a[q][i][0]);
                            a[q][i][1] = fmaf(kv, xc[jc].y, a[q][i][1]);
                            a[q][i][2] = fmaf(kv, xc[jc].z, a[q][i][2]);
                            a[q][i][3] = fmaf(kv, xc[jc].w, a[q][i][3]);
                        }
                }
            }
        }
        if (!ok) break;
        __syncwarp();
        if (more) issue();
        ++consumed;
        cslot = nslot;
        cpar = npar;
        curN = nxtN;
        have = haveN;
    }
    if (ok) {
        if (sl >= sFirst) finish();
    } else {
        // a copy did not land in time: flag it, give the copies still in
        // flight a bounded chance to land, and leave the shared memory
        if (lane == 0) atomicExch(&bs->fault, 1);
        const unsigned long long drain = global_ns() + kDrainNs;
        for (int k = consumed; k < issued; ++k)
            mbar_wait(bars + k % NS, (uint32_t)(k / NS) & 1u, drain);
        __syncwarp();
    }
    // the block's sums: rows sit in slots 0 .. 15 of pass 0, so the trees over
    // the 32 slots start eight slots apart
    __shared__ float wsum[MB][kSpmvWarps];
#pragma unroll
    for (int j = 0; j < 4; ++j) {
#pragma unroll
        for (int o = 8; o > 0; o >>= 1)
            part[j] += __shfl_xor_sync(0xffffffffu, part[j], o * LPS);
        if (lane < LPS) wsum[4 * lane + j][warp] = part[j];
    }
    __syncthreads();
    double blkSum = 0.0;
    if (threadIdx.x < MB) {
        float w[8];
#pragma unroll
        for (int i = 0; i < 8; ++i) w[i] = wsum[threadIdx.x][i];
        blkSum = (double)sum_of_8(w);
    }
    double tot;
    ColumnLoads in;
    if (grid_sum_lanes<MB>(blkSum, args.partials, &bs->ticket[0], tot, blk, nblk,
                           [&] { in.load(bs, m); }) &&
        threadIdx.x < 32) {
        if (!in.fault)
            batch_finalize(bs, m, fin, tot, in);
        else if (threadIdx.x == 0)
            bs->done = kFault;
    }
}

template <int MB, bool RES>
__global__ void __launch_bounds__(kSpmvThreads, 3) k_spmm(SpmmArgs a) {
    extern __shared__ __align__(128) unsigned char smem[];
    spmm_body<MB, RES>(a, (int)blockIdx.x, (int)gridDim.x, smem);
}

template <int MB>
__global__ void __launch_bounds__(kSpmvThreads, 3)
k_spmm_sys(const SpmmArgs *__restrict__ tab, const int *__restrict__ off, int nSys) {
    extern __shared__ __align__(128) unsigned char smem[];
    const int s = sys_of(off, nSys, (int)blockIdx.x);
    const int b0 = __ldg(off + s);
    spmm_body<MB, false>(tab[s], (int)blockIdx.x - b0, __ldg(off + s + 1) - b0, smem);
}

template <int MB>
void launch_spmm(const SpmmArgs &a, cudaStream_t st) {
    const int smem = spmv_smem_bytes<float, 0>();
    launch_pdl(a.fin ? k_spmm<MB, true> : k_spmm<MB, false>, a.A.grid, kSpmvThreads, smem, st, a);
}

template <typename K>
static bool set_smem(K k, int smem) {
    return cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, smem) ==
           cudaSuccess;
}

int spmm_persistent_grid(int MB, int nSlicesTotal) {
    if (!spmm_prepare()) return -1;
    int dev = 0, sms = device_sm_count(), nb = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || sms < 1) return -1;
    const int smem = spmv_smem_bytes<float, 0>();
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(
            &nb, MB == 4 ? k_spmm<4, false> : k_spmm<8, false>, kSpmvThreads, smem) !=
            cudaSuccess ||
        nb < 1)
        return -1;
    const int need = (nSlicesTotal + kSpmvWarps - 1) / kSpmvWarps;
    return std::max(1, std::min(nb * sms, need));
}


// ---- batched restriction + update ---------------------------------------------

// Sums v over the block's threads that share t % MB; thread t = j * NV + c
// (t < MB * NV) receives the total of value c for column j, added warp by
// warp in warp order.  Within a warp the lanes MB, 2 MB, ... apart are added by
// halving exchanges (each keeps half of the values at every level).
template <int MB, int NV>
__device__ __forceinline__ float block_sum_by_column(const float (&in)[NV]) {
    constexpr int P = NV <= 16 ? 16 : 32;
    static_assert(NV <= P, "");
    __shared__ float wred[kThreads / 32][MB][NV];
    const int w = threadIdx.x >> 5, l = threadIdx.x & 31;
    float v[P];
#pragma unroll
    for (int i = 0; i < P; ++i) v[i] = i < NV ? in[i < NV ? i : 0] : 0.0f;
    int base = 0, cnt = P;
#pragma unroll
    for (int o = MB; o < 32; o <<= 1) {
        cnt >>= 1;
        const bool hi = (l & o) != 0;
#pragma unroll
        for (int i = 0; i < P / 2; ++i) {
            if (i >= cnt) break;
            const float send = hi ? v[i] : v[i + cnt];
            const float mine = hi ? v[i + cnt] : v[i];
            v[i] = mine + __shfl_xor_sync(0xffffffffu, send, o);
        }
        if (hi) base += cnt;
    }
    constexpr int kLeft = P / (32 / MB);
#pragma unroll
    for (int i = 0; i < kLeft; ++i)
        if (base + i < NV) wred[w][l % MB][base + i] = v[i];
    __syncthreads();
    float s = 0.0f;
    if ((int)threadIdx.x < MB * NV) {
        const int j = threadIdx.x / NV, c = threadIdx.x % NV;
#pragma unroll
        for (int ww = 0; ww < kThreads / 32; ++ww) s += wred[ww][j][c];
    }
    __syncthreads();
    return s;
}

// A unit's staged set-up data: its rows of Z~ (own rows) then W~ (coupled rows),
// M floats each, then the coupled rows' dofs; at most kUnitRowsBatch rows, half
// as many with 12 columns.
constexpr int kStageBytesB = kUnitRowsBatch * (6 + 1) * (int)sizeof(float);

template <int M>
__device__ __forceinline__ void row_times(const float *z, float rn, float *acc) {
    if (M == 12) {
#pragma unroll
        for (int c = 0; c < M; c += 4) {
            const float4 v = *reinterpret_cast<const float4 *>(z + c);
            acc[c] = fmaf(v.x, rn, acc[c]);
            acc[c + 1] = fmaf(v.y, rn, acc[c + 1]);
            acc[c + 2] = fmaf(v.z, rn, acc[c + 2]);
            acc[c + 3] = fmaf(v.w, rn, acc[c + 3]);
        }
    } else {
#pragma unroll
        for (int c = 0; c < M; c += 2) {
            const float2 v = *reinterpret_cast<const float2 *>(z + c);
            acc[c] = fmaf(v.x, rn, acc[c]);
            acc[c + 1] = fmaf(v.y, rn, acc[c + 1]);
        }
    }
}

// One unit (own rows, then coupled rows, of one box); thread t handles column
// j = t % MB of rows t / MB, t / MB + 256 / MB, ...  acc: Z~^T r (M), W~^T r (M),
// ||r||^2 of its column.  Mode 0 updates the running columns (r' = r -
// alpha_j q, u += alpha_j p) and copies the residual of the others.
//
// The unit's rows of Z~ and W~ and its dof map, shared by the columns, are
// copied into shared memory before the wait for the product (set-up data);
// four rows' entries of r, q, p and u are in flight at a time.  8 columns at
// 32^3 (599 units): 30.4 us before, 18.0 now (four blocks
// per SM).
template <int MB, int M>
__device__ __forceinline__ bool restrict_b_unit(const RestrictBArgs &a, int unit, float *stage,
                                                float *rrs) {
    constexpr int kRowStep = kThreads / MB, U = 4;
    const RowBoxDev &B = a.B;
    const BatchScalars *bs = a.bs;
    const int mode = a.mode;
    const int s = B.unitBox[unit];
    const int j = threadIdx.x % MB, row0 = threadIdx.x / MB;
    const uint64_t keep = l2_keep_policy();
    const int o0 = B.ownRowPtr[s], RO = B.ownRowPtr[s + 1] - o0;
    const int e0 = B.extRowPtr[s], RE = B.extRowPtr[s + 1] - e0;
    const int ob = B.unitOwnBegin[unit], nOwn = B.unitOwnEnd[unit] - ob;
    const int eb = B.unitExtBegin[unit], nExt = mode != 2 ? B.unitExtEnd[unit] - eb : 0;
    float *zs = stage, *ws = stage + (size_t)nOwn * M;
    float *dmap = ws + (size_t)nExt * M;
    {
        const float *Z = B.Z + B.zBase[s] + (ob - o0), *W = B.W + B.wBase[s] + (eb - e0);
        for (int r = threadIdx.x; r < nOwn; r += kThreads)
#pragma unroll
            for (int c = 0; c < M; ++c) cp_keep(zs + r * M + c, Z + (size_t)c * RO + r, keep);
        for (int r = threadIdx.x; r < nExt; r += kThreads) {
#pragma unroll
            for (int c = 0; c < M; ++c) cp_keep(ws + r * M + c, W + (size_t)c * RE + r, keep);
            cp_keep(dmap + r, reinterpret_cast<const float *>(B.extRowDof + eb + r), keep);
        }
    }
    pdl_wait();
    cp_wait_all();
    if (!batch_runs(bs, mode == 0)) return false;
    __syncthreads();
    const int its = bs->its;
    // iteration: the product advanced its, so buffer (its - 1) & 1 is read
    const float *r_cur = mode == 2 ? a.f : (((its & 1) != (mode == 0)) ? a.rB : a.rA);
    float *r_next = mode == 0 ? ((its & 1) ? a.rB : a.rA) : nullptr;
    float *u = a.u;
    const float *p = a.p, *q = a.q;
    const bool run = mode == 0 && col_runs(bs, j, a.m);
    const float alpha = run ? (float)bs->alpha[j] : 0.0f;
    float acc[2 * M + 1];
#pragma unroll
    for (int c = 0; c <= 2 * M; ++c) acc[c] = 0.0f;
    for (int r = row0; r < nOwn; r += U * kRowStep) {
        float rv[U], qv[U], pv[U], uv[U];
#pragma unroll
        for (int i = 0; i < U; ++i) {
            const int ri = r + i * kRowStep;
            const bool ok = ri < nOwn;
            const size_t e = (size_t)(ob + ri) * MB + j;
            rv[i] = ok ? r_cur[e] : 0.0f;
            qv[i] = ok && run ? q[e] : 0.0f;
            pv[i] = ok && run ? p[e] : 0.0f;
            uv[i] = ok && run ? u[e] : 0.0f;
        }
#pragma unroll
        for (int i = 0; i < U; ++i) {
            const int ri = r + i * kRowStep;
            if (ri < nOwn) {
                const size_t e = (size_t)(ob + ri) * MB + j;
                float rn = rv[i];
                if (mode == 0) {
                    if (run) {
                        rn = fmaf(-alpha, qv[i], rn);
                        u[e] = fmaf(alpha, pv[i], uv[i]);
                    }
                    r_next[e] = rn;
                }
                acc[2 * M] = fmaf(rn, rn, acc[2 * M]);
                row_times<M>(zs + ri * M, rn, acc);
            }
        }
    }
    for (int r = row0; r < nExt; r += U * kRowStep) {
        float rv[U], qv[U];
#pragma unroll
        for (int i = 0; i < U; ++i) {
            const int ri = r + i * kRowStep;
            const bool ok = ri < nExt;
            const size_t e = ok ? (size_t)__float_as_int(dmap[ri]) * MB + j : 0;
            rv[i] = ok ? r_cur[e] : 0.0f;
            qv[i] = ok && run ? q[e] : 0.0f;
        }
#pragma unroll
        for (int i = 0; i < U; ++i) {
            const int ri = r + i * kRowStep;
            if (ri < nExt) {
                const float rn = run ? fmaf(-alpha, qv[i], rv[i]) : rv[i];
                row_times<M>(ws + ri * M, rn, acc + M);
            }
        }
    }
    const float tsum = block_sum_by_column<MB, 2 * M + 1>(acc);
    // thread t < MB * (2M + 1): column tj = t / (2M + 1), value tc = t % (2M + 1)
    const int tj = threadIdx.x / (2 * M + 1), tc = threadIdx.x % (2 * M + 1);
    const bool holder = (int)threadIdx.x < MB * (2 * M + 1);
    if (holder && tc == 2 * M) rrs[tj] = tsum;
    const int u0 = B.boxUnit[s], nu = B.boxUnit[s + 1] - u0;
    const int c0 = B.col0[s];
    double *G = a.G, *ZR = a.ZR, *unitPart = a.unitPart;
    float *G32 = a.G32;
    __shared__ float red[MB][2 * 12];
    __shared__ bool lastUnit;
    if (nu == 1) {
        if (holder && tc < 2 * M) red[tj][tc] = tsum;
        __syncthreads();
        if ((int)threadIdx.x < MB * M) {
            const int jj = threadIdx.x / M, c = threadIdx.x % M;
            const double zsum = red[jj][c], wsum = red[jj][M + c];
            G[(size_t)(c0 + c) * MB + jj] = zsum - wsum;
            G32[(size_t)jj * a.gld + c0 + c] = (float)(zsum - wsum);
            if (ZR) ZR[(size_t)(c0 + c) * MB + jj] = zsum;
        }
    } else {
        if (holder && tc < 2 * M)
            unitPart[((size_t)unit * MB + tj) * 24 + tc] = (double)tsum;
        __threadfence();
        __syncthreads();
        if (threadIdx.x == 0)
            lastUnit = atomicAdd(&B.boxTicket[s], 1u) == (unsigned int)nu - 1;
        __syncthreads();
        if (lastUnit) {
            __threadfence();
            if ((int)threadIdx.x < MB * M) {
                const int jj = threadIdx.x / M, c = threadIdx.x % M;
                double zsum = 0.0, wsum = 0.0;
                const double *up = unitPart + ((size_t)u0 * MB + jj) * 24 + c;
                for (int v = 0; v < nu; v += 4) {   // four units' loads in flight
                    double zv[4], wv[4];
#pragma unroll
                    for (int i = 0; i < 4; ++i) {
                        zv[i] = v + i < nu ? __ldcg(up + (size_t)(v + i) * MB * 24) : 0.0;
                        wv[i] = v + i < nu ? __ldcg(up + (size_t)(v + i) * MB * 24 + M) : 0.0;
                    }
                    zsum = v == 0 ? zv[0] : zsum + zv[0];
                    wsum = v == 0 ? wv[0] : wsum + wv[0];
#pragma unroll
                    for (int i = 1; i < 4; ++i)
                        if (v + i < nu) {
                            zsum += zv[i];
                            wsum += wv[i];
                        }
                }
                G[(size_t)(c0 + c) * MB + jj] = zsum - wsum;
                G32[(size_t)jj * a.gld + c0 + c] = (float)(zsum - wsum);
                if (ZR) ZR[(size_t)(c0 + c) * MB + jj] = zsum;
            }
            if (threadIdx.x == 0) B.boxTicket[s] = 0u;
        }
    }
    __syncthreads();
    return true;
}

// mode 0 (iteration): r' = r - alpha_j q, u += alpha_j p for the running
// columns, G from r'; the last block sets rr_j of the running columns and
// holds those at their trigger or at the iteration limit.  mode 1: G and
// rr_j of the columns being replaced from the current residual.  mode 2:
// G = Z~^T f only.
template <int MB>
__device__ __forceinline__ void restrict_b_body(const RestrictBArgs &a, int blk, int nblk) {
    extern __shared__ __align__(16) float stageB[];
    __shared__ float rrs[MB];
    BatchScalars *bs = a.bs;
    const int m = a.m, mode = a.mode;
    const bool went = a.B.menr[a.B.unitBox[blk]] ? restrict_b_unit<MB, 12>(a, blk, stageB, rrs)
                                                 : restrict_b_unit<MB, 6>(a, blk, stageB, rrs);
    if (!went || mode == 2) return;
    // lane j of warp 0 adds column j's ||r||^2
    const double rr = threadIdx.x < MB ? (double)rrs[threadIdx.x] : 0.0;
    double tot;
    ColumnLoads in;
    if (grid_sum_lanes<MB>(rr, a.partials, &bs->ticket[2], tot, blk, nblk,
                           [&] { in.load(bs, m); }) &&
        threadIdx.x < 32) {
        const int j = threadIdx.x;   // one column per lane
        if (mode == 1) {
            if (in.repl) bs->rr[j] = tot;
            return;
        }
        bool any = false;
        if (in.runs) {
            bs->rr[j] = tot;
            bool hold = tot <= in.trig || !isfinite(tot);
            if (in.its >= in.maxIt) {
                hold = true;
                bs->last[j] = 1;
            }
            if (hold) bs->pend[j] = 1;
            any = !hold;
        }
        any = __any_sync(0xffffffffu, any);
        if (j == 0 && !any) bs->done = kConverged;
    }
}

template <int MB>
__global__ void __launch_bounds__(kThreads, 4) k_restrict_b(RestrictBArgs a) {
    restrict_b_body<MB>(a, (int)blockIdx.x, (int)gridDim.x);
}

template <int MB>
__global__ void __launch_bounds__(kThreads, 4)
k_restrict_b_sys(const RestrictBArgs *__restrict__ tab, const int *__restrict__ off, int nSys) {
    const int s = sys_of(off, nSys, (int)blockIdx.x);
    const int b0 = __ldg(off + s);
    restrict_b_body<MB>(tab[s], (int)blockIdx.x - b0, __ldg(off + s + 1) - b0);
}

template <int MB>
void launch_restrict_b(const RestrictBArgs &a, cudaStream_t st) {
    launch_pdl(k_restrict_b<MB>, a.B.nUnits, kThreads, kStageBytesB, st, a);
}

// ---- batched coarse solve NU = E^-1 G -----------------------------------------

// Sums NV values over the warp's lanes by halving exchanges (fixed tree):
// afterwards lane L holds in v[0 .. NV / 32) the totals of values
// (NV / 32) L + i.
template <int NV>
__device__ __forceinline__ void lane_reduce_scatter(float (&v)[NV], int lane) {
    static_assert(NV >= 32 && NV % 32 == 0, "NV: a multiple of 32");
#pragma unroll
    for (int st = 0; st < 5; ++st) {
        const int o = 16 >> st, half = (NV >> st) >> 1;
        const bool hi = (lane & o) != 0;
#pragma unroll
        for (int i = 0; i < half; ++i) {
            const float send = hi ? v[i] : v[i + half];
            const float keep = hi ? v[i + half] : v[i];
            v[i] = keep + __shfl_xor_sync(0xffffffffu, send, o);
        }
    }
}

// rows of E^-1 per block of the batched coarse solve (RB * MB = 32 partial
// sums per lane)
template <int MB>
__host__ __device__ constexpr int coarse_rows_b() { return 32 / MB; }
constexpr int kCoarseChunkB = 128;   // columns of G per chunk (4 per lane)

// One chunk's entries of E^-1 for a lane: 4 consecutive columns (one 16-byte
// load per row, V = 4) or 4 columns 32 apart (V = 1) of each of the RB rows.
template <int RB, int V>
__device__ __forceinline__ void coarse_load_e(const float *Eb, int k, int rLast, int lc, int clen,
                                              int lane, uint64_t keep, float (&e)[RB][4]) {
#pragma unroll
    for (int r = 0; r < RB; ++r) {
        const float *row = Eb + (size_t)min(r, rLast) * k + lc;
        if (V == 4) {
            float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
            if (4 * lane < clen) v = ld_keep(reinterpret_cast<const float4 *>(row + 4 * lane), keep);
            e[r][0] = v.x;
            e[r][1] = v.y;
            e[r][2] = v.z;
            e[r][3] = v.w;
        } else {
#pragma unroll
            for (int q = 0; q < 4; ++q)
                e[r][q] = lane + 32 * q < clen ? ld_keep(row + lane + 32 * q, keep) : 0.0f;
        }
    }
}

// NU = E^-1 G for the MB columns, then the scalars.  mode 0: nu only; mode 1
// (start, every column): rho_j = rr_j + nu_j^T zr_j, beta_j = 0; mode 2
// (iteration, running columns): the same rho_new, beta_j = rho_new / rho_j;
// mode 3 (replacement, the replaced columns): as 2, with beta_j = 0 for a
// column that leaves, that broke down or whose residual the replacement
// lengthened by more than 2x.  A block takes 32 / MB consecutive rows of
// E^-1 and its warps split the columns into segments (multiples of 4).  Each
// warp walks its segment in chunks of kCoarseChunkB columns (the first chunk's
// entries of E^-1 loaded before the wait for the restriction: E^-1 does not
// depend on it); G, stored column by column, is read through L1, where the SM's
// blocks find it after the first.  The partial sums are reduced over the lanes,
// then over the warps in order.  8 columns, k =
// 3150: 29.9 us before (G staged by each warp in shared memory through bulk
// copies and barriers), 22.2 now (three blocks of 80 registers per SM; four of 64
// spill, 39).
template <int MB, int V>
__device__ __forceinline__ void coarse_b_body(const CoarseBArgs &a, int blk, int nblk) {
    constexpr int RB = coarse_rows_b<MB>(), NV = RB * MB, P = NV / 32, CH = kCoarseChunkB;
    __shared__ float red[kWarps][NV];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int k = a.k;
    const int i0 = blk * RB;
    const int seg = (k + 4 * kWarps - 1) / (4 * kWarps) * 4;
    const int l0 = warp * seg, l1 = min(k, l0 + seg);
    const uint64_t keep = l2_keep_policy();
    const float *Eb = a.Einv + (size_t)i0 * k;
    const int rLast = k - 1 - i0;
    float e[RB][4];
    if (l0 < l1) coarse_load_e<RB, V>(Eb, k, rLast, l0, min(CH, l1 - l0), lane, keep, e);
    pdl_wait();
    BatchScalars *bs = a.bs;
    if (!batch_runs(bs, a.mode == 2)) return;
    const int m = a.m, mode = a.mode;
    float acc[NV];
#pragma unroll
    for (int t = 0; t < NV; ++t) acc[t] = 0.0f;
    for (int lc = l0; lc < l1; lc += CH) {
        const int clen = min(CH, l1 - lc);
        if (lc > l0) coarse_load_e<RB, V>(Eb, k, rLast, lc, clen, lane, keep, e);
        const float *g0 = a.G32 + lc;
#pragma unroll
        for (int j = 0; j < MB; ++j) {
            float g[4] = {0.0f, 0.0f, 0.0f, 0.0f};
            if (V == 4) {
                if (4 * lane < clen) {
                    const float4 v =
                        ld_dep(reinterpret_cast<const float4 *>(g0 + (size_t)j * a.gld + 4 * lane));
                    g[0] = v.x;
                    g[1] = v.y;
                    g[2] = v.z;
                    g[3] = v.w;
                }
            } else {
#pragma unroll
                for (int q = 0; q < 4; ++q)
                    if (lane + 32 * q < clen) g[q] = ld_dep(g0 + (size_t)j * a.gld + lane + 32 * q);
            }
#pragma unroll
            for (int r = 0; r < RB; ++r) {
                float t = fmaf(e[r][0], g[0], acc[r * MB + j]);
                t = fmaf(e[r][1], g[1], t);
                t = fmaf(e[r][2], g[2], t);
                acc[r * MB + j] = fmaf(e[r][3], g[3], t);
            }
        }
    }
    lane_reduce_scatter<NV>(acc, lane);
#pragma unroll
    for (int i = 0; i < P; ++i) red[warp][P * lane + i] = acc[i];
    __syncthreads();
    // warp 0 (lane = r * MB + j): nu_i for row i = i0 + r, column j, and its
    // share of nu_j^T zr_j, summed over the block's rows
    static_assert(NV == 32, "one lane per (row, column) of the block");
    double pj = 0.0;
    if (warp == 0) {
        float sum = 0.0f;
#pragma unroll
        for (int w = 0; w < kWarps; ++w) sum += red[w][lane];
        const int r = lane / MB, j = lane % MB, i = i0 + r;
        if (i < k) {
            a.NU[(size_t)i * MB + j] = (double)sum;
            a.NU32[(size_t)i * MB + j] = sum;
            if (mode != 0) pj = (double)sum * a.ZR[(size_t)i * MB + j];
        }
#pragma unroll
        for (int o = MB; o < 32; o <<= 1) pj += __shfl_xor_sync(0xffffffffu, pj, o);
    }
    double tot;
    ColumnLoads in;
    if (grid_sum_lanes<MB>(pj, a.partials, &bs->ticket[3], tot, blk, nblk,
                           [&] { in.load(bs, m); }) &&
        threadIdx.x < 32) {
        const int j = threadIdx.x;   // one column per lane
        if (in.fault) {
            if (j == 0) bs->done = kFault;
        } else if (mode != 0 && j < m &&
                   (mode == 2 ? in.runs : (mode == 1 || in.repl))) {
            const double rho_new = in.rr + tot;
            if (mode == 1 || !in.active ||
                (mode == 3 && (in.broken || in.rr > 4.0 * in.rrRep)))
                bs->beta[j] = 0.0;
            else
                bs->beta[j] = rho_new / in.rho;
            bs->rho[j] = rho_new;
            if (mode == 3) bs->broken[j] = 0;
        }
    }
}

template <int MB, int V>
__global__ void __launch_bounds__(kThreads, MB == 8 ? 3 : 2) k_coarse_b(CoarseBArgs a) {
    coarse_b_body<MB, V>(a, (int)blockIdx.x, (int)gridDim.x);
}

template <int MB>
__global__ void __launch_bounds__(kThreads, MB == 8 ? 3 : 2)
k_coarse_b_sys(const CoarseBArgs *__restrict__ tab, const int *__restrict__ off, int nSys) {
    const int s = sys_of(off, nSys, (int)blockIdx.x);
    const int b0 = __ldg(off + s), nb = __ldg(off + s + 1) - b0;
    const CoarseBArgs &a = tab[s];
    if ((a.k & 3) == 0)
        coarse_b_body<MB, 4>(a, (int)blockIdx.x - b0, nb);
    else
        coarse_b_body<MB, 1>(a, (int)blockIdx.x - b0, nb);
}

int coarse_b_blocks(int k, int MB) {
    const int rb = MB == 4 ? coarse_rows_b<4>() : coarse_rows_b<8>();
    const int grid = (k + rb - 1) / rb;
    return grid > 0 ? grid : 1;
}

template <int MB>
void launch_coarse_b(const CoarseBArgs &a, cudaStream_t st) {
    launch_pdl(a.k % 4 == 0 ? k_coarse_b<MB, 4> : k_coarse_b<MB, 1>, coarse_b_blocks(a.k, MB),
               kThreads, 0, st, a);
}

// ---- batched prolongation -----------------------------------------------------

// mode 0 (iteration, running columns) and mode 3 (replacement, the replaced
// columns): p = y + Z~ nu + beta_j p, 0 for a replaced column that leaves;
// mode 1 (start): p = Z~ nu; mode 2 (start): p = y + Z~ nu.  y is the current
// residual buffer.
//
// A thread's rows are all in flight at once: their rows of Z~ before the wait
// for the coarse solve, their entries of y and p after it, beside those of nu.
// (Not before: in a launch over several systems a held system's replacement, on
// a stream of its own, writes both, and the count that picks y's buffer; 8
// columns at 32^3: 9.2 us, 9.0 with both before the wait, and 16.4 with every
// warp asking L2 first whether the system is held.)
template <int MB, int M>
__device__ __forceinline__ void prolong_b_unit(const ProlongBArgs &a, int unit) {
    constexpr int kRowStep = kThreads / MB, R = (kProlongRowsBatch + kRowStep - 1) / kRowStep;
    const RowBoxDev &B = a.B;
    const BatchScalars *bs = a.bs;
    const int s = B.pUnitBox[unit], mode = a.mode;
    const int j = threadIdx.x % MB, row0 = threadIdx.x / MB;
    const int c0 = B.col0[s], r0 = B.ownRowPtr[s], RO = B.ownRowPtr[s + 1] - r0;
    const float *Z = B.Z + B.zBase[s] - r0;
    const int rb = B.pUnitBegin[unit] + row0, re = B.pUnitEnd[unit];
    const uint64_t keep = l2_keep_policy();
    float z[R][M], yv[R], pv[R];
#pragma unroll
    for (int i = 0; i < R; ++i) {
        const int r = rb + i * kRowStep;
#pragma unroll
        for (int c = 0; c < M; ++c)
            z[i][c] = r < re ? ld_keep(Z + (size_t)c * RO + r, keep) : 0.0f;
    }
    pdl_wait();
    if (!batch_runs(bs, mode == 0)) return;
    bool leaves = false;
    if (mode == 0) {
        if (!col_runs(bs, j, a.m)) return;   // no block-wide step follows
    } else if (mode == 3) {
        if (j >= a.m || !bs->repl[j]) return;
        leaves = !bs->active[j];
    }
    const float *y = (bs->its & 1) ? a.rB : a.rA;
#pragma unroll
    for (int i = 0; i < R; ++i) {
        const int r = rb + i * kRowStep;
        const size_t e = (size_t)r * MB + j;
        yv[i] = r < re && mode != 1 ? y[e] : 0.0f;
        pv[i] = r < re && (mode == 0 || mode == 3) ? a.p[e] : 0.0f;
    }
    const float beta = (mode == 0 || mode == 3) && !leaves ? (float)bs->beta[j] : 0.0f;
    float nv[M];
#pragma unroll
    for (int c = 0; c < M; ++c) nv[c] = a.NU32[(size_t)(c0 + c) * MB + j];
#pragma unroll
    for (int i = 0; i < R; ++i) {
        const int r = rb + i * kRowStep;
        if (r >= re) break;
        float zv = 0.0f;
#pragma unroll
        for (int c = 0; c < M; ++c) zv = fmaf(z[i][c], nv[c], zv);
        const size_t e = (size_t)r * MB + j;
        if (mode == 0 || mode == 3)
            a.p[e] = leaves ? 0.0f : yv[i] + zv + beta * pv[i];
        else if (mode == 1)
            a.p[e] = zv;
        else
            a.p[e] = yv[i] + zv;
    }
}

template <int MB>
__device__ __forceinline__ void prolong_b_body(const ProlongBArgs &a, int blk) {
    if (a.B.menr[a.B.pUnitBox[blk]])
        prolong_b_unit<MB, 12>(a, blk);
    else
        prolong_b_unit<MB, 6>(a, blk);
}

template <int MB>
__global__ void __launch_bounds__(kThreads) k_prolong_b(ProlongBArgs a) {
    prolong_b_body<MB>(a, (int)blockIdx.x);
}

template <int MB>
__global__ void __launch_bounds__(kThreads)
k_prolong_b_sys(const ProlongBArgs *__restrict__ tab, const int *__restrict__ off, int nSys) {
    const int s = sys_of(off, nSys, (int)blockIdx.x);
    prolong_b_body<MB>(tab[s], (int)blockIdx.x - __ldg(off + s));
}

template <int MB>
void launch_prolong_b(const ProlongBArgs &a, cudaStream_t st) {
    launch_pdl(k_prolong_b<MB>, a.B.nPUnits, kThreads, 0, st, a);
}

// Before each iteration over several systems: whether it runs each system
// (running and not held), read once so that every block of the iteration's
// four kernels agrees.  A replacement's last kernel releases the hold after
// its other writes (k_batch_arm), so a gate that sees the release sees them.
__global__ void k_batch_gate(const SpmmArgs *__restrict__ tab, int nSys) {
    for (int s = threadIdx.x; s < nSys; s += blockDim.x) {
        BatchScalars *bs = tab[s].bs;
        const int held = *reinterpret_cast<volatile const int *>(&bs->hold);
        __threadfence();
        const int done = *reinterpret_cast<volatile const int *>(&bs->done);
        bs->go = done == kRunning && !held;
    }
}

// one FP32 iteration of every system of the table: the gate, then four launches
template <int MB>
void launch_iteration_sys(const BatchSysTab &t, cudaStream_t st) {
    k_batch_gate<<<1, 128, 0, st>>>(t.spmm, t.nSys);
    const int smem = spmv_smem_bytes<float, 0>();
    launch_pdl(k_spmm_sys<MB>, t.blocks[0], kSpmvThreads, smem, st, t.spmm, t.off[0], t.nSys);
    launch_pdl(k_restrict_b_sys<MB>, t.blocks[1], kThreads, kStageBytesB, st, t.rst, t.off[1], t.nSys);
    launch_pdl(k_coarse_b_sys<MB>, t.blocks[2], kThreads, 0, st, t.crs, t.off[2], t.nSys);
    launch_pdl(k_prolong_b_sys<MB>, t.blocks[3], kThreads, 0, st, t.pro, t.off[3], t.nSys);
}

// ---- column scalars -------------------------------------------------------------

__device__ __forceinline__ void fresh_slot(Scalars *sc) {
    Scalars z{};
    z.tol2ff = -1.0;
    z.max_it = INT_MAX;
    *sc = z;
}

__global__ void k_batch_slots(Scalars *slots, unsigned mask) {
    const int j = threadIdx.x;
    if (j < kMaxBatch && ((mask >> j) & 1u)) fresh_slot(slots + j);
}

// repl_j = column j is in mask, fresh reduction slots for them; the
// replacement's kernels run (done = kRunning) unless a wait has failed
__global__ void k_batch_open(BatchScalars *bs, Scalars *slots, unsigned mask) {
    const int j = threadIdx.x;
    if (j < kMaxBatch) {
        const int r = (mask >> j) & 1u;
        bs->repl[j] = r;
        if (r) fresh_slot(slots + j);
    }
    if (j == 0 && bs->done != kFault) bs->done = kRunning;
}

// the replaced columns' FP64 residuals ||f_j - K u_j||^2 (slot j, scratch 0):
// a column leaves converged (<= tol^2 ||f_j||^2), not finite, or at its last
// cycle (iteration limit or max_outer replacements)
__global__ void k_batch_judge(BatchScalars *bs, const Scalars *slots, int m) {
    if (threadIdx.x != 0 || blockIdx.x != 0) return;
    for (int j = 0; j < m; ++j) {
        if (!bs->repl[j]) continue;
        if (slots[j].done == kFault) {
            bs->fault = 1;
            bs->done = kFault;
        }
        const double rn2 = slots[j].scratch[0];
        bs->rn2[j] = rn2;
        bs->cycles[j] += 1;
        bs->rrRep[j] = bs->rr[j];
        if (!isfinite(rn2)) {
            bs->active[j] = 0;
            bs->outcome[j] = kColBad;
        } else if (rn2 <= bs->tol * bs->tol * bs->ff[j]) {
            bs->active[j] = 0;
        } else if (bs->last[j] || bs->cycles[j] >= bs->max_outer) {
            bs->active[j] = 0;
            bs->outcome[j] = kColLimit;
        }
    }
}

// Triggers of the columns being replaced (first: every column, after the
// start): the next replacement of column j once its recursive residual has
// dropped by delta (squared: delta2), or to the floor below which the FP32
// recursion no longer tracks the true residual (a quarter of the target
// relative to the last replacement's ratio of recursive to true residual),
// but at least by kMinGroupDrop2; then release them.
__global__ void k_batch_arm(BatchScalars *bs, int m, int first) {
    if (threadIdx.x != 0 || blockIdx.x != 0) return;
    bool any = false;
    for (int j = 0; j < m; ++j) {
        if (first || bs->repl[j]) {
            if (!bs->active[j]) {
                bs->trig[j] = -1.0;
            } else if (first) {
                bs->trig[j] = bs->delta2 * bs->rr[j];
            } else {
                const double sj = bs->scale[j], rr = bs->rr[j], tol = bs->tol;
                const double gamma2 = rr / (sj * sj * bs->rn2[j]);
                const double f1 = 0.25 * tol * tol * bs->ff[j] * sj * sj * gamma2;
                const double f2 = kMinGroupDrop2 * rr;
                const double floor2 = f2 < f1 ? f2 : f1;
                const double t = bs->delta2 * rr;
                bs->trig[j] = floor2 > t ? floor2 : t;
            }
            bs->pend[j] = 0;
            bs->last[j] = 0;
            bs->repl[j] = 0;
        }
        any |= bs->active[j] && !bs->pend[j];
    }
    if (bs->done != kFault) bs->done = any ? kRunning : kConverged;
    __threadfence();   // every write of the replacement before the release
    *reinterpret_cast<volatile int *>(&bs->hold) = 0;
}

__global__ void k_batch_hold(BatchScalars *bs) {
    if (threadIdx.x == 0 && blockIdx.x == 0) bs->hold = 1;
}

void launch_batch_slots(Scalars *slots, unsigned mask, cudaStream_t st) {
    k_batch_slots<<<1, 32, 0, st>>>(slots, mask);
}
void launch_batch_open(BatchScalars *bs, Scalars *slots, unsigned mask, cudaStream_t st) {
    k_batch_open<<<1, 32, 0, st>>>(bs, slots, mask);
}
void launch_batch_judge(BatchScalars *bs, const Scalars *slots, int m, cudaStream_t st) {
    k_batch_judge<<<1, 32, 0, st>>>(bs, slots, m);
}
void launch_batch_arm(BatchScalars *bs, int m, int first, cudaStream_t st) {
    k_batch_arm<<<1, 32, 0, st>>>(bs, m, first);
}
void launch_batch_hold(BatchScalars *bs, cudaStream_t st) { k_batch_hold<<<1, 32, 0, st>>>(bs); }

// ---- FP64 <-> FP32 transforms of several columns --------------------------------

// out[(ot[I] + i) * MB + j] = scale_j (L^-1 r_j)_i for the columns being
// replaced (repl_j; every column at the start), 0 for those that leave and
// for padding columns; r_j = r + j * ldr in the caller's numbering (nat).
// out is the current residual buffer (outA, or outB when its is odd).  One
// thread per (node, column).
template <int MB>
__global__ void k_fwd_scale_b(int nNodes, int m, const int *nat, const int *ot, FacDev F,
                              const double *r, long long ldr, const BatchScalars *bs,
                              float *outA, float *outB) {
    const long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    if (t >= (long long)nNodes * MB) return;
    const int I = (int)(t / MB), j = (int)(t % MB);
    if (j < m && !bs->repl[j]) return;
    float *out = (bs->its & 1) ? outB : outA;
    const int b = nat[I + 1] - nat[I], d0 = nat[I], o0 = ot[I];
    const bool on = j < m && bs->active[j];
    const double sj = on ? bs->scale[j] : 0.0;
    const int q = F.nodeIdx[I];
    with_node_size(b, [&](auto Bc) {
        constexpr int B = decltype(Bc)::value;
        double x[B];
#pragma unroll
        for (int i = 0; i < B; ++i) x[i] = on ? r[j * ldr + d0 + i] : 0.0;
        if (on) fwd_solve_fixed<B>(F, q, x);
#pragma unroll
        for (int i = 0; i < B; ++i) out[(size_t)(o0 + i) * MB + j] = (float)(sj * x[i]);
    });
}

// u_j += (L^-T ut_j)_i / scale_j, then ut_j = 0, for the columns being
// replaced; one thread per (node, column)
template <int MB>
__global__ void k_bwd_accum_b(int nNodes, int m, const int *nat, const int *in, FacDev F,
                              float *ut, const BatchScalars *bs, double *u, long long ldu) {
    // one division per column and block, not one per thread (FP64)
    __shared__ double inv[MB];
    if (threadIdx.x < MB) inv[threadIdx.x] = 1.0 / bs->scale[threadIdx.x];
    __syncthreads();
    const long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    if (t >= (long long)nNodes * MB) return;
    const int I = (int)(t / MB), j = (int)(t % MB);
    if (j >= m || !bs->repl[j]) return;
    const int b = nat[I + 1] - nat[I], d0 = in[I], o0 = nat[I];
    const int q = F.nodeIdx[I];
    with_node_size(b, [&](auto Bc) {
        constexpr int B = decltype(Bc)::value;
        double x[B], uv[B];
#pragma unroll
        for (int i = 0; i < B; ++i) {
            x[i] = (double)ut[(size_t)(d0 + i) * MB + j];
            uv[i] = u[j * ldu + o0 + i];
        }
        bwd_solve_fixed<B>(F, q, x);
#pragma unroll
        for (int i = 0; i < B; ++i) {
            ut[(size_t)(d0 + i) * MB + j] = 0.0f;
            u[j * ldu + o0 + i] = uv[i] + inv[j] * x[i];
        }
    });
}

template <int MB>
void launch_fwd_scale_b(int nNodes, int m, const int *nat, const int *ot, const FacDev &F,
                        const double *r, long long ldr, const BatchScalars *bs, float *outA,
                        float *outB, cudaStream_t st) {
    const long long nt = (long long)nNodes * MB;
    k_fwd_scale_b<MB><<<(unsigned)((nt + 127) / 128), 128, 0, st>>>(nNodes, m, nat, ot, F, r, ldr,
                                                                     bs, outA, outB);
}

template <int MB>
void launch_bwd_accum_b(int nNodes, int m, const int *nat, const int *in, const FacDev &F,
                        float *ut, const BatchScalars *bs, double *u, long long ldu,
                        cudaStream_t st) {
    const long long nt = (long long)nNodes * MB;
    k_bwd_accum_b<MB><<<(unsigned)((nt + 127) / 128), 128, 0, st>>>(nNodes, m, nat, in, F, ut, bs,
                                                                     u, ldu);
}

// dynamic shared memory limits of the batched kernels (once per process)
bool spmm_prepare() {
    const int smem = spmv_smem_bytes<float, 0>();
    return set_smem(k_spmm<4, false>, smem) && set_smem(k_spmm<4, true>, smem) &&
           set_smem(k_spmm<8, false>, smem) && set_smem(k_spmm<8, true>, smem) &&
           set_smem(k_spmm_sys<4>, smem) && set_smem(k_spmm_sys<8>, smem);
}

#define XDCG_BATCH_INST(MB)                                                                    \
    template void launch_spmm<MB>(const SpmmArgs &, cudaStream_t);                             \
    template void launch_restrict_b<MB>(const RestrictBArgs &, cudaStream_t);                  \
    template void launch_coarse_b<MB>(const CoarseBArgs &, cudaStream_t);                      \
    template void launch_prolong_b<MB>(const ProlongBArgs &, cudaStream_t);                    \
    template void launch_iteration_sys<MB>(const BatchSysTab &, cudaStream_t);                 \
    template void launch_fwd_scale_b<MB>(int, int, const int *, const int *, const FacDev &,   \
                                         const double *, long long, const BatchScalars *,      \
                                         float *, float *, cudaStream_t);                      \
    template void launch_bwd_accum_b<MB>(int, int, const int *, const int *, const FacDev &,   \
                                         float *, const BatchScalars *, double *, long long,    \
                                         cudaStream_t);
XDCG_BATCH_INST(4)
XDCG_BATCH_INST(8)
#undef XDCG_BATCH_INST

}  // namespace xdcg

// Box-level kernels of Algorithm 3: the restriction g = Z^T r - W^T y
// (right-hand sides of both coarse solves, merged) and the prolongation
// p = y + Z nu (+ beta p).
//
// Z is applied matrix-free from the node position relative to the box
// centre (Eqs. dcg_deflation_space, dcg_deflation_space_enr_std,
// dcg_deflation_space_enr_enr) in the FP64 path (or by value, when the caller
// gave Z), and from the explicit scaled basis Z~ = L^T Z in the FP32
// block-scaled path.
#include <algorithm>

#include "cache.cuh"
#include "reduce.cuh"

namespace xdcg {

// ---- restriction (FP64) ------------------------------------------------------
//
// One CTA per six coarse columns of a box (BoxDev::unit), the units with the
// most rows first.  The lanes of a warp form five groups of six lanes; lane
// (group, column c) accumulates column c over every slots-th node of the box
// (box_slots), so every lane keeps one running sum and the only cross-lane
// step is a short, fixed-order sum in shared memory.  Warps 0-3 take Z^T r
// over the box's own nodes, warps 4-7 W^T y over the nodes coupled to it.
//
// What bounds it is not the 42 MB of W (48^3) but the chains: a lane's sum is
// a serial chain of FP64 operations.  So a chain touches no dependent global
// load: the entries of r and y are gathered into shared memory by the whole
// CTA, a chunk at a time, the positions of the nodes' blocks likewise, and a
// lane keeps kAhead groups of W (three rows of a node each; an enriched node
// is two or five groups, so all lanes do the same thing) in flight.  Records,
// node geometry and the first groups of W are set-up data, loaded before the
// wait for the kernel that wrote r and y.  A box of twelve columns is two
// CTAs because the FP64 units of one SM need ~25 us for the 3,591 coupled rows
// of the largest box at 48^3, all twelve columns.
//
// 48^3 (512 boxes, 373k dofs): 82.9 us before (one CTA of 128 threads per box,
// one warp set doing both sums, loads exposed per four nodes, a six-way
// divergent switch per node), 47.8 now; 24^3 (64 boxes): 56.6 before, 28.8 now;
// 12^3 (8 boxes): 61.9 before, 30.9 now.  Two CTAs per SM: with three the longest
// chains share their SM's FP64 units with more of the others (57.5 us at 48^3),
// with one the gathers are exposed (58.9).

constexpr int kBoxThreads = 256;
constexpr int kExtChunk = 880, kOwnChunk = 240;   // records / nodes per chunk: multiples of 20, 8
constexpr int kOwnRecChunk = 560;                 // records of Z by value (the same memory)
constexpr int kAhead = 12;                         // groups of W in flight per lane

struct OwnGeo {
    double a[kOwnChunk * 6], x[kOwnChunk * 3];
    signed char h[kOwnChunk];                     // H(x_I), or 2 H where the node has jump dofs
};
struct OwnRec {
    double v[kOwnRecChunk * 3];
    int off[kOwnRecChunk];
};

// One lane's share of sum_I blk_I^T v_I over nSteps steps of a staged chunk,
// a record per slot and step (off: block position / 6, -1 for padding; v: three
// entries per record, zero for padding, whose products then add nothing: no
// branch stands between the steps of the chain).
struct RecChain {
    double w[kAhead][3];
    const double *base;
    int M, slots, slot;
    __device__ __forceinline__ void load(int u, int step, const int *off, int nSteps) {
        const int o = step < nSteps ? off[slot + step * slots] : -1;
        const double *b = base + 6LL * max(o, 0);
#pragma unroll
        for (int i = 0; i < 3; ++i) w[u][i] = o >= 0 ? __ldg(b + i * M) : 0.0;
    }
    __device__ __forceinline__ void start(const int *off, int nSteps) {
#pragma unroll
        for (int u = 0; u < kAhead; ++u) load(u, u, off, nSteps);
    }
    __device__ __forceinline__ void run(const int *off, const double *v, int nSteps, double &acc) {
        int st = 0;
        for (; st + kAhead <= nSteps; st += kAhead) {
#pragma unroll
            for (int u = 0; u < kAhead; ++u) {
                const double *x = v + 3 * (slot + (st + u) * slots);
#pragma unroll
                for (int i = 0; i < 3; ++i) acc = fma(w[u][i], x[i], acc);
                load(u, st + u + kAhead, off, nSteps);
            }
        }
#pragma unroll
        for (int u = 0; u < kAhead; ++u) {
            if (st + u >= nSteps) break;
            const double *x = v + 3 * (slot + (st + u) * slots);
#pragma unroll
            for (int i = 0; i < 3; ++i) acc = fma(w[u][i], x[i], acc);
        }
    }
};

// Column c (0..5) of R(x)^T a, R the rigid block of Eq. dcg_deflation_space:
// a_c for c < 3, then -z a1 + y a2, z a0 - x a2, -y a0 + x a1, the pair of
// positions and entries picked per column so that the columns of a warp do
// not diverge.
__device__ __forceinline__ double rigid_col(int c, const double *a, const double *x) {
    const double P = c == 3 ? x[1] : (c == 4 ? x[2] : x[0]);
    const double s = c == 3 ? a[2] : (c == 4 ? a[0] : a[1]);
    const double Q = c == 3 ? -x[2] : (c == 4 ? -x[0] : -x[1]);
    const double q = c == 3 ? a[1] : (c == 4 ? a[2] : a[0]);
    const double lin = __fma_rn(P, s, __dmul_rn(Q, q));
    return c == 0 ? a[0] : (c == 1 ? a[1] : (c == 2 ? a[2] : lin));
}

template <bool EXPL>
__global__ void __launch_bounds__(kBoxThreads, 2)
k_restrict(BoxDev<double> B, const double *a, const double *b, int withW, double *g, double *zr,
           const Scalars *sc) {
    __shared__ double sv[kExtChunk * 3];
    __shared__ int soff[kExtChunk];
    __shared__ union {
        OwnGeo geo;
        OwnRec rec;
    } own;
    __shared__ double red[2][20 * 6];
    const int2 unit = B.unit[blockIdx.x];
    const int s = unit.x, M = B.menr[s] ? 12 : 6, slots = box_slots(M);
    const bool enr = unit.y != 0;                 // the enriched six columns
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const bool ownWarp = warp < 4;
    // eight slots fill two warps: the own nodes' on another pair of the SM's
    // four FP64 units than the coupled nodes'
    const int c = lane % 6, slot = ((warp + (ownWarp && M == 12 ? 2 : 0)) & 3) * 5 + lane / 6;
    const bool act = lane < 30 && slot < slots;
    const long long e0 = B.ext.ptr[s], nExt = withW ? B.ext.ptr[s + 1] - e0 : 0;
    const int o0 = B.ownPtr[s];
    const long long z0 = EXPL ? B.own.ptr[s] : 0;
    const long long nOwn = EXPL ? B.own.ptr[s + 1] - z0 : B.ownPtr[s + 1] - o0;
    const int CE = kExtChunk, CO = EXPL ? kOwnRecChunk : kOwnChunk;
    constexpr int kE = (kExtChunk + kBoxThreads - 1) / kBoxThreads;
    constexpr int kO = ((EXPL ? kOwnRecChunk : kOwnChunk) + kBoxThreads - 1) / kBoxThreads;
    int ed[kE], od[kO];
    bool jump[kO];
    double acc = 0.0;
    RecChain ch;
    ch.base = (EXPL && ownWarp ? B.Zt : B.W) + c + (enr ? 6 : 0);
    ch.M = M;
    ch.slots = slots;
    ch.slot = slot;
    const int *choff = EXPL && ownWarp ? own.rec.off : soff;
    const bool records = act && (EXPL || !ownWarp);
    for (long long ch0 = 0;; ++ch0) {
        const int ne = (int)max(0LL, min((long long)CE, nExt - ch0 * CE));
        const int no = (int)max(0LL, min((long long)CO, nOwn - ch0 * CO));
        if (ch0 > 0 && ne == 0 && no == 0) break;
        if (ch0 > 0) __syncthreads();             // the previous chunk has been used
        // set-up data of the chunk
#pragma unroll
        for (int q = 0; q < kE; ++q) {
            const int i = threadIdx.x + q * kBoxThreads;
            ed[q] = -1;
            if (i < ne) {
                const int2 r = __ldg(B.ext.rec + e0 + ch0 * CE + i);
                ed[q] = r.y;
                soff[i] = r.y >= 0 ? r.x : -1;
            }
        }
#pragma unroll
        for (int q = 0; q < kO; ++q) {
            const int i = threadIdx.x + q * kBoxThreads;
            od[q] = -1;
            jump[q] = false;
            if (i < no) {
                if (EXPL) {
                    const int2 r = __ldg(B.own.rec + z0 + ch0 * CO + i);
                    od[q] = r.y;
                    own.rec.off[i] = r.y >= 0 ? r.x : -1;
                } else {
                    const long long t = o0 + ch0 * CO + i;
                    od[q] = B.ownDof[t];
                    jump[q] = enr && B.ownB[t] == 6;
                    own.geo.h[i] = (signed char)(B.ownH[t] * (jump[q] ? 2 : 1));
#pragma unroll
                    for (int e = 0; e < 3; ++e) own.geo.x[3 * i + e] = B.ownX[3 * t + e];
                }
            }
        }
        __syncthreads();
        const int nSteps = (ownWarp ? no : ne) / slots;   // of a list of records
        if (records) ch.start(choff, nSteps);
        if (ch0 == 0) {
            pdl_wait();
            if (sc && sc->done != kRunning) return;
        }
        // the entries of r and y
#pragma unroll
        for (int q = 0; q < kE; ++q) {
            const int i = threadIdx.x + q * kBoxThreads;
            if (i < ne)
#pragma unroll
                for (int e = 0; e < 3; ++e) sv[3 * i + e] = ed[q] >= 0 ? b[ed[q] + e] : 0.0;
        }
#pragma unroll
        for (int q = 0; q < kO; ++q) {
            const int i = threadIdx.x + q * kBoxThreads;
            if (i < no)
#pragma unroll
                for (int e = 0; e < 3; ++e) {
                    if (EXPL) {
                        own.rec.v[3 * i + e] = od[q] >= 0 ? a[od[q] + e] : 0.0;
                    } else {
                        own.geo.a[6 * i + e] = a[od[q] + e];
                        if (jump[q]) own.geo.a[6 * i + 3 + e] = a[od[q] + 3 + e];
                    }
                }
        }
        __syncthreads();
        if (records) {
            ch.run(choff, EXPL && ownWarp ? own.rec.v : sv, nSteps, acc);
        } else if (act && !enr) {
#pragma unroll 4
            for (int i = slot; i < no; i += slots)
                acc += rigid_col(c, own.geo.a + 6 * i, own.geo.x + 3 * i);
        } else if (act) {
#pragma unroll 2
            for (int i = slot; i < no; i += slots) {
                const int h = own.geo.h[i];
                double z = rigid_col(c, own.geo.a + 6 * i, own.geo.x + 3 * i);
                z = h > 0 ? z : -z;
                if (h == 2 || h == -2)
                    z += rigid_col(c, own.geo.a + 6 * i + 3, own.geo.x + 3 * i);
                acc += z;
            }
        }
    }
    if (act) red[ownWarp ? 0 : 1][slot * 6 + c] = acc;
    __shared__ double wtot[6];
    __syncthreads();
    double tot = 0.0;
    if (warp < 2 && lane < 6) {
#pragma unroll
        for (int q = 0; q < 20; ++q)
            if (q < slots) tot += red[warp][q * 6 + lane];
        if (warp == 1) wtot[lane] = tot;
    }
    __syncthreads();
    if (threadIdx.x < 6) {
        const int i = B.col0[s] + (enr ? 6 : 0) + threadIdx.x;
        g[i] = tot - wtot[threadIdx.x];
        if (zr) zr[i] = tot;
    }
}

void launch_restrict(const BoxDev<double> &B, const double *a, const double *b, int withW,
                     double *g, double *zr, const Scalars *sc, cudaStream_t st) {
    // Z by value (B.Zt) or from the geometry
    launch_pdl(B.Zt ? k_restrict<true> : k_restrict<false>, B.nUnits, kBoxThreads, 0, st, B, a, b,
               withW, g, zr, sc);
}


// ---- prolongation (FP64) -----------------------------------------------------

// mode 0: p = y + Z nu + beta p;  mode 1: p = Z nu;  mode 2: p = y + Z nu
template <typename T>
__device__ __forceinline__ T emitted(T yv, T pv, T zv, int mode, T beta) {
    return mode == 0 ? yv + zv + beta * pv : (mode == 1 ? zv : yv + zv);
}

constexpr int kProThreads = 128;

// One thread per own node, parts CTAs per box (so that a box of several
// hundred nodes is one round of threads).  A node's geometry is loaded before
// the wait for the coarse solve, its entries of y and p after it, three at a
// time, loads first.  (Before the wait they would have to come from L2, where
// the three loads of a node's entries share no line of L1: solves at 1e-8
// 23.290 ms so, 23.249 as it is, at 48^3; 4.716 and 4.695 at 12^3.)
template <int M, bool EXPL>
__device__ __forceinline__ void prolong_box(const BoxDev<double> &B, int s, int t, int step,
                                            const double *nu, const double *y, double *p,
                                            int mode, const Scalars *sc) {
    const int o1 = B.ownPtr[s + 1], c0 = B.col0[s];
    int d0 = 0, bI = 0;
    double X = 0.0, Y = 0.0, Z = 0.0, H = 0.0, yv[3], pv[3];
    auto load3 = [&](int d) {
#pragma unroll
        for (int i = 0; i < 3; ++i) {
            yv[i] = mode != 1 ? y[d + i] : 0.0;
            pv[i] = mode == 0 ? p[d + i] : 0.0;
        }
    };
    auto load_node = [&]() {
        d0 = B.ownDof[t];
        bI = B.ownB[t];
        if (!EXPL) {
            X = B.ownX[3 * (size_t)t];
            Y = B.ownX[3 * (size_t)t + 1];
            Z = B.ownX[3 * (size_t)t + 2];
            H = (double)B.ownH[t];
        }
    };
    if (t < o1) load_node();
    pdl_wait();
    if (blockIdx.x == 0 && blockIdx.y == 0 && threadIdx.x == 0) report(sc);
    if (sc->done != kRunning) return;
    if (t >= o1) return;
    load3(d0);
    const double beta = sc->beta;
    double n[M];
#pragma unroll
    for (int c = 0; c < M; ++c) n[c] = nu[c0 + c];
    while (true) {
        double v[3], ve[3] = {0.0, 0.0, 0.0};
        if (!EXPL) {
            v[0] = n[0] + Z * n[4] - Y * n[5];
            v[1] = n[1] - Z * n[3] + X * n[5];
            v[2] = n[2] + Y * n[3] - X * n[4];
            if (M == 12) {
                ve[0] = n[6] + Z * n[10] - Y * n[11];
                ve[1] = n[7] - Z * n[9] + X * n[11];
                ve[2] = n[8] + Y * n[9] - X * n[10];
#pragma unroll
                for (int i = 0; i < 3; ++i) v[i] += H * ve[i];
            }
        }
        for (int i0 = 0; i0 < bI; i0 += 3) {
            if (i0) load3(d0 + i0);
            double zv[3];
            if (EXPL) {
                const double *Zb = B.Zt + B.ownZ[t] + (size_t)i0 * M;
                double z[3][M];
#pragma unroll
                for (int i = 0; i < 3; ++i)
#pragma unroll
                    for (int c = 0; c < M; ++c) z[i][c] = Zb[i * M + c];
#pragma unroll
                for (int i = 0; i < 3; ++i) {
                    zv[i] = 0.0;
#pragma unroll
                    for (int c = 0; c < M; ++c) zv[i] = fma(z[i][c], n[c], zv[i]);
                }
            } else {
                // standard rows; jump rows (bI = 6); branch rows: 0
#pragma unroll
                for (int i = 0; i < 3; ++i)
                    zv[i] = i0 == 0 ? v[i] : (bI == 6 && M == 12 ? ve[i] : 0.0);
            }
#pragma unroll
            for (int i = 0; i < 3; ++i)
                p[d0 + i0 + i] = emitted(yv[i], pv[i], zv[i], mode, beta);
        }
        t += step;
        if (t >= o1) return;
        load_node();
        load3(d0);
    }
}

// Bound by latency (15 MB at 48^3): 21.6 us before (one CTA of 128 threads per
// box, each entry's loads behind the previous entry's store), 13.3 now;
// 12^3: 17.7 before, 10.2 now.
template <bool EXPL>
__global__ void __launch_bounds__(kProThreads)
k_prolong(BoxDev<double> B, const double *nu, const double *y, double *p, int mode, Scalars *sc) {
    const int s = blockIdx.x, step = kProThreads * gridDim.y;
    const int t = B.ownPtr[s] + blockIdx.y * kProThreads + threadIdx.x;
    if (B.menr[s])
        prolong_box<12, EXPL>(B, s, t, step, nu, y, p, mode, sc);
    else
        prolong_box<6, EXPL>(B, s, t, step, nu, y, p, mode, sc);
}

void launch_prolong(const BoxDev<double> &B, const double *nu, const double *y, double *p,
                    int mode, Scalars *sc, cudaStream_t st) {
    // enough CTAs per box for one round over an average box, and for a box
    // of up to twice the average in a second
    const int parts = std::min(16, std::max(1, (B.nOwn / B.nBox + kProThreads) / kProThreads));
    launch_pdl(B.Zt ? k_prolong<true> : k_prolong<false>, dim3(B.nBox, parts), kProThreads, 0, st,
               B, nu, y, p, mode, sc);
}


// ---- row-parallel box kernels of the block-scaled FP32 path -----------------

constexpr int kRowThreads = 256;

// A thread's rows of a unit that are in flight before the wait: OWN own rows
// and EXT coupled rows (the later ones are loaded in batches after it).  Their
// rows of Z~ and W~ (set-up data) are copied asynchronously into shared memory
// (kStageFloats per thread), their entries of r, p and u, which the kernel
// before the product wrote at the latest, and their dof map go to registers.
// Units of a large system share an SM by fours; with at most one unit per SM
// the whole unit is in flight.
template <int M, bool FEW> struct RowStage;
template <> struct RowStage<6, false> { static constexpr int OWN = 3, EXT = 6; };
template <> struct RowStage<12, false> { static constexpr int OWN = 1, EXT = 2; };
template <> struct RowStage<6, true> { static constexpr int OWN = 5, EXT = 9; };
template <> struct RowStage<12, true> { static constexpr int OWN = 4, EXT = 7; };
template <bool FEW>
constexpr int kStageFloats = FEW ? 132 : 54;

// One restriction unit: own rows [ownBegin, ownEnd) and coupled rows
// [extBegin, extEnd) of one box (most boxes are one unit).  acc[0..M): Z~^T r
// over its own rows, acc[M..2M): W~^T r over its coupled rows, acc[2M]:
// ||r||^2; returns (in thread 0) the unit's ||r||^2.  YV (caller blocks, mode
// 3): the coupled rows take W~^T of y = M~^-1 r.  alpha_of() waits for the
// previous kernel and gives alpha, or false if there is nothing to do.
template <int M, bool YV, bool FEW, typename F>
__device__ __forceinline__ bool restrict_update_unit(const RowBoxDev &B, int unit, float *u,
                                                     const float *r_cur, float *r_next,
                                                     const float *p, const float *q,
                                                     const float *yv, int mode, double *g,
                                                     double *zr, const Scalars *sc, float *stage,
                                                     float (*red)[32], F &&alpha_of,
                                                     float &rr) {
    constexpr int OWN = RowStage<M, FEW>::OWN, EXT = RowStage<M, FEW>::EXT, T = kRowThreads;
    static_assert((OWN + EXT) * M <= kStageFloats<FEW>, "");
    const int s = B.unitBox[unit], tid = threadIdx.x;
    const int o0 = B.ownRowPtr[s], RO = B.ownRowPtr[s + 1] - o0;
    const int e0 = B.extRowPtr[s], RE = B.extRowPtr[s + 1] - e0;
    const int oBegin = B.unitOwnBegin[unit] + tid, oEnd = B.unitOwnEnd[unit];
    const int eBegin = B.unitExtBegin[unit] + tid;
    const int eEnd = mode != 2 ? B.unitExtEnd[unit] : 0;
    const float *Z = B.Z + B.zBase[s] - o0, *W = B.W + B.wBase[s] - e0;
    const uint64_t keep = l2_keep_policy();
    float *zs = stage + tid, *ws = stage + OWN * M * T + tid;
    int ed[EXT];
    float ro[OWN], po[OWN], uo[OWN], re[EXT];
    // set-up data, and in an iteration the vectors that the product only read
    auto load_static = [&]() {
#pragma unroll
        for (int i = 0; i < EXT; ++i)
            ed[i] = eBegin + i * T < eEnd ? ld_keep(B.extRowDof + eBegin + i * T, keep) : -1;
#pragma unroll
        for (int i = 0; i < OWN; ++i)
            if (oBegin + i * T < oEnd)
#pragma unroll
                for (int c = 0; c < M; ++c)
                    cp_keep(zs + (i * M + c) * T, Z + (size_t)c * RO + oBegin + i * T, keep);
#pragma unroll
        for (int i = 0; i < EXT; ++i)
            if (ed[i] >= 0)
#pragma unroll
                for (int c = 0; c < M; ++c)
                    cp_keep(ws + (i * M + c) * T, W + (size_t)c * RE + eBegin + i * T, keep);
    };
    auto load_vectors = [&]() {
#pragma unroll
        for (int i = 0; i < OWN; ++i) {
            const int r = oBegin + i * T;
            const bool ok = r < oEnd;
            ro[i] = ok ? ld_early(r_cur + r) : 0.0f;
            po[i] = ok && mode == 0 ? ld_early(p + r) : 0.0f;
            uo[i] = ok && mode == 0 ? ld_early(u + r) : 0.0f;
        }
#pragma unroll
        for (int i = 0; i < EXT; ++i) re[i] = ed[i] >= 0 ? ld_early((YV ? yv : r_cur) + ed[i]) : 0.0f;
    };
    // launches queued past a stop load nothing early (a read that may be
    // stale; the one after the wait decides)
    const bool early = __ldcg(&sc->done) == kRunning;
    if (early) {
        load_static();
        if (mode == 0) load_vectors();
    }
    pdl_wait();
    if (sc->done != kRunning) {
        cp_wait_all();
        return false;
    }
    if (!early) load_static();
    if (!early || mode != 0) load_vectors();
    float qo[OWN], qe[EXT];
    if (mode == 0) {
#pragma unroll
        for (int i = 0; i < OWN; ++i) qo[i] = oBegin + i * T < oEnd ? q[oBegin + i * T] : 0.0f;
        if (!YV)
#pragma unroll
            for (int i = 0; i < EXT; ++i) qe[i] = ed[i] >= 0 ? q[ed[i]] : 0.0f;
    }
    float alpha = 0.0f;
    if (!alpha_of(alpha)) {
        cp_wait_all();
        return false;
    }
    float acc[2 * M + 1];
#pragma unroll
    for (int c = 0; c <= 2 * M; ++c) acc[c] = 0.0f;
    cp_wait_all();
#pragma unroll
    for (int i = 0; i < OWN; ++i) {
        const int r = oBegin + i * T;
        if (r < oEnd) {
            float rn = ro[i];
            if (mode == 0) {
                rn = fmaf(-alpha, qo[i], rn);
                r_next[r] = rn;
                u[r] = fmaf(alpha, po[i], uo[i]);
            }
            acc[2 * M] = fmaf(rn, rn, acc[2 * M]);
#pragma unroll
            for (int c = 0; c < M; ++c) acc[c] = fmaf(zs[(i * M + c) * T], rn, acc[c]);
        }
    }
    // the remaining own rows, two at a time, loads first
    for (int r = oBegin + OWN * T; r < oEnd; r += 2 * T) {
        float z[2][M], rv[2], pv[2], uv[2], qv[2];
#pragma unroll
        for (int i = 0; i < 2; ++i) {
            const int rr2 = r + i * T;
            const bool ok = rr2 < oEnd;
            rv[i] = ok ? r_cur[rr2] : 0.0f;
            qv[i] = ok && mode == 0 ? q[rr2] : 0.0f;
            pv[i] = ok && mode == 0 ? p[rr2] : 0.0f;
            uv[i] = ok && mode == 0 ? u[rr2] : 0.0f;
#pragma unroll
            for (int c = 0; c < M; ++c)
                z[i][c] = ok ? ld_keep(Z + (size_t)c * RO + rr2, keep) : 0.0f;
        }
#pragma unroll
        for (int i = 0; i < 2; ++i) {
            const int rr2 = r + i * T;
            if (rr2 < oEnd) {
                float rn = rv[i];
                if (mode == 0) {
                    rn = fmaf(-alpha, qv[i], rn);
                    r_next[rr2] = rn;
                    u[rr2] = fmaf(alpha, pv[i], uv[i]);
                }
                acc[2 * M] = fmaf(rn, rn, acc[2 * M]);
#pragma unroll
                for (int c = 0; c < M; ++c) acc[c] = fmaf(z[i][c], rn, acc[c]);
            }
        }
    }
#pragma unroll
    for (int i = 0; i < EXT; ++i) {
        if (ed[i] >= 0) {
            const float rn = !YV && mode == 0 ? fmaf(-alpha, qe[i], re[i]) : re[i];
#pragma unroll
            for (int c = 0; c < M; ++c) acc[M + c] = fmaf(ws[(i * M + c) * T], rn, acc[M + c]);
        }
    }
    for (int r = eBegin + EXT * T; r < eEnd; r += 2 * T) {
        float w[2][M], rv[2], qv[2];
        int d[2];
#pragma unroll
        for (int i = 0; i < 2; ++i)
            d[i] = r + i * T < eEnd ? ld_keep(B.extRowDof + r + i * T, keep) : -1;
#pragma unroll
        for (int i = 0; i < 2; ++i) {
            rv[i] = d[i] >= 0 ? (YV ? yv[d[i]] : r_cur[d[i]]) : 0.0f;
            qv[i] = d[i] >= 0 && !YV && mode == 0 ? q[d[i]] : 0.0f;
#pragma unroll
            for (int c = 0; c < M; ++c)
                w[i][c] = d[i] >= 0 ? ld_keep(W + (size_t)c * RE + r + i * T, keep) : 0.0f;
        }
#pragma unroll
        for (int i = 0; i < 2; ++i) {
            if (d[i] >= 0) {
                const float rn = !YV && mode == 0 ? fmaf(-alpha, qv[i], rv[i]) : rv[i];
#pragma unroll
                for (int c = 0; c < M; ++c) acc[M + c] = fmaf(w[i][c], rn, acc[M + c]);
            }
        }
    }
    // the block's sums: each warp's by halving exchanges, the eight warps' by
    // one lane per column
    constexpr int P = M == 6 ? 16 : 32;
    const int warp = tid >> 5, lane = tid & 31;
    const float mine = warp_sum_scatter<P, 2 * M + 1>(acc);
    if (P == 32 || (lane & 1) == 0) red[warp][P == 32 ? lane : lane >> 1] = mine;
    __syncthreads();
    rr = 0.0f;
    if (warp == 0) {
        auto total = [&](int c) {
            float x[8];
#pragma unroll
            for (int w = 0; w < 8; ++w) x[w] = red[w][c];
            return sum_of_8(x);
        };
        if (lane == 0) rr = total(2 * M);
        const int u0 = B.boxUnit[s], nu = B.boxUnit[s + 1] - u0;
        const int c = lane, c0 = B.col0[s];
        double zsum = 0.0, wsum = 0.0;
        if (c < M) {
            zsum = total(c);
            wsum = total(M + c);
        }
        bool finish = nu == 1;
        if (nu > 1) {
            // the box's last unit adds their sums in unit order
            if (c < M) {
                B.unitPart[(size_t)unit * 24 + c] = zsum;
                B.unitPart[(size_t)unit * 24 + M + c] = wsum;
                __threadfence();
            }
            __syncwarp();
            unsigned int t = 0;
            if (lane == 0) t = atomicAdd(&B.boxTicket[s], 1u);
            finish = __shfl_sync(0xffffffffu, t, 0) == (unsigned int)nu - 1;
            if (finish) {
                __threadfence();
                zsum = wsum = 0.0;
                if (c < M)
                    for (int v = u0; v < u0 + nu; ++v) {
                        zsum += __ldcg(B.unitPart + (size_t)v * 24 + c);
                        wsum += __ldcg(B.unitPart + (size_t)v * 24 + M + c);
                    }
                if (lane == 0) B.boxTicket[s] = 0u;
            }
        }
        if (finish && c < M) {
            g[c0 + c] = zsum - wsum;
            B.g32[c0 + c] = (float)(zsum - wsum);
            if (zr) zr[c0 + c] = zsum;
        }
    }
    return true;
}

// Mode 0 (an iteration): the product left its blocks' sums of p^T q in pqPart
// instead of reducing them itself; every block adds them (block_total_t0), takes
// alpha = rho / pq, and block 0 records pq, alpha and counts the iteration (its
// += 1: the launch's arguments do not depend on the iteration, so a captured
// batch of iterations can be replayed), or the breakdown (or a failed wait of
// the product).  Its blocks' sums of ||r||^2 stay in partials, for the coarse
// solve; mode 1 (start, replacement) adds them itself.
//
// Bound by latency: 51 MB at 48^3, most of it from L2, between two grid-wide
// dependencies.  48^3 (543 units): 28.8 us before (dependent loads after the
// wait, every warp dividing in FP64, a reduction across the blocks), 22.1 now;
// 12^3 (11 units): 19.8 before, 12.3 now.
template <bool YV, bool FEW>
__global__ void __launch_bounds__(kRowThreads, FEW ? 1 : 4)
k_restrict_update(RowBoxDev B, float *u, const float *r_cur, float *r_next, const float *p,
                  const float *q, const float *yv, int mode, double *g, double *zr,
                  double *partials, Scalars *sc, const float2 *pqPart, int pqN) {
    extern __shared__ __align__(16) float stage[];
    __shared__ float red[8][32];
    const int unit = blockIdx.x;
    // after the wait: alpha, the same for every thread; false: nothing to do
    auto alpha_of = [&](float &alpha) -> bool {
        if (mode != 0) return true;   // no update: alpha stays 0
        __shared__ float sAlpha;
        __shared__ bool sGo;
        const double pq = block_total_t0(pqPart, pqN);
        if (threadIdx.x == 0) {
            const bool fault = sc->fault != 0;
            const bool broken = !(pq > 0.0) || !isfinite(pq);
            const double a = sc->rho / pq;
            sAlpha = (float)a;
            sGo = !fault && !broken;
            if (blockIdx.x == 0) {
                if (fault) {
                    sc->done = kFault;
                } else {
                    sc->pq = pq;
                    sc->its += 1;
                    if (broken)
                        sc->done = kBreakdown;
                    else
                        sc->alpha = a;
                }
            }
        }
        __syncthreads();
        alpha = sAlpha;
        return sGo;
    };
    float rr = 0.0f;
    const bool went =
        B.menr[B.unitBox[unit]]
            ? restrict_update_unit<12, YV, FEW>(B, unit, u, r_cur, r_next, p, q, yv, mode, g, zr,
                                                sc, stage, red, alpha_of, rr)
            : restrict_update_unit<6, YV, FEW>(B, unit, u, r_cur, r_next, p, q, yv, mode, g, zr,
                                               sc, stage, red, alpha_of, rr);
    if (!went || mode >= 2) return;
    if (threadIdx.x == 0) partials[blockIdx.x] = (double)rr;
    if (mode == 0) return;
    if (!last_block(&sc->ticket[2])) return;
    const double tot = sum_slots<kRowThreads>(partials, (int)gridDim.x);
    if (threadIdx.x == 0) {
        sc->rr = tot;
        sc->ry = tot;
        if (tot <= sc->tol2ff)
            sc->done = kConverged;
        else if (sc->its >= sc->max_it)
            sc->done = kMaxIter;
        else if (!isfinite(tot))
            sc->done = kBreakdown;
    }
}

template <bool YV, bool FEW>
static void launch_restrict_rows(const RowBoxDev &B, float *u, const float *r_cur, float *r_next,
                                 const float *p, const float *q, const float *y, int mode,
                                 double *g, double *zr, double *partials, Scalars *sc,
                                 const float2 *pqPart, int pqN, cudaStream_t st) {
    launch_pdl(k_restrict_update<YV, FEW>, B.nUnits, kRowThreads,
               kStageFloats<FEW> * kRowThreads * sizeof(float), st, B, u, r_cur, r_next, p, q, y,
               mode, g, zr, partials, sc, pqPart, pqN);
}

// dynamic shared memory of the restriction's staging (once per context)
bool restrict_rows_prepare() {
    auto set = [](auto k, int floats) {
        return cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                    floats * kRowThreads * (int)sizeof(float)) == cudaSuccess;
    };
    return set(k_restrict_update<false, false>, kStageFloats<false>) &&
           set(k_restrict_update<true, false>, kStageFloats<false>) &&
           set(k_restrict_update<false, true>, kStageFloats<true>) &&
           set(k_restrict_update<true, true>, kStageFloats<true>);
}

// FEW when every unit has an SM to itself
void launch_restrict_start(const RowBoxDev &B, const float *r, int mode, double *g, double *zr,
                           double *partials, Scalars *sc, cudaStream_t st, const float *y) {
    const bool few = B.nUnits <= device_sm_count();
    auto launch = mode == 3 ? (few ? launch_restrict_rows<true, true> : launch_restrict_rows<true, false>)
                            : (few ? launch_restrict_rows<false, true> : launch_restrict_rows<false, false>);
    launch(B, nullptr, r, nullptr, nullptr, nullptr, y, mode, g, zr, partials, sc, nullptr, 0, st);
}

void launch_restrict_update(const RowBoxDev &B, float *u, const float *r_cur, float *r_next,
                            const float *p, const float *q, double *g, double *zr,
                            double *rrPart, Scalars *sc, const float2 *pqPart, int pqN,
                            cudaStream_t st) {
    auto launch = B.nUnits <= device_sm_count() ? launch_restrict_rows<false, true>
                                                : launch_restrict_rows<false, false>;
    launch(B, u, r_cur, r_next, p, q, nullptr, 0, g, zr, rrPart, sc, pqPart, pqN, st);
}

// Triggers its dependent, the next product, only while its grid is small: the
// product's blocks fill the SMs as they are, and a large prolongation finishes
// later beside them (32^3, 512 blocks: 46.3 us per iteration with, 47.0
// without; 48^3, 1,066 blocks: 79.4 and 78.0; nothing was measured between).
constexpr int kTriggerBlocks = 608;   // four for each of 152 SMs

// Prolongation over one unit's own rows, kProlongRows / kRowThreads rows a
// thread, all in flight before the wait for the coarse solve: their rows of
// Z~, and their entries of y and p, which no kernel still running writes.
template <int M>
__device__ __forceinline__ void prolong_rows_unit(const RowBoxDev &B, int unit,
                                                  const float *nu32, const float *y, float *p,
                                                  int mode, const Scalars *sc) {
    constexpr int R = (kProlongRows + kRowThreads - 1) / kRowThreads;
    const int s = B.pUnitBox[unit];
    const int c0 = B.col0[s], r0 = B.ownRowPtr[s], RO = B.ownRowPtr[s + 1] - r0;
    const float *Z = B.Z + B.zBase[s] - r0;
    const int rb = B.pUnitBegin[unit] + threadIdx.x, re = B.pUnitEnd[unit];
    const uint64_t keep = l2_keep_policy();
    float z[R][M], yv[R], pv[R];
    auto load = [&]() {
#pragma unroll
        for (int i = 0; i < R; ++i) {
            const int r = rb + i * kRowThreads;
            const bool ok = r < re;
#pragma unroll
            for (int c = 0; c < M; ++c)
                z[i][c] = ok ? ld_keep(Z + (size_t)c * RO + r, keep) : 0.0f;
            yv[i] = ok && mode != 1 ? ld_early(y + r) : 0.0f;
            pv[i] = ok && mode == 0 ? ld_early(p + r) : 0.0f;
        }
    };
    const bool early = __ldcg(&sc->done) == kRunning;   // may be stale, as above
    if (early) load();
    pdl_wait();
    if ((int)gridDim.x <= kTriggerBlocks) pdl_trigger();
    if (blockIdx.x == 0 && threadIdx.x == 0) report(sc);
    if (sc->done != kRunning) return;
    if (!early) load();
    const float beta = (float)sc->beta;
    float n[M];
#pragma unroll
    for (int c = 0; c < M; ++c) n[c] = nu32[c0 + c];
#pragma unroll
    for (int i = 0; i < R; ++i) {
        const int r = rb + i * kRowThreads;
        if (r < re) {
            float zv = 0.0f;
#pragma unroll
            for (int c = 0; c < M; ++c) zv = fmaf(z[i][c], n[c], zv);
            p[r] = emitted(yv[i], pv[i], zv, mode, beta);
        }
    }
}

// 48^3: 12.2 us before, 10.3 now; 12^3: 8.3 before, 6.5 now
__global__ void __launch_bounds__(kRowThreads)
k_prolong_rows(RowBoxDev B, const float *nu32, const float *y, float *p, int mode, Scalars *sc) {
    const int unit = blockIdx.x;
    if (B.menr[B.pUnitBox[unit]])
        prolong_rows_unit<12>(B, unit, nu32, y, p, mode, sc);
    else
        prolong_rows_unit<6>(B, unit, nu32, y, p, mode, sc);
}

void launch_prolong_rows(const RowBoxDev &B, const float *nu32, const float *y, float *p,
                         int mode, Scalars *sc, cudaStream_t st) {
    launch_pdl(k_prolong_rows, B.nPUnits, kRowThreads, 0, st, B, nu32, y, p, mode, sc);
}

// set-up: row-major per-item blocks (b x M at srcOff) to the per-box
// column-major layout
__global__ void k_to_colmajor(int nItems, const int *itemBox, const int *rowStart,
                              const unsigned char *itemB, const long long *srcOff,
                              const int *boxRowPtr, const long long *boxBase, const int *menr,
                              const float *src, float *dst) {
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= nItems) return;
    const int s = itemBox[t], M = menr[s] ? 12 : 6, b = itemB[t];
    const int R = boxRowPtr[s + 1] - boxRowPtr[s];
    const int rl0 = rowStart[t] - boxRowPtr[s];
    for (int i = 0; i < b; ++i)
        for (int c = 0; c < M; ++c)
            dst[boxBase[s] + (long long)c * R + rl0 + i] = src[srcOff[t] + i * M + c];
}

void launch_to_colmajor(int nItems, const int *itemBox, const int *rowStart,
                        const unsigned char *itemB, const long long *srcOff,
                        const int *boxRowPtr, const long long *boxBase, const int *menr,
                        const float *src, float *dst, cudaStream_t st) {
    if (nItems == 0) return;
    k_to_colmajor<<<(nItems + 127) / 128, 128, 0, st>>>(nItems, itemBox, rowStart, itemB, srcOff,
                                                        boxRowPtr, boxBase, menr, src, dst);
}

}  // namespace xdcg

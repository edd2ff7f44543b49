// FP64 block Thomas elimination with explicit block inverses (the plain FP64 path, and the mixed
// path's FP64 route): Gauss-Jordan with implicit partial pivoting in panels of 8 columns, one
// persistent cooperative launch, both ends of the column at once on two halves of the grid.
//
// This part issues about two FP64 fused operations per clock and SM, so a panel of several hundred
// rows factored by one CTA, with a block barrier pair per column, is most of the time: 51 us per
// panel at 594 species (of which the other 75 SMs idle through about 40), 22 us at 96.  Here
//  - the panel belongs to a thread-block cluster, its rows spread over the cluster's CTAs, one row
//    per thread (two beyond 512 rows of a CTA) in registers.  Per column every warp sends its best candidate row (the reciprocal of
//    its pivot and the row's panel entries) to all CTAs as asynchronous stores that complete on the
//    receiver's mbarrier, and each picks the winner from its own copy: no barrier of the cluster or
//    the block.  The loop over the panel's columns is rolled (the finished column moves to the end):
//    unrolled, its code ran out of the instruction cache and a column took 1,900 clocks;
//  - the other CTAs apply the previous panels to their columns meanwhile.  k_factor64_flow: a CTA
//    keeps its columns of the layer in shared memory, takes each panel as its flag appears and hands
//    the columns of panel p + 2 over once panel p has been applied to them; grid barriers only at a
//    layer's end.  k_factor64: columns too many for shared memory (a small share of the SMs in a
//    batch) stay in global memory, with one grid barrier per panel.
// Bound by the FP64 updates at 594 species (8 S^2 fused operations per panel over the chain's SMs,
// 24,400 clocks), by the chain of columns below some 300.
// The pivot is the unused row of largest magnitude to 20 bits (the high word of the double), the
// lowest row among equals.
//
// Pivoting is implicit: rows never move, perm_k[c] is the row that served as pivot of column c and
// iperm_k its inverse.  After factorization D holds B_k with D'^-1_k[i][j] = B_k[perm_k(i)][iperm_k(j)].
#include <cuda_runtime.h>
#include <math.h>

#include <algorithm>

#include "xk_mbar.cuh"

namespace xk {

namespace {

constexpr int kNB = 8;
constexpr int kThreads = 512;
constexpr int kWarps = kThreads / 32;
constexpr int kPS = kNB + 1;              // padded row of the panel in shared memory
constexpr size_t kSmemMax = 227 * 1024;

// A warp's best candidate for a pivot: the reciprocal of the pivot and the rest of the row's panel
// entries, the magnitude's high word, the row.
struct __align__(16) Cand {
    double row[kNB];
    unsigned key;
    int idx;                              // -1: the warp has no unused row
    int pad[2];
};
constexpr int kCandParts = sizeof(Cand) / 16;

__device__ __forceinline__ void st_cluster(uint32_t addr, int v)
{
    asm volatile("st.shared::cluster.b32 [%0], %1;" ::"r"(addr), "r"(v) : "memory");
}
// Asynchronous store of 16 bytes into a CTA of the cluster, counted by that CTA's mbarrier.
__device__ __forceinline__ void st_async(uint32_t addr, uint4 v, uint32_t mbar)
{
    asm volatile("st.async.shared::cluster.mbarrier::complete_tx::bytes.v4.b32 [%0], {%1, %2, %3, %4}, [%5];" ::"r"(addr),
                 "r"(v.x), "r"(v.y), "r"(v.z), "r"(v.w), "r"(mbar)
                 : "memory");
}
// Bounded wait for a counter that other CTAs raise, as mbar_wait.
__device__ __forceinline__ void wait_count(const unsigned *word, unsigned target, Ctl *ctl)
{
    const unsigned long long limit = ctl->wait_polls ? ctl->wait_polls : kSyncPolls;
    for (unsigned long long i = 0; i < limit; ++i) {
        unsigned v;
        asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(word) : "memory");
        if ((int)(v - target) >= 0) return;
        if ((i & 63) == 63 && *(volatile int *)&ctl->err_timeout) return;
    }
    atomicExch(&ctl->err_timeout, 1);
}
__device__ __forceinline__ void raise_count(unsigned *word)
{
    __threadfence();
    asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(word) : "memory");
}

__device__ __forceinline__ void cluster_sync(int cs)
{
    if (cs == 1) {
        __syncthreads();
    } else {
        asm volatile("barrier.cluster.arrive.release;" ::: "memory");
        asm volatile("barrier.cluster.wait.acquire;" ::: "memory");
    }
}

// Barrier over the clusters of a chain.  The first CTA of each cluster arrives and polls (bounded, as
// GridSync) and hands the outcome to the others, so that the CTAs of a cluster always leave together:
// none writes into the shared memory of one that has gone.
struct ChainSync {
    unsigned *word, *left;
    Ctl *ctl;
    int cs, nclus, crank;
    int *go;                              // shared memory, the same offset in every CTA
    unsigned target;
    __device__ __forceinline__ bool sync()
    {
        target += (unsigned)nclus;
        __threadfence();
        cluster_sync(cs);
        if (crank == 0 && threadIdx.x == 0) {
            int ok = 1;
            __threadfence();
            asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(word) : "memory");
            const unsigned long long limit = ctl->wait_polls ? ctl->wait_polls : kSyncPolls;
            volatile int *vto = &ctl->err_timeout;
            for (unsigned long long i = 0;; ++i) {
                unsigned v;
                asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(word) : "memory");
                // exactly this barrier's count or the arrivals of the next: a held counter never is
                if (v - target < (unsigned)nclus) break;
                if (i > limit || ((i & 63) == 63 && *vto)) {
                    atomicExch(&ctl->err_timeout, 1);
                    ok = 0;
                    break;
                }
            }
            __threadfence();
            // complete, but a wait of somebody's may have given up on the way here
            tell(ok && !*vto);
        }
        cluster_sync(cs);
        return *go != 0;
    }
    __device__ __forceinline__ void tell(int ok)
    {
        if (cs == 1) *go = ok;
        else
            for (int r = 0; r < cs; ++r) st_cluster(map_rank(smem_u32(go), r), ok);
    }
    // at the start, after a barrier of the cluster: false if a wait of an earlier launch has given up.  One
    // CTA looks: another that looked for itself might see a wait of this launch give up and leave alone.
    __device__ __forceinline__ bool open()
    {
        if (crank == 0 && threadIdx.x == 0) tell(!*(volatile int *)&ctl->err_timeout);
        cluster_sync(cs);
        return *go != 0;
    }
    // after the last sync; the last cluster out clears the words
    __device__ __forceinline__ void leave()
    {
        cluster_sync(cs);
        if (crank == 0 && threadIdx.x == 0 && atomicAdd(left, 1u) == (unsigned)nclus - 1) {
            *word = 0u;
            *left = 0u;
            __threadfence();
        }
    }
};

// The panel's share of one CTA of its cluster.
struct Panel {
    int S, ld, cs, crank, rpc, r0, nr, nw, ncand;
    double *P, *G;                // [rpc][kPS]: the panel's rows, the previous panel's result
    double *us;                   // [kNB * kNB]: the previous panel's pivot rows in this panel
    Cand *stage, *cand;           // [kWarps], [2][32]
    int *piv;                     // [2][kNB]
    uint32_t mbar;                // two mbarriers, one per candidate buffer
    unsigned col;                 // columns done in this launch: buffer col & 1, phase (col / 2) & 1
    Ctl *ctl;
};

// Panel p of layer block D: takes its columns from D (the panels before p - 1 are applied), applies
// panel p - 1, factors it and leaves G in D's panel columns and in G.
template <int RPT>
__device__ __forceinline__ void panel_step(Panel &q, double *D, int *perm, int *iperm, int p, unsigned &used)
{
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int c0 = p * kNB, nb = min(kNB, q.S - c0);
    const int *pp = q.piv + ((p + 1) & 1) * kNB;   // the previous panel's pivot rows
    int *pc = q.piv + (p & 1) * kNB;
    for (int e = tid; e < q.nr * kNB; e += kThreads) {
        const int r = e / kNB, j = e % kNB;
        q.P[r * kPS + j] = j < nb ? __ldcg(D + (size_t)(q.r0 + r) * q.ld + c0 + j) : 0.0;
    }
    if (p > 0 && tid < kNB * kNB) {
        const int l = tid / kNB, j = tid % kNB;
        q.us[tid] = j < nb ? __ldcg(D + (size_t)pp[l] * q.ld + c0 + j) : 0.0;
    }
    __syncthreads();
    if (p > 0) {
        for (int e = tid; e < q.nr * kNB; e += kThreads) {
            const int r = e / kNB, j = e % kNB;
            bool piv = false;
#pragma unroll
            for (int l = 0; l < kNB; ++l) piv |= pp[l] == q.r0 + r;
            double acc = piv ? 0.0 : q.P[r * kPS + j];
#pragma unroll
            for (int l = 0; l < kNB; ++l) acc = fma(q.G[r * kPS + l], q.us[l * kNB + j], acc);
            q.P[r * kPS + j] = acc;
        }
        __syncthreads();
    }
    if (warp < q.nw) {
        double x[RPT][kNB];
#pragma unroll
        for (int i = 0; i < RPT; ++i) {
            const int r = tid + i * kThreads;
#pragma unroll
            for (int j = 0; j < kNB; ++j) x[i][j] = r < q.nr ? q.P[r * kPS + j] : 0.0;
        }
        // column c is always x[.][0]: each step shifts the others down one and puts the finished column
        // last, so that after eight steps they are in their places again
#pragma unroll 1
        for (int c = 0; c < kNB; ++c) {
            if (c >= nb) {                      // a ragged panel's missing columns
#pragma unroll
                for (int i = 0; i < RPT; ++i) {
                    const double t = x[i][0];
#pragma unroll
                    for (int j = 1; j < kNB; ++j) x[i][j - 1] = x[i][j];
                    x[i][kNB - 1] = t;
                }
                continue;
            }
            const int par = q.col & 1;
            const uint32_t bar = q.mbar + 8u * par, phase = (q.col >> 1) & 1u;
            ++q.col;
            Cand *cb = q.cand + 32 * par;
            if (tid == 0) mbar_expect(bar, (uint32_t)(q.ncand * sizeof(Cand)));
            // this warp's best unused row (and its reciprocal, while the reduction runs)
            unsigned key = 0u;
            int bi = -1;
#pragma unroll
            for (int i = 0; i < RPT; ++i) {
                const unsigned m = (unsigned)__double2hiint(x[i][0]) & 0x7fffffffu;
                if (!((used >> i) & 1u) && (bi < 0 || m > key)) { key = m; bi = i; }
            }
            double mine_row[kNB];
#pragma unroll
            for (int j = 0; j < kNB; ++j) mine_row[j] = RPT > 1 && bi == RPT - 1 ? x[RPT - 1][j] : x[0][j];
            // (a column without a nonzero candidate is singular: the bookkeeping goes on)
            mine_row[0] = key == 0u ? 0.0 : reciprocal_newton(mine_row[0]);
            const unsigned best = __reduce_max_sync(0xffffffffu, bi >= 0 ? key + 1u : 0u);
            const unsigned who = __ballot_sync(0xffffffffu, bi >= 0 && key + 1u == best);
            const int src = who ? __ffs(who) - 1 : 0;
            if (lane == src) {
                Cand &o = q.stage[warp];
#pragma unroll
                for (int j = 0; j < kNB; j += 2) *(double2 *)&o.row[j] = make_double2(mine_row[j], mine_row[j + 1]);
                o.key = key;
                o.idx = who ? q.r0 + tid + bi * kThreads : -1;
            }
            __syncwarp();
            for (int it = lane; it < q.cs * kCandParts; it += 32) {
                const int dst = it / kCandParts, part = it % kCandParts;
                st_async(map_rank(smem_u32(&cb[q.crank * q.nw + warp]) + 16u * part, dst), ((const uint4 *)&q.stage[warp])[part],
                         map_rank(bar, dst));
            }
            mbar_wait(bar, phase, q.ctl);
            __syncwarp();
            const bool have = lane < q.ncand && cb[lane].idx >= 0;
            const unsigned ck = have ? cb[lane].key : 0u;
            const unsigned top = __reduce_max_sync(0xffffffffu, have ? ck + 1u : 0u);
            const unsigned win = __ballot_sync(0xffffffffu, have && ck + 1u == top);
            const Cand &w = cb[win ? __ffs(win) - 1 : 0];
            const int row = min(max(w.idx, 0), q.S - 1);
            double pr[kNB];
#pragma unroll
            for (int j = 0; j < kNB; j += 2) {
                const double2 v = *(const double2 *)&w.row[j];
                pr[j] = v.x;
                pr[j + 1] = v.y;
            }
            if (tid == 0) {
                pc[c] = row;
                if (q.crank == 0 && top <= 1u) atomicExch(&q.ctl->err_singular, 1);
            }
#pragma unroll
            for (int i = 0; i < RPT; ++i) {
                const bool mine = q.r0 + tid + i * kThreads == row && tid + i * kThreads < q.nr;
                if (mine) {
                    used |= 1u << i;
                    perm[c0 + c] = row;
                    iperm[row] = c0 + c;
                }
                // the pivot row starts from zero and takes the multiplier that leaves it scaled
                const double f = mine ? -pr[0] : x[i][0] * pr[0];
#pragma unroll
                for (int j = 1; j < kNB; ++j) x[i][j - 1] = fma(-f, pr[j], mine ? 0.0 : x[i][j]);
                x[i][kNB - 1] = -f;
            }
        }
        // the panel's columns become G
#pragma unroll
        for (int i = 0; i < RPT; ++i) {
            const int r = tid + i * kThreads;
            if (r >= q.nr) continue;
            double *Dr = D + (size_t)(q.r0 + r) * q.ld + c0;
#pragma unroll
            for (int j = 0; j < kNB; ++j) {
                q.G[r * kPS + j] = j < nb ? x[i][j] : 0.0;
                if (j < nb) __stcg(Dr + j, x[i][j]);
            }
        }
    }
}

// A pivot's row, or its place among them.  Where a wait has given up the list may hold anything: kept in
// bounds until the chain's next barrier ends the launch.
__device__ __forceinline__ int row_at(const int *p, int S) { return min(max(__ldcg(p), 0), S - 1); }

// Which layers a chain takes, and in which order.
struct Order {
    int nsteps, k0, dk;
};
__device__ __forceinline__ Order order_of(int mode, int half, int L, int mid)
{
    if (mode == 1) return half == 0 ? Order{mid, 0, 1} : Order{L - 1 - mid, L - 1, -1};
    if (mode == 2) return Order{1, mid, 0};
    return Order{L, 0, 1};
}

// Schur terms of layer k: f(n, rowc, colc) for each neighbour n already eliminated,
// D_k -= diag(rowc) D'^-1_n diag(colc).
template <typename F>
__device__ __forceinline__ bool schur_terms(const BlockSys<double> &a, int mode, int step, int dk, int k, F f)
{
    const size_t S = a.S;
    const bool below = mode == 2 ? k > 0 : step > 0 && dk > 0;
    const bool above = mode == 2 ? k + 1 < a.L : step > 0 && dk < 0;
    if (below) f(k - 1, a.lo + k * S, a.up + (k - 1) * S);
    if (above) f(k + 1, a.up + k * S, a.lo + (k + 1) * S);
    return below || above;
}

struct PanelShared {
    Cand stage[kWarps], cand[2][32];
    double us[kNB * kNB];
    int piv[2][kNB], go;
    unsigned long long mbar[2];
};

__device__ __forceinline__ Panel make_panel(PanelShared &sh, double *dyn, const BlockSys<double> &a, Ctl *ctl, int cs, int crank)
{
    Panel q;
    q.S = a.S;
    q.ld = a.ld;
    q.cs = cs;
    q.crank = crank;
    q.rpc = (a.S + cs - 1) / cs;
    q.r0 = crank * q.rpc;
    q.nr = max(0, min(a.S, q.r0 + q.rpc) - q.r0);
    q.nw = min(kWarps, (q.rpc + 31) / 32);
    q.ncand = cs * q.nw;
    q.P = dyn;
    q.G = q.P + (size_t)q.rpc * kPS;
    q.us = sh.us;
    q.stage = sh.stage;
    q.cand = sh.cand[0];
    q.piv = sh.piv[0];
    q.mbar = smem_u32(sh.mbar);
    q.col = 0;
    q.ctl = ctl;
    // every CTA's mbarriers stand before another CTA sends to them
    if (threadIdx.x == 0) {
        for (int i = 0; i < 2; ++i) mbar_init(q.mbar + 8u * i);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    cluster_sync(cs);
    return q;
}

template <int RPT>
__device__ __forceinline__ unsigned unused_rows(const Panel &q)
{
    unsigned used = 0;                           // bit i: this thread's row i has been a pivot, or is none
#pragma unroll
    for (int i = 0; i < RPT; ++i)
        if ((int)threadIdx.x + i * kThreads >= q.nr) used |= 1u << i;
    return used;
}

// mode 0: all layers top-down on the whole grid.  mode 1 (twisted): two chains on the two halves of
// the grid, layers 0 .. mid-1 top-down and L-1 .. mid+1 bottom-up.  mode 2: the middle layer on the
// whole grid, with both Schur terms.  RPT: panel rows per thread.
template <int RPT>
__global__ void __launch_bounds__(kThreads, 1)
k_factor64(BlockSys<double> a, Ctl *ctl, const int *skip, int mode, int mid, int cs)
{
    if (ctl->finished || (skip && *skip)) return;
    extern __shared__ __align__(16) unsigned char dyn[];
    __shared__ PanelShared sh;
    const int S = a.S, ld = a.ld;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int half = mode == 1 ? (int)(blockIdx.x >= gridDim.x / 2) : 0;
    const int nblk = mode == 1 ? (int)gridDim.x / 2 : (int)gridDim.x;
    const int bid = (int)blockIdx.x - half * nblk;
    const int crank = (int)cluster_rank(), cidx = bid / cs, nclus = nblk / cs;
    // trailing updates: the CTAs of the other clusters, or everyone where there is only one
    const int ntrail = nclus > 1 ? nblk - cs : nblk, tq = nclus > 1 ? bid - cs : bid;
    ChainSync chain{a.bar + 2 * half, a.bar + 6 + half, ctl, cs, nclus, crank, &sh.go, 0u};
    Panel q = make_panel(sh, (double *)dyn, a, ctl, cs, crank);
    if (!chain.open()) return;
    double *U = q.G + (size_t)q.rpc * kPS;                // [kNB][cw]: pivot rows in this CTA's columns
    double *rowbuf = (double *)dyn + (size_t)warp * S;    // Schur term: a source row per warp
    const Order o = order_of(mode, half, a.L, mid);
    const int npan = (S + kNB - 1) / kNB;
    for (int step = 0; step < o.nsteps; ++step) {
        const int k = o.k0 + step * o.dk;
        double *D = a.D + (size_t)k * S * ld;
        int *perm = a.perm + (size_t)k * S, *iperm = a.iperm + (size_t)k * S;
        // D'^-1_n[i][j] = B_n[perm_n(i)][iperm_n(j)]: a warp per row, the source row through shared memory
        const bool touched = schur_terms(a, mode, step, o.dk, k, [&](int nbr, const double *rowc, const double *colc) {
            const double *Bn = a.D + (size_t)nbr * S * ld;
            const int *pn = a.perm + (size_t)nbr * S, *ipn = a.iperm + (size_t)nbr * S;
            for (int i = bid * kWarps + warp; i < S; i += nblk * kWarps) {
                const double *src = Bn + (size_t)row_at(pn + i, S) * ld;
                const double rc = rowc[i];
                __syncwarp();
                for (int j = lane; j < S; j += 32) rowbuf[j] = __ldcg(src + j);
                __syncwarp();
                double *Di = D + (size_t)i * ld;
                for (int j = lane; j < S; j += 32) Di[j] -= rc * rowbuf[row_at(ipn + j, S)] * colc[j];
            }
        });
        if (touched && !chain.sync()) return;
        unsigned used = unused_rows<RPT>(q);
        for (int p = 0; p <= npan; ++p) {
            if (cidx == 0 && p < npan) panel_step<RPT>(q, D, perm, iperm, p, used);
            if (p > 0 && tq >= 0) {
                // panel p - 1 applied to every column but its own and panel p's (the cluster's)
                const int q0 = (p - 1) * kNB, nb = min(kNB, S - q0);
                const int c1 = q0 + nb + (p < npan ? min(kNB, S - q0 - kNB) : 0);
                const int ncol = S - (c1 - q0), per = ncol / ntrail, rest = ncol - per * ntrail;
                const int j0 = tq * per + min(tq, rest), cw = per + (tq < rest ? 1 : 0);
                if (cw > 0) {
                    int pr[kNB];
#pragma unroll
                    for (int l = 0; l < kNB; ++l) pr[l] = l < nb ? row_at(perm + q0 + l, S) : -1;
                    auto col = [&](int c) { return j0 + c < q0 ? j0 + c : j0 + c + (c1 - q0); };
                    __syncthreads();
                    for (int e = tid; e < kNB * cw; e += kThreads) {
                        const int l = e / cw, c = e - l * cw;
                        U[e] = l < nb ? __ldcg(D + (size_t)row_at(perm + q0 + l, S) * ld + col(c)) : 0.0;
                    }
                    __syncthreads();
                    // one element per thread, three of them in flight
                    const int total = S * cw;
                    for (int e0 = tid; e0 < total; e0 += 3 * kThreads) {
                        double acc[3], g[3][kNB];
                        int rr[3], qq[3];
#pragma unroll
                        for (int u = 0; u < 3; ++u) {
                            const int e = min(e0 + u * kThreads, total - 1);
                            rr[u] = e / cw;
                            qq[u] = e - rr[u] * cw;
                            const double *Dr = D + (size_t)rr[u] * ld;
                            acc[u] = __ldcg(Dr + col(qq[u]));
                            if (nb == kNB) {
#pragma unroll
                                for (int l = 0; l < kNB; l += 2) {
                                    const double2 v = __ldcg((const double2 *)(Dr + q0 + l));
                                    g[u][l] = v.x;
                                    g[u][l + 1] = v.y;
                                }
                            } else {
#pragma unroll
                                for (int l = 0; l < kNB; ++l) g[u][l] = l < nb ? __ldcg(Dr + q0 + l) : 0.0;
                            }
                        }
#pragma unroll
                        for (int u = 0; u < 3; ++u) {
                            bool piv = false;
#pragma unroll
                            for (int l = 0; l < kNB; ++l) piv |= pr[l] == rr[u];
                            double v = piv ? 0.0 : acc[u];
#pragma unroll
                            for (int l = 0; l < kNB; ++l) v = fma(g[u][l], U[l * cw + qq[u]], v);
                            if (e0 + u * kThreads < total) __stcg(D + (size_t)rr[u] * ld + col(qq[u]), v);
                        }
                    }
                }
            }
            if (!chain.sync()) return;
        }
    }
    chain.leave();
}

// The same elimination with every CTA beyond the panel's cluster keeping its columns [j0, j0 + cw) of
// the layer in shared memory.  Flags of a chain (they only grow; cleared by the last cluster out):
// flag[0] counts the panels' CTAs that have finished a panel, flag[1 + q] the owners that have handed
// panel q's columns over.  Panel p needs its columns with the panels before p - 1 applied; its G stays
// in D's panel columns until the layer's end, when every CTA has read it, and the columns follow.
constexpr int kMaxPanels = 2 * kThreads / kNB;
__global__ void __launch_bounds__(kThreads, 1)
k_factor64_flow(BlockSys<double> a, Ctl *ctl, const int *skip, int mode, int mid, int cs)
{
    if (ctl->finished || (skip && *skip)) return;
    extern __shared__ __align__(16) unsigned char dyn[];
    __shared__ PanelShared sh;
    const int S = a.S, ld = a.ld;
    const int tid = threadIdx.x;
    const int half = mode == 1 ? (int)(blockIdx.x >= gridDim.x / 2) : 0;
    const int nblk = mode == 1 ? (int)gridDim.x / 2 : (int)gridDim.x;
    const int bid = (int)blockIdx.x - half * nblk;
    const int crank = (int)cluster_rank(), cidx = bid / cs, nclus = nblk / cs;
    ChainSync chain{a.bar + 2 * half, a.bar + 6 + half, ctl, cs, nclus, crank, &sh.go, 0u};
    unsigned *flag = a.bar + 8 + half * (kMaxPanels + 8);
    const Order o = order_of(mode, half, a.L, mid);
    const int npan = (S + kNB - 1) / kNB;
    // columns of the owners: the first `rest` of them have one more
    const int ntrail = nblk - cs, tq = bid - cs, per = S / ntrail, rest = S - per * ntrail;
    const int j0 = tq * per + min(tq, rest), cw = tq >= 0 ? per + (tq < rest ? 1 : 0) : 0;
    auto owner = [&](int j) { return j < rest * (per + 1) ? j / (per + 1) : rest + (j - rest * (per + 1)) / max(per, 1); };
    Panel q = make_panel(sh, (double *)dyn, a, ctl, cs, crank);
    if (!chain.open()) return;
    const int ws = cw | 1;                        // odd row stride: a row per thread without conflicts
    double *W = (double *)dyn;                    // [S][ws]: this CTA's columns
    double *U = W + (size_t)S * ws;               // [kNB][cw]
    bool ok = true;
    for (int step = 0; step < o.nsteps && ok; ++step) {
        const int k = o.k0 + step * o.dk;
        double *D = a.D + (size_t)k * S * ld;
        int *perm = a.perm + (size_t)k * S, *iperm = a.iperm + (size_t)k * S;
        if (cidx == 0) {
            unsigned used = unused_rows<1>(q);
            for (int p = 0; p < npan; ++p) {
                if (tid == 0) {
                    const int c0 = p * kNB, owners = owner(min(c0 + kNB, S) - 1) - owner(c0) + 1;
                    wait_count(flag + 1 + p, (unsigned)(owners * (step + 1)), ctl);
                }
                __syncthreads();
                panel_step<1>(q, D, perm, iperm, p, used);
                __syncthreads();
                if (tid == 0) raise_count(flag);
            }
        } else {
            // hand the columns of panel p over: they are in W, every thread's rows
            auto hand_over = [&](int p) {
                const int a0 = max(j0, p * kNB), a1 = min(j0 + cw, min(p * kNB + kNB, S));
                if (p >= npan || a0 >= a1) return;
                for (int r = tid; r < S; r += kThreads)
                    for (int j = a0; j < a1; ++j) __stcg(D + (size_t)r * ld + j, W[r * ws + j - j0]);
                __syncthreads();
                if (tid == 0) raise_count(flag + 1 + p);
            };
            for (int e = tid; e < S * cw; e += kThreads) {
                const int i = e / cw, c = e - i * cw;
                W[i * ws + c] = D[(size_t)i * ld + j0 + c];
            }
            schur_terms(a, mode, step, o.dk, k, [&](int nbr, const double *rowc, const double *colc) {
                const double *Bn = a.D + (size_t)nbr * S * ld;
                const int *pn = a.perm + (size_t)nbr * S, *ipn = a.iperm + (size_t)nbr * S;
                for (int e = tid; e < S * cw; e += kThreads) {
                    const int i = e / cw, c = e - i * cw;
                    W[i * ws + c] -= rowc[i] * __ldcg(Bn + (size_t)row_at(pn + i, S) * ld + row_at(ipn + j0 + c, S)) * colc[j0 + c];
                }
            });
            __syncthreads();
            hand_over(0);
            hand_over(1);
            for (int p = 0; p < npan; ++p) {
                const int c0 = p * kNB, nb = min(kNB, S - c0);
                if (tid == 0) wait_count(flag, (unsigned)(cs * (step * npan + p + 1)), ctl);
                __syncthreads();
                int pr[kNB];
#pragma unroll
                for (int l = 0; l < kNB; ++l) pr[l] = l < nb ? row_at(perm + c0 + l, S) : -1;
                // G of this thread's first row on its way while the pivot rows are copied
                double g[kNB];
                auto load_g = [&](int r) {
                    const double *Dr = D + (size_t)r * ld + c0;
                    if (nb == kNB) {
#pragma unroll
                        for (int l = 0; l < kNB; l += 2) {
                            const double2 v = __ldcg((const double2 *)(Dr + l));
                            g[l] = v.x;
                            g[l + 1] = v.y;
                        }
                    } else {
#pragma unroll
                        for (int l = 0; l < kNB; ++l) g[l] = l < nb ? __ldcg(Dr + l) : 0.0;
                    }
                };
                if (tid < S) load_g(tid);
                for (int e = tid; e < kNB * cw; e += kThreads) {
                    const int l = e / cw, c = e - l * cw;
                    int row = 0;
#pragma unroll
                    for (int m = 0; m < kNB; ++m)
                        if (m == l) row = pr[m];
                    U[e] = l < nb ? W[row * ws + c] : 0.0;
                }
                __syncthreads();
                // own columns: those of panel p become G, those of panel p + 1 are the cluster's
                const int s0 = min(max(c0 - j0, 0), cw), s1 = min(max(c0 + nb - j0, 0), cw);
                const int s2 = min(max(c0 + 2 * kNB - j0, s1), cw);
                for (int r = tid; r < S; r += kThreads) {
                    if (r != tid) load_g(r);
                    bool piv = false;
#pragma unroll
                    for (int l = 0; l < kNB; ++l) piv |= pr[l] == r;
                    double *Wr = W + (size_t)r * ws;
                    auto run = [&](int b, int e) {
                        int c = b;
                        for (; c + 2 < e; c += 3) {
                            double v0 = piv ? 0.0 : Wr[c], v1 = piv ? 0.0 : Wr[c + 1], v2 = piv ? 0.0 : Wr[c + 2];
#pragma unroll
                            for (int l = 0; l < kNB; ++l) {
                                const double *u = U + l * cw + c;
                                v0 = fma(g[l], u[0], v0);
                                v1 = fma(g[l], u[1], v1);
                                v2 = fma(g[l], u[2], v2);
                            }
                            Wr[c] = v0; Wr[c + 1] = v1; Wr[c + 2] = v2;
                        }
                        for (; c < e; ++c) {
                            double v = piv ? 0.0 : Wr[c];
#pragma unroll
                            for (int l = 0; l < kNB; ++l) v = fma(g[l], U[l * cw + c], v);
                            Wr[c] = v;
                        }
                    };
                    run(0, s0);
                    run(s2, cw);
                    if (s0 < s1) {
#pragma unroll
                        for (int l = 0; l < kNB; ++l) {
                            const int c = c0 + l - j0;
                            if (c >= s0 && c < s1) Wr[c] = g[l];
                        }
                    }
                }
                hand_over(p + 2);
                __syncthreads();
            }
        }
        // every CTA has read the panels' G: the columns themselves follow
        ok = chain.sync();
        if (!ok) break;
        for (int e = tid; e < S * cw; e += kThreads) {
            const int i = e / cw, c = e - i * cw;
            __stcg(D + (size_t)i * ld + j0 + c, W[i * ws + c]);
        }
        ok = chain.sync();
    }
    if (!ok) return;
    // the flags too are zero again when the last cluster has left
    cluster_sync(cs);
    if (crank == 0 && tid == 0 && atomicAdd(chain.left, 1u) == (unsigned)nclus - 1) {
        for (int i = 0; i <= npan; ++i) flag[i] = 0u;
        *chain.word = 0u;
        *chain.left = 0u;
        __threadfence();
    }
}

size_t smem_general(int S, int cs, int ntrail)
{
    const size_t rpc = (S + cs - 1) / cs, cw = (S + ntrail - 1) / ntrail;
    const size_t panel = (2 * rpc * kPS + kNB * cw) * sizeof(double);
    const size_t rows = (size_t)kWarps * S * sizeof(double);
    return (std::max(panel, rows) + 255) & ~(size_t)255;
}

size_t smem_flow(int S, int cs, int ntrail)
{
    const size_t rpc = (S + cs - 1) / cs, cw = (S + ntrail - 1) / ntrail;
    const size_t panel = 2 * rpc * kPS * sizeof(double), slice = ((size_t)S * (cw | 1) + kNB * cw) * sizeof(double);
    return (std::max(panel, slice) + 255) & ~(size_t)255;
}

using FactorFn = void (*)(BlockSys<double>, Ctl *, const int *, int, int, int);
FactorFn kernel_of(int S, const FactorPlan &p)
{
    if (p.flow64) return k_factor64_flow;
    return (S + p.cs - 1) / p.cs <= kThreads ? k_factor64<1> : k_factor64<2>;
}

cudaError_t launch_mode(const BlockSys<double> &sys, const FactorPlan &plan, Ctl *ctl, cudaStream_t st, const int *skip,
                        int mode, int mid, int ctas)
{
    FactorFn fn = kernel_of(sys.S, plan);
    cudaError_t e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)plan.smem64);
    if (e != cudaSuccess) return e;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(ctas);
    cfg.blockDim = dim3(kThreads);
    cfg.dynamicSmemBytes = plan.smem64;
    cfg.stream = st;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeCooperative;
    attr[0].val.cooperative = 1;
    attr[1].id = cudaLaunchAttributeClusterDimension;
    attr[1].val.clusterDim.x = plan.cs;
    attr[1].val.clusterDim.y = 1;
    attr[1].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 2;
    count_launches(1);
    return cudaLaunchKernelEx(&cfg, fn, sys, ctl, skip, mode, mid, plan.cs);
}

// CTAs of one chain when `ctas` are launched (two chains at once need both halves whole).
int chain_of(int ctas, int cs) { return ctas / 2 / cs * cs; }

}  // namespace

size_t factor64_words() { return 8 + 2 * (kMaxPanels + 8); }

int factor64_plan(int S, int want, FactorPlan *p)
{
    if (S <= 0 || S > 2 * kThreads || want < 1) return -1;
    // The panel's cluster: the rows it spreads against the cost of an exchange across CTAs and of the SMs
    // taken from the updates.  Measured (ms with clusters of 1, 2, 4, 8): S = 20 (8 steps of 40 layers)
    // 8.4, 8.7, 8.7, 8.8; 96 (4 steps of 150) 52.6, 49.7, 48.6, 48.8; 131 (60 layers) 8.8, 7.8, 7.3, 7.2;
    // 250 (60) 21.1, 15.5, 13.7, 13.4; 400 (60) 46, 31, 22.9, 21.7; 594 (150) 275, 140, 102, 121.
    const int largest = S <= 32 ? 1 : S <= 128 || S > 500 ? 4 : 8;
    // CTAs of a launch: to each beyond the cluster at least about four columns
    auto ctas_of = [&](int cs) { return std::min(want, 2 * (cs + std::max(1, (S + 3) / 4 / cs) * cs)) / cs * cs; };
    auto fits = [&](int cs, int flow) {
        FactorPlan t = *p;
        t.cs = cs;
        t.flow64 = flow;
        t.ctas64 = ctas_of(cs);
        for (int pass = 0; pass < 2; ++pass) {
            const int half = chain_of(t.ctas64, cs);
            if (flow && half <= cs) return false;
            t.smem64 = flow ? smem_flow(S, cs, half - cs) : smem_general(S, cs, std::max(1, half - cs));
            if (t.smem64 > kSmemMax - sizeof(PanelShared)) return false;
            FactorFn fn = kernel_of(S, t);
            cudaLaunchConfig_t cfg = {};
            cfg.gridDim = dim3(cs);
            cfg.blockDim = dim3(kThreads);
            cfg.dynamicSmemBytes = t.smem64;
            cudaLaunchAttribute attr[1];
            attr[0].id = cudaLaunchAttributeClusterDimension;
            attr[0].val.clusterDim.x = cs;
            attr[0].val.clusterDim.y = 1;
            attr[0].val.clusterDim.z = 1;
            cfg.attrs = attr;
            cfg.numAttrs = 1;
            int n = 0;
            if (allow_smem(fn, t.smem64) != cudaSuccess || cudaOccupancyMaxActiveClusters(&n, fn, &cfg) != cudaSuccess ||
                n < 1) {
                cudaGetLastError();
                return false;
            }
            // fewer clusters than wanted fit at once: plan again for those
            if (n * cs >= t.ctas64) {
                *p = t;
                return true;
            }
            t.ctas64 = n * cs;
        }
        return false;
    };
    // columns in shared memory where they fit, a quarter of the launch (half a chain) at most to the panel,
    // before a larger cluster without (250 species, 40 layers on 8 CTAs 44 ms so, 30 with one CTA to the
    // panel; 400, 30 layers on 16 64 and 46; 594, 24 layers on 38 62 and 51)
    for (int cs = largest; cs >= 1; cs /= 2)
        if ((S + cs - 1) / cs <= kThreads && (cs == 1 || want >= 4 * cs) && fits(cs, 1)) return 0;
    // else in global memory, the CTAs of a small share of the SMs: the cluster that leaves a chain the
    // most of them, the largest of equals (all of a chain's CTAs, if need be: the panel is then everyone's
    // and so are the updates).  With half a chain to the panel, as above, and so: 250 species, 40 layers on
    // 4 CTAs 82 and 53 ms; 400, 30 layers on 8 123 and 75; 594, 24 layers on 4 637 and 359, on 8 323 and
    // 187.  A larger cluster that leaves CTAs over is no gain (on 6: 250 species
    // 44 ms with 1, 52 with 2; 594 325 and 347; on 12 167 with 2, 181 with 4).
    int best = 1, most = 0;
    for (int cs = largest; cs >= 1; cs /= 2)
        if (want >= 2 * cs && (cs == 1 || (S + cs - 1) / cs <= kThreads) && chain_of(ctas_of(cs), cs) > most) {
            best = cs;
            most = chain_of(ctas_of(cs), cs);
        }
    return fits(best, 0) || fits(1, 0) ? 0 : -1;
}

cudaError_t launch_factor64(const BlockSys<double> &sys, const FactorPlan &plan, Ctl *ctl, cudaStream_t st, const int *skip)
{
    // both ends at once on two halves of the grid, then the middle layer on all of it
    const int half = chain_of(plan.ctas64, plan.cs);
    if (!(plan.twisted && sys.L >= 3 && half >= 1)) return launch_mode(sys, plan, ctl, st, skip, 0, 0, plan.ctas64);
    const int mid = sys.L / 2;
    cudaError_t e = launch_mode(sys, plan, ctl, st, skip, 1, mid, 2 * half);
    if (e == cudaSuccess) e = launch_mode(sys, plan, ctl, st, skip, 2, mid, plan.ctas64);
    return e;
}

}  // namespace xk

// FP64 block Thomas elimination with explicit block inverses (the plain FP64 path, and the mixed
// path's FP64 route): Gauss-Jordan with implicit partial pivoting in panels of 8 columns, one
// persistent cooperative launch, both ends of the column at once on two halves of the grid.
//
// This part issues about two FP64 fused operations per clock and SM, so a panel of several hundred
// rows factored by one CTA, with a block barrier pair per column, is most of the time: 51 us per
// panel at 594 species (of which the other 75 SMs idle through about 40), 22 us at 96.  Here
//  - the panel belongs to a thread-block cluster, its rows spread over the cluster's CTAs, one row
//    per thread in registers.  A column costs one cluster barrier: every warp pushes its best
//    candidate row (value and the row's 8 panel entries) to all CTAs through distributed shared
//    memory, and after the barrier each CTA picks the winner from its own copy;
//  - the other CTAs apply the previous panel to their columns meanwhile (look-ahead): the cluster
//    applies it to the next panel itself.  One grid barrier per panel instead of two.
// The pivot is the unused row of largest magnitude to 20 bits (the high word of the double), the
// lowest row among equals.
//
// Pivoting is implicit: rows never move, perm_k[c] is the row that served as pivot of column c and
// iperm_k its inverse.  After factorization D holds B_k with D'^-1_k[i][j] = B_k[perm_k(i)][iperm_k(j)].
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>

#include <algorithm>

#include "xk_internal.cuh"

namespace xk {

namespace {

constexpr int kNB = 8;
constexpr int kThreads = 512;
constexpr int kWarps = kThreads / 32;
constexpr int kPS = kNB + 1;              // padded row of the panel in shared memory
constexpr size_t kSmemMax = 227 * 1024;

// A warp's best candidate for a pivot: the row's panel entries, the magnitude's high word, the row.
struct __align__(16) Cand {
    double row[kNB];
    unsigned key;
    int idx;                              // -1: the warp has no unused row
    int pad[2];
};
constexpr int kCandParts = sizeof(Cand) / 16;

__device__ __forceinline__ uint32_t smem_u32(const void *p) { return (uint32_t)__cvta_generic_to_shared(p); }
__device__ __forceinline__ uint32_t cluster_rank()
{
    uint32_t r;
    asm("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}
__device__ __forceinline__ uint32_t map_rank(uint32_t addr, int rank)
{
    uint32_t r;
    asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(rank));
    return r;
}
__device__ __forceinline__ void st_cluster(uint32_t addr, uint4 v)
{
    asm volatile("st.shared::cluster.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(addr), "r"(v.x), "r"(v.y), "r"(v.z), "r"(v.w)
                 : "memory");
}
__device__ __forceinline__ void st_cluster(uint32_t addr, int v)
{
    asm volatile("st.shared::cluster.b32 [%0], %1;" ::"r"(addr), "r"(v) : "memory");
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

// 1 / x by two Newton-Raphson steps from the hardware's approximation; the quotient itself where the
// approximation's range ends.
__device__ __forceinline__ double reciprocal(double x)
{
    const double ax = fabs(x);
    if (!(ax > 1e-290 && ax < 1e290)) return 1.0 / x;
    double y;
    asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
    y = fma(y, fma(-x, y, 1.0), y);
    return fma(y, fma(-x, y, 1.0), y);
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
            if (cs == 1) *go = ok;
            else
                for (int r = 0; r < cs; ++r) st_cluster(map_rank(smem_u32(go), r), ok);
        }
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

// mode 0: all layers top-down on the whole grid.  mode 1 (twisted): two chains on the two halves of
// the grid, layers 0 .. mid-1 top-down and L-1 .. mid+1 bottom-up.  mode 2: the middle layer on the
// whole grid, with both Schur terms.  RPT: panel rows per thread.
template <int RPT>
__global__ void __launch_bounds__(kThreads, 1)
k_factor64(BlockSys<double> a, Ctl *ctl, const int *skip, int mode, int mid, int cs)
{
    if (ctl->finished || ctl->err_timeout || (skip && *skip)) return;
    extern __shared__ __align__(16) unsigned char dyn[];
    __shared__ Cand stage[kWarps];
    __shared__ Cand cand[2][32];
    __shared__ double us[kNB * kNB];
    __shared__ int s_piv[2][kNB], s_go;
    const int S = a.S, ld = a.ld, L = a.L;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int half = mode == 1 ? (int)(blockIdx.x >= gridDim.x / 2) : 0;
    const int nblk = mode == 1 ? (int)gridDim.x / 2 : (int)gridDim.x;
    const int bid = (int)blockIdx.x - half * nblk;
    const int crank = (int)cluster_rank(), cidx = bid / cs, nclus = nblk / cs;
    const bool panel_cta = cidx == 0;
    // trailing updates: the CTAs of the other clusters, or everyone where there is only one
    const int ntrail = nclus > 1 ? nblk - cs : nblk, tq = nclus > 1 ? bid - cs : bid;
    int *pinfo = a.pinfo + 64 * half;
    ChainSync chain{a.bar + 2 * half, a.bar + 6 + half, ctl, cs, nclus, crank, &s_go, 0u};

    const int rpc = (S + cs - 1) / cs, r0 = crank * rpc, nr = max(0, min(S, r0 + rpc) - r0);
    const int nw = min(kWarps, (rpc + 31) / 32), ncand = cs * nw;     // warps with panel rows, per CTA and in all
    double *P = (double *)dyn;                       // [rpc][kPS]: the panel's rows of this CTA
    double *G = P + (size_t)rpc * kPS;               // [rpc][kPS]: the previous panel's
    double *U = G + (size_t)rpc * kPS;               // [kNB][cw]: pivot rows in this CTA's columns
    double *rowbuf = (double *)dyn + (size_t)warp * S;    // Schur term: a source row per warp

    int nsteps = L, k0 = 0, dk = 1;
    if (mode == 1) {
        nsteps = half == 0 ? mid : L - 1 - mid;
        k0 = half == 0 ? 0 : L - 1;
        dk = half == 0 ? 1 : -1;
    } else if (mode == 2) {
        nsteps = 1;
        k0 = mid;
        dk = 0;
    }
    const int npan = (S + kNB - 1) / kNB;
    int par = 0;                                     // candidate buffer of the next column
    for (int step = 0; step < nsteps; ++step) {
        const int k = k0 + step * dk;
        double *D = a.D + (size_t)k * S * ld;
        int *perm = a.perm + (size_t)k * S, *iperm = a.iperm + (size_t)k * S;
        // D_k -= diag(rowc) D'^-1_n diag(colc), D'^-1_n[i][j] = B_n[perm_n(i)][iperm_n(j)]: a warp per
        // row, the source row through shared memory
        auto schur = [&](int nbr, const double *rowc, const double *colc) {
            const double *Bn = a.D + (size_t)nbr * S * ld;
            const int *pn = a.perm + (size_t)nbr * S, *ipn = a.iperm + (size_t)nbr * S;
            for (int i = bid * kWarps + warp; i < S; i += nblk * kWarps) {
                const double *src = Bn + (size_t)__ldcg(pn + i) * ld;
                const double rc = rowc[i];
                __syncwarp();
                for (int j = lane; j < S; j += 32) rowbuf[j] = __ldcg(src + j);
                __syncwarp();
                double *Di = D + (size_t)i * ld;
                for (int j = lane; j < S; j += 32) Di[j] -= rc * rowbuf[__ldcg(ipn + j)] * colc[j];
            }
        };
        bool touched = true;
        if (mode == 2) {
            if (k > 0) schur(k - 1, a.lo + (size_t)k * S, a.up + (size_t)(k - 1) * S);
            if (k + 1 < L) schur(k + 1, a.up + (size_t)k * S, a.lo + (size_t)(k + 1) * S);
        } else if (step > 0) {
            if (dk > 0) schur(k - 1, a.lo + (size_t)k * S, a.up + (size_t)(k - 1) * S);
            else schur(k + 1, a.up + (size_t)k * S, a.lo + (size_t)(k + 1) * S);
        } else {
            touched = false;
        }
        if (touched && !chain.sync()) return;

        unsigned used = 0;                           // bit i: this thread's row i has been a pivot
#pragma unroll
        for (int i = 0; i < RPT; ++i)
            if (tid + i * kThreads >= nr) used |= 1u << i;
        for (int p = 0; p <= npan; ++p) {
            if (panel_cta && p < npan) {
                const int c0 = p * kNB, nb = min(kNB, S - c0);
                const int *pp = s_piv[(p + 1) & 1];  // the previous panel's pivot rows
                int *pc = s_piv[p & 1];
                for (int e = tid; e < nr * kNB; e += kThreads) {
                    const int r = e / kNB, j = e % kNB;
                    P[r * kPS + j] = j < nb ? __ldcg(D + (size_t)(r0 + r) * ld + c0 + j) : 0.0;
                }
                if (p > 0 && tid < kNB * kNB) {
                    const int l = tid / kNB, j = tid % kNB;
                    us[tid] = j < nb ? __ldcg(D + (size_t)pp[l] * ld + c0 + j) : 0.0;
                }
                __syncthreads();
                if (p > 0) {
                    for (int e = tid; e < nr * kNB; e += kThreads) {
                        const int r = e / kNB, j = e % kNB;
                        bool piv = false;
#pragma unroll
                        for (int l = 0; l < kNB; ++l) piv |= pp[l] == r0 + r;
                        double acc = piv ? 0.0 : P[r * kPS + j];
#pragma unroll
                        for (int l = 0; l < kNB; ++l) acc = fma(G[r * kPS + l], us[l * kNB + j], acc);
                        P[r * kPS + j] = acc;
                    }
                    __syncthreads();
                }
                double x[RPT][kNB];
#pragma unroll
                for (int i = 0; i < RPT; ++i) {
                    const int r = tid + i * kThreads;
#pragma unroll
                    for (int j = 0; j < kNB; ++j) x[i][j] = r < nr ? P[r * kPS + j] : 0.0;
                }
#pragma unroll
                for (int lc = 0; lc < kNB; ++lc) {
                    if (lc >= nb) break;
                    Cand *cb = cand[par];
                    par ^= 1;
                    if (warp < nw) {
                        // this warp's best unused row
                        unsigned key = 0u;
                        int bi = -1;
#pragma unroll
                        for (int i = 0; i < RPT; ++i) {
                            const unsigned m = (unsigned)__double2hiint(x[i][lc]) & 0x7fffffffu;
                            if (!((used >> i) & 1u) && (bi < 0 || m > key)) { key = m; bi = i; }
                        }
                        const unsigned best = __reduce_max_sync(0xffffffffu, bi >= 0 ? key + 1u : 0u);
                        const unsigned who = __ballot_sync(0xffffffffu, bi >= 0 && key + 1u == best);
                        const int src = who ? __ffs(who) - 1 : 0;
                        if (lane == src) {
                            Cand &c = stage[warp];
#pragma unroll
                            for (int i = 0; i < RPT; ++i)
                                if (i == bi || (i == 0 && bi < 0)) {
#pragma unroll
                                    for (int j = 0; j < kNB; ++j) c.row[j] = x[i][j];
                                }
                            c.key = key;
                            c.idx = who ? r0 + tid + bi * kThreads : -1;
                        }
                        __syncwarp();
                        for (int it = lane; it < cs * kCandParts; it += 32) {
                            const int dst = it / kCandParts, part = it % kCandParts;
                            const uint4 v = ((const uint4 *)&stage[warp])[part];
                            if (cs == 1) ((uint4 *)&cb[warp])[part] = v;
                            else st_cluster(map_rank(smem_u32(&cb[crank * nw + warp]) + 16u * part, dst), v);
                        }
                    }
                    cluster_sync(cs);
                    if (warp < nw) {
                        const bool have = lane < ncand && cb[lane].idx >= 0;
                        const unsigned ck = have ? cb[lane].key : 0u;
                        const unsigned top = __reduce_max_sync(0xffffffffu, have ? ck + 1u : 0u);
                        const unsigned who = __ballot_sync(0xffffffffu, have && ck + 1u == top);
                        const Cand &c = cb[who ? __ffs(who) - 1 : 0];
                        const int row = c.idx;
                        double pr[kNB];
#pragma unroll
                        for (int j = 0; j < kNB; j += 2) {
                            const double2 v = *(const double2 *)&c.row[j];
                            pr[j] = v.x;
                            pr[j + 1] = v.y;
                        }
                        // a column without a nonzero candidate: singular; the bookkeeping goes on
                        const bool zero = top <= 1u;
                        const double rcp = zero ? 0.0 : reciprocal(pr[lc]);
                        if (tid == 0) {
                            pc[lc] = row;
                            if (crank == 0) {
                                __stcg(pinfo + (p & 1) * kNB + lc, row);
                                if (zero) atomicExch(&ctl->err_singular, 1);
                            }
                        }
#pragma unroll
                        for (int i = 0; i < RPT; ++i) {
                            const int r = r0 + tid + i * kThreads;
                            const bool mine = r == row && tid + i * kThreads < nr;
                            if (mine) {
                                used |= 1u << i;
                                perm[c0 + lc] = row;
                                iperm[row] = c0 + lc;
                            }
                            // the pivot row starts from zero and takes the multiplier that leaves it scaled
                            const double f = mine ? -rcp : x[i][lc] * rcp;
#pragma unroll
                            for (int q = 1; q < kNB; ++q) {
                                const int j = (lc + q) % kNB;
                                x[i][j] = fma(-f, pr[j], mine ? 0.0 : x[i][j]);
                            }
                            x[i][lc] = -f;
                        }
                    }
                }
                // the panel's columns become G
#pragma unroll
                for (int i = 0; i < RPT; ++i) {
                    const int r = tid + i * kThreads;
                    if (r >= nr) continue;
                    double *Dr = D + (size_t)(r0 + r) * ld + c0;
#pragma unroll
                    for (int j = 0; j < kNB; ++j) {
                        G[r * kPS + j] = j < nb ? x[i][j] : 0.0;
                        if (j < nb) __stcg(Dr + j, x[i][j]);
                    }
                }
            }
            if (p > 0 && tq >= 0) {
                // panel p - 1 applied to every column but its own and panel p's (the cluster's)
                const int q0 = (p - 1) * kNB, nb = min(kNB, S - q0);
                const int c1 = q0 + nb + (p < npan ? min(kNB, S - q0 - kNB) : 0);
                const int ncol = S - (c1 - q0), per = ncol / ntrail, rest = ncol - per * ntrail;
                const int j0 = tq * per + min(tq, rest), cw = per + (tq < rest ? 1 : 0);
                if (cw > 0) {
                    const int *pq = pinfo + ((p - 1) & 1) * kNB;
                    int pr[kNB];
#pragma unroll
                    for (int l = 0; l < kNB; ++l) pr[l] = l < nb ? __ldcg(pq + l) : -1;
                    auto col = [&](int q) { return j0 + q < q0 ? j0 + q : j0 + q + (c1 - q0); };
                    __syncthreads();
                    for (int e = tid; e < kNB * cw; e += kThreads) {
                        const int l = e / cw, q = e - l * cw;
                        U[e] = l < nb ? __ldcg(D + (size_t)__ldcg(pq + l) * ld + col(q)) : 0.0;
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

size_t smem_of(int S, int cs, int ntrail)
{
    const size_t rpc = (S + cs - 1) / cs, cw = (S + ntrail - 1) / ntrail;
    const size_t panel = (2 * rpc * kPS + kNB * cw) * sizeof(double);
    const size_t rows = (size_t)kWarps * S * sizeof(double);
    return (std::max(panel, rows) + 255) & ~(size_t)255;
}

cudaError_t launch_mode(const BlockSys<double> &sys, const FactorPlan &plan, Ctl *ctl, cudaStream_t st, const int *skip,
                        int mode, int mid, int ctas)
{
    const int rpc = (sys.S + plan.cs - 1) / plan.cs;
    auto fn = rpc <= kThreads ? k_factor64<1> : k_factor64<2>;
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

}  // namespace

int factor64_plan(int S, int want, FactorPlan *p)
{
    if (S <= 0 || S > 2 * kThreads || want < 1) return -1;
    // The panel's cluster: a column's barrier costs more across CTAs than the rows it spreads save until
    // there are about 130 rows (S = 96: 52 ms for four steps with one CTA, 59 with 4 or 8); beyond 500
    // rows the trailing updates want the CTAs (S = 594: 118 ms a solve with 4, 135 with 8; S = 250 at 60
    // layers: 17.3 and 16.7, 21.7 with one).
    for (int cs = S <= 128 ? 1 : S <= 500 ? 8 : 4; cs >= 1; cs /= 2) {
        if (want < 4 * cs && cs > 1) continue;
        const int rpc = (S + cs - 1) / cs;
        if (cs > 1 && rpc > kThreads) continue;
        // a chain beyond the cluster has at most a CTA per 4 columns
        const int chain = cs + std::max(1, (S + 3) / 4 / cs) * cs;
        int ctas = std::min(want, 2 * chain) / cs * cs;
        const size_t smem = smem_of(S, cs, std::max(1, ctas / 2 / cs * cs - cs));
        if (smem > kSmemMax) continue;
        auto fn = rpc <= kThreads ? k_factor64<1> : k_factor64<2>;
        if (cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) != cudaSuccess) {
            cudaGetLastError();
            continue;
        }
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3(cs);
        cfg.blockDim = dim3(kThreads);
        cfg.dynamicSmemBytes = smem;
        cudaLaunchAttribute attr[1];
        attr[0].id = cudaLaunchAttributeClusterDimension;
        attr[0].val.clusterDim.x = cs;
        attr[0].val.clusterDim.y = 1;
        attr[0].val.clusterDim.z = 1;
        cfg.attrs = attr;
        cfg.numAttrs = 1;
        int n = 0;
        if (cudaOccupancyMaxActiveClusters(&n, fn, &cfg) != cudaSuccess || n < 1) {
            cudaGetLastError();
            continue;
        }
        ctas = std::min(ctas, n * cs);
        p->cs = cs;
        p->ctas64 = ctas;
        p->smem64 = std::max(smem, smem_of(S, cs, std::max(1, ctas / 2 / cs * cs - cs)));
        if (p->smem64 > kSmemMax) continue;
        return 0;
    }
    return -1;
}

cudaError_t launch_factor64(const BlockSys<double> &sys, const FactorPlan &plan, Ctl *ctl, cudaStream_t st, const int *skip)
{
    // both ends at once on two halves of the grid, then the middle layer on all of it
    const int half = plan.ctas64 / 2 / plan.cs * plan.cs;
    if (!(plan.twisted && sys.L >= 3 && half >= 1)) return launch_mode(sys, plan, ctl, st, skip, 0, 0, plan.ctas64);
    const int mid = sys.L / 2;
    cudaError_t e = launch_mode(sys, plan, ctl, st, skip, 1, mid, 2 * half);
    if (e == cudaSuccess) e = launch_mode(sys, plan, ctl, st, skip, 2, mid, plan.ctas64);
    return e;
}

}  // namespace xk

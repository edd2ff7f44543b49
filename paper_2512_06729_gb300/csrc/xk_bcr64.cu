// Block cyclic reduction in FP64 (the plain FP64 path's factorization for blocks of at most 152 rows).
//
// The block elimination from both ends (xk_factor64.cu) is a chain of L / 2 layers with S columns
// each, and at these sizes it is all latency: 2,900 clocks per column, 11 ms for 96 species and 150
// layers, of which the arithmetic would take 0.25.  The reduction does four times the arithmetic, but
// in a chain of log2 L inversions: every second layer of a level is inverted at once, and the products
// that eliminate them are spread over the chip.  It pays while a block fits in the shared memory of a
// cluster and the arithmetic stays short against the chain: the factorization takes 1.8 ms at 96
// species and 150 layers (nine inversions in a row of 195 to 90 us, products 0.84 ms), and a step
// 11.9 ms with the elimination, 2.2 with the reduction (17.4 and 3.1 at 120 species and 90 layers).
//
// k_inv64: one block per cluster, columns dealt out over its CTAs, Gauss-Jordan in place with implicit
// partial pivoting.  The owner of column c sends it, as it stands, to every CTA of the cluster
// (asynchronous stores that complete on the receiver's mbarrier); there a lead warp turns it into the
// multipliers, applies them to the next column this CTA will have to send, and hands them to the other
// warps, which update the rest of its columns behind it.  Every column has its own place and its own
// barriers, each used once, so nobody waits for room.  A column costs one trip between CTAs, a
// reciprocal (beside the pivot search) and three dependent products: 0.9 us, which bounds every level
// but the lowest two, where there are too few SMs for 96 columns of 75 blocks.
#include <algorithm>
#include <cstring>

#include "xk_bcr.cuh"
#include "xk_mbar.cuh"

namespace xk {

namespace {

constexpr int kInvThreads = 256;
constexpr int kInvBusy = 96;              // FP64 instructions of a step above which warp 4 works too
constexpr size_t kInvSmemMax = 220 * 1024;

// Asynchronous store of 8 bytes into a CTA of the cluster, counted by that CTA's mbarrier.
__device__ __forceinline__ void st_async(uint32_t addr, unsigned long long v, uint32_t mbar)
{
    asm volatile("st.async.shared::cluster.mbarrier::complete_tx::bytes.b64 [%0], %1, [%2];" ::"r"(addr), "l"(v), "r"(mbar)
                 : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint32_t bar)
{
    asm volatile("mbarrier.arrive.release.cta.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ void cluster_sync()
{
    asm volatile("barrier.cluster.arrive.release;" ::: "memory");
    asm volatile("barrier.cluster.wait.acquire;" ::: "memory");
}
__device__ __forceinline__ void grid_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void grid_trigger() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

// Shared memory of one CTA: its columns, every column's message (S rows, then the pivot's row as an
// integer and the pivot's reciprocal), the barriers of messages, multipliers and handed-over columns, pivots by column and by row.
struct InvLayout {
    int ncol, slot;                        // columns of a CTA, words of a message
    size_t slots, bars, ints, bytes;
};
__host__ __device__ inline InvLayout inv_layout(int S, int cs)
{
    InvLayout l;
    l.ncol = (S + cs - 1) / cs;
    l.slot = S + 2;
    l.slots = (size_t)l.ncol * S;
    l.bars = l.slots + (size_t)S * l.slot;
    l.ints = l.bars + 2 * (size_t)S + l.ncol;
    l.bytes = (l.ints + S) * 8;
    return l;
}

template <int RPT>
__global__ void __launch_bounds__(kInvThreads, 1) k_inv64(const Bcr64Inv *tasks, int S, int ldin, int ld, int cs, Ctl *ctl)
{
    grid_trigger();
    grid_wait();
    if (ctl->finished) return;
    extern __shared__ __align__(16) double sm[];
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, rank = (int)cluster_rank();
    const Bcr64Inv task = tasks[blockIdx.x / cs];
    const InvLayout lay = inv_layout(S, cs);
    double *cols = sm, *slots = sm + lay.slots;
    const uint32_t bar0 = smem_u32(sm + lay.bars), ready0 = bar0 + 8 * S, handed0 = ready0 + 8 * S;
    int *prow = (int *)(sm + lay.ints), *rcol = prow + S;
    const int ncol = (S - rank + cs - 1) / cs;         // columns rank, rank + cs, ...
    for (int i = tid; i < S; i += kInvThreads) {
        mbar_init(bar0 + 8 * i);
        mbar_init(ready0 + 8 * i);
        if (i < lay.ncol) mbar_init(handed0 + 8 * i);
        rcol[i] = prow[i] = 0;
    }
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    for (int i = tid; i < S; i += kInvThreads) mbar_expect(bar0 + 8 * i, 8 * (S + 2));
    for (int e = tid; e < ncol * S; e += kInvThreads) {
        const int i = e / ncol, l = e - i * ncol;
        cols[l * S + i] = task.in[(size_t)i * ldin + rank + cs * l];
    }
    __syncthreads();
    cluster_sync();                                     // every CTA's barriers stand
    if (warp == 0) {
        // the lead: own column j in registers, taken from the others cs steps before it is the pivot's
        int j = rank, l = 0;
        double a[RPT];
        unsigned used = 0;                              // bit t: row 32 t + lane was a pivot
#pragma unroll
        for (int t = 0; t < RPT; ++t) a[t] = j < S && t * 32 + lane < S ? cols[t * 32 + lane] : 0.0;
        for (int c = 0; c < S; ++c) {
            if (c == j) {
                unsigned key = 0;
                int bi = 0;
                double best = 1.0;
#pragma unroll
                for (int t = 0; t < RPT; ++t) {
                    const unsigned k = t * 32 + lane < S && !(used >> t & 1)
                                           ? ((unsigned)__double2hiint(a[t]) & 0x7fffffffu) + 1u : 0u;
                    if (k > key) {
                        key = k;
                        bi = t * 32 + lane;
                        if (k > 1u) best = a[t];
                    }
                }
                // every candidate's reciprocal beside the search
                const double rbest = reciprocal64(best);
                const unsigned top = __reduce_max_sync(0xffffffffu, key);
                const int win = __ffs(__ballot_sync(0xffffffffu, key == top)) - 1;
                const int p = __shfl_sync(0xffffffffu, bi, win);
                if (top <= 1u && lane == 0) atomicExch(&ctl->err_singular, 1);
                const uint32_t to = smem_u32(slots + (size_t)c * lay.slot);
                const double rsend = __shfl_sync(0xffffffffu, rbest, win);
                for (int q = 1; q <= cs; ++q) {         // the next column's owner first
                    const int r = (rank + q) & (cs - 1);
                    const uint32_t addr = map_rank(to, r), mb = map_rank(bar0 + 8 * c, r);
#pragma unroll
                    for (int t = 0; t < RPT; ++t)
                        if (t * 32 + lane < S)
                            st_async(addr + 8 * (t * 32 + lane), (unsigned long long)__double_as_longlong(a[t]), mb);
                    if (lane == 0) {
                        st_async(addr + 8 * S, (unsigned long long)p, mb);
                        st_async(addr + 8 * S + 8, (unsigned long long)__double_as_longlong(rsend), mb);
                    }
                }
            }
            double *v = slots + (size_t)c * lay.slot;
            mbar_wait(bar0 + 8 * c, 0u, ctl);
            const int p = min(max(((const int *)(v + S))[0], 0), S - 1);
            const double rp = v[S + 1];
            double w[RPT];
#pragma unroll
            for (int t = 0; t < RPT; ++t) w[t] = t * 32 + lane < S ? v[t * 32 + lane] : 0.0;
#pragma unroll
            for (int t = 0; t < RPT; ++t) {
                const bool piv = t * 32 + lane == p;
                w[t] = piv ? rp : -(w[t] * rp);
                if (piv) used |= 1u << t;
            }
            __syncwarp();
#pragma unroll
            for (int t = 0; t < RPT; ++t)
                if (t * 32 + lane < S) {
                    v[t * 32 + lane] = w[t];
                    if (c == j) cols[l * S + t * 32 + lane] = w[t];
                }
            if (lane == 0) {
                prow[c] = p;
                rcol[p] = c;
            }
            __syncwarp();
            if (lane == 0) mbar_arrive(ready0 + 8 * c);
            if (c == j) {
                j += cs;
                ++l;
                if (j < S) {
                    if (c > 0) mbar_wait(handed0 + 8 * l, 0u, ctl);   // all steps before c are in it
#pragma unroll
                    for (int t = 0; t < RPT; ++t) a[t] = t * 32 + lane < S ? cols[l * S + t * 32 + lane] : 0.0;
                }
            }
            // step c on the lead's column
            double ap = a[0];
#pragma unroll
            for (int t = 1; t < RPT; ++t)
                if (p >> 5 == t) ap = a[t];
            ap = __shfl_sync(0xffffffffu, ap, p & 31);
#pragma unroll
            for (int t = 0; t < RPT; ++t) a[t] = fma(w[t], ap, t * 32 + lane == p ? 0.0 : a[t]);
        }
    } else {
        // column l belongs to one warp throughout; of its columns, the ones due next come first
        // (warp 4 shares the lead's FP64 unit: it works only where the units are what bounds the step)
        const bool four = ncol * RPT > kInvBusy;
        const int nwk = four ? 7 : 6, wk = warp == 4 ? (four ? 3 : ncol) : warp - 1 - (warp > 4 && !four);
        const int own = wk < ncol ? (ncol - wk + nwk - 1) / nwk : 0;
        int first = 0, m0 = 0;                          // the lead's column (first after c), own's first behind it
        for (int c = 0; c < S; ++c) {
            if (rank + cs * first <= c) ++first;
            while (m0 < own && wk + nwk * m0 <= first) ++m0;
            mbar_wait(ready0 + 8 * c, 0u, ctl);
            const double *v = slots + (size_t)c * lay.slot;
            const int p = prow[c];
            double w[RPT];
#pragma unroll
            for (int t = 0; t < RPT; ++t) w[t] = t * 32 + lane < S ? v[t * 32 + lane] : 0.0;
            for (int q = 0; q < own; ++q) {
                int m = m0 + q;
                if (m >= own) m -= own;
                const int l = wk + nwk * m, j = rank + cs * l;
                if (l == first || j == c) continue;     // the lead's
                double *x = cols + l * S;
                const double ap = x[p];
                double y[RPT];
#pragma unroll
                for (int t = 0; t < RPT; ++t) y[t] = t * 32 + lane < S && t * 32 + lane != p ? x[t * 32 + lane] : 0.0;
                __syncwarp();
#pragma unroll
                for (int t = 0; t < RPT; ++t)
                    if (t * 32 + lane < S) x[t * 32 + lane] = fma(w[t], ap, y[t]);
                __syncwarp();
                if (j - cs - 1 == c && lane == 0) mbar_arrive(handed0 + 8 * l);
            }
        }
    }
    __syncthreads();
    // A^-1[c][prow[d]] = W[prow[c]][d]
    for (int e = tid; e < ncol * S; e += kInvThreads) {
        const int l = e / S, i = e - l * S;
        task.out[(size_t)rcol[i] * ld + prow[rank + cs * l]] = cols[e];
    }
    cluster_sync();                                     // none leaves while another may still send to it
}

// Level 0 (diagonal couplings), for each kept even layer i with eliminated neighbours l = i-1, r = i+1:
//   D_i -= diag(lo_i) INV_l diag(up_l) + diag(up_i) INV_r diag(lo_r)
//   CP(1, i/2) = [ -diag(lo_i) INV_l diag(lo_l) | -diag(up_i) INV_r diag(up_r) ]
__global__ void __launch_bounds__(256) k_level0_64(double *D, const double *INV, double *CP, const double *lo,
                                                    const double *up, int L, int S, int ldd, int ld, const Ctl *ctl)
{
    grid_trigger();
    grid_wait();
    if (ctl->finished) return;
    const int i = 2 * blockIdx.y, e = blockIdx.x * 256 + threadIdx.x;
    if (e >= S * S) return;
    const int y = e / S, c = e - y * S;
    const size_t blk = (size_t)S * ld, at = (size_t)y * ld + c;
    double *cp = CP + (size_t)(i / 2) * 2 * blk + (size_t)y * 2 * ld + c;
    double upd = 0.0;
    if (i >= 1) {
        const double g = lo[(size_t)i * S + y] * INV[(i - 1) * blk + at];
        upd += g * up[(size_t)(i - 1) * S + c];
        if (i >= 2) cp[0] = -(g * lo[(size_t)(i - 1) * S + c]);
    }
    if (i + 1 < L) {
        const double g = up[(size_t)i * S + y] * INV[(i + 1) * blk + at];
        upd += g * lo[(size_t)(i + 1) * S + c];
        if (i + 2 < L) cp[ld] = -(g * up[(size_t)(i + 1) * S + c]);
    }
    D[(size_t)i * S * ldd + (size_t)y * ldd + c] -= upd;
}

// C = src + sign (A0 B0 + A1 B1), S x S each: one 16 x 16 tile of one task per CTA, two entries per
// thread, both operands' panels in shared memory whole.  Bound by FP64 issue (two multiply-adds per
// thread and k); tiles this small because a level of the reduction has few blocks, and because shared
// memory has time to spare beside FP64 units of this rate.  The lowest level's 221 products of 96 rows
// take 360 us, which is that rate; the last levels' 13 us are the latency of one tile.
constexpr int kTile = 16;
__global__ void __launch_bounds__(128) k_gemm64(const Bcr64Gemm *tasks, int S, const Ctl *ctl)
{
    grid_trigger();
    grid_wait();
    if (ctl->finished) return;
    extern __shared__ __align__(16) double sm[];
    const int nt = (S + kTile - 1) / kTile, per = nt * nt, tid = threadIdx.x;
    const Bcr64Gemm t = tasks[blockIdx.x / per];
    const int tile = blockIdx.x % per, i0 = tile / nt * kTile, j0 = tile % nt * kTile;
    const int lda = S + 1, nseg = t.a1 ? 2 : 1;        // odd or even, rows lie in different banks
    double *As = sm, *Bs = sm + (size_t)2 * kTile * lda;
    auto fetch = [](double *dst, const double *src, bool in) {
        const int bytes = in ? 8 : 0;                  // zero outside
        asm volatile("cp.async.ca.shared.global [%0], [%1], 8, %2;" ::"r"(smem_u32(dst)), "l"(src), "r"(bytes) : "memory");
    };
    for (int s = 0; s < nseg; ++s) {
        const double *A = s ? t.a1 : t.a0, *B = s ? t.b1 : t.b0;
        for (int e = tid; e < kTile * S; e += 128) {
            const int i = e / S, k = e - i * S;
            const bool in = i0 + i < S;
            fetch(As + (s * kTile + i) * lda + k, in ? A + (size_t)(i0 + i) * t.lda + k : A, in);
        }
        for (int e = tid; e < kTile * S; e += 128) {
            const int k = e / kTile, j = e % kTile;
            const bool in = j0 + j < S;
            fetch(Bs + ((size_t)s * S + k) * kTile + j, in ? B + (size_t)k * t.ldb + j0 + j : B, in);
        }
    }
    asm volatile("cp.async.commit_group;\n\tcp.async.wait_group 0;" ::: "memory");
    __syncthreads();
    const int j = tid % kTile, i = tid / kTile;
    double c0[2] = {0.0, 0.0}, c1[2] = {0.0, 0.0};
    for (int s = 0; s < nseg; ++s) {
        const double *a0 = As + (s * kTile + i) * lda, *a1 = a0 + kTile / 2 * lda, *b = Bs + (size_t)s * S * kTile + j;
        int k = 0;
#pragma unroll 4
        for (; k + 2 <= S; k += 2) {
            const double b0 = b[k * kTile], b1 = b[(k + 1) * kTile];
            c0[0] = fma(a0[k], b0, c0[0]);
            c1[0] = fma(a1[k], b0, c1[0]);
            c0[1] = fma(a0[k + 1], b1, c0[1]);
            c1[1] = fma(a1[k + 1], b1, c1[1]);
        }
        if (k < S) {
            c0[0] = fma(a0[k], b[k * kTile], c0[0]);
            c1[0] = fma(a1[k], b[k * kTile], c1[0]);
        }
    }
    if (j0 + j < S) {
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int r = i0 + i + h * (kTile / 2);
            if (r >= S) continue;
            const double v = h ? c1[0] + c1[1] : c0[0] + c0[1];
            const size_t at = (size_t)r * t.ldc + j0 + j;
            t.c[at] = (t.src ? t.src[at] : 0.0) + t.sign * v;
        }
    }
}

// The factorization's stages and tasks; pointers into arrays that may not exist yet (sizes only).
void build(Bcr64Plan &p, int L, int S, int ldd)
{
    p.L = L;
    p.S = S;
    const int ld = p.ld = (S + 1) / 2 * 2;
    p.ldd = ldd;
    p.inv.clear(); p.gemm.clear(); p.mv.clear(); p.fac.clear(); p.sol.clear();
    const BcrLevels lv(L);
    const auto &lists = lv.lists;
    p.levels = (int)lists.size() - 1;
    const size_t blk = (size_t)S * ld;
    auto D = [&](int k) { return p.D + (size_t)k * S * ldd; };
    auto INV = [&](int k) { return p.INV + k * blk; };
    auto CP = [&](int q, int half) { return p.CP + q * 2 * blk + half * ld; };
    auto PQ = [&](int k, int half) { return p.PQ + k * 2 * blk + half * ld; };
    auto stage = [&](int kind, int off, int count, int level) { p.fac.push_back(BcrStage{kind, off, count, 0, 0, level}); };
    for (int l = 0; l < p.levels; ++l) {
        const auto &a = lists[l];
        const int i0 = (int)p.inv.size();
        for (size_t q = 1; q < a.size(); q += 2) p.inv.push_back(Bcr64Inv{D(a[q]), INV(a[q])});
        stage(kBcrLeafStage, i0, (int)p.inv.size() - i0, l);
        if (l == 0) {
            stage(kBcrLevel0, 0, (L + 1) / 2, 0);
            continue;
        }
        const int g0 = (int)p.gemm.size(), off = lv.cp_off[l];
        // [P_j | Q_j] = D_j^-1 [L_j | U_j]
        for (size_t q = 1; q < a.size(); q += 2)
            for (int half = 0; half < (q + 1 < a.size() ? 2 : 1); ++half)
                p.gemm.push_back(Bcr64Gemm{INV(a[q]), CP(off + (int)q, half), nullptr, nullptr, nullptr, PQ(a[q], half), 1.0,
                                           ld, 2 * ld, 2 * ld});
        stage(kBcrGemm, g0, (int)p.gemm.size() - g0, l);
        const int g1 = (int)p.gemm.size();
        // Schur complements and the couplings of the next level
        for (size_t q = 0; q < a.size(); q += 2) {
            const bool hl = q >= 1, hr = q + 1 < a.size();
            if (!hl && !hr) continue;
            const int cpi = off + (int)q, cpn = lv.cp_off[l + 1] + (int)(q / 2);
            Bcr64Gemm t{nullptr, nullptr, nullptr, nullptr, D(a[q]), D(a[q]), -1.0, 2 * ld, 2 * ld, ldd};
            if (hr) { t.a0 = CP(cpi, 1); t.b0 = PQ(a[q + 1], 0); }                       // U_i P_r
            if (hl) { (hr ? t.a1 : t.a0) = CP(cpi, 0); (hr ? t.b1 : t.b0) = PQ(a[q - 1], 1); }   // L_i Q_l
            p.gemm.push_back(t);
            if (hl && q >= 2)                            // L_i <- -L_i P_l
                p.gemm.push_back(Bcr64Gemm{CP(cpi, 0), PQ(a[q - 1], 0), nullptr, nullptr, nullptr, CP(cpn, 0), -1.0,
                                           2 * ld, 2 * ld, 2 * ld});
            if (hr && q + 2 < a.size())                  // U_i <- -U_i Q_r
                p.gemm.push_back(Bcr64Gemm{CP(cpi, 1), PQ(a[q + 1], 1), nullptr, nullptr, nullptr, CP(cpn, 1), -1.0,
                                           2 * ld, 2 * ld, 2 * ld});
        }
        stage(kBcrGemm, g1, (int)p.gemm.size() - g1, l);
    }
    const int i0 = (int)p.inv.size(), root = lists.back()[0];
    p.inv.push_back(Bcr64Inv{D(root), INV(root)});
    stage(kBcrLeafStage, i0, 1, p.levels);
    bcr_solve_tasks(lv, BcrArrays<double>{p.INV, p.CP, p.PQ, p.lo, p.up, p.bw, p.tw, p.xw, L, S, S, ld}, p.mv, p.sol);
}

// CTAs to a cluster: as many as leave every block of the level a cluster at once, of those that hold
// the block; a block of 32 rows is quicker on one (no trip between CTAs).
int inv_cluster(int S, int count)
{
    int cs = 1;
    while (cs < 8 && inv_layout(S, cs).bytes > kInvSmemMax) cs *= 2;
    if (S > 32)
        while (cs < 8 && cs * 2 * count <= 152) cs *= 2;
    return cs;
}

template <int RPT>
cudaError_t launch_inv_rpt(const Bcr64Plan &p, const BcrStage &s, Ctl *ctl, cudaStream_t st)
{
    const int S = p.S, count = s.count;
    const int cs = inv_cluster(S, count);
    const InvLayout lay = inv_layout(S, cs);
    const cudaError_t e = allow_smem(k_inv64<RPT>, kInvSmemMax);
    if (e != cudaSuccess) return e;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(count * cs);
    cfg.blockDim = dim3(kInvThreads);
    cfg.dynamicSmemBytes = lay.bytes;
    cfg.stream = st;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = cs;
    at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    count_launches(1);
    return cudaLaunchKernelEx(&cfg, k_inv64<RPT>, (const Bcr64Inv *)(p.inv_d + s.off), S, p.ldd, p.ld, cs, ctl);
}

size_t gemm_bytes(int S) { return (size_t)2 * kTile * (S + 1 + S) * sizeof(double); }

}  // namespace

Bcr64Sizes bcr64_sizes(int L, int S)
{
    Bcr64Plan p;
    build(p, L, S, S);
    const size_t ld = p.ld, blk = S * ld;
    const BcrLevels lv(L);
    return Bcr64Sizes{(int)p.inv.size(), (int)p.gemm.size(), (int)p.mv.size(), (int)p.sol.size(),
                      L * blk, std::max(lv.ncp, 1) * 2 * blk, (size_t)L * 2 * blk, (size_t)L * ld};
}

cudaError_t bcr64_build(Bcr64Plan &p, int L, int S, int ldd, cudaStream_t st)
{
    if (S > kBcr64Max || ldd < S) return cudaErrorInvalidValue;
    build(p, L, S, ldd);
    // the task lists lie one behind the other (with the allocator's gaps): one copy for the four
    std::vector<char> image;
    auto put = [&](const auto *dst, const auto &v) {
        const size_t at = (const char *)dst - (const char *)p.inv_d, bytes = v.size() * sizeof(v[0]);
        if (image.size() < at + bytes) image.resize(at + bytes);
        if (bytes) memcpy(image.data() + at, v.data(), bytes);
    };
    put(p.inv_d, p.inv);
    put(p.gemm_d, p.gemm);
    put(p.mv_d, p.mv);
    put(p.sol_d, p.sol);
    cudaError_t e = cudaMemcpyAsync(p.inv_d, image.data(), image.size(), cudaMemcpyHostToDevice, st);
    // a padding column is read by the solve and written by nobody
    if (p.ld != S) {
        const size_t blk = (size_t)S * p.ld, vec = (size_t)L * p.ld;
        double *arr[] = {p.INV, p.CP, p.PQ, p.bw, p.tw, p.xw};
        const size_t len[] = {L * blk, std::max(BcrLevels(L).ncp, 1) * 2 * blk, 2 * L * blk, vec, vec, vec};
        for (int i = 0; i < 6; ++i)
            if (e == cudaSuccess) e = cudaMemsetAsync(arr[i], 0, len[i] * sizeof(double), st);
    }
    // the host copy must outlive the asynchronous one
    return e == cudaSuccess ? cudaStreamSynchronize(st) : e;
}

cudaError_t bcr64_factor(const Bcr64Plan &p, Ctl *ctl, cudaStream_t st)
{
    cudaError_t e = allow_smem(k_gemm64, gemm_bytes(kBcr64Max));
    if (e != cudaSuccess) return e;
    const int nt = (p.S + kTile - 1) / kTile;
    for (const BcrStage &s : p.fac) {
        if (s.kind == kBcrLeafStage) {
            switch ((p.S + 31) / 32) {
            case 1: e = launch_inv_rpt<1>(p, s, ctl, st); break;
            case 2: e = launch_inv_rpt<2>(p, s, ctl, st); break;
            case 3: e = launch_inv_rpt<3>(p, s, ctl, st); break;
            case 4: e = launch_inv_rpt<4>(p, s, ctl, st); break;
            default: e = launch_inv_rpt<5>(p, s, ctl, st); break;
            }
        } else if (s.kind == kBcrGemm) {
            count_launches(1);
            e = launch_dependent(k_gemm64, dim3(s.count * nt * nt), dim3(128), gemm_bytes(p.S), st, p.gemm_d + s.off, p.S,
                                 (const Ctl *)ctl);
        } else {
            count_launches(1);
            e = launch_dependent(k_level0_64, dim3((p.S * p.S + 255) / 256, s.count), dim3(256), 0, st, p.D,
                                 (const double *)p.INV, p.CP, p.lo, p.up, p.L, p.S, p.ldd, p.ld, (const Ctl *)ctl);
        }
        if (e != cudaSuccess) return e;
    }
    return cudaGetLastError();
}

}  // namespace xk

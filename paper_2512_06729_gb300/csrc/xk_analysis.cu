// Chemical-equilibrium initial state (Sec. 2.5, option (i)) and the reaction-pathway analyser
// (Sec. 4) on the GPU.
//
// Equilibrium: one CTA per layer finds the ideal-gas mixture of minimum Gibbs energy at the layer's
// T and P for given element totals.  The unknowns are ln N_y of every species, the total ln N and
// one potential pi_e per element; each Newton iteration reduces to an (E+1) x (E+1) system (the
// reduced Gibbs iteration of the NASA equilibrium program, Gordon & McBride 1994).  The species
// loop (exp, chemical potentials, the update) is spread over the CTA's threads, the system's sums
// over species over its lanes in sublists of fixed order, and one warp solves the small system with
// partial pivoting.  At convergence the mole fractions are rebuilt from the
// potentials, x_y = exp(sum_e pi_e a_ey - G_y/RT - ln P), so trace species keep full relative
// accuracy however small.
//
// Pathways: one warp per (source, layer) runs Dijkstra on the layer's reaction graph with edge
// weights 1/rate (the kinetically fastest route minimises the summed inverse rates).  The graph is
// the same in every layer (built on the host from the network); the weights come from that
// layer's forward and reverse rates.  Distances, the predecessor tree and each path's slowest step
// are kept in shared memory until the warp writes them out.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>

#include "xk_internal.cuh"

namespace xk {
namespace {

constexpr int kEqThreads = 256;
constexpr int kEqMaxE = 31;              // E + 1 rows of the Newton system fit one warp
constexpr double kLnMajor = -18.420680743952367;   // ln 1e-8: species above this fraction are "major"
constexpr double kTraceCap = 9.2103;               // a trace species may rise to about 1e-4 of N per step

constexpr int kEqWarps = kEqThreads / 32;

struct EqShared {
    double A[kEqMaxE + 1][kEqMaxE + 2];  // the (E+1) x (E+1) system with its right-hand side
    double sol[kEqMaxE + 1];
    double bk[kEqMaxE];
    double red[2][kEqWarps];
    unsigned long long kred[2][kEqWarps];
    double lntot, bsum;
    int eact[kEqMaxE], ired[kEqWarps];
    int singular;
};

__device__ __forceinline__ double warp_sum(double v)
{
    for (int o = 16; o; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

// Largest (least) bit pattern of the warp: non-negative doubles order like them, and two integer
// reductions take a tenth of an FP64 comparison tree.
__device__ __forceinline__ unsigned long long warp_max_key(unsigned long long k)
{
    const unsigned h = (unsigned)(k >> 32), mh = __reduce_max_sync(0xffffffffu, h);
    const unsigned ml = __reduce_max_sync(0xffffffffu, h == mh ? (unsigned)k : 0u);
    return (unsigned long long)mh << 32 | ml;
}
__device__ __forceinline__ unsigned long long key_of(double d) { return (unsigned long long)__double_as_longlong(d); }

// Block-wide sums of two values, the same in every thread.
__device__ void block_sum2(EqShared &sh, double &a, double &b)
{
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    a = warp_sum(a);
    b = warp_sum(b);
    if (lane == 0) {
        sh.red[0][w] = a;
        sh.red[1][w] = b;
    }
    __syncthreads();
    // both sums in one tree: lanes 0 .. 7 the first, 8 .. 15 the second
    double v = lane < 2 * kEqWarps ? sh.red[lane / kEqWarps][lane % kEqWarps] : 0.0;
    for (int o = kEqWarps / 2; o; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    a = __shfl_sync(0xffffffffu, v, 0);
    b = __shfl_sync(0xffffffffu, v, kEqWarps);
    __syncthreads();
}

// Gauss-Jordan with implicit partial pivoting of the M x (M+1) augmented system on the first four
// warps, one to each FP64 unit of the SM: lane r stands for row r, warp w updates the columns j = w
// (mod 4), pivot and multipliers are found by all four alike.  Eliminating above the pivot costs no
// more instructions than below and leaves no back substitution (M (M+1) / 2 dependent results on one
// lane before).  The pivot is the unused row of largest magnitude by its high word, the first among
// equals.  Column c is only read in step c, so one barrier per step does.
constexpr int kSolveWarps = 4;
__device__ void warps_solve(EqShared &sh, int M)
{
    const int lane = threadIdx.x & 31, wrp = threadIdx.x >> 5;
    bool used = lane >= M;
    int mycol = 0;
    double myrcp = 0.0;
    for (int c = 0; c < M; ++c) {
        const double v = lane < M ? sh.A[lane][c] : 0.0;
        const unsigned key = used ? 0u : (unsigned)__double2hiint(v) & 0x7fffffffu;
        const unsigned top = __reduce_max_sync(0xffffffffu, key);
        if (top == 0u || top > 0x7ff00000u) {          // nothing left, or not a number: in all four warps
            if (lane == 0) sh.singular = 1;
            return;
        }
        const int p = __ffs(__ballot_sync(0xffffffffu, !used && key == top)) - 1;
        const double rcp = reciprocal64(sh.A[p][c]);
        if (lane == p) {
            used = true;
            mycol = c;
            myrcp = rcp;
        }
        if (lane < M && lane != p) {
            const double l = -(v * rcp);
            for (int j = c + 1 + ((wrp - c - 1) & (kSolveWarps - 1)); j <= M; j += kSolveWarps)
                sh.A[lane][j] = fma(l, sh.A[p][j], sh.A[lane][j]);
        }
        asm volatile("bar.sync 1, %0;" ::"n"(32 * kSolveWarps) : "memory");
    }
    if (wrp == 0 && lane < M) sh.sol[mycol] = sh.A[lane][M] * myrcp;
}

// Dynamic shared memory: lnN, nj, mu [S] doubles, the entries' parts [2 nsub] doubles (sums of nj and
// of nj mu), then the activity flags [S] as bytes.  Bound by FP64 issue (a warp instruction holds its
// unit, one to four warps, for 65 clocks whatever its lanes do): per iteration the exponentials, then
// the system's chain of M pivots.  At 594 species x 150 layers an iteration takes 25 us; with one thread
// to an entry (the longest some 550 terms), divisions and a back substitution on one lane it took 110.
__global__ void __launch_bounds__(kEqThreads) k_equilibrium(Col c, EqIndex ix, const double *b, double *x,
                                                             double *nout, int max_iter, double tol, int *iters,
                                                             int *status)
{
    __shared__ EqShared sh;
    extern __shared__ double eq_dyn[];
    const int S = c.S, E = c.E, M = c.E + 1, k = blockIdx.x, tid = threadIdx.x, lane = tid & 31, wrp = tid >> 5;
    double *lnN = eq_dyn, *nj = lnN + S, *mu = nj + S, *part = mu + S;
    unsigned char *act = (unsigned char *)(part + 2 * ix.nsub);
    const double *g = c.grt + (size_t)k * S;
    const double lnP = log(c.P[k]);

    // element totals: a warp per element
    for (int e = wrp; e < E; e += kEqWarps) {
        double v = 0.0;
        if (b) v = b[(size_t)k * E + e];
        else {
            for (int y = lane; y < S; y += 32) v += (double)c.elem[y * E + e] * c.n[(size_t)k * S + y];
            v = warp_sum(v);
        }
        if (lane == 0) {
            sh.bk[e] = v;
            sh.eact[e] = v > 0.0;
        }
    }
    __syncthreads();
    if (tid == 0) {
        double s = 0.0;
        for (int e = 0; e < E; ++e)
            if (sh.eact[e]) s += sh.bk[e];
        sh.bsum = s;
        sh.lntot = 0.0;
        sh.singular = 0;
    }
    int cnt = 0;
    for (int y = tid; y < S; y += kEqThreads) {
        int on = 1;
        for (int q = ix.sp[y]; q < ix.sp[y + 1]; ++q)
            if (!sh.eact[ix.se[q]]) on = 0;
        act[y] = (unsigned char)on;
        cnt += on;
    }
    cnt = __reduce_add_sync(0xffffffffu, cnt);
    if (lane == 0) sh.ired[wrp] = cnt;
    __syncthreads();
    int nact = 0;
    for (int i = 0; i < kEqWarps; ++i) nact += sh.ired[i];
    if (nact == 0 || !(sh.bsum > 0.0)) {
        if (tid == 0) {
            iters[k] = 0;
            status[k] = -1;
        }
        return;
    }
    for (int y = tid; y < S; y += kEqThreads) {
        lnN[y] = act[y] ? log(1.0 / nact) : 0.0;
        if (!act[y]) nj[y] = mu[y] = 0.0;
    }
    __syncthreads();

    int it = 0, done = 0;
    for (; it < max_iter; ++it) {
        const double lntot = sh.lntot, ntot = exp(lntot), shift = lnP - lntot;
        double sn = 0.0, snm = 0.0;
        for (int y = tid; y < S; y += kEqThreads) {
            if (!act[y]) continue;
            const double n = exp(lnN[y]), m = g[y] + lnN[y] + shift;
            const double nm = n * m;
            nj[y] = n;
            mu[y] = nm;
            sn += n;
            snm += nm;
        }
        // the system starts from zero (pairs of elements no species shares stay zero)
        for (int t = tid; t < M * (M + 1); t += kEqThreads) sh.A[t / (M + 1)][t % (M + 1)] = 0.0;
        block_sum2(sh, sn, snm);
        // each entry's sublists, a lane each; element sums take nj mu along
        for (int q = wrp; q < ix.ngrp; q += kEqWarps) {
            double sv = 0.0, dv = 0.0;
            for (int r = ix.gp[q]; r < ix.gp[q + 1]; ++r) {
                const int y = ix.ent[32 * r + lane];
                if (y >= 0) {
                    const double a = ix.ec[32 * r + lane];
                    sv = fma(a, nj[y], sv);
                    dv = fma(a, mu[y], dv);
                }
            }
            const int to = ix.part[32 * q + lane];
            if (to >= 0) {
                part[to] = sv;
                part[ix.nsub + to] = dv;
            }
        }
        __syncthreads();
        for (int t = tid; t < ix.nent; t += kEqThreads) {
            const int code = ix.eij[t];
            double sv = 0.0, dv = 0.0;
            for (int q = ix.ep[t]; q < ix.ep[t + 1]; ++q) {
                sv += part[q];
                if (code < 0) dv += part[ix.nsub + q];
            }
            if (code >= 0) {
                const int i = code >> 5, j = code & 31;
                if (sh.eact[i] && sh.eact[j]) {
                    sh.A[i][j] = sv;
                    sh.A[j][i] = sv;
                }
            } else {
                const int i = -1 - code;
                if (sh.eact[i]) {
                    sh.A[i][E] = sv;
                    sh.A[E][i] = sv;
                    sh.A[i][M] = sh.bk[i] / sh.bsum - sv + dv;
                }
            }
        }
        if (tid == 0) {
            sh.A[E][E] = sn - ntot;
            sh.A[E][M] = ntot - sn + snm;
        }
        __syncthreads();
        if (tid < E && !sh.eact[tid]) sh.A[tid][tid] = 1.0;
        __syncthreads();
        if (wrp < kSolveWarps) warps_solve(sh, M);
        __syncthreads();
        if (sh.singular) break;
        const double dlntot = sh.sol[E];
        // step limit (the largest of non-negative values by their bit patterns) and convergence measure
        unsigned long long big = key_of(5.0 * fabs(dlntot)), rise = 0ull;
        double conv = 0.0;
        for (int y = tid; y < S; y += kEqThreads) {
            if (!act[y]) continue;
            double d = dlntot - (g[y] + lnN[y] + shift);
            for (int q = ix.sp[y]; q < ix.sp[y + 1]; ++q) d = fma(sh.sol[ix.se[q]], ix.sc[q], d);
            mu[y] = d;
            const double lx = lnN[y] - lntot;
            const unsigned long long kd = key_of(d) & 0x7fffffffffffffffull;
            // ln x is negative at these magnitudes: above ln 1e-8 means a smaller bit pattern
            if (!(lx < 0.0) || key_of(lx) < key_of(kLnMajor)) big = max(big, kd);
            else if (d - dlntot > 0.0)
                rise = max(rise, key_of((d - dlntot) * reciprocal64(-lx - kTraceCap)) & 0x7fffffffffffffffull);
            conv = fma(nj[y], __longlong_as_double((long long)kd), conv);
        }
        big = warp_max_key(big);
        rise = warp_max_key(rise);
        conv = warp_sum(conv);
        if (lane == 0) {
            sh.kred[0][wrp] = big;
            sh.kred[1][wrp] = rise;
            sh.red[0][wrp] = conv;
        }
        __syncthreads();
        conv = 0.0;
        for (int i = 0; i < kEqWarps; ++i) {   // same order in every thread: identical results everywhere
            big = max(big, sh.kred[0][i]);
            rise = max(rise, sh.kred[1][i]);
            conv += sh.red[0][i];
        }
        const double bigd = __longlong_as_double((long long)big), rised = __longlong_as_double((long long)rise);
        double lam = bigd > 2.0 ? 2.0 / bigd : 1.0;
        if (rised > 1.0) lam = fmin(lam, 1.0 / rised);
        for (int y = tid; y < S; y += kEqThreads)
            if (act[y]) lnN[y] = fma(lam, mu[y], lnN[y]);
        __syncthreads();
        if (tid == 0) sh.lntot = lntot + lam * dlntot;
        if (conv / sn < tol && fabs(dlntot) < tol) {
            ++it;
            done = 1;   // same decision in every thread (block-reduced values)
            break;
        }
        __syncthreads();
    }
    __syncthreads();
    if (tid == 0) {
        iters[k] = it;
        status[k] = sh.singular ? -1 : (done ? 0 : 1);
    }
    if (sh.singular) return;
    // mole fractions from the potentials of the last solve, normalised
    double amax = -INFINITY;
    for (int y = tid; y < S; y += kEqThreads) {
        if (!act[y]) continue;
        double v = -g[y] - lnP;
        for (int q = ix.sp[y]; q < ix.sp[y + 1]; ++q) v += sh.sol[ix.se[q]] * ix.sc[q];
        mu[y] = v;
        amax = fmax(amax, v);
    }
    for (int o = 16; o; o >>= 1) amax = fmax(amax, __shfl_xor_sync(0xffffffffu, amax, o));
    if (lane == 0) sh.red[0][wrp] = amax;
    __syncthreads();
    for (int i = 0; i < kEqWarps; ++i) amax = fmax(amax, sh.red[0][i]);
    __syncthreads();
    double z = 0.0, zero = 0.0;
    for (int y = tid; y < S; y += kEqThreads)
        if (act[y]) z += exp(mu[y] - amax);
    block_sum2(sh, z, zero);
    const double lz = log(z);
    const double ng = c.ngas[k];
    for (int y = tid; y < S; y += kEqThreads) {
        const double v = act[y] ? exp(mu[y] - amax - lz) : 0.0;
        if (x) x[(size_t)k * S + y] = v;
        if (nout) nout[(size_t)k * S + y] = v * ng;
    }
}

__global__ void k_fluxes(Col c, const double *n, double *q)
{
    const long long total = (long long)c.L * c.R;
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < total;
         i += (long long)gridDim.x * blockDim.x) {
        const int k = (int)(i / c.R), r = (int)(i % c.R);
        const double *nk = n + (size_t)k * c.S;
        double wf, wb;
        if (c.rtype[r] == XK_RX_PHOTO) {
            wf = c.kph[(size_t)k * c.Rph + c.prow[r]];
            wb = 0.0;
        } else {
            wf = c.kf[i];
            wb = c.kr[i];
        }
        for (int s = 0; s < 3; ++s) {
            const int a = c.reac[3 * r + s], p = c.prod[3 * r + s];
            if (a >= 0) wf *= nk[a];
            if (p >= 0) wb *= nk[p];
        }
        q[2 * i] = wf;
        q[2 * i + 1] = wb;
    }
}

// Edge weight of every reaction direction in every layer: 1/q for q > 0, +inf otherwise (no edge).
// Computed once per layer and shared by every source's search.
__global__ void k_path_weights(long long n, const double *q, double *wq)
{
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
        const double r = q[i];
        wq[i] = r > 0.0 ? 1.0 / r : INFINITY;
    }
}

// Distances are non-negative doubles (or +inf): their bit patterns order like the values, so the
// search compares them (key_of) on the integer pipes: FP64 compares are scarce on this GPU.

// Least weight of every group of parallel edges (source u, target v) in every layer.  Rounding is
// monotone, so du + (least weight) is the least of du + (weight) over the group: the search needs no
// other weight to know whether and to what v's distance falls.
__global__ void k_path_groups(PathGraph gr, int ng, int L, long long LR2, const double *wq, double *gmin)
{
    const long long n = (long long)L * ng, R2 = LR2 / L;
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
        const int k = (int)(i / ng), g = (int)(i - (long long)k * ng);
        const double *wk = wq + (size_t)k * R2;
        unsigned long long m = key_of(INFINITY);
        for (int t = gr.gs[g]; t < gr.gs[g + 1]; ++t) m = min(m, key_of(wk[gr.gcode[t]]));
        gmin[i] = __longlong_as_double((long long)m);
    }
}

// Per-warp shared memory of the pathway search: the distances' bit patterns [S], then the group of the
// edge into a species [S] ints, its predecessor and the finishing order [S] 16-bit words.  A finished
// species' distance has its sign bit set: the scan compares unsigned words, the relaxation signed ones,
// so that neither takes it up.
__host__ __device__ inline size_t path_warp_bytes(int S)
{
    return ((size_t)S * (8 + 4 + 2 + 2) + 15) / 16 * 16;
}

// One warp per search, the searches of a layer side by side (they read the same weights).  What a
// finished species costs is a chain of latencies: the scan for the least open distance, then the
// species' groups and their least weights (contiguous, one trip to L2), one FP64 addition.  The edge
// of a group that gave the distance is looked up once per species at the end, from the distance of
// its predecessor, which no longer changes: scanning the codes at every relaxation (three dependent
// trips) took 10,800 clocks per species, and the slowest steps by one lane in global memory a
// seventh of the whole.  Rates, weights and eight searches in each of 150 layers of 594 species take
// 1.25 ms so, 3.42 before.
__global__ void k_pathways(Col c, PathGraph gr, int ng, const double *wq, const double *gmin, int nsrc, const int *src,
                           int wpb, double *dist_out, int *pred_out, int *edge_out, int *lim_out, double *limw_out)
{
    extern __shared__ double path_dyn[];
    const int S = c.S, L = c.L, lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const long long prob = (long long)blockIdx.x * wpb + w;
    if (w >= wpb || prob >= (long long)nsrc * L) return;
    const int k = (int)(prob / nsrc), j = (int)(prob - (long long)k * nsrc);
    const int s0 = src[j];
    char *base = (char *)path_dyn + path_warp_bytes(S) * w;
    unsigned long long *dist = (unsigned long long *)base;
    int *pg = (int *)(dist + S);
    unsigned short *pred = (unsigned short *)(pg + S), *order = pred + S;
    const double *wk = wq + (size_t)k * c.R * 2, *gk = gmin + (size_t)k * ng;
    const unsigned long long kinf = key_of(INFINITY), kdone = 1ull << 63;
    for (int y = lane; y < S; y += 32) {
        dist[y] = y == s0 ? 0ull : kinf;
        pg[y] = -1;
    }
    __syncwarp();
    int nord = 0;
    for (;;) {
        // the unfinished species of least distance, the lower index on ties
        unsigned long long bd = kinf;
        int bi = S;
#pragma unroll 4
        for (int y = lane; y < S; y += 32) {
            const unsigned long long ky = dist[y];
            if (ky < bd) {
                bd = ky;
                bi = y;
            }
        }
        const unsigned hi = (unsigned)(bd >> 32), mh = __reduce_min_sync(0xffffffffu, hi);
        const unsigned lo = hi == mh ? (unsigned)bd : 0xffffffffu, ml = __reduce_min_sync(0xffffffffu, lo);
        if (mh >= (unsigned)(kinf >> 32)) break;
        const int u = (int)__reduce_min_sync(0xffffffffu, hi == mh && (unsigned)bd == ml ? (unsigned)bi : 0xffffffffu);
        const double du = __longlong_as_double((long long)((unsigned long long)mh << 32 | ml));
        if (lane == 0) {
            dist[u] |= kdone;
            order[nord] = (unsigned short)u;
        }
        ++nord;
        // relax: one lane per target species
        const int g1 = gr.gp[u + 1];
        for (int g = gr.gp[u] + lane; g < g1; g += 32) {
            const int v = gr.gv[g];
            const long long cand = (long long)key_of(du + gk[g]);
            if (cand < (long long)dist[v]) {
                dist[v] = (unsigned long long)cand;
                pred[v] = (unsigned short)u;
                pg[v] = g;
            }
        }
        __syncwarp();
    }
    // the first edge, codes increasing, that gives the least distance
    const size_t o = ((size_t)j * L + k) * S;
    for (int y = lane; y < S; y += 32) {
        int be = -1;
        const int g = pg[y];
        if (g >= 0) {
            const double du = __longlong_as_double((long long)(dist[pred[y]] & ~kdone));
            unsigned long long kb = kinf;
            for (int t = gr.gs[g]; t < gr.gs[g + 1]; ++t) {
                const int e = gr.gcode[t];
                const unsigned long long kc = key_of(du + wk[e]);
                if (kc < kb) {
                    kb = kc;
                    be = e;
                }
            }
        }
        if (dist_out) dist_out[o + y] = __longlong_as_double((long long)(dist[y] & ~kdone));
        if (pred_out) pred_out[o + y] = g >= 0 ? (int)pred[y] : -1;
        if (edge_out) edge_out[o + y] = be;
        pg[y] = be;
    }
    if (!lim_out) return;
    __syncwarp();
    // the edge's weight takes the distance's place
    for (int y = lane; y < S; y += 32) dist[y] = pg[y] >= 0 ? key_of(wk[pg[y]]) : 0ull;
    __syncwarp();
    // slowest step of each path, in the order the species were finished: a species' weight and edge
    // become those of its path's slowest step
    if (lane == 0)
        for (int i = 1; i < nord; ++i) {
            const int v = order[i], u = pred[v];
            if (u != s0 && !(dist[v] > dist[u])) {
                dist[v] = dist[u];
                pg[v] = pg[u];
            }
        }
    __syncwarp();
    for (int y = lane; y < S; y += 32) {
        lim_out[o + y] = pg[y];
        limw_out[o + y] = __longlong_as_double((long long)dist[y]);
    }
}

}  // namespace

cudaError_t launch_equilibrium(const Col &c, const EqIndex &ix, const double *b, double *x, double *nout,
                               int max_iter, double tol, int *iters, int *status, cudaStream_t st)
{
    if (c.E + 1 > kEqMaxE) return cudaErrorInvalidValue;
    const size_t species = (size_t)c.S * (3 * sizeof(double) + 1), smem = species + 2 * (size_t)ix.nsub * sizeof(double);
    if (species > 200 * 1024) return cudaErrorInvalidValue;   // with the parts (kEqMaxSub) and EqShared: 227 KB
    if (smem > 48 * 1024) {
        cudaError_t e = cudaFuncSetAttribute(k_equilibrium, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return e;
    }
    k_equilibrium<<<c.L, kEqThreads, smem, st>>>(c, ix, b, x, nout, max_iter, tol, iters, status);
    count_launches(1);
    return cudaGetLastError();
}

void launch_fluxes(const Col &c, const double *n, double *q, cudaStream_t st)
{
    const long long total = (long long)c.L * c.R;
    const int blocks = (int)std::min<long long>((total + 255) / 256, 152LL * 8);
    k_fluxes<<<std::max(blocks, 1), 256, 0, st>>>(c, n, q);
    count_launches(1);
}

cudaError_t launch_pathways(const Col &c, const PathGraph &g, int ngroups, const double *q, double *wbuf, double *gbuf,
                            int nsrc, const int *src, double *dist, int *pred_sp, int *pred_edge, int *lim_edge,
                            double *lim_w, cudaStream_t st)
{
    const long long nw = (long long)c.L * c.R * 2, ngl = (long long)c.L * ngroups;
    if (nw > 0) {
        k_path_weights<<<(int)std::min<long long>((nw + 255) / 256, 152LL * 8), 256, 0, st>>>(nw, q, wbuf);
        count_launches(1);
    }
    if (ngl > 0) {
        k_path_groups<<<(int)std::min<long long>((ngl + 255) / 256, 152LL * 16), 256, 0, st>>>(g, ngroups, c.L, nw, wbuf, gbuf);
        count_launches(1);
    }
    const size_t per = path_warp_bytes(c.S), cap = 200 * 1024;
    if (per > cap) return cudaErrorInvalidValue;
    // searches of one layer to a CTA, as few as leave no SM without one
    const long long probs = (long long)nsrc * c.L;
    const int wpb = (int)std::max<long long>(1, std::min<long long>(std::min<long long>(8, cap / per), (probs + 151) / 152));
    const size_t smem = per * wpb;
    if (smem > 48 * 1024) {
        cudaError_t e = cudaFuncSetAttribute(k_pathways, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return e;
    }
    const int blocks = (int)((probs + wpb - 1) / wpb);
    k_pathways<<<blocks, 32 * wpb, smem, st>>>(c, g, ngroups, wbuf, gbuf, nsrc, src, wpb, dist, pred_sp, pred_edge, lim_edge,
                                              lim_w);
    count_launches(1);
    return cudaGetLastError();
}

}  // namespace xk

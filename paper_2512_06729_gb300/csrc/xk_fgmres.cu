// The reduction's solve and the FGMRES around it, each as one persistent cooperative launch.
//
// A preconditioner application walks the levels of the block cyclic reduction forward and back: a
// chain of about 3 log2(L) dependent stages of matrix-vector products that together read every
// inverse and coupling block once (the level-0 inverses twice).  It is bound by that read (771 MB
// at 594 species x 150 layers, 113 us at the measured copy rate) and, in small columns, by the
// barriers between the stages.  An iteration adds the matrix-free Jacobian product and two
// Gram-Schmidt passes, a few microseconds each when nothing is launched between them.  So the whole
// solve is one launch of one CTA per SM (a share of them in a batch): every scalar of the iteration
// (rotations, residual, when to stop) is computed by each CTA for itself from the same sums, in the
// same order, and a solve that is not needed costs one launch that returns at once, not one per
// kernel of every iteration slot.
#include <math.h>

#include <algorithm>

#include "xk_bcr.cuh"
#include "xk_gmres.cuh"
#include "xk_layer.cuh"

namespace xk {

namespace {

constexpr int kThreads = 512;
constexpr int kWarps = kThreads / 32;

// The right-hand side as the reduction reads it: (float)(b * mult * bscale).
struct Rhs {
    const double *b, *bscale;
    double mult;
};

template <typename T>
struct ApplyArgs {
    const BcrStage *stages;
    const BcrMvT<T> *mv;
    int nstages, S, rows, ld;
};
// Four floats or two doubles of a row at a time.
template <typename T>
struct Wide;
template <>
struct Wide<float> {
    using type = float4;
    static __device__ __forceinline__ float dot(float acc, float4 a, float4 x)
    {
        return acc + (a.x * x.x + a.y * x.y + a.z * x.z + a.w * x.w);
    }
};
template <>
struct Wide<double> {
    using type = double2;
    static __device__ __forceinline__ double dot(double acc, double2 a, double2 x) { return fma(a.y, x.y, fma(a.x, x.x, acc)); }
};

// Entry k of a task's vector: the right-hand side of a layer or a work vector, less diagonal
// coupling terms (level 0) on the first S entries.
template <typename T>
__device__ __forceinline__ T rhs_term(const Rhs &r, int layer, const T *v, int k, int S, const T *d0, const T *w0,
                                      const T *d1, const T *w1)
{
    T val;
    if (layer >= 0) {
        val = T(0);
        if (k < S) {
            const long long q = (long long)layer * S + k;
            const double b = r.b[q] * r.mult;
            val = (T)(r.bscale ? b * r.bscale[q] : b);
        }
    } else {
        val = v ? v[k] : T(0);
    }
    if (k < S) {
        if (d0) val -= d0[k] * w0[k];
        if (d1) val -= d1[k] * w1[k];
    }
    return val;
}

// Rows [row, row + RPW) of M v, one warp: all of a lane's loads of RPW rows in flight together.
template <int RPW, typename T>
__device__ __forceinline__ void mv_rows(const BcrMvT<T> &t, const T *v, int row, int nrow, T (&out)[RPW])
{
    using V = typename Wide<T>::type;
    const int lane = threadIdx.x & 31;
    const V *m[RPW];
    T acc[RPW];
#pragma unroll
    for (int i = 0; i < RPW; ++i) {
        m[i] = (const V *)(t.M + (long long)(row + min(i, nrow - 1)) * t.ld);
        acc[i] = T(0);
    }
    const int n4 = t.K * (int)sizeof(T) / 16;
#pragma unroll 4
    for (int q = lane; q < n4; q += 32) {
        const V x = ((const V *)v)[q];
#pragma unroll
        for (int i = 0; i < RPW; ++i) acc[i] = Wide<T>::dot(acc[i], __ldg(m[i] + q), x);
    }
#pragma unroll
    for (int i = 0; i < RPW; ++i) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) acc[i] += __shfl_xor_sync(0xffffffffu, acc[i], o);
        out[i] = acc[i];
    }
}

// One stage: chunks of kWarps * RPW rows of every task's block, contiguous chunks to a CTA so that
// the task's vector in shared memory is filled once for several of them.
template <int RPW, typename T>
__device__ __forceinline__ void mv_stage(const ApplyArgs<T> &a, const BcrStage &st, const Rhs &rhs, double *x,
                                         const double *xscale, T *v)
{
    const int S = a.S, Sp = a.ld, warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int rows = kWarps * RPW, chunks = (a.rows + rows - 1) / rows, items = st.count * chunks;
    const int G = gridDim.x, per = items / G, rest = items - per * G, b = blockIdx.x;
    const int i0 = b * per + min(b, rest), i1 = i0 + per + (b < rest ? 1 : 0);
    int have = -1;
    for (int item = i0; item < i1; ++item) {
        const int ti = item / chunks, chunk = item - ti * chunks;
        const BcrMvT<T> &t = a.mv[st.off + ti];
        if (ti != have) {
            __syncthreads();
            for (int k = threadIdx.x; k < t.K; k += kThreads)
                v[k] = k < Sp ? rhs_term<T>(rhs, t.in, t.v0, k, S, t.d0, t.w0, t.d1, t.w1) : t.v1[k - Sp];
            __syncthreads();
            have = ti;
        }
        const int row = chunk * rows + warp * RPW, nrow = min(RPW, a.rows - row);
        if (nrow <= 0) continue;
        T out[RPW];
        mv_rows<RPW, T>(t, v, row, nrow, out);
        T mine = out[0];
#pragma unroll
        for (int i = 1; i < RPW; ++i)
            if (lane == i) mine = out[i];
        if (lane < nrow) {
            const int r = row + lane;
            T base = T(0);
            if (t.bin >= 0 || t.base) base = rhs_term<T>(rhs, t.bin, t.base, r, S, t.e0, t.f0, t.e1, t.f1);
            const T y = base + t.sign * mine;
            t.y[r] = y;
            if (t.out >= 0 && r < S) {
                const long long q = (long long)t.out * S + r;
                x[q] = xscale ? (double)y * xscale[q] : (double)y;
            }
        }
    }
}

// x = M^-1 rhs: every stage, a grid barrier after each but the last.  false: a wait gave up.
template <typename T>
__device__ __forceinline__ bool bcr_apply(const ApplyArgs<T> &a, const Rhs &rhs, double *x, const double *xscale, T *v,
                                          GridSync &gs)
{
    for (int si = 0; si < a.nstages; ++si) {
        const BcrStage st = a.stages[si];
        // four rows to a warp where the stage has that much work for every CTA, else one
        const int total = st.count * a.rows;
        if (total >= 4 * kWarps * (int)gridDim.x) mv_stage<4, T>(a, st, rhs, x, xscale, v);
        else mv_stage<1, T>(a, st, rhs, x, xscale, v);
        if (si + 1 < a.nstages && !gs.sync()) return false;
    }
    return true;
}

__device__ __forceinline__ bool stopped(const int *skip, const Ctl *ctl)
{
    return (ctl && (ctl->finished || ctl->err_timeout)) || (skip && *skip);
}

template <typename T>
__global__ void __launch_bounds__(kThreads, 1)
k_bcr_solve(ApplyArgs<T> a, const double *b, const double *bscale, double *x, const double *xscale, unsigned *words,
            const int *skip, Ctl *ctl)
{
    if (stopped(skip, ctl)) return;
    extern __shared__ __align__(16) unsigned char dyn[];
    GridSync gs(words, ctl);
    bcr_apply<T>(a, Rhs{b, bscale, 1.0}, x, xscale, (T *)dyn, gs);
    gs.leave();
}

// ---------------------------------------------------------------------------
// FGMRES(m) in FP64 on the scaled, row-equilibrated operator, preconditioned by the reduction.  The
// same iteration as enqueue_fgmres (cycles of m within max_iter, one short spare cycle, convergence
// decided on the true residual at each cycle's start).  A CTA owns whole layers of every vector.
// ---------------------------------------------------------------------------
template <typename T>
struct FgArgs {
    Col c;
    ApplyArgs<T> ap;
    const double *b, *rowd;
    double *x, *V, *Z, *w, *partials;
    unsigned *words;
    GmState *gm;
    Ctl *ctl;
    const int *skip;
    double tol;
    int m, max_iter, rates_in_smem, role;
};

struct FgShared {
    double H[(kMaxBasis + 1) * kMaxBasis];
    double g[kMaxBasis + 1], cs[kMaxBasis], sn[kMaxBasis], h1[kMaxBasis + 1], h2[kMaxBasis + 1], y[kMaxBasis];
    double beta, hn, resid;
    int stop, failed;
};

__device__ __forceinline__ double warp_sum(double v)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

// h[i] = <V_i, w>, i < nv, and with nv < 0 h[0] = <w, w>: a warp per basis vector and layer of this
// CTA, then (after the barrier) every CTA adds the layers' parts in the same order, so that the sums
// do not depend on how many CTAs the launch has.  The parts alternate between two buffers: a CTA past
// the barrier may write its next parts while another still adds the last ones.
template <typename T>
__device__ __forceinline__ bool fg_dots(const FgArgs<T> &a, int nv, const double *w, double *h, GridSync &gs, int &buf)
{
    const int S = a.c.S, L = a.c.L, warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    double *parts = a.partials + (long long)(buf ^= 1) * L * (kMaxBasis + 1);
    const long long N = (long long)L * S;
    const int n = nv < 0 ? 1 : nv;
    __syncthreads();
    for (int k = blockIdx.x; k < L; k += gridDim.x) {
        const long long o = (long long)k * S;
        for (int i = warp; i < n; i += kWarps) {
            const double *vi = nv < 0 ? w : a.V + (long long)i * N;
            double acc = 0.0;
#pragma unroll 4
            for (int e = lane; e < S; e += 32) acc += vi[o + e] * w[o + e];
            acc = warp_sum(acc);
            if (lane == 0) parts[(long long)k * (kMaxBasis + 1) + i] = acc;
        }
    }
    if (!gs.sync()) return false;
    for (int i = warp; i < n; i += kWarps) {
        double acc = 0.0;
        for (int k = lane; k < L; k += 32) acc += parts[(long long)k * (kMaxBasis + 1) + i];
        acc = warp_sum(acc);
        if (lane == 0) h[i] = acc;
    }
    __syncthreads();
    return true;
}

template <typename T>
__global__ void __launch_bounds__(kThreads, 1) k_fgmres(FgArgs<T> a)
{
    if (stopped(a.skip, a.ctl)) return;
    extern __shared__ __align__(16) unsigned char dyn[];
    __shared__ FgShared sh;
    const Col &c = a.c;
    const int S = c.S, L = c.L, G = gridDim.x, tid = threadIdx.x;
    const long long N = (long long)L * S;
    GridSync gs(a.words, a.ctl);
    T *v = (T *)dyn;
    double *jv = (double *)dyn;

    // f(e) for every element this CTA owns, the same thread for the same element each time
    auto own = [&](auto f) {
        for (int k = blockIdx.x; k < L; k += G)
            for (int e = tid; e < S; e += kThreads) f((long long)k * S + e);
    };
    auto matvec = [&](const double *x) {
        for (int k = blockIdx.x; k < L; k += G) {
            __syncthreads();
            jv_layer_body(c, a.ctl, x, a.w, a.rowd, k, jv, a.rates_in_smem != 0);
        }
        __syncthreads();
    };
    own([&](long long e) { a.x[e] = 0.0; });
    const int m = a.m, full = (a.max_iter + m - 1) / m, spare = min(m, 8), cycles = full + 1;
    int iters = 0, done = 0, failed = 0, buf = 0;
    double bnorm = 0.0, resid = 0.0;
    const bool lead = blockIdx.x == 0 && tid == 0;
    bool ok = true;
    for (int cyc = 0; cyc < cycles && !done; ++cyc) {
        // r = b - A x, its norm; r in w (cycle 0: x = 0)
        if (cyc > 0) {
            // x of the neighbouring layers is needed
            if (!(ok = gs.sync())) break;
            matvec(a.x);
        }
        own([&](long long e) { a.w[e] = cyc == 0 ? a.b[e] : a.b[e] - a.w[e]; });
        if (!(ok = fg_dots(a, -1, a.w, sh.h1, gs, buf))) break;
        const double beta = sqrt(sh.h1[0]);
        if (cyc == 0) bnorm = beta;
        resid = bnorm > 0.0 ? beta / bnorm : 0.0;
        if (!(beta > 0.0) || resid <= a.tol || !isfinite(beta) || iters >= a.max_iter) {
            done = 1;
            if (!isfinite(beta)) failed = 1;
            break;
        }
        __syncthreads();
        if (tid == 0) {
            for (int i = 0; i <= kMaxBasis; ++i) sh.g[i] = 0.0;
            sh.g[0] = beta;
        }
        const int mc = cyc < full ? min(m, a.max_iter - cyc * m) : spare;
        double scale = 1.0 / beta;             // V_j = w * scale
        int j = 0;
        bool end = false;
        while (!end) {
            // every CTA's part of w is written (the barrier of the norm above); V_j is this CTA's copy
            double *vj = a.V + (long long)j * N, *zj = a.Z + (long long)j * N;
            own([&](long long e) { vj[e] = a.w[e] * scale; });
            if (!(ok = bcr_apply<T>(a.ap, Rhs{a.w, a.rowd, scale}, zj, nullptr, v, gs))) break;
            if (!(ok = gs.sync())) break;
            matvec(zj);
            if (!(ok = fg_dots(a, j + 1, a.w, sh.h1, gs, buf))) break;
            own([&](long long e) {
                double acc = a.w[e];
                for (int i = 0; i <= j; ++i) acc -= sh.h1[i] * a.V[(long long)i * N + e];
                a.w[e] = acc;
            });
            if (!(ok = fg_dots(a, j + 1, a.w, sh.h2, gs, buf))) break;
            own([&](long long e) {
                double acc = a.w[e];
                for (int i = 0; i <= j; ++i) acc -= sh.h2[i] * a.V[(long long)i * N + e];
                a.w[e] = acc;
            });
            // ||w||^2 into y[0]
            if (!(ok = fg_dots(a, -1, a.w, sh.y, gs, buf))) break;
            if (tid == 0) {
                double *H = sh.H + j * (kMaxBasis + 1);
                for (int i = 0; i <= j; ++i) H[i] = sh.h1[i] + sh.h2[i];
                const double hn = sqrt(sh.y[0]);
                H[j + 1] = hn;
                sh.hn = hn;
                for (int i = 0; i < j; ++i) {
                    const double p = sh.cs[i] * H[i] + sh.sn[i] * H[i + 1];
                    const double q = -sh.sn[i] * H[i] + sh.cs[i] * H[i + 1];
                    H[i] = p;
                    H[i + 1] = q;
                }
                const double p = H[j], q = H[j + 1], r = hypot(p, q);
                const double cc = r > 0.0 ? p / r : 1.0, ss = r > 0.0 ? q / r : 0.0;
                sh.cs[j] = cc;
                sh.sn[j] = ss;
                H[j] = r;
                H[j + 1] = 0.0;
                sh.g[j + 1] = -ss * sh.g[j];
                sh.g[j] = cc * sh.g[j];
                sh.resid = fabs(sh.g[j + 1]) / bnorm;
                const int bad = !isfinite(sh.resid);
                sh.failed = bad;
                sh.stop = bad || sh.resid <= a.tol || iters + 1 >= a.max_iter || j + 1 >= mc || !(hn > 0.0);
            }
            __syncthreads();
            resid = sh.resid;
            end = sh.stop != 0;
            scale = 1.0 / sh.hn;
            if (sh.failed) {
                failed = 1;
                done = 1;
            }
            ++iters;
            ++j;
        }
        if (!ok) break;
        // x += Z y, H y = g
        if (tid == 0)
            for (int i = j - 1; i >= 0; --i) {
                double s = sh.g[i];
                for (int q = i + 1; q < j; ++q) s -= sh.H[q * (kMaxBasis + 1) + i] * sh.y[q];
                sh.y[i] = s / sh.H[i * (kMaxBasis + 1) + i];
            }
        __syncthreads();
        own([&](long long e) {
            double acc = a.x[e];
            for (int i = 0; i < j; ++i) acc += sh.y[i] * a.Z[(long long)i * N + e];
            a.x[e] = acc;
        });
    }
    if (ok && !done) {
        // the last cycle ended on the recurrence estimate: the residual it left
        if ((ok = gs.sync())) {
            matvec(a.x);
            own([&](long long e) { a.w[e] = a.b[e] - a.w[e]; });
            if ((ok = fg_dots(a, -1, a.w, sh.h1, gs, buf))) resid = bnorm > 0.0 ? sqrt(sh.h1[0]) / bnorm : 0.0;
        }
    }
    if (lead) {
        GmState *gm = a.gm;
        gm->iters = iters;
        gm->resid = resid;
        gm->tol = a.tol;
        gm->bnorm = bnorm;
        gm->done = 1;
        gm->failed = failed;
        Ctl *ctl = a.ctl;
        ctl->solver_iters = iters;
        ctl->solver_resid = resid;
        ctl->total_iters += iters;
        // a solve around the FP32 factors that did not reach the tolerance hands the step to the FP64
        // factorization, and so does every later step at this dt or above
        if (a.role == 0 && (failed || !(resid <= a.tol))) {
            ctl->skip64 = 0;
            ctl->used_fp64 = 1;
            if (ctl->dt < ctl->dt_fp64) ctl->dt_fp64 = ctl->dt;
        }
    }
    gs.leave();
}

// One CTA per SM, or the column's share of them in a batch.
int solve_ctas(int share) { return share > 0 ? std::min(share, device_sms()) : device_sms(); }

template <typename T>
ApplyArgs<T> apply_args(const BcrSolveT<T> &p) { return {p.stages, p.mv, p.nstages, p.S, p.rows, p.ld}; }

}  // namespace

template <typename T>
cudaError_t bcr_solve(const BcrSolveT<T> &p, const double *b, double *x, const double *bscale, const double *xscale,
                      const int *skip, Ctl *ctl, cudaStream_t st)
{
    cudaError_t e = allow_smem(k_bcr_solve<T>, kJvSmemMax);
    if (e != cudaSuccess) return e;
    ApplyArgs<T> a = apply_args(p);
    unsigned *words = p.bar;
    void *args[] = {(void *)&a, (void *)&b, (void *)&bscale, (void *)&x, (void *)&xscale, (void *)&words, (void *)&skip,
                    (void *)&ctl};
    count_launches(1);
    return cudaLaunchCooperativeKernel((const void *)k_bcr_solve<T>, dim3(solve_ctas(p.ctas)), dim3(kThreads), args,
                                       (size_t)2 * p.ld * sizeof(T), st);
}

template <typename T>
cudaError_t bcr_fgmres(const BcrSolveT<T> &p, const Col &c, const GmArgs &g, const double *rowd, cudaStream_t st)
{
    cudaError_t e = allow_smem(k_fgmres<T>, kJvSmemMax);
    if (e != cudaSuccess) return e;
    FgArgs<T> a;
    a.c = c;
    a.ap = apply_args(p);
    a.b = g.b;
    a.rowd = rowd;
    a.x = g.x; a.V = g.V; a.Z = g.Z; a.w = g.w; a.partials = g.partials;
    a.words = p.bar;
    a.gm = g.gm;
    a.ctl = g.ctl;
    a.skip = g.skip_solve;
    a.tol = g.tol;
    a.m = std::min(g.m, kMaxBasis);
    a.max_iter = g.max_iter;
    a.role = g.role;
    a.rates_in_smem = jv_rates_in_smem(c) ? 1 : 0;
    const size_t smem = std::max((size_t)2 * p.ld * sizeof(T), jv_smem_doubles(c, a.rates_in_smem != 0) * sizeof(double));
    if (smem > kJvSmemMax) return cudaErrorInvalidValue;
    void *args[] = {(void *)&a};
    count_launches(1);
    return cudaLaunchCooperativeKernel((const void *)k_fgmres<T>, dim3(solve_ctas(p.ctas)), dim3(kThreads), args, smem, st);
}

template cudaError_t bcr_solve<float>(const BcrSolveT<float> &, const double *, double *, const double *, const double *,
                                      const int *, Ctl *, cudaStream_t);
template cudaError_t bcr_solve<double>(const BcrSolveT<double> &, const double *, double *, const double *, const double *,
                                       const int *, Ctl *, cudaStream_t);
template cudaError_t bcr_fgmres<float>(const BcrSolveT<float> &, const Col &, const GmArgs &, const double *, cudaStream_t);
template cudaError_t bcr_fgmres<double>(const BcrSolveT<double> &, const Col &, const GmArgs &, const double *, cudaStream_t);

}  // namespace xk

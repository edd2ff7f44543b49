// Lagrangian parcel scheme (Sec. 2, Fig. 1 and Fig. 2): one global iteration carries an air
// parcel from the bottom layer to the top and back (layers 0 .. L-1, then L-2 .. 0).  In layer k
// the parcel's densities x evolve for the eddy mixing time tau_k = dz_k^2 / K_zz,k under that
// layer's chemistry (Sec. 2.3) and molecular diffusion written as a pseudo-reaction pair with the
// stored densities of layers k -+ 1 (Sec. 2.1, after Eq. 4: the molecular part of Eq. 2's flux);
// eddy diffusion is the parcel's motion and has no term.  Within a visit: linearly implicit Euler
// steps (I/h - dF/dx) delta = F under the step controller of the Eulerian path, each solved by
// Gaussian elimination with partial pivoting plus two sweeps of FP64 iterative refinement.  The
// parcel keeps its mixing ratios from layer to layer, and each visit leaves its densities as the
// layer's.
//
// The sweep is sequential in the layers, so one CTA runs a whole iteration: every reduction,
// pivot search and elimination step stays inside the block (no grid-wide wait).  Systems whose two
// S x S matrices (the system and its factors) fit in shared memory (S up to 112, small_layout against
// kSmemLimit) have a kernel of their own; larger ones keep them in global memory, where they stay in L2.
#include <cfloat>

#include "xk_internal.cuh"
#include "xk_layer.cuh"

namespace xk {

namespace {

constexpr int kMaxWarps = 32;
constexpr int kRefineSweeps = 2;          // FP64 iterative-refinement sweeps of every implicit step
constexpr size_t kSmemLimit = 208 * 1024; // dynamic shared memory the kernel may ask for

struct Shared {
    double red[kMaxWarps];
    int ired[kMaxWarps];
    double h, t, hs;
    int last, done;
    int piv[2];
};

__device__ __forceinline__ int nwarps() { return blockDim.x >> 5; }

// max over the block; every thread gets the result
__device__ double block_max(double v, Shared &sh)
{
    for (int o = 16; o > 0; o >>= 1) v = fmax(v, __shfl_xor_sync(0xffffffffu, v, o));
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    __syncthreads();
    if (lane == 0) sh.red[warp] = v;
    __syncthreads();
    v = lane < nwarps() ? sh.red[lane] : -DBL_MAX;
    for (int o = 16; o > 0; o >>= 1) v = fmax(v, __shfl_xor_sync(0xffffffffu, v, o));
    return v;
}

__device__ int block_or(int v, Shared &sh)
{
    v = __any_sync(0xffffffffu, v) ? 1 : 0;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    __syncthreads();
    if (lane == 0) sh.ired[warp] = v;
    __syncthreads();
    v = lane < nwarps() ? sh.ired[lane] : 0;
    return __any_sync(0xffffffffu, v) ? 1 : 0;
}

// Row of the largest |A[i][c]|, i >= c (the first on ties, as a sequential scan picks it), or -1.
__device__ int pivot_row(const double *A, int S, int c, Shared &sh)
{
    double best = -1.0;
    int bi = S;
    for (int i = c + threadIdx.x; i < S; i += blockDim.x) {
        const double v = fabs(A[(long long)i * S + c]);
        if (v > best) { best = v; bi = i; }
    }
    for (int o = 16; o > 0; o >>= 1) {
        const double ov = __shfl_xor_sync(0xffffffffu, best, o);
        const int oi = __shfl_xor_sync(0xffffffffu, bi, o);
        if (ov > best || (ov == best && oi < bi)) { best = ov; bi = oi; }
    }
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    __syncthreads();
    if (lane == 0) { sh.red[warp] = best; sh.ired[warp] = bi; }
    __syncthreads();
    best = lane < nwarps() ? sh.red[lane] : -1.0;
    bi = lane < nwarps() ? sh.ired[lane] : S;
    for (int o = 16; o > 0; o >>= 1) {
        const double ov = __shfl_xor_sync(0xffffffffu, best, o);
        const int oi = __shfl_xor_sync(0xffffffffu, bi, o);
        if (ov > best || (ov == best && oi < bi)) { best = ov; bi = oi; }
    }
    return best > 0.0 ? bi : -1;
}

// A <- its LU factors with partial pivoting (whole rows swapped; row c of the factors came from
// row piv[c] of the rows as they stood at step c).  0, or -1 on a zero pivot column.
__device__ int lu_factor(double *A, int *piv, int S, Shared &sh)
{
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, nw = nwarps();
    for (int c = 0; c < S; ++c) {
        const int p = pivot_row(A, S, c, sh);
        if (p < 0) return -1;
        if (threadIdx.x == 0) piv[c] = p;
        if (p != c)
            for (int j = threadIdx.x; j < S; j += blockDim.x) {
                const double t = A[(long long)c * S + j];
                A[(long long)c * S + j] = A[(long long)p * S + j];
                A[(long long)p * S + j] = t;
            }
        __syncthreads();
        const double inv = 1.0 / A[(long long)c * S + c];
        // a warp per row below the pivot: its multiplier, then the row update along the lanes
        for (int i = c + 1 + warp; i < S; i += nw) {
            double *Ai = A + (long long)i * S;
            const double l = Ai[c] * inv;
            __syncwarp();
            if (lane == 0) Ai[c] = l;
            for (int j = c + 1 + lane; j < S; j += 32) Ai[j] -= l * A[(long long)c * S + j];
        }
        __syncthreads();
    }
    return 0;
}

// x <- (LU)^-1 P x with the factors of lu_factor.
__device__ void lu_solve(const double *A, const int *piv, double *x, int S)
{
    if (threadIdx.x == 0)
        for (int c = 0; c < S; ++c) {
            const int p = piv[c];
            if (p != c) { const double t = x[c]; x[c] = x[p]; x[p] = t; }
        }
    __syncthreads();
    for (int c = 0; c < S; ++c) {            // unit lower triangle, column by column
        const double xc = x[c];
        for (int i = c + 1 + threadIdx.x; i < S; i += blockDim.x) x[i] -= A[(long long)i * S + c] * xc;
        __syncthreads();
    }
    for (int c = S - 1; c >= 0; --c) {       // upper triangle
        const double xc = x[c] * (1.0 / A[(long long)c * S + c]);
        __syncthreads();
        if (threadIdx.x == 0) x[c] = xc;
        for (int i = threadIdx.x; i < c; i += blockDim.x) x[i] -= A[(long long)i * S + c] * xc;
        __syncthreads();
    }
}

// d <- A0^-1 F: LU with partial pivoting of A (a copy of A0), then kRefineSweeps sweeps of FP64
// iterative refinement r = F - A0 d, d += (LU)^-1 P r.  0, or -1 on a zero pivot column.
__device__ int dense_solve(const double *A0, double *A, int *piv, const double *F, double *d, double *r, int S,
                           Shared &sh)
{
    for (long long e = threadIdx.x; e < (long long)S * S; e += blockDim.x) A[e] = A0[e];
    for (int y = threadIdx.x; y < S; y += blockDim.x) d[y] = F[y];
    __syncthreads();
    if (lu_factor(A, piv, S, sh) != 0) return -1;
    lu_solve(A, piv, d, S);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, nw = nwarps();
    for (int sweep = 0; sweep < kRefineSweeps; ++sweep) {
        for (int i = warp; i < S; i += nw) {
            const double *Ai = A0 + (long long)i * S;
            double acc = 0.0;
            for (int j = lane; j < S; j += 32) acc += Ai[j] * d[j];
            for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
            if (lane == 0) r[i] = F[i] - acc;
        }
        __syncthreads();
        lu_solve(A, piv, r, S);
        for (int y = threadIdx.x; y < S; y += blockDim.x) d[y] += r[y];
        __syncthreads();
    }
    return 0;
}

// The step size and what the controller says of a step with largest relative change mr (thread 0).
__device__ void step_size(Shared &sh, const Policy &pol, double tau)
{
    const double rest = tau - sh.t;
    double hs = sh.h < rest ? sh.h : rest;
    if (hs > pol.dt_max) hs = pol.dt_max;
    sh.hs = hs;
    sh.last = hs >= rest;
}
__device__ void step_control(Shared &sh, const Policy &pol, double tau, double hs, double mr, bool ok, int visit_steps,
                             int max_visit_steps)
{
    if (ok) {
        sh.t = sh.last ? tau : sh.t + hs;
        double fac = mr > 0.0 ? pol.rel_target / mr : pol.grow_max;
        if (fac > pol.grow_max) fac = pol.grow_max;
        if (fac < pol.shrink_min) fac = pol.shrink_min;
        double next = hs * fac;
        if (hs < sh.h && fac >= 1.0 && next < sh.h) next = sh.h;   // cut short by the visit's end
        sh.h = next;
        sh.done = 0;
    } else {
        sh.h = 0.5 * hs;
        sh.done = sh.h < pol.dt_min ? XK_ENEG : 0;
    }
    if (visit_steps > max_visit_steps && !sh.done) sh.done = XK_ENOCONV;
}

__global__ void __launch_bounds__(1024, 1) k_parcel_iteration(Col c, ParcelArgs a)
{
    __shared__ Shared sh;
    extern __shared__ double dyn[];
    const int S = c.S, L = c.L, R = c.R;
    const int tid = threadIdx.x, nt = blockDim.x;
    const int warp = tid >> 5, lane = tid & 31, nw = nwarps();
    const Policy &pol = a.pol;
    ParcelState *st = a.st;
    double *x = dyn, *F = x + S, *d = F + S, *r = d + S;
    int *piv = (int *)(r + S);
    double *A0 = a.A, *A = a.A + (long long)S * S;
    for (long long i = tid; i < (long long)L * S; i += nt) a.Nold[i] = a.N[i];
    for (int y = tid; y < S; y += nt) a.vmr[y] = a.N[y] / c.ngas[0];
    if (tid == 0) sh.h = st->h;
    long long steps = 0, rejected = 0;
    __syncthreads();
    for (int v = 0; v < 2 * L - 1; ++v) {
        const int k = v < L ? v : 2 * L - 2 - v;
        const double nk = c.ngas[k], dzk = c.dz[k];
        const double tau = dzk * dzk / c.Kzz[k];
        for (int y = tid; y < S; y += nt) x[y] = a.vmr[y] * nk;
        if (tid == 0) sh.t = 0.0;
        __syncthreads();
        int visit_steps = 0;
        while (sh.t < tau) {
            if (tid == 0) step_size(sh, pol, tau);
            __syncthreads();
            const double hs = sh.hs;
            // reaction terms at the parcel's densities (Sec. 2.3)
            for (int rr = tid; rr < R; rr += nt) reaction_terms_at(c, k, rr, x, a.w + rr, a.dd + (long long)rr * 6);
            __syncthreads();
            // right-hand side: chemistry plus the molecular-diffusion pair
            for (int y = tid; y < S; y += nt) {
                double f = 0.0;
                for (int e = c.yp[y]; e < c.yp[y + 1]; ++e) {
                    const int code = c.yent[e];
                    if ((code & 15) - 8 < 0) f -= a.w[code >> 4];
                    else f += a.w[code >> 4];
                }
                double loss = 0.0, gain = 0.0;
                if (k + 1 < L) {
                    loss += a.um[(long long)k * S + y];
                    gain += a.vm[(long long)k * S + y] * a.N[(long long)(k + 1) * S + y];
                }
                if (k > 0) {
                    loss += a.vm[(long long)(k - 1) * S + y];
                    gain += a.um[(long long)(k - 1) * S + y] * a.N[(long long)(k - 1) * S + y];
                }
                F[y] = f + (gain - loss * x[y]) / dzk;
            }
            // matrix I/h - dF/dx: one warp per row, entries of the pattern summed in a fixed order
            for (int i = warp; i < S; i += nw) {
                double *Ar = A0 + (long long)i * S;
                for (int j = lane; j < S; j += 32) Ar[j] = 0.0;
                __syncwarp();
                for (int q = c.jp[i] + lane; q < c.jp[i + 1]; q += 32) Ar[c.jcol[q]] = jac_entry(c, q, a.dd);
                __syncwarp();
                if (lane == 0) {
                    double loss = 0.0;
                    if (k + 1 < L) loss += a.um[(long long)k * S + i];
                    if (k > 0) loss += a.vm[(long long)(k - 1) * S + i];
                    Ar[i] += 1.0 / hs + loss / dzk;
                }
            }
            __syncthreads();
            if (dense_solve(A0, A, piv, F, d, r, S, sh) != 0) {
                if (tid == 0) { st->status = XK_ESINGULAR; st->visit = v; }
                return;
            }
            // the Eulerian step controller: reject on a negative or a too large relative change
            double mr = 0.0;
            int bad = 0;
            for (int y = tid; y < S; y += nt) {
                const double xv = x[y], dv = d[y], nn = xv + dv;
                if (!isfinite(nn) || nn < -pol.neg_tol * nk) bad = 1;
                if (xv > pol.f_floor * nk) mr = fmax(mr, fabs(dv) / xv);
            }
            bad = block_or(bad, sh);
            mr = block_max(mr, sh);
            const int ok = !bad && !(mr > pol.rel_reject);
            if (ok)
                for (int y = tid; y < S; y += nt) {
                    const double nn = x[y] + d[y];
                    x[y] = nn < 0.0 ? 0.0 : nn;
                }
            __syncthreads();
            ++visit_steps;
            if (tid == 0) step_control(sh, pol, tau, hs, mr, ok, visit_steps, a.max_visit_steps);
            if (ok) ++steps;
            else ++rejected;
            __syncthreads();
            if (sh.done) {
                if (tid == 0) { st->status = sh.done; st->visit = v; st->steps += steps; st->rejected += rejected; }
                return;
            }
        }
        for (int y = tid; y < S; y += nt) {
            a.N[(long long)k * S + y] = x[y];
            a.vmr[y] = x[y] / nk;
        }
        __syncthreads();
    }
    double ch = 0.0;
    for (long long i = tid; i < (long long)L * S; i += nt) {
        const int k = (int)(i / S);
        const double nv = a.N[i];
        if (nv > pol.f_floor * c.ngas[k]) ch = fmax(ch, fabs(nv - a.Nold[i]) / nv);
    }
    ch = block_max(ch, sh);
    if (tid == 0) {
        st->max_change = ch;
        st->h = sh.h;
        st->steps += steps;
        st->rejected += rejected;
        st->status = 0;
    }
}

// ---------------------------------------------------------------------------
// systems of at most kSmallS species: matrices in shared memory
// ---------------------------------------------------------------------------
// A step is a chain of small dependent operations.  An FP64 instruction holds its unit (one to four
// warps) for 65 clocks, whatever the lanes do, and its result takes no longer; a division is ten of
// them, a comparison as much as a product.  So pivots are compared as bit patterns; the column that is
// pivoted next is a warp's own business while the others eliminate; its reciprocals are kept for the
// triangular solves, which one warp does with the vector in registers; and every sum is formed in the
// order of the general kernel, whose results these are bit for bit (a parcel carries a rounding
// through hundreds of steps, grown many orders of magnitude).  A step of 40 species takes 60 us, on the
// general kernel (its matrices in shared memory) 187: the elimination has two fifths of it, the three
// solves over a third, the assembly and the residuals a tenth each.
constexpr int kSmallS = 128;
constexpr int kSmallThreads = 256;
constexpr int kSmallWarps = kSmallThreads / 32;

// Order of |v| among pivot candidates as a bit pattern; 0 for zero and for what is not a number, which
// no pivot search takes.
__device__ __forceinline__ unsigned long long pivot_key(double v)
{
    const unsigned long long k = (unsigned long long)__double_as_longlong(v) & 0x7fffffffffffffffull;
    return k > 0x7ff0000000000000ull ? 0ull : k;
}

// Shared-memory layout of the small kernel (doubles): the matrices' rows are an odd number of words
// apart, so that 32 rows of a column lie in 32 banks.
struct SmallLayout {
    int ld;
    size_t mats, rates, bytes;
};
__host__ __device__ inline SmallLayout small_layout(int S, int R, bool rates_in_smem)
{
    SmallLayout l;
    l.ld = S | 1;
    // before the matrices: x, F, d, r, gain, loss, loss / dz, 1 / pivots, two columns; then the row order
    l.mats = 10 * (size_t)S + (size_t)(S + 1) / 2;
    l.rates = l.mats + 2 * (size_t)S * l.ld;
    l.bytes = (l.rates + (rates_in_smem ? 7 * (size_t)R : 0)) * sizeof(double);
    return l;
}

// A <- its LU factors, order[i] the original row at place i, inv the pivots' reciprocals; l: two columns
// of multipliers.  Warp 0 runs one column ahead: while the others apply step c to the columns from c + 2
// on, it applies it to column c + 1, finds that column's pivot (the first row of largest magnitude) and
// multipliers, and leaves them for the next step.  It has its FP64 unit to itself: warp 4, on the same
// one, only exchanges the rows of the finished columns.  Rows are read where they were and written where
// the exchange puts them.  One barrier per column.  0, or -1 on a zero pivot column, in every thread.
template <int kC>
__device__ int small_factor_rows(double *A, int ld, int *order, double *inv, double *l, int S, Shared &sh)
{
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    for (int c = -1; c + 1 < S; ++c) {
        const int p = c >= 0 ? sh.piv[c & 1] : 0;
        const double *lc = l + (c & 1) * S;
        if (warp == 0) {
            const int j = c + 1;
            double *ln = l + (j & 1) * S;
            const double ap = c >= 0 ? A[p * ld + j] : 0.0, ac = c >= 0 ? A[c * ld + j] : 0.0;
            double v[kC];
            unsigned long long best = 0ull;
            int bi = S;
#pragma unroll
            for (int t = 0; t < kC; ++t) {
                v[t] = 0.0;
                if (j + t * 32 >= S) continue;
                const int i = j + t * 32 + lane, ii = min(i, S - 1);
                v[t] = A[ii * ld + j];
                if (c >= 0) v[t] = fma(-lc[ii], ap, ii == p ? ac : v[t]);
                const unsigned long long k = i < S ? pivot_key(v[t]) : 0ull;
                bi = k > best ? i : bi;
                best = k > best ? k : best;
            }
            const unsigned hi = (unsigned)(best >> 32), mh = __reduce_max_sync(0xffffffffu, hi);
            const unsigned lo = hi == mh ? (unsigned)best : 0u, ml = __reduce_max_sync(0xffffffffu, lo);
            const int q = (int)__reduce_min_sync(0xffffffffu, hi == mh && (unsigned)best == ml ? (unsigned)bi : 0xffffffffu);
            if ((mh | ml) == 0u) {
                if (lane == 0) sh.piv[j & 1] = -1;
            } else {
                double vp = v[0];
#pragma unroll
                for (int t = 1; t < kC; ++t)
                    if (j + t * 32 < S && (q - j) >> 5 == t) vp = v[t];
                vp = __shfl_sync(0xffffffffu, vp, (q - j) & 31);
                const double vc = __shfl_sync(0xffffffffu, v[0], 0), ipv = reciprocal_rn(vp);
                if (lane == 0) {
                    if (c >= 0) A[c * ld + j] = ap;
                    A[j * ld + j] = vp;
                    inv[j] = ipv;
                    const int o = order[j];
                    order[j] = order[q];
                    order[q] = o;
                    sh.piv[j & 1] = q;
                }
#pragma unroll
                for (int t = 0; t < kC; ++t) {
                    if (j + t * 32 >= S) continue;
                    const int i = j + t * 32 + lane;
                    const double m = (i == q ? vc : v[t]) * ipv;
                    if (i > j && i < S) A[i * ld + j] = ln[i] = m;
                }
            }
        } else if (warp == 4) {
            if (c > 0 && p != c)
                for (int j = lane; j < c; j += 32) {
                    const double t = A[c * ld + j];
                    A[c * ld + j] = A[p * ld + j];
                    A[p * ld + j] = t;
                }
        } else if (c >= 0) {
            double m[kC];
#pragma unroll
            for (int t = 0; t < kC; ++t) m[t] = c + 1 + t * 32 < S ? lc[min(c + 1 + t * 32 + lane, S - 1)] : 0.0;
            for (int j = c + 2 + (warp < 4 ? warp - 1 : warp - 2); j < S; j += kSmallWarps - 2) {
                const double ap = A[p * ld + j], ac = A[c * ld + j];
                __syncwarp();
                if (lane == 0) A[c * ld + j] = ap;
#pragma unroll
                for (int t = 0; t < kC; ++t) {
                    if (c + 1 + t * 32 >= S) continue;
                    const int i = c + 1 + t * 32 + lane;
                    if (i < S) A[i * ld + j] = fma(-m[t], ap, i == p ? ac : A[i * ld + j]);
                }
            }
        }
        __syncthreads();
        if (sh.piv[(c + 1) & 1] < 0) return -1;
    }
    return 0;
}

__device__ int small_factor(double *A, int ld, int *order, double *inv, double *l, int S, Shared &sh)
{
    if (S <= 32) return small_factor_rows<1>(A, ld, order, inv, l, S, sh);
    if (S <= 64) return small_factor_rows<2>(A, ld, order, inv, l, S, sh);
    return small_factor_rows<4>(A, ld, order, inv, l, S, sh);
}

// x <- (LU)^-1 P f on one warp, T words of the vector to a lane.
template <int T>
__device__ void warp_lu_solve(const double *A, int ld, const int *order, const double *inv, const double *f, double *x,
                              int S)
{
    const int lane = threadIdx.x & 31;
    double v[T], iv[T];
#pragma unroll
    for (int t = 0; t < T; ++t) {
        const int i = t * 32 + lane;
        v[t] = i < S ? f[order[i]] : 0.0;
        iv[t] = i < S ? inv[i] : 0.0;
    }
#pragma unroll
    for (int t = 0; t < T; ++t) {                  // unit lower triangle, column by column
        const int n = min(32, S - 32 * t);
        for (int q = 0; q < n; ++q) {
            const int c = 32 * t + q;
            double m[T];
#pragma unroll
            for (int u = t; u < T; ++u) {
                const int i = u * 32 + lane;
                m[u] = i > c && i < S ? A[i * ld + c] : 0.0;
            }
            const double xc = __shfl_sync(0xffffffffu, v[t], q);
#pragma unroll
            for (int u = t; u < T; ++u)
                if (u * 32 + lane > c) v[u] = fma(-m[u], xc, v[u]);
        }
    }
#pragma unroll
    for (int t = T - 1; t >= 0; --t) {             // upper triangle
        const int n = min(32, S - 32 * t);
        for (int q = n - 1; q >= 0; --q) {
            const int c = 32 * t + q;
            double m[T];
#pragma unroll
            for (int u = 0; u <= t; ++u) m[u] = u * 32 + lane < c ? A[(u * 32 + lane) * ld + c] : 0.0;
            const double own = v[t] * iv[t];
            const double xc = __shfl_sync(0xffffffffu, own, q);
            if (lane == q) v[t] = xc;
#pragma unroll
            for (int u = 0; u <= t; ++u)
                if (u * 32 + lane < c) v[u] = fma(-m[u], xc, v[u]);
        }
    }
    __syncwarp();                                  // f may be x
#pragma unroll
    for (int t = 0; t < T; ++t)
        if (t * 32 + lane < S) x[t * 32 + lane] = v[t];
    __syncwarp();
}

__device__ void small_solve(const double *A, int ld, const int *order, const double *inv, const double *f, double *x, int S)
{
    if (S <= 32) warp_lu_solve<1>(A, ld, order, inv, f, x, S);
    else if (S <= 64) warp_lu_solve<2>(A, ld, order, inv, f, x, S);
    else warp_lu_solve<4>(A, ld, order, inv, f, x, S);
}

__global__ void __launch_bounds__(kSmallThreads, 1) k_parcel_small(Col c, ParcelArgs a, int rates_in_smem)
{
    __shared__ Shared sh;
    __shared__ double rh;                          // 1 / (step size)
    extern __shared__ double dyn[];
    const int S = c.S, L = c.L, R = c.R;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const Policy &pol = a.pol;
    ParcelState *st = a.st;
    const SmallLayout lay = small_layout(S, R, rates_in_smem);
    const int ld = lay.ld;
    double *x = dyn, *F = x + S, *d = F + S, *r = d + S, *gain = r + S, *loss = gain + S, *ldz = loss + S, *inv = ldz + S;
    double *lbuf = inv + S;
    int *order = (int *)(lbuf + 2 * S);
    double *A0 = dyn + lay.mats, *A = A0 + (size_t)S * ld;
    double *w = rates_in_smem ? dyn + lay.rates : a.w, *dd = rates_in_smem ? w + R : a.dd;
    // places of the pattern's entries in the matrices (-1 - place: on the diagonal); the general
    // kernel's matrices hold them
    int *place = (int *)a.A;
    for (int i = warp; i < S; i += kSmallWarps)
        for (int q = c.jp[i] + lane; q < c.jp[i + 1]; q += 32) {
            const int j = c.jcol[q], e = i * ld + j;
            place[q] = i == j ? -1 - e : e;
        }
    const int nnz = c.jp[S];
    for (long long i = tid; i < (long long)L * S; i += kSmallThreads) a.Nold[i] = a.N[i];
    for (int y = tid; y < S; y += kSmallThreads) a.vmr[y] = a.N[y] / c.ngas[0];
    if (tid == 0) sh.h = st->h;
    long long steps = 0, rejected = 0;
    // the species' sums go to the first warp, the matrix to the others
    const int fw = 1;
    __syncthreads();
    for (int v = 0; v < 2 * L - 1; ++v) {
        const int k = v < L ? v : 2 * L - 2 - v;
        const double nk = c.ngas[k], dzk = c.dz[k];
        const double tau = dzk * dzk / c.Kzz[k];
        for (int y = tid; y < S; y += kSmallThreads) {
            x[y] = a.vmr[y] * nk;
            // the molecular-diffusion pair: the neighbours' densities stay during a visit
            double ls = 0.0, gn = 0.0;
            if (k + 1 < L) {
                ls += a.um[(long long)k * S + y];
                gn += a.vm[(long long)k * S + y] * a.N[(long long)(k + 1) * S + y];
            }
            if (k > 0) {
                ls += a.vm[(long long)(k - 1) * S + y];
                gn += a.um[(long long)(k - 1) * S + y] * a.N[(long long)(k - 1) * S + y];
            }
            gain[y] = gn;
            loss[y] = ls;
            ldz[y] = ls / dzk;
        }
        if (tid == 0) {
            sh.t = 0.0;
            step_size(sh, pol, tau);
        }
        __syncthreads();
        int visit_steps = 0;
        while (sh.t < tau) {
            const double hs = sh.hs;
            // reaction terms at the parcel's densities (Sec. 2.3)
            for (int rr = tid; rr < R; rr += kSmallThreads) reaction_terms_at(c, k, rr, x, w + rr, dd + (long long)rr * 6);
            if (tid == kSmallThreads - 1) rh = 1.0 / hs;
            for (int e = tid; e < 2 * S * ld; e += kSmallThreads) A0[e] = 0.0;      // A follows A0
            for (int y = tid; y < S; y += kSmallThreads) order[y] = y;
            __syncthreads();
            if (warp < fw) {
                for (int y = tid; y < S; y += 32 * fw) {
                    double f = 0.0;
                    const int e1 = c.yp[y + 1];
#pragma unroll 4
                    for (int e = c.yp[y]; e < e1; ++e) {
                        const int code = c.yent[e];
                        f += signed_by(w[code >> 4], (code & 15) >= 8);
                    }
                    F[y] = f + (gain[y] - loss[y] * x[y]) / dzk;
                    if (c.jdq[y] < 0) A0[y * ld + y] = A[y * ld + y] = rh + ldz[y];
                }
            } else {
                // matrix I/h - dF/dx, entries of the pattern summed in a fixed order
                for (int q = tid - 32 * fw; q < nnz; q += kSmallThreads - 32 * fw) {
                    double acc = 0.0;
                    const int t1 = c.jtp[q + 1];
#pragma unroll 4
                    for (int t = c.jtp[q]; t < t1; ++t) {
                        const int code = c.jrs[t], rs = code >> 1;
                        acc += signed_by(dd[(rs >> 3) * 6 + (rs & 7)], code & 1);
                    }
                    int e = place[q];
                    if (e < 0) {
                        e = -1 - e;
                        acc += rh + ldz[e / (ld + 1)];
                    }
                    A0[e] = acc;
                    A[e] = acc;
                }
            }
            __syncthreads();
            if (small_factor(A, ld, order, inv, lbuf, S, sh) != 0) {
                if (tid == 0) { st->status = XK_ESINGULAR; st->visit = v; }
                return;
            }
            if (warp == 0) small_solve(A, ld, order, inv, F, d, S);
            for (int sweep = 0; sweep < kRefineSweeps; ++sweep) {
                __syncthreads();
                for (int i = warp; i < S; i += kSmallWarps) {
                    const double *Ai = A0 + i * ld;
                    double acc = 0.0;
                    for (int j = lane; j < S; j += 32) acc += Ai[j] * d[j];
                    for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
                    if (lane == 0) r[i] = F[i] - acc;
                }
                __syncthreads();
                if (warp == 0) {
                    small_solve(A, ld, order, inv, r, r, S);
                    for (int y = lane; y < S; y += 32) d[y] += r[y];
                    __syncwarp();
                }
            }
            // the Eulerian step controller: reject on a negative or a too large relative change
            if (warp == 0) {
                unsigned long long mk = 0ull;
                int bad = 0;
                for (int y = lane; y < S; y += 32) {
                    const double xv = x[y], dv = d[y], nn = xv + dv;
                    if (!isfinite(nn) || nn < -pol.neg_tol * nk) bad = 1;
                    if (xv > pol.f_floor * nk) mk = max(mk, pivot_key(fabs(dv) / xv));
                }
                bad = __any_sync(0xffffffffu, bad);
                const unsigned hi = (unsigned)(mk >> 32), mh = __reduce_max_sync(0xffffffffu, hi);
                const unsigned ml = __reduce_max_sync(0xffffffffu, hi == mh ? (unsigned)mk : 0u);
                const double mr = __longlong_as_double((long long)((unsigned long long)mh << 32 | ml));
                const bool ok = !bad && !(mr > pol.rel_reject);
                if (ok)
                    for (int y = lane; y < S; y += 32) {
                        const double nn = x[y] + d[y];
                        x[y] = nn < 0.0 ? 0.0 : nn;
                    }
                if (ok) ++steps;
                else ++rejected;
                ++visit_steps;
                if (lane == 0) {
                    step_control(sh, pol, tau, hs, mr, ok, visit_steps, a.max_visit_steps);
                    if (sh.t < tau) step_size(sh, pol, tau);
                }
            }
            __syncthreads();
            if (sh.done) {
                if (tid == 0) { st->status = sh.done; st->visit = v; st->steps += steps; st->rejected += rejected; }
                return;
            }
        }
        for (int y = tid; y < S; y += kSmallThreads) {
            a.N[(long long)k * S + y] = x[y];
            a.vmr[y] = x[y] / nk;
        }
        __syncthreads();
    }
    double ch = 0.0;
    for (long long i = tid; i < (long long)L * S; i += kSmallThreads) {
        const int k = (int)(i / S);
        const double nv = a.N[i];
        if (nv > pol.f_floor * c.ngas[k]) ch = fmax(ch, fabs(nv - a.Nold[i]) / nv);
    }
    ch = block_max(ch, sh);
    if (tid == 0) {
        st->max_change = ch;
        st->h = sh.h;
        st->steps += steps;
        st->rejected += rejected;
        st->status = 0;
    }
}

}  // namespace

cudaError_t launch_parcel_iteration(const Col &c, const ParcelArgs &a, cudaStream_t st)
{
    const int S = c.S;
    SmallLayout small = small_layout(S, c.R, true);
    const bool rates = small.bytes <= kSmemLimit;
    if (!rates) small = small_layout(S, c.R, false);
    count_launches(1);
    if (S <= kSmallS && small.bytes <= kSmemLimit) {
        // eight warps: what a barrier waits for, and two to each FP64 unit
        cudaError_t e = cudaFuncSetAttribute(k_parcel_small, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)small.bytes);
        if (e != cudaSuccess) return e;
        k_parcel_small<<<1, kSmallThreads, small.bytes, st>>>(c, a, rates ? 1 : 0);
        return cudaGetLastError();
    }
    const size_t smem = sizeof(double) * 4 * (size_t)S + sizeof(int) * (size_t)((S + 1) & ~1);
    // fewer warps while the system is small, so that each barrier waits on less; then the whole SM
    const int threads = S <= 160 ? 256 : 1024;
    cudaError_t e = cudaFuncSetAttribute(k_parcel_iteration, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    k_parcel_iteration<<<1, threads, smem, st>>>(c, a);
    return cudaGetLastError();
}

}  // namespace xk

// Chemistry and transport rows of the implicit step: grid, thermochemistry,
// rate coefficients, photolysis, reaction rates and their derivatives,
// residual F(n) (Eq. 1 with the flux of Eq. 2), Jacobian blocks, the
// matrix-free Jacobian-vector product, and device-side step control.
#include <math.h>

#include <algorithm>

#include <atomic>

#include "xk_layer.cuh"

namespace xk {

namespace {

constexpr int kThreads = 256;

inline int nblocks(long long n, int t = kThreads) { return (int)((n + t - 1) / t); }
// Grid of a kernel that a device flag may skip: a grid-stride loop over at most a few waves, so
// that a skipped launch (an FGMRES slot past convergence, an FP64 route not taken) schedules a
// few thousand threads, not one per element.
constexpr int kGatedBlocks = 152 * 8;

// ---------------------------------------------------------------------------
// grid (Sec. 2.1): n_gas = P / (k_B T); hydrostatic altitudes; layer widths
// ---------------------------------------------------------------------------
__global__ void k_grid(Col c)
{
    int L = c.L;
    for (int k = threadIdx.x; k < L; k += blockDim.x)
        c.ngas[k] = c.P[k] * kBarToCgs / (kBoltz * c.T[k]);
    __syncthreads();
    if (threadIdx.x == 0) {
        double z = 0.0;
        c.z[0] = 0.0;
        for (int k = 0; k + 1 < L; ++k) {
            double Th = 0.5 * (c.T[k] + c.T[k + 1]);
            double H = kBoltz * Th / (c.mbar * kAmu * c.g);
            z = z + H * log(c.P[k] / c.P[k + 1]);
            c.z[k + 1] = z;
        }
    }
    __syncthreads();
    for (int k = threadIdx.x; k < L; k += blockDim.x) {
        if (k + 1 < L) c.dzi[k] = c.z[k + 1] - c.z[k];
        double w;
        if (L == 1) w = 1.0;
        else if (k == 0) w = c.z[1] - c.z[0];
        else if (k == L - 1) w = c.z[L - 1] - c.z[L - 2];
        else w = 0.5 * (c.z[k + 1] - c.z[k - 1]);
        c.dz[k] = w;
    }
}

// Eq. 2 at interface k+1/2: phi = u n_k - v n_{k+1}; eddy part in mixing-ratio
// form -K n_gas d(n/n_gas)/dz, molecular part -D (dn/dz + n (1/H_y + (1+alpha_T) T'/T)).
__global__ void k_transport(Col c)
{
    long long idx = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    int S = c.S;
    if (idx >= (long long)(c.L - 1) * S) return;
    int k = (int)(idx / S), y = (int)(idx % S);
    double Th = 0.5 * (c.T[k] + c.T[k + 1]);
    double nh = 0.5 * (c.ngas[k] + c.ngas[k + 1]);
    double Kh = 0.5 * (c.Kzz[k] + c.Kzz[k + 1]);
    double h = c.dzi[k];
    double dTdz = (c.T[k + 1] - c.T[k]) / h;
    double D = c.dcoef[y] * pow(Th, 0.75) / nh;
    double Hy = kBoltz * Th / (c.mass[y] * kAmu * c.g);
    double a = 1.0 / Hy + (1.0 + c.alpha_T) * dTdz / Th;
    c.u[idx] = Kh * nh / (h * c.ngas[k]) + D * (1.0 / h - 0.5 * a);
    c.v[idx] = Kh * nh / (h * c.ngas[k + 1]) + D * (1.0 / h + 0.5 * a);
}

// ---------------------------------------------------------------------------
// thermochemistry (Appendix A) and rate coefficients (Sec. 2.3)
// ---------------------------------------------------------------------------
__device__ __forceinline__ double gibbs_rt(const double *nasa15, double T)
{
    const double *a = (T < nasa15[0]) ? nasa15 + 1 : nasa15 + 8;
    return a[0] * (1.0 - log(T)) - a[1] * T / 2.0 - a[2] * T * T / 6.0
         - a[3] * T * T * T / 12.0 - a[4] * T * T * T * T / 20.0 + a[5] / T - a[6];
}

__global__ void k_gibbs(Col c)
{
    long long idx = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (idx >= (long long)c.L * c.S) return;
    int k = (int)(idx / c.S), y = (int)(idx % c.S);
    c.grt[idx] = gibbs_rt(c.nasa + 15 * y, c.T[k]);
}

__device__ __forceinline__ double arrh(double al, double be, double ga, double T, int form)
{
    double Tb = (form == 0) ? T / 300.0 : T;
    return al * pow(Tb, be) * exp(-ga / T);
}

__device__ __forceinline__ double troe_f(const double *tr, double T, double Pr)
{
    if (tr[0] == 0.0 || Pr <= 0.0) return 1.0;
    double Fc = (1.0 - tr[0]) * exp(-T / tr[1]) + tr[0] * exp(-T / tr[2]);
    if (tr[3] != 0.0) Fc += exp(-tr[3] / T);
    double lFc = log10(Fc);
    double cc = -0.4 - 0.67 * lFc;
    double N = 0.75 - 1.27 * lFc;
    double x = log10(Pr) + cc;
    double q = x / (N - 0.14 * x);
    return pow(10.0, lFc / (1.0 + q * q));
}

// k_f, k_r and ln K_c per (layer, reaction); ln K_c = -sum nu G/RT + dnu ln(p0 / k_B T).
__global__ void k_rates(Col c)
{
    long long idx = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (idx >= (long long)c.L * c.R) return;
    int k = (int)(idx / c.R), r = (int)(idx % c.R);
    double T = c.T[k];
    int t = c.rtype[r];
    const double *grt = c.grt + (long long)k * c.S;
    double dG = 0.0;
    int dnu = 0;
#pragma unroll
    for (int s = 0; s < 3; ++s) {
        int i = c.reac[3 * r + s];
        if (i >= 0) { dG -= grt[i]; dnu -= 1; }
        int j = c.prod[3 * r + s];
        if (j >= 0) { dG += grt[j]; dnu += 1; }
    }
    double lnk = (t == XK_RX_PHOTO) ? 0.0 : -dG + dnu * log(kP0 / (kBoltz * T));
    const double *a = c.arr + 9 * r;
    double f = 0.0, b = 0.0;
    if (t == XK_RX_TWO_BODY) {
        f = arrh(a[0], a[1], a[2], T, c.form[r]);
    } else if (t == XK_RX_THREE_BODY) {
        double k0 = arrh(a[3], a[4], a[5], T, c.form[r]);
        double ki = arrh(a[6], a[7], a[8], T, c.form[r]);
        double M = c.ngas[k];
        double Pr = k0 * M / ki;
        f = k0 * M / (1.0 + k0 * M / ki) * troe_f(c.troe + 4 * r, T, Pr);
    }
    if (t != XK_RX_PHOTO) b = f / exp(lnk);
    c.kf[idx] = f;
    c.kr[idx] = b;
    if (c.lnkc) c.lnkc[idx] = lnk;
}

// ---------------------------------------------------------------------------
// photolysis (Sec. 2.3.3): extinction by absorption and Rayleigh scattering, direct beam with the
// optical depth to the layer midpoint, and optionally the diffuse field J_diff = (J_up + J_down) / 2
// ---------------------------------------------------------------------------
constexpr int kExtLayers = 4;    // layers per thread of the extinction sums (sigma loaded once for them)
constexpr int kExtChunk = 128;   // species whose densities are staged at a time

// alpha (absorption) and alpha_s (scattering) per (layer, wavelength): one thread per wavelength and
// kExtLayers consecutive layers, reading each cross section once for all of them (coalesced in w).
// The densities come from shared memory: fetched through the species' index in the loop, they were
// its latency.  Bound by FP64 issue (one multiply-add per species, layer and wavelength): 57 us at 154
// species, 1,000 wavelengths and 150 layers (97 before, some 45 at the rate k_photo_k reaches).
__global__ void __launch_bounds__(128) k_photo_alpha(Col c, const double *n)
{
    __shared__ __align__(16) double sn[kExtChunk][kExtLayers];
    const int w = blockIdx.x * blockDim.x + threadIdx.x;
    const int k0 = blockIdx.y * kExtLayers;
    const int nk = min(kExtLayers, c.L - k0);
    for (int scatter = 0; scatter < 2; ++scatter) {
        const int cnt = scatter ? c.Ssca : c.Sabs;
        const int *sp = scatter ? c.sca_sp : c.abs_sp;
        const double *sig = (scatter ? c.sig_sca : c.sig_abs) + w;
        double *out = (scatter ? c.alpha_s : c.alpha) + (long long)k0 * c.W + w;
        double s[kExtLayers];
#pragma unroll
        for (int j = 0; j < kExtLayers; ++j) s[j] = 0.0;
        for (int i0 = 0; i0 < cnt; i0 += kExtChunk) {
            const int m = min(kExtChunk, cnt - i0);
            __syncthreads();
            for (int t = threadIdx.x; t < m * kExtLayers; t += blockDim.x) {
                const int i = t / kExtLayers, j = t % kExtLayers;
                sn[i][j] = j < nk ? n[(long long)(k0 + j) * c.S + sp[i0 + i]] : 0.0;
            }
            __syncthreads();
            if (w < c.W) {
                const double *sg = sig + (long long)i0 * c.W;
#pragma unroll 4
                for (int i = 0; i < m; ++i) {
                    const double v = sg[(long long)i * c.W];
#pragma unroll
                    for (int j = 0; j < kExtLayers; ++j) s[j] += v * sn[i][j];
                }
            }
        }
#pragma unroll
        for (int j = 0; j < kExtLayers; ++j)
            if (w < c.W && j < nk) out[(long long)j * c.W] = s[j];
    }
}

// The diffuse field.  In layer k the diffuse fluxes leaving it, D_k down through its bottom and U_k up
// through its top, obey
//     D_k = T_k D_{k+1} + r_k U_{k-1} + P_k / 2,   U_k = T_k U_{k-1} + r_k D_{k+1} + P_k / 2,
// with D_L = 0 and U_{-1} = albedo (D_0 + beam at the bottom); r_k = (1 - t) omega / 2,
// T_k = t + (1 - t) omega / 2, t = exp(-2 dtau_k), omega_k = dtau_s / dtau, and P_k = omega_k mu J0
// (e^{-tau_top/mu} - e^{-tau_bot/mu}) the beam photons the layer scatters.
//
// First kernel: the direct beam into Jw and r, T, P / 2 of every layer, which depend on the layers
// above only through the optical depth.  A CTA takes 32 wavelengths, a warp a run of layers counted
// from the top.  Bound by the FP64 issue of three exponentials a layer (a layer's bottom is the next
// one's top).  Both kernels in one, a thread per wavelength, left half of the SMs' schedulers without
// a warp and the rest waiting for one exponential after the other.  327 us at 10,000 wavelengths and
// 150 layers, and 176 for the second.
constexpr int kPhotoRuns = 16;
__global__ void __launch_bounds__(32 * kPhotoRuns) k_photo_layers(Col c)
{
    __shared__ double runs[kPhotoRuns][33];
    const int lane = threadIdx.x & 31, g = threadIdx.x >> 5, w = blockIdx.x * 32 + lane;
    const bool on = w < c.W;
    const int per = (c.L + kPhotoRuns - 1) / kPhotoRuns;
    const int i0 = min(c.L, g * per), i1 = min(c.L, i0 + per);   // positions from the top: layer L-1-i
    const long long LW = (long long)c.L * c.W;
    double run = 0.0;
    if (on)
        for (int i = i0; i < i1; ++i) {
            const int k = c.L - 1 - i;
            const long long idx = (long long)k * c.W + w;
            run += (c.alpha[idx] + c.alpha_s[idx]) * c.dz[k];
        }
    runs[g][lane] = run;
    __syncthreads();
    double above = 0.0;
    for (int h = 0; h < g; ++h) above += runs[h][lane];
    if (!on || i0 >= i1) return;
    const double J0 = c.J0[w], mu = c.mu, rmu = reciprocal_rn(mu);
    double top = exp(-over(above, mu, rmu));
    for (int i = i0; i < i1; ++i) {
        const int k = c.L - 1 - i;
        const long long idx = (long long)k * c.W + w;
        const double ta = c.alpha[idx] * c.dz[k], ts = c.alpha_s[idx] * c.dz[k], dt = ta + ts;
        c.Jw[idx] = J0 * exp(-over(fma(0.5, dt, above), mu, rmu));
        above += dt;
        const double bot = exp(-over(above, mu, rmu));
        const double om = __double_as_longlong(dt) > 0 ? over(ts, dt, reciprocal_rn(dt)) : 0.0;
        const double t = exp(-2.0 * dt), r = (0.5 - 0.5 * t) * om;
        c.rt[idx] = r;
        c.rt[LW + idx] = t + r;
        c.rt[2 * LW + idx] = 0.5 * (om * mu * J0 * (top - bot));
        top = bot;
    }
}

// Second kernel: one thread per wavelength.  Going down, each layer's fluxes are written in terms of
// the flux entering from below: D_k = p_k U_{k-1} + h0_k, U_k = q_k U_{k-1} + h1_k (p_k is the
// reflectance of the layers from k up, as in the adding method), in the places of r, T and P; going
// up, U_{-1} is found from the boundary and the fluxes follow layer by layer, with J dlambda for the
// sums over wavelength.  Bound by the chain of a reciprocal and four products per layer; the loads run
// kPhotoAhead layers ahead of it.
constexpr int kPhotoAhead = 4;
__global__ void __launch_bounds__(32) k_photo_diffuse(Col c)
{
    const int w = blockIdx.x * 32 + threadIdx.x;
    if (w >= c.W) return;
    const long long W = c.W, LW = (long long)c.L * W;
    double *rt = c.rt + w;
    double pn = 0.0, h0n = 0.0;
    for (int k0 = c.L - 1; k0 >= 0; k0 -= kPhotoAhead) {
        double r[kPhotoAhead], T[kPhotoAhead], P[kPhotoAhead];
#pragma unroll
        for (int j = 0; j < kPhotoAhead; ++j) {
            const double *q = rt + max(k0 - j, 0) * W;
            r[j] = q[0];
            T[j] = q[LW];
            P[j] = q[2 * LW];
        }
#pragma unroll
        for (int j = 0; j < kPhotoAhead; ++j) {
            if (k0 - j < 0) break;
            double *o = rt + (k0 - j) * W;
            const double rd = reciprocal64(fma(-r[j], pn, 1.0));
            const double q = T[j] * rd, h1 = fma(r[j], h0n, P[j]) * rd, tp = T[j] * pn;
            pn = fma(tp, q, r[j]);
            h0n = fma(tp, h1, fma(T[j], h0n, P[j]));
            o[0] = pn;
            o[LW] = q;
            o[2 * LW] = h0n;
            o[3 * LW] = h1;
        }
    }
    double above = 0.0;
    for (int k = c.L - 1; k >= 0; --k) {
        const long long i = (long long)k * W + w;
        above += c.alpha[i] * c.dz[k] + c.alpha_s[i] * c.dz[k];
    }
    const double A = c.albedo, bottom = c.mu * c.J0[w] * exp(-above / c.mu), dl = c.dlam[w];
    // U_{-1} = A (D_0 + bottom), D_0 = p_0 U_{-1} + h0_0
    double Ub = A * (h0n + bottom) / (1.0 - A * pn), Dk = fma(pn, Ub, h0n);
    for (int k0 = 0; k0 < c.L; k0 += kPhotoAhead) {
        double p[kPhotoAhead], q[kPhotoAhead], h0[kPhotoAhead], h1[kPhotoAhead], J[kPhotoAhead];
#pragma unroll
        for (int j = 0; j < kPhotoAhead; ++j) {
            const int k = min(k0 + j, c.L - 1), u = min(k + 1, c.L - 1);
            q[j] = rt[LW + k * W];
            h1[j] = rt[3 * LW + k * W];
            p[j] = k + 1 < c.L ? rt[u * W] : 0.0;              // of the layer above: D_L = 0
            h0[j] = k + 1 < c.L ? rt[2 * LW + u * W] : 0.0;
            J[j] = c.Jw[k * W + w];
        }
#pragma unroll
        for (int j = 0; j < kPhotoAhead; ++j) {
            if (k0 + j >= c.L) break;
            const double Uk = fma(q[j], Ub, h1[j]), Dn = fma(p[j], Uk, h0[j]);
            const double Jk = fma(0.25, (Ub + Uk) + (Dk + Dn), J[j]);
            const long long i = (k0 + j) * W + w;
            c.Jw[i] = Jk;
            c.Jd[i] = Jk * dl;
            Ub = Uk;
            Dk = Dn;
        }
    }
}

// Direct beam only: one warp per wavelength.  Lane l takes a run of consecutive layers counted
// from the top, sums their optical thicknesses, and a warp scan gives the optical depth above its
// run; the lane then walks its run (32x the parallelism of a thread per wavelength, which left
// 1,000 bins on 8 SMs).
__global__ void k_photo_J_direct(Col c)
{
    const int w = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int lane = threadIdx.x & 31;
    if (w >= c.W) return;
    const int per = (c.L + 31) / 32;
    const int i0 = lane * per, i1 = min(c.L, i0 + per);   // positions from the top: layer L-1-i
    double run = 0.0;
    for (int i = i0; i < i1; ++i) {
        const int k = c.L - 1 - i;
        const long long idx = (long long)k * c.W + w;
        run += (c.alpha[idx] + c.alpha_s[idx]) * c.dz[k];
    }
    double incl = run;
    for (int o = 1; o < 32; o <<= 1) {
        const double v = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += v;
    }
    double above = __shfl_up_sync(0xffffffffu, incl, 1);   // sum over the runs above this one
    if (lane == 0) above = 0.0;
    const double J0 = c.J0[w], mu = c.mu, rmu = reciprocal_rn(mu), dl = c.dlam[w];
    for (int i = i0; i < i1; ++i) {
        const int k = c.L - 1 - i;
        const long long idx = (long long)k * c.W + w;
        const double dt = (c.alpha[idx] + c.alpha_s[idx]) * c.dz[k];
        const double J = J0 * exp(-over(fma(0.5, dt, above), mu, rmu));
        c.Jw[idx] = J;
        c.Jd[idx] = J * dl;
        above += dt;
    }
}

// k_ph = t_f sum_w J(k, w) sigma(w) dlambda(w): a CTA takes KT layers x kPhotoQ reactions, its four
// warps every fourth run of 32 wavelengths; the lanes' sums are folded with each exchange halving what
// a lane holds (one FP64 addition per output and warp, where a warp per output added 32 one after the
// other), then the warps' in order.  Bound by FP64 issue, one multiply-add per layer, reaction and
// wavelength (J dlambda comes ready from the kernel before): 65 us at 200 reactions, 1,000 wavelengths
// and 150 layers (199 before), 513 at 10,000.
//
// Below kPhotoFaint the order of a product decides how many bits are left of it: a term loses at most
// half the smallest double, 2.5e-324, times dlambda, and thousands of them are seen in sums below some
// 1e-305 only.  There the sum is formed again with the products as the definition has them, (J sigma)
// dlambda (a few rates in the layers where the beam ends, 10 us; sums of such numbers are exact or nearly).
constexpr int kPhotoQ = 8;
constexpr double kPhotoFaint = 1e-302;
template <int KT>
__global__ void __launch_bounds__(128) k_photo_k(Col c)
{
    __shared__ double part[4][KT * kPhotoQ];
    __shared__ int faint[KT * kPhotoQ];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nq = (c.Rph + kPhotoQ - 1) / kPhotoQ;
    const int k0 = blockIdx.x / nq * KT, q0 = blockIdx.x % nq * kPhotoQ;
    const double *J[KT], *sg[kPhotoQ];
#pragma unroll
    for (int i = 0; i < KT; ++i) J[i] = c.Jd + (long long)min(k0 + i, c.L - 1) * c.W;
#pragma unroll
    for (int q = 0; q < kPhotoQ; ++q) sg[q] = c.sigma + (long long)min(q0 + q, c.Rph - 1) * c.W;
    double acc[KT][kPhotoQ];
#pragma unroll
    for (int i = 0; i < KT; ++i)
#pragma unroll
        for (int q = 0; q < kPhotoQ; ++q) acc[i][q] = 0.0;
    for (int w = threadIdx.x; w < c.W; w += 128) {
        double j[KT];
#pragma unroll
        for (int i = 0; i < KT; ++i) j[i] = J[i][w];
#pragma unroll
        for (int q = 0; q < kPhotoQ; ++q) {
            const double v = sg[q][w];
#pragma unroll
            for (int i = 0; i < KT; ++i) acc[i][q] = fma(j[i], v, acc[i][q]);
        }
    }
#pragma unroll
    for (int i = 0; i < KT; ++i) {
        double v[kPhotoQ];
#pragma unroll
        for (int q = 0; q < kPhotoQ; ++q) v[q] = acc[i][q];
#pragma unroll
        for (int h = kPhotoQ / 2, o = 16; h; h >>= 1, o >>= 1)
#pragma unroll
            for (int q = 0; q < h; ++q) {
                const bool hi = lane & o;
                const double give = hi ? v[q] : v[q + h], keep = hi ? v[q + h] : v[q];
                v[q] = keep + __shfl_xor_sync(0xffffffffu, give, o);
            }
        double t = v[0];
        t += __shfl_xor_sync(0xffffffffu, t, 2);
        t += __shfl_xor_sync(0xffffffffu, t, 1);
        // a lane's output: bits 4, 3, 2 of its number
        if ((lane & 3) == 0) part[warp][i * kPhotoQ + (lane >> 2)] = t;
    }
    __syncthreads();
    if (threadIdx.x < KT * kPhotoQ) {
        const int k = k0 + threadIdx.x / kPhotoQ, q = q0 + threadIdx.x % kPhotoQ;
        double t = 0.0;
        for (int i = 0; i < 4; ++i) t += part[i][threadIdx.x];
        const bool in = k < c.L && q < c.Rph;
        if (in) c.kph[(long long)k * c.Rph + q] = c.tf * t;
        faint[threadIdx.x] = in && t > 0.0 && t < kPhotoFaint;
    }
    __syncthreads();
    for (int e = warp; e < KT * kPhotoQ; e += 4) {
        if (!faint[e]) continue;
        const int k = k0 + e / kPhotoQ, q = q0 + e % kPhotoQ;
        const double *Jk = c.Jw + (long long)k * c.W, *sq = c.sigma + (long long)q * c.W;
        double t = 0.0;
#pragma unroll 8
        for (int w = lane; w < c.W; w += 32) t += Jk[w] * sq[w] * c.dlam[w];
        for (int o = 16; o; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
        if (lane == 0) c.kph[(long long)k * c.Rph + q] = c.tf * t;
    }
}

// one warp per (layer, reaction), lanes striding the wavelengths, partial sums added in lane order: the
// parcel scheme's, whose sweep grows a rounding of the rates by eight orders of magnitude and more, so
// that its results stand or fall with the order of this sum.  200 us against k_photo_k's 65 at 200
// reactions, 1,000 wavelengths and 150 layers, of an iteration's 260 ms.
__global__ void k_photo_k_ordered(Col c)
{
    const int warp = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, lane = threadIdx.x & 31;
    if (warp >= c.L * c.Rph) return;
    const double *J = c.Jw + (long long)(warp / c.Rph) * c.W, *sg = c.sigma + (long long)(warp % c.Rph) * c.W;
    double s = 0.0;
    for (int w = lane; w < c.W; w += 32) s += J[w] * sg[w] * c.dlam[w];
    double tot = 0.0;
    for (int l = 0; l < 32; ++l) tot += __shfl_sync(0xffffffffu, s, l);
    if (lane == 0) c.kph[warp] = c.tf * tot;
}

// ---------------------------------------------------------------------------
// reaction rates w = k_f prod n_reac - k_r prod n_prod and partial derivatives
// d[slot] = d(k_f prod n_reac)/d n_reac[slot] (slots 0-2) and
//           -d(k_r prod n_prod)/d n_prod[slot] (slots 3-5)
// ---------------------------------------------------------------------------
// Layer k of the step's right-hand side, by one CTA: the reaction rates and derivatives
// (reaction_terms_at), then F = sum_r nu w_r - (phi_{k+1/2} - phi_{k-1/2}) / dz_k from the rates in
// shared memory, the solve scaling s = max(n, f_floor n_gas) with b = F / s, and, when diag is
// given, the rows' equilibration: diag = max(|I/dt - dF/dn|_ii, 1/dt) and bhat = b / diag, the
// diagonal entry summed from the derivatives just written.  A kernel per quantity with a thread per
// species took 170 us at 594 species x 150 layers, most of it in the few threads that hold the bath
// gas's thousands of entries one after the other.
__global__ void __launch_bounds__(512)
k_layer_terms(Col c, const double *n, double *F, const Ctl *ctl, double f_floor, double *diag, double *bhat,
              int rates_in_smem)
{
    if (ctl && ctl->finished) return;
    extern __shared__ double lt_sm[];
    const int S = c.S, R = c.R, L = c.L;
    for (int k = blockIdx.x; k < L; k += gridDim.x) {
        double *sn = lt_sm, *part = sn + S, *w = rates_in_smem ? part + c.nsub : c.w + (long long)k * R;
        const long long row0 = (long long)k * S;
        __syncthreads();
        for (int i = threadIdx.x; i < S; i += blockDim.x) sn[i] = n[row0 + i];
        __syncthreads();
        double *dk = c.d + (long long)k * R * 6;
        for (int r = threadIdx.x; r < R; r += blockDim.x) {
            double wr, d[6];
            reaction_terms_at(c, k, r, sn, &wr, d);
            w[r] = wr;
            double2 *o = (double2 *)(dk + (long long)r * 6);
            o[0] = make_double2(d[0], d[1]);
            o[1] = make_double2(d[2], d[3]);
            o[2] = make_double2(d[4], d[5]);
        }
        __syncthreads();
        species_parts(c, w, part);
        __syncthreads();
        for (int i = threadIdx.x; i < S; i += blockDim.x) {
            const long long idx = row0 + i;
            const double nk = sn[i];
            double f = -species_sum(c, part, i);
            double upf = 0.0, dnf = 0.0;
            if (k + 1 < L) upf = c.u[idx] * nk - c.v[idx] * n[idx + S];
            if (k > 0) dnf = c.u[idx - S] * n[idx - S] - c.v[idx - S] * nk;
            f += -(upf - dnf) / c.dz[k];
            if (c.fshift) f -= c.fshift[idx];
            F[idx] = f;
            if (c.s) {
                const double sc = fmax(nk, f_floor * c.ngas[k]);
                c.s[idx] = sc;
                c.b[idx] = f / sc;
                c.rs[idx] = 1.0 / sc;
            }
        }
        if (!diag) continue;
        __syncthreads();
        // diagonal entries: the same sublists over the terms of each species' own column
        const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
        for (int g = warp; g < c.ndg; g += nw) {
            double acc = 0.0;
            const int q1 = c.dgp[g + 1];
#pragma unroll 4
            for (int q = c.dgp[g]; q < q1; ++q) {
                const int code = c.dent[32 * q + lane];
                if (code >= 0) acc += signed_by(dk[code >> 1], code & 1);
            }
            const int to = c.dpart[32 * g + lane];
            if (to >= 0) part[to] = acc;
        }
        __syncthreads();
        const double rdt = 1.0 / ctl->dt;
        for (int i = threadIdx.x; i < S; i += blockDim.x) {
            const long long idx = row0 + i;
            double acc = 0.0;
            for (int q = c.dsp[i]; q < c.dsp[i + 1]; ++q) acc += part[q];
            const double dg = fmax(fabs(rdt + acc + c.tdg[idx]), rdt);
            diag[idx] = dg;
            bhat[idx] = c.b[idx] / dg;
        }
    }
}

// Dense diagonal blocks A_k = I/dt - dF_k/dn_k, couplings lo/up.  scaled != 0 writes
// diag(1/s) A diag(s) and the matching couplings.
//
// A row's non-zeros come from the reactions its species is in, about fifty of a network's thousands.
// A warp loads those reactions' derivatives (48 contiguous bytes each) into shared memory once and
// its lanes then sum whole columns of the row from there, each in a fixed order, eight rows to a
// CTA; a species in more than kJacOcc reactions (the bath gas is in thousands) takes a whole CTA.
// Gathering every term of every entry from global memory instead is bound by its latency: 1,290 us
// at 594 species x 150 layers, this 390.  Bound by FP64 issue and latency: the additions of the terms
// (4.2e7, about 75 us if every lane had the same number) and two products and a conversion per non-zero
// entry; beside them the write of the blocks (222 MB in FP32, 33 us).  An entry of more than kJacLong
// terms (the diagonal has one per reaction of the row) is summed by the warp, four of them together,
// since one lane's chain held up the other 31 (541 us).
template <typename T>
__global__ void __launch_bounds__(kJacWarps * 32)
k_jacobian(Col c, const Ctl *ctl, double dt_override, int scaled, T *A, T *lo, T *up, const int *skip, long long lstride)
{
    if ((ctl && ctl->finished) || (skip && *skip)) return;
    extern __shared__ __align__(16) unsigned char jac_sm[];
    const int S = c.S, L = c.L, ld = c.ld;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    double *dall = (double *)jac_sm;                                  // kJacHeavyOcc * 6: the tiles' derivatives
    double *hrow = dall + kJacHeavyOcc * 6;                           // S: a heavy row
    T *row = (T *)(hrow + S) + (long long)warp * S;                   // S: this warp's light row
    double *dbuf = dall + warp * kJacOcc * 6;
    const double rdt = 1.0 / (dt_override > 0.0 ? dt_override : ctl->dt);
    if (lstride <= 0) lstride = (long long)S * ld;

    // derivatives of tile t's reactions, by nt threads of which this is number id
    auto load_tile = [&](const double2 *dk, int t, double *dst, int id, int nt) {
        const int o0 = c.jto[t], n = (c.jto[t + 1] - o0) * 3;
        for (int b = id; b < n; b += 8 * nt) {
            double2 v[8];
#pragma unroll
            for (int u = 0; u < 8; ++u) {
                const int e = min(b + u * nt, n - 1), occ = e / 3;
                v[u] = dk[3 * (long long)(c.yent[o0 + occ] >> 4) + (e - 3 * occ)];
            }
#pragma unroll
            for (int u = 0; u < 8; ++u)
                if (b + u * nt < n) ((double2 *)dst)[b + u * nt] = v[u];
        }
    };
    // every step-th term from t to t1 (an addition of nothing costs as much as any other: the first
    // term is taken as it is)
    auto lane_sum = [&](const double *src, int t, int t1, int step) {
        double acc = 0.0;
        if (t < t1) {
            const int code = c.jterm[t];
            acc = signed_by(src[code >> 1], code & 1);
            t += step;
        }
#pragma unroll 4
        for (; t < t1; t += step) {
            const int code = c.jterm[t];
            acc += signed_by(src[code >> 1], code & 1);
        }
        return acc;
    };
    auto group_sum = [&](const double *src, int g) { return lane_sum(src, c.jge[g], c.jge[g + 1], 1); };
    // the sums of long groups g .. g + 3 (those below g1), by the warp: a lane's terms, then exchanges
    // of which the first two halve the groups a lane holds; lane l gets group g + l / 8
    auto long_sums = [&](const double *src, int g, int g1) {
        double v[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) v[q] = g + q < g1 ? lane_sum(src, c.jge[g + q] + lane, c.jge[g + q + 1], 32) : 0.0;
        const bool h16 = lane & 16, h8 = lane & 8;
        const double a0 = (h16 ? v[2] : v[0]) + __shfl_xor_sync(0xffffffffu, h16 ? v[0] : v[2], 16);
        const double a1 = (h16 ? v[3] : v[1]) + __shfl_xor_sync(0xffffffffu, h16 ? v[1] : v[3], 16);
        double t = (h8 ? a1 : a0) + __shfl_xor_sync(0xffffffffu, h8 ? a0 : a1, 8);
        for (int o = 4; o; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
        return t;
    };
    auto is_long = [&](int g) { return c.jge[g + 1] - c.jge[g] > kJacLong; };
    auto couplings = [&](int k, int i) {
        const long long q = (long long)k * S + i;
        double lov = c.tlo[q], upv = c.tup[q];
        if (scaled) {
            const double ri = c.rs[q];
            if (k > 0) lov *= c.s[q - S] * ri;
            if (k + 1 < L) upv *= c.s[q + S] * ri;
        }
        lo[q] = (T)lov;
        up[q] = (T)upv;
    };

    const long long items = (long long)c.nji * L;
    for (long long it = blockIdx.x; it < items; it += gridDim.x) {
        const int q = (int)(it / L), k = (int)(it - (long long)q * L);
        const double2 *dk = (const double2 *)(c.d + (long long)k * c.R * 6);
        const double *sk = c.s + (long long)k * S;
        if (c.jit[kJacWarps * q + 1] != -2) {
            const int i = c.jit[kJacWarps * q + warp];
            if (i < 0) continue;
            for (int j = lane; j < S; j += 32) row[j] = (T)0;
            const double diag = rdt + c.tdg[(long long)k * S + i];
            const double inv = scaled ? c.rs[(long long)k * S + i] : 1.0;
            __syncwarp();
            const int t = c.jrt[i];
            if (t < c.jrt[i + 1]) {                       // one tile at most
                load_tile(dk, t, dbuf, lane, 32);
                __syncwarp();
                const int g1 = c.jtg[t + 1];
                for (int g = c.jtg[t]; g < g1;) {
                    // the longest come first: up to 32 of them one after the other, a lane keeping
                    // each, then a lane for each of the next 32
                    const int g0 = g;
                    double v = 0.0;
                    int n = 0;
                    for (; n < 32 && g < g1 && is_long(g); n += 4, g += 4) {
                        const double s = long_sums(dbuf, g, g1);
                        const double mine = __shfl_sync(0xffffffffu, s, (lane & 3) * 8);
                        if (lane >> 2 == n >> 2) v = mine;
                    }
                    if (g > g1) {
                        n -= g - g1;
                        g = g1;
                    }
                    if (n == 0) {
                        n = min(32, g1 - g);
                        if (lane < n) v = group_sum(dbuf, g + lane);
                        g += n;
                    }
                    if (lane < n) {
                        const int j = c.jgc[g0 + lane];
                        if (j == i) v += diag;
                        if (scaled && j != i) v = v * sk[j] * inv;
                        row[j] = (T)v;
                    }
                }
            }
            if (lane == 0) {
                if (c.jdq[i] < 0) row[i] = (T)diag;       // no reaction holds it
                couplings(k, i);
            }
            __syncwarp();
            T *Ar = A + (long long)k * lstride + (long long)i * ld;
            for (int j = lane; j < ld; j += 32) Ar[j] = j < S ? row[j] : (T)0;
            __syncwarp();
        } else {
            const int i = c.jit[kJacWarps * q];
            const double diag = rdt + c.tdg[(long long)k * S + i];
            const double inv = scaled ? c.rs[(long long)k * S + i] : 1.0;
            __syncthreads();
            for (int j = threadIdx.x; j < S; j += blockDim.x) hrow[j] = j == i ? diag : 0.0;
            for (int t = c.jrt[i]; t < c.jrt[i + 1]; ++t) {
                __syncthreads();
                load_tile(dk, t, dall, threadIdx.x, blockDim.x);
                __syncthreads();
                // long groups four to a warp, the others a thread each (the longest come first)
                const int g1 = c.jtg[t + 1];
                const int g0 = c.jtg[t];
                for (int g = g0 + 4 * warp; g < g1 && is_long(g); g += 4 * kJacWarps) {
                    const double v = long_sums(dall, g, g1);
                    if (!(lane & 7) && g + (lane >> 3) < g1) hrow[c.jgc[g + (lane >> 3)]] += v;
                }
                // (a group of four that began with a long one is done)
                for (int g = g0 + threadIdx.x; g < g1; g += blockDim.x)
                    if (!is_long(g0 + ((g - g0) & ~3))) hrow[c.jgc[g]] += group_sum(dall, g);
            }
            __syncthreads();
            T *Ar = A + (long long)k * lstride + (long long)i * ld;
            for (int j = threadIdx.x; j < ld; j += blockDim.x) {
                double v = j < S ? hrow[j] : 0.0;
                if (scaled && j < S && j != i) v = v * sk[j] * inv;
                Ar[j] = (T)v;
            }
            if (threadIdx.x == 0) couplings(k, i);
            __syncthreads();
        }
    }
}

// ---------------------------------------------------------------------------
// photolysis rates in the Jacobian (cfg.photo_jacobian): the change of k_ph along the physical
// direction v = s x of J v.  The direct beam J = J0 exp(-tau/mu) changes by -J dtau/mu, with dtau
// the optical depth of the extinction change sum_i sigma_i v_i above the layer (half the layer's
// own), so dk_ph = t_f sum_w dJ sigma dlambda; the rate w = k_ph n_A then changes by dk_ph n_A.
// ---------------------------------------------------------------------------
__global__ void k_photo_beta(Col c, const Ctl *ctl, const double *x, const int *skip)
{
    if ((ctl && ctl->finished) || (skip && *skip)) return;
    const int w = blockIdx.x * blockDim.x + threadIdx.x;
    const int k0 = blockIdx.y * kExtLayers;
    if (w >= c.W) return;
    const int nk = min(kExtLayers, c.L - k0);
    double sb[kExtLayers];
#pragma unroll
    for (int j = 0; j < kExtLayers; ++j) sb[j] = 0.0;
    for (int i = 0; i < c.Sabs; ++i) {
        const double sg = c.sig_abs[(long long)i * c.W + w];
        const int y = c.abs_sp[i];
#pragma unroll
        for (int j = 0; j < kExtLayers; ++j)
            if (j < nk) {
                const long long e = (long long)(k0 + j) * c.S + y;
                sb[j] += sg * c.s[e] * x[e];
            }
    }
    for (int i = 0; i < c.Ssca; ++i) {
        const double sg = c.sig_sca[(long long)i * c.W + w];
        const int y = c.sca_sp[i];
#pragma unroll
        for (int j = 0; j < kExtLayers; ++j)
            if (j < nk) {
                const long long e = (long long)(k0 + j) * c.S + y;
                sb[j] += sg * c.s[e] * x[e];
            }
    }
#pragma unroll
    for (int j = 0; j < kExtLayers; ++j)
        if (j < nk) c.pbeta[(long long)(k0 + j) * c.W + w] = sb[j];
}

// one warp per wavelength, the same run-and-scan layout as the direct beam
__global__ void k_photo_dJ(Col c, const Ctl *ctl, const int *skip)
{
    if ((ctl && ctl->finished) || (skip && *skip)) return;
    const int w = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int lane = threadIdx.x & 31;
    if (w >= c.W) return;
    const int per = (c.L + 31) / 32;
    const int i0 = lane * per, i1 = min(c.L, i0 + per);
    double run = 0.0;
    for (int i = i0; i < i1; ++i) {
        const int k = c.L - 1 - i;
        run += c.pbeta[(long long)k * c.W + w] * c.dz[k];
    }
    double incl = run;
    for (int o = 1; o < 32; o <<= 1) {
        const double v = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += v;
    }
    double above = __shfl_up_sync(0xffffffffu, incl, 1);
    if (lane == 0) above = 0.0;
    for (int i = i0; i < i1; ++i) {
        const int k = c.L - 1 - i;
        const long long idx = (long long)k * c.W + w;
        const double db = c.pbeta[idx] * c.dz[k];
        c.pdJ[idx] = -c.Jw[idx] * (above + 0.5 * db) / c.mu;
        above += db;
    }
}

// dk_ph = t_f sum_w dJ sigma dlambda; one warp per (layer, reaction)
__global__ void k_photo_dk(Col c, const Ctl *ctl, const int *skip)
{
    if ((ctl && ctl->finished) || (skip && *skip)) return;
    const int warp = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int lane = threadIdx.x & 31;
    if (warp >= c.L * c.Rph) return;
    const int k = warp / c.Rph, q = warp % c.Rph;
    const double *dJ = c.pdJ + (long long)k * c.W;
    const double *sg = c.sigma + (long long)q * c.W;
    double s = 0.0;
    for (int w = lane; w < c.W; w += 32) s += dJ[w] * sg[w] * c.dlam[w];
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if (lane == 0) c.pdk[(long long)k * c.Rph + q] = c.tf * s;
}

// y = diag(1/s) (I/dt - J) diag(s) x, one CTA per layer (xk_layer.cuh)
__global__ void __launch_bounds__(512) k_jv_layer(Col c, const Ctl *ctl, const double *x, double *y,
                                                  const double *rowdiv, const int *skip, int rates_in_smem)
{
    if ((ctl && ctl->finished) || (skip && *skip)) return;
    extern __shared__ double jv_sm[];
    for (int k = blockIdx.x; k < c.L; k += gridDim.x) {
        __syncthreads();
        jv_layer_body(c, ctl, x, y, rowdiv, k, jv_sm, rates_in_smem != 0);
    }
}

__global__ void k_unscale(Col c, const double *xs, double *delta)
{
    long long idx = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (idx >= (long long)c.L * c.S) return;
    delta[idx] = xs[idx] * c.s[idx];
}

// ---------------------------------------------------------------------------
// step control on the device
// ---------------------------------------------------------------------------
__global__ void k_check(Col c, Ctl *ctl, Policy pol)
{
    if (ctl->finished) return;
    long long idx = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    int S = c.S;
    double rel = 0.0;
    int bad = 0, neg = 0;
    if (idx < (long long)c.L * S) {
        int k = (int)(idx / S);
        double nv = c.n[idx], dv = c.delta[idx];
        double nn = nv + dv;
        double ng = c.ngas[k];
        if (!isfinite(nn)) bad = 1;
        else {
            if (nn < -pol.neg_tol * ng) bad = 1;
            if (nn < 0.0) neg = 1;
            if (nv > pol.f_floor * ng) rel = fabs(dv) / nv;
        }
    }
    // warp-level combine, one atomic per warp
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        rel = fmax(rel, __shfl_xor_sync(0xffffffffu, rel, o));
        bad |= __shfl_xor_sync(0xffffffffu, bad, o);
        neg += __shfl_xor_sync(0xffffffffu, neg, o);
    }
    if ((threadIdx.x & 31) == 0) {
        if (rel > 0.0) atomicMax(&ctl->max_rel_bits, (unsigned long long)__double_as_longlong(rel));
        if (bad) atomicOr(&ctl->bad, 1);
        if (neg) atomicAdd(&ctl->n_neg, neg);
    }
}

// Mixed precision routing at the start of a step: steps at dt at or above the
// smallest dt where the FP32-preconditioned solve failed go straight to FP64.
__global__ void k_route(Ctl *ctl)
{
    ctl->skip32 = ctl->dt >= ctl->dt_fp64 ? 1 : 0;
    const int reuse = ctl->skip32 && ctl->have64 && ctl->reuse_enabled;
    ctl->skip_reuse = reuse ? 0 : 1;
    ctl->skip64 = (ctl->skip32 && !reuse) ? 0 : 1;
    ctl->used_fp64 = ctl->skip32;
}

// Scalings of the reused FP64 factorization: input rowd * s / s64, output s64 / s.
__global__ void k_reuse_scales(long long N, const double *rowd, const double *s, const double *s64, double *pin,
                               double *pout, const Ctl *ctl)
{
    if (ctl->finished || ctl->skip_reuse) return;
    long long idx = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (idx >= N) return;
    pin[idx] = rowd[idx] * s[idx] / s64[idx];
    pout[idx] = s64[idx] / s[idx];
}

// After an FP64 factorization: remember its scaling, mark the factors valid.
__global__ void k_after_refactor(long long N, const double *s, double *s64, Ctl *ctl)
{
    if (ctl->finished || ctl->skip64) return;
    long long idx = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (idx < N) s64[idx] = s[idx];
    if (idx == 0) {
        ctl->have64 = !ctl->err_timeout;     // pivots and blocks of one that gave up are not complete
        ctl->refactors += 1;
    }
}

__global__ void k_begin(Ctl *ctl)
{
    if (ctl->finished) {
        ctl->accepted = 0;
        return;
    }
    ctl->max_rel_bits = 0ull;
    ctl->solver_iters = 0;
    ctl->solver_resid = 0.0;
    ctl->bad = 0;
    ctl->n_neg = 0;
    ctl->accepted = 0;
    ctl->converged = 0;
}

__global__ void k_decide(Ctl *ctl, Policy pol)
{
    if (ctl->finished) return;
    double dt = ctl->dt;
    double maxrel = __longlong_as_double((long long)ctl->max_rel_bits);
    int ok = !ctl->bad && !ctl->err_singular && !ctl->err_timeout;
    if (ok && maxrel > pol.rel_reject) ok = 0;
    ctl->max_rel = maxrel;
    ctl->last_dt = dt;
    ctl->steps += 1;
    if (ctl->used_fp64) ctl->fp64_steps += 1;
    if (ok) {
        double fac = (maxrel > 0.0) ? pol.rel_target / maxrel : pol.grow_max;
        if (fac > pol.grow_max) fac = pol.grow_max;
        if (fac < pol.shrink_min) fac = pol.shrink_min;
        double dn = dt * fac;
        ctl->dt_next = (dn > pol.dt_max) ? pol.dt_max : dn;
        ctl->accepted = 1;
        ctl->n_acc += 1;
        ctl->t += dt;
        if (dt >= pol.ss_dt && maxrel < pol.ss_tol) {
            ctl->converged = 1;
            ctl->finished = 1;
        }
    } else {
        ctl->dt_next = 0.5 * dt;
        ctl->accepted = 0;
        ctl->n_neg = 0;
        ctl->n_rej += 1;
        if (ctl->err_timeout) { ctl->status = XK_ETIMEOUT; ctl->finished = 1; }
        else if (ctl->dt_next < pol.dt_min) { ctl->status = XK_ENEG; ctl->finished = 1; }
    }
    ctl->dt = ctl->dt_next;
}

// n <- max(n + delta, 0) on an accepted step (reads the decision of this step).
__global__ void k_apply(Col c, Ctl *ctl)
{
    if (!ctl->accepted) return;
    long long idx = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (idx >= (long long)c.L * c.S) return;
    double nn = c.n[idx] + c.delta[idx];
    c.n[idx] = nn < 0.0 ? 0.0 : nn;
}

__global__ void k_set_mixing(Col c, const double *f, double *n)
{
    long long idx = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (idx >= (long long)c.L * c.S) return;
    n[idx] = f[idx] * c.ngas[idx / c.S];
}

}  // namespace

static std::atomic<long long> g_launches{0};
void count_launches(long long n) { g_launches.fetch_add(n, std::memory_order_relaxed); }
long long launches() { return g_launches.load(std::memory_order_relaxed); }

__global__ void k_convert32(const double *src, size_t lds, float *dst, size_t ldd, size_t rows, size_t cols)
{
    long long idx = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (idx >= (long long)(rows * cols)) return;
    size_t r = idx / cols, j = idx - r * cols;
    dst[r * ldd + j] = (float)src[r * lds + j];
}

void launch_convert32(const double *src, size_t lds, float *dst, size_t ldd, size_t rows, size_t cols, cudaStream_t st)
{
    if (rows * cols == 0) return;
    count_launches(1);
    k_convert32<<<nblocks((long long)(rows * cols)), kThreads, 0, st>>>(src, lds, dst, ldd, rows, cols);
}

void launch_set_mixing(const Col &c, const double *f, double *n, cudaStream_t st)
{
    if (((long long)c.L * c.S) > 0) { count_launches(1); k_set_mixing<<<nblocks((long long)c.L * c.S), kThreads, 0, st>>>(c, f, n); }
}

// ---------------------------------------------------------------------------
// Transport terms of the rows of I/dt - dF/dn, once per atmosphere: read by the rows' equilibration, the
// Jacobian's assembly and J v.
__global__ void k_transport_rows(Col c)
{
    const long long idx = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    const int S = c.S, L = c.L;
    if (idx >= (long long)L * S) return;
    const int k = (int)(idx / S), i = (int)(idx % S);
    double dg = 0.0;
    if (k + 1 < L) dg += c.u[(long long)k * S + i] / c.dz[k];
    if (k > 0) dg += c.v[(long long)(k - 1) * S + i] / c.dz[k];
    c.tdg[idx] = dg;
    c.tlo[idx] = (k > 0) ? -c.u[(long long)(k - 1) * S + i] / c.dz[k] : 0.0;
    c.tup[idx] = (k + 1 < L) ? -c.v[(long long)k * S + i] / c.dz[k] : 0.0;
}

void launch_transport_coeffs(const Col &c, const double *Kzz, double *u, double *v, cudaStream_t st)
{
    if (c.L < 2) return;
    Col t = c;
    t.Kzz = Kzz;
    t.u = u;
    t.v = v;
    count_launches(1);
    k_transport<<<nblocks((long long)(c.L - 1) * c.S), kThreads, 0, st>>>(t);
}

void launch_grid(const Col &c, cudaStream_t st)
{
    count_launches(1); k_grid<<<1, 256, 0, st>>>(c);
    if (c.L > 1) { count_launches(1); k_transport<<<nblocks((long long)(c.L - 1) * c.S), kThreads, 0, st>>>(c); }
    if ((long long)c.L * c.S > 0) { count_launches(1); k_transport_rows<<<nblocks((long long)c.L * c.S), kThreads, 0, st>>>(c); }
}

void launch_thermo(const Col &c, cudaStream_t st)
{
    if (((long long)c.L * c.S) > 0) { count_launches(1); k_gibbs<<<nblocks((long long)c.L * c.S), kThreads, 0, st>>>(c); }
}

void launch_rates(const Col &c, cudaStream_t st)
{
    if (((long long)c.L * c.S) > 0) { count_launches(1); k_gibbs<<<nblocks((long long)c.L * c.S), kThreads, 0, st>>>(c); }
    if (((long long)c.L * c.R) > 0) { count_launches(1); k_rates<<<nblocks((long long)c.L * c.R), kThreads, 0, st>>>(c); }
}

void launch_photolysis(const Col &c, const double *n, cudaStream_t st, bool ordered)
{
    if (c.Rph == 0) return;
    if (c.W > 0) {
        if (c.L > 0) {
            count_launches(1);
            dim3 grid(nblocks(c.W, 128), (c.L + kExtLayers - 1) / kExtLayers);
            k_photo_alpha<<<grid, 128, 0, st>>>(c, n);
        }
        count_launches(1);
        if (c.diffuse) {
            k_photo_layers<<<nblocks(c.W, 32), 32 * kPhotoRuns, 0, st>>>(c);
            count_launches(1);
            k_photo_diffuse<<<nblocks(c.W, 32), 32, 0, st>>>(c);
        } else k_photo_J_direct<<<nblocks((long long)c.W * 32, 128), 128, 0, st>>>(c);
    }
    if (ordered && c.L > 0) {
        count_launches(1);
        k_photo_k_ordered<<<nblocks((long long)c.L * c.Rph * 32), kThreads, 0, st>>>(c);
    } else if (c.L > 0) {
        // layers to a tile: those that leave the fullest SM the least to do, a tile's folding and loads
        // counted as half a layer
        const auto tiles = [&](int kt) { return (long long)((c.L + kt - 1) / kt) * ((c.Rph + kPhotoQ - 1) / kPhotoQ); };
        const auto cost = [&](int kt) { return (double)((tiles(kt) + 151) / 152) * (kt + 0.5); };
        int kt = 2;
        for (int t = 3; t <= 5; ++t)
            if (cost(t) < cost(kt)) kt = t;
        count_launches(1);
        const int nt = (int)tiles(kt);
        if (kt == 2) k_photo_k<2><<<nt, 128, 0, st>>>(c);
        else if (kt == 3) k_photo_k<3><<<nt, 128, 0, st>>>(c);
        else if (kt == 4) k_photo_k<4><<<nt, 128, 0, st>>>(c);
        else k_photo_k<5><<<nt, 128, 0, st>>>(c);
    }
}

void launch_layer_terms(const Col &c, const double *n, double *F, const Ctl *ctl, double f_floor, double *diag,
                        double *bhat, cudaStream_t st)
{
    if ((long long)c.L * c.S <= 0) return;
    const bool rates = jv_rates_in_smem(c);
    const size_t sm = jv_smem_doubles(c, rates) * sizeof(double);
    allow_smem(k_layer_terms, kJvSmemMax);
    count_launches(1);
    k_layer_terms<<<std::min(c.L, kGatedBlocks), 512, sm, st>>>(c, n, F, ctl, f_floor, diag, bhat, rates ? 1 : 0);
}

// Blocks of few items each, the longest rows in the first: the hardware's order of them evens out what
// rows of unequal length leave (1,216 blocks of three to an SM end in a third of a wave).
constexpr long long kJacBlocks = 152 * 24;

template <typename T>
static void launch_jacobian_t(const Col &c, const Ctl *ctl, double dt_override, int scaled, T *A, T *lo, T *up,
                              cudaStream_t st, const int *skip, long long lstride)
{
    if ((long long)c.L * c.S <= 0) return;
    const size_t sm = sizeof(double) * ((size_t)kJacHeavyOcc * 6 + c.S) + sizeof(T) * (size_t)kJacWarps * c.S;
    cudaFuncSetAttribute(k_jacobian<T>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
    const long long items = (long long)c.nji * c.L;
    count_launches(1);
    k_jacobian<T><<<(int)std::min<long long>(items, kJacBlocks), kJacWarps * 32, sm, st>>>(c, ctl, dt_override, scaled, A, lo,
                                                                                         up, skip, lstride);
}

void launch_jacobian64(const Col &c, const Ctl *ctl, double dt_override, int scaled, double *A, double *lo, double *up,
                       cudaStream_t st, const int *skip)
{
    launch_jacobian_t<double>(c, ctl, dt_override, scaled, A, lo, up, st, skip, 0);
}

void launch_jacobian32(const Col &c, const Ctl *ctl, float *A, float *lo, float *up, cudaStream_t st, const int *skip,
                       long long lstride)
{
    launch_jacobian_t<float>(c, ctl, 0.0, 1, A, lo, up, st, skip, lstride);
}

void launch_jv(const Col &c, const Ctl *ctl, const double *xs, double *ys, const double *rowdiv, const int *skip,
               cudaStream_t st)
{
    if ((long long)c.L * c.S <= 0) return;
    if (c.photo_jac) {
        count_launches(3);
        dim3 grid(nblocks(c.W, 128), (c.L + kExtLayers - 1) / kExtLayers);
        k_photo_beta<<<grid, 128, 0, st>>>(c, ctl, xs, skip);
        k_photo_dJ<<<nblocks((long long)c.W * 32, 128), 128, 0, st>>>(c, ctl, skip);
        k_photo_dk<<<nblocks((long long)c.L * c.Rph * 32), kThreads, 0, st>>>(c, ctl, skip);
    }
    const bool rates = jv_rates_in_smem(c);
    const size_t sm = jv_smem_doubles(c, rates) * sizeof(double);
    allow_smem(k_jv_layer, kJvSmemMax);
    count_launches(1);
    k_jv_layer<<<std::min(c.L, kGatedBlocks), 512, sm, st>>>(c, ctl, xs, ys, rowdiv, skip, rates ? 1 : 0);
}

void launch_unscale(const Col &c, const double *xs, double *delta, cudaStream_t st)
{
    if (((long long)c.L * c.S) > 0) { count_launches(1); k_unscale<<<nblocks((long long)c.L * c.S), kThreads, 0, st>>>(c, xs, delta); }
}

void launch_check(const Col &c, Ctl *ctl, const Policy &pol, cudaStream_t st)
{
    if (((long long)c.L * c.S) > 0) { count_launches(1); k_check<<<nblocks((long long)c.L * c.S), kThreads, 0, st>>>(c, ctl, pol); }
}

void launch_decide(const Col &c, Ctl *ctl, const Policy &pol, cudaStream_t st)
{
    (void)c;
    count_launches(1); k_decide<<<1, 1, 0, st>>>(ctl, pol);
}

void launch_apply(const Col &c, Ctl *ctl, cudaStream_t st)
{
    if (((long long)c.L * c.S) > 0) { count_launches(1); k_apply<<<nblocks((long long)c.L * c.S), kThreads, 0, st>>>(c, ctl); }
}

void launch_reuse_scales(long long N, const double *rowd, const double *s, const double *s64, double *pin, double *pout,
                         const Ctl *ctl, cudaStream_t st)
{
    count_launches(1);
    k_reuse_scales<<<nblocks(N), kThreads, 0, st>>>(N, rowd, s, s64, pin, pout, ctl);
}

void launch_after_refactor(long long N, const double *s, double *s64, Ctl *ctl, cudaStream_t st)
{
    count_launches(1);
    k_after_refactor<<<nblocks(N), kThreads, 0, st>>>(N, s, s64, ctl);
}

void launch_route(Ctl *ctl, cudaStream_t st)
{
    count_launches(1);
    k_route<<<1, 1, 0, st>>>(ctl);
}

void launch_begin(Ctl *ctl, cudaStream_t st)
{
    count_launches(1);
    k_begin<<<1, 1, 0, st>>>(ctl);
}

}  // namespace xk

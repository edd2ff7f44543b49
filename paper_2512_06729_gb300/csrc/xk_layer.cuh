// Per-layer device code shared by the kernels that give a layer to one CTA.
#pragma once

#include "xk_internal.cuh"

namespace xk {

// v or -v by flipping the sign bit: a negation on the FP64 unit would cost as much as an addition
// (this part issues about two FP64 operations per clock and SM).
__device__ __forceinline__ double signed_by(double v, bool plus)
{
    return __hiloint2double(__double2hiint(v) ^ (plus ? 0 : (int)0x80000000), __double2loint(v));
}

// Species sums of one layer over its reactions: for every species, the sum over its entries of
// +val[reaction] for reactant entries and -val[reaction] for product entries.  Each lane sums one
// sublist serially (Col::sgp): FP64 additions are what this costs, so there are as few as entries,
// none for padding lanes of a warp-wide tree.  The caller adds a species' parts in order
// (species_sum) after a block barrier: every sum has a fixed order.
__device__ __forceinline__ void species_parts(const Col &c, const double *val, double *part)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    for (int g = warp; g < c.nsg; g += nw) {
        double acc = 0.0;
        const int q1 = c.sgp[g + 1];
#pragma unroll 4
        for (int q = c.sgp[g]; q < q1; ++q) {
            const int code = c.sent[32 * q + lane];
            if (code >= 0) acc += signed_by(val[code >> 1], code & 1);
        }
        const int to = c.spart[32 * g + lane];
        if (to >= 0) part[to] = acc;
    }
}

__device__ __forceinline__ double species_sum(const Col &c, const double *part, int i)
{
    double acc = 0.0;
    for (int q = c.ssp[i]; q < c.ssp[i + 1]; ++q) acc += part[q];
    return acc;
}

// the photolysis rate's extra change along v (0 unless photo_jacobian): dk_ph n_A
__device__ __forceinline__ double photo_jv_term(const Col &c, int k, int r)
{
    if (!c.photo_jac || c.rtype[r] != XK_RX_PHOTO) return 0.0;
    return c.pdk[(long long)k * c.Rph + c.prow[r]] * c.n[(long long)k * c.S + c.reac[3 * r]];
}

// Doubles of shared memory that jv_layer_body needs: v = s x of the layer,
// the partial sums, and the rates' changes where they fit (otherwise they go through c.dw).
__host__ __device__ inline size_t jv_smem_doubles(const Col &c, bool rates)
{
    return (size_t)c.S + 1 + (size_t)c.nsub + (rates ? (size_t)c.R : 0);
}

// The rates' changes stay in shared memory up to this size of everything together (R about 20,000);
// larger networks take them through c.dw, written and read by the same CTA.
constexpr size_t kJvSmemMax = 200 * 1024;
__host__ inline bool jv_rates_in_smem(const Col &c) { return jv_smem_doubles(c, true) * sizeof(double) <= kJvSmemMax; }

// Layer k of y = diag(1/s) (I/dt - J) diag(s) x (rows divided by rowdiv when given), by one CTA,
// matrix-free from the reaction derivatives d: first the change of every rate along v = s x (six
// derivatives per reaction, three 16-byte loads, and gathers of v from shared memory), then the
// species sums from shared memory, then transport.  Bound by the read of d (48 bytes per reaction
// and layer).  Ends with every thread's rows written; sm must not be reused before a barrier.
__device__ __forceinline__ void jv_layer_body(const Col &c, const Ctl *ctl, const double *x, double *y,
                                              const double *rowdiv, int k, double *sm, bool rates_in_smem)
{
    const int S = c.S, R = c.R, L = c.L;
    double *sx = sm, *part = sx + S + 1, *dws = rates_in_smem ? part + c.nsub : c.dw + (long long)k * R;
    const long long row0 = (long long)k * S;
    for (int i = threadIdx.x; i < S; i += blockDim.x) sx[i] = c.s[row0 + i] * x[row0 + i];
    __syncthreads();
    const double2 *dk = (const double2 *)(c.d + (long long)k * R * 6);
    // four reactions per thread at a time, all their loads before the first use
    for (int r0 = threadIdx.x; r0 < R; r0 += 4 * blockDim.x) {
        uint4 q[4];
        double2 d01[4], d23[4], d45[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const int r = min(r0 + u * (int)blockDim.x, R - 1);
            q[u] = c.rx[r];
            d01[u] = dk[3 * r];
            d23[u] = dk[3 * r + 1];
            d45[u] = dk[3 * r + 2];
        }
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const int r = r0 + u * (int)blockDim.x;
            if (r >= R) break;
            // reactions of a kind stand together, so the slots a kind does not use are skipped by whole warps
            double acc = 0.0;
            auto slot = [&](double d, unsigned j) { if (j != (unsigned)S) acc += d * sx[j]; };
            slot(d01[u].x, q[u].x & 0xffffu);
            slot(d23[u].y, q[u].y >> 16);
            slot(d01[u].y, q[u].x >> 16);
            slot(d45[u].x, q[u].z & 0xffffu);
            slot(d23[u].x, q[u].y & 0xffffu);
            slot(d45[u].y, q[u].z >> 16);
            if (c.photo_jac) acc += photo_jv_term(c, k, r);
            dws[r] = acc;
        }
    }
    __syncthreads();
    species_parts(c, dws, part);
    __syncthreads();
    const double rdt = 1.0 / ctl->dt;
    for (int i = threadIdx.x; i < S; i += blockDim.x) {
        const long long q = row0 + i;
        const double ri = c.rs[q];
        double r = species_sum(c, part, i) * ri + (rdt + c.tdg[q]) * x[q];
        if (k > 0) r += c.tlo[q] * c.s[q - S] * ri * x[q - S];
        if (k + 1 < L) r += c.tup[q] * c.s[q + S] * ri * x[q + S];
        if (rowdiv) r /= rowdiv[q];
        y[q] = r;
    }
}

}  // namespace xk

// Block cyclic reduction (odd-even elimination of layers) of the block-tridiagonal
// system (I/dt - J) x = b, in FP32 on the tensor cores: the mixed path's
// preconditioner, a block LU of the system with its layers ordered odd before
// even, level by level.
//
// Rows of the system: L_k x_{k-1} + D_k x_k + U_k x_{k+1} = b_k.  At each level the
// layers at odd positions j of the current list are eliminated:
//   x_j = D_j^-1 (b_j - L_j x_{j-1} - U_j x_{j+1});
// each kept neighbour i takes the Schur complement
//   D_i <- D_i - L_i Q_l - U_i P_r,  P = D^-1 L,  Q = D^-1 U,
// and couples to the next kept layers through L_i <- -L_i P_l, U_i <- -U_i Q_r.
// At level 0 the couplings are the diagonal transport terms, so the updates are
// element-wise; from level 1 on they are dense S x S blocks and every update is a
// product on the tensor cores (xk_tc.cu), batched over the layers of the level.
// The inverses D_j^-1 come from a recursive 2 x 2 block inversion (Schur
// complement of the leading block), whose products are batched the same way,
// down to blocks of at most 160 rows inverted by one CTA each (Gauss-Jordan
// with partial pivoting).  The work per factorization is about 4x that of
// block Thomas, but instead of a chain of L dependent inversions there are
// about log2(L) levels, each filling the GPU.
//
// Blocks are padded to Sp = round_up(S, 32) rows and columns with the identity
// in the padding, so that every product has dimensions that are multiples of 32.
#include <cuda_runtime.h>

#include <stdint.h>

#include <algorithm>

#include "xk_bcr.cuh"

namespace xk {

namespace {

constexpr int kArrD = 0, kArrINV = 1, kArrTMP = 2, kArrCP = 3, kArrPQ = 4, kArrays = 5;

__device__ __forceinline__ bool stop(const int *skip, const Ctl *ctl)
{
    return (ctl && (ctl->finished || ctl->err_timeout)) || (skip && *skip);
}

// Leading (upper-left) part of a block of n rows in the recursive inversion: a multiple of 32.
int split_of(int n) { return 32 * ((n + 63) / 64); }

// ---------------------------------------------------------------------------
// Gauss-Jordan inversion with partial pivoting of one N x N block per CTA
// (N = 32 RG <= 160), in panels of 8 columns with look-ahead.  Pivoting is
// implicit: rows never move; the pivot of column c is the unused row p(c) of
// largest |value|, and the in-place elimination leaves row p(k) holding row k
// of (P M)^-1, so M^-1[k][p(c)] = W[p(k)][c].
//
// Warps 0 .. RG-1 factor the panels, a row per lane with its 8 entries in
// registers.  A column costs a warp reduction (the warp's best row), a barrier
// among these warps (each leaves its best row, already scaled, in shared
// memory) and 8 FMAs.  The result G (N x 8) turns the other columns by one
// rank-8 update,
//   W[r][j] <- W[r][j] + sum_l G[r][l] U[l][j],   U the panel's pivot rows,
// (the pivot rows themselves without their old value), which the other warps
// apply one panel behind, in registers: a warp owns quads of columns (all of
// their rows) and writes them to the block's image in shared memory after each
// update, where it then reads the next panel's pivot rows; a quad belongs to one
// panel, and the only block barrier is one per panel.  The panel warps apply the
// previous panel's update to their next panel themselves.  Panels travel through
// the block's image in shared memory (row stride N + 4: rows are read 16 bytes a
// lane without conflicts), G also with every value twice, as the packed FMAs
// (two columns to an instruction) want it.
//
// What bounds it: the chain of N dependent columns, then the issue slots of the
// updates (2 N^3 flop on one SM's FP32 pipe).  The loop over a panel's columns is
// rolled and no branch depends on where the pivot is: with a jump per pivot row
// a column took 720 clocks, 300 of them there, and with all of the panel's rows
// on one warp 400, most of them selects.  The panel is 8 wide because 16 doubles
// the panel warps' work per column and 4 doubles the updates' loads and stores.
// ---------------------------------------------------------------------------
constexpr int kLeafPanel = 8;
constexpr int kLeafThreads = 512;
constexpr int leaf_trail(int RG) { return kLeafThreads / 32 - RG; }                 // warps of the trailing update
constexpr int leaf_quads(int RG) { return (8 * RG + leaf_trail(RG) - 1) / leaf_trail(RG); }   // of one warp, at most
constexpr int kLeafGd = 20;                                  // row stride of the doubled G
// the block (row stride N + 4) with room for the quads past its end, two panels' doubled G
constexpr size_t leaf_smem(int RG)
{
    return sizeof(float) * ((size_t)32 * RG * (32 * RG + 4) + 2 * 32 * RG * kLeafGd);
}

// A predicated store: which of a lane's rows is the pivot is known at run time only, and a branch
// per candidate (or a jump table) costs a few hundred clocks each time.
__device__ __forceinline__ void store4_if(bool p, float *dst, float4 v)
{
    asm volatile("{\n\t.reg .pred q;\n\tsetp.ne.b32 q, %0, 0;\n\t@q st.shared.v4.f32 [%1], {%2, %3, %4, %5};\n\t}"
                 ::"r"((int)p), "r"((uint32_t)__cvta_generic_to_shared(dst)), "f"(v.x), "f"(v.y), "f"(v.z), "f"(v.w)
                 : "memory");
}

// Two FMAs (products) in one instruction, on both halves.
__device__ __forceinline__ void fma2(float2 &d, float2 a, float2 b)
{
    unsigned long long &dd = reinterpret_cast<unsigned long long &>(d);
    asm("fma.rn.f32x2 %0, %1, %2, %0;"
        : "+l"(dd)
        : "l"(reinterpret_cast<unsigned long long &>(a)), "l"(reinterpret_cast<unsigned long long &>(b)));
}
__device__ __forceinline__ void mul2(float2 &d, float2 a)
{
    unsigned long long &dd = reinterpret_cast<unsigned long long &>(d);
    asm("mul.rn.f32x2 %0, %0, %1;" : "+l"(dd) : "l"(reinterpret_cast<unsigned long long &>(a)));
}

struct __align__(16) LeafCand {
    float row[kLeafPanel];        // 1 / pivot, then the rest of the row times it
};

template <int RG>
__global__ void __launch_bounds__(kLeafThreads, 1) k_leaf_inverse(const BcrLeaf *tasks, const int *skip, const Ctl *ctl)
{
    constexpr int N = 32 * RG, NP = kLeafPanel, NPAN = N / NP, LD = N + 4, TW = leaf_trail(RG), NQ = leaf_quads(RG);
    extern __shared__ __align__(16) float sm[];
    float *tile = sm;                          // [N][LD]
    float *Gd = tile + N * LD;                 // [2][N][kLeafGd]
    __shared__ LeafCand cand[2][RG];
    __shared__ __align__(16) unsigned keys[2][8];
    __shared__ int piv[2][NP], perm[N];
    const int ln = threadIdx.x & 31, wv = threadIdx.x >> 5;
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    const BcrLeaf t = tasks[blockIdx.x];
    if (threadIdx.x < 16) keys[threadIdx.x >> 3][threadIdx.x & 7] = 0u;
    asm volatile("griddepcontrol.wait;" ::: "memory");
    if (stop(skip, ctl)) return;
#pragma unroll 10
    for (int e = threadIdx.x; e < N * N; e += kLeafThreads) {
        const int r = e / N, j = e - r * N;
        tile[r * LD + j] = t.in[(long long)r * t.ldin + j];
    }
    __syncthreads();
    if (wv < RG) {
        const int me = 32 * wv + ln;                       // this lane's row
        unsigned live = 0x7fffff00u, code = 255u - me;     // of the pivot search: zero once the row has been a pivot
        bool last = false;                                 // a pivot of the previous panel
        float2 g[NP];                                      // the row of the previous panel's G, doubled
        for (int p = 0; p < NPAN; ++p) {
            float *at = tile + me * LD + p * NP;
            float x[NP];
            {
                const float4 v0 = *(const float4 *)at, v1 = *(const float4 *)(at + 4);
                float2 xx[4] = {{v0.x, v0.y}, {v0.z, v0.w}, {v1.x, v1.y}, {v1.z, v1.w}};
                if (p > 0) {
                    if (last) xx[0] = xx[1] = xx[2] = xx[3] = float2{0.f, 0.f};
                    const int *pp = piv[(p - 1) & 1];
#pragma unroll
                    for (int l = 0; l < NP; ++l) {
                        const float *ur = tile + pp[l] * LD + p * NP;
                        const float4 u0 = *(const float4 *)ur, u1 = *(const float4 *)(ur + 4);
                        fma2(xx[0], g[l], float2{u0.x, u0.y});
                        fma2(xx[1], g[l], float2{u0.z, u0.w});
                        fma2(xx[2], g[l], float2{u1.x, u1.y});
                        fma2(xx[3], g[l], float2{u1.z, u1.w});
                    }
                }
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    x[2 * j] = xx[j].x;
                    x[2 * j + 1] = xx[j].y;
                }
            }
            last = false;
            // column c is always x[0]: each step shifts the others down one and puts the finished column
            // last, so that after eight steps they are in their places again
#pragma unroll 1
            for (int c = 0; c < NP; ++c) {
                // pivot: the unused row of largest |value| (its float bits without the low eight, which
                // hold the row so that one reduction finds both; the lowest row among near-equals)
                const unsigned k = (__float_as_uint(x[0]) & live) | code;
                unsigned top = __reduce_max_sync(0xffffffffu, k);
                // meanwhile this lane's own row, scaled (a singular block: the FP64 Krylov solve sees a
                // poor preconditioner)
                float s[NP];
                s[0] = reciprocal32(x[0] == 0.0f ? 1e-30f : x[0]);
#pragma unroll
                for (int j = 1; j < NP; ++j) s[j] = x[j] * s[0];
                LeafCand *cb = cand[c & 1];
                const bool best = k == top;
                store4_if(best, cb[wv].row, make_float4(s[0], s[1], s[2], s[3]));
                store4_if(best, cb[wv].row + 4, make_float4(s[4], s[5], s[6], s[7]));
                if (RG > 1) {
                    if (ln == 0) keys[c & 1][wv] = top;
                    asm volatile("bar.sync 1, %0;" ::"n"(32 * RG) : "memory");
                    const uint4 k0 = *(const uint4 *)keys[c & 1];
                    top = max(max(k0.x, k0.y), max(k0.z, k0.w));
                    if (RG > 4) top = max(top, keys[c & 1][4]);
                } else {
                    __syncwarp();
                }
                const int row = 255 - (int)(top & 0xffu);
                const float4 r0 = *(const float4 *)cb[row >> 5].row, r1 = *(const float4 *)(cb[row >> 5].row + 4);
                const float pr[NP] = {r0.x, r0.y, r0.z, r0.w, r1.x, r1.y, r1.z, r1.w};
                const bool is = k == top;                  // the pivot row becomes the scaled row
                const float f = x[0];
#pragma unroll
                for (int j = 1; j < NP; ++j) {
                    const float v = fmaf(-f, pr[j], x[j]);
                    x[j - 1] = is ? s[j] : v;
                }
                x[NP - 1] = is ? s[0] : -f * pr[0];
                if (is) {
                    live = code = 0u;
                    last = true;
                    piv[p & 1][c] = row;
                    perm[p * NP + c] = row;
                }
            }
            *(float4 *)at = make_float4(x[0], x[1], x[2], x[3]);
            *(float4 *)(at + 4) = make_float4(x[4], x[5], x[6], x[7]);
            float *gd = Gd + ((p & 1) * N + me) * kLeafGd;
#pragma unroll
            for (int j = 0; j < NP; j += 2) *(float4 *)(gd + 2 * j) = make_float4(x[j], x[j], x[j + 1], x[j + 1]);
#pragma unroll
            for (int j = 0; j < NP; ++j) g[j] = float2{x[j], x[j]};
            __syncthreads();
        }
        __syncthreads();
    } else {
        const int tw = wv - RG;
        float2 w[NQ][RG][2];                   // this warp's quads tw + TW i: rows ln + 32 a
#pragma unroll
        for (int i = 0; i < NQ; ++i) {
            const int q = tw + TW * i;
#pragma unroll
            for (int a = 0; a < RG; ++a) {
                const float4 v = q < N / 4 ? *(const float4 *)(tile + (ln + 32 * a) * LD + 4 * q) : make_float4(0.f, 0.f, 0.f, 0.f);
                w[i][a][0] = float2{v.x, v.y};
                w[i][a][1] = float2{v.z, v.w};
            }
        }
        __syncthreads();
        for (int p = 1; p <= NPAN; ++p) {      // panel p - 1 is done; the panel warps are at panel p
            const int *pp = piv[(p - 1) & 1];
            unsigned mine = 0;                 // bit a: row ln + 32 a is a pivot row of the panel
#pragma unroll
            for (int l = 0; l < NP; ++l) mine |= ln == (pp[l] & 31) ? 1u << (pp[l] >> 5) : 0u;
            // the pivot rows start from zero in the update
#pragma unroll
            for (int a = 0; a < RG; ++a) {
                const float z = (mine >> a) & 1u ? 0.0f : 1.0f;
#pragma unroll
                for (int i = 0; i < NQ; ++i) {
                    mul2(w[i][a][0], float2{z, z});
                    mul2(w[i][a][1], float2{z, z});
                }
            }
            const float *gp = Gd + (((p - 1) & 1) * N + ln) * kLeafGd;
#pragma unroll
            for (int h = 0; h < 4; ++h) {      // two of the panel's columns at a time
                float4 g4[RG];
#pragma unroll
                for (int a = 0; a < RG; ++a) g4[a] = *(const float4 *)(gp + 32 * a * kLeafGd + 4 * h);
#pragma unroll
                for (int l = 0; l < 2; ++l) {
                    const float *ur = tile + pp[2 * h + l] * LD + 4 * tw;      // the pivot row as it was
#pragma unroll
                    for (int i = 0; i < NQ; ++i) {
                        const float4 u = *(const float4 *)(ur + 4 * TW * i);
#pragma unroll
                        for (int a = 0; a < RG; ++a) {
                            const float2 gl = l == 0 ? float2{g4[a].x, g4[a].y} : float2{g4[a].z, g4[a].w};
                            fma2(w[i][a][0], gl, float2{u.x, u.y});
                            fma2(w[i][a][1], gl, float2{u.z, u.w});
                        }
                    }
                }
            }
            __syncwarp();                      // every lane has read the pivot rows
            // the tile follows: the next panel's pivot rows are read there, and the panel warps read
            // their panels there.  The quads of panel p - 1 are G already; those of panel p are theirs
#pragma unroll
            for (int i = 0; i < NQ; ++i) {
                const int q = tw + TW * i, pq = q / (NP / 4);
                float *at = tile + ln * LD + 4 * q;
                if (q < N / 4 && pq == p - 1) {
#pragma unroll
                    for (int a = 0; a < RG; ++a) {
                        const float4 v = *(const float4 *)(at + 32 * a * LD);
                        w[i][a][0] = float2{v.x, v.y};
                        w[i][a][1] = float2{v.z, v.w};
                    }
                } else if (q < N / 4 && pq != p) {
#pragma unroll
                    for (int a = 0; a < RG; ++a)
                        *(float4 *)(at + 32 * a * LD) = make_float4(w[i][a][0].x, w[i][a][0].y, w[i][a][1].x, w[i][a][1].y);
                }
            }
            __syncthreads();
        }
        // M^-1[k][p(c)] = W[p(k)][c]: columns permuted here, rows on the way out
#pragma unroll
        for (int i = 0; i < NQ; ++i) {
            const int q = tw + TW * i;
            if (q < N / 4) {
                const int c0 = perm[4 * q], c1 = perm[4 * q + 1], c2 = perm[4 * q + 2], c3 = perm[4 * q + 3];
#pragma unroll
                for (int a = 0; a < RG; ++a) {
                    float *at = tile + (ln + 32 * a) * LD;
                    at[c0] = w[i][a][0].x;
                    at[c1] = w[i][a][0].y;
                    at[c2] = w[i][a][1].x;
                    at[c3] = w[i][a][1].y;
                }
            }
        }
    }
    __syncthreads();
#pragma unroll 10
    for (int e = threadIdx.x; e < N * N; e += kLeafThreads) {
        const int k = e / N, j = e - k * N;
        t.out[(long long)k * t.ldout + j] = tile[perm[k] * LD + j];
    }
}

template <int RG>
cudaError_t launch_leaf_rg(const BcrLeaf *tasks, int count, const int *skip, const Ctl *ctl, cudaStream_t st)
{
    constexpr size_t smem = leaf_smem(RG);
    const cudaError_t e = allow_smem(k_leaf_inverse<RG>, smem);
    if (e != cudaSuccess) return e;
    count_launches(1);
    return launch_dependent(k_leaf_inverse<RG>, dim3(count), dim3(kLeafThreads), smem, st, tasks, skip, ctl);
}

// One CTA per block; every block of a launch has the same n, a multiple of 32 up to kBcrLeafMax.
cudaError_t launch_leaf(const BcrLeaf *tasks, int count, int n, const int *skip, const Ctl *ctl, cudaStream_t st)
{
    switch (n / 32) {
    case 1: return launch_leaf_rg<1>(tasks, count, skip, ctl, st);
    case 2: return launch_leaf_rg<2>(tasks, count, skip, ctl, st);
    case 3: return launch_leaf_rg<3>(tasks, count, skip, ctl, st);
    case 4: return launch_leaf_rg<4>(tasks, count, skip, ctl, st);
    case 5: return launch_leaf_rg<5>(tasks, count, skip, ctl, st);
    default: return cudaErrorInvalidValue;
    }
}

// Level 0 (diagonal couplings), for each kept even layer i with eliminated neighbours l = i-1, r = i+1:
//   D_i -= diag(lo_i) INV_l diag(up_l) + diag(up_i) INV_r diag(lo_r)
//   CP(1, i/2) = [ -diag(lo_i) INV_l diag(lo_l) | -diag(up_i) INV_r diag(up_r) ]
// Four columns to a thread.  Bound by memory: at 594 species x 150 layers 555 MB, 81 us at the copy
// rate if the second reading of each inverse comes from L2, and takes 98; entry by entry it took 221.
__global__ void __launch_bounds__(256) k_bcr_level0(float *D, const float *INV, float *CP, const float *lo,
                                                     const float *up, const int *kept, int L, int S, int Sp,
                                                     const int *skip, const Ctl *ctl)
{
    if (stop(skip, ctl)) return;
    const int i = kept[blockIdx.y], q = blockIdx.x * 256 + threadIdx.x, w4 = Sp / 4;
    if (q >= Sp * w4) return;
    const int y = q / w4, c = (q - y * w4) * 4;
    const long long blk = (long long)Sp * Sp, e = (long long)y * Sp + c;
    const bool hasl = i >= 1, hasr = i + 1 < L;
    float4 gl = make_float4(0, 0, 0, 0), gr = gl, d = *(const float4 *)(D + i * blk + e);
    if (hasl) gl = *(const float4 *)(INV + (i - 1) * blk + e);
    if (hasr) gr = *(const float4 *)(INV + (i + 1) * blk + e);
    const float loi = (hasl && y < S) ? lo[(long long)i * S + y] : 0.0f;
    const float upi = (hasr && y < S) ? up[(long long)i * S + y] : 0.0f;
    auto at = [&](const float *a, int k, int j) { return c + j < S ? a[(long long)k * S + c + j] : 0.0f; };
    float *cp = CP + (long long)(i / 2) * Sp * 2 * Sp + (long long)y * 2 * Sp + c;
    float upd[4] = {0.0f, 0.0f, 0.0f, 0.0f}, o[4];
    if (hasl) {
        const float g[4] = {gl.x, gl.y, gl.z, gl.w};
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            upd[j] += loi * g[j] * at(up, i - 1, j);
            o[j] = -loi * g[j] * at(lo, i - 1, j);
        }
        if (i >= 2) *(float4 *)cp = make_float4(o[0], o[1], o[2], o[3]);
    }
    if (hasr) {
        const float g[4] = {gr.x, gr.y, gr.z, gr.w};
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            upd[j] += upi * g[j] * at(lo, i + 1, j);
            o[j] = -upi * g[j] * at(up, i + 1, j);
        }
        if (i + 2 <= L - 1) *(float4 *)(cp + Sp) = make_float4(o[0], o[1], o[2], o[3]);
    }
    d.x -= upd[0];
    d.y -= upd[1];
    d.z -= upd[2];
    d.w -= upd[3];
    *(float4 *)(D + i * blk + e) = d;
}

__global__ void k_bcr_pad(float *D, int L, int S, int Sp)
{
    const long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    const int padr = Sp - S;
    if (padr <= 0 || e >= (long long)L * padr * Sp) return;
    const int k = (int)(e / ((long long)padr * Sp));
    const long long rem = e - (long long)k * padr * Sp;
    const int y = S + (int)(rem / Sp), c = (int)(rem % Sp);
    D[((long long)k * Sp + y) * Sp + c] = (c == y) ? 1.0f : 0.0f;
}

unsigned nblk(long long n, int t) { return (unsigned)((n + t - 1) / t); }

// ---------------------------------------------------------------------------
// Host: the plan (stages of task lists), built from the layer structure alone.
// ---------------------------------------------------------------------------
struct View {
    int arr, r0, c0;
};

struct Builder {
    BcrPlan &p;
    int L, S, Sp;
    std::vector<int> depth_col;

    int cols(int arr) const
    {
        switch (arr) {
        case kArrD: case kArrINV: return Sp;
        case kArrTMP: return p.Wt;
        default: return 2 * Sp;
        }
    }
    float *base(int arr) const
    {
        switch (arr) {
        case kArrD: return p.D;
        case kArrINV: return p.INV;
        case kArrTMP: return p.TMP;
        case kArrCP: return p.CP;
        default: return p.PQ;
        }
    }
    float *ptr(int arr, int z, int r, int c) const
    {
        float *b = base(arr);
        if (!b) return nullptr;
        return b + ((size_t)z * Sp + r) * (size_t)cols(arr) + c;
    }
    TcOut out(int arr, int z, int r, int c, float alpha, float beta, int n, bool accumulate) const
    {
        TcOut o;
        o.ptr = ptr(arr, z, r, c);
        o.src = accumulate ? o.ptr : nullptr;
        o.ld = o.lds = cols(arr);
        o.alpha = alpha;
        o.beta = accumulate ? beta : 0.0f;
        o.n = n;
        return o;
    }
    // one product task C = A B: A (m x k) at (ai, az, ar, ac), B (k x n) at (bi, bz, br, bc)
    static TcTask product(int m, int n, int k, View a, int az, View b, int bz, TcOut o)
    {
        TcTask t{};
        t.nseg = 1;
        t.seg[0] = TcSeg{a.arr, a.c0, a.r0, az, b.arr, b.c0, b.r0, bz, k};
        t.nout = 1;
        t.out[0] = o;
        t.m = m;
        t.n = n;
        return t;
    }
    void gemm_stage(std::vector<TcTask> &ts, int level)
    {
        if (ts.empty()) return;
        BcrStage s{kBcrGemm, (int)p.gemm.size(), (int)ts.size(), (int)p.tile_task.size(),
                   tc_number_tiles(ts.data(), (int)ts.size()), level};
        for (int q = 0; q < (int)ts.size(); ++q) p.tile_task.insert(p.tile_task.end(), ts[q].tiles, q);
        p.gemm.insert(p.gemm.end(), ts.begin(), ts.end());
        p.fac.push_back(s);
    }
    // Widths of the temporaries at each recursion depth: X (h x r), Y (r x h), Sc (r x r) side by side.
    void widths(int n, int d, std::vector<int> &w) const
    {
        if (n <= kBcrLeafMax) return;
        const int h = split_of(n), r = n - h;
        if ((int)w.size() <= d) w.resize(d + 1, 0);
        w[d] = std::max(w[d], 2 * r + h);
        widths(h, d + 1, w);
        widths(r, d + 1, w);
    }
    // Inverse of the n x n blocks in (layer zin[b]) into out (layer zout[b]); temporaries in TMP layer b.
    void inverse(int n, View in, const std::vector<int> &zin, View out, const std::vector<int> &zout, int d, int level)
    {
        const int B = (int)zin.size();
        if (n <= kBcrLeafMax) {
            BcrStage s{kBcrLeafStage, (int)p.leaf.size(), B, 0, n, level};
            for (int b = 0; b < B; ++b)
                p.leaf.push_back(BcrLeaf{ptr(in.arr, zin[b], in.r0, in.c0), ptr(out.arr, zout[b], out.r0, out.c0),
                                         cols(in.arr), cols(out.arr), n});
            p.fac.push_back(s);
            return;
        }
        const int h = split_of(n), r = n - h, cd = depth_col[d];
        const View A{in.arr, in.r0, in.c0}, Bv{in.arr, in.r0, in.c0 + h}, Cv{in.arr, in.r0 + h, in.c0},
            Dv{in.arr, in.r0 + h, in.c0 + h};
        const View TL{out.arr, out.r0, out.c0}, TR{out.arr, out.r0, out.c0 + h}, BL{out.arr, out.r0 + h, out.c0},
            BR{out.arr, out.r0 + h, out.c0 + h};
        const View X{kArrTMP, 0, cd}, Y{kArrTMP, 0, cd + r}, Sc{kArrTMP, 0, cd + r + h};
        std::vector<int> zt(B);
        for (int b = 0; b < B; ++b) zt[b] = b;
        // 1. A^-1 into TL
        inverse(h, A, zin, TL, zout, d + 1, level);
        std::vector<TcTask> ts;
        // 2. X = A^-1 B, Y = C A^-1
        for (int b = 0; b < B; ++b) {
            ts.push_back(product(h, r, h, TL, zout[b], Bv, zin[b], out_of(X, b, 1.0f, 0.0f, r, false)));
            ts.push_back(product(r, h, h, Cv, zin[b], TL, zout[b], out_of(Y, b, 1.0f, 0.0f, h, false)));
        }
        gemm_stage(ts, level);
        ts.clear();
        // 3. Sc = D - C X
        for (int b = 0; b < B; ++b) {
            TcTask t = product(r, r, h, Cv, zin[b], X, zt[b], out_of(Sc, b, -1.0f, 1.0f, r, false));
            t.out[0].src = ptr(Dv.arr, zin[b], Dv.r0, Dv.c0);
            t.out[0].lds = cols(Dv.arr);
            t.out[0].beta = 1.0f;
            ts.push_back(t);
        }
        gemm_stage(ts, level);
        ts.clear();
        // 4. Sc^-1 into BR
        inverse(r, Sc, zt, BR, zout, d + 1, level);
        // 5. TR = -X Sc^-1, BL = -Sc^-1 Y
        for (int b = 0; b < B; ++b) {
            ts.push_back(product(h, r, r, X, zt[b], BR, zout[b], out_view(TR, zout[b], -1.0f, r)));
            ts.push_back(product(r, h, r, BR, zout[b], Y, zt[b], out_view(BL, zout[b], -1.0f, h)));
        }
        gemm_stage(ts, level);
        ts.clear();
        // 6. TL = A^-1 - X BL
        for (int b = 0; b < B; ++b) {
            TcTask t = product(h, h, r, X, zt[b], BL, zout[b], out_view(TL, zout[b], -1.0f, h));
            t.out[0].src = t.out[0].ptr;
            t.out[0].beta = 1.0f;
            ts.push_back(t);
        }
        gemm_stage(ts, level);
    }
    TcOut out_of(View v, int z, float alpha, float beta, int n, bool acc) const
    {
        return out(v.arr, z, v.r0, v.c0, alpha, beta, n, acc);
    }
    TcOut out_view(View v, int z, float alpha, int n) const { return out(v.arr, z, v.r0, v.c0, alpha, 0.0f, n, false); }

    void build()
    {
        std::vector<int> w;
        widths(Sp, 0, w);
        depth_col.assign(w.size() + 1, 0);
        for (size_t d = 0; d < w.size(); ++d) depth_col[d + 1] = depth_col[d] + w[d];
        p.Wt = std::max(32, (depth_col.back() + 31) / 32 * 32);
        const BcrLevels lv(L);
        const auto &lists = lv.lists;
        const auto &cp_off = lv.cp_off;
        p.levels = (int)lists.size() - 1;
        p.Ncp = std::max(lv.ncp, 1);
        int zt = 1;
        for (int l = 0; l < p.levels; ++l) zt = std::max(zt, (int)lists[l].size() / 2);
        p.Zt = zt;
        p.level0_kept.clear();
        for (int k = 0; k < L; k += 2) p.level0_kept.push_back(k);
        const View Dfull{kArrD, 0, 0}, Ifull{kArrINV, 0, 0};
        // factorization
        for (int l = 0; l < p.levels; ++l) {
            const auto &a = lists[l];
            std::vector<int> elim;
            for (size_t q = 1; q < a.size(); q += 2) elim.push_back(a[q]);
            inverse(Sp, Dfull, elim, Ifull, elim, 0, l);
            if (l == 0) {
                p.fac.push_back(BcrStage{kBcrLevel0, 0, (int)p.level0_kept.size(), 0, 0, 0});
                continue;
            }
            std::vector<TcTask> ts;
            // [P_j | Q_j] = D_j^-1 [L_j | U_j]
            for (size_t q = 1; q < a.size(); q += 2) {
                const int j = a[q];
                const bool right = q + 1 < a.size();
                const int n = right ? 2 * Sp : Sp;
                ts.push_back(product(Sp, n, Sp, Ifull, j, View{kArrCP, 0, 0}, cp_off[l] + (int)q,
                                     out(kArrPQ, j, 0, 0, 1.0f, 0.0f, n, false)));
            }
            gemm_stage(ts, l);
            ts.clear();
            // Schur complements and the couplings of the next level
            for (size_t q = 0; q < a.size(); q += 2) {
                const int i = a[q];
                const int cpi = cp_off[l] + (int)q;
                const bool hl = q >= 1, hr = q + 1 < a.size();
                if (!hl && !hr) continue;
                TcTask t{};
                t.nseg = 0;
                if (hr) t.seg[t.nseg++] = TcSeg{kArrCP, Sp, 0, cpi, kArrPQ, 0, 0, a[q + 1], Sp};       // U_i P_r
                if (hl) t.seg[t.nseg++] = TcSeg{kArrCP, 0, 0, cpi, kArrPQ, Sp, 0, a[q - 1], Sp};       // L_i Q_l
                t.nout = 1;
                t.out[0] = out(kArrD, i, 0, 0, -1.0f, 1.0f, Sp, true);
                t.m = Sp;
                t.n = Sp;
                ts.push_back(t);
                const int cpn = cp_off[l + 1] + (int)(q / 2);
                if (hl && q >= 2)       // L_i <- -L_i P_l
                    ts.push_back(product(Sp, Sp, Sp, View{kArrCP, 0, 0}, cpi, View{kArrPQ, 0, 0}, a[q - 1],
                                         out(kArrCP, cpn, 0, 0, -1.0f, 0.0f, Sp, false)));
                if (hr && q + 2 < a.size())   // U_i <- -U_i Q_r
                    ts.push_back(product(Sp, Sp, Sp, View{kArrCP, 0, Sp}, cpi, View{kArrPQ, 0, Sp}, a[q + 1],
                                         out(kArrCP, cpn, 0, Sp, -1.0f, 0.0f, Sp, false)));
            }
            gemm_stage(ts, l);
        }
        const int root = lists.back()[0];
        inverse(Sp, Dfull, std::vector<int>{root}, Ifull, std::vector<int>{root}, 0, p.levels);
        bcr_solve_tasks(lv, BcrArrays<float>{p.INV, p.CP, p.PQ, p.lo, p.up, p.bw, p.tw, p.xw, L, S, Sp, Sp}, p.mv, p.sol);
    }
};

}  // namespace

// Right-hand sides are read where they are first needed, and those of the layers kept at level 0 with
// the coupling terms to their eliminated neighbours taken off on the way.
template <typename T>
void bcr_solve_tasks(const BcrLevels &lv, const BcrArrays<T> &p, std::vector<BcrMvT<T>> &out, std::vector<BcrStage> &sol)
{
    using Mv = BcrMvT<T>;
    const auto &lists = lv.lists;
    const auto &cp_off = lv.cp_off;
    const int L = p.L, S = p.S, Sp = p.ld, levels = (int)lists.size() - 1, root = lists.back()[0];
    const size_t blk = (size_t)p.rows * Sp;
    // the lists are also sized before the arrays exist
    auto inv = [&](int k) { return p.INV ? p.INV + k * blk : nullptr; };
    auto cp = [&](int q, int c) { return p.CP ? p.CP + q * 2 * blk + c : nullptr; };
    auto pq = [&](int k) { return p.PQ ? p.PQ + k * 2 * blk : nullptr; };
    auto vec = [&](T *a, int k) { return a ? a + (size_t)k * Sp : nullptr; };
    auto row = [&](const T *a, int k) { return a ? a + (size_t)k * S : nullptr; };
    auto mv_stage = [&](std::vector<Mv> &ts, int level) {
        if (ts.empty()) return;
        sol.push_back(BcrStage{kBcrMv, (int)out.size(), (int)ts.size(), 0, 0, level});
        out.insert(out.end(), ts.begin(), ts.end());
    };
    auto rhs0 = [&](int i, int &layer, const T *&c0, const T *&w0, const T *&c1, const T *&w1) {
        layer = i;
        if (i >= 1) { c0 = row(p.lo, i); w0 = vec(p.tw, i - 1); }
        if (i + 1 < L) { c1 = row(p.up, i); w1 = vec(p.tw, i + 1); }
    };
    auto mv = [](const T *M, int ld, int K, T sign, T *y) {
        Mv t{};
        t.M = M; t.ld = ld; t.K = K; t.sign = sign; t.y = y;
        t.in = t.bin = t.out = -1;
        return t;
    };
    for (int l = 0; l < levels; ++l) {
        const auto &a = lists[l];
        std::vector<Mv> ts;
        for (size_t q = 1; q < a.size(); q += 2) {       // t_j = D_j^-1 b_j
            const int j = a[q];
            Mv t = mv(inv(j), Sp, Sp, T(1), vec(p.tw, j));
            if (l == 0) t.in = j;
            else if (l == 1) rhs0(j, t.in, t.d0, t.w0, t.d1, t.w1);
            else t.v0 = vec(p.bw, j);
            ts.push_back(t);
        }
        mv_stage(ts, l);
        if (l == 0) continue;
        ts.clear();
        for (size_t q = 0; q < a.size(); q += 2) {       // b_i -= L_i t_l + U_i t_r
            const int i = a[q];
            const int cpi = cp_off[l] + (int)q;
            const bool hl = q >= 1, hr = q + 1 < a.size();
            if (!hl && !hr) continue;
            Mv t = mv(cp(cpi, hl ? 0 : Sp), 2 * Sp, hl && hr ? 2 * Sp : Sp, -T(1), vec(p.bw, i));
            if (l == 1) rhs0(i, t.bin, t.e0, t.f0, t.e1, t.f1);
            else t.base = vec(p.bw, i);
            t.v0 = vec(p.tw, hl ? a[q - 1] : a[q + 1]);
            if (hl && hr) t.v1 = vec(p.tw, a[q + 1]);
            ts.push_back(t);
        }
        mv_stage(ts, l);
    }
    {
        Mv t = mv(inv(root), Sp, Sp, T(1), vec(p.xw, root));
        if (levels == 0) t.in = root;
        else if (levels == 1) rhs0(root, t.in, t.d0, t.w0, t.d1, t.w1);
        else t.v0 = vec(p.bw, root);
        t.out = root;
        std::vector<Mv> ts{t};
        mv_stage(ts, levels);
    }
    for (int l = levels - 1; l >= 0; --l) {
        const auto &a = lists[l];
        std::vector<Mv> ts;
        for (size_t q = 1; q < a.size(); q += 2) {
            const int j = a[q];
            const bool hr = q + 1 < a.size();
            Mv t;
            if (l == 0) {      // x_j = D_j^-1 (b_j - lo_j x_{j-1} - up_j x_{j+1})
                t = mv(inv(j), Sp, Sp, T(1), vec(p.xw, j));
                t.in = j;
                t.d0 = row(p.lo, j); t.w0 = vec(p.xw, a[q - 1]);
                if (hr) { t.d1 = row(p.up, j); t.w1 = vec(p.xw, a[q + 1]); }
            } else {           // x_j = t_j - [P_j | Q_j] [x_l; x_r]
                t = mv(pq(j), 2 * Sp, hr ? 2 * Sp : Sp, -T(1), vec(p.xw, j));
                t.v0 = vec(p.xw, a[q - 1]);
                t.v1 = hr ? vec(p.xw, a[q + 1]) : nullptr;
                t.base = vec(p.tw, j);
            }
            t.out = j;
            ts.push_back(t);
        }
        mv_stage(ts, l);
    }
}

template void bcr_solve_tasks<float>(const BcrLevels &, const BcrArrays<float> &, std::vector<BcrMv> &, std::vector<BcrStage> &);
template void bcr_solve_tasks<double>(const BcrLevels &, const BcrArrays<double> &, std::vector<BcrMvT<double>> &,
                                      std::vector<BcrStage> &);

BcrSizes bcr_sizes(int L, int S)
{
    BcrPlan p;
    p.L = L;
    p.S = S;
    p.Sp = (S + 31) / 32 * 32;
    Builder b{p, L, S, p.Sp, {}};
    b.build();
    BcrSizes z;
    z.Sp = p.Sp;
    z.Wt = p.Wt;
    z.Zt = p.Zt;
    z.Ncp = p.Ncp;
    z.ngemm = (int)p.gemm.size();
    z.ntile = (int)p.tile_task.size();
    z.nleaf = (int)p.leaf.size();
    z.nmv = (int)p.mv.size();
    z.nsol = (int)p.sol.size();
    const size_t blk = (size_t)p.Sp * p.Sp;
    z.floats_D = (size_t)L * blk;
    z.floats_INV = (size_t)L * blk;
    z.floats_TMP = (size_t)p.Zt * p.Sp * p.Wt;
    z.floats_CP = (size_t)p.Ncp * 2 * blk;
    z.floats_PQ = (size_t)L * 2 * blk;
    z.floats_vec = (size_t)L * p.Sp;
    return z;
}

int bcr_build(BcrPlan &p, int L, int S, cudaStream_t st)
{
    p.L = L;
    p.S = S;
    p.Sp = (S + 31) / 32 * 32;
    p.gemm.clear(); p.tile_task.clear(); p.leaf.clear(); p.mv.clear(); p.fac.clear(); p.sol.clear();
    Builder b{p, L, S, p.Sp, {}};
    b.build();
    // tensor maps of the five arrays
    const TcArray arrs[kArrays] = {{p.D, L, p.Sp, p.Sp}, {p.INV, L, p.Sp, p.Sp}, {p.TMP, p.Zt, p.Sp, p.Wt},
                                   {p.CP, p.Ncp, p.Sp, 2 * p.Sp}, {p.PQ, L, p.Sp, 2 * p.Sp}};
    p.maps.assign(2 * kArrays, CUtensorMap{});
    for (int a = 0; a < kArrays; ++a)
        if (tc_make_maps(arrs[a], &p.maps[2 * a], &p.maps[2 * a + 1]) != 0) return -1;
    if (!p.gemm.empty() && cudaMemcpyAsync(p.gemm_d, p.gemm.data(), p.gemm.size() * sizeof(TcTask), cudaMemcpyHostToDevice, st))
        return -1;
    if (!p.tile_task.empty() &&
        cudaMemcpyAsync(p.tile_task_d, p.tile_task.data(), p.tile_task.size() * sizeof(int), cudaMemcpyHostToDevice, st))
        return -1;
    if (!p.leaf.empty() && cudaMemcpyAsync(p.leaf_d, p.leaf.data(), p.leaf.size() * sizeof(BcrLeaf), cudaMemcpyHostToDevice, st))
        return -1;
    if (!p.mv.empty() && cudaMemcpyAsync(p.mv_d, p.mv.data(), p.mv.size() * sizeof(BcrMv), cudaMemcpyHostToDevice, st))
        return -1;
    if (cudaMemcpyAsync(p.maps_d, p.maps.data(), p.maps.size() * sizeof(CUtensorMap), cudaMemcpyHostToDevice, st))
        return -1;
    if (cudaMemcpyAsync(p.l0_d, p.level0_kept.data(), p.level0_kept.size() * sizeof(int), cudaMemcpyHostToDevice, st))
        return -1;
    if (cudaMemcpyAsync(p.sol_d, p.sol.data(), p.sol.size() * sizeof(BcrStage), cudaMemcpyHostToDevice, st)) return -1;
    // the host copies of the task lists must outlive the asynchronous copies
    if (cudaStreamSynchronize(st) != cudaSuccess) return -1;
    return 0;
}

void bcr_init_pad(const BcrPlan &p, cudaStream_t st)
{
    const long long n = (long long)p.L * (p.Sp - p.S) * p.Sp;
    if (n <= 0) return;
    count_launches(1);
    k_bcr_pad<<<nblk(n, 256), 256, 0, st>>>(p.D, p.L, p.S, p.Sp);
}

void bcr_work(const BcrPlan &p, double *mma_flops, double *leaf_flops)
{
    double m = 0.0, l = 0.0;
    for (const TcTask &t : p.gemm) {
        long long k = 0;
        for (int s = 0; s < t.nseg; ++s) k += t.seg[s].k;
        m += 2.0 * t.m * (double)t.n * (double)k;
    }
    for (const BcrLeaf &f : p.leaf) l += 2.0 * (double)f.n * f.n * f.n;
    if (mma_flops) *mma_flops = m;
    if (leaf_flops) *leaf_flops = l;
}

cudaError_t bcr_factor(const BcrPlan &p, const int *skip, Ctl *ctl, cudaStream_t st, BcrTimer *timer)
{
    for (const BcrStage &s : p.fac) {
        switch (s.kind) {
        case kBcrLeafStage: {
            if (timer) timer->begin(s.kind);
            cudaError_t e = launch_leaf(p.leaf_d + s.off, s.count, s.tiles, skip, ctl, st);
            if (timer) timer->end(s.kind);
            if (e != cudaSuccess) return e;
            break;
        }
        case kBcrGemm: {
            if (timer) timer->begin(s.kind);
            cudaError_t e = launch_tc_gemm(p.gemm_d + s.off, p.tile_task_d + s.tile, s.tiles, p.maps_d, skip, ctl, st);
            if (timer) timer->end(s.kind);
            if (e != cudaSuccess) return e;
            break;
        }
        case kBcrLevel0:
            count_launches(1);
            k_bcr_level0<<<dim3(nblk((long long)p.Sp * p.Sp / 4, 256), s.count), 256, 0, st>>>(
                p.D, p.INV, p.CP, p.lo, p.up, p.l0_d, p.L, p.S, p.Sp, skip, ctl);
            break;
        default:
            break;
        }
    }
    return cudaGetLastError();
}

}  // namespace xk

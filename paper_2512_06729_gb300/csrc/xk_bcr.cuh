// Block cyclic reduction of the block-tridiagonal system on the tensor cores:
// the mixed path's FP32 factorization and its solve.
#pragma once

#include <vector>

#include "xk_tc.cuh"

namespace xk {

constexpr int kBcrLeafMax = 160;   // largest block inverted directly by one CTA

// One block inverted by Gauss-Jordan with partial pivoting in one CTA (n <= kBcrLeafMax).
struct BcrLeaf {
    const float *in;
    float *out;
    int ldin, ldout, n;
};

// y = base + sign * M v for the rows [0, Sp) of one block: M is Sp x K row-major (ld).  v is the
// right-hand side of layer `in` (in >= 0) or the work vector v0, less d0 w0 and d1 w1 on the first S
// entries (the diagonal couplings of level 0), and behind it v1 when K = 2 Sp.  The base likewise:
// layer `bin` of the right-hand side or the vector base, less e0 f0 and e1 f1.  out >= 0: y is also
// the solution of that layer.
template <typename T>
struct BcrMvT {
    const T *M;
    const T *v0, *v1, *d0, *w0, *d1, *w1, *base, *e0, *f0, *e1, *f1;
    T *y;
    int ld, K;
    T sign;
    int in, bin, out;
};
using BcrMv = BcrMvT<float>;

struct BcrStage {
    int kind;          // BcrKind
    int off, count;    // range in the task list of that kind
    int tile;          // GEMM: first entry of its tiles in the tile list
    int tiles;         // GEMM: output tiles of the launch; leaf inversions: the blocks' order n
    int level;         // the reduction level it belongs to
};
enum BcrKind { kBcrLeafStage = 0, kBcrGemm = 1, kBcrLevel0 = 2, kBcrMv = 3 };

// The levels of the reduction of L layers: lists[0] all of them, then every second one, down to one.
// Layer lists[l][q] of a level l >= 1 has its couplings in block cp_off[l] + q of the coupling array.
struct BcrLevels {
    std::vector<std::vector<int>> lists;
    std::vector<int> cp_off;
    int ncp;
    explicit BcrLevels(int L) : lists{std::vector<int>(L)}, ncp(0)
    {
        for (int k = 0; k < L; ++k) lists[0][k] = k;
        while (lists.back().size() > 1) {
            std::vector<int> kept;
            for (size_t q = 0; q < lists.back().size(); q += 2) kept.push_back(lists.back()[q]);
            lists.push_back(kept);
        }
        cp_off.assign(lists.size(), 0);
        for (size_t l = 1; l < lists.size(); ++l) {
            cp_off[l] = ncp;
            ncp += (int)lists[l].size();
        }
    }
};

// Where the blocks and vectors of a reduction lie: INV [L] and PQ [L] ([P | Q] side by side) by layer,
// CP by coupling block ([L | U]), `rows` rows of ld (2 ld) entries to a block; vectors ld apart.
template <typename T>
struct BcrArrays {
    const T *INV, *CP, *PQ, *lo, *up;
    T *bw, *tw, *xw;
    int L, S, rows, ld;
};
// The solve's tasks and stages.
template <typename T>
void bcr_solve_tasks(const BcrLevels &lv, const BcrArrays<T> &a, std::vector<BcrMvT<T>> &mv, std::vector<BcrStage> &sol);

// What the persistent solve reads.
template <typename T>
struct BcrSolveT {
    const BcrStage *stages;
    const BcrMvT<T> *mv;
    int nstages, S, rows, ld;
    unsigned *bar;         // its GridSync words (2, zero between calls)
    int ctas;              // CTAs of the launch (0: one per SM)
};

// The plan of one column's factorization and solve.  Built on the host once per workspace; the
// task lists live in the workspace.
struct BcrPlan {
    int L = 0, S = 0, Sp = 0, Wt = 0, Zt = 0, Ncp = 0, levels = 0;
    // arrays: D (the FP32 blocks, padded to Sp x Sp per layer), INV (inverses), TMP (inversion
    // temporaries), CP (dense couplings [L | U] of the levels >= 1), PQ (D^-1 [L | U])
    float *D = nullptr, *INV = nullptr, *TMP = nullptr, *CP = nullptr, *PQ = nullptr;
    float *bw = nullptr, *tw = nullptr, *xw = nullptr;      // [L][Sp] vectors of the solve
    const float *lo = nullptr, *up = nullptr;                // level-0 couplings [L][S] (FP32)
    std::vector<TcTask> gemm;
    std::vector<int> tile_task;    // per product stage: the stage's task of each output tile
    std::vector<BcrLeaf> leaf;
    std::vector<BcrMv> mv;
    std::vector<BcrStage> fac, sol;
    std::vector<int> level0_kept;                            // even layers kept at level 0
    TcTask *gemm_d = nullptr;
    int *tile_task_d = nullptr;
    BcrLeaf *leaf_d = nullptr;
    BcrMv *mv_d = nullptr;
    CUtensorMap *maps_d = nullptr;
    std::vector<CUtensorMap> maps;
    int *l0_d = nullptr;
    BcrStage *sol_d = nullptr;     // the solve's stages, walked by one persistent kernel
    unsigned *bar = nullptr;       // its GridSync words (2, zero between calls)
    int solve_ctas = 0;            // CTAs of that kernel (0: one per SM)
};

// Sizes of the device arrays and task lists of an L-layer, S-species column (no pointers).
struct BcrSizes {
    int Sp, Wt, Zt, Ncp, ngemm, ntile, nleaf, nmv, nsol;
    size_t floats_D, floats_INV, floats_TMP, floats_CP, floats_PQ, floats_vec;
};
BcrSizes bcr_sizes(int L, int S);
// Fill the plan for arrays already laid out (p.D ... p.xw, p.lo, p.up, and the task storage
// pointers set); uploads task lists and tensor maps on st.  0 or -1.
int bcr_build(BcrPlan &p, int L, int S, cudaStream_t st);
// Pad rows of D to the identity (once per workspace).
void bcr_init_pad(const BcrPlan &p, cudaStream_t st);
// Optional marks around the factorization's launches (tracing).
struct BcrTimer {
    virtual void begin(int kind) = 0;
    virtual void end(int kind) = 0;
    virtual ~BcrTimer() = default;
};
// Factorization: every level's inversions and Schur updates (D is overwritten).
cudaError_t bcr_factor(const BcrPlan &p, const int *skip, Ctl *ctl, cudaStream_t st, BcrTimer *timer = nullptr);
// Flops of one factorization: 2 m n k over the products, 2 n^3 over the leaves.
void bcr_work(const BcrPlan &p, double *mma_flops, double *leaf_flops);
inline BcrSolveT<float> solve_of(const BcrPlan &p)
{
    return {p.sol_d, p.mv_d, (int)p.sol.size(), p.S, p.Sp, p.Sp, p.bar, p.solve_ctas};
}

// The same reduction in FP64 (xk_bcr64.cu): blocks of S rows, S at most kBcr64Max.
constexpr int kBcr64Max = 152;    // rows of a block that a cluster of 8 CTAs holds (inv_layout)
struct Bcr64Inv {
    const double *in;
    double *out;
};
// C = src + sign (A0 B0 + A1 B1), all S x S
struct Bcr64Gemm {
    const double *a0, *b0, *a1, *b1, *src;
    double *c;
    double sign;
    int lda, ldb, ldc;
};
struct Bcr64Plan {
    int L = 0, S = 0, ld = 0, ldd = 0, levels = 0;    // ldd: of D, ld: of the others
    double *D = nullptr, *INV = nullptr, *CP = nullptr, *PQ = nullptr, *bw = nullptr, *tw = nullptr, *xw = nullptr;
    const double *lo = nullptr, *up = nullptr;
    std::vector<Bcr64Inv> inv;
    std::vector<Bcr64Gemm> gemm;
    std::vector<BcrMvT<double>> mv;
    std::vector<BcrStage> fac, sol;
    Bcr64Inv *inv_d = nullptr;
    Bcr64Gemm *gemm_d = nullptr;
    BcrMvT<double> *mv_d = nullptr;
    BcrStage *sol_d = nullptr;
    unsigned *bar = nullptr;
    int solve_ctas = 0;
};
struct Bcr64Sizes {
    int ninv, ngemm, nmv, nsol;
    size_t inv, cp, pq, vec;       // doubles
};
Bcr64Sizes bcr64_sizes(int L, int S);
// Fill the plan for arrays already laid out (the task lists in the order inv, gemm, mv, sol); uploads the
// lists and clears the arrays' padding.
cudaError_t bcr64_build(Bcr64Plan &p, int L, int S, int ldd, cudaStream_t st);
cudaError_t bcr64_factor(const Bcr64Plan &p, Ctl *ctl, cudaStream_t st);
inline BcrSolveT<double> solve_of(const Bcr64Plan &p)
{
    return {p.sol_d, p.mv_d, (int)p.sol.size(), p.S, p.S, p.ld, p.bar, p.solve_ctas};
}

// x = M^-1 (b * bscale) (* xscale) with the factorization, FP64 in and out (xk_fgmres.cu).
template <typename T>
cudaError_t bcr_solve(const BcrSolveT<T> &p, const double *b, double *x, const double *bscale, const double *xscale,
                      const int *skip, Ctl *ctl, cudaStream_t st);

struct GmArgs;
// The whole FGMRES of enqueue_fgmres preconditioned by the reduction (role 0 or 2), in one cooperative
// launch; its matrix-vector product is launch_jv's with the rows divided by rowd, its preconditioner
// bcr_solve's with bscale = rowd.  Not for cfg.photo_jacobian, whose product needs launches of its own.
template <typename T>
cudaError_t bcr_fgmres(const BcrSolveT<T> &p, const Col &c, const GmArgs &g, const double *rowd, cudaStream_t st);

}  // namespace xk

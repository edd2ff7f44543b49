// Batched products C = A B on the tcgen05 tensor cores with FP32 accuracy.
//
// A tile of 128 x 128 of one task's output at a time.  Warp 0 streams
// the operands into shared memory with TMA: A (row-major) in 128-byte swizzled
// rows, B (row-major, i.e. N-major) as a plain [32 k][128 n] tile.  The split
// warps turn every FP32 element x into a TF32 head h (x rounded to nearest at 10
// explicit mantissa bits, exact in TF32) and tail l = x - h (exact in FP32, at
// most 2^-11 |x|), itself rounded to TF32: A into tensor memory, a row per
// thread (the swizzle makes those row reads conflict-free), B transposed into
// the K-major swizzled layout that the TF32 kind reads (16-byte chunk c of row n
// stored at chunk c ^ (n mod 8)).  Warp 1 issues, per K step of 8, the three
// products A_h B_h + A_h B_l + A_l B_h into one FP32 accumulator in tensor
// memory (the 3xTF32 scheme: the rounding of the tails and the dropped A_l B_l
// term leave at most about 3 * 2^-22 of |a||b| per product, a dozen FP32 units,
// far below TF32's 2^-11).  The epilogue warps read the accumulator back
// (tcgen05.ld) and apply alpha, beta and the column routing of the task, while
// the other warps are at the next tile: a CTA per SM takes the launch's tiles in
// turn, two accumulators alternating.
//
// What bounds it is the traffic of one SM's shared memory, 128 bytes a clock,
// per 32-deep stage: with A's halves in shared memory too it is 32 KB landing,
// 32 KB read by the split, 64 KB written by it and 96 KB read by the twelve
// products, 1,800 clocks beside the products' own 900, and a stage measured 1.2
// us.  A in tensor memory takes 16 KB of the writes and 48 KB of the products'
// reads away, and two groups of eight split warps on alternate stages hide each
// other's latencies.
//
// The launches of a factorization follow one another (programmatic dependent
// launch): barriers, tensor memory and the task are set up while the previous
// launch drains.
//
// Every wait on an mbarrier is bounded; a wait that gives up records
// ctl->err_timeout, and the CTA still waits (bounded) for its own tensor-core
// work and frees its tensor memory before returning.
#include <cuda.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include <algorithm>
#include <mutex>

#include "xk_tc.cuh"

namespace xk {

namespace {

constexpr int kRaw = 4;                                   // stages as loaded: A and B tiles
constexpr int kSplit = 3;                                 // stages split: B head and tail, A in tensor memory
constexpr int kGroups = 2;                                // groups of split warps, on alternate stages
// a group must see every phase of the slots it waits for: a wait for phase n + 1 passes while phase n
// is still open
static_assert(kRaw % kGroups == 0, "a raw slot belongs to one group");
constexpr int kGroupWarps = 8;                            // of a group: four on A, four on B
constexpr int kSplitWarps = kGroups * kGroupWarps;        // warps 2-17: split
constexpr int kEpiWarps = 4;                              // warps 18-21: epilogue
constexpr int kThreads = 32 * (2 + kSplitWarps + kEpiWarps);   // warp 0 TMA, warp 1 MMA
constexpr int kMaxTiles = 64;                             // output tiles of one CTA
constexpr uint32_t kTileBytes = kTcTileM * kTcStageK * 4; // 16 KB: A tile (128 x 32) or B tile (32 x 128)
constexpr uint32_t kTmemCols = 512;                       // two accumulators of 128, 64 per split stage for A
constexpr uint32_t kTmemA = 256;
constexpr size_t kSmemBytes = (2 * kRaw + 2 * kSplit) * kTileBytes + 1024 + 256;
constexpr unsigned long long kWaitPolls = 1ull << 26;

__device__ __forceinline__ uint32_t smem_u32(const void *p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count)
{
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
}

__device__ __forceinline__ void mbar_expect_tx(uint32_t bar, uint32_t bytes)
{
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}

__device__ __forceinline__ void mbar_arrive(uint32_t bar)
{
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}

__device__ __forceinline__ bool mbar_try(uint32_t bar, uint32_t parity)
{
    uint32_t done;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(done)
        : "r"(bar), "r"(parity)
        : "memory");
    return done != 0;
}

// Bounded wait for the phase of the given parity; false (and the error flag) when it gives up
// or another thread of the CTA already gave up.
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity, volatile int *abort, Ctl *ctl)
{
    for (unsigned long long i = 0; i < kWaitPolls; ++i) {
        if (mbar_try(bar, parity)) return true;
        if (*abort) return false;
    }
    *abort = 1;
    if (ctl) atomicExch(&ctl->err_timeout, 1);
    return false;
}

__device__ __forceinline__ void tma_load_3d(uint32_t dst, const CUtensorMap *map, int x, int y, int z, uint32_t bar)
{
    asm volatile(
        "cp.async.bulk.tensor.3d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4}], [%5];"
        ::"r"(dst), "l"((uint64_t)map), "r"(x), "r"(y), "r"(z), "r"(bar)
        : "memory");
}

// Shared-memory matrix descriptor, 128-byte swizzle: start, leading and stride byte offsets.
__device__ __forceinline__ uint64_t sw128_desc(uint32_t saddr, uint32_t lbo, uint32_t sbo)
{
    uint64_t d = 0;
    d |= (uint64_t)((saddr >> 4) & 0x3FFFu);
    d |= (uint64_t)((lbo >> 4) & 0x3FFFu) << 16;
    d |= (uint64_t)((sbo >> 4) & 0x3FFFu) << 32;
    d |= (uint64_t)1 << 46;          // descriptor version of the 5th-generation tensor core
    d |= (uint64_t)2 << 61;          // 128-byte swizzle
    return d;
}

// Instruction descriptor: kind::tf32, FP32 accumulator, A and B K-major, M x N.
__host__ __device__ constexpr uint32_t tf32_idesc(int M, int N)
{
    return (1u << 4)                  // accumulator FP32
         | (2u << 7)                  // A: TF32
         | (2u << 10)                 // B: TF32
         | ((uint32_t)(N >> 3) << 17)
         | ((uint32_t)(M >> 4) << 24);
}

// D += A B with A (128 x 8, a lane per row, a column per k) in tensor memory.
__device__ __forceinline__ void mma_tf32(uint32_t tmem, uint32_t atmem, uint64_t bd, uint32_t idesc, uint32_t acc)
{
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "setp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::tf32 [%0], [%1], %2, %3, p;\n\t}"
        ::"r"(tmem), "r"(atmem), "l"(bd), "r"(idesc), "r"(acc)
        : "memory");
}

// 16 columns of this warp's 32 lanes.
__device__ __forceinline__ void tmem_st16(uint32_t taddr, const float (&r)[16])
{
    asm volatile(
        "tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], "
        "{%1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, %16};"
        ::"r"(taddr), "f"(r[0]), "f"(r[1]), "f"(r[2]), "f"(r[3]), "f"(r[4]), "f"(r[5]), "f"(r[6]), "f"(r[7]), "f"(r[8]),
          "f"(r[9]), "f"(r[10]), "f"(r[11]), "f"(r[12]), "f"(r[13]), "f"(r[14]), "f"(r[15])
        : "memory");
}

__device__ __forceinline__ void mma_commit(uint32_t bar)
{
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar) : "memory");
}

__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }

__device__ __forceinline__ void tmem_ld16(uint32_t taddr, uint32_t (&r)[16])
{
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 "
        "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
          "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
        : "r"(taddr));
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
}

// x rounded to the nearest TF32 value (ties away from zero), low 13 bits cleared: exact in TF32.
__device__ __forceinline__ float tf32_round(float x) { return __uint_as_float((__float_as_uint(x) + 0x1000u) & 0xFFFFE000u); }

__global__ void __launch_bounds__(kThreads, 1)
k_tc_gemm(const TcTask *__restrict__ tasks, const int *__restrict__ tile_task, int total,
          const CUtensorMap *__restrict__ maps, const int *skip, Ctl *ctl)
{
    extern __shared__ uint8_t smem_raw[];
    __shared__ uint32_t tmem_sh;
    __shared__ int abort_sh, s_task[kMaxTiles], s_nk[kMaxTiles];
    // the next launch may set up; its own wait holds it until this one has finished
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    const uint32_t raw_u = smem_u32(smem_raw);
    uint8_t *smem = smem_raw + (((raw_u + 1023u) & ~1023u) - raw_u);     // 1024-byte aligned tiles
    const uint32_t sbase = smem_u32(smem);
    // raw stage r: A at 2 r tiles, B behind it; split stage s: B head at kSplitAt + 2 s tiles, tail behind it
    constexpr uint32_t kSplitAt = 2 * kRaw * kTileBytes;
    const uint32_t bars = sbase + kSplitAt + 2 * kSplit * kTileBytes;
    auto full = [&](int r) { return bars + 8u * r; };
    auto taken = [&](int r) { return bars + 8u * (kRaw + r); };
    auto ready = [&](int s) { return bars + 8u * (2 * kRaw + s); };
    auto empty = [&](int s) { return bars + 8u * (2 * kRaw + kSplit + s); };
    auto accf = [&](int b) { return bars + 8u * (2 * kRaw + 2 * kSplit + b); };       // accumulator b is complete
    auto acce = [&](int b) { return bars + 8u * (2 * kRaw + 2 * kSplit + 2 + b); };   // ... has been read
    const uint32_t drain = bars + 8u * (2 * kRaw + 2 * kSplit + 4);

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int ntile = (total - 1 - (int)blockIdx.x) / (int)gridDim.x + 1;     // tiles of this CTA (the host sees to <= kMaxTiles)
    volatile int *abort = &abort_sh;

    for (int i = threadIdx.x; i < ntile; i += kThreads) {
        const int q = tile_task ? tile_task[blockIdx.x + i * gridDim.x] : 0;
        const TcTask &t = tasks[q];
        s_task[i] = q;
        s_nk[i] = (t.seg[0].k + (t.nseg > 1 ? t.seg[1].k : 0)) / kTcStageK;
    }
    if (threadIdx.x == 0) {
        abort_sh = 0;
        for (int r = 0; r < kRaw; ++r) {
            mbar_init(full(r), 1);
            mbar_init(taken(r), kGroupWarps);
        }
        for (int s = 0; s < kSplit; ++s) {
            mbar_init(ready(s), kGroupWarps);
            mbar_init(empty(s), 1);
        }
        for (int b = 0; b < 2; ++b) {
            mbar_init(accf(b), 1);
            mbar_init(acce(b), kEpiWarps);
        }
        mbar_init(drain, 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_sh)),
                     "r"(kTmemCols)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = tmem_sh;
    bool mma_issued = false;

    // what the previous launches wrote is visible from here on
    asm volatile("griddepcontrol.wait;" ::: "memory");
    const bool off = (ctl && (ctl->finished || ctl->err_timeout)) || (skip && *skip);

    if (off) {
        // nothing to do: free the tensor memory below
    } else if (warp == 0) {
        if (lane == 0) {
            bool go = true;
            for (int i = 0, it = 0; i < ntile && go; ++i) {
                const TcTask &t = tasks[s_task[i]];
                const int local = (int)blockIdx.x + i * (int)gridDim.x - t.tile0;
                const int tm = local / t.tiles_n, tn = local - tm * t.tiles_n;
                for (int sg = 0; sg < t.nseg && go; ++sg) {
                    const TcSeg g = t.seg[sg];
                    for (int kk = 0; kk < g.k; kk += kTcStageK, ++it) {
                        const int r = it % kRaw;
                        if (it >= kRaw && !mbar_wait(taken(r), ((uint32_t)(it / kRaw) & 1u) ^ 1u, abort, ctl)) {
                            go = false;
                            break;
                        }
                        const uint32_t st = sbase + 2 * r * kTileBytes;
                        mbar_expect_tx(full(r), 2 * kTileBytes);
                        tma_load_3d(st, maps + 2 * g.amap, g.ax + kk, g.ay + tm * kTcTileM, g.az, full(r));
                        tma_load_3d(st + kTileBytes, maps + 2 * g.bmap + 1, g.bx + tn * kTcTileN, g.by + kk, g.bz, full(r));
                    }
                }
            }
        }
    } else if (warp == 1) {
        if (lane == 0) {
            constexpr uint32_t idesc = tf32_idesc(kTcTileM, kTcTileN);
            bool go = true;
            for (int i = 0, it = 0; i < ntile && go; ++i) {
                const int b = i & 1;
                const uint32_t acc = tmem + 128u * b;
                if (i >= 2 && !mbar_wait(acce(b), ((uint32_t)(i / 2) & 1u) ^ 1u, abort, ctl)) break;
                tc_fence_after();
                for (int j = 0; j < s_nk[i]; ++j, ++it) {
                    const int s = it % kSplit;
                    if (!mbar_wait(ready(s), (uint32_t)(it / kSplit) & 1u, abort, ctl)) {
                        go = false;
                        break;
                    }
                    tc_fence_after();
                    const uint32_t bt = sbase + kSplitAt + 2 * s * kTileBytes;
                    const uint32_t at = tmem + kTmemA + 64u * s;
#pragma unroll
                    for (int ks = 0; ks < kTcStageK / 8; ++ks) {
                        // B K-major: rows of 32 FP32 (128 B), 8-row groups 1024 B apart, K step of 8 = 32 B
                        const uint64_t bh = sw128_desc(bt + ks * 32u, 16u, 1024u);
                        const uint64_t bl = sw128_desc(bt + kTileBytes + ks * 32u, 16u, 1024u);
                        const uint32_t ah = at + 8u * ks, al = at + 32u + 8u * ks;
                        mma_tf32(acc, ah, bh, idesc, (j | ks) ? 1u : 0u);
                        mma_tf32(acc, ah, bl, idesc, 1u);
                        mma_tf32(acc, al, bh, idesc, 1u);
                    }
                    mma_issued = true;
                    mma_commit(empty(s));
                }
                if (go) mma_commit(accf(b));
            }
        }
    } else if (warp < 2 + kSplitWarps) {
        const int sw = warp - 2, group = sw / kGroupWarps, gw = sw % kGroupWarps;
        const int quad = warp & 3;                 // the tensor-memory lanes this warp may touch: 32 quad ..
        int stages = 0;
        for (int i = 0; i < ntile; ++i) stages += s_nk[i];
        for (int it = group; it < stages; it += kGroups) {
            const int r = it % kRaw, s = it % kSplit;
            bool ok = mbar_wait(full(r), (uint32_t)(it / kRaw) & 1u, abort, ctl);
            if (ok && it >= kSplit) ok = mbar_wait(empty(s), ((uint32_t)(it / kSplit) & 1u) ^ 1u, abort, ctl);
            if (!__all_sync(0xffffffffu, ok)) break;
            const uint8_t *raw = smem + 2 * r * kTileBytes;
            float h[16], l[16];
            auto split = [&] {
#pragma unroll
                for (int k = 0; k < 16; ++k) {
                    h[k] = tf32_round(l[k]);
                    l[k] = tf32_round(l[k] - h[k]);
                }
            };
            if (gw < 4) {
                // A: row m of the tile, chunk c of its eight at c ^ (m mod 8)
                tc_fence_after();
                const int m = quad * 32 + lane;
                const float4 *row = (const float4 *)(raw + m * 128);
                const uint32_t at = tmem + ((uint32_t)(quad * 32) << 16) + kTmemA + 64u * s;
#pragma unroll
                for (int half = 0; half < 2; ++half) {
#pragma unroll
                    for (int c = 0; c < 4; ++c) {
                        const float4 v = row[(4 * half + c) ^ (m & 7)];
                        l[4 * c] = v.x; l[4 * c + 1] = v.y; l[4 * c + 2] = v.z; l[4 * c + 3] = v.w;
                    }
                    split();
                    tmem_st16(at + 16u * half, h);
                    tmem_st16(at + 32u + 16u * half, l);
                }
                asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
                tc_fence_before();
            } else {
                // B: column n of the [32 k][128 n] tile
                const int n = (gw - 4) * 32 + lane;
                const float *b = (const float *)(raw + kTileBytes) + n;
                uint8_t *bh = smem + kSplitAt + 2 * s * kTileBytes + n * 128, *bl = bh + kTileBytes;
#pragma unroll
                for (int half = 0; half < 2; ++half) {
#pragma unroll
                    for (int k = 0; k < 16; ++k) l[k] = b[(16 * half + k) * kTcTileN];
                    split();
#pragma unroll
                    for (int c = 0; c < 4; ++c) {
                        const int off16 = ((4 * half + c) ^ (n & 7)) * 16;
                        *(float4 *)(bh + off16) = make_float4(h[4 * c], h[4 * c + 1], h[4 * c + 2], h[4 * c + 3]);
                        *(float4 *)(bl + off16) = make_float4(l[4 * c], l[4 * c + 1], l[4 * c + 2], l[4 * c + 3]);
                    }
                }
                asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            }
            __syncwarp();
            if (lane == 0) {
                mbar_arrive(taken(r));
                mbar_arrive(ready(s));
            }
        }
    } else {
        // epilogue: 32 rows (the warp's lanes of tensor memory), 16 columns at a time; beta's operand of
        // the next 16 is read while these are written
        const int quad = warp & 3;
        for (int i = 0; i < ntile; ++i) {
            const TcTask &t = tasks[s_task[i]];
            const int local = (int)blockIdx.x + i * (int)gridDim.x - t.tile0;
            const int tm = local / t.tiles_n, tn = local - tm * t.tiles_n;
            const int row = tm * kTcTileM + quad * 32 + lane, n0 = tn * kTcTileN;
            const bool live = row < t.m;
            const int nc = min(kTcTileN, t.n - n0) / 16;
            float4 old[4];
            // where columns n .. n + 15 go (destinations change at multiples of 32)
            auto dest = [&](int c, const float *&src, float &alpha, float &beta) {
                const int n = n0 + 16 * c, o = (t.nout > 1 && n >= t.out[0].n) ? 1 : 0;
                const TcOut &O = t.out[o];
                const int nn = o ? n - t.out[0].n : n;
                alpha = O.alpha;
                beta = O.src ? O.beta : 0.0f;
                src = O.src + (long long)row * O.lds + nn;
                return O.ptr + (long long)row * O.ld + nn;
            };
            auto fetch = [&](int c) {
                const float *src;
                float alpha, beta;
                dest(c, src, alpha, beta);
                if (live && beta != 0.0f) {
#pragma unroll
                    for (int j = 0; j < 4; ++j) old[j] = ((const float4 *)src)[j];
                }
            };
            if (nc > 0) fetch(0);
            const bool ok = mbar_wait(accf(i & 1), (uint32_t)(i / 2) & 1u, abort, ctl);
            if (!__all_sync(0xffffffffu, ok)) break;
            tc_fence_after();
            for (int c = 0; c < nc; ++c) {
                uint32_t r[16];
                tmem_ld16(tmem + 128u * (i & 1) + ((uint32_t)(quad * 32) << 16) + 16u * c, r);
                const float *src;
                float alpha, beta;
                float4 *dst = (float4 *)dest(c, src, alpha, beta);
                if (live) {
#pragma unroll
                    for (int j = 0; j < 4; ++j) {
                        float4 v = make_float4(alpha * __uint_as_float(r[4 * j]), alpha * __uint_as_float(r[4 * j + 1]),
                                               alpha * __uint_as_float(r[4 * j + 2]), alpha * __uint_as_float(r[4 * j + 3]));
                        if (beta != 0.0f) {
                            v.x += beta * old[j].x; v.y += beta * old[j].y; v.z += beta * old[j].z; v.w += beta * old[j].w;
                        }
                        dst[j] = v;
                    }
                }
                if (c + 1 < nc) fetch(c + 1);
            }
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(acce(i & 1));
        }
    }
    __syncwarp();
    // an aborted CTA waits (bounded) for the tensor-core work it issued before freeing TMEM
    if (warp == 1 && lane == 0 && *abort && mma_issued) {
        mma_commit(drain);
        for (unsigned long long i = 0; i < kWaitPolls && !mbar_try(drain, 0u); ++i) {
        }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 1) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(kTmemCols) : "memory");
    }
}

using EncodeTiled = CUresult (*)(CUtensorMap *, CUtensorMapDataType, cuuint32_t, void *, const cuuint64_t *,
                                 const cuuint64_t *, const cuuint32_t *, const cuuint32_t *, CUtensorMapInterleave,
                                 CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

EncodeTiled encode_fn()
{
    static std::once_flag once;
    static EncodeTiled fn = nullptr;
    std::call_once(once, [] {
        void *p = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) == cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            fn = (EncodeTiled)p;
        else
            cudaGetLastError();
    });
    return fn;
}

}  // namespace

int tc_make_maps(const TcArray &a, CUtensorMap *amap, CUtensorMap *bmap)
{
    EncodeTiled enc = encode_fn();
    if (!enc || !a.base || a.C % 32 || a.R <= 0 || a.Z <= 0 || ((uintptr_t)a.base & 255)) return -1;
    const cuuint64_t dims[3] = {(cuuint64_t)a.C, (cuuint64_t)a.R, (cuuint64_t)a.Z};
    const cuuint64_t strides[2] = {(cuuint64_t)a.C * 4, (cuuint64_t)a.C * a.R * 4};
    const cuuint32_t elem[3] = {1, 1, 1};
    const cuuint32_t box_a[3] = {32, (cuuint32_t)kTcTileM, 1};
    const cuuint32_t box_b[3] = {(cuuint32_t)kTcTileN, (cuuint32_t)kTcStageK, 1};
    if (enc(amap, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 3, a.base, dims, strides, box_a, elem, CU_TENSOR_MAP_INTERLEAVE_NONE,
            CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_128B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
        return -1;
    if (enc(bmap, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 3, a.base, dims, strides, box_b, elem, CU_TENSOR_MAP_INTERLEAVE_NONE,
            CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_128B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
        return -1;
    return 0;
}

int tc_number_tiles(TcTask *tasks, int ntasks)
{
    int total = 0;
    for (int i = 0; i < ntasks; ++i) {
        TcTask &t = tasks[i];
        t.tiles_n = (t.n + kTcTileN - 1) / kTcTileN;
        t.tiles = ((t.m + kTcTileM - 1) / kTcTileM) * t.tiles_n;
        t.tile0 = total;
        total += t.tiles;
    }
    return total;
}

cudaError_t launch_tc_gemm(const TcTask *tasks, const int *tile_task, int total_tiles, const CUtensorMap *maps,
                           const int *skip, Ctl *ctl, cudaStream_t st)
{
    if (total_tiles <= 0) return cudaSuccess;
    const cudaError_t e = allow_smem(k_tc_gemm, kSmemBytes);
    if (e != cudaSuccess) return e;
    // a CTA per SM; more where one would get over kMaxTiles tiles
    const int ctas = std::max(std::min(total_tiles, device_sms()), (total_tiles + kMaxTiles - 1) / kMaxTiles);
    count_launches(1);
    return launch_dependent(k_tc_gemm, dim3(ctas), dim3(kThreads), kSmemBytes, st, tasks, tile_task, total_tiles, maps, skip,
                            ctl);
}

}  // namespace xk

// ---------------------------------------------------------------------------
// C-ABI: one product, to check the tensor-core contraction on its own.
// ---------------------------------------------------------------------------
namespace {
__device__ xk::TcTask g_tc_task;
__device__ CUtensorMap g_tc_maps[4];
std::mutex g_tc_mu;
}  // namespace

extern "C" int xk_tc_gemm(int M, int N, int K, const float *A, int lda, const float *B, int ldb, float *C, int ldc,
                          float alpha, float beta, void *stream)
{
    using namespace xk;
    if (M <= 0 || N <= 0 || K <= 0 || M % 32 || N % 32 || K % 32 || lda % 32 || ldb % 32 || ldc % 32 || lda < K ||
        ldb < N || ldc < N || !A || !B || !C)
        return XK_EINVAL;
    if (((uintptr_t)A & 255) || ((uintptr_t)B & 255) || ((uintptr_t)C & 15)) return XK_EINVAL;
    cudaStream_t st = (cudaStream_t)stream;
    TcArray aa{const_cast<float *>(A), 1, M, lda}, bb{const_cast<float *>(B), 1, K, ldb};
    CUtensorMap maps[4];
    if (tc_make_maps(aa, &maps[0], &maps[1]) || tc_make_maps(bb, &maps[2], &maps[3])) return XK_EINVAL;
    TcTask t{};
    t.nseg = 1;
    t.seg[0] = TcSeg{0, 0, 0, 0, 1, 0, 0, 0, K};
    t.nout = 1;
    t.out[0] = TcOut{C, C, ldc, ldc, alpha, beta, N};
    t.m = M;
    t.n = N;
    int tiles = tc_number_tiles(&t, 1);
    std::lock_guard<std::mutex> lock(g_tc_mu);
    void *dtask = nullptr, *dmaps = nullptr;
    if (cudaGetSymbolAddress(&dtask, g_tc_task) != cudaSuccess || cudaGetSymbolAddress(&dmaps, g_tc_maps) != cudaSuccess ||
        cudaMemcpyAsync(dtask, &t, sizeof t, cudaMemcpyHostToDevice, st) != cudaSuccess ||
        cudaMemcpyAsync(dmaps, maps, sizeof maps, cudaMemcpyHostToDevice, st) != cudaSuccess) {
        cudaGetLastError();
        return XK_ECUDA;
    }
    cudaError_t e = launch_tc_gemm((const TcTask *)dtask, nullptr, tiles, (const CUtensorMap *)dmaps, nullptr, nullptr, st);
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    if (e != cudaSuccess) {
        cudaGetLastError();
        return XK_ECUDA;
    }
    return XK_OK;
}

// 16-bit GEMM for the decoder's projections on the 5th-generation tensor cores, with the WEIGHT rows on the accumulator
// lanes:  D^T[feature, row] = W[feature, :] . X[row, :],  float accumulation in TMEM.
//
// Why this orientation.  A decode step has few activation rows and streams every weight once.  With the weights on the
// MMA's M axis (128 features per CTA, always full) the rows sit on its N axis, whose width follows the batch in steps of
// 16: 71 rows cost an 80-wide MMA and an 80-row operand tile, not 128.  And a warp's 32 lanes hold 32 consecutive
// features of one row, so every epilogue access to the residual stream, the activations or the logits is coalesced.
//
//   CG = 2   two CTAs of a cluster form one 256-feature tile (cta_group::2): each loads its own 128 weight rows and HALF
//            of the activation tile, 32 KB per 64-deep k-block at 256 rows instead of 48 KB.  The projections at more than
//            128 rows are bound by the bytes that flow from L2 into shared memory, not by the MMA.
//   splits   the CTAs of a cluster share a tile and take a K range each (small batches: 12 or 16 feature tiles would
//            otherwise keep 12 or 16 SMs busy).  Every CTA leaves its partial tile in its own shared memory and reduces a
//            share of the rows over distributed shared memory, slices added in order: complete sums inside the kernel, so
//            the epilogues below can be fused at every batch size, and the result does not depend on timing.
//
// Roles: warp 0 = TMA producer, warp 1 = MMA issuer (and TMEM owner), warps 2..9 = epilogue, two warps per 32-lane quarter
// of the accumulator (two groups of 128 threads, each taking every other chunk of rows).
//
// Programmatic dependent launch: the kernel may start while the one before it runs.  Until grid_dep_wait() it sets up
// barriers and TMEM and requests weight tiles; it releases its own dependents only after its wait, so whatever runs two
// kernels back has finished when a kernel starts.
//
// What it measured when it replaced the rows-on-lanes kernel with separate norm and post-processing kernels (four projections and
// what lies between them, per layer, B200): 16 rows 46 -> 34 us, 71 rows 50 -> 41, 237 rows 80 -> 57, 336 rows 78 -> 68.  Whole decode
// steps then and now: 1.5B shape, 16 rows 2.03 -> 1.32 ms, 237 rows 3.76 -> 2.57 ms; 8B shape, 64 rows 6.28 -> 4.43 ms.
// What bounds it: up to about 128 rows the weight stream (gate/up of 16 rows: 55 MB in the 11.5 us from its first request to its
// last tile, 4.8 TB/s of 6.55 copy rate, 5 us of it before its turn) and a fixed chain per launch (hand-over 0.7 us, first tile 0.5,
// drain 1-2; where K is split about 1 more for the hand-over of the partial tiles).  From 512 rows on the MMAs and,
// beside them, the epilogue's instructions (gate/up of 10,184 rows: 405 us, without any epilogue 350).  Counters, alone on the GPU:
// gate/up 64 rows 17.6 us, tensor pipe 13 %, DRAM 38 %; 1,024 rows 49.1 us, 70 %, 15 %; 10,240 rows 368 us, 91 %.
//
// All waits on mbarriers are bounded; one that runs out raises DEV_ERR_WAIT_TIMEOUT, every role leaves its loop, and the
// CTA frees its TMEM before it returns.
#pragma once

#include <cuda.h>
#include <cuda_fp16.h>

#include "common.cuh"
#include "gemm_tc.cuh"
#include "kernels_basic.cuh"

namespace pc {
namespace wt {

using tc::mbar_arrive;
using tc::mbar_arrive_expect_tx;
using tc::mbar_init;
using tc::smem_u32;
using tc::tc_fence_after;
using tc::tc_fence_before;
using tc::tma_load_2d;

constexpr int FT = 128;                // features per CTA
constexpr int BK = 64;                 // k-block: 64 16-bit values = one 128-byte swizzle row
constexpr int W_BYTES = FT * BK * 2;
constexpr int EPI_WARPS = 8, EPI_THREADS = 32 * EPI_WARPS;
constexpr int THREADS = 64 + EPI_THREADS;
constexpr int MAX_STAGES = 12;
constexpr int MAX_ROWS_TILE = 256;
constexpr int MAX_SPLITS = 8;
constexpr int SMEM_BUDGET = 222 * 1024;          // of 227 KB
constexpr uint64_t WAIT_NS = 1000000000ull;      // no wait of a pass is longer than its kernel, which takes milliseconds at most

// What the host fixes for a launch.
struct Geom {
    int M, N, K;         // row bound, features, depth
    int nt;              // activation rows per tile: a multiple of 16 (CG 1) or 32 (CG 2), at most 256
    int splits;          // K ranges = CTAs (CG 1) or CTA pairs (CG 2) per tile
    int stages;
    int n_acc;           // accumulators: 2 when a cluster walks several tiles
    int half;            // operands IEEE half (1) or bfloat16 (0)
    int tiles_r, n_tiles;          // row tiles, all tiles
    uint32_t tmem_cols;            // accumulator columns: a power of two, 32 .. 512
    int share;                     // rows of a tile one CTA finishes
    int k_blocks;
    uint64_t tiles_r_inv, splits_inv;      // floor(2^32 / x) + 1: exact quotients of values below 65,536 without a division
};

// Fills in the derived members.
inline Geom make_geom(int M, int N, int K, int cg, int nt, int splits, int stages, int n_acc, bool half) {
    Geom g{M, N, K, nt, splits, stages, n_acc, half ? 1 : 0, 0, 0, 32, 0, 0, 0, 0};
    g.tiles_r = (M + nt - 1) / nt;
    g.n_tiles = g.tiles_r * ((N + cg * FT - 1) / (cg * FT));
    while (g.tmem_cols < (uint32_t)(((nt + 31) & ~31) * n_acc)) g.tmem_cols <<= 1;
    g.share = (nt + splits - 1) / splits;
    g.k_blocks = K / BK;
    g.tiles_r_inv = (1ull << 32) / (uint32_t)g.tiles_r + 1;
    g.splits_inv = (1ull << 32) / (uint32_t)splits + 1;
    return g;
}

template <bool DUAL> __host__ __device__ constexpr int x_bytes(int nt, int cg) { return (nt / cg) * BK * 2 * (DUAL ? 2 : 1); }
constexpr int SCALE_FLOATS = 2 * MAX_ROWS_TILE + 32;        // row scales of two tiles; rows behind the last are read, not used
constexpr int SMEM_FIXED = 1024 /*align*/ + 512 /*barriers*/ + 2 * SCALE_FLOATS * 4 /*row scales, row slots*/;
// Rows of a chunk of one epilogue group (unsplit tiles): NR for each of its four warps, or half of the tile when that is less.
__host__ __device__ constexpr int chunk_rows(int nt, int nr) { return nt >= 32 ? 4 * nr : 8; }
template <bool DUAL> __host__ __device__ constexpr int smem_bytes(int nt, int nr, int cg, int splits, int stages) {
    return stages * (W_BYTES + x_bytes<DUAL>(nt, cg)) + SMEM_FIXED + (splits == 1 ? 2 * chunk_rows(nt, nr) * FT * 4 : 0);
}

// ---------------------------------------------------------------------------------------------
// PTX wrappers this kernel needs beyond gemm_tc.cuh's
// ---------------------------------------------------------------------------------------------
__device__ __forceinline__ uint32_t cluster_rank() { uint32_t r; asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r)); return r; }
__device__ __forceinline__ uint32_t map_rank(uint32_t addr, uint32_t rank) {
    uint32_t r;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(rank));
    return r;
}
__device__ __forceinline__ void cluster_sync() {
    asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}
__device__ __forceinline__ float4 ld_cluster_f32x4(uint32_t addr) {
    float4 v;
    asm volatile("ld.shared::cluster.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "r"(addr) : "memory");
    return v;
}
__device__ __forceinline__ void mbar_arrive_cluster(uint32_t addr) {
    asm volatile("mbarrier.arrive.release.cluster.shared::cluster.b64 _, [%0];" ::"r"(addr) : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(uint32_t bar, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok) : "r"(bar), "r"(parity) : "memory");
    return ok != 0;
}
// Bounded wait; false when it gave up or another role raised the abort flag.  Only the first poll is inlined: the code of a
// launch runs once or twice, so its size is latency.
__device__ __noinline__ bool mbar_wait_slow(uint32_t bar, uint32_t parity, volatile int* abort_flag) {
    uint64_t began = 0;
#pragma unroll 1
    for (uint32_t it = 0; it < tc::WAIT_LIMIT; ++it) {
        if (mbar_try_wait(bar, parity)) return true;
        if ((it & 63u) == 63u) {
            uint64_t now;
            asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(now));
            if (began == 0) began = now;
            if (*abort_flag || now - began > WAIT_NS) return false;
            __nanosleep(64);
        }
    }
    return false;
}
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity, volatile int* abort_flag) {
    return mbar_try_wait(bar, parity) || mbar_wait_slow(bar, parity, abort_flag);
}
__device__ __forceinline__ bool mbar_test(uint32_t bar, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok) : "r"(bar), "r"(parity) : "memory");
    return ok != 0;
}
// The whole warp waits; the same answer in every lane.
__device__ __forceinline__ bool mbar_wait_warp(uint32_t bar, uint32_t parity, volatile int* abort_flag) {
    return __all_sync(0xffffffffu, mbar_wait(bar, parity, abort_flag)) != 0;
}
// True in one lane, the same one each time.  The producer and the MMA issuer run their loops with the whole warp and elect a lane
// where they issue: control and addresses stay in uniform registers, and the compiler knows that one thread issues.  A loop of
// lane 0 alone took 0.34 us per k-block whatever the tile, which bounded every pass (gate/up of 16 rows: 8.2 us for 24 k-blocks).
__device__ __forceinline__ bool elect_one() {
    uint32_t r;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "elect.sync _|p, 0xffffffff;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(r) :: "memory");
    return r != 0;
}
template <int CG> __device__ __forceinline__ void tmem_alloc(uint32_t dst, uint32_t cols) {
    if constexpr (CG == 1) {
        tc::tmem_alloc(dst, cols);
    } else {
        asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(dst), "r"(cols) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
    }
}
template <int CG> __device__ __forceinline__ void tmem_dealloc(uint32_t addr, uint32_t cols) {
    if constexpr (CG == 1) tc::tmem_dealloc(addr, cols);
    else asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(addr), "r"(cols) : "memory");
}
template <int CG> __device__ __forceinline__ void mma(uint32_t d, uint64_t a, uint64_t b, uint32_t idesc, uint32_t accumulate) {
    if constexpr (CG == 1) {
        tc::umma_bf16(d, a, b, idesc, accumulate);
    } else {
        const uint32_t zero = 0;
        asm volatile(
            "{\n\t.reg .pred p;\n\t"
            "setp.ne.b32 p, %4, 0;\n\t"
            "tcgen05.mma.cta_group::2.kind::f16 [%0], %1, %2, %3, {%5, %5, %5, %5, %5, %5, %5, %5}, p;\n\t}"
            ::"r"(d), "l"(a), "l"(b), "r"(idesc), "r"(accumulate), "r"(zero) : "memory");
    }
}
// Arrives on the barrier (in both CTAs of the pair for CG 2) once the MMAs issued so far have completed.
template <int CG> __device__ __forceinline__ void commit(uint32_t bar, uint32_t pair_mask) {
    if constexpr (CG == 1) {
        tc::umma_commit(bar);
    } else {
        const uint16_t m = (uint16_t)pair_mask;
        asm volatile("tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], %1;"
                     ::"r"(bar), "h"(m) : "memory");
    }
}
// A tile load; for CG 2 the completion is counted on the barrier of the pair's even CTA.
template <int CG> __device__ __forceinline__ void load_tile(uint32_t dst, const CUtensorMap* map, uint32_t bar, int c0, int c1) {
    if constexpr (CG == 1) {
        tma_load_2d(dst, map, bar, c0, c1);
    } else {
        asm volatile(
            "cp.async.bulk.tensor.2d.cta_group::2.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4}], [%2];"
            ::"r"(dst), "l"(map), "r"(bar), "r"(c0), "r"(c1) : "memory");
    }
}
// A weight tile that is read once.
template <int CG> __device__ __forceinline__ void load_weights_once(uint32_t dst, const CUtensorMap* map, uint32_t bar, int c0, int c1, uint64_t policy) {
    if constexpr (CG == 1) {
        asm volatile("cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes.L2::cache_hint [%0], [%1, {%3, %4}], [%2], %5;"
                     ::"r"(dst), "l"(map), "r"(bar), "r"(c0), "r"(c1), "l"(policy) : "memory");
    } else {
        asm volatile("cp.async.bulk.tensor.2d.cta_group::2.shared::cluster.global.mbarrier::complete_tx::bytes.L2::cache_hint [%0], [%1, {%3, %4}], [%2], %5;"
                     ::"r"(dst), "l"(map), "r"(bar), "r"(c0), "r"(c1), "l"(policy) : "memory");
    }
}
// 8 consecutive accumulator columns of this thread's TMEM lane
__device__ __forceinline__ void tmem_ld8(uint32_t taddr, float* v) {
    uint32_t r[8];
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]) : "r"(taddr) : "memory");
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
    for (int i = 0; i < 8; ++i) v[i] = __uint_as_float(r[i]);
}
// The epilogue threads meet; true when all of them got what they waited for.
__device__ __forceinline__ bool epi_all(bool ok) {
    uint32_t r;
    asm volatile(
        "{\n\t.reg .pred p, q;\n\t"
        "setp.ne.u32 p, %1, 0;\n\t"
        "barrier.cta.red.and.pred q, 1, %2, p;\n\t"
        "selp.u32 %0, 1, 0, q;\n\t}"
        : "=r"(r) : "r"(ok ? 1u : 0u), "n"(EPI_THREADS) : "memory");
    return r != 0;
}
__device__ __forceinline__ void group_sync(int group) {
    if (group == 0) asm volatile("bar.sync 2, %0;" ::"n"(EPI_THREADS / 2) : "memory");
    else asm volatile("bar.sync 3, %0;" ::"n"(EPI_THREADS / 2) : "memory");
}

// ---------------------------------------------------------------------------------------------
// Epilogues.  The accumulator has a feature per lane; a warp of the epilogue finishes whole rows of the tile, NR at a time,
// a lane holding the four consecutive features f0 + 4 lane .. + 3.  The values change hands through shared memory (staging
// memory of 4 NR rows, or the partial tiles when the cluster splits K).  Row-wise every access is a 16-byte vector and what
// belongs to a row is warp-uniform: about 45 instructions per row, where one feature per thread took 240, and the epilogue's
// instructions are what bounds large batches (two warps per scheduler beside the MMA).
//
// Code is kept short and without branches around arithmetic: a layer alternates between four such kernels, each running its
// epilogue a few times per launch, so instructions are instruction-cache misses first.
// ---------------------------------------------------------------------------------------------
struct Ctx {
    int lane;
    int f0;                 // first feature of the CTA's tile
    int f;                  // first of this lane's four features
    bool fv;                // they exist (the number of features is a multiple of 4, except for logits)
    int row0;               // first row of the tile
    const float* scale;     // per row of the tile: RMSNorm factor (ResNorm: power of two of the operand)
    const int* slot;        // where each row of the tile goes (epilogues with kSlots)
};
// Rows r + j * step, j < NR, of the tile; those below `end` exist.
struct Rows {
    int r, step, end;
    __device__ __forceinline__ int at(int j) const { return r + j * step; }
    __device__ __forceinline__ bool has(int j) const { return r + j * step < end; }
};

// The RMSNorm a ResNorm epilogue left unfinished.  It wrote half(h * gain * used) with a power of two per row and the row's sum of
// squares per feature tile; what the accumulators still lack is rstd / used, rstd = rsqrt(sum / d + eps).
//
// The power of two keeps the operand inside half's range whatever the size of the residual stream: it is 2^-4 / rms, rounded down,
// of the row one norm earlier (operand_scale), so the mantissas are those of half(h * gain) and the values are about 2^-4 times
// the normalised ones.  That leaves room for an rms that grows 2^10-fold within a sublayer at a gain of 8 and a row whose
// whole weight sits in one element, and for one that shrinks 2^6-fold (factor 2^10) before half's subnormals cost more than 2^-15 of
// the row's rms, an eighth of its rounding.  A row outside that room is not multiplied from its operand: the ResNorm tile that met an
// overflow leaves its sum with the sign set, row_factor answers with -rstd, and the consumer's epilogue takes the row's products
// from the residual stream itself (rescue_rows), rounded as the plain norm rounds them.
// Measured beside the same kernels without any of this: no case differs by more than two runs of one side (16 rows 10.51 -> 10.52 ms
// per eight steps, 351-token prefill 2.10 -> 2.06 ms); the same rescue per row inside the chunk loop cost 2 % at 16-351 rows.
struct RowScale {
    const float* ssq; int n, stride, d; float eps;      // ssq[n][stride]; n == 0: the operand is complete
    const float* used;             // per row: the power of two in the operand (nullptr: none).  ResNorm: the one to put there
    float* next;                   // per row: operand_scale of this norm, for the ResNorm that follows (or nullptr)
    const void* w; const float* h; const float* gain;      // weights, residual stream and gain for rescue_rows
};

constexpr float MAX_FACTOR = 1024.f;
// What the accumulators of `row` are to be multiplied with, or -rstd (never zero) when the operand does not hold the row.  The
// entries are added in order (every consumer gets the same bits), sixteen loads in flight at a time.
__device__ __forceinline__ float row_factor(const RowScale& r, int row, bool keep_next) {
    const float* __restrict__ p = r.ssq + row;
    const float u = r.used != nullptr ? r.used[row] : 1.f;
    float s = 0.f, low = 0.f;
#pragma unroll 1
    for (int e = 0; e < r.n; e += 16) {
        float x[16];
#pragma unroll
        for (int i = 0; i < 16; ++i) x[i] = e + i < r.n ? p[(size_t)(e + i) * r.stride] : 0.f;
#pragma unroll
        for (int i = 0; i < 16; ++i) { s += fabsf(x[i]); low = fminf(low, x[i]); }
    }
    const float rstd = rsqrtf(s / (float)r.d + r.eps);
    if (keep_next && r.next != nullptr) r.next[row] = operand_scale(rstd);
    if (r.used == nullptr) return rstd;
    const float f = rstd * __uint_as_float(0x7f000000u - __float_as_uint(u));       // 1 / u of a power of two
    return (low < 0.f) | !(f <= MAX_FACTOR) ? -fmaxf(rstd, 1e-37f) : f;             // (a NaN row too)
}

// Rows of a complete accumulator tile whose operand does not hold them (scale < 0, that is -rstd): this CTA's share k0 .. k1 of their
// products from the residual stream, the operand rounded as the plain norm rounds it (half, range-guarded), put in the place of
// the accumulators, and the factor left is 1.  All epilogue threads; a thread has a feature, its group every other row.
__device__ __forceinline__ void rescue_rows(const __half* __restrict__ w_row, const float* __restrict__ h, const float* __restrict__ gain, int K,
                                            int k0, int k1, int live, float* scale, uint32_t taddr, int group, int32_t* err) {
    int bad = 0;
#pragma unroll 1
    for (int p = group; p < live; p += 2) {
        const float rstd = -scale[p];
        if (!(rstd > 0.f)) continue;
        const float* __restrict__ h_row = h + (size_t)p * K;
        float y[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll 1
        for (int k = k0; k < k1; k += 4) {
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const float v = h_row[k + i] * rstd * gain[k + i];
                bad |= half_bad(v);
                const float a = __half2float(__float2half_rn(half_clamp(v)));
                if (w_row != nullptr) y[i] = fmaf(a, __half2float(w_row[k + i]), y[i]);
            }
        }
        const uint32_t sum = __float_as_uint((y[0] + y[1]) + (y[2] + y[3]));
        __syncwarp();
        asm volatile("tcgen05.st.sync.aligned.32x32b.x1.b32 [%0], {%1};" ::"r"(taddr + p), "r"(sum) : "memory");
    }
    asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
    if (bad) set_error(err, DEV_ERR_HALF_RANGE);
    tc_fence_before();
    asm volatile("bar.sync 1, %0;" ::"n"(EPI_THREADS) : "memory");
    tc_fence_after();
    for (int p = (int)threadIdx.x - 64; p < live; p += EPI_THREADS)
        if (scale[p] < 0.f) scale[p] = 1.f;
    asm volatile("bar.sync 1, %0;" ::"n"(EPI_THREADS) : "memory");
}

// A 16-bit GEMM operand: IEEE half (range-guarded), or bfloat16 with an optional rounding remainder.
struct Operand {
    void* p; void* lo;
};
__device__ __forceinline__ uint32_t pack_half(float a, float b) {
    const __half2 p = __floats2half2_rn(a, b);
    return *reinterpret_cast<const uint32_t*>(&p);
}
__device__ __forceinline__ uint32_t pack_half_clamped(float a, float b) { return pack_half(half_clamp(a), half_clamp(b)); }
__device__ __forceinline__ uint32_t pack_bf16(float a, float b) {
    const __nv_bfloat162 p = __floats2bfloat162_rn(a, b);
    return *reinterpret_cast<const uint32_t*>(&p);
}
__device__ __forceinline__ float bf16_rest(float v) { return v - __bfloat162float(__float2bfloat16_rn(v)); }
__device__ __forceinline__ float4 f4(float a, float b, float c, float d) { return make_float4(a, b, c, d); }
// Element products, two per instruction.
__device__ __forceinline__ float4 mul4(float4 a, float4 b) {
    float4 y;
    asm("{\n\t.reg .b64 a, b;\n\t"
        "mov.b64 a, {%4, %5}; mov.b64 b, {%8, %9}; mul.rn.f32x2 a, a, b; mov.b64 {%0, %1}, a;\n\t"
        "mov.b64 a, {%6, %7}; mov.b64 b, {%10, %11}; mul.rn.f32x2 a, a, b; mov.b64 {%2, %3}, a;\n\t}"
        : "=f"(y.x), "=f"(y.y), "=f"(y.z), "=f"(y.w)
        : "f"(a.x), "f"(a.y), "f"(a.z), "f"(a.w), "f"(b.x), "f"(b.y), "f"(b.z), "f"(b.w));
    return y;
}
// Largest magnitude, NaN when there is one: one instruction per value finds whether a batch fits half; only a batch that does
// not is clamped.
__device__ __forceinline__ float max_mag(float m, float v) {
    float r;
    asm("max.NaN.f32 %0, %1, %2;" : "=f"(r) : "f"(m), "f"(fabsf(v)));
    return r;
}
__device__ __forceinline__ bool beyond_half(float m) { return !(m <= HALF_MAX_F); }

// logits[row, f] = acc times the row's RMSNorm factor
struct EpiStore {
    static constexpr bool kDual = true;       // may take its activations as value + rounding remainder
    static constexpr bool kScaled = true;     // the operand may lack its norm's factor
    static constexpr bool kSplit = false;      // K may be split over a cluster
    static constexpr bool kSlots = false;
    static constexpr int NR = 4;
    float* C; int ld;
    RowScale rs;
    __device__ __forceinline__ void begin(const Ctx&) {}
    __device__ __forceinline__ void prefetch(const Ctx&, const Rows&) {}
    __device__ __forceinline__ void rows(const Ctx& c, const float4* x, const Rows& R, const Rows&) {
        float* dst = C + (size_t)(c.row0 + R.r) * ld + c.f;
        const size_t step = (size_t)R.step * ld;
        const bool vec = c.fv && (ld & 3) == 0;
#pragma unroll
        for (int j = 0; j < NR; ++j, dst += step) {
            const float s = c.scale[R.at(j)];
            const float4 y = f4(x[j].x * s, x[j].y * s, x[j].z * s, x[j].w * s);
            if (vec & R.has(j)) *reinterpret_cast<float4*>(dst) = y;
            if (((ld & 3) != 0) & R.has(j)) {            // a vocabulary that is no multiple of 4
                if (c.f < ld) dst[0] = y.x;
                if (c.f + 1 < ld) dst[1] = y.y;
                if (c.f + 2 < ld) dst[2] = y.z;
                if (c.f + 3 < ld) dst[3] = y.w;
            }
        }
    }
    __device__ __forceinline__ void end() {}
};

// g / (1 + e^-g) with the hardware exponential and reciprocal.  For g >= 0 good to 2^-21; below, the rounding of the exponent's argument
// counts |g| times, 2^-20 at g = -10.  The product is rounded to 2^-11 (half) or 2^-8 (bfloat16) next.  Against 64 bits the logits
// of the 1.5B and 8B shapes are as far off as with expf and a division (decode 16-560 rows: 0.991 to 1.005 times; a prefill's K and V
// with either are the same distance away to four digits).
__device__ __forceinline__ float silu(float g) {
    float e, r;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(e) : "f"(g * -1.4426950408889634f));
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(1.f + e));
    return g * r;
}

// act[row, j] = silu(gate_j) * up_j with gate / up rows interleaved (features 2j, 2j + 1) and the row's RMSNorm factor applied
template <bool HALF>
struct EpiSwiGLU {
    static constexpr bool kDual = false;       // may take its activations as value + rounding remainder
    static constexpr bool kScaled = HALF;
    static constexpr bool kSplit = false;      // K may be split over a cluster
    static constexpr bool kSlots = false;
    static constexpr int NR = 4;
    Operand act; int ld;
    RowScale rs;
    int32_t* err;
    bool bad;
    __device__ __forceinline__ void begin(const Ctx&) { bad = false; }
    __device__ __forceinline__ void prefetch(const Ctx&, const Rows&) {}
    __device__ __forceinline__ void rows(const Ctx& c, const float4* x, const Rows& R, const Rows&) {
        float a[NR], b[NR], m = 0.f;
        uint32_t y[NR];
#pragma unroll
        for (int j = 0; j < NR; ++j) {
            const float s = c.scale[R.at(j)];
            a[j] = silu(x[j].x * s) * (x[j].y * s);
            b[j] = silu(x[j].z * s) * (x[j].w * s);
            if (HALF) m = max_mag(max_mag(m, a[j]), b[j]);
            y[j] = HALF ? pack_half(a[j], b[j]) : pack_bf16(a[j], b[j]);
        }
        if (HALF && beyond_half(m)) {
#pragma unroll
            for (int j = 0; j < NR; ++j) {
                bad |= R.has(j) & (beyond_half(a[j]) | beyond_half(b[j]));      // rows behind the last hold anything
                y[j] = pack_half_clamped(a[j], b[j]);
            }
        }
        uint16_t* dst = reinterpret_cast<uint16_t*>(act.p) + (size_t)(c.row0 + R.r) * ld + (c.f >> 1);
        const size_t step = (size_t)R.step * ld;
#pragma unroll
        for (int j = 0; j < NR; ++j, dst += step)
            if (c.fv & R.has(j)) *reinterpret_cast<uint32_t*>(dst) = y[j];
    }
    __device__ __forceinline__ void end() { if (HALF && bad) set_error(err, DEV_ERR_HALF_RANGE); }
};

// h[row, f] += acc;  the next norm's operand a[row, f] = h * gain (half: times the row's power of two) WITHOUT its 1/rms factor;
// ssq[f / 128][row] = the tile's share of the row's sum of squares, with the sign set where the operand left half's range (see
// RowScale).  gain == nullptr: only the residual add.
template <bool HALF>
struct EpiResNorm {
    static constexpr bool kDual = !HALF;       // may take its activations as value + rounding remainder
    static constexpr bool kScaled = false;
    static constexpr bool kSplit = true;      // K may be split over a cluster (CTA pairs: never)
    static constexpr bool kSlots = false;
    static constexpr int NR = 4;
    float* h; int ld;
    const float* gain;
    Operand a;
    float* ssq; int ssq_stride;
    RowScale rs;                     // only `used`: the operand of these projections is complete
    float4 g, res[NR];
    __device__ __forceinline__ void begin(const Ctx& c) {
        g = gain != nullptr && c.fv ? *reinterpret_cast<const float4*>(gain + c.f) : f4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
        for (int j = 0; j < NR; ++j) res[j] = f4(0.f, 0.f, 0.f, 0.f);
    }
    __device__ __forceinline__ void prefetch(const Ctx& c, const Rows& R) {
        const float* src = h + (size_t)(c.row0 + R.r) * ld + c.f;
        const size_t step = (size_t)R.step * ld;
#pragma unroll
        for (int j = 0; j < NR; ++j, src += step)
            if (c.fv & R.has(j)) res[j] = *reinterpret_cast<const float4*>(src);
    }
    __device__ __forceinline__ void rows(const Ctx& c, const float4* x, const Rows& R, const Rows& next) {
        float4 v[NR];
#pragma unroll
        for (int j = 0; j < NR; ++j) v[j] = f4(x[j].x + res[j].x, x[j].y + res[j].y, x[j].z + res[j].z, x[j].w + res[j].w);
        prefetch(c, next);           // the residual of the next rows travels while these are finished
        const size_t at = (size_t)(c.row0 + R.r) * ld + c.f, step = (size_t)R.step * ld;
        float* dst = h + at;
#pragma unroll
        for (int j = 0; j < NR; ++j, dst += step)
            if (c.fv & R.has(j)) *reinterpret_cast<float4*>(dst) = v[j];
        if (gain == nullptr) return;
        uint16_t* op = reinterpret_cast<uint16_t*>(a.p) + at;
        float s[NR], m = 0.f;
        uint2 y[NR];
#pragma unroll
        for (int j = 0; j < NR; ++j) {
            s[j] = v[j].x * v[j].x + v[j].y * v[j].y + v[j].z * v[j].z + v[j].w * v[j].w;
            v[j] = mul4(v[j], g);
            if (HALF) { const float u = c.scale[R.at(j)]; v[j] = mul4(v[j], f4(u, u, u, u)); }
            if (HALF) m = max_mag(max_mag(max_mag(max_mag(m, v[j].x), v[j].y), v[j].z), v[j].w);
            y[j] = HALF ? make_uint2(pack_half(v[j].x, v[j].y), pack_half(v[j].z, v[j].w)) : make_uint2(pack_bf16(v[j].x, v[j].y), pack_bf16(v[j].z, v[j].w));
        }
        uint32_t sign = 0;               // of the sum this lane stores: set when its row does not fit half
        if (HALF && __any_sync(0xffffffffu, beyond_half(m))) {
            uint32_t over = 0;           // bit j: row j (rows behind the last hold anything and store nothing)
#pragma unroll
            for (int j = 0; j < NR; ++j) {
                if (c.fv & (beyond_half(v[j].x) | beyond_half(v[j].y) | beyond_half(v[j].z) | beyond_half(v[j].w))) over |= 1u << j;
                y[j] = make_uint2(pack_half_clamped(v[j].x, v[j].y), pack_half_clamped(v[j].z, v[j].w));
            }
            sign = __reduce_or_sync(0xffffffffu, over) >> (c.lane >> 3) << 31;
        }
#pragma unroll
        for (int j = 0; j < NR; ++j, op += step)
            if (c.fv & R.has(j)) *reinterpret_cast<uint2*>(op) = y[j];
        if (!HALF && a.lo != nullptr) {
            op = reinterpret_cast<uint16_t*>(a.lo) + at;
#pragma unroll
            for (int j = 0; j < NR; ++j, op += step)
                if (c.fv & R.has(j))
                    *reinterpret_cast<uint2*>(op) = make_uint2(pack_bf16(bf16_rest(v[j].x), bf16_rest(v[j].y)), pack_bf16(bf16_rest(v[j].z), bf16_rest(v[j].w)));
        }
        // four row sums over the warp: two exchanges leave a lane with one row, three more add it up
        const bool u16 = c.lane & 16, u8 = c.lane & 8;
        float p = (u16 ? s[2] : s[0]) + __shfl_xor_sync(0xffffffffu, u16 ? s[0] : s[2], 16);
        float q = (u16 ? s[3] : s[1]) + __shfl_xor_sync(0xffffffffu, u16 ? s[1] : s[3], 16);
        float t = (u8 ? q : p) + __shfl_xor_sync(0xffffffffu, u8 ? p : q, 8);
        t += __shfl_xor_sync(0xffffffffu, t, 4);
        t += __shfl_xor_sync(0xffffffffu, t, 2);
        t += __shfl_xor_sync(0xffffffffu, t, 1);
        const int j = c.lane >> 3;                       // lane bits 4 and 3 chose the row
        if (HALF) t = __uint_as_float(__float_as_uint(t) ^ sign);
        if (((c.lane & 7) == 0) & R.has(j)) ssq[(size_t)(c.f0 / FT) * ssq_stride + c.row0 + R.at(j)] = t;
    }
    __device__ __forceinline__ void end() {}
};

// QKV projection, head_dim 128 = one feature tile per head: RMSNorm factor of the row, bias, per-head RMSNorm of q and k,
// RoPE, q to its buffer, K / V to the row's KV slot (all IEEE half) -- the arithmetic of qkv_post_kernel.
struct EpiQkv {
    static constexpr bool kDual = true;       // may take its activations as value + rounding remainder
    static constexpr bool kScaled = true;
    static constexpr bool kSplit = true;      // K may be split over a cluster (CTA pairs: never)
    static constexpr bool kSlots = true;
    static constexpr int NR = 2;       // rotary factors of the rows in hand and of the next ones take registers
    int Hq, Hkv, layer;
    const float* bias;                 // [(Hq + 2 Hkv) * 128] or nullptr
    const float* q_gain;               // [128] or nullptr (no QK-norm)
    const float* k_gain;
    float eps;
    const float2* rope;                // [rows, 64] (cos, sin)
    RowGeom geo;
    KvArena prompt_arena, suffix_arena;
    __half* q_out;
    RowScale rs;
    int32_t* err;
    float4 b, g, cs[NR][2];            // bias, gain; rotary factors of the rows in hand
    __half *base_s, *base_p;           // this head's plane of the two arenas; q: its column of the q buffer (base_s)
    int pitch;                         // elements from one slot (q: row) to the next
    bool is_q, turn, norm, bad;
    __device__ __forceinline__ void begin(const Ctx& c) {
        const int head = c.f0 / FT;
        bad = false;
        is_q = head < Hq;
        turn = head < Hq + Hkv;                          // V rows are not rotated
        const float* gain = is_q ? q_gain : (turn ? k_gain : nullptr);
        norm = gain != nullptr;
        b = bias != nullptr && c.fv ? *reinterpret_cast<const float4*>(bias + c.f) : f4(0.f, 0.f, 0.f, 0.f);
        g = norm ? *reinterpret_cast<const float4*>(gain + 4 * c.lane) : f4(1.f, 1.f, 1.f, 1.f);
        const int64_t plane = ((int64_t)layer * 2 + (turn ? 0 : 1)) * Hkv + (turn ? head - Hq : head - Hq - Hkv);
        base_s = (is_q ? q_out + (size_t)head * FT : reinterpret_cast<__half*>(suffix_arena.base) + plane * suffix_arena.n_slots * FT) + 4 * c.lane;
        base_p = reinterpret_cast<__half*>(prompt_arena.base) + plane * prompt_arena.n_slots * FT + 4 * c.lane;
        pitch = is_q ? Hq * FT : FT;
#pragma unroll
        for (int j = 0; j < NR; ++j) cs[j][0] = cs[j][1] = f4(1.f, 0.f, 1.f, 0.f);
    }
    // 2 * slot + (1: suffix arena or q buffer, 0: prompt arena), negative: nowhere.  Taken once per tile by a thread per row: the
    // lookup per row and chunk put two dependent loads into every chunk (the projection over 10,184 rows: 184 -> 147 us).
    __device__ __forceinline__ int slot_of(int row) const {
        if (is_q) return 2 * row + 1;
        const int64_t w = geo.wslot[row];
        return (int)(2 * w) + (geo.warena[row] ? 1 : 0);
    }
    __device__ __forceinline__ void prefetch(const Ctx& c, const Rows& R) {
#pragma unroll
        for (int j = 0; j < NR; ++j) {
            if (c.fv & R.has(j) & turn) {
                const float4* p = reinterpret_cast<const float4*>(rope + (size_t)(c.row0 + R.at(j)) * 64) + 2 * (c.lane & 15);
                cs[j][0] = p[0];
                cs[j][1] = p[1];
            }
        }
    }
    __device__ __forceinline__ void rows(const Ctx& c, const float4* x, const Rows& R, const Rows& next) {
        const float sign = c.lane < 16 ? -1.f : 1.f;
        float4 v[NR];
        uint2 y[NR];
        float m = 0.f;
#pragma unroll
        for (int j = 0; j < NR; ++j) {
            const float s = c.scale[R.at(j)];
            v[j] = f4(x[j].x * s + b.x, x[j].y * s + b.y, x[j].z * s + b.z, x[j].w * s + b.w);
        }
        if (norm) {
            float ss[NR];
#pragma unroll
            for (int j = 0; j < NR; ++j) ss[j] = v[j].x * v[j].x + v[j].y * v[j].y + v[j].z * v[j].z + v[j].w * v[j].w;
#pragma unroll
            for (int o = 16; o > 0; o >>= 1)
#pragma unroll
                for (int j = 0; j < NR; ++j) ss[j] += __shfl_xor_sync(0xffffffffu, ss[j], o);
#pragma unroll
            for (int j = 0; j < NR; ++j) {
                const float r = rsqrtf(ss[j] / (float)FT + eps);
                v[j] = f4(v[j].x * r * g.x, v[j].y * r * g.y, v[j].z * r * g.z, v[j].w * r * g.w);
            }
        }
#pragma unroll
        for (int j = 0; j < NR; ++j) {
            // rotary partner of feature i < 64 is i + 64: sixteen lanes on
            const float4 o = f4(__shfl_xor_sync(0xffffffffu, v[j].x, 16), __shfl_xor_sync(0xffffffffu, v[j].y, 16),
                                __shfl_xor_sync(0xffffffffu, v[j].z, 16), __shfl_xor_sync(0xffffffffu, v[j].w, 16));
            const float4 p = cs[j][0], q = cs[j][1];
            v[j] = f4(v[j].x * p.x + sign * (o.x * p.y), v[j].y * p.z + sign * (o.y * p.w), v[j].z * q.x + sign * (o.z * q.y), v[j].w * q.z + sign * (o.w * q.w));
            m = max_mag(max_mag(max_mag(max_mag(m, v[j].x), v[j].y), v[j].z), v[j].w);
            y[j] = make_uint2(pack_half(v[j].x, v[j].y), pack_half(v[j].z, v[j].w));
        }
        if (beyond_half(m)) {
#pragma unroll
            for (int j = 0; j < NR; ++j) {
                bad |= R.has(j) & (beyond_half(v[j].x) | beyond_half(v[j].y) | beyond_half(v[j].z) | beyond_half(v[j].w));
                y[j] = make_uint2(pack_half_clamped(v[j].x, v[j].y), pack_half_clamped(v[j].z, v[j].w));
            }
        }
        prefetch(c, next);
#pragma unroll
        for (int j = 0; j < NR; ++j) {
            const int slot = c.slot[R.at(j)];
            if (c.fv & R.has(j) & (slot >= 0)) *reinterpret_cast<uint2*>((slot & 1 ? base_s : base_p) + (int64_t)(slot >> 1) * pitch) = y[j];
        }
    }
    __device__ __forceinline__ void end() { if (bad) set_error(err, DEV_ERR_HALF_RANGE); }
};

// ---------------------------------------------------------------------------------------------
// Kernel
// ---------------------------------------------------------------------------------------------
__device__ __forceinline__ int quotient(int x, uint64_t inverse) { return (int)(((uint64_t)(uint32_t)x * inverse) >> 32); }

// ONCE: one row tile, every weight is read once per pass (with a choice at run time in the loop the 8B shape lost 2 %, large prefills 1 %).
template <int CG, bool DUAL, bool ONCE, class Epi>
__global__ void __launch_bounds__(THREADS, 1)
gemm_wt_kernel(const __grid_constant__ CUtensorMap map_w, const __grid_constant__ CUtensorMap map_x,
               const __grid_constant__ CUtensorMap map_x_lo, const StepDesc* __restrict__ sd, const Geom G, Epi epi, int32_t* err) {
    extern __shared__ uint8_t smem_raw[];
    uint8_t* tiles = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
    const int X1 = (G.nt / CG) * BK * 2, stage_bytes = W_BYTES + X1 * (DUAL ? 2 : 1);
    float* scale = reinterpret_cast<float*>(tiles + G.stages * stage_bytes);
    int* slots = reinterpret_cast<int*>(scale + SCALE_FLOATS);
    uint64_t* bars = reinterpret_cast<uint64_t*>(slots + SCALE_FLOATS);
    float* staging = reinterpret_cast<float*>(bars + 64);
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars + 2 * MAX_STAGES + 4);
    volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);
    volatile int* outside_tile = abort_flag + 1;       // [2] the last tile (plus one) of this parity that has rows its operand does not hold

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const bool splitting = Epi::kSplit && CG == 1 && G.splits > 1;
    const uint32_t rank = cluster_rank();
    const uint32_t peer = CG == 2 ? rank & 1u : 0u, leader = rank - peer;
    const int split = (int)rank / CG;
    const uint32_t full0 = smem_u32(bars), empty0 = full0 + 8 * MAX_STAGES, tfull0 = empty0 + 8 * MAX_STAGES, tempty0 = tfull0 + 16;
    const uint32_t tiles_u32 = smem_u32(tiles);
    const int acc_cols = (G.nt + 31) & ~31;
    const uint32_t tmem_cols = G.tmem_cols;

    const int cluster = quotient(CG == 2 ? blockIdx.x >> 1 : blockIdx.x, G.splits_inv), n_clusters = quotient(CG == 2 ? gridDim.x >> 1 : gridDim.x, G.splits_inv);
    const int tiles_r = G.tiles_r, n_tiles = G.n_tiles;
    const int kb0 = quotient(split * G.k_blocks, G.splits_inv), kb1 = quotient((split + 1) * G.k_blocks, G.splits_inv);
    // tile t: rows fastest, so that clusters running together share a weight tile
    auto place = [&](int t, int& f0, int& r0) {
        const int ft = quotient(t, G.tiles_r_inv);
        f0 = (ft * CG + (int)peer) * FT;
        r0 = (t - ft * tiles_r) * G.nt;
    };

    if (threadIdx.x == 0) {
#pragma unroll 1
        for (int s = 0; s < G.stages; ++s) { mbar_init(full0 + 8 * s, 1); mbar_init(empty0 + 8 * s, 1); }
        mbar_init(tfull0, 1); mbar_init(tfull0 + 8, 1);
        mbar_init(tempty0, CG * EPI_WARPS); mbar_init(tempty0 + 8, CG * EPI_WARPS);
        *abort_flag = 0;
        outside_tile[0] = outside_tile[1] = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    }
    if (CG == 2) cluster_sync();                    // the peer's loads are counted on the leader's barriers
    const uint32_t full_at = CG == 2 ? map_rank(full0, leader) : full0;

    if (warp == 0) {
        __syncwarp();
        if (lane == 1) {
            asm volatile("prefetch.tensormap [%0];" ::"l"(&map_x) : "memory");
            if (DUAL) asm volatile("prefetch.tensormap [%0];" ::"l"(&map_x_lo) : "memory");
        }
        asm volatile("bar.arrive 4, %0;" ::"n"(THREADS) : "memory");      // the barriers exist; the others meet here, this warp goes on
        // ---------------- TMA producer ----------------
        // Before the wait for the previous kernel the weight tile of every stage is requested, and nothing else.
        {
            bool ok = true;
            const uint64_t policy = ONCE ? policy_evict_first() : 0;
            auto weights = [&](uint32_t dst, uint32_t bar, int c0, int c1) {
                if constexpr (ONCE) load_weights_once<CG>(dst, &map_w, bar, c0, c1, policy);
                else load_tile<CG>(dst, &map_w, bar, c0, c1);
            };
            int tile = cluster, kb = kb0, f0, r0;
            place(tile, f0, r0);
            const int stages = G.stages;
            int s = 0;
#pragma unroll 1
            for (; s < stages && tile < n_tiles; ++s) {
                if (elect_one()) {
                    if (peer == 0) mbar_arrive_expect_tx(full0 + 8 * s, CG * stage_bytes);
                    weights(tiles_u32 + s * stage_bytes, full_at + 8 * s, kb * BK, f0);
                }
                if (++kb == kb1) { kb = kb0; tile += n_clusters; place(tile, f0, r0); }
            }
            int ahead = s;                          // stages whose weights are requested
            grid_dep_wait();                        // the activations are the previous kernel's output
            grid_dep_launch_dependents();           // the next kernel may start: whatever runs two kernels back has finished
            tile = cluster; kb = kb0;
            place(tile, f0, r0);
            uint32_t phase = 1;
            s = 0;
#pragma unroll 1
            while (tile < n_tiles) {
                const uint32_t at = tiles_u32 + s * stage_bytes, bar = full_at + 8 * s;
                const bool requested = ahead > 0;
                --ahead;
                if (!requested && !mbar_wait_warp(empty0 + 8 * s, phase, abort_flag)) { ok = false; break; }
                if (elect_one()) {
                    if (!requested) {
                        if (peer == 0) mbar_arrive_expect_tx(full0 + 8 * s, CG * stage_bytes);
                        weights(at, bar, kb * BK, f0);
                    }
                    const int r = r0 + (int)peer * (G.nt / CG);
                    load_tile<CG>(at + W_BYTES, &map_x, bar, kb * BK, r);
                    if (DUAL) load_tile<CG>(at + W_BYTES + X1, &map_x_lo, bar, kb * BK, r);
                }
                if (++s == stages) { s = 0; phase ^= 1u; }
                if (++kb == kb1) { kb = kb0; tile += n_clusters; place(tile, f0, r0); }
            }
            if (!ok && lane == 0) { *abort_flag = 1; set_error(err, DEV_ERR_WAIT_TIMEOUT); }
        }
        __syncwarp();
    }
    uint32_t tmem_base = 0;
    if (warp != 0) {
        if (warp == 1) tmem_alloc<CG>(smem_u32(tmem_slot), tmem_cols);
        tc_fence_before();
        asm volatile("bar.sync 4, %0;" ::"n"(THREADS) : "memory");
        tc_fence_after();
        tmem_base = *tmem_slot;
        grid_dep_wait();                            // residual stream, row geometry, buffers to be overwritten
    }
    if (warp == 1) {
        if (peer == 0) {
            // ---------------- MMA issuer ----------------
            const uint32_t idesc = tc::make_idesc(FT * CG, G.nt, G.half != 0);
            const uint32_t pair = 3u << leader;
            const uint64_t dw0 = tc::make_smem_desc(tiles_u32);          // of stage 0; only the address field (16-byte units) changes
            const uint32_t step = stage_bytes >> 4;
            uint32_t stage = 0, phase = 0, acc = 0, acc_phase = 0;
            bool ok = true;
#pragma unroll 1
            for (int t = cluster; t < n_tiles && ok; t += n_clusters) {
                if (!mbar_wait_warp(tempty0 + 8 * acc, acc_phase ^ 1u, abort_flag)) { ok = false; break; }
                tc_fence_after();
                const uint32_t d = tmem_base + acc * acc_cols;
                uint32_t add = 0;
                bool ready = false;                                  // the next stage was seen full while this one was issued
#pragma unroll 1
                for (int kb = kb0; kb < kb1; ++kb) {
                    if (!__all_sync(0xffffffffu, ready) && !mbar_wait_warp(full0 + 8 * stage, phase, abort_flag)) { ok = false; break; }
                    tc_fence_after();
                    const uint32_t here = stage;
                    if (++stage == (uint32_t)G.stages) { stage = 0; phase ^= 1u; }
                    ready = mbar_test(full0 + 8 * stage, phase);
                    if (elect_one()) {
                        const uint64_t dw = dw0 + here * step, dx = dw + (W_BYTES >> 4);
#pragma unroll
                        for (int kk = 0; kk < BK / 16; ++kk) mma<CG>(d, dw + 2 * kk, dx + 2 * kk, idesc, kk > 0 ? 1u : add);
                        if (DUAL) {
                            const uint64_t dl = dx + (X1 >> 4);
#pragma unroll
                            for (int kk = 0; kk < BK / 16; ++kk) mma<CG>(d, dw + 2 * kk, dl + 2 * kk, idesc, 1u);
                        }
                        commit<CG>(empty0 + 8 * here, pair);
                    }
                    add = 1;
                }
                if (!ok) break;
                if (elect_one()) commit<CG>(tfull0 + 8 * acc, pair);
                if (++acc == (uint32_t)G.n_acc) { acc = 0; acc_phase ^= 1u; }
            }
            if (!ok && lane == 0) { *abort_flag = 1; set_error(err, DEV_ERR_WAIT_TIMEOUT); }
        }
        __syncwarp();
    } else if (warp > 1) {
        // ---------------- epilogue ----------------
        const int tid = threadIdx.x - 64;
        const int quarter = warp & 3, group = (warp - 2) >> 2;
        Ctx c;
        c.lane = lane;
        const int lane128 = quarter * 32 + lane;
        const int m_live = sd != nullptr ? min(G.M, sd->n_rows) : G.M;
        const uint32_t tempty_at = CG == 2 ? map_rank(tempty0, leader) : tempty0;
        const int share = G.share;                               // rows of a tile this CTA finishes (all, or its share of a split)
        constexpr int NR = Epi::NR;
        constexpr bool kRescue = Epi::kScaled && !DUAL;
        const int cw = chunk_rows(G.nt, NR);
        float* stage = staging + group * cw * FT;
        uint32_t acc = 0, acc_phase = 0;
        bool ok = true;
        int turn = 0;
#pragma unroll 1
        for (int t = cluster; t < n_tiles; t += n_clusters, turn ^= 1) {
            // a warp may be one tile ahead of another (not more: all meet once per tile), so the row scales alternate
            float* tile_scale = scale + turn * MAX_ROWS_TILE;
            c.scale = tile_scale;
            c.slot = slots + turn * MAX_ROWS_TILE;
            place(t, c.f0, c.row0);
            c.f = c.f0 + 4 * lane; c.fv = c.f < G.N;
            const int live = max(0, min(G.nt, m_live - c.row0));
            const int begin = min(live, split * share), end = min(live, begin + share);
            // The rows of this warp.  Whole tile: the groups take chunks of cw rows in turn, a warp every fourth row of a chunk.
            // Split tile: a warp takes every eighth row of the share.
            int at = splitting ? begin + warp - 2 : group * cw;
            const int advance = splitting ? 8 * NR : 2 * cw;
            auto rows_of = [&](int p) { return splitting ? Rows{p, 8, end} : Rows{p + quarter, 4, min(live, p + cw)}; };
            epi.begin(c);
            epi.prefetch(c, rows_of(at));
            if (tid < live) {                                     // at most 256 rows: a thread each
                const RowScale& r = epi.rs;
                const int row = c.row0 + tid;
                const float s = r.n > 0 ? row_factor(r, row, c.f0 == 0 && split == 0) : (r.used != nullptr ? r.used[row] : 1.f);
                tile_scale[tid] = s;
                if (kRescue && s < 0.f) outside_tile[turn] = t + 1;
                if constexpr (Epi::kSlots) slots[turn * MAX_ROWS_TILE + tid] = epi.slot_of(row);
            }
            // the accumulator is complete, the row scales are in place
            ok = epi_all(mbar_wait(tfull0 + 8 * acc, acc_phase, abort_flag));
            if (!ok) break;
            tc_fence_after();
            const uint32_t taddr = tmem_base + ((uint32_t)(quarter * 32) << 16) + acc * acc_cols;
            if constexpr (kRescue)
                if (outside_tile[turn] == t + 1)
                    rescue_rows(c.f0 + lane128 < G.N ? reinterpret_cast<const __half*>(epi.rs.w) + (size_t)(c.f0 + lane128) * G.K : nullptr,
                                epi.rs.h + (size_t)c.row0 * G.K, epi.rs.gain, G.K, kb0 * BK, kb1 * BK, live, tile_scale, taddr, group, err);
            if (splitting) {
                // leave the partial tile in this CTA's shared memory (the operand ring is drained) for the cluster
                float* part = reinterpret_cast<float*>(tiles) + lane128;
#pragma unroll 1
                for (int p0 = group * 8; p0 < live; p0 += 16) {
                    float v[8];
                    tmem_ld8(taddr + p0, v);
#pragma unroll
                    for (int i = 0; i < 8; ++i) part[(p0 + i) * FT] = v[i];
                }
                cluster_sync();
            }
            const int stop = splitting ? end : live;
#pragma unroll 1
            for (; at < stop; at += advance) {
                const Rows R = rows_of(at);
                float4 x[NR];
                if (splitting) {
                    // the K ranges' partial sums of these rows, added in range order; all ranges of two rows are in flight together (a
                    // read of another CTA's memory takes a quarter of a microsecond: one range after another took 1.2 us with six and
                    // 1.8 us with eight, eight decode steps of 16 rows 10.51 -> 9.93 ms, of 237 rows 20.06 -> 19.73)
#pragma unroll
                    for (int j = 0; j < NR; ++j) x[j] = f4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
                    for (int j = 0; j < NR; j += 2) {
                        if (!R.has(j)) break;
                        const bool both = R.has(j + 1);
                        const uint32_t at_row = tiles_u32 + (uint32_t)(R.at(j) * FT + 4 * lane) * 4;
                        float4 y[MAX_SPLITS][2];
#pragma unroll
                        for (int s = 0; s < MAX_SPLITS; ++s) {
                            y[s][0] = y[s][1] = f4(0.f, 0.f, 0.f, 0.f);
                            if (s < G.splits) {
                                const uint32_t from = map_rank(at_row, (uint32_t)s);
                                y[s][0] = ld_cluster_f32x4(from);
                                if (both) y[s][1] = ld_cluster_f32x4(from + 8 * FT * 4);
                            }
                        }
#pragma unroll
                        for (int s = 0; s < MAX_SPLITS; ++s)
#pragma unroll
                            for (int i = 0; i < 2; ++i) {
                                x[j + i] = f4(x[j + i].x + y[s][i].x, x[j + i].y + y[s][i].y, x[j + i].z + y[s][i].z, x[j + i].w + y[s][i].w);
                            }
                    }
                } else {
                    group_sync(group);                           // the previous chunk has been read
#pragma unroll 1
                    for (int p0 = 0; p0 < cw; p0 += 8) {
                        float v[8];
                        tmem_ld8(taddr + at + p0, v);
#pragma unroll
                        for (int i = 0; i < 8; ++i) stage[(p0 + i) * FT + lane128] = v[i];
                    }
                    group_sync(group);
#pragma unroll
                    for (int j = 0; j < NR; ++j) x[j] = *reinterpret_cast<const float4*>(stage + ((quarter + 4 * j) & (cw - 1)) * FT + 4 * lane);
                }
                epi.rows(c, x, R, rows_of(at + advance));
            }
            if (!splitting) {
                tc_fence_before();
                __syncwarp();
                if (lane == 0) { if (CG == 2) mbar_arrive_cluster(tempty_at + 8 * acc); else mbar_arrive(tempty0 + 8 * acc); }
            }
            epi.end();
            if (++acc == (uint32_t)G.n_acc) { acc = 0; acc_phase ^= 1u; }
        }
        if (!ok) {
            if (lane == 0) { *abort_flag = 1; set_error(err, DEV_ERR_WAIT_TIMEOUT); }
            if (splitting) cluster_sync();                    // the meeting point this role would have reached
        }
    }
    if (splitting && warp < 2) cluster_sync();                // partial tiles are in place
    tc_fence_before();
    __syncthreads();
    if (*abort_flag) {
#pragma unroll 1
        for (int i = 0; i < 2000; ++i) __nanosleep(1000);        // copies in flight land before the shared memory is released
        __syncthreads();
    }
    if (splitting || CG == 2) cluster_sync();                 // nobody leaves while a peer reads its memory or signals it
    if (warp == 1) {
        __syncwarp();
        tc_fence_after();
        tmem_dealloc<CG>(tmem_base, tmem_cols);
    }
}

template <int CG, bool DUAL, class Epi>
inline cudaError_t configure() {
    const cudaError_t e = cudaFuncSetAttribute(gemm_wt_kernel<CG, DUAL, false, Epi>, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024);
    return e != cudaSuccess ? e : cudaFuncSetAttribute(gemm_wt_kernel<CG, DUAL, true, Epi>, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024);
}

// map_w: boxes of 128 weight rows; map_x (and map_x_lo when DUAL): boxes of nt / CG activation rows.
template <int CG, bool DUAL, class Epi>
inline cudaError_t launch(cudaStream_t st, const CUtensorMap& map_w, const CUtensorMap& map_x, const CUtensorMap& map_x_lo,
                          const StepDesc* sd, const Geom& g, int n_clusters, Epi epi, int32_t* err, bool programmatic) {
    cudaLaunchConfig_t cfg;
    memset(&cfg, 0, sizeof(cfg));
    cfg.gridDim = dim3((unsigned)(n_clusters * CG * g.splits)); cfg.blockDim = dim3(THREADS);
    cfg.dynamicSmemBytes = smem_bytes<DUAL>(g.nt, Epi::NR, CG, g.splits, g.stages); cfg.stream = st;
    cudaLaunchAttribute attr[2];
    int n = 0;
    if (CG * g.splits > 1) {
        attr[n].id = cudaLaunchAttributeClusterDimension;
        attr[n].val.clusterDim.x = CG * g.splits; attr[n].val.clusterDim.y = 1; attr[n].val.clusterDim.z = 1;
        ++n;
    }
    if (programmatic) {
        attr[n].id = cudaLaunchAttributeProgrammaticStreamSerialization;
        attr[n].val.programmaticStreamSerializationAllowed = 1;
        ++n;
    }
    cfg.attrs = attr; cfg.numAttrs = n;
    return cudaLaunchKernelEx(&cfg, g.tiles_r == 1 ? gemm_wt_kernel<CG, DUAL, true, Epi> : gemm_wt_kernel<CG, DUAL, false, Epi>, map_w, map_x, map_x_lo, sd, g, epi, err);
}

}  // namespace wt
}  // namespace pc

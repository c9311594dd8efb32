// Shared-prefix decode attention for bf16 models, on tensor cores, with K/V tiles staged by TMA.
//
// The K/V arenas are viewed as 2-D tensors of 16-bit elements (IEEE half) [planes * n_slots, head_dim]; a tile of TP consecutive
// slots is fetched as head_dim/64 boxes of [TP rows x 64 columns] with the 128-byte swizzle, which makes
// the ldmatrix reads below bank-conflict free.
//
//   attn_group_kernel   one CTA per (64 query rows of a group, KV head).  The query rows are all live
//                       rollouts of the group times the query heads sharing the KV head, so the group's
//                       prompt K/V is read once per 64 query rows instead of once per rollout
//                       (S = Q K^T and O = P V as m16n8k16 MMAs, online softmax in registers).  Every
//                       query row carries its own number of visible prompt slots, which also makes this
//                       the causal prefill kernel.  Decode: leaves (m, l, unnormalised O) per query row
//                       in scratch.  Prefill: writes the normalised output.
//   attn_suffix_kernel  teams of two or four warps claim (rollout, KV head) items and stream their suffix K/V through
//                       3-stage TMA rings, beside the shared-prefix kernel.  Positions sit on the MMA M axis (S^T = K Q^T,
//                       O^T = V^T P^T), so the 6-8 query heads fill the N = 8 axis and no MMA work is
//                       padded; P is transposed between the two MMAs with movmatrix.  A team merges its warps' shares
//                       and the shared-prefix records into the attention output.
//
// Scores are kept in the log2 domain (scaled by log2(e) / sqrt(head_dim)) so that exp2f is the only
// transcendental.  Waits on mbarriers are bounded (see gemm_tc.cuh).
#pragma once

#include <cuda_fp16.h>

#include "common.cuh"
#include "gemm_tc.cuh"
#include "kernels_basic.cuh"

namespace pc {
namespace am {

using tc::mbar_arrive;
using tc::mbar_arrive_expect_tx;
using tc::mbar_init;
using tc::mbar_wait;
using tc::smem_u32;
using tc::tma_load_2d;

__device__ __forceinline__ void ldsm_x4(uint32_t addr, uint32_t& r0, uint32_t& r1, uint32_t& r2, uint32_t& r3) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0, %1, %2, %3}, [%4];"
                 : "=r"(r0), "=r"(r1), "=r"(r2), "=r"(r3) : "r"(addr));
}
__device__ __forceinline__ void ldsm_x4_t(uint32_t addr, uint32_t& r0, uint32_t& r1, uint32_t& r2, uint32_t& r3) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0, %1, %2, %3}, [%4];"
                 : "=r"(r0), "=r"(r1), "=r"(r2), "=r"(r3) : "r"(addr));
}
__device__ __forceinline__ uint32_t movmatrix_t(uint32_t a) {
    uint32_t d;
    asm volatile("movmatrix.sync.aligned.m8n8.trans.b16 %0, %1;" : "=r"(d) : "r"(a));
    return d;
}
__device__ __forceinline__ void mma_bf16(float* c, uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t b0, uint32_t b1) {
    asm volatile(
        "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, {%0, %1, %2, %3};"
        : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
        : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}
// Both attention products take IEEE half operands: q, K and V are stored as half (see qkv_post_kernel), P is rounded to half
__device__ __forceinline__ void mma_f16(float* c, uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t b0, uint32_t b1) {
    asm volatile(
        "mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, {%0, %1, %2, %3};"
        : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
        : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}
__device__ __forceinline__ uint32_t pack_f16(float lo, float hi) {
    const __half2 p = __floats2half2_rn(lo, hi);
    return *reinterpret_cast<const uint32_t*>(&p);
}
// The same for values that leave the kernel as a GEMM operand: out-of-range values are saturated and reported.
__device__ __forceinline__ uint32_t pack_f16_guard(float lo, float hi, int32_t* err) {
    return pack_f16(half_guard(lo, err), half_guard(hi, err));
}
__device__ __forceinline__ uint32_t pack_bf16(float lo, float hi) {
    const __nv_bfloat162 p = __floats2bfloat162_rn(lo, hi);
    return *reinterpret_cast<const uint32_t*>(&p);
}
// exp2 that maps -inf to 0 without producing NaN when both operands are -inf
__device__ __forceinline__ float exp2_safe(float x, float m) { return m == -INFINITY ? 0.f : exp2f(x - m); }

// K and V of one tile of consecutive slots in one request: the arena as [K|V][64-dim half][row][64], row counted from plane 0
// (make_kv_tile_map).
__device__ __forceinline__ void tma_load_kv(uint32_t dst, const CUtensorMap* map, uint32_t bar, int row) {
    asm volatile(
        "cp.async.bulk.tensor.4d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4, %3, %3}], [%2];"
        ::"r"(dst), "l"(map), "r"(bar), "r"(0), "r"(row)
        : "memory");
}
// The same for tiles that are read once.
__device__ __forceinline__ void tma_load_kv_once(uint32_t dst, const CUtensorMap* map, uint32_t bar, int row, uint64_t policy) {
    asm volatile(
        "cp.async.bulk.tensor.4d.shared::cluster.global.mbarrier::complete_tx::bytes.L2::cache_hint [%0], [%1, {%3, %4, %3, %3}], [%2], %5;"
        ::"r"(dst), "l"(map), "r"(bar), "r"(0), "r"(row), "l"(policy)
        : "memory");
}
// Byte offset of (row r, dim d) (d a multiple of 8) in a swizzled tile of ROWS rows: boxes of 64 dims,
// rows of 128 bytes, 16-byte chunk index XORed with (r mod 8).
template <int ROWS>
__device__ __forceinline__ uint32_t tile_off(int r, int d) {
    return (uint32_t)((d >> 6) * (ROWS * 128) + r * 128 + ((((d & 63) >> 3) ^ (r & 7)) << 4));
}

// Prefix part of the attention, per (row, query head): running max (log2 domain), sum, unnormalised output.
// When a group has few query rows its prompt is cut into n_parts ranges handled by different CTAs; every range
// leaves its own record and the suffix kernel merges all of them.
struct PrefixPartial {
    float* m;               // [n_parts][stride]
    float* l;               // [n_parts][stride]
    float* o;               // [n_parts][stride * head_dim]
    int n_parts;
    size_t stride;          // rows capacity * Hq
    int32_t* done;          // CTAs of the shared-prefix kernel that have left their records (a hint), or nullptr
};
constexpr int MAX_PREFIX_PARTS = 8, MAX_MERGED_PARTS = 4;      // (the second where attn_suffix_kernel merges)
constexpr int MAX_RECORDS = MAX_PREFIX_PARTS > MAX_MERGED_PARTS + 1 ? MAX_PREFIX_PARTS : MAX_MERGED_PARTS + 1;

// ---------------------------------------------------------------------------------------------
// Group (shared-prefix / causal-prefill) kernel
// ---------------------------------------------------------------------------------------------
constexpr int G_THREADS = 128;      // 4 warps x 16 query rows; two such CTAs share an SM
constexpr int G_QROWS = 64;
constexpr int G_TK = 64;            // KV positions per stage
constexpr int G_STAGES = 3;
template <int HD> constexpr int group_smem_bytes() { return G_STAGES * 2 * G_TK * HD * 2 + 1024 + 128; }

template <int HD, bool FINAL>
__global__ void __launch_bounds__(G_THREADS, 2)
attn_group_kernel(const __grid_constant__ CUtensorMap kv_map, const StepDesc* __restrict__ sd, int64_t n_slots, int Hq, int Hkv,
                  int layer, const __nv_bfloat16* __restrict__ q, const int32_t* __restrict__ group_row_start, RowGeom g,
                  float scale_log2, PrefixPartial part, __nv_bfloat16* __restrict__ out, __nv_bfloat16* __restrict__ out_lo,
                  int32_t* err) {
    constexpr int KS = HD / 16;          // k-steps of Q K^T
    constexpr int NT = G_TK / 8;         // position n-tiles per stage
    constexpr int DT = HD / 8;           // dim n-tiles of the output
    constexpr int TILE_BYTES = G_TK * HD * 2;
    const int grp = blockIdx.z, kvh = blockIdx.y;
    // Decode steps launch this kernel as a programmatic dependent of the QKV post-processing: the step descriptor, the row
    // geometry and the prompt K/V were all written before that kernel started, so the first K/V tiles are requested while
    // it still runs; q is read after grid_dep_wait().  Every CTA waits on every path (a grid that ended before the kernel
    // it depends on would let the next kernel start too early).  The prefill form reads K/V of this very pass: it waits first.
    if (FINAL) grid_dep_wait();
    if (grp >= sd->n_groups) { grid_dep_wait(); return; }
    // group_row_start holds this pass's groups from entry 0 on (decode: the copy in the workspace)
    const int row0 = group_row_start[grp], n_rows = group_row_start[grp + 1] - row0;
    const int n_rep = Hq / Hkv;
    const int n_parts = FINAL ? 1 : part.n_parts;
    const int q_tiles = gridDim.x / n_parts;
    const int my_part = blockIdx.x / q_tiles;
    const int q0 = (blockIdx.x - my_part * q_tiles) * G_QROWS;
    if (q0 >= n_rows * n_rep) { grid_dep_wait(); return; }

    extern __shared__ uint8_t smem_raw[];
    uint8_t* tiles = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
    uint64_t* bars = reinterpret_cast<uint64_t*>(tiles + G_STAGES * 2 * TILE_BYTES);
    __shared__ int s_abort;
    __shared__ int s_maxlen;
    const uint32_t tiles_u32 = smem_u32(tiles), full0 = smem_u32(bars), empty0 = full0 + 8 * G_STAGES;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;

    if (threadIdx.x == 0) {
        for (int s = 0; s < G_STAGES; ++s) { mbar_init(full0 + 8 * s, 1); mbar_init(empty0 + 8 * s, G_THREADS / 32); }
        s_abort = 0;
        s_maxlen = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    }
    __syncthreads();

    // Decode: the rows of a group share their prompt, so the visible prompt length is known from the group's first
    // row and the first K/V tiles are requested before anything else is loaded.  Prefill: every row sees its own
    // prefix; the longest one of the tile is found below.
    const int64_t kv_start = g.p_start[row0];
    const int64_t krow0 = (((int64_t)layer * 2 + 0) * Hkv + kvh) * n_slots + kv_start;
    const int64_t vrow0 = (((int64_t)layer * 2 + 1) * Hkv + kvh) * n_slots + kv_start;
    auto issue = [&](int tile, int stage) {
        const uint32_t kb = tiles_u32 + stage * 2 * TILE_BYTES, vb = kb + TILE_BYTES;
        mbar_arrive_expect_tx(full0 + 8 * stage, 2 * TILE_BYTES);
#pragma unroll
        for (int b = 0; b < HD / 64; ++b) {
            tma_load_2d(kb + b * (G_TK * 128), &kv_map, full0 + 8 * stage, b * 64, (int)(krow0 + (int64_t)tile * G_TK));
            tma_load_2d(vb + b * (G_TK * 128), &kv_map, full0 + 8 * stage, b * 64, (int)(vrow0 + (int64_t)tile * G_TK));
        }
    };
    int max_len = 0, tile0 = 0, n_tiles = 0;
    auto set_range = [&](int len) {
        max_len = len;
        const int n_tiles_all = (max_len + G_TK - 1) / G_TK;
        const int tiles_per_part = (n_tiles_all + n_parts - 1) / n_parts;
        tile0 = my_part * tiles_per_part;                                // this CTA covers tiles [tile0, tile0 + n_tiles)
        n_tiles = max(0, min(n_tiles_all, tile0 + tiles_per_part) - tile0);
    };
    if (!FINAL) {
        set_range(g.p_len[row0]);
        if (threadIdx.x == 0)
            for (int t = 0; t < G_STAGES && t < n_tiles; ++t) issue(tile0 + t, t);
        grid_dep_wait();
    }

    // this thread's two query rows: qr = q0 + warp*16 + lane/4 (+8); query row qr = (rollout row qr / n_rep, head qr % n_rep)
    int lim[2], grow[2], head[2];
#pragma unroll
    for (int i = 0; i < 2; ++i) {
        const int qr = q0 + warp * 16 + (lane >> 2) + 8 * i;
        const bool valid = qr < n_rows * n_rep;
        grow[i] = valid ? row0 + qr / n_rep : -1;
        head[i] = kvh * n_rep + (valid ? qr % n_rep : 0);
        lim[i] = valid ? g.p_len[grow[i]] : 0;
        if (!FINAL) lim[i] = min(lim[i], max_len);
    }
    if (FINAL) {
        int mx = max(lim[0], lim[1]);
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) mx = max(mx, __shfl_xor_sync(0xffffffffu, mx, o));
        if (lane == 0) atomicMax(&s_maxlen, mx);
    }
    // Q fragments (A operand), straight from global memory
    uint32_t qa[KS][4];
#pragma unroll
    for (int ks = 0; ks < KS; ++ks) {
#pragma unroll
        for (int i = 0; i < 2; ++i) {
            uint32_t lo = 0, hi = 0;
            if (grow[i] >= 0) {
                const __nv_bfloat16* p = q + ((size_t)grow[i] * Hq + head[i]) * HD + ks * 16 + (lane & 3) * 2;
                lo = *reinterpret_cast<const uint32_t*>(p);
                hi = *reinterpret_cast<const uint32_t*>(p + 8);
            }
            qa[ks][i] = lo;          // a0 (row), a1 (row + 8)
            qa[ks][2 + i] = hi;      // a2, a3: dims + 8
        }
    }
    if (FINAL) {
        __syncthreads();
        set_range(s_maxlen);
        if (threadIdx.x == 0)
            for (int t = 0; t < G_STAGES && t < n_tiles; ++t) issue(tile0 + t, t);
    }

    float o[DT][4];
#pragma unroll
    for (int t = 0; t < DT; ++t) { o[t][0] = o[t][1] = o[t][2] = o[t][3] = 0.f; }
    float mrow[2] = {-INFINITY, -INFINITY}, lrow[2] = {0.f, 0.f};
    bool ok = true;

    for (int lt = 0; lt < n_tiles; ++lt) {
        const int tile = tile0 + lt;
        const int stage = lt % G_STAGES;
        const uint32_t phase = (uint32_t)(lt / G_STAGES) & 1u;
        if (!mbar_wait(full0 + 8 * stage, phase, &s_abort)) { ok = false; break; }
        const uint32_t kb = tiles_u32 + stage * 2 * TILE_BYTES, vb = kb + TILE_BYTES;
        // S = Q K^T for 64 positions
        float s[NT][4];
#pragma unroll
        for (int nt = 0; nt < NT; ++nt) { s[nt][0] = s[nt][1] = s[nt][2] = s[nt][3] = 0.f; }
#pragma unroll
        for (int ks = 0; ks < KS; ++ks) {
#pragma unroll
            for (int np = 0; np < NT / 2; ++np) {
                const int mat = lane >> 3;
                const int r = np * 16 + (lane & 7) + ((mat >> 1) << 3), d = ks * 16 + ((mat & 1) << 3);
                uint32_t b0, b1, b2, b3;
                ldsm_x4(kb + tile_off<G_TK>(r, d), b0, b1, b2, b3);
                mma_f16(s[2 * np], qa[ks][0], qa[ks][1], qa[ks][2], qa[ks][3], b0, b1);
                mma_f16(s[2 * np + 1], qa[ks][0], qa[ks][1], qa[ks][2], qa[ks][3], b2, b3);
            }
        }
        // mask, online softmax (rows lane/4 and lane/4 + 8; a row lives in the four lanes of a quad)
        const int pos0 = tile * G_TK + (lane & 3) * 2;
        float bmax[2] = {-INFINITY, -INFINITY};
#pragma unroll
        for (int nt = 0; nt < NT; ++nt) {
#pragma unroll
            for (int c = 0; c < 4; ++c) {
                const int pos = pos0 + nt * 8 + (c & 1);
                const float v = pos < lim[c >> 1] ? s[nt][c] * scale_log2 : -INFINITY;
                s[nt][c] = v;
                bmax[c >> 1] = fmaxf(bmax[c >> 1], v);
            }
        }
        float corr[2];
#pragma unroll
        for (int i = 0; i < 2; ++i) {
            bmax[i] = fmaxf(bmax[i], __shfl_xor_sync(0xffffffffu, bmax[i], 1));
            bmax[i] = fmaxf(bmax[i], __shfl_xor_sync(0xffffffffu, bmax[i], 2));
            const float mnew = fmaxf(mrow[i], bmax[i]);
            corr[i] = exp2_safe(mrow[i], mnew);
            mrow[i] = mnew;
            lrow[i] *= corr[i];
        }
#pragma unroll
        for (int t = 0; t < DT; ++t) { o[t][0] *= corr[0]; o[t][1] *= corr[0]; o[t][2] *= corr[1]; o[t][3] *= corr[1]; }
        uint32_t pa[NT / 2][4];
#pragma unroll
        for (int nt = 0; nt < NT; ++nt) {
            float p[4];
#pragma unroll
            for (int c = 0; c < 4; ++c) { p[c] = exp2_safe(s[nt][c], mrow[c >> 1]); lrow[c >> 1] += p[c]; }
            pa[nt >> 1][(nt & 1) * 2 + 0] = pack_f16(p[0], p[1]);
            pa[nt >> 1][(nt & 1) * 2 + 1] = pack_f16(p[2], p[3]);
        }
        // rows of V beyond the longest visible prefix of this CTA may be uninitialised memory: their P is 0, but
        // 0 * NaN would poison the sum, so positions >= max_len are never multiplied (k-steps past it are skipped)
        const int valid_in_tile = min(G_TK, max_len - tile * G_TK);
#pragma unroll
        for (int kk = 0; kk < G_TK / 16; ++kk) {
            if (kk * 16 >= valid_in_tile) break;
            const bool ragged = kk * 16 + 16 > valid_in_tile;      // block-uniform
#pragma unroll
            for (int dp = 0; dp < DT / 2; ++dp) {
                const int mat = lane >> 3;
                const int r = kk * 16 + (lane & 7) + ((mat & 1) << 3), d = dp * 16 + ((mat >> 1) << 3);
                uint32_t b0, b1, b2, b3;
                ldsm_x4_t(vb + tile_off<G_TK>(r, d), b0, b1, b2, b3);
                if (ragged) {
                    // zero the V values of positions >= valid_in_tile: after the transposing load a thread holds
                    // positions kk*16 + (lane%4)*2 + {0,1} in b0/b2 and + 8 in b1/b3
                    const int p = kk * 16 + (lane & 3) * 2;
                    const uint32_t m_lo = (p < valid_in_tile ? 0x0000ffffu : 0u) | (p + 1 < valid_in_tile ? 0xffff0000u : 0u);
                    const uint32_t m_hi = (p + 8 < valid_in_tile ? 0x0000ffffu : 0u) | (p + 9 < valid_in_tile ? 0xffff0000u : 0u);
                    b0 &= m_lo; b2 &= m_lo; b1 &= m_hi; b3 &= m_hi;
                }
                mma_f16(o[2 * dp], pa[kk][0], pa[kk][1], pa[kk][2], pa[kk][3], b0, b1);
                mma_f16(o[2 * dp + 1], pa[kk][0], pa[kk][1], pa[kk][2], pa[kk][3], b2, b3);
            }
        }
        __syncwarp();
        if (lane == 0) mbar_arrive(empty0 + 8 * stage);
        if (threadIdx.x == 0 && lt + G_STAGES < n_tiles) {
            if (!mbar_wait(empty0 + 8 * stage, phase, &s_abort)) { ok = false; break; }
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            issue(tile + G_STAGES, stage);
        }
    }
    if (!ok) { s_abort = 1; set_error(err, DEV_ERR_WAIT_TIMEOUT); }

    // row sums live spread over the quad
#pragma unroll
    for (int i = 0; i < 2; ++i) {
        lrow[i] += __shfl_xor_sync(0xffffffffu, lrow[i], 1);
        lrow[i] += __shfl_xor_sync(0xffffffffu, lrow[i], 2);
    }
#pragma unroll
    for (int i = 0; i < 2; ++i) {
        if (grow[i] < 0) continue;
        const size_t rh = (size_t)grow[i] * Hq + head[i];
        if (FINAL) {
            const float inv = lrow[i] > 0.f ? 1.f / lrow[i] : 0.f;
#pragma unroll
            for (int t = 0; t < DT; ++t) {
                const float y0 = o[t][2 * i] * inv, y1 = o[t][2 * i + 1] * inv;
                const size_t at = rh * HD + t * 8 + (lane & 3) * 2;
                if (out_lo == nullptr) {         // the output projection takes IEEE half operands
                    *reinterpret_cast<uint32_t*>(out + at) = pack_f16_guard(y0, y1, err);
                } else {
                    *reinterpret_cast<uint32_t*>(out + at) = pack_bf16(y0, y1);
                    // rounding remainder, consumed as a second bf16 operand by the output projection
                    *reinterpret_cast<uint32_t*>(out_lo + at) = pack_bf16(y0 - __bfloat162float(__float2bfloat16_rn(y0)),
                                                                          y1 - __bfloat162float(__float2bfloat16_rn(y1)));
                }
            }
        } else {
            const size_t ph = (size_t)my_part * part.stride + rh;
            if ((lane & 3) == 0) { part.m[ph] = mrow[i]; part.l[ph] = lrow[i]; }
            if (n_tiles > 0) {          // an empty range leaves (m, l) = (-inf, 0); its output is never read
#pragma unroll
                for (int t = 0; t < DT; ++t)
                    *reinterpret_cast<float2*>(part.o + ph * HD + t * 8 + (lane & 3) * 2) = make_float2(o[t][2 * i], o[t][2 * i + 1]);
            }
        }
    }
    if (s_abort) {      // let copies still in flight land before the shared memory is released
        for (int i = 0; i < 2000; ++i) __nanosleep(1000);
    }
    __syncthreads();
}

// ---------------------------------------------------------------------------------------------
// Suffix kernel
// ---------------------------------------------------------------------------------------------
// A warp's tile -- ldmatrix, two rounds of MMAs, the softmax between them -- is one chain of about 900 clocks for 8 KB, so a warp
// of its own per scheduler cannot keep up with HBM (4 warps, 32 positions at a time: 4.35 TB/s at 237 rows x 512); two per
// scheduler can.  192 KB of tiles are in flight per SM, in two CTAs, so that one fits beside a CTA of the shared-prefix kernel.
constexpr int S_WARPS = 4;
constexpr int S_CTAS = 2;           // per SM
constexpr int S_TP = 16;            // positions per stage: one MMA tile
constexpr int S_STAGES = 3;
constexpr int S_SLOTS = 8;          // items a CTA knows of: the one in hand and those its rings reach into
template <int HD> __host__ __device__ constexpr int suffix_smem_need() { return S_WARPS * (S_STAGES * 2 * S_TP * HD * 2 + 8 * HD * 4) + 768; }
constexpr int SUFFIX_SMEM_BYTES = 113 * 1024;      // half of an SM's 228 KB less the reserved KB
static_assert(suffix_smem_need<128>() <= SUFFIX_SMEM_BYTES, "suffix buffers");

// One tile of 16 positions: K fragments against the heads' queries, online softmax, V.  loaded() is called once the tile is in
// registers (its ring slot is free).
template <int HD, class Loaded>
__device__ __forceinline__ void suffix_tile(uint32_t kb, uint32_t vb, int lane, int valid, float scale_log2, const uint32_t (&qb)[HD / 16][2],
                                            float (&o)[HD / 16][4], float (&mh)[2], float (&lh)[2], Loaded loaded) {
    constexpr int KS = HD / 16, DT = HD / 16;
    const int mat = lane >> 3;
    // All fragments of the tile first: the loads are in flight together, and the ring slot is free again before any
    // arithmetic.  (Interleaved, every MMA waits for its own ldmatrix.)
    uint32_t ka[KS][4], va[DT][4];
#pragma unroll
    for (int ks = 0; ks < KS; ++ks) {
        const int r = (lane & 7) + ((mat & 1) << 3), d = ks * 16 + ((mat >> 1) << 3);
        ldsm_x4(kb + tile_off<S_TP>(r, d), ka[ks][0], ka[ks][1], ka[ks][2], ka[ks][3]);
    }
#pragma unroll
    for (int dt = 0; dt < DT; ++dt) {
        const int r = (lane & 7) + ((mat >> 1) << 3), d = dt * 16 + ((mat & 1) << 3);
        ldsm_x4_t(vb + tile_off<S_TP>(r, d), va[dt][0], va[dt][1], va[dt][2], va[dt][3]);
    }
    loaded();
    // S^T = K Q^T : 16 positions on M, heads on N; two chains so that consecutive MMAs do not wait for one another
    float s[4] = {0.f, 0.f, 0.f, 0.f}, s2[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
    for (int ks = 0; ks < KS; ++ks) mma_f16((ks & 1) ? s2 : s, ka[ks][0], ka[ks][1], ka[ks][2], ka[ks][3], qb[ks][0], qb[ks][1]);
    // mask + per-head tile max (a head's column is spread over the 8 lanes sharing lane % 4)
    float bmax[2] = {-INFINITY, -INFINITY};
#pragma unroll
    for (int c = 0; c < 4; ++c) {
        const int pos = (lane >> 2) + ((c >> 1) << 3);
        s[c] = pos < valid ? (s[c] + s2[c]) * scale_log2 : -INFINITY;
        bmax[c & 1] = fmaxf(bmax[c & 1], s[c]);
    }
    float corr[2];
#pragma unroll
    for (int i = 0; i < 2; ++i) {
        bmax[i] = fmaxf(bmax[i], __shfl_xor_sync(0xffffffffu, bmax[i], 4));
        bmax[i] = fmaxf(bmax[i], __shfl_xor_sync(0xffffffffu, bmax[i], 8));
        bmax[i] = fmaxf(bmax[i], __shfl_xor_sync(0xffffffffu, bmax[i], 16));
        const float mnew = fmaxf(mh[i], bmax[i]);          // finite: a tile has a position
        corr[i] = exp2f(mh[i] - mnew);
        mh[i] = mnew;
        lh[i] *= corr[i];
    }
#pragma unroll
    for (int t = 0; t < DT; ++t) { o[t][0] *= corr[0]; o[t][1] *= corr[1]; o[t][2] *= corr[0]; o[t][3] *= corr[1]; }
    // O^T += V^T P^T; P^T fragments come from S^T through movmatrix
    float p[4];
#pragma unroll
    for (int c = 0; c < 4; ++c) { p[c] = exp2f(s[c] - mh[c & 1]); lh[c & 1] += p[c]; }
    const uint32_t b0 = movmatrix_t(pack_f16(p[0], p[1])), b1 = movmatrix_t(pack_f16(p[2], p[3]));
    if (valid < S_TP) {
        // slots past the rollout's last token may be uninitialised: zero them (0 * NaN = NaN).  After the transposing
        // load a thread holds positions (lane%4)*2 + {0,1} in registers 0 and 1, + 8 in 2 and 3.
        const int pp = (lane & 3) * 2;
        const uint32_t m_lo = (pp < valid ? 0x0000ffffu : 0u) | (pp + 1 < valid ? 0xffff0000u : 0u);
        const uint32_t m_hi = (pp + 8 < valid ? 0x0000ffffu : 0u) | (pp + 9 < valid ? 0xffff0000u : 0u);
#pragma unroll
        for (int dt = 0; dt < DT; ++dt) { va[dt][0] &= m_lo; va[dt][1] &= m_lo; va[dt][2] &= m_hi; va[dt][3] &= m_hi; }
    }
#pragma unroll
    for (int dt = 0; dt < DT; ++dt) mma_f16(o[dt], va[dt][0], va[dt][1], va[dt][2], va[dt][3], b0, b1);
}
// A warp's share of an item: m8 / l8 [8 heads], obuf [8 heads][HD] unnormalised.
template <int HD>
__device__ __forceinline__ void suffix_finish(int lane, const float (&o)[HD / 16][4], const float (&mh)[2], float (&lh)[2], float* m8, float* l8, float* obuf) {
    constexpr int DT = HD / 16;
    // reduce the per-thread partial sums of each head over the 8 lanes sharing lane % 4
#pragma unroll
    for (int i = 0; i < 2; ++i) {
        lh[i] += __shfl_xor_sync(0xffffffffu, lh[i], 4);
        lh[i] += __shfl_xor_sync(0xffffffffu, lh[i], 8);
        lh[i] += __shfl_xor_sync(0xffffffffu, lh[i], 16);
    }
    if (lane < 4) {
        m8[lane * 2] = mh[0]; m8[lane * 2 + 1] = mh[1];
        l8[lane * 2] = lh[0]; l8[lane * 2 + 1] = lh[1];
    }
    // O^T fragment (dims dt*16 + lane/4 (+8), heads (lane%4)*2 + {0,1}) -> obuf[head][dim]
#pragma unroll
    for (int dt = 0; dt < DT; ++dt) {
        const int d = dt * 16 + (lane >> 2), hh = (lane & 3) * 2;
        obuf[hh * HD + d] = o[dt][0];
        obuf[(hh + 1) * HD + d] = o[dt][1];
        obuf[hh * HD + d + 8] = o[dt][2];
        obuf[(hh + 1) * HD + d + 8] = o[dt][3];
    }
}

// Normalises and stores one (row, query head): IEEE half, or bf16 with its rounding remainder (second operand of the O projection).
// A lane holds dims lane * HD/32 ...
template <int HD>
__device__ __forceinline__ void store_attention(int lane, size_t rh, float* acc, float denom, __nv_bfloat16* __restrict__ out,
                                                __nv_bfloat16* __restrict__ out_lo, int32_t* err) {
    constexpr int EPL = HD / 32;
    const float inv = denom > 0.f ? 1.f / denom : 0.f;
    float lo[EPL];
#pragma unroll
    for (int e = 0; e < EPL; ++e) {
        acc[e] *= inv;
        lo[e] = acc[e] - __bfloat162float(__float2bfloat16_rn(acc[e]));
    }
    __nv_bfloat16* dst = out + rh * HD + lane * EPL;
    if (out_lo == nullptr) {                 // the output projection takes IEEE half operands: no remainder needed
        if (EPL == 4) *reinterpret_cast<uint2*>(dst) = make_uint2(pack_f16_guard(acc[0], acc[1], err), pack_f16_guard(acc[EPL - 2], acc[EPL - 1], err));
        else *reinterpret_cast<uint32_t*>(dst) = pack_f16_guard(acc[0], acc[1], err);
        return;
    }
    __nv_bfloat16* dst_lo = out_lo + rh * HD + lane * EPL;
    if (EPL == 4) {
        *reinterpret_cast<uint2*>(dst) = make_uint2(pack_bf16(acc[0], acc[1]), pack_bf16(acc[EPL - 2], acc[EPL - 1]));
        *reinterpret_cast<uint2*>(dst_lo) = make_uint2(pack_bf16(lo[0], lo[1]), pack_bf16(lo[EPL - 2], lo[EPL - 1]));
    } else {
        *reinterpret_cast<uint32_t*>(dst) = pack_bf16(acc[0], acc[1]);
        *reinterpret_cast<uint32_t*>(dst_lo) = pack_bf16(lo[0], lo[1]);
    }
}

// Suffix attention of batches with more than two (row, KV head) items per SM (smaller ones take attn_suffix_team_kernel).  A team of
// T warps takes an item at a time, each warp every T-th tile, and merges the warps' shares and the item's shared-prefix records
// by their log-sum-exp:  M = max m_i,  out = sum_i O_i 2^(m_i - M) / sum_i l_i 2^(m_i - M).  T: suffix_team_warps in pc_api.cu.
//
// The items are claimed as the teams get to them.  A CTA that starts beside the shared-prefix kernel (113 KB each) streams while
// that one computes and takes more of them than one that has to wait for its place; an item that is finished before the shared-prefix
// records are there is left as a record too and merged at the end.  A warp's ring runs on into the next item while its team merges.
//
// What bounds it: HBM, but for the first and the last few microseconds.  237 rows x 512 (118 MB, 18 us at the copy rate): from the end of the
// projection before 33 us with the shared-prefix kernel inside (12 of them); first tile at 4, last item begun at 24.  With one
// 192 KB CTA per SM, which had to wait for the shared-prefix CTAs, and a suffix per warp cut into ranges, merged between two ranges by the last
// warp (5-13 us, every warp at the same time), eight steps took: 237 rows x 512 19.8 -> 19.1 ms, 336 x 900 30.6 -> 29.0, 2,048 x 512 101.2 -> 95.5.
// Halving the last items so that the CTAs end closer together cost more (records, fences, a second merge) than it gave.
struct SuffixWork {
    int32_t* next;              // the layer's next item; 0 at the start of a step
    int32_t* link;              // [rows capacity * Hkv]: items put off, a list per CTA
    int prefix_ctas;            // value of part.done once the shared-prefix records are there
    __nv_bfloat16* out;
    __nv_bfloat16* out_lo;
};
struct SuffixItem {
    int64_t krow;               // first K row of the suffix in the arena's (plane, slot) rows
    int item, n;                // (row, KV head), or -1: there are no more; suffix length
};

template <int HD, int T>
__global__ void __launch_bounds__(S_WARPS * 32, S_CTAS)
attn_suffix_kernel(const __grid_constant__ CUtensorMap kv_map, const StepDesc* __restrict__ sd, int64_t n_slots, int Hq, int Hkv,
                   int layer, const __nv_bfloat16* __restrict__ q, RowGeom g, float scale_log2, PrefixPartial part, SuffixWork wk, int32_t* err) {
    constexpr int KS = HD / 16;                   // k-steps of K Q^T
    constexpr int DT = HD / 16;                   // 16-dim m-tiles of O^T
    constexpr int EPL = HD / 32;
    constexpr int H = 8 / T;                      // heads of an item a warp merges
    constexpr int TILE_BYTES = S_TP * HD * 2;
    constexpr int RING_BYTES = S_STAGES * 2 * TILE_BYTES;
    extern __shared__ uint8_t smem_raw[];
    uint8_t* base = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, team = warp / T, me = warp % T;
    float* obufs = reinterpret_cast<float*>(base + S_WARPS * RING_BYTES);              // [warp][8 heads][HD]
    float* mls = obufs + S_WARPS * 8 * HD;                                              // [warp][m of 8 heads, l of 8 heads]
    float *obuf = obufs + team * T * 8 * HD, *ml = mls + team * T * 16;                // of the team
    SuffixItem* all_slots = reinterpret_cast<SuffixItem*>(mls + S_WARPS * 16);
    SuffixItem* slots = all_slots + team * S_SLOTS;
    uint64_t* all_bars = reinterpret_cast<uint64_t*>(all_slots + S_WARPS / T * S_SLOTS);
    uint64_t* bars = all_bars + warp * S_STAGES;
    // of the team: a wait ran out, items entered in the slots so far, the shared-prefix records are there
    volatile int* abort_flag = reinterpret_cast<volatile int*>(all_bars + S_WARPS * S_STAGES) + team * 4;
    volatile int *known = abort_flag + 1, *records_there = abort_flag + 2;
    auto team_sync = [&]() { asm volatile("bar.sync %0, %1;" ::"r"(1 + team), "n"(T * 32) : "memory"); };
    if ((int)(base - smem_raw) + suffix_smem_need<HD>() > SUFFIX_SMEM_BYTES) {        // (the shared memory window is not where it should be)
        if (threadIdx.x == 0) set_error(err, DEV_ERR_GROUP_RANGE);
        grid_dep_wait();
        return;
    }
    // A team's last warp, which has the fewest tiles, claims: lane 0 asks for the item after the one in hand while that one's last tiles are
    // requested, and enters it when the ring gets there, between two tiles or behind the last.  (Short items were claimed as far ahead as the
    // ring reaches, by the warp that has their one tile: the CTAs that start first took four, the others one, and a claim and its look-up, 1.4 us,
    // stood in front of each tile.  Eight steps of 64 groups with prompts of 16-64: 320 rows x 2 slots 17.9 -> 16.9 ms, 512 x 16 22.3 -> 21.3.)
    const bool claims = me == T - 1;
    int claim = 0, asked = 1;                     // asked: claims so far, at most two more than the items done
    auto request = [&]() { if (lane == 0) claim = atomicAdd(wk.next, 1); };
    if (claims) request();
    const uint32_t tiles_u32 = smem_u32(base + warp * RING_BYTES), full0 = smem_u32(bars);
    const int n_rep = Hq / Hkv, n_items = sd->n_rows * Hkv;

    if (threadIdx.x == 32) asm volatile("prefetch.tensormap [%0];" ::"l"(&kv_map) : "memory");
    if (claims && lane == 0) { *abort_flag = 0; *known = 0; *records_there = part.done == nullptr; }
    if (lane == 0) {
        for (int s = 0; s < S_STAGES; ++s) mbar_init(full0 + 8 * s, 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    }
    auto enter = [&](int seq) {                   // slot of the seq-th item of this team
        int item = __shfl_sync(0xffffffffu, claim, 0), n = 0;
        int64_t start = 0;
        while (item < n_items) {
            const int row = item / Hkv;
            n = g.s_len[row]; start = g.s_start[row];
            if (n > 0) break;                     // (a row that was refused has no suffix and its outputs are not defined)
            request();
            item = __shfl_sync(0xffffffffu, claim, 0);
        }
        if (lane == 0) {
            const int kvh = item % Hkv;
            slots[seq % S_SLOTS] = SuffixItem{((int64_t)layer * 2 * Hkv + kvh) * n_slots + start, item < n_items ? item : -1, n};
            __threadfence_block();
            *known = seq + 1;
        }
        __syncwarp();
    };
    if (claims) enter(0);
    __syncthreads();

    // item in hand; producer cursor: item p_seq, tile p_tile (tracked identically by every lane; lane 0 issues)
    const uint64_t policy = policy_evict_first();
    int seq = 0, p_seq = 0, p_tile = me, p_tiles = 0, issued = 0, consumed = 0;
    int64_t p_krow = 0;
    bool p_open = false;
    auto refill = [&](bool may_enter) {           // may_enter: the warp that claims may wait for its claim
        while (issued - consumed < S_STAGES) {
            if (claims && asked == seq + 1 && (p_seq > seq || (p_open && p_tile + 2 * T >= p_tiles))) { request(); ++asked; }
            if (!p_open) {
                if (p_seq > seq + 1) return;
                if (p_seq >= __shfl_sync(0xffffffffu, *known, 0)) {
                    if (!claims || !may_enter) return;       // again at the next tile or item
                    enter(p_seq);
                }
                __syncwarp();
                const SuffixItem s = slots[p_seq % S_SLOTS];
                if (s.item < 0) return;
                p_krow = s.krow; p_tiles = (s.n + S_TP - 1) / S_TP; p_tile = me;
                p_open = true;
            }
            if (p_tile >= p_tiles) { ++p_seq; p_open = false; continue; }
            const int stage = issued % S_STAGES;
            if (lane == 0) {
                asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                mbar_arrive_expect_tx(full0 + 8 * stage, 2 * TILE_BYTES);
                tma_load_kv_once(tiles_u32 + stage * 2 * TILE_BYTES, &kv_map, full0 + 8 * stage, (int)(p_krow + (int64_t)p_tile * S_TP), policy);
            }
            ++issued;
            p_tile += T;
        }
    };

    bool waited = false, ok = true;
    int later = -1;                               // first lane of the team: head of the list of items put off
    auto wait_prefix = [&]() {
        grid_dep_wait();
        grid_dep_launch_dependents();          // the output projection may request its weights once there is room for it
        waited = true;
    };
    // Merges: heads me, me + T, ... of an item, side by side.  Lane 8 h + i holds m and l of source i of the h-th of them: up to four
    // shared-prefix records and, as source OWN, the suffix.  The team's shares are folded into that one source first, whether it then stays in
    // registers or is put off as a record: which of the two an item meets is a matter of timing, its sums are not.
    constexpr int OWN = MAX_MERGED_PARTS;
    float rec[H][OWN + 1][EPL], rm = -INFINITY, rl = 0.f;
    auto fetch_records = [&](size_t rh0, bool own) {        // own: the suffix too, which was put off
        const int np = part.n_parts;
#pragma unroll
        for (int h = 0; h < H; ++h)
#pragma unroll
            for (int i = 0; i <= OWN; ++i) {
                const bool on = (i < OWN ? i < np : own) && me + T * h < n_rep;
                const float* src = part.o + ((size_t)(i < OWN ? i : np) * part.stride + rh0 + me + T * h) * HD + lane * EPL;
                if (EPL == 4) {
                    const float4 x = on ? __ldcg(reinterpret_cast<const float4*>(src)) : make_float4(0.f, 0.f, 0.f, 0.f);
                    rec[h][i][0] = x.x; rec[h][i][1] = x.y; rec[h][i][EPL - 2] = x.z; rec[h][i][EPL - 1] = x.w;
                } else {
                    const float2 x = on ? __ldcg(reinterpret_cast<const float2*>(src)) : make_float2(0.f, 0.f);
                    rec[h][i][0] = x.x; rec[h][i][1] = x.y;
                }
            }
        const int i = lane & 7, j = me + T * (lane >> 3);
        const bool on = (i < OWN ? i < np : i == OWN && own) && lane < 8 * H && j < n_rep;
        const size_t at = (size_t)(i < OWN ? i : np) * part.stride + rh0 + j;
        rm = on ? __ldcg(part.m + at) : -INFINITY;
        rl = on ? __ldcg(part.l + at) : 0.f;
    };
    // over the eight lanes of a head, the same bits in each
    auto head_max = [&](float m) {
#pragma unroll
        for (int d = 1; d < 8; d <<= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, d));
        return m;
    };
    auto head_sum = [&](float l) {
#pragma unroll
        for (int d = 1; d < 8; d <<= 1) l = __fadd_rn(l, __shfl_xor_sync(0xffffffffu, l, d));
        return l;
    };
    auto fold_shares = [&]() {                    // the shares of the team's warps -> source OWN
        const bool on = (lane & 7) < T && lane < 8 * H;
        const float* at = ml + (lane & (T - 1)) * 16 + ((me + T * (lane >> 3)) & 7);
        const float m = on ? at[0] : -INFINITY, l = on ? at[8] : 0.f;
        const float M = head_max(m), w = exp2_safe(m, M), sum = head_sum(__fmul_rn(l, w));
        if ((lane & 7) == OWN) { rm = M; rl = sum; }
#pragma unroll
        for (int h = 0; h < H; ++h) {
#pragma unroll
            for (int e = 0; e < EPL; ++e) rec[h][OWN][e] = 0.f;
#pragma unroll
            for (int i = 0; i < T; ++i) {
                const float x = __shfl_sync(0xffffffffu, w, 8 * h + i);
                const float* src = obuf + (i * 8 + ((me + T * h) & 7)) * HD + lane * EPL;
#pragma unroll
                for (int e = 0; e < EPL; ++e) rec[h][OWN][e] = __fmaf_rn(src[e], x, rec[h][OWN][e]);      // (a warp without tiles left zeros)
            }
        }
    };
    auto put_off = [&](size_t rh0) {              // source OWN -> record n_parts
#pragma unroll
        for (int h = 0; h < H; ++h) {
            const int j = me + T * h;
            const float m = __shfl_sync(0xffffffffu, rm, 8 * h + OWN), l = __shfl_sync(0xffffffffu, rl, 8 * h + OWN);
            if (j >= n_rep) break;
            const size_t at = (size_t)part.n_parts * part.stride + rh0 + j;
            if (lane == 0) { part.m[at] = m; part.l[at] = l; }
            float* dst = part.o + at * HD + lane * EPL;
            if (EPL == 4) *reinterpret_cast<float4*>(dst) = make_float4(rec[h][OWN][0], rec[h][OWN][1], rec[h][OWN][EPL - 2], rec[h][OWN][EPL - 1]);
            else *reinterpret_cast<float2*>(dst) = make_float2(rec[h][OWN][0], rec[h][OWN][1]);
        }
    };
    auto merge = [&](size_t rh0) {                // all sources -> the item's output
        const float M = head_max(rm), w = exp2_safe(rm, M), denom = head_sum(__fmul_rn(rl, w));
#pragma unroll
        for (int h = 0; h < H; ++h) {
            float acc[EPL];
#pragma unroll
            for (int e = 0; e < EPL; ++e) acc[e] = 0.f;
#pragma unroll
            for (int i = 0; i <= OWN; ++i) {
                const float f = __shfl_sync(0xffffffffu, w, 8 * h + i);
                // a record with m = -inf was left by an empty range: its output is not defined
#pragma unroll
                for (int e = 0; e < EPL; ++e) acc[e] = __fmaf_rn(f > 0.f ? rec[h][i][e] : 0.f, f, acc[e]);
            }
            const float dh = __shfl_sync(0xffffffffu, denom, 8 * h);
            if (me + T * h >= n_rep) break;
            store_attention<HD>(lane, rh0 + me + T * h, acc, dh, wk.out, wk.out_lo, err);
        }
    };

    uint32_t qn[KS][2];                           // Q^T fragments (B operand) of item q_seq: head = lane / 4, dims ks*16 + (lane%4)*2 (+8)
    int q_seq = -1;
    auto fetch_q = [&](int seq) {
        const int item = slots[seq % S_SLOTS].item;
        if (item < 0) return;
        const int row = item / Hkv, kvh = item - row * Hkv, hq = lane >> 2;
        const __nv_bfloat16* qp = q + ((size_t)row * Hq + (size_t)kvh * n_rep + hq) * HD + (lane & 3) * 2;
#pragma unroll
        for (int ks = 0; ks < KS; ++ks) {
            qn[ks][0] = hq < n_rep ? *reinterpret_cast<const uint32_t*>(qp + ks * 16) : 0u;
            qn[ks][1] = hq < n_rep ? *reinterpret_cast<const uint32_t*>(qp + ks * 16 + 8) : 0u;
        }
        q_seq = seq;
    };
    refill(false);
    for (;; ++seq) {
        const SuffixItem it = slots[seq % S_SLOTS];
        if (it.item < 0) break;
        const int row = it.item / Hkv, kvh = it.item - row * Hkv, tiles = (it.n + S_TP - 1) / S_TP;
        if (q_seq != seq) fetch_q(seq);
        uint32_t qb[KS][2];
#pragma unroll
        for (int ks = 0; ks < KS; ++ks) { qb[ks][0] = qn[ks][0]; qb[ks][1] = qn[ks][1]; }
        refill(false);
        float o[DT][4];
#pragma unroll
        for (int t = 0; t < DT; ++t) { o[t][0] = o[t][1] = o[t][2] = o[t][3] = 0.f; }
        float mh[2] = {-INFINITY, -INFINITY}, lh[2] = {0.f, 0.f};      // heads (lane%4)*2 + {0, 1}
#pragma unroll 1
        for (int tile = me; tile < tiles; tile += T) {
            const int stage = consumed % S_STAGES;
            if (!__all_sync(0xffffffffu, mbar_wait(full0 + 8 * stage, (uint32_t)(consumed / S_STAGES) & 1u, abort_flag))) { ok = false; break; }
            const uint32_t kb = tiles_u32 + stage * 2 * TILE_BYTES;
            suffix_tile<HD>(kb, kb + TILE_BYTES, lane, min(S_TP, it.n - tile * S_TP), scale_log2, qb, o, mh, lh, [&]() {
                ++consumed;
                __syncwarp();
                refill(tile + T < tiles);
            });
        }
        if (claims && ok) refill(true);           // (the next item may not have been looked up)
        if (me == 0 && lane == 0 && *records_there == 0 && *reinterpret_cast<volatile int32_t*>(part.done) >= wk.prefix_ctas) *records_there = 1;
        if (!ok) *abort_flag = 1;
        const size_t rh0 = (size_t)row * Hq + (size_t)kvh * n_rep;
        if (waited) fetch_records(rh0, false);    // (they travel while the warps meet)
        team_sync();                              // the item before has been merged; the next is known
        if (*abort_flag) { ok = false; break; }
        refill(false);
        suffix_finish<HD>(lane, o, mh, lh, ml + me * 16, ml + me * 16 + 8, obuf + me * 8 * HD);
        if (*known > seq + 1) fetch_q(seq + 1);
        const bool now = *records_there != 0;
        if (now && !waited) {
            wait_prefix();
            fetch_records(rh0, false);
        }
        team_sync();
        fold_shares();
        if (now) {
            merge(rh0);
        } else {
            put_off(rh0);
            if (me == 0 && lane == 0) { wk.link[it.item] = later; later = it.item; }
        }
    }
    if (!ok && lane == 0) { *abort_flag = 1; set_error(err, DEV_ERR_WAIT_TIMEOUT); }
    if (!waited) wait_prefix();                   // (every CTA waits on every path)
    if (me == 0 && lane == 0) *known = later;
    team_sync();
    // items put off: a head was left by the warp that merges it now
    for (int item = *known; item >= 0 && ok;) {
        const int row = item / Hkv, kvh = item - row * Hkv;
        const size_t rh0 = (size_t)row * Hq + (size_t)kvh * n_rep;
        const int next = __ldcg(wk.link + item);
        fetch_records(rh0, true);
        merge(rh0);
        item = next;
    }
    // drain: tiles issued but not consumed must land before the shared memory is released
    while (ok && consumed < issued) {
        const int stage = consumed % S_STAGES;
        if (!mbar_wait(full0 + 8 * stage, (uint32_t)(consumed / S_STAGES) & 1u, abort_flag)) break;
        ++consumed;
    }
    __syncthreads();
    if (*abort_flag) {
        for (int i = 0; i < 2000; ++i) __nanosleep(1000);
    }
    __syncthreads();
}

}  // namespace am
}  // namespace pc

// Shared-prefix and causal-prefill attention on the 5th-generation tensor cores, head_dim 128.
//
// One CTA takes 128 query rows of a group (rollouts x the query heads that share a KV head) and a range of the group's prompt,
// 64 keys at a time:  S = Q K^T (128 x 64 in TMEM), softmax by four warps with a query row per thread, P to shared memory as
// IEEE half, O += P V (128 x 128 in TMEM).  K and V arrive by TMA as they lie in the arena: K is the K-major operand of the
// first product, V the MN-major operand of the second.  Two S accumulators let the next S run under the softmax, and two CTAs
// per SM (113 KB, 256 TMEM columns each) overlap one's softmax with the other's MMAs.
//
// The running reference of a row's softmax is its maximum so far; when that grows, O is rescaled in TMEM.  A reference that lags
// behind it by up to 2^8 saves most of the rescaling (prefill of 351 tokens 2 %, 2,048 rows 1 %, fewer rows nothing) but costs precision:
// the large P then lie anywhere between powers of two instead of just below 1, where half rounds finest, and the K and V of a prefill
// were 0.22 % (+- 0.02) further from 64 bits.
//
// What bounds it: chains, not a pipe.  Alone on the GPU (cold) a launch of 96-128 CTAs takes 12.8 us with three tiles a CTA (64 rows x
// 640 keys) and 22.5 us with ten (1,024 rows): about 1.4 us or 2,700 clocks a tile, of which the exponentials (16 per clock and
// SM) would be 512, and 9 us that no tile explains (launch, q, first K, record).  Prefill of 16 x 640 tokens, 960 CTAs of 5.5 tiles:
// 71.3 us, 2.0 us of an SM's time per tile with a CTA's start and end in it.  Tensor pipe 8 / 15 / 17 %, DRAM 10 / 8 / 7 % busy.
// The mma.sync kernel (attn_group_kernel, kept for head_dim 64) needs 5,000 clocks for a tile of half the rows.
#pragma once

#include "attention_mma.cuh"
#include "gemm_wt.cuh"

namespace pc {
namespace at {

using am::PrefixPartial;
using tc::mbar_arrive;
using tc::mbar_arrive_expect_tx;
using tc::mbar_init;
using tc::smem_u32;
using tc::tc_fence_after;
using tc::tc_fence_before;
using tc::tma_load_2d;
using wt::mbar_wait;

constexpr int HD = 128;
constexpr int QROWS = 128;          // query rows of a CTA
constexpr int TK = am::G_TK;        // keys per tile (64: one MMA of 64 columns, four of 16 keys)
constexpr int STAGES = 2;           // K / V tiles in flight
constexpr int Q_BYTES = QROWS * HD * 2, P_BYTES = QROWS * TK * 2, KV_BYTES = TK * HD * 2;
constexpr int THREADS = 192;        // warps 0..3 softmax (TMEM lane quarter = warp), 4 MMA issuer, 5 TMA producer
constexpr int TMEM_COLS = 256;      // O: columns 0..127, S: 128..191 and 192..255
constexpr int REC_PITCH = HD * 4 + 16;      // rows of an output on its way out: eight threads' 16 bytes in different banks
static_assert(QROWS * REC_PITCH <= Q_BYTES + P_BYTES + STAGES * 2 * KV_BYTES, "rows of a record");
constexpr int SMEM_BYTES = Q_BYTES + P_BYTES + STAGES * 2 * KV_BYTES + 1024;      // 113 KB: half of an SM's 228 KB less the reserved KB

// Shared-memory descriptor of an MN-major 128-byte-swizzled operand: rows of 64 values along MN (128 bytes), 8-row groups along K
// 1024 bytes apart, blocks of 64 along MN `mn_stride` bytes apart.
__device__ __forceinline__ uint64_t make_mn_desc(uint32_t saddr, uint32_t mn_stride) {
    return (uint64_t)((saddr & 0x3FFFFu) >> 4) | ((uint64_t)(mn_stride >> 4) << 16) | ((uint64_t)(1024 >> 4) << 32) | (1ull << 46) | (2ull << 61);
}
__device__ __forceinline__ void tmem_st32(uint32_t taddr, const float* v) {
    uint32_t r[32];
#pragma unroll
    for (int i = 0; i < 32; ++i) r[i] = __float_as_uint(v[i]);
    asm volatile(
        "tcgen05.st.sync.aligned.32x32b.x32.b32 [%0], "
        "{%1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, %16, "
        "%17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31, %32};"
        ::"r"(taddr), "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]), "r"(r[8]), "r"(r[9]),
          "r"(r[10]), "r"(r[11]), "r"(r[12]), "r"(r[13]), "r"(r[14]), "r"(r[15]), "r"(r[16]), "r"(r[17]), "r"(r[18]), "r"(r[19]),
          "r"(r[20]), "r"(r[21]), "r"(r[22]), "r"(r[23]), "r"(r[24]), "r"(r[25]), "r"(r[26]), "r"(r[27]), "r"(r[28]), "r"(r[29]),
          "r"(r[30]), "r"(r[31])
        : "memory");
    asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ float ex2(float x) {
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
// Byte offset of 16-byte chunk c (8 values) of row r in a block of 64 columns, 128-byte swizzle.
__device__ __forceinline__ uint32_t chunk_off(int r, int c) { return (uint32_t)(r * 128 + ((c ^ (r & 7)) << 4)); }

// Units of work: (group, KV head, 128 query rows, range of the prompt), range fastest; one CTA each.
// FINAL (prefill): every query row sees its own prefix, the normalised output is written.  Otherwise (decode): the rows of a group
// see the whole prompt and a record (m, l, unnormalised O) per query row is left for the merge.
template <bool FINAL>
__global__ void __launch_bounds__(THREADS, 2)
attn_prefix_kernel(const __grid_constant__ CUtensorMap kv_map, const StepDesc* __restrict__ sd, int64_t n_slots, int Hq, int Hkv,
                   int layer, const __nv_bfloat16* __restrict__ q, const int32_t* __restrict__ group_row_start, RowGeom g,
                   float scale_log2, PrefixPartial part, int q_tiles, __nv_bfloat16* __restrict__ out,
                   __nv_bfloat16* __restrict__ out_lo, int32_t* err) {
    extern __shared__ uint8_t smem_raw[];
    uint8_t* base = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
    const int slack = (int)(base - smem_raw);
    uint64_t* bars = reinterpret_cast<uint64_t*>(base + Q_BYTES + P_BYTES + STAGES * 2 * KV_BYTES);
    const uint32_t q_u32 = smem_u32(base), p_u32 = q_u32 + Q_BYTES, kv_u32 = p_u32 + P_BYTES;
    // K full, V full, K empty, V empty [STAGES each]; S full [2]; P ready; O done; Q ready
    const uint32_t kfull0 = smem_u32(bars), vfull0 = kfull0 + 8 * STAGES, kempty0 = vfull0 + 8 * STAGES, vempty0 = kempty0 + 8 * STAGES;
    const uint32_t sfull0 = vempty0 + 8 * STAGES, pready = sfull0 + 16, odone = pready + 8, qready = odone + 8;
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars + 4 * STAGES + 5);
    volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);
    int* s_maxlen = reinterpret_cast<int*>(tmem_slot + 2);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;

    const int n_rep = Hq / Hkv;
    const int n_parts = FINAL ? 1 : part.n_parts;
    const int unit = blockIdx.x;
    const int my_part = unit % n_parts, q0 = (unit / n_parts) % q_tiles * QROWS;
    const int kvh = unit / (n_parts * q_tiles) % Hkv, grp = unit / (n_parts * q_tiles * Hkv);
    int row0 = 0, n_q = 0;
    if (grp < sd->n_groups) {
        row0 = group_row_start[grp];
        n_q = (group_row_start[grp + 1] - row0) * n_rep;
    }
    if (q0 >= n_q || slack + Q_BYTES + P_BYTES + STAGES * 2 * KV_BYTES + 256 > SMEM_BYTES) {
        if (q0 < n_q && threadIdx.x == 0) set_error(err, DEV_ERR_GROUP_RANGE);        // (the shared memory window is not where it should be)
        grid_dep_wait();
        grid_dep_launch_dependents();
        if (!FINAL && part.done != nullptr && threadIdx.x == 0) atomicAdd(part.done, 1);
        return;
    }

    if (threadIdx.x == 0) {
        for (int s = 0; s < STAGES; ++s) { mbar_init(kfull0 + 8 * s, 1); mbar_init(vfull0 + 8 * s, 1); mbar_init(kempty0 + 8 * s, 1); mbar_init(vempty0 + 8 * s, 1); }
        mbar_init(sfull0, 1); mbar_init(sfull0 + 8, 1);
        mbar_init(pready, 4); mbar_init(odone, 1); mbar_init(qready, 4);
        *abort_flag = 0;
        *s_maxlen = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    }
    if (warp == 4) tc::tmem_alloc(smem_u32(tmem_slot), TMEM_COLS);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *tmem_slot;

    // the visible prefix: of the whole group (decode), of the longest row of the tile (prefill)
    int max_len;
    const int qr = q0 + threadIdx.x;        // softmax threads: this thread's query row = (rollout row qr / n_rep, head qr % n_rep)
    const bool valid = threadIdx.x < QROWS && qr < n_q;
    const int row = row0 + (valid ? qr / n_rep : 0), head = kvh * n_rep + (valid ? qr % n_rep : 0);
    int lim = 0;
    if (FINAL) {
        if (threadIdx.x < QROWS) {
            lim = valid ? g.p_len[row] : 0;
            int mx = lim;
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) mx = max(mx, __shfl_xor_sync(0xffffffffu, mx, o));
            if (lane == 0) atomicMax(s_maxlen, mx);
        }
        __syncthreads();
        max_len = *s_maxlen;
    } else {
        max_len = g.p_len[row0];
        lim = valid ? max_len : 0;
    }
    const int tiles_all = (max_len + TK - 1) / TK, per_part = (tiles_all + n_parts - 1) / n_parts;
    const int tile0 = my_part * per_part, n_tiles = max(0, min(tiles_all, tile0 + per_part) - tile0);

    bool ok = true;
    // one answer per warp: tensor-memory accesses need all its lanes, and producer and issuer elect one where they issue
    auto warp_wait = [&](uint32_t bar, uint32_t parity) { return __all_sync(0xffffffffu, mbar_wait(bar, parity, abort_flag)) != 0; };
    if (warp == 5) {
        {
            // ---------------- TMA producer ----------------
            if (FINAL) grid_dep_wait();             // K and V of this very pass; decode: the prompt's were written by an earlier call
            const int64_t kv_start = g.p_start[row0];
            const int64_t krow = (((int64_t)layer * 2 + 0) * Hkv + kvh) * n_slots + kv_start, vrow = (((int64_t)layer * 2 + 1) * Hkv + kvh) * n_slots + kv_start;
#pragma unroll 1
            for (int t = 0; t < n_tiles; ++t) {
                const int s = t % STAGES;
                const uint32_t kb = kv_u32 + s * 2 * KV_BYTES, vb = kb + KV_BYTES, ph = (uint32_t)(t / STAGES - 1) & 1u;
                if (t >= STAGES && !warp_wait(kempty0 + 8 * s, ph)) { ok = false; break; }
                if (wt::elect_one()) {
                    mbar_arrive_expect_tx(kfull0 + 8 * s, KV_BYTES);
                    tma_load_2d(kb, &kv_map, kfull0 + 8 * s, 0, (int)(krow + (int64_t)(tile0 + t) * TK));
                    tma_load_2d(kb + TK * 128, &kv_map, kfull0 + 8 * s, 64, (int)(krow + (int64_t)(tile0 + t) * TK));
                }
                if (t >= STAGES && !warp_wait(vempty0 + 8 * s, ph)) { ok = false; break; }
                if (wt::elect_one()) {
                    mbar_arrive_expect_tx(vfull0 + 8 * s, KV_BYTES);
                    tma_load_2d(vb, &kv_map, vfull0 + 8 * s, 0, (int)(vrow + (int64_t)(tile0 + t) * TK));
                    tma_load_2d(vb + TK * 128, &kv_map, vfull0 + 8 * s, 64, (int)(vrow + (int64_t)(tile0 + t) * TK));
                }
            }
        }
        __syncwarp();
    } else if (warp == 4) {
        if (n_tiles > 0) {
            // ---------------- MMA issuer: S of the next tile goes ahead of this tile's P V ----------------
            const uint32_t idesc_s = tc::make_idesc(QROWS, TK, true), idesc_o = tc::make_idesc(QROWS, HD, true) | (1u << 16) /* V: MN-major */;
            auto issue_s = [&](int t) {
                const int s = t % STAGES;
                if (!warp_wait(kfull0 + 8 * s, (uint32_t)(t / STAGES) & 1u)) return false;
                tc_fence_after();
                if (wt::elect_one()) {
                    const uint64_t dq = tc::make_smem_desc(q_u32), dk = tc::make_smem_desc(kv_u32 + s * 2 * KV_BYTES);
#pragma unroll
                    for (int kk = 0; kk < HD / 16; ++kk) {
                        // 64-column blocks of Q (128 rows) and K (TK rows), 32 bytes per 16 columns inside a block
                        const uint32_t aq = (kk >> 2) * (QROWS * 128 >> 4) + (kk & 3) * 2, ak = (kk >> 2) * (TK * 128 >> 4) + (kk & 3) * 2;
                        tc::umma_bf16(tmem + HD + (t & 1) * TK, dq + aq, dk + ak, idesc_s, kk > 0 ? 1u : 0u);
                    }
                    tc::umma_commit(kempty0 + 8 * s);
                    tc::umma_commit(sfull0 + 8 * (t & 1));
                }
                return true;
            };
            ok = warp_wait(qready, 0);
            tc_fence_after();
            if (ok) ok = issue_s(0);
#pragma unroll 1
            for (int t = 0; t < n_tiles && ok; ++t) {
                if (t + 1 < n_tiles && !issue_s(t + 1)) { ok = false; break; }
                const int s = t % STAGES;
                if (!warp_wait(vfull0 + 8 * s, (uint32_t)(t / STAGES) & 1u) || !warp_wait(pready, (uint32_t)t & 1u)) { ok = false; break; }
                tc_fence_after();
                if (wt::elect_one()) {
                    const uint64_t dp = tc::make_smem_desc(p_u32), dv = make_mn_desc(kv_u32 + s * 2 * KV_BYTES + KV_BYTES, TK * 128);
                    const int steps = (max_len - (tile0 + t) * TK + 15) / 16;       // groups of 16 keys that hold a visible one
#pragma unroll
                    for (int kk = 0; kk < TK / 16; ++kk)
                        if (kk < steps) tc::umma_bf16(tmem, dp + kk * 2, dv + kk * (16 * 128 >> 4), idesc_o, (t > 0 || kk > 0) ? 1u : 0u);
                    tc::umma_commit(vempty0 + 8 * s);
                    tc::umma_commit(odone);
                }
            }
        }
        __syncwarp();
    } else {
        // ---------------- softmax: one query row per thread ----------------
        grid_dep_wait();                     // q: the kernel before this one
        grid_dep_launch_dependents();
        {
            const uint4* src = reinterpret_cast<const uint4*>(q + ((size_t)row * Hq + head) * HD);
#pragma unroll
            for (int c = 0; c < HD / 8; ++c) {
                const uint4 v = valid ? src[c] : make_uint4(0u, 0u, 0u, 0u);
                *reinterpret_cast<uint4*>(base + (c >> 3) * (QROWS * 128) + chunk_off(threadIdx.x, c & 7)) = v;
            }
        }
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        __syncwarp();
        if (lane == 0) mbar_arrive(qready);
        const uint32_t lanes = tmem + ((uint32_t)(warp * 32) << 16);
        float m = -INFINITY, l = 0.f;
#pragma unroll 1
        for (int t = 0; t < n_tiles; ++t) {
            if (!warp_wait(sfull0 + 8 * (t & 1), (uint32_t)(t >> 1) & 1u)) { ok = false; break; }
            tc_fence_after();
            float s[TK];
            tc::tmem_ld32(lanes + HD + (t & 1) * TK, s);
            tc::tmem_ld32(lanes + HD + (t & 1) * TK + 32, s + 32);
            const int see = lim - (tile0 + t) * TK;          // visible keys of the tile (may be <= 0 or > TK)
            if (__any_sync(0xffffffffu, see < TK)) {
#pragma unroll
                for (int i = 0; i < TK; ++i) s[i] = i < see ? s[i] : -INFINITY;
            }
            float x4[4] = {-INFINITY, -INFINITY, -INFINITY, -INFINITY};
#pragma unroll
            for (int i = 0; i < TK; ++i) x4[i & 3] = fmaxf(x4[i & 3], s[i]);
            const float mx = fmaxf(fmaxf(x4[0], x4[1]), fmaxf(x4[2], x4[3])) * scale_log2;      // (the scale is positive; -inf stays -inf)
            // P's buffer and O are free once the previous P V is done
            if (t > 0 && !warp_wait(odone, (uint32_t)(t - 1) & 1u)) { ok = false; break; }
            tc_fence_after();
            const bool move = mx > m;
            if (__any_sync(0xffffffffu, move)) {
                const float corr = move ? (m == -INFINITY ? 0.f : ex2(m - mx)) : 1.f;
                if (move) m = mx;
                l *= corr;
                if (t > 0) {
#pragma unroll 1
                    for (int c = 0; c < HD; c += 32) {
                        float o[32];
                        tc::tmem_ld32(lanes + c, o);
#pragma unroll
                        for (int i = 0; i < 32; ++i) o[i] *= corr;
                        tmem_st32(lanes + c, o);
                    }
                }
            }
            const float ref = m == -INFINITY ? 0.f : m;      // a row that has seen no key yet: every P is 2^-inf = 0
            float l4[4] = {l, 0.f, 0.f, 0.f};
#pragma unroll
            for (int i = 0; i < TK; ++i) {
                s[i] = ex2(s[i] * scale_log2 - ref);
                l4[i & 3] += s[i];
            }
            l = (l4[0] + l4[1]) + (l4[2] + l4[3]);
#pragma unroll
            for (int c = 0; c < TK / 8; ++c) {
                const uint32_t w0 = am::pack_f16(s[8 * c], s[8 * c + 1]), w1 = am::pack_f16(s[8 * c + 2], s[8 * c + 3]);
                const uint32_t w2 = am::pack_f16(s[8 * c + 4], s[8 * c + 5]), w3 = am::pack_f16(s[8 * c + 6], s[8 * c + 7]);
                asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(p_u32 + chunk_off(threadIdx.x, c)), "r"(w0), "r"(w1), "r"(w2), "r"(w3) : "memory");
            }
            // values of V behind the last visible key may be anything: their P is 0, but 0 * NaN would poison the sum, so the
            // rows up to the next multiple of 16 are zeroed (groups of 16 behind that are not multiplied)
            const int left = max_len - (tile0 + t) * TK;
            if (left < TK && (left & 15) != 0) {
                if (!warp_wait(vfull0 + 8 * (t % STAGES), (uint32_t)(t / STAGES) & 1u)) { ok = false; break; }
                uint8_t* vb = base + Q_BYTES + P_BYTES + (t % STAGES) * 2 * KV_BYTES + KV_BYTES;
                for (int i = threadIdx.x; i < (16 - (left & 15)) * 16; i += QROWS)
                    *reinterpret_cast<uint4*>(vb + ((i >> 3) & 1) * (TK * 128) + (left + (i >> 4)) * 128 + (i & 7) * 16) = make_uint4(0u, 0u, 0u, 0u);
            }
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(pready);
        }
        if (ok && n_tiles > 0 && !warp_wait(odone, (uint32_t)(n_tiles - 1) & 1u)) ok = false;
        tc_fence_after();
        if (ok) {
            const size_t rh = (size_t)row * Hq + head;
            const size_t ph = (size_t)my_part * part.stride + rh;
            const float inv = FINAL ? (l > 0.f ? 1.f / l : 0.f) : 1.f;
            if (!FINAL && valid) { part.m[ph] = m; part.l[ph] = l; }
            // a record's output (512 bytes, a row per thread) leaves through shared memory, where nothing is in use any more: stored by
            // the threads, 16 bytes each of 32 rows at a time, it took 2 us
            float* rec_row = reinterpret_cast<float*>(base + threadIdx.x * REC_PITCH);
            if (n_tiles > 0) {               // an empty range leaves (m, l) = (-inf, 0); its output is never read
#pragma unroll 1
                for (int c = 0; c < HD; c += 32) {
                    float o[32];
                    tc::tmem_ld32(lanes + c, o);
                    if (!valid) continue;
                    if (!FINAL) {
                        float4* dst = reinterpret_cast<float4*>(rec_row + c);
#pragma unroll
                        for (int i = 0; i < 8; ++i) dst[i] = make_float4(o[4 * i], o[4 * i + 1], o[4 * i + 2], o[4 * i + 3]);
                        continue;
                    }
                    uint4* dst = reinterpret_cast<uint4*>(out + rh * HD + c);
#pragma unroll
                    for (int i = 0; i < 32; ++i) o[i] *= inv;
                    if (out_lo == nullptr) {         // the output projection takes IEEE half operands
#pragma unroll
                        for (int i = 0; i < 4; ++i)
                            dst[i] = make_uint4(am::pack_f16_guard(o[8 * i], o[8 * i + 1], err), am::pack_f16_guard(o[8 * i + 2], o[8 * i + 3], err),
                                                am::pack_f16_guard(o[8 * i + 4], o[8 * i + 5], err), am::pack_f16_guard(o[8 * i + 6], o[8 * i + 7], err));
                    } else {
                        uint4* lo = reinterpret_cast<uint4*>(out_lo + rh * HD + c);      // rounding remainder: second operand of the projection
#pragma unroll
                        for (int i = 0; i < 4; ++i) {
                            dst[i] = make_uint4(am::pack_bf16(o[8 * i], o[8 * i + 1]), am::pack_bf16(o[8 * i + 2], o[8 * i + 3]),
                                                am::pack_bf16(o[8 * i + 4], o[8 * i + 5]), am::pack_bf16(o[8 * i + 6], o[8 * i + 7]));
#pragma unroll
                            for (int k = 0; k < 8; ++k) o[8 * i + k] = wt::bf16_rest(o[8 * i + k]);
                            lo[i] = make_uint4(am::pack_bf16(o[8 * i], o[8 * i + 1]), am::pack_bf16(o[8 * i + 2], o[8 * i + 3]),
                                               am::pack_bf16(o[8 * i + 4], o[8 * i + 5]), am::pack_bf16(o[8 * i + 6], o[8 * i + 7]));
                        }
                    }
                }
                if (!FINAL && valid) {
                    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                    asm volatile("cp.async.bulk.global.shared::cta.bulk_group [%0], [%1], %2;"
                                 ::"l"(__cvta_generic_to_global(part.o + ph * HD)), "r"(smem_u32(rec_row)), "r"(HD * 4) : "memory");
                    asm volatile("cp.async.bulk.commit_group;" ::: "memory");
                    asm volatile("cp.async.bulk.wait_group 0;" ::: "memory");
                }
            } else if (FINAL && valid) {
                for (int c = 0; c < HD; c += 8) {
                    *reinterpret_cast<uint4*>(out + rh * HD + c) = make_uint4(0u, 0u, 0u, 0u);
                    if (out_lo != nullptr) *reinterpret_cast<uint4*>(out_lo + rh * HD + c) = make_uint4(0u, 0u, 0u, 0u);
                }
            }
        }
    }
    if (!ok && lane == 0) { *abort_flag = 1; set_error(err, DEV_ERR_WAIT_TIMEOUT); }
    tc_fence_before();
    __syncthreads();
    // Tells suffix warps that started beside this kernel when to stop putting off their merges.  (They still wait for the kernel's end.)
    if (!FINAL && part.done != nullptr && threadIdx.x == 0) atomicAdd(part.done, 1);
    if (*abort_flag) {
#pragma unroll 1
        for (int i = 0; i < 2000; ++i) __nanosleep(1000);    // copies in flight land before the shared memory is released
        __syncthreads();
    }
    if (warp == 4) {
        __syncwarp();
        tc_fence_after();
        tc::tmem_dealloc(tmem, TMEM_COLS);
    }
}

}  // namespace at
}  // namespace pc

// Attention of small decode batches: a cluster of C CTAs (C = 1, 2, 4 or 8) takes one (rollout, KV head), its 4 C warps
// stream the item's tiles in turn, and the cluster merges their partial softmaxes over distributed shared memory into the attention
// output -- no records of its own, no merge kernel (a launch and three L2 round trips: 5 us of a 60 us layer at 16 rows).
//
//   JOINT   the tiles are the prompt's and then the suffix's, from two arenas: the kernel is the whole attention of a layer.  It follows the
//           QKV projection; every tile but the one that projection writes into is requested before the wait.
//   else    the tiles are the suffix's, and the item's shared-prefix records join the merge.  At 113 KB a CTA fits beside one of the
//           shared-prefix kernel, whose programmatic dependent it is: the two run side by side and this one waits for the records
//           only when it merges.
// When which is taken: joint_attention in pc_api.cu.
//
// What bounds it: latency.  16 rows, 640 + 1,100 positions, four CTAs: seven tiles per warp (0.5 us each), the hand-over, and the chain
// partial softmax -> weights -> output.
#pragma once

#include <type_traits>

#include "attention_mma.cuh"
#include "gemm_wt.cuh"

namespace pc {
namespace am {

constexpr int T_WARPS = 4, T_STAGES = 3;
template <int HD> __host__ __device__ constexpr int team_smem_need() { return T_WARPS * (T_STAGES * 2 * S_TP * HD * 2 + 8 * HD * 4) + 512; }
constexpr int TEAM_SMEM_BYTES = 113 * 1024;      // half of an SM's 228 KB less the reserved KB
static_assert(team_smem_need<128>() <= TEAM_SMEM_BYTES, "team buffers");

// floats `at` of lane of a CTA's output buffer in the cluster
template <int EPL> __device__ __forceinline__ void ld_cluster(uint32_t addr, float* v) {
    if (EPL == 4) {
        const float4 x = wt::ld_cluster_f32x4(addr);
        v[0] = x.x; v[1] = x.y; v[EPL - 2] = x.z; v[EPL - 1] = x.w;
    } else {
        asm volatile("ld.shared::cluster.v2.f32 {%0, %1}, [%2];" : "=f"(v[0]), "=f"(v[1]) : "r"(addr) : "memory");
    }
}

template <int HD, bool JOINT>
__global__ void __launch_bounds__(T_WARPS * 32, 2)
attn_suffix_team_kernel(const __grid_constant__ CUtensorMap kv_map, const __grid_constant__ CUtensorMap prompt_map, int64_t prompt_slots, const StepDesc* __restrict__ sd, int64_t n_slots, int Hq, int Hkv,
                        int layer, const __nv_bfloat16* __restrict__ q, RowGeom g, float scale_log2, PrefixPartial part, int team_ctas,
                        __nv_bfloat16* __restrict__ out, __nv_bfloat16* __restrict__ out_lo, int32_t* err) {
    constexpr int KS = HD / 16, DT = HD / 16, EPL = HD / 32;
    constexpr int TILE_BYTES = S_TP * HD * 2, WARP_BYTES = T_STAGES * 2 * TILE_BYTES;
    extern __shared__ uint8_t smem_raw[];
    uint8_t* base = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int item = blockIdx.x / team_ctas, rank = blockIdx.x % team_ctas;
    const bool fits = (int)(base - smem_raw) + team_smem_need<HD>() <= TEAM_SMEM_BYTES;
    if (item >= sd->n_rows * Hkv || !fits) {               // (the same for the whole cluster)
        if (!fits && threadIdx.x == 0) set_error(err, DEV_ERR_GROUP_RANGE);
        grid_dep_wait();
        return;
    }
    float* obuf = reinterpret_cast<float*>(base + T_WARPS * WARP_BYTES);                         // [warp][8 heads][HD]
    float* ml = obuf + T_WARPS * 8 * HD;                                                          // [warp][m of 8 heads, l of 8 heads]
    uint64_t* bars = reinterpret_cast<uint64_t*>(ml + T_WARPS * 16) + warp * T_STAGES;
    volatile int* abort_flag = reinterpret_cast<volatile int*>(ml + T_WARPS * 16 + 2 * T_WARPS * T_STAGES);
    const uint32_t tiles_u32 = smem_u32(base + warp * WARP_BYTES), full0 = smem_u32(bars);
    const int n_rep = Hq / Hkv, row = item / Hkv, kvh = item - row * Hkv;

    if (threadIdx.x == 0) *abort_flag = 0;
    if (lane == 0) {
        for (int s = 0; s < T_STAGES; ++s) mbar_init(full0 + 8 * s, 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    }
    __syncthreads();

    const int n = g.s_len[row], n_prompt = JOINT ? g.p_len[row] : 0;
    const int p_tiles = (n_prompt + S_TP - 1) / S_TP, tiles = p_tiles + (n + S_TP - 1) / S_TP;      // the prompt's tiles first
    const int workers = team_ctas * T_WARPS, me = rank * T_WARPS + warp;
    const int64_t krow = ((int64_t)layer * 2 * Hkv + kvh) * n_slots + g.s_start[row];
    const int64_t prow = JOINT ? ((int64_t)layer * 2 * Hkv + kvh) * prompt_slots + g.p_start[row] : 0;
    const uint64_t policy = policy_evict_first();
    int next = me, issued = 0, consumed = 0;
    auto issue = [&]() {
        const int stage = issued % T_STAGES;
        if (lane == 0) {
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            mbar_arrive_expect_tx(full0 + 8 * stage, 2 * TILE_BYTES);
            if (JOINT && next < p_tiles) tma_load_kv(tiles_u32 + stage * 2 * TILE_BYTES, &prompt_map, full0 + 8 * stage, (int)(prow + (int64_t)next * S_TP));
            else tma_load_kv_once(tiles_u32 + stage * 2 * TILE_BYTES, &kv_map, full0 + 8 * stage, (int)(krow + (int64_t)(next - p_tiles) * S_TP), policy);
        }
        ++issued;
        next += workers;
    };
    if (JOINT) {
        // all but the last tile, which holds the position the QKV projection is writing, were there before this step
        while (issued < T_STAGES && next < tiles - 1) issue();
        grid_dep_wait();
        grid_dep_launch_dependents();          // the output projection may request its weights
    }
    while (issued < T_STAGES && next < tiles) issue();
    uint32_t qb[KS][2];
    {
        const int hq = lane >> 2;
        const __nv_bfloat16* qp = q + ((size_t)row * Hq + (size_t)kvh * n_rep + hq) * HD + (lane & 3) * 2;
#pragma unroll
        for (int ks = 0; ks < KS; ++ks) {
            qb[ks][0] = hq < n_rep ? *reinterpret_cast<const uint32_t*>(qp + ks * 16) : 0u;
            qb[ks][1] = hq < n_rep ? *reinterpret_cast<const uint32_t*>(qp + ks * 16 + 8) : 0u;
        }
    }
    float o[DT][4], mh[2] = {-INFINITY, -INFINITY}, lh[2] = {0.f, 0.f};
#pragma unroll
    for (int t = 0; t < DT; ++t) { o[t][0] = o[t][1] = o[t][2] = o[t][3] = 0.f; }
    bool ok = true;
#pragma unroll 1
    for (int tile = me; tile < tiles; tile += workers) {
        const int stage = consumed % T_STAGES;
        if (!mbar_wait(full0 + 8 * stage, (uint32_t)(consumed / T_STAGES) & 1u, abort_flag)) { ok = false; break; }
        const uint32_t kb = tiles_u32 + stage * 2 * TILE_BYTES;
        suffix_tile<HD>(kb, kb + TILE_BYTES, lane, min(S_TP, tile < p_tiles ? n_prompt - tile * S_TP : n - (tile - p_tiles) * S_TP), scale_log2, qb, o, mh, lh, [&]() {
            ++consumed;
            __syncwarp();
            if (next < tiles) issue();
        });
    }
    suffix_finish<HD>(lane, o, mh, lh, ml + warp * 16, ml + warp * 16 + 8, obuf + warp * 8 * HD);
    if (!ok) { *abort_flag = 1; if (lane == 0) set_error(err, DEV_ERR_WAIT_TIMEOUT); }

    if (!JOINT) {
        grid_dep_wait();                       // the shared-prefix kernel's records
        grid_dep_launch_dependents();          // the output projection may request its weights
    }
    const size_t rh0 = (size_t)row * Hq + (size_t)kvh * n_rep;
    const int np = JOINT ? 0 : part.n_parts;
    // this warp's heads: me, me + workers, ...; the records of the first are requested before the cluster meets
    auto records = [&](int j, float& pm, float& pl, float (&v)[MAX_PREFIX_PARTS][EPL]) {
        pm = lane < np ? __ldcg(part.m + (size_t)lane * part.stride + rh0 + j) : -INFINITY;
        pl = lane < np ? __ldcg(part.l + (size_t)lane * part.stride + rh0 + j) : 0.f;
#pragma unroll
        for (int i = 0; i < MAX_PREFIX_PARTS; ++i) {
            const float* p = part.o + ((size_t)i * part.stride + rh0 + j) * HD + lane * EPL;
            if (EPL == 4) {
                const float4 x = i < np ? __ldcg(reinterpret_cast<const float4*>(p)) : make_float4(0.f, 0.f, 0.f, 0.f);
                v[i][0] = x.x; v[i][1] = x.y; v[i][EPL - 2] = x.z; v[i][EPL - 1] = x.w;
            } else {
                const float2 x = i < np ? __ldcg(reinterpret_cast<const float2*>(p)) : make_float2(0.f, 0.f);
                v[i][0] = x.x; v[i][1] = x.y;
            }
        }
    };
    float pm = -INFINITY, pl = 0.f, v[MAX_PREFIX_PARTS][EPL];
    if (!JOINT && me < n_rep) records(me, pm, pl, v);
    if (team_ctas > 1) wt::cluster_sync(); else __syncthreads();
    for (int j = me; j < n_rep; j += workers) {
        if (!JOINT && j != me) records(j, pm, pl, v);
        // lane w holds m and l of worker w (at most 32)
        float tm = -INFINITY, tl = 0.f;
        if (lane < workers) {
            const uint32_t at = wt::map_rank(smem_u32(ml + (lane % T_WARPS) * 16 + j), (uint32_t)(lane / T_WARPS));
            asm volatile("ld.shared::cluster.f32 %0, [%1];" : "=f"(tm) : "r"(at) : "memory");
            asm volatile("ld.shared::cluster.f32 %0, [%1];" : "=f"(tl) : "r"(at + 32) : "memory");
        }
        const float M = warp_max(fmaxf(pm, tm));
        const float wp = exp2_safe(pm, M), wt_ = exp2_safe(tm, M);
        const float denom = warp_sum(pl * wp + tl * wt_);
        float acc[EPL];
#pragma unroll
        for (int e = 0; e < EPL; ++e) acc[e] = 0.f;
#pragma unroll
        for (int i = 0; i < (JOINT ? 0 : MAX_PREFIX_PARTS); ++i) {
            const float w = __shfl_sync(0xffffffffu, wp, i);
            if (w > 0.f) {                     // a record with m = -inf was left by an empty range: its output is not defined
#pragma unroll
                for (int e = 0; e < EPL; ++e) acc[e] = __fmaf_rn(v[i][e], w, acc[e]);
            }
        }
        // sixteen reads in flight where a cluster shares the item: a read of another CTA's memory takes a quarter of a microsecond
        auto add = [&](auto batch) {
            constexpr int N = decltype(batch)::value;
#pragma unroll 1
            for (int k0 = 0; k0 < workers; k0 += N) {
                float x[N][EPL];
#pragma unroll
                for (int i = 0; i < N; ++i)
                    ld_cluster<EPL>(wt::map_rank(smem_u32(obuf + ((i % T_WARPS) * 8 + j) * HD + lane * EPL), (uint32_t)min((k0 + i) / T_WARPS, team_ctas - 1)), x[i]);
#pragma unroll
                for (int i = 0; i < N; ++i) {
                    const float w = __shfl_sync(0xffffffffu, wt_, (k0 + i) & 31);      // 0 from `workers` on
#pragma unroll
                    for (int e = 0; e < EPL; ++e) acc[e] = __fmaf_rn(x[i][e], w, acc[e]);      // (a worker without tiles left zeros)
                }
            }
        };
        if (team_ctas > 1) add(std::integral_constant<int, 16>{}); else add(std::integral_constant<int, T_WARPS>{});
        store_attention<HD>(lane, rh0 + j, acc, denom, out, out_lo, err);
    }
    // drain: tiles issued but not consumed must land before the shared memory is released
    while (ok && consumed < issued) {
        const int stage = consumed % T_STAGES;
        if (!mbar_wait(full0 + 8 * stage, (uint32_t)(consumed / T_STAGES) & 1u, abort_flag)) break;
        ++consumed;
    }
    __syncthreads();
    if (*abort_flag) {
#pragma unroll 1
        for (int i = 0; i < 2000; ++i) __nanosleep(1000);
    }
    if (team_ctas > 1) wt::cluster_sync();     // nobody leaves while a peer reads its memory
}

}  // namespace am
}  // namespace pc

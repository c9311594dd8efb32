// Plain-FP32 attention for float32 models, prefill and decode: one query position per row, a (row, KV head) block walks the
// row's prompt slots and then its suffix slots with an online softmax, serving all query heads that share the KV head.
//
// Positions are taken eight at a time by a warp: their K and V rows are loaded together, the eight scores of a head are summed
// over the lanes in nine exchanges (every exchange halves the scores a lane carries) and the running softmax moves once per
// eight positions.  One position at a time -- five exchanges, an exponential and a rescaling in a chain per head -- took 19.7 us
// at 96 rows x 110 positions.  Warp w takes chunks w, w + 8, ... of the prompt, then of the suffix, so a row's result does not
// depend on its batch mates.
#pragma once

#include "common.cuh"
#include "kernels_basic.cuh"

namespace pc {

constexpr int ATTN_MAX_REP = 8;   // query heads per KV head supported
constexpr int ATTN_WARPS = 8;
constexpr int ATTN_CHUNK = 8;     // positions a warp works on together

// POST (decode): the q|k|v projection comes as it left its GEMM, and the block finishes its own heads first -- bias, QK-norm, RoPE, q to
// its buffer, K and V to the row's slot, which no other row attends (a kernel of its own was 4 us per layer).
// HD = head_dim (64 or 128); each lane owns EPL = HD / 32 consecutive dims of every K/V row.  REP: query heads per KV head, rounded
// up to 2, 4 or 8.
template <int HD, int REP, bool POST>
__global__ void __launch_bounds__(32 * ATTN_WARPS) attn_row_simt_kernel(const StepDesc* __restrict__ sd, int Hq, int Hkv, int layer, const float* q,
                                                                        RowGeom g, KvArena prompt_arena, KvArena suffix_arena,
                                                                        float scale, float* __restrict__ out, QkvPostArgs<float> post) {
    constexpr int EPL = HD / 32, CH = ATTN_CHUNK;
    const int r = blockIdx.x, kvh = blockIdx.y;
    grid_dep_wait();
    grid_dep_launch_dependents();
    if (r >= sd->n_rows) return;
    const int n_rep = Hq / Hkv;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;

    if (POST) {
        for (int j = warp; j < n_rep + 2; j += ATTN_WARPS) {
            const int head = j < n_rep ? kvh * n_rep + j : Hq + kvh + (j - n_rep) * Hkv;
            qkv_post_items_warp<float, 1>(lane, post, &r, &head, 1);
        }
        __syncthreads();
    }
    float qf[REP][EPL], acc[REP][EPL], mx[REP], ls[REP];
#pragma unroll
    for (int j = 0; j < REP; ++j) {
        mx[j] = -INFINITY; ls[j] = 0.f;
#pragma unroll
        for (int e = 0; e < EPL; ++e) { acc[j][e] = 0.f; qf[j][e] = 0.f; }
        if (j < n_rep) {
            VecLoad<float, EPL>::load(q + ((size_t)r * Hq + (size_t)kvh * n_rep + j) * HD + lane * EPL, qf[j]);
#pragma unroll
            for (int e = 0; e < EPL; ++e) qf[j][e] *= scale;
        }
    }

    const int64_t kplane = ((int64_t)layer * 2 + 0) * Hkv + kvh, vplane = ((int64_t)layer * 2 + 1) * Hkv + kvh;
    const int mine = lane >> 2;                   // the position of a chunk whose score this lane ends up with
#pragma unroll 1
    for (int part = 0; part < 2; ++part) {
        const KvArena ar = part ? suffix_arena : prompt_arena;
        const int64_t start = part ? g.s_start[r] : g.p_start[r];
        const int n = part ? g.s_len[r] : g.p_len[r];
        const float* kb = reinterpret_cast<const float*>(ar.base) + (kplane * ar.n_slots + start) * HD + lane * EPL;
        const float* vb = reinterpret_cast<const float*>(ar.base) + (vplane * ar.n_slots + start) * HD + lane * EPL;
#pragma unroll 1
        for (int t0 = warp * CH; t0 < n; t0 += ATTN_WARPS * CH) {
            float kf[CH][EPL], vf[CH][EPL];
#pragma unroll
            for (int i = 0; i < CH; ++i) {
#pragma unroll
                for (int e = 0; e < EPL; ++e) kf[i][e] = vf[i][e] = 0.f;
                if (t0 + i < n) {
                    VecLoad<float, EPL>::load(kb + (size_t)(t0 + i) * HD, kf[i]);
                    VecLoad<float, EPL>::load(vb + (size_t)(t0 + i) * HD, vf[i]);
                }
            }
#pragma unroll
            for (int j = 0; j < REP; ++j) {
                if (j >= n_rep) break;
                float s[CH];
#pragma unroll
                for (int i = 0; i < CH; ++i) {
                    s[i] = 0.f;
#pragma unroll
                    for (int e = 0; e < EPL; ++e) s[i] = fmaf(qf[j][e], kf[i][e], s[i]);
                }
                // lane bits 4, 3, 2 choose a position, bits 1, 0 are added up
#pragma unroll
                for (int w = 4; w >= 1; w >>= 1) {
                    const bool up = lane & (w * 4);
#pragma unroll
                    for (int i = 0; i < w; ++i) {
                        const float keep = up ? s[w + i] : s[i], give = up ? s[i] : s[w + i];
                        s[i] = keep + __shfl_xor_sync(0xffffffffu, give, w * 4);
                    }
                }
                float x = s[0];
                x += __shfl_xor_sync(0xffffffffu, x, 2);
                x += __shfl_xor_sync(0xffffffffu, x, 1);
                if (t0 + mine >= n) x = -INFINITY;
                float m = x;
#pragma unroll
                for (int o = 4; o <= 16; o <<= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
                const float mnew = fmaxf(mx[j], m);            // finite: the chunk has a position
                const float corr = expf(mx[j] - mnew);          // exp(-inf) = 0 on the first chunk
                const float p = expf(x - mnew);
                mx[j] = mnew;
#pragma unroll
                for (int e = 0; e < EPL; ++e) acc[j][e] *= corr;
                float l = ls[j] * corr;
#pragma unroll
                for (int i = 0; i < CH; ++i) {
                    const float pi = __shfl_sync(0xffffffffu, p, i * 4);
                    l += pi;
#pragma unroll
                    for (int e = 0; e < EPL; ++e) acc[j][e] = fmaf(pi, vf[i][e], acc[j][e]);
                }
                ls[j] = l;
            }
        }
    }

    // merge the warps' partial softmaxes
    __shared__ float s_m[ATTN_WARPS][REP], s_l[ATTN_WARPS][REP];
    __shared__ float s_acc[ATTN_WARPS][REP][HD];
#pragma unroll
    for (int j = 0; j < REP; ++j) {
        if (j < n_rep) {
            if (lane == 0) { s_m[warp][j] = mx[j]; s_l[warp][j] = ls[j]; }
#pragma unroll
            for (int e = 0; e < EPL; ++e) s_acc[warp][j][lane * EPL + e] = acc[j][e];
        }
    }
    __syncthreads();
    for (int idx = threadIdx.x; idx < n_rep * HD; idx += blockDim.x) {
        const int j = idx / HD, e = idx - j * HD;
        float M = -INFINITY;
#pragma unroll
        for (int w = 0; w < ATTN_WARPS; ++w) M = fmaxf(M, s_m[w][j]);
        float L = 0.f, O = 0.f;
#pragma unroll
        for (int w = 0; w < ATTN_WARPS; ++w) {
            const float c = s_m[w][j] == -INFINITY ? 0.f : expf(s_m[w][j] - M);
            L += s_l[w][j] * c;
            O += s_acc[w][j][e] * c;
        }
        out[((size_t)r * Hq + (size_t)kvh * n_rep + j) * HD + e] = L > 0.f ? O / L : 0.f;
    }
}

template <int HD, bool POST>
inline cudaError_t launch_attn_row_simt(cudaStream_t st, bool dep, const StepDesc* sd, int M, int Hq, int Hkv, int layer, const float* q, RowGeom g,
                                        KvArena prompt_arena, KvArena suffix_arena, float scale, float* out, const QkvPostArgs<float>& post) {
    const int rep = Hq / Hkv;
    cudaLaunchConfig_t cfg;
    memset(&cfg, 0, sizeof(cfg));
    cfg.gridDim = dim3(M, Hkv); cfg.blockDim = dim3(32 * ATTN_WARPS); cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr; cfg.numAttrs = dep ? 1 : 0;
    return cudaLaunchKernelEx(&cfg, rep <= 2 ? attn_row_simt_kernel<HD, 2, POST> : rep <= 4 ? attn_row_simt_kernel<HD, 4, POST> : attn_row_simt_kernel<HD, 8, POST>,
                              sd, Hq, Hkv, layer, q, g, prompt_arena, suffix_arena, scale, out, post);
}

}  // namespace pc

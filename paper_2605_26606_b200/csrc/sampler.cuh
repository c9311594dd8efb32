// Seeded Gumbel-max sampling over the whole vocabulary (temperature T, top_p = 1: an exact categorical draw).
// Philox4x32-10 follows the published definition (Salmon et al., SC'11): one 128-bit block per four
// vocabulary ids, key = seed, counter = (v >> 2, step, rollout, prompt).
#pragma once

#include "common.cuh"

namespace pc {

struct Philox4 { uint32_t x, y, z, w; };

__device__ __forceinline__ Philox4 philox4x32_10(uint32_t c0, uint32_t c1, uint32_t c2, uint32_t c3, uint32_t k0, uint32_t k1) {
    constexpr uint32_t M0 = 0xD2511F53u, M1 = 0xCD9E8D57u, W0 = 0x9E3779B9u, W1 = 0xBB67AE85u;
#pragma unroll
    for (int r = 0; r < 10; ++r) {
        // one 32 x 32 -> 64 bit product per multiplier (high and low word of the same multiplication)
        const uint64_t p0 = (uint64_t)M0 * c0, p1 = (uint64_t)M1 * c2;
        const uint32_t hi0 = (uint32_t)(p0 >> 32), lo0 = (uint32_t)p0;
        const uint32_t hi1 = (uint32_t)(p1 >> 32), lo1 = (uint32_t)p1;
        const uint32_t n0 = hi1 ^ c1 ^ k0, n2 = hi0 ^ c3 ^ k1;
        c0 = n0; c1 = lo1; c2 = n2; c3 = lo0;
        k0 += W0; k1 += W1;
    }
    return Philox4{c0, c1, c2, c3};
}

// The same with the round keys in registers (as the compiler would have it, they are added up again in every block: 18 of 100
// instructions).
struct PhiloxKeys {
    uint32_t a[10], b[10];
    __device__ __forceinline__ PhiloxKeys(uint32_t k0, uint32_t k1) {
#pragma unroll
        for (int r = 0; r < 10; ++r) {
            a[r] = k0 + (uint32_t)r * 0x9E3779B9u;
            b[r] = k1 + (uint32_t)r * 0xBB67AE85u;
            asm volatile("" : "+r"(a[r]), "+r"(b[r]));
        }
    }
};
__device__ __forceinline__ Philox4 philox4x32_10(uint32_t c0, uint32_t c1, uint32_t c2, uint32_t c3, const PhiloxKeys& k) {
#pragma unroll
    for (int r = 0; r < 10; ++r) {
        const uint64_t p0 = (uint64_t)0xD2511F53u * c0, p1 = (uint64_t)0xCD9E8D57u * c2;
        const uint32_t n0 = (uint32_t)(p1 >> 32) ^ c1 ^ k.a[r], n2 = (uint32_t)(p0 >> 32) ^ c3 ^ k.b[r];
        c0 = n0; c1 = (uint32_t)p1; c2 = n2; c3 = (uint32_t)p0;
    }
    return Philox4{c0, c1, c2, c3};
}

// u = ((w >> 9) + 1/2) / 2^23 is exact in float and lies strictly inside (0, 1).
__device__ __forceinline__ float gumbel_from_word(uint32_t w) {
    const float u = ((float)(w >> 9) + 0.5f) * 1.1920928955078125e-07f;   // 2^-23
    return -logf(-logf(u));
}

struct Top2 {
    float best, second;
    int idx;
};

__device__ __forceinline__ void top2_push(Top2& t, float s, int v) {
    // strict ">" keeps the lowest id among equal scores because ids arrive in increasing order per thread
    if (s > t.best) { t.second = t.best; t.best = s; t.idx = v; }
    else if (s > t.second) t.second = s;
}

// Same fold when candidates arrive in arbitrary id order: equal scores keep the lowest id.
__device__ __forceinline__ void top2_push_unordered(Top2& t, float s, int v) {
    if (s > t.best || (s == t.best && v < t.idx)) { t.second = t.best; t.best = s; t.idx = v; }
    else if (s > t.second) t.second = s;
}

__device__ __forceinline__ Top2 top2_merge(const Top2& a, const Top2& b) {
    Top2 o;
    const bool a_wins = a.best > b.best || (a.best == b.best && a.idx < b.idx);
    o.best = a_wins ? a.best : b.best;
    o.idx = a_wins ? a.idx : b.idx;
    o.second = fmaxf(a_wins ? b.best : a.best, fmaxf(a.second, b.second));
    return o;
}

__device__ __forceinline__ Top2 top2_warp_reduce(Top2 t) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        Top2 other;
        other.best = __shfl_xor_sync(0xffffffffu, t.best, o);
        other.second = __shfl_xor_sync(0xffffffffu, t.second, o);
        other.idx = __shfl_xor_sync(0xffffffffu, t.idx, o);
        t = top2_merge(t, other);
    }
    return t;
}

// Scores the 4-id blocks b_begin .. b_end - 1 of one row (a thread block of SAMPLE_THREADS) and folds them into t.
//
// Almost every candidate is rejected without evaluating its Gumbel noise.  v can enter the row's top two only if
// logit_v / T + g_v > s for every lower bound s of the row's second-best score, that is only if
// 1 - u_v < 1 - exp(-x), x = exp(logit_v / T - s), and 1 - exp(-x) <= x.  u_v is an affine function of the random word, so a block of four
// ids costs one exponential (of its largest logit) and one comparison (of its largest word).  s is the best second-best score any warp
// of the thread block has found, through one word of shared memory.  The bound carries a slack far above the float error of its
// evaluation, a comparison with a NaN passes, and candidates that pass are scored in full, so the result is identical to scoring
// everything.
//
// What bounds it: the issue slots (123 instructions per 128 ids; Philox is 20 multiplications and 20 three-way XORs of them, the 32 x 32 -> 64
// multiplications alone half of the time), then the logits, which are read once.  With one bound per warp from the largest logit of the whole
// range -- a pass of its own over the row -- most blocks of 128 ids still held a candidate, and voting on, queueing and scoring those was
// half of the 245 instructions.  Vocabulary 151,936, both kernels of a draw, then and now: 16 rows 26 -> 16 us, 71 rows 57 -> 30,
// 256 rows 127 -> 69, 2,048 rows 577 -> 375.
constexpr int SAMPLE_THREADS = 256;
constexpr int SAMPLE_BLOCKS = 4;        // resident per SM
constexpr int SAMPLE_QUEUE = 160;       // per-warp queue of candidates that passed the bound: 32 waiting + up to 128 new

// Bound of the words (as 2^23 + (w >> 9)) below which no candidate with a logit up to l can beat the score s; unit = log2(e) / T and
// shift = -s log2(e) plus a slack of 5e-4 (18 + |s|).  (The noise lies between -2.9 and 16.7, so only where |l / T| < |s| + 18 does the slack have to
// cover the float error of l / T - s, which is 1e-6 of the two.)  With a finite shift a logit of -inf is refused, and one that overflows to it:
// masked ids cost what others do (when they passed, as a NaN: 256 rows, 90 % of 151,936 ids at -inf, 441 us against 73).
__device__ __forceinline__ float word_limit(float l, float unit, float shift) {
    float x;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(x) : "f"(fmaf(l, unit, shift)));
    return fmaf(x, -8388608.f * 1.001f, 16777214.f);       // 2^24 - (2^23 x 1.001 + 2)
}
__device__ __forceinline__ float word_value(uint32_t w) { return __uint_as_float(0x4b000000u | (w >> 9)); }       // 2^23 + (w >> 9)

__device__ __forceinline__ void scan_blocks(Top2& t, const float* __restrict__ lg, int vocab, int b_begin, int b_end,
                                            float temperature, uint32_t c1, uint32_t c2, uint32_t c3, uint32_t k0, uint32_t k1,
                                            uint2* __restrict__ queue /*this warp's SAMPLE_QUEUE slots*/, volatile int32_t* bound /*of the thread block, ordered form; -inf*/) {
    constexpr int U = 2;                        // blocks of a thread in hand; as many more are on their way from memory
    constexpr float LOG2E = 1.4426950408889634f;
    const int lane = threadIdx.x & 31;
    const uint32_t lt_mask = (1u << lane) - 1u;
    const PhiloxKeys keys(k0, k1);
    // While no bound is known every id passes: shift = +inf, or ALL_BUT_INF once seed() has noted the lowest id that could be the answer
    // where every score is -inf (unit is then small enough for every other logit to pass).
    constexpr float ALL_BUT_INF = 3e38f;
    int32_t bound_for = score_to_ordered(-INFINITY);
    float unit = 1e-3f, shift = INFINITY;
    int queued = 0;                             // warp-uniform
    auto set_bound = [&](int32_t b) {
        bound_for = b;
        const float s = ordered_to_score(b);
        unit = LOG2E / temperature;
        // (a temperature without a reciprocal: everything passes; two certain ids: only such ids do -- everything took 242 us instead of 75, 256 rows)
        shift = !(unit < INFINITY) ? NAN : s < INFINITY ? fmaf(-s, LOG2E, 5e-4f * LOG2E * (18.f + fabsf(s))) : -INFINITY;
    };
    auto share_bound = [&](float best, float second) {          // second-best of the warp's scores: a lower bound of the row's
        const float now = ordered_to_score(bound_for);
        if (__popc(__ballot_sync(0xffffffffu, best > now)) + __popc(__ballot_sync(0xffffffffu, second > now)) < 2) return;
        const Top2 w = top2_warp_reduce(Top2{best, second, 0});
        if (w.second > now) {
            const int32_t b = score_to_ordered(w.second);
            if (lane == 0) atomicMax(const_cast<int32_t*>(bound), b);
            set_bound(b);
        }
    };
    auto drain = [&](int keep) {                // scores queued candidates, 32 at a time, until at most `keep` remain
        while (queued > keep) {
            const int take = min(32, queued);
            __syncwarp();
            if (lane < take) {
                const uint2 c = queue[queued - take + lane];
                top2_push_unordered(t, lg[c.x] / temperature + gumbel_from_word(c.y), (int)c.x);
            }
            queued -= take;
            share_bound(t.best, t.second);
            __syncwarp();
        }
    };
    // One candidate per lane, the one with the largest word, for a first bound (not folded: it is scored again later), and the lowest id of
    // each lane that is a number, as a candidate of score -inf.
    auto seed = [&](bool in, int b, const Philox4& w, const float4& l) {
        const uint32_t top = max(max(w.x, w.y), max(w.z, w.w));
        const float at = top == w.x ? l.x : (top == w.y ? l.y : (top == w.z ? l.z : l.w));
        const float s = in ? at / temperature + gumbel_from_word(top) : -INFINITY;
        const float ll[4] = {l.x, l.y, l.z, l.w};
#pragma unroll
        for (int i = 3; i >= 0; --i)
            if (in && b * 4 + i < vocab && ll[i] == ll[i]) t.idx = b * 4 + i;
        if (bound_for == score_to_ordered(-INFINITY) && __any_sync(0xffffffffu, t.idx != 0x7fffffff)) shift = ALL_BUT_INF;
        share_bound(s > -INFINITY ? s : -INFINITY /*NaN too*/, -INFINITY);
    };
    auto consider = [&](bool in, int b, const Philox4& w, const float4& l) {
        const uint32_t top = max(max(w.x, w.y), max(w.z, w.w));
        const float most = fmaxf(fmaxf(l.x, l.y), fmaxf(l.z, l.w));
        if (!__any_sync(0xffffffffu, in && !(word_value(top) <= word_limit(most, unit, shift)))) return;
        const uint32_t ww[4] = {w.x, w.y, w.z, w.w};
        const float ll[4] = {l.x, l.y, l.z, l.w};
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const int v = b * 4 + i;
            const bool pass = in && v < vocab && !(word_value(ww[i]) <= word_limit(ll[i], unit, shift));
            const uint32_t m = __ballot_sync(0xffffffffu, pass);
            if (pass) queue[queued + __popc(m & lt_mask)] = make_uint2((uint32_t)v, ww[i]);
            queued += __popc(m);
        }
        drain(31);
    };
    auto refresh = [&]() {
        const int32_t b = *bound;
        if (__any_sync(0xffffffffu, b > bound_for)) set_bound(__reduce_max_sync(0xffffffffu, b));
    };
    bool first = true;
    int base = b_begin + (int)(threadIdx.x - lane);          // trip counts are warp-uniform (shuffles and ballots need every lane)
    // rounds in which all of the warp's blocks are whole and their logits can be read as vectors
    const int whole = (reinterpret_cast<uintptr_t>(lg) & 15u) == 0 ? min(b_end, vocab >> 2) - ((U - 1) * SAMPLE_THREADS + 31) : 0;
    if (base < whole) {
        const float4* p = reinterpret_cast<const float4*>(lg) + base + lane;
        float4 next[U];
#pragma unroll
        for (int u = 0; u < U; ++u) next[u] = p[u * SAMPLE_THREADS];
#pragma unroll 1
        for (; base < whole; base += U * SAMPLE_THREADS) {
            float4 l[U];
            Philox4 w[U];
#pragma unroll
            for (int u = 0; u < U; ++u) l[u] = next[u];
            p += U * SAMPLE_THREADS;
            if (base + U * SAMPLE_THREADS < whole)
#pragma unroll
                for (int u = 0; u < U; ++u) next[u] = p[u * SAMPLE_THREADS];
#pragma unroll
            for (int u = 0; u < U; ++u) w[u] = philox4x32_10((uint32_t)(base + u * SAMPLE_THREADS + lane), c1, c2, c3, keys);
            refresh();
            if (first) { first = false; seed(true, base + lane, w[0], l[0]); }
#pragma unroll
            for (int u = 0; u < U; ++u) consider(true, base + u * SAMPLE_THREADS + lane, w[u], l[u]);
        }
    }
#pragma unroll 1
    for (; base < b_end; base += SAMPLE_THREADS) {
        const int b = base + lane;
        float l[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) l[i] = b < b_end && 4 * b + i < vocab ? lg[4 * b + i] : -INFINITY;
        const float4 l4 = make_float4(l[0], l[1], l[2], l[3]);
        const Philox4 w = philox4x32_10((uint32_t)b, c1, c2, c3, keys);
        refresh();
        if (first) { first = false; seed(b < b_end, b, w, l4); }
        consider(b < b_end, b, w, l4);
    }
    drain(0);
}

// Largest logit / T of v0 <= v < v1 (block-wide); `red` is 33 floats of shared memory.
__device__ __forceinline__ float range_max(const float* __restrict__ lg, int v0, int v1, float temperature, float* red) {
    float m = -INFINITY;
    // 16-byte loads, four in flight per thread: a row is hundreds of KB and one scalar load per thread at a time would
    // leave the pass bound by memory latency
    int v = v0;
    while (v < v1 && (reinterpret_cast<uintptr_t>(lg + v) & 15u) != 0) { if (threadIdx.x == 0) m = fmaxf(m, lg[v]); ++v; }
    const int n4 = (v1 - v) >> 2;
    const float4* p4 = reinterpret_cast<const float4*>(lg + v);
    int i = threadIdx.x;
    for (; i + 3 * (int)blockDim.x < n4; i += 4 * blockDim.x) {
        const float4 a = p4[i], b = p4[i + blockDim.x], c = p4[i + 2 * blockDim.x], d = p4[i + 3 * blockDim.x];
        m = fmaxf(m, fmaxf(fmaxf(fmaxf(a.x, a.y), fmaxf(a.z, a.w)), fmaxf(fmaxf(b.x, b.y), fmaxf(b.z, b.w))));
        m = fmaxf(m, fmaxf(fmaxf(fmaxf(c.x, c.y), fmaxf(c.z, c.w)), fmaxf(fmaxf(d.x, d.y), fmaxf(d.z, d.w))));
    }
    for (; i < n4; i += blockDim.x) { const float4 a = p4[i]; m = fmaxf(m, fmaxf(fmaxf(a.x, a.y), fmaxf(a.z, a.w))); }
    for (int t = v + 4 * n4 + threadIdx.x; t < v1; t += blockDim.x) m = fmaxf(m, lg[t]);
    m = warp_max(m) / temperature;          // temperature > 0: the division is monotone
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (lane == 0) red[warp] = m;
    __syncthreads();
    if (warp == 0) {
        float x = lane < (int)(blockDim.x >> 5) ? red[lane] : -INFINITY;
        x = warp_max(x);
        if (lane == 0) red[32] = x;
    }
    __syncthreads();
    return red[32];
}

// One block per row.
__global__ void __launch_bounds__(SAMPLE_THREADS, SAMPLE_BLOCKS) sample_kernel(const StepDesc* __restrict__ sd, int vocab, const float* __restrict__ logits,
                                                     const int32_t* __restrict__ logits_row, float temperature,
                                                     uint32_t k0, uint32_t k1, const int32_t* __restrict__ row_prompt,
                                                     const int32_t* __restrict__ row_rollout, const int32_t* __restrict__ row_step,
                                                     int step_offset, int32_t* __restrict__ out_tokens,
                                                     const int64_t* __restrict__ out_index, int64_t out_index_offset,
                                                     float* __restrict__ out_gap, const int32_t* __restrict__ prompt_key,
                                                     const DecodeArgsDev* __restrict__ da) {
    grid_dep_wait();
    grid_dep_launch_dependents();
    const int r = blockIdx.x;
    const int64_t ro = r;                   // index into the row arrays
    if (sd != nullptr && r >= sd->n_rows) return;
    if (da != nullptr) {                    // decode step: token buffer, temperature and seed from the device-resident arguments
        out_tokens = da->tokens; temperature = da->temperature; k0 = da->k0; k1 = da->k1;
    }
    const float* lg = logits + (size_t)(logits_row ? logits_row[ro] : r) * vocab;
    const uint32_t c1 = (uint32_t)(row_step[ro] + step_offset), c2 = (uint32_t)row_rollout[ro],
                   c3 = (uint32_t)(prompt_key ? prompt_key[row_prompt[ro]] : row_prompt[ro]);    // key id of the prompt
    Top2 t{-INFINITY, -INFINITY, 0x7fffffff};
    const int n_blocks = (vocab + 3) >> 2;
    __shared__ int32_t bound;
    __shared__ uint2 queue[SAMPLE_THREADS / 32][SAMPLE_QUEUE];
    if (threadIdx.x == 0) bound = score_to_ordered(-INFINITY);
    __syncthreads();
    scan_blocks(t, lg, vocab, 0, n_blocks, temperature, c1, c2, c3, k0, k1, queue[threadIdx.x >> 5], &bound);
    t = top2_warp_reduce(t);
    __shared__ Top2 sh[8];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (lane == 0) sh[warp] = t;
    __syncthreads();
    if (warp == 0) {
        Top2 u = lane < (int)(blockDim.x >> 5) ? sh[lane] : Top2{-INFINITY, -INFINITY, 0x7fffffff};
        u = top2_warp_reduce(u);
        if (lane == 0) {
            const int64_t at = out_index ? out_index[ro] + out_index_offset : (int64_t)r;
            if (at >= 0) out_tokens[at] = u.idx;
            if (out_gap) out_gap[r] = u.best - u.second;
        }
    }
}

// ---------------------------------------------------------------------------------------------
// Two-pass form for small batches: with few rows one block per row leaves most SMs idle, so the vocabulary of a row is
// cut into n_chunks ranges scored by different blocks.  Every range leaves its (best, second, arg-best) in scratch and a
// second kernel folds the ranges in order.  Maxima are exact, so the result is identical to the one-pass kernel's.
// ---------------------------------------------------------------------------------------------
struct Top2Rec { float best, second; int idx; int pad; };

__global__ void __launch_bounds__(SAMPLE_THREADS, SAMPLE_BLOCKS) sample_partial_kernel(const StepDesc* __restrict__ sd, int vocab, int n_chunks,
                                                             const float* __restrict__ logits, const int32_t* __restrict__ logits_row,
                                                             float temperature, uint32_t k0, uint32_t k1,
                                                             const int32_t* __restrict__ row_prompt, const int32_t* __restrict__ row_rollout,
                                                             const int32_t* __restrict__ row_step, int step_offset, Top2Rec* __restrict__ scratch,
                                                             const int32_t* __restrict__ prompt_key, const DecodeArgsDev* __restrict__ da) {
    grid_dep_wait();
    grid_dep_launch_dependents();
    const int r = blockIdx.x, chunk = blockIdx.y;
    const int64_t ro = r;
    if (sd != nullptr && r >= sd->n_rows) return;
    if (da != nullptr) { temperature = da->temperature; k0 = da->k0; k1 = da->k1; }
    const float* lg = logits + (size_t)(logits_row ? logits_row[ro] : r) * vocab;
    const uint32_t c1 = (uint32_t)(row_step[ro] + step_offset), c2 = (uint32_t)row_rollout[ro],
                   c3 = (uint32_t)(prompt_key ? prompt_key[row_prompt[ro]] : row_prompt[ro]);    // key id of the prompt
    Top2 t{-INFINITY, -INFINITY, 0x7fffffff};
    const int n_blocks = (vocab + 3) >> 2;
    const int per_chunk = (n_blocks + n_chunks - 1) / n_chunks;
    const int b_end = min(n_blocks, (chunk + 1) * per_chunk);
    __shared__ int32_t bound;
    __shared__ uint2 queue[SAMPLE_THREADS / 32][SAMPLE_QUEUE];
    if (threadIdx.x == 0) bound = score_to_ordered(-INFINITY);
    __syncthreads();
    scan_blocks(t, lg, vocab, chunk * per_chunk, b_end, temperature, c1, c2, c3, k0, k1, queue[threadIdx.x >> 5], &bound);
    t = top2_warp_reduce(t);
    __shared__ Top2 sh[8];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (lane == 0) sh[warp] = t;
    __syncthreads();
    if (warp == 0) {
        Top2 u = lane < (int)(blockDim.x >> 5) ? sh[lane] : Top2{-INFINITY, -INFINITY, 0x7fffffff};
        u = top2_warp_reduce(u);
        if (lane == 0) scratch[(size_t)r * n_chunks + chunk] = Top2Rec{u.best, u.second, u.idx, 0};
    }
}

// A warp per row, a record per lane (at most SAMPLE_MAX_CHUNKS = 32; the merge is order-independent: equal scores keep the lowest id).
constexpr int REDUCE_ROWS = 4;          // rows (warps) of a block
__global__ void __launch_bounds__(32 * REDUCE_ROWS) sample_reduce_kernel(const StepDesc* __restrict__ sd, int n_rows, int n_chunks,
                                     const Top2Rec* __restrict__ scratch, int32_t* __restrict__ out_tokens, const int64_t* __restrict__ out_index,
                                     int64_t out_index_offset, float* __restrict__ out_gap, const DecodeArgsDev* __restrict__ da) {
    grid_dep_wait();
    grid_dep_launch_dependents();
    const int r = blockIdx.x * REDUCE_ROWS + (threadIdx.x >> 5), lane = threadIdx.x & 31;
    const int64_t ro = r;
    if (r >= (sd != nullptr ? sd->n_rows : n_rows)) return;
    if (da != nullptr) out_tokens = da->tokens;
    Top2 t{-INFINITY, -INFINITY, 0x7fffffff};
    if (lane < n_chunks) {
        const Top2Rec x = scratch[(size_t)r * n_chunks + lane];
        t = Top2{x.best, x.second, x.idx};
    }
    t = top2_warp_reduce(t);
    if (lane != 0) return;
    const int64_t at = out_index ? out_index[ro] + out_index_offset : (int64_t)r;
    if (at >= 0) out_tokens[at] = t.idx;
    if (out_gap) out_gap[r] = t.best - t.second;
}

// log softmax(logits / T)[token]: the behaviour log-probability of an already drawn token.  One block per row;
// max and sum of exponentials are block reductions in a fixed shape, so the value does not depend on timing.
__global__ void __launch_bounds__(256) token_logprob_kernel(const StepDesc* __restrict__ sd, int vocab, const float* __restrict__ logits,
                                                            const int32_t* __restrict__ logits_row, float temperature,
                                                            const int32_t* __restrict__ tokens, const int64_t* __restrict__ tok_index,
                                                            int64_t tok_index_offset, float* __restrict__ out,
                                                            const int64_t* __restrict__ out_index, int64_t out_index_offset,
                                                            const DecodeArgsDev* __restrict__ da) {
    grid_dep_wait();
    grid_dep_launch_dependents();
    const int r = blockIdx.x;
    const int64_t ro = r;
    if (sd != nullptr && r >= sd->n_rows) return;
    if (da != nullptr) { tokens = da->tokens; out = da->logprobs; temperature = da->temperature; }
    const float* lg = logits + (size_t)(logits_row ? logits_row[ro] : r) * vocab;
    __shared__ float red[33];
    const float mx = range_max(lg, 0, vocab, temperature, red);          // max of logits / T
    const float inv_t = 1.f / temperature;
    float s = 0.f;
    {
        // 16-byte loads, four in flight per thread (one scalar load at a time leaves the pass bound by memory latency);
        // every thread adds its elements in a fixed order, so the sum does not depend on timing
        int v = 0;
        while (v < vocab && (reinterpret_cast<uintptr_t>(lg + v) & 15u) != 0) { if (threadIdx.x == 0) s += expf(lg[v] * inv_t - mx); ++v; }
        const int n4 = (vocab - v) >> 2;
        const float4* p4 = reinterpret_cast<const float4*>(lg + v);
        auto add4 = [&](const float4 a) {
            s += expf(a.x * inv_t - mx); s += expf(a.y * inv_t - mx); s += expf(a.z * inv_t - mx); s += expf(a.w * inv_t - mx);
        };
        int i = threadIdx.x;
        for (; i + 3 * (int)blockDim.x < n4; i += 4 * blockDim.x) {
            const float4 a = p4[i], b = p4[i + blockDim.x], c = p4[i + 2 * blockDim.x], d = p4[i + 3 * blockDim.x];
            add4(a); add4(b); add4(c); add4(d);
        }
        for (; i < n4; i += blockDim.x) add4(p4[i]);
        for (int t = v + 4 * n4 + threadIdx.x; t < vocab; t += blockDim.x) s += expf(lg[t] * inv_t - mx);
    }
    s = block_sum(s, red);
    if (threadIdx.x == 0) {
        const int64_t ti = tok_index ? tok_index[ro] + tok_index_offset : (int64_t)r;
        if (ti < 0) return;
        const int tok = tokens[ti];
        const float lp = (tok >= 0 && tok < vocab) ? lg[tok] * inv_t - mx - logf(s) : -INFINITY;
        out[out_index ? out_index[ro] + out_index_offset : (int64_t)r] = lp;
    }
}

constexpr int SAMPLE_MAX_CHUNKS = 32;
// Ranges per row: the number that minimises (waves of the grid) x (a range's ids + the fixed cost of a block, as long as 3,000 ids take);
// 1 means the one-pass kernel.  (As many as give four blocks per SM or the next more: 768 blocks in two waves at 256 rows.  With a fixed
// cost of 2 % of the row whatever its length, 1,024 rows of 2,048 ids were cut into 4,096 ranges: 41 us, one pass 22; 600 rows of 8,192 44 against 33.)
inline int sample_chunks(int n_rows, int vocab, int num_sms) {
    const long long slots = (long long)SAMPLE_BLOCKS * num_sms;
    int best = 1;
    double best_cost = -1.;
    for (int c = 1; c <= SAMPLE_MAX_CHUNKS; ++c) {
        const double cost = (double)(((long long)n_rows * c + slots - 1) / slots) * (1. / c + 3000. / vocab);
        if (best_cost < 0. || cost < best_cost * 0.98) { best_cost = cost; best = c; }
    }
    return best;
}

}  // namespace pc

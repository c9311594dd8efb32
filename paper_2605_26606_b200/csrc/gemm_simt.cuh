// C[M, N] = A[M, K] * W[N, K]^T with float accumulation on the plain FP32 pipes.
// Used for float32 models (TF32 tensor cores would break their 1e-4 logit tolerance) and as the
// reference the tensor-core GEMMs are checked against.  Each output element sums its K products in
// a fixed order that does not depend on M, so a row's result does not depend on its batch mates.
//
// These GEMMs are latency: a decode step of the small float32 configuration multiplies up to a hundred rows with matrices
// that sit in L2.  So a CTA takes few rows (RT = 8 or 16; 64 for prefills) x 32 columns, keeps eight k-blocks of 64 in flight
// (cp.async), and its eight warps share the k-blocks: warp w adds the k = 8 w .. 8 w + 7 of every block, and the eight partial
// sums of an element are added in warp order.  With one 64 x 64 tile per CTA and a serial k loop of two barriers per 16 k
// (4 .. 32 CTAs) the down projection took 28.6 us at 96 rows; it takes a tenth of that now.
#pragma once

#include <cstring>

#include "common.cuh"

namespace pc {

// Epilogues receive four consecutive columns [col0, col0+4) of one row; n_valid of them are inside N.
struct EpiStoreF32 {            // C = acc (+ bias)
    static constexpr bool kNorm = true;       // the activations are a residual stream whose RMSNorm is applied here
    float* C; int ldc; const float* bias;
    __device__ __forceinline__ void operator()(int row, int col0, const float* acc, int n_valid) const {
        float* dst = C + (size_t)row * ldc + col0;
        if (n_valid == 4 && (ldc & 3) == 0 && bias == nullptr) {
            *reinterpret_cast<float4*>(dst) = make_float4(acc[0], acc[1], acc[2], acc[3]);
            return;
        }
        for (int i = 0; i < n_valid; ++i) dst[i] = acc[i] + (bias ? bias[col0 + i] : 0.f);
    }
};
struct EpiResidual {            // H += acc   (float residual stream; N is a multiple of 8)
    static constexpr bool kNorm = false;
    float* H; int ldc;
    __device__ __forceinline__ void operator()(int row, int col0, const float* acc, int n_valid) const {
        float4* dst = reinterpret_cast<float4*>(H + (size_t)row * ldc + col0);
        float4 h = *dst;
        h.x += acc[0]; h.y += acc[1]; h.z += acc[2]; h.w += acc[3];
        *dst = h;
    }
};
struct EpiSwiGLU {              // columns (2j, 2j+1) = (gate_j, up_j)  ->  out[row, j] = silu(gate) * up
    static constexpr bool kNorm = true;
    float* out; int ld;
    __device__ __forceinline__ void operator()(int row, int col0, const float* acc, int n_valid) const {
        for (int i = 0; i + 1 < n_valid; i += 2) {
            const float g = acc[i], u = acc[i + 1];
            out[(size_t)row * ld + ((col0 + i) >> 1)] = g / (1.f + expf(-g)) * u;
        }
    }
};

constexpr int SIMT_BN = 32, SIMT_BK = 64, SIMT_WARPS = 8;
constexpr int SIMT_LD = SIMT_BK + 4;        // padded row of a tile: eight lanes' 16-byte loads of different rows hit different banks
template <int RT> __host__ __device__ constexpr int simt_stages() { return RT >= 64 ? 4 : 8; }
template <int RT> __host__ __device__ constexpr int simt_stage_floats() { return (RT + SIMT_BN + 1) * SIMT_LD; }      // activations, weights, gain
template <int RT> __host__ __device__ constexpr int simt_smem_bytes() { return simt_stages<RT>() * simt_stage_floats<RT>() * 4; }
// A launch of more CTAs than two per SM gets only the stages it fills (K = 256: four), so that more of them fit an SM: vocabulary 2,048 x
// 128 rows are 512 CTAs, on 148 SMs two rounds with eight stages (11.6 us), one with four (6.6).  Smaller launches keep them all: a dependent
// CTA that settles beside those still at work slows them (down projection of 128 rows 4.0 -> 5.2 us).
template <int RT> inline int simt_smem_bytes(int K, long long ctas, int num_sms) {
    if (ctas <= 2 * num_sms) return simt_smem_bytes<RT>();
    const int blocks = (K + SIMT_BK - 1) / SIMT_BK, used = blocks < simt_stages<RT>() ? blocks : simt_stages<RT>();
    const int tiles = used * simt_stage_floats<RT>() * 4, sums = SIMT_WARPS * RT * (SIMT_BN + 1) * 4;
    return tiles > sums ? tiles : sums;
}
// RMSNorm in front of a GEMM (Epi::kNorm):  RMSNorm(x; gain) W^T = rstd * (x (gain * W)^T).  Every CTA has its rows' squares in hand anyway; a
// norm kernel of its own was 4 us of a float32 decode step, five times.
struct SimtNorm {
    const float* gain; float eps;
    const int32_t* src;             // row src[r] of the activations instead of r, or nullptr
};

// 16 bytes into shared memory, zeros where the source is outside its matrix
__device__ __forceinline__ void cp_async16(uint32_t dst, const void* src, bool inside) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(inside ? 16 : 0) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N> __device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }

// Launched as a programmatic dependent: the weight tiles are requested while the kernel before this one still runs, and the next kernel
// may start as soon as that one has ended.
template <int RT, class Epi>
__global__ void __launch_bounds__(32 * SIMT_WARPS) gemm_simt_kernel(const StepDesc* __restrict__ sd, const float* __restrict__ A, const float* __restrict__ W,
                                                                    int M, int N, int K, SimtNorm nm, Epi epi) {
    constexpr int STAGES = simt_stages<RT>(), X_ROWS = RT, STAGE_FLOATS = simt_stage_floats<RT>(), QUADS = SIMT_BK / 4;
    extern __shared__ __align__(16) float smem[];
    const int m0 = blockIdx.y * RT, n0 = blockIdx.x * SIMT_BN, tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int blocks = (K + SIMT_BK - 1) / SIMT_BK;
    auto load_w = [&](int kb) {
        const uint32_t base = (uint32_t)__cvta_generic_to_shared(smem + (kb % STAGES) * STAGE_FLOATS + X_ROWS * SIMT_LD);
#pragma unroll
        for (int i = 0; i < SIMT_BN * QUADS / (32 * SIMT_WARPS); ++i) {
            const int u = tid + i * 32 * SIMT_WARPS, r = u / QUADS, k = kb * SIMT_BK + (u % QUADS) * 4;
            const bool in = n0 + r < N && k < K;
            cp_async16(base + (r * SIMT_LD + (u % QUADS) * 4) * 4, W + (in ? (size_t)(n0 + r) * K + k : 0), in);
        }
        if (Epi::kNorm && tid < QUADS) {
            const int k = kb * SIMT_BK + tid * 4;
            cp_async16(base + (SIMT_BN * SIMT_LD + tid * 4) * 4, nm.gain + (k < K ? k : 0), k < K);
        }
    };
    auto load_x = [&](int kb) {
        const uint32_t base = (uint32_t)__cvta_generic_to_shared(smem + (kb % STAGES) * STAGE_FLOATS);
#pragma unroll
        for (int i = 0; i < (X_ROWS * QUADS + 32 * SIMT_WARPS - 1) / (32 * SIMT_WARPS); ++i) {
            const int u = tid + i * 32 * SIMT_WARPS, r = u / QUADS, k = kb * SIMT_BK + (u % QUADS) * 4;
            if (X_ROWS * QUADS % (32 * SIMT_WARPS) != 0 && u >= X_ROWS * QUADS) break;
            const bool in = m0 + r < M && k < K;
            cp_async16(base + (r * SIMT_LD + (u % QUADS) * 4) * 4, A + (in ? (size_t)(Epi::kNorm && nm.src != nullptr ? nm.src[m0 + r] : m0 + r) * K + k : 0), in);
        }
    };
    const int first = min(STAGES - 1, blocks);
    for (int kb = 0; kb < first; ++kb) load_w(kb);
    grid_dep_wait();
    grid_dep_launch_dependents();
    if (sd != nullptr) M = sd->n_rows;          // live row count; the grid was sized for an upper bound
    if (m0 >= M) { cp_async_commit(); cp_async_wait<0>(); return; }
    for (int kb = 0; kb < STAGES - 1; ++kb) {
        if (kb < first) load_x(kb);
        cp_async_commit();                      // (a group per block, empty ones too: the count below stays the same)
    }
    float acc[RT], ss[(RT + 31) / 32];          // ss: squares of rows lane, lane + 32 over this warp's k
#pragma unroll
    for (int r = 0; r < RT; ++r) acc[r] = 0.f;
#pragma unroll
    for (int r = 0; r < (RT + 31) / 32; ++r) ss[r] = 0.f;
    for (int kb = 0; kb < blocks; ++kb) {
        cp_async_wait<STAGES - 2>();
        __syncthreads();                        // block kb has arrived for everybody, and everybody is done with block kb - 1
        if (kb + STAGES - 1 < blocks) { load_w(kb + STAGES - 1); load_x(kb + STAGES - 1); }
        cp_async_commit();
        const float* xs = smem + (kb % STAGES) * STAGE_FLOATS + warp * 8;
        const float* ws = smem + (kb % STAGES) * STAGE_FLOATS + (X_ROWS + lane) * SIMT_LD + warp * 8;
#pragma unroll
        for (int q = 0; q < 8; q += 4) {
            float4 w = *reinterpret_cast<const float4*>(ws + q);
            if (Epi::kNorm) {
                const float4 g = *reinterpret_cast<const float4*>(ws + (SIMT_BN - lane) * SIMT_LD + q);
                w.x *= g.x; w.y *= g.y; w.z *= g.z; w.w *= g.w;
#pragma unroll
                for (int i = 0; i < (RT + 31) / 32; ++i) {
                    if (lane + 32 * i < RT) {
                        const float4 x = *reinterpret_cast<const float4*>(xs + (lane + 32 * i) * SIMT_LD + q);
                        ss[i] = fmaf(x.x, x.x, fmaf(x.y, x.y, fmaf(x.z, x.z, fmaf(x.w, x.w, ss[i]))));
                    }
                }
            }
#pragma unroll
            for (int r = 0; r < RT; ++r) {
                const float4 x = *reinterpret_cast<const float4*>(xs + r * SIMT_LD + q);
                acc[r] = fmaf(x.x, w.x, acc[r]);
                acc[r] = fmaf(x.y, w.y, acc[r]);
                acc[r] = fmaf(x.z, w.z, acc[r]);
                acc[r] = fmaf(x.w, w.w, acc[r]);
            }
        }
    }
    cp_async_wait<0>();
    __syncthreads();
#pragma unroll
    for (int r = 0; r < RT; ++r) smem[(warp * RT + r) * SIMT_BN + lane] = acc[r];
    float* squares = smem + SIMT_WARPS * RT * SIMT_BN;          // [warp][row]
    if (Epi::kNorm) {
#pragma unroll
        for (int i = 0; i < (RT + 31) / 32; ++i)
            if (lane + 32 * i < RT) squares[warp * RT + lane + 32 * i] = ss[i];
    }
    __syncthreads();
    for (int u = tid; u < RT * SIMT_BN / 4; u += 32 * SIMT_WARPS) {
        const int r = u / (SIMT_BN / 4), c = u % (SIMT_BN / 4) * 4;
        if (m0 + r >= M || n0 + c >= N) continue;
        float s[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
        for (int w = 0; w < SIMT_WARPS; ++w) {
            const float4 v = *reinterpret_cast<const float4*>(smem + (w * RT + r) * SIMT_BN + c);
            s[0] += v.x; s[1] += v.y; s[2] += v.z; s[3] += v.w;
        }
        if (Epi::kNorm) {
            float t = 0.f;
#pragma unroll
            for (int w = 0; w < SIMT_WARPS; ++w) t += squares[w * RT + r];
            const float rstd = rsqrtf(t / (float)K + nm.eps);
#pragma unroll
            for (int i = 0; i < 4; ++i) s[i] *= rstd;
        }
        epi(m0 + r, n0 + c, s, min(4, N - (n0 + c)));
    }
}

// Must run once per epilogue and device before its first launch (raises the dynamic shared memory limits).
template <class Epi>
inline cudaError_t configure_gemm_simt() {
    cudaError_t e = cudaFuncSetAttribute(gemm_simt_kernel<64, Epi>, cudaFuncAttributeMaxDynamicSharedMemorySize, simt_smem_bytes<64>());
    if (e == cudaSuccess) e = cudaFuncSetAttribute(gemm_simt_kernel<16, Epi>, cudaFuncAttributeMaxDynamicSharedMemorySize, simt_smem_bytes<16>());
    if (e == cudaSuccess) e = cudaFuncSetAttribute(gemm_simt_kernel<8, Epi>, cudaFuncAttributeMaxDynamicSharedMemorySize, simt_smem_bytes<8>());
    return e;
}

template <int RT, class Epi>
inline cudaError_t launch_gemm_simt_rt(cudaStream_t st, bool dep, int num_sms, const StepDesc* sd, const float* A, const float* W, int M, int N, int K, SimtNorm nm, Epi epi) {
    cudaLaunchConfig_t cfg;
    memset(&cfg, 0, sizeof(cfg));
    cfg.gridDim = dim3((N + SIMT_BN - 1) / SIMT_BN, (M + RT - 1) / RT); cfg.blockDim = dim3(32 * SIMT_WARPS);
    cfg.dynamicSmemBytes = simt_smem_bytes<RT>(K, (long long)cfg.gridDim.x * cfg.gridDim.y, num_sms); cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr; cfg.numAttrs = dep ? 1 : 0;
    return cudaLaunchKernelEx(&cfg, gemm_simt_kernel<RT, Epi>, sd, A, W, M, N, K, nm, epi);
}

// Rows per CTA: 64 read the weights fewest times and are for passes with several waves of such tiles (at one wave, 2048 columns x
// 128 rows, the tile's own latency shows: 11.5 us); 16 from about a CTA per SM on.
template <class Epi>
inline cudaError_t launch_gemm_simt(cudaStream_t st, bool dep, int num_sms, const StepDesc* sd, const float* A, const float* W, int M, int N, int K, SimtNorm nm, Epi epi) {
    if (M <= 0 || N <= 0) return cudaSuccess;
    const long long cols = (N + SIMT_BN - 1) / SIMT_BN;
    if (cols * ((M + 63) / 64) >= 512) return launch_gemm_simt_rt<64>(st, dep, num_sms, sd, A, W, M, N, K, nm, epi);
    if (cols * ((M + 15) / 16) >= 128) return launch_gemm_simt_rt<16>(st, dep, num_sms, sd, A, W, M, N, K, nm, epi);
    return launch_gemm_simt_rt<8>(st, dep, num_sms, sd, A, W, M, N, K, nm, epi);
}

}  // namespace pc

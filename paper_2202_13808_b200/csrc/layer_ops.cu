// The parts of a Linear layer's backward pass around the weight gradient: the derivative of the GELU in front of it, the bias
// gradient and the rounding of the weight gradient to the parameter's type (see layer_ops.h).
#include "layer_ops.h"

#include "common.cuh"
#include "sm100_ptx.cuh"

namespace dropit {

namespace {

__device__ __forceinline__ float bf16_to_float(uint32_t bits) { return __uint_as_float(bits << 16); }
// Two floats as packed bf16, round to nearest even.
__device__ __forceinline__ uint32_t pack_bf16(float lo, float hi) {
    uint32_t r;
    asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(r) : "f"(hi), "f"(lo));
    return r;
}

// GELU'(x) = Phi(x) + x phi(x)
__device__ __forceinline__ float gelu_derivative(float x) {
    return 0.5f * (1.0f + erff(x * 0.70710678f)) + x * 0.39894228f * expf(-0.5f * x * x);
}

// The derivative is looked up: x is bf16, and the patterns of 2^-9 <= |x| < 8 (all but a few per mille of a GELU's inputs) fill
// 12 KB of shared memory.  Bound by HBM (two reads, one write, 58 MB at 3152 x 3072: 9 us); evaluated per element the arithmetic sets the
// pace: 16 us with PyTorch's kernel at that size, 13.7 us here, the wait for the kernel in front included.
constexpr uint32_t kKeyLo = 118u << 7, kKeyHi = 130u << 7, kSpan = kKeyHi - kKeyLo;
constexpr int kGeluThreads = 512;
__global__ void __launch_bounds__(kGeluThreads)
gelu_backward_kernel(const uint4* __restrict__ dy, const uint4* __restrict__ x, uint4* __restrict__ dx, int64_t n) {
    __shared__ float table[2 * kSpan];
    for (uint32_t i = threadIdx.x; i < 2 * kSpan; i += kGeluThreads)
        table[i] = gelu_derivative(bf16_to_float(i < kSpan ? kKeyLo + i : 0x8000u | (kKeyLo + i - kSpan)));
    __syncthreads();
    ptx::grid_dependency_wait();
    auto derivative = [&](uint32_t bits) {
        const uint32_t i = (bits & 0x7FFFu) - kKeyLo;
        return i < kSpan ? table[i + (bits >> 15) * kSpan] : gelu_derivative(bf16_to_float(bits));
    };
    auto two = [&](uint32_t g, uint32_t v) {
        return pack_bf16(bf16_to_float(g & 0xFFFFu) * derivative(v & 0xFFFFu), bf16_to_float(g >> 16) * derivative(v >> 16));
    };
    const int64_t vecs = n / 8, stride = (int64_t)gridDim.x * kGeluThreads;
    int64_t i = (int64_t)blockIdx.x * kGeluThreads + threadIdx.x;
    for (; i + stride < vecs; i += 2 * stride) {        // two vectors in flight
        const uint4 g0 = ld_stream(dy + i), v0 = ld_stream(x + i), g1 = ld_stream(dy + i + stride), v1 = ld_stream(x + i + stride);
        dx[i] = make_uint4(two(g0.x, v0.x), two(g0.y, v0.y), two(g0.z, v0.z), two(g0.w, v0.w));
        dx[i + stride] = make_uint4(two(g1.x, v1.x), two(g1.y, v1.y), two(g1.z, v1.z), two(g1.w, v1.w));
    }
    if (i < vecs) {
        const uint4 g = ld_stream(dy + i), v = ld_stream(x + i);
        dx[i] = make_uint4(two(g.x, v.x), two(g.y, v.y), two(g.z, v.z), two(g.w, v.w));
    }
    const int64_t e = vecs * 8 + (int64_t)blockIdx.x * kGeluThreads + threadIdx.x;      // the last n mod 8 elements
    if (e < n)
        reinterpret_cast<uint16_t*>(dx)[e] = (uint16_t)pack_bf16(bf16_to_float(reinterpret_cast<const uint16_t*>(dy)[e]) *
                                                                 derivative(reinterpret_cast<const uint16_t*>(x)[e]), 0.f);
}

// Clusters of eight CTAs.  The first ones sum 64 columns of dy each: a CTA takes an eighth of the rows, its threads (row group,
// 8 columns), the partial sums meet in shared memory and then in the first CTA, in order.  The others round dw to bf16.  Bound by latency:
// 6.3 us at 3152 tokens, 768 x 3072, where a fill, a column sum and a cast in sequence took 16 us.
constexpr int kSumCtas = 8, kSumThreads = 256, kSumCols = 64;
__global__ void __cluster_dims__(kSumCtas, 1, 1) __launch_bounds__(kSumThreads)
finish_linear_kernel(const float* __restrict__ dw, uint16_t* __restrict__ dw_out, int64_t count, const uint16_t* __restrict__ dy, int64_t M,
                     int64_t Cz, uint16_t* __restrict__ db, int sum_clusters) {
    __shared__ __align__(16) float rows[kSumThreads / 8][kSumCols];
    __shared__ __align__(16) float ctas[kSumCtas][kSumCols];      // of the first CTA: what the others found
    const int cluster = blockIdx.x / kSumCtas, rank = blockIdx.x % kSumCtas;
    if (cluster < sum_clusters) ptx::cluster_sync_all();          // the first CTA runs before the others write to its shared memory
    ptx::grid_dependency_wait();
    if (cluster < sum_clusters) {
        const int group = threadIdx.x / 8, c8 = (threadIdx.x % 8) * 8;
        const int64_t col = (int64_t)cluster * kSumCols + c8;
        float acc[8] = {};
        if (col < Cz) {
            const int64_t step = (int64_t)kSumCtas * (kSumThreads / 8);
            auto add = [&](const uint4& v) {
                const uint32_t w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    acc[2 * e] += bf16_to_float(w[e] & 0xFFFFu);
                    acc[2 * e + 1] += bf16_to_float(w[e] >> 16);
                }
            };
            int64_t r = (int64_t)rank * (kSumThreads / 8) + group;
            for (; r + 3 * step < M; r += 4 * step) {             // four rows in flight
                uint4 v[4];
#pragma unroll
                for (int u = 0; u < 4; ++u) v[u] = ld_stream(reinterpret_cast<const uint4*>(dy + (r + u * step) * Cz + col));
#pragma unroll
                for (int u = 0; u < 4; ++u) add(v[u]);
            }
            for (; r < M; r += step) add(ld_stream(reinterpret_cast<const uint4*>(dy + r * Cz + col)));
        }
#pragma unroll
        for (int e = 0; e < 8; ++e) rows[group][c8 + e] = acc[e];
        __syncthreads();
        if (threadIdx.x < kSumCols) {
            float s = 0.f;
            for (int g = 0; g < kSumThreads / 8; ++g) s += rows[g][threadIdx.x];
            ptx::st_cluster_u32(ptx::map_shared_to_cta(ptx::smem_u32(&ctas[rank][threadIdx.x]), 0), __float_as_uint(s));
        }
        ptx::cluster_sync_all();
        if (rank == 0 && threadIdx.x < kSumCols) {
            const int64_t c = (int64_t)cluster * kSumCols + threadIdx.x;
            float s = 0.f;
            for (int k = 0; k < kSumCtas; ++k) s += ctas[k][threadIdx.x];
            if (c < Cz) db[c] = (uint16_t)pack_bf16(s, 0.f);
        }
    } else {
        const int64_t vecs = count / 8, stride = (int64_t)(gridDim.x - sum_clusters * kSumCtas) * kSumThreads;
        const int64_t first = (int64_t)(blockIdx.x - sum_clusters * kSumCtas) * kSumThreads + threadIdx.x;
        const float4* src = reinterpret_cast<const float4*>(dw);
        for (int64_t i = first; i < vecs; i += stride) {
            const float4 a = __ldcs(src + 2 * i), b = __ldcs(src + 2 * i + 1);
            reinterpret_cast<uint4*>(dw_out)[i] = make_uint4(pack_bf16(a.x, a.y), pack_bf16(a.z, a.w), pack_bf16(b.x, b.y), pack_bf16(b.z, b.w));
        }
        for (int64_t e = vecs * 8 + first; e < count; e += stride) dw_out[e] = (uint16_t)pack_bf16(dw[e], 0.f);
    }
}

template <typename... Args>
dropit_status launch_programmatic(void (*kernel)(Args...), int64_t blocks, int threads, cudaStream_t stream, Args... args) {
    cudaLaunchAttribute pdl[1];
    pdl[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    pdl[0].val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)blocks);
    cfg.blockDim = dim3((unsigned)threads);
    cfg.stream = stream;
    cfg.attrs = pdl;
    cfg.numAttrs = 1;
    if (cudaLaunchKernelEx(&cfg, kernel, args...) != cudaSuccess) {
        (void)cudaGetLastError();
        return DROPIT_ERR_CUDA;
    }
    return check_launch();
}

}  // namespace

dropit_status gelu_backward_bf16(const void* dy, const void* x, void* dx, int64_t n, void* cuda_stream) {
    if (n <= 0) return DROPIT_OK;
    int64_t blocks = (n / 8 + kGeluThreads - 1) / kGeluThreads;
    const int64_t resident = (int64_t)sm_count() * 4;
    if (blocks > resident) blocks = resident;
    if (blocks < 1) blocks = 1;
    return launch_programmatic(gelu_backward_kernel, blocks, kGeluThreads, as_stream(cuda_stream), reinterpret_cast<const uint4*>(dy),
                               reinterpret_cast<const uint4*>(x), reinterpret_cast<uint4*>(dx), n);
}

dropit_status finish_linear_backward(const float* dw, void* dw_out, int64_t count, const void* dy, int64_t M, int64_t Cz, void* db,
                                     void* cuda_stream) {
    const int sums = db ? (int)((Cz + kSumCols - 1) / kSumCols) : 0;
    int64_t casts = (count / 8 + kSumThreads * kSumCtas - 1) / (kSumThreads * kSumCtas);
    if (casts > (int64_t)sm_count() / 2) casts = sm_count() / 2;
    if (casts < 1) casts = 1;
    return launch_programmatic(finish_linear_kernel, (sums + casts) * kSumCtas, kSumThreads, as_stream(cuda_stream), dw,
                               reinterpret_cast<uint16_t*>(dw_out), count, reinterpret_cast<const uint16_t*>(dy), M, Cz,
                               reinterpret_cast<uint16_t*>(db), sums);
}

}  // namespace dropit

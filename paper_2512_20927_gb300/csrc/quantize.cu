// Storage formats of the feature table (not in the paper): BF16, and FP8 E4M3
// with one FP32 scale per Gaussian.  The blend and dense kernels decode both
// in registers and accumulate in FP32.
//
// BF16: round to nearest, ties to even (__float2bfloat16_rn).
// FP8:  scale_i = max_c |f_ic| / 448 (1 for an all-zero row), computed in FP32;
//       code_ic = E4M3(f_ic / scale_i) with the division rounded to nearest and
//       the conversion rounding to nearest even and saturating to +-448.
//
// GB300 design: both formats are bound by HBM (each input read once, each
// output written once), so a pass reads 16 bytes per lane and load, with
// several loads of a thread in flight.  FP8 keeps the row in registers
// between its maximum and its codes (one warp per row, rows of up to 1024
// channels) and divides by the row's scale with one reciprocal per row and
// exact FMA corrections per element (quotient() below).
// FP8, 500k rows of 512 (1.28 GB): 360.4 us with 4-byte loads, the row read
// twice and a divide per element; 188.2 us now, 1.00 of a plain copy's rate.
// Rows that 16-byte loads cannot cover (a length that is no multiple of 4, a
// pointer that is not aligned) and longer rows take the element-wise kernels.
#include <cuda_bf16.h>
#include <cuda_fp8.h>

#include "qr_internal.cuh"

namespace qr {
namespace {

__global__ void __launch_bounds__(256)
bf16_kernel(const float *__restrict__ in, int64_t count, uint16_t *__restrict__ out) {
    const int64_t stride = int64_t(gridDim.x) * blockDim.x;
    for (int64_t i = int64_t(blockIdx.x) * blockDim.x + threadIdx.x; i < count; i += stride) {
        const __nv_bfloat16 b = __float2bfloat16_rn(in[i]);
        out[i] = *reinterpret_cast<const uint16_t *>(&b);
    }
}

// Four elements per load; a CTA takes 4 x 256 consecutive loads at a time, so
// each thread has four in flight.  `quads` whole quads, then `rest` elements
// (fewer than 4) by the first threads.
__global__ void __launch_bounds__(256)
bf16_quads_kernel(const float4 *__restrict__ in, int64_t quads, int rest, uint2 *__restrict__ out) {
    const int64_t step = int64_t(gridDim.x) * 1024;
    for (int64_t b = int64_t(blockIdx.x) * 1024 + threadIdx.x; b < quads; b += step) {
        float4 v[4];
#pragma unroll
        for (int u = 0; u < 4; ++u)
            if (b + 256 * u < quads) v[u] = __ldcs(in + b + 256 * u);
#pragma unroll
        for (int u = 0; u < 4; ++u)
            if (b + 256 * u < quads) {
                const __nv_bfloat162 lo = __floats2bfloat162_rn(v[u].x, v[u].y);
                const __nv_bfloat162 hi = __floats2bfloat162_rn(v[u].z, v[u].w);
                __stcs(out + b + 256 * u, make_uint2(*reinterpret_cast<const uint32_t *>(&lo),
                                                     *reinterpret_cast<const uint32_t *>(&hi)));
            }
    }
    if (blockIdx.x == 0 && int(threadIdx.x) < rest) {
        const __nv_bfloat16 t = __float2bfloat16_rn(reinterpret_cast<const float *>(in + quads)[threadIdx.x]);
        reinterpret_cast<uint16_t *>(out + quads)[threadIdx.x] = *reinterpret_cast<const uint16_t *>(&t);
    }
}

__global__ void __launch_bounds__(256)
fp8_rows_kernel(const float *__restrict__ in, int64_t rows, int C, uint8_t *__restrict__ codes,
                float *__restrict__ scale) {
    const int lane = threadIdx.x & 31;
    const int64_t warp = (int64_t(blockIdx.x) * blockDim.x + threadIdx.x) >> 5;
    const int64_t nwarps = (int64_t(gridDim.x) * blockDim.x) >> 5;
    for (int64_t r = warp; r < rows; r += nwarps) {
        const float *f = in + r * C;
        float mx = 0.f;
        for (int c = lane; c < C; c += 32) mx = fmaxf(mx, fabsf(f[c]));
        for (int o = 16; o > 0; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
        const float s = mx > 0.f ? __fdiv_rn(mx, 448.0f) : 1.0f;
        if (lane == 0) scale[r] = s;
        uint8_t *q = codes + r * C;
        for (int c = lane; c < C; c += 32)
            q[c] = uint8_t(__nv_cvt_float_to_fp8(__fdiv_rn(f[c], s), __NV_SATFINITE, __NV_E4M3));
    }
}

// f / s rounded to nearest as far as an E4M3 code can tell, from r = 1 / s
// rounded to nearest: two residual corrections (Markstein, "Computation of
// elementary functions on the IBM RISC System/6000 processor", 1990: a
// quotient within one ulp, corrected once with a correctly rounded
// reciprocal, is the correctly rounded quotient; the first step brings f r
// within one ulp).  The residuals are exact for 2^-64 <= s <= 2^64 unless
// |f / s| is below 2^-60, where the code is a zero of f's sign either way.
__device__ __forceinline__ float quotient(float f, float s, float r) {
    float q = __fmul_rn(f, r);
    q = __fmaf_rn(__fmaf_rn(-q, s, f), r, q);
    q = __fmaf_rn(__fmaf_rn(-q, s, f), r, q);
    return copysignf(q, f);   // f = -0: the corrections lose the sign
}
__device__ __forceinline__ uint32_t codes4(float a, float b, float c, float d) {
    const uint32_t lo = __nv_cvt_float2_to_fp8x2(make_float2(a, b), __NV_SATFINITE, __NV_E4M3);
    const uint32_t hi = __nv_cvt_float2_to_fp8x2(make_float2(c, d), __NV_SATFINITE, __NV_E4M3);
    return lo | hi << 16;
}

// One warp per row of `quads` quads (4 channels), at most 32 V: lane l holds
// quads l, l + 32, ... of the row, so loads are 512 and stores 128 contiguous
// bytes a warp.
template <int V>
__global__ void __launch_bounds__(256)
fp8_quads_kernel(const float4 *__restrict__ in, int64_t rows, int quads,
                 uint32_t *__restrict__ codes, float *__restrict__ scale) {
    const int lane = threadIdx.x & 31;
    const int64_t warp = (int64_t(blockIdx.x) * blockDim.x + threadIdx.x) >> 5;
    const int64_t nwarps = (int64_t(gridDim.x) * blockDim.x) >> 5;
    for (int64_t r = warp; r < rows; r += nwarps) {
        const float4 *f = in + r * quads;
        float4 x[V];
#pragma unroll
        for (int v = 0; v < V; ++v)
            x[v] = lane + 32 * v < quads ? __ldcs(f + lane + 32 * v) : make_float4(0.f, 0.f, 0.f, 0.f);
        float mx = 0.f;
#pragma unroll
        for (int v = 0; v < V; ++v)
            mx = fmaxf(fmaxf(fmaxf(mx, fabsf(x[v].x)), fmaxf(fabsf(x[v].y), fabsf(x[v].z))), fabsf(x[v].w));
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
        const float s = mx > 0.f ? __fdiv_rn(mx, 448.0f) : 1.0f;
        if (lane == 0) scale[r] = s;
        uint32_t *q = codes + r * quads;
        const bool fast = s >= 0x1p-64f && s <= 0x1p64f;
        const float inv = __frcp_rn(s);
#pragma unroll
        for (int v = 0; v < V; ++v) {
            float4 y;
            if (fast) {
                y = make_float4(quotient(x[v].x, s, inv), quotient(x[v].y, s, inv),
                                quotient(x[v].z, s, inv), quotient(x[v].w, s, inv));
            } else {
                y = make_float4(__fdiv_rn(x[v].x, s), __fdiv_rn(x[v].y, s), __fdiv_rn(x[v].z, s),
                                __fdiv_rn(x[v].w, s));
            }
            if (lane + 32 * v < quads) __stcs(q + lane + 32 * v, codes4(y.x, y.y, y.z, y.w));
        }
    }
}

int grid_for(int64_t work, int threads) {
    int dev = 0, sms = 152;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    const int64_t want = (work + threads - 1) / threads;
    return int(want < 1 ? 1 : (want > int64_t(sms) * 8 ? int64_t(sms) * 8 : want));
}

// One CTA per `per` units of work: the CTAs of a pass this even need no
// persistent loop, and a grid that is no multiple of what is resident leaves
// no half-empty last wave (the kernels loop where the grid is capped).
unsigned whole_grid(int64_t work, int per) {
    const int64_t want = (work + per - 1) / per;
    return unsigned(want < 1 ? 1 : (want > (int64_t(1) << 30) ? int64_t(1) << 30 : want));
}
bool aligned(const void *p, uintptr_t bytes) { return (reinterpret_cast<uintptr_t>(p) & (bytes - 1)) == 0; }

}  // namespace
}  // namespace qr

using namespace qr;

extern "C" qr_status qr_quantize_bf16(const float *in, int64_t count, uint16_t *out,
                                      qr_stream stream) {
    if (count < 0 || (count > 0 && (!in || !out))) return QR_ERR_INVALID_ARG;
    if (count == 0) return QR_OK;
    const cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
    if (aligned(in, 16) && aligned(out, 8))
        bf16_quads_kernel<<<whole_grid(count / 4, 1024), 256, 0, st>>>(
            reinterpret_cast<const float4 *>(in), count / 4, int(count % 4), reinterpret_cast<uint2 *>(out));
    else
        bf16_kernel<<<grid_for(count, 256), 256, 0, st>>>(in, count, out);
    count_launch();
    return cudaGetLastError() == cudaSuccess ? QR_OK : QR_ERR_CUDA;
}

extern "C" qr_status qr_quantize_fp8(const float *in, int64_t rows, int32_t C, uint8_t *codes,
                                     float *scale, qr_stream stream) {
    if (rows < 0 || C < 1 || (rows > 0 && (!in || !codes || !scale))) return QR_ERR_INVALID_ARG;
    if (rows == 0) return QR_OK;
    const cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
    auto quads = [&](auto kern) {
        kern<<<whole_grid(rows, 8), 256, 0, st>>>(reinterpret_cast<const float4 *>(in), rows, C / 4,
                                   reinterpret_cast<uint32_t *>(codes), scale);
    };
    if (C % 4 != 0 || C > 1024 || !aligned(in, 16) || !aligned(codes, 4))
        fp8_rows_kernel<<<grid_for(rows * 32, 256), 256, 0, st>>>(in, rows, C, codes, scale);
    else if (C <= 128) quads(fp8_quads_kernel<1>);
    else if (C <= 256) quads(fp8_quads_kernel<2>);
    else if (C <= 512) quads(fp8_quads_kernel<4>);
    else quads(fp8_quads_kernel<8>);
    count_launch();
    return cudaGetLastError() == cudaSuccess ? QR_OK : QR_ERR_CUDA;
}

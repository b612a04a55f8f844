// E4M3 operands for the offloaded product (the paper's Limitations / Future Work list FP8 next to FP16; Eq. 2 is the
// product that runs on the untrusted accelerator, so that is the one whose operands are narrowed):
//   per-tensor quantiser   scale = max|x| / 448 (binary32),  code = nearest-even E4M3 of x / scale (binary32 division)
//   product                Y' = (s_U s_W) (U8 W8), fp32 accumulation on the tensor cores, stored in bf16
// The quantiser is two launches after the clearing of the maximum: |x| maximum (integer atomic on the bit pattern, exact and
// order-free) and the cast, in which every thread works the scale out for itself.  Both are bound by reading x (16 bits: 2 bytes in,
// 1 out per value); a thread keeps the loads of four rows in flight.  2150 x 4096 in bf16: 27 us with one row at a time, a launch for
// the scale and one conversion instruction per value, 17 us.
#include <cuda_fp8.h>

#include "common.cuh"

namespace gelo {

namespace {

__device__ __forceinline__ float widen8(const __nv_bfloat16* e, int j) { return __bfloat162float(e[j]); }
__device__ __forceinline__ float widen8(const __half* e, int j) { return __half2float(e[j]); }

// Eight consecutive values of a row
template <typename T>
struct Eight {
    uint4 raw[sizeof(T) / 2];
    __device__ __forceinline__ void load(const T* p)
    {
#pragma unroll
        for (int i = 0; i < (int)sizeof(T) / 2; ++i) raw[i] = reinterpret_cast<const uint4*>(p)[i];
    }
    __device__ __forceinline__ void widen(float (&v)[8]) const
    {
        if constexpr (sizeof(T) == 4) {
#pragma unroll
            for (int j = 0; j < 8; ++j) v[j] = reinterpret_cast<const float*>(raw)[j];
        } else {
#pragma unroll
            for (int j = 0; j < 8; ++j) v[j] = widen8(reinterpret_cast<const T*>(raw), j);
        }
    }
};
constexpr int kQuantRows = 4;                                 // rows a thread has in flight

template <typename T>
__global__ void __launch_bounds__(256) amax_kernel(const T* __restrict__ x, int rows, int cols, int ld, unsigned* __restrict__ amax_bits)
{
    chain_next();
    chain_wait();
    float m = 0.0f;
    const int g = blockIdx.x * 256 + threadIdx.x;
    if (8 * g < cols) {                                       // cols is a multiple of 8
        for (int r = blockIdx.y; r < rows; r += kQuantRows * gridDim.y) {
            Eight<T> e[kQuantRows];
#pragma unroll
            for (int u = 0; u < kQuantRows; ++u) e[u].load(x + (size_t)min(r + u * (int)gridDim.y, rows - 1) * ld + 8 * g);   // (a row twice is harmless)
#pragma unroll
            for (int u = 0; u < kQuantRows; ++u) {
                float v[8];
                e[u].widen(v);
#pragma unroll
                for (int j = 0; j < 8; ++j) m = fmaxf(m, fabsf(v[j]));
            }
        }
    }
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, off));
    __shared__ float part[8];
    if ((threadIdx.x & 31) == 0) part[threadIdx.x >> 5] = m;
    __syncthreads();
    if (threadIdx.x == 0) {
#pragma unroll
        for (int i = 1; i < 8; ++i) m = fmaxf(m, part[i]);
        if (m > 0.0f) atomicMax(amax_bits, __float_as_uint(m));   // non-negative floats order like their bits
    }
}

template <typename T>
__global__ void __launch_bounds__(256) cast_e4m3_kernel(const T* __restrict__ x, int rows, int cols, int ld,
                                                        const unsigned* __restrict__ amax_bits, float* __restrict__ scale,
                                                        uint8_t* __restrict__ out, int ldo)
{
    chain_next();
    chain_wait();
    const float amax = __uint_as_float(*amax_bits);
    const float s = amax > 0.0f ? __fdiv_rn(amax, 448.0f) : 1.0f;
    const int g = blockIdx.x * 256 + threadIdx.x;
    if (g == 0 && blockIdx.y == 0) *scale = s;
    if (8 * g >= cols) return;
    for (int r = blockIdx.y; r < rows; r += kQuantRows * gridDim.y) {
        Eight<T> e[kQuantRows];
#pragma unroll
        for (int u = 0; u < kQuantRows; ++u) e[u].load(x + (size_t)min(r + u * (int)gridDim.y, rows - 1) * ld + 8 * g);
#pragma unroll
        for (int u = 0; u < kQuantRows; ++u) {
            const int row = r + u * (int)gridDim.y;
            float v[8];
            e[u].widen(v);
            uint32_t c[2] = {0u, 0u};
#pragma unroll
            for (int j = 0; j < 8; j += 2)
                c[j >> 2] |= (uint32_t)__nv_cvt_float2_to_fp8x2(make_float2(__fdiv_rn(v[j], s), __fdiv_rn(v[j + 1], s)), __NV_SATFINITE, __NV_E4M3)
                             << (8 * (j & 3));
            if (row < rows) *reinterpret_cast<uint2*>(out + (size_t)row * ldo + 8 * g) = make_uint2(c[0], c[1]);
        }
    }
}

template <typename T>
int quantize_typed(gelo_ctx* ctx, const void* x, int rows, int cols, int ld, uint8_t* out, int ldo, float* scale, cudaStream_t st)
{
    unsigned* amax_bits = reinterpret_cast<unsigned*>(scale + 1);
    GELO_CUDA_OK(cudaMemsetAsync(amax_bits, 0, sizeof(unsigned), st));
    const int gx = ceil_div(cols, 8 * 256);
    int gy = ceil_div(8 * ctx->sm_count, gx);                 // eight CTAs of 256 threads per SM
    if (gy > ceil_div(rows, kQuantRows)) gy = ceil_div(rows, kQuantRows);
    GELO_TRY(launch_chained(ctx, amax_kernel<T>, dim3(gx, gy), 256, 0, st, static_cast<const T*>(x), rows, cols, ld, amax_bits));
    GELO_TRY(after_launch(ctx));
    GELO_TRY(launch_chained(ctx, cast_e4m3_kernel<T>, dim3(gx, gy), 256, 0, st, static_cast<const T*>(x), rows, cols, ld, amax_bits, scale,
                           out, ldo));
    return after_launch(ctx);
}

}  // namespace

// out (rows x cols E4M3 codes, row stride ldo bytes) and scale[0] from x (rows x cols of `dtype`, row stride ld);
// scale[1] is scratch for the maximum.  cols a multiple of 8, ld a multiple of 8 (4 for fp32 pairs of loads), ldo a multiple of 8.
int launch_quantize_e4m3(gelo_ctx* ctx, const void* x, int rows, int cols, int ld, int dtype, void* out, int ldo, float* scale,
                         cudaStream_t st)
{
    if (rows <= 0 || cols <= 0) return GELO_OK;
    if ((cols % 8) || (ld % 8) || (ldo % 8) || ld < cols || ldo < cols) return GELO_ERR_INVALID;
    if (dtype == GELO_BF16) return quantize_typed<__nv_bfloat16>(ctx, x, rows, cols, ld, static_cast<uint8_t*>(out), ldo, scale, st);
    if (dtype == GELO_F16) return quantize_typed<__half>(ctx, x, rows, cols, ld, static_cast<uint8_t*>(out), ldo, scale, st);
    return quantize_typed<float>(ctx, x, rows, cols, ld, static_cast<uint8_t*>(out), ldo, scale, st);
}

}  // namespace gelo

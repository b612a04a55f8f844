// Shared-memory tiled FFMA GEMM: C = alpha * op(A) op(B) + beta * C with fp32
// accumulation.  It is the fp32-exact path of the three products of the offload
// (Eq. 1-3) and the workhorse of the trailing updates in the blocked QR and LU.
// The B operand may be the vertical stack of two matrices (Eq. 8: H_full = [H; S])
// and the output may be split into column thirds (Q | K | V).
//
// Two kernels: gemm_f32_kernel for fp32 matrices with 16-byte rows where the tiles are few, gemm_simt_kernel for everything else.
#include "common.cuh"

namespace gelo {

namespace {

constexpr int BK = 16;
constexpr int kThreads = 256;

struct GemmParams {
    int M, N, K;
    const void* A; int lda;
    const void* B; int ldb;
    const void* B2; int b_split;
    void* C0; void* C1; void* C2; int ldc; int csplit;
    float alpha, beta, diag;
    int kper; size_t plane;                                  // K slice blockIdx.z covers [z kper, z kper + kper) and writes plane z
};

__device__ __forceinline__ float ldf(const float* p) { return __ldg(p); }
__device__ __forceinline__ float ldf(const __nv_bfloat16* p) { return __bfloat162float(*p); }
__device__ __forceinline__ float ldf(const __half* p) { return __half2float(*p); }
__device__ __forceinline__ float ldc(const __half* p) { return __half2float(*p); }
__device__ __forceinline__ void stf(__half* p, float v) { *p = __float2half_rn(v); }
__device__ __forceinline__ float ldc(const float* p) { return *p; }
__device__ __forceinline__ float ldc(const __nv_bfloat16* p) { return __bfloat162float(*p); }
__device__ __forceinline__ void stf(float* p, float v) { *p = v; }
__device__ __forceinline__ void stf(__nv_bfloat16* p, float v) { *p = __float2bfloat16_rn(v); }

template <typename T, bool TA, bool TB, int BM, int BN>
__global__ void __launch_bounds__(kThreads) gemm_simt_kernel(const GemmParams prm)
{
    constexpr int RM = BM / 64, RN = BN / 64;
    constexpr int LA = BM * BK / kThreads, LB = BN * BK / kThreads;
    __shared__ __align__(16) float As[BK][BM + 4];
    __shared__ __align__(16) float Bs[BK][BN + 4];

    const T* __restrict__ A = static_cast<const T*>(prm.A);
    const T* __restrict__ B = static_cast<const T*>(prm.B);
    const T* __restrict__ B2 = static_cast<const T*>(prm.B2);
    const int tid = threadIdx.x;
    const int m0 = blockIdx.y * BM, n0 = blockIdx.x * BN;
    const int ty = tid >> 4, tx = tid & 15;

    float acc[RM * 4][RN * 4];
#pragma unroll
    for (int i = 0; i < RM * 4; ++i)
#pragma unroll
        for (int j = 0; j < RN * 4; ++j) acc[i][j] = 0.0f;

    float ra[LA], rb[LB];

    auto fetch = [&](int k0) {
#pragma unroll
        for (int i = 0; i < LA; ++i) {
            const int idx = tid + i * kThreads;
            int r, kk;
            if (TA) { r = idx % BM; kk = idx / BM; } else { kk = idx % BK; r = idx / BK; }
            const int gm = m0 + r, gk = k0 + kk;
            float v = 0.0f;
            if (gm < prm.M && gk < prm.K)
                v = TA ? ldf(A + (size_t)gk * prm.lda + gm) : ldf(A + (size_t)gm * prm.lda + gk);
            ra[i] = v;
        }
#pragma unroll
        for (int i = 0; i < LB; ++i) {
            const int idx = tid + i * kThreads;
            int c, kk;
            if (TB) { kk = idx % BK; c = idx / BK; } else { c = idx % BN; kk = idx / BN; }
            const int gn = n0 + c, gk = k0 + kk;
            float v = 0.0f;
            if (gn < prm.N && gk < prm.K) {
                if (TB) v = ldf(B + (size_t)gn * prm.ldb + gk);
                else if (gk < prm.b_split) v = ldf(B + (size_t)gk * prm.ldb + gn);
                else v = ldf(B2 + (size_t)(gk - prm.b_split) * prm.ldb + gn);
            }
            rb[i] = v;
        }
    };
    auto stash = [&]() {
#pragma unroll
        for (int i = 0; i < LA; ++i) {
            const int idx = tid + i * kThreads;
            int r, kk;
            if (TA) { r = idx % BM; kk = idx / BM; } else { kk = idx % BK; r = idx / BK; }
            As[kk][r] = ra[i];
        }
#pragma unroll
        for (int i = 0; i < LB; ++i) {
            const int idx = tid + i * kThreads;
            int c, kk;
            if (TB) { kk = idx % BK; c = idx / BK; } else { c = idx % BN; kk = idx / BN; }
            Bs[kk][c] = rb[i];
        }
    };

    const int k_lo = blockIdx.z * prm.kper, k_hi = min(prm.K, k_lo + prm.kper);
    fetch(k_lo);
    for (int k0 = k_lo; k0 < k_hi; k0 += BK) {
        stash();
        __syncthreads();
        if (k0 + BK < k_hi) fetch(k0 + BK);
#pragma unroll
        for (int kk = 0; kk < BK; ++kk) {
            float a[RM * 4], b[RN * 4];
#pragma unroll
            for (int i = 0; i < RM; ++i) {
                const float4 v = *reinterpret_cast<const float4*>(&As[kk][ty * 4 + i * 64]);
                a[4 * i] = v.x; a[4 * i + 1] = v.y; a[4 * i + 2] = v.z; a[4 * i + 3] = v.w;
            }
#pragma unroll
            for (int j = 0; j < RN; ++j) {
                const float4 v = *reinterpret_cast<const float4*>(&Bs[kk][tx * 4 + j * 64]);
                b[4 * j] = v.x; b[4 * j + 1] = v.y; b[4 * j + 2] = v.z; b[4 * j + 3] = v.w;
            }
#pragma unroll
            for (int i = 0; i < RM * 4; ++i)
#pragma unroll
                for (int j = 0; j < RN * 4; ++j) acc[i][j] = fmaf(a[i], b[j], acc[i][j]);
        }
        __syncthreads();
    }

    T* const Cs[3] = { static_cast<T*>(prm.C0), static_cast<T*>(prm.C1), static_cast<T*>(prm.C2) };
#pragma unroll
    for (int i = 0; i < RM * 4; ++i) {
        const int gm = m0 + ty * 4 + (i >> 2) * 64 + (i & 3);
        if (gm >= prm.M) continue;
#pragma unroll
        for (int j = 0; j < RN * 4; ++j) {
            const int gn = n0 + tx * 4 + (j >> 2) * 64 + (j & 3);
            if (gn >= prm.N) continue;
            const int chunk = gn / prm.csplit;
            T* p = Cs[chunk] + blockIdx.z * prm.plane + (size_t)gm * prm.ldc + (gn - chunk * prm.csplit);
            float v = prm.alpha * acc[i][j] + (gm == gn ? prm.diag : 0.0f);
            if (prm.beta != 0.0f) v += prm.beta * ldc(p);
            stf(p, v);
        }
    }
}

// ---- fp32, 64 x kN tiles, the k range of a stage shared out to four groups of threads ---------------------------
//
// A warp's 16-byte read of shared memory takes four cycles whatever it broadcasts, so what counts is values read per multiply-add:
// 8 x 8 entries per thread read a value per four multiply-adds, which balances the two pipes, 4 x 4 entries twice that.  A
// 64 x 64 tile then has only 64 threads; four such groups take 16 of the 64 k of a stage each and their sums are added at the end
// (in order), which also shortens the chain of a product with a deep K and few tiles.  32 columns per tile where 64 would leave SMs idle.
// 512 x 512 x 512: 39 us with 4 x 4 entries per thread and single-word loads, 15 us.
constexpr int kF32K = 64;                      // k of a stage
constexpr int kF32M = 64;

template <int kN>
struct F32Shared {
    float A[2][kF32K][kF32M + 4];
    float B[2][kF32K][kN + 4];
};

template <bool TA, int kN>
__global__ void __launch_bounds__(kThreads) gemm_f32_kernel(const GemmParams prm)
{
    constexpr int kC = kN / 32;                // column quads per thread
    extern __shared__ __align__(16) uint8_t f32_smem[];
    F32Shared<kN>& s = *reinterpret_cast<F32Shared<kN>*>(f32_smem);
    const float* __restrict__ A = static_cast<const float*>(prm.A);
    const float* __restrict__ B = static_cast<const float*>(prm.B);
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int group = tid >> 6, ty = (tid & 63) >> 3, tx = tid & 7;
    const int m0 = blockIdx.y * kF32M, n0 = blockIdx.x * kN;
    const int k_lo = blockIdx.z * prm.kper, k_hi = min(prm.K, k_lo + prm.kper);

    float4 ra[4], rb[2 * kC];
    const float4 zero = make_float4(0.f, 0.f, 0.f, 0.f);
    auto fetch = [&](int k0) {
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            ra[i] = zero;
            if (TA) {                          // 16 quads of columns, 16 rows of k at a time
                const int k = k0 + 16 * i + (tid >> 4), c = m0 + 4 * (tid & 15);
                if (k < k_hi && c < prm.M) ra[i] = *reinterpret_cast<const float4*>(A + (size_t)k * prm.lda + c);
            } else {                           // a row per lane, so that the transposed stores fall into different banks
                const int k = k0 + 16 * i + 4 * (warp >> 1), r = m0 + 32 * (warp & 1) + lane;
                if (k < k_hi && r < prm.M) {
                    ra[i] = *reinterpret_cast<const float4*>(A + (size_t)r * prm.lda + k);
                    if (k + 1 >= k_hi) ra[i].y = 0.0f;
                    if (k + 2 >= k_hi) ra[i].z = 0.0f;
                    if (k + 3 >= k_hi) ra[i].w = 0.0f;
                }
            }
        }
#pragma unroll
        for (int i = 0; i < 2 * kC; ++i) {
            const int idx = tid + kThreads * i, k = k0 + idx / (kN / 4), c = n0 + 4 * (idx % (kN / 4));
            rb[i] = (k < k_hi && c < prm.N) ? *reinterpret_cast<const float4*>(B + (size_t)k * prm.ldb + c) : zero;
        }
    };
    auto stash = [&](int b) {
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            if (TA) {
                *reinterpret_cast<float4*>(&s.A[b][16 * i + (tid >> 4)][4 * (tid & 15)]) = ra[i];
            } else {
                const int k = 16 * i + 4 * (warp >> 1), r = 32 * (warp & 1) + lane;
                s.A[b][k][r] = ra[i].x; s.A[b][k + 1][r] = ra[i].y; s.A[b][k + 2][r] = ra[i].z; s.A[b][k + 3][r] = ra[i].w;
            }
        }
#pragma unroll
        for (int i = 0; i < 2 * kC; ++i) {
            const int idx = tid + kThreads * i;
            *reinterpret_cast<float4*>(&s.B[b][idx / (kN / 4)][4 * (idx % (kN / 4))]) = rb[i];
        }
    };

    float acc[8][4 * kC];
#pragma unroll
    for (int i = 0; i < 8; ++i)
#pragma unroll
        for (int j = 0; j < 4 * kC; ++j) acc[i][j] = 0.0f;

    fetch(k_lo);
    stash(0);
    __syncthreads();
    int b = 0;
    for (int k0 = k_lo; k0 < k_hi; k0 += kF32K, b ^= 1) {
        const bool more = k0 + kF32K < k_hi;
        if (more) fetch(k0 + kF32K);
#pragma unroll
        for (int kk = 0; kk < 16; ++kk) {
            const int k = 16 * group + kk;
            float x[8], y[4 * kC];
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const float4 v = *reinterpret_cast<const float4*>(&s.A[b][k][32 * h + 4 * ty]);
                x[4 * h] = v.x; x[4 * h + 1] = v.y; x[4 * h + 2] = v.z; x[4 * h + 3] = v.w;
            }
#pragma unroll
            for (int h = 0; h < kC; ++h) {
                const float4 v = *reinterpret_cast<const float4*>(&s.B[b][k][32 * h + 4 * tx]);
                y[4 * h] = v.x; y[4 * h + 1] = v.y; y[4 * h + 2] = v.z; y[4 * h + 3] = v.w;
            }
#pragma unroll
            for (int i = 0; i < 8; ++i)
#pragma unroll
                for (int j = 0; j < 4 * kC; ++j) acc[i][j] = fmaf(x[i], y[j], acc[i][j]);
        }
        if (more) stash(b ^ 1);
        __syncthreads();
    }

    // ---- the four groups' sums, tile by tile in shared memory; then 256 threads add and store quads of columns ----
    float* const sum = &s.A[0][0][0];          // 4 tiles of 64 x kN (the operands have been read)
    static_assert(sizeof(F32Shared<kN>) >= 4 * kF32M * kN * sizeof(float), "the sums fit where the operands were");
#pragma unroll
    for (int i = 0; i < 8; ++i)
#pragma unroll
        for (int h = 0; h < kC; ++h)
            *reinterpret_cast<float4*>(sum + (group * kF32M + 32 * (i >> 2) + 4 * ty + (i & 3)) * kN + 32 * h + 4 * tx) =
                make_float4(acc[i][4 * h], acc[i][4 * h + 1], acc[i][4 * h + 2], acc[i][4 * h + 3]);
    __syncthreads();
    float* const Cs[3] = { static_cast<float*>(prm.C0), static_cast<float*>(prm.C1), static_cast<float*>(prm.C2) };
    for (int idx = tid; idx < kF32M * kN / 4; idx += kThreads) {
        const int r = idx / (kN / 4), c = 4 * (idx % (kN / 4)), gm = m0 + r, gn = n0 + c;
        if (gm >= prm.M || gn >= prm.N) continue;
        float v[4] = {0.0f, 0.0f, 0.0f, 0.0f};
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const float4 t = *reinterpret_cast<const float4*>(sum + (q * kF32M + r) * kN + c);
            v[0] += t.x; v[1] += t.y; v[2] += t.z; v[3] += t.w;
        }
        const int part = gn / prm.csplit;      // (a multiple of four)
        float* p = Cs[part] + blockIdx.z * prm.plane + (size_t)gm * prm.ldc + (gn - part * prm.csplit);
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            v[j] = prm.alpha * v[j] + (gm == gn + j ? prm.diag : 0.0f);
            if (prm.beta != 0.0f && gn + j < prm.N) v[j] += prm.beta * p[j];
        }
        if (gn + 3 < prm.N) {
            *reinterpret_cast<float4*>(p) = make_float4(v[0], v[1], v[2], v[3]);
        } else {
#pragma unroll
            for (int j = 0; j < 4; ++j)
                if (gn + j < prm.N) p[j] = v[j];
        }
    }
}

template <bool TA, int kN>
int launch_f32(gelo_ctx* ctx, const GemmParams& p, int slices, cudaStream_t st)
{
    static bool attr_done[64] = {};
    if (ctx->device >= 0 && ctx->device < 64 && !attr_done[ctx->device]) {
        GELO_CUDA_OK(cudaFuncSetAttribute(gemm_f32_kernel<TA, kN>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(F32Shared<kN>)));
        attr_done[ctx->device] = true;
    }
    // (not chained: 512 rows in fp32, non-orthogonal sample 700 us like this, 753 us chained)
    gemm_f32_kernel<TA, kN><<<dim3(ceil_div(p.N, kN), ceil_div(p.M, kF32M), slices), kThreads, sizeof(F32Shared<kN>), st>>>(p);
    return after_launch(ctx);
}

bool aligned_rows(const void* p, int ld) { return (reinterpret_cast<uintptr_t>(p) & 15u) == 0 && (ld % 4) == 0; }

template <typename T, bool TA, bool TB>
void launch_tiles(const GemmParams& p, bool small, int slices, cudaStream_t st)
{
    if (small) {
        dim3 grid(ceil_div(p.N, 64), ceil_div(p.M, 64), slices);
        gemm_simt_kernel<T, TA, TB, 64, 64><<<grid, kThreads, 0, st>>>(p);
    } else {
        dim3 grid(ceil_div(p.N, 128), ceil_div(p.M, 128), slices);
        gemm_simt_kernel<T, TA, TB, 128, 128><<<grid, kThreads, 0, st>>>(p);
    }
}

}  // namespace

int launch_gemm_simt(gelo_ctx* ctx, const GemmArgs& g, cudaStream_t st)
{
    if (g.M <= 0 || g.N <= 0) return GELO_OK;
    if (g.K < 0 || !g.A || !g.B || !g.C[0] || g.nsplit < 1 || g.nsplit > 3 || g.N % g.nsplit != 0)
        return GELO_ERR_INVALID;
    if (g.B2 && g.transB) return GELO_ERR_INVALID;
    if (g.ksplit < 1 || (g.ksplit > 1 && (g.beta != 0.0f || g.nsplit != 1))) return GELO_ERR_INVALID;
    for (int i = 0; i < g.nsplit; ++i)
        if (!g.C[i]) return GELO_ERR_INVALID;
    GemmParams p;
    p.M = g.M; p.N = g.N; p.K = g.K;
    p.A = g.A; p.lda = g.lda; p.B = g.B; p.ldb = g.ldb;
    p.B2 = g.B2 ? g.B2 : g.B; p.b_split = g.B2 ? g.b_split : g.K;
    p.C0 = g.C[0]; p.C1 = g.C[g.nsplit > 1 ? 1 : 0]; p.C2 = g.C[g.nsplit > 2 ? 2 : 0];
    p.ldc = g.ldc; p.csplit = g.N / g.nsplit;
    p.alpha = g.alpha; p.beta = g.beta; p.diag = g.diag;
    p.kper = ceil_div(ceil_div(g.K, g.ksplit), BK) * BK;      // (the caller's slices: whole steps, none of them empty)
    p.plane = g.plane;
    const int slices = g.ksplit;
    // gemm_f32_kernel is made for products that leave SMs idle: up to one of its 64 x 64 tiles per SM it takes 0.3 to 0.9 of the time of
    // the tiles below (4096 x 4096 by 64 rows 268 -> 109 us, 127 rows 269 -> 187 us).  Beyond, a plain product runs faster on those, which
    // hold four CTAs per SM instead of one: 4096 x 12288 by 127 rows 496 us there, 586 us here; 1000 x 1000 by 4096 columns
    // 281 and 320 us.  In a second round of tiles it depends: this kernel loses what its last stage of 64 k leaves empty (200 x 200 by 4096 columns
    // 24.8 us there, 26.9 here) and cannot hide the latency of a B that comes from DRAM (64 rows, 4096 x 12288: 371 and 384 us; 512 x 12288
    // 51.5 and 49.4), except that it does not load rows past M (17 rows, 4096 x 16384: 365 and 340 us; a third round, by 24576
    // columns, 490 and 516 us).  The sampler's products (transposed, in slices, or adding to C) stay here: 3000 rows orthogonal 9.7 ms
    // like this, 9.5 ms on the tiles below, but 1075 rows 1.14 and 1.18 ms.
    const long tiles64 = (long)ceil_div(g.N, 64) * ceil_div(g.M, kF32M) * slices;
    const bool plain = !g.transA && g.beta == 0.0f && g.diag == 0.0f && slices == 1;
    const bool two_rounds = ceil_div(g.K, kF32K) * kF32K - g.K <= g.K / 16 && (g.M <= 32 || (size_t)g.K * g.N * sizeof(float) <= (72u << 20));
    const bool few_tiles = !plain || tiles64 <= (two_rounds ? 2L : 1L) * ctx->sm_count;
    if (few_tiles && g.dtype == GELO_F32 && !g.transB && !g.B2 && aligned_rows(g.A, g.lda) && aligned_rows(g.B, g.ldb) && aligned_rows(g.C[0], g.ldc) &&
        (g.nsplit == 1 || (p.csplit % 4 == 0 && aligned_rows(p.C1, g.ldc) && aligned_rows(p.C2, g.ldc))) && g.plane % 4 == 0) {
        // rows of A and B are read in whole quads: the last one of a row may reach past its end, but not past its stride
        const bool wide = tiles64 >= ctx->sm_count;
        if (g.transA) return wide ? launch_f32<true, 64>(ctx, p, slices, st) : launch_f32<true, 32>(ctx, p, slices, st);
        return wide ? launch_f32<false, 64>(ctx, p, slices, st) : launch_f32<false, 32>(ctx, p, slices, st);
    }
    const long tiles128 = (long)ceil_div(g.M, 128) * ceil_div(g.N, 128) * slices;
    const bool small = g.M <= 64 || g.N <= 64 || tiles128 < 2L * ctx->sm_count;
    if (g.dtype == GELO_BF16) {
        if (g.transA || g.transB) return GELO_ERR_UNSUPPORTED;
        launch_tiles<__nv_bfloat16, false, false>(p, small, slices, st);
    } else if (g.dtype == GELO_F16) {
        if (g.transA || g.transB) return GELO_ERR_UNSUPPORTED;
        launch_tiles<__half, false, false>(p, small, slices, st);
    } else {
        if (!g.transA && !g.transB) launch_tiles<float, false, false>(p, small, slices, st);
        else if (g.transA && !g.transB) launch_tiles<float, true, false>(p, small, slices, st);
        else if (!g.transA && g.transB) launch_tiles<float, false, true>(p, small, slices, st);
        else launch_tiles<float, true, true>(p, small, slices, st);
    }
    return after_launch(ctx);
}

}  // namespace gelo

// 2-norm condition number estimate of the non-orthogonal mixing matrix (paper, Mitigation 1: a
// non-orthogonal A is to be checked for good conditioning after it is drawn, a bound of 100 being the example).
// kappa_2(A) = sigma_max(A) * sigma_max(A^-1); each factor is the square root of the largest Ritz value of
// Op^T Op after a few Lanczos steps from a Gaussian start vector, with Op = A (z = 0) and Op = A^-1 (z = 1), both
// run in the same launches.  (Six Lanczos steps are as close as twelve steps of the power iteration: the Ritz value
// is the best estimate the Krylov space holds, the power iterate only its last vector.  A Ritz value never exceeds
// lambda_max, so the estimate is a lower one.)
// The operators are the matrices as stored (bf16 or fp32), i.e. exactly what the mixing and unmixing products
// read.  All sums have a fixed order, so the estimate is bit-reproducible.
//
// Where the rows of a matrix fit the shared memory of eight CTAs (16 bits: up to 920 rows, fp32: 656) all steps are one launch, cond_small_kernel.
// Beyond, a step is two: cond_step_kernel, bound by reading both operators (74 MB at 4300 rows in bf16, which stay in
// L2 from step to step), and cond_reduce_kernel, whose last CTA also does the Lanczos recurrence.  What counts is
// loads in flight: slabs of 16 rows (538 CTAs at 4300 rows) with two rows per warp and whole-vector loads of x, the
// slab sums spread over sixteen threads per column, the eigenvalues searched by 32 lanes at a time.  Against 32-row
// slabs with scalar loads of x, a thread per column in the sums, a launch of its own for the recurrence and bisection by
// a single thread: 630 -> 250 us per estimate at 4300 rows (the pass over both operators 63 -> 23 us).
#include <cfloat>

#include "common.cuh"
#include "philox.cuh"
#include "tc_ptx.cuh"

namespace gelo {

namespace {

constexpr int kCondRows = 16;        // rows of a slab (one CTA each), as long as that makes no more than ...
constexpr int kCondSlabsMax = 512;   // ... this many slabs
constexpr int kCondChunkCols = 64;   // entries per CTA of the reduction over slabs
constexpr int kCondParts = 16;       // threads that share an entry's sum
constexpr int kLanczosSteps = 6;     // the estimate is within about 6% of kappa_2 (measured at m = 64 .. 4300, gamma 0.5 .. 3)

struct CondViews {
    const void* op[2];
    int ld, m, mpad, slabs, rows_per;
    float* v;         // [2][mpad]  current Lanczos vector (unit length)
    float* vprev;     // [2][mpad]  the one before
    float* w;         // [2][mpad]  Op^T Op v
    float* partial;   // [2][slabs][mpad]
    float* tri;       // [2][2][kLanczosSteps]  diagonal and off-diagonal of the Lanczos tridiagonal matrices
    unsigned* done;   // [2]  CTAs of the current reduction that have finished (zero between launches)
};

// The start vector, as the only slab of a first reduction.
__global__ void cond_init_kernel(CondViews v, uint64_t seed, uint32_t attempt)
{
    chain_next();
    chain_wait();
    const int z = blockIdx.y;
    const int i4 = (blockIdx.x * blockDim.x + threadIdx.x) * 4;
    if (i4 == 0) v.done[z] = 0;
    if (i4 >= v.mpad) return;
    float g[4];
    gaussian_block(seed, ((uint64_t)z * v.mpad + i4) >> 2, GELO_STREAM_POWER, attempt, g);
    for (int t = 0; t < 4; ++t) {
        const int i = i4 + t;
        if (i < v.mpad) v.partial[(size_t)z * v.slabs * v.mpad + i] = i < v.m ? g[t] : 0.0f;
    }
}

// Sum over the CTA's threads in a fixed order; every thread receives it.
__device__ __forceinline__ float cond_block_sum(float local, float* red)
{
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) local += __shfl_xor_sync(0xffffffffu, local, off);
    __syncthreads();                                         // red may still be read from the previous sum
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = local;
    __syncthreads();
    float t = red[threadIdx.x & 31];
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) t += __shfl_xor_sync(0xffffffffu, t, off);
    return t;
}

// step < 0: v = w / |w| (the start vector), vprev = 0.  Otherwise the Lanczos recurrence
//   alpha = v . w,  r = w - alpha v - beta_prev vprev,  beta = |r|,  vprev <- v,  v <- r / beta.
// Run by all 1024 threads of one CTA.
__device__ __forceinline__ void cond_lanczos(const CondViews& v, int z, int step, float* red)
{
    float* vc = v.v + (size_t)z * v.mpad;
    float* vp = v.vprev + (size_t)z * v.mpad;
    float* w = v.w + (size_t)z * v.mpad;
    float* alpha = v.tri + (size_t)z * 2 * kLanczosSteps;
    float* beta = alpha + kLanczosSteps;
    if (step < 0) {
        float local = 0.0f;
        for (int i = threadIdx.x; i < v.m; i += 1024) local = fmaf(w[i], w[i], local);
        const float nrm = sqrtf(cond_block_sum(local, red));
        const float inv = nrm > 0.0f ? 1.0f / nrm : 0.0f;
        for (int i = threadIdx.x; i < v.mpad; i += 1024) { vc[i] = i < v.m ? w[i] * inv : 0.0f; vp[i] = 0.0f; }
        return;
    }
    float local = 0.0f;
    for (int i = threadIdx.x; i < v.m; i += 1024) local = fmaf(vc[i], w[i], local);
    const float a = cond_block_sum(local, red);
    const float bprev = step > 0 ? beta[step - 1] : 0.0f;
    local = 0.0f;
    for (int i = threadIdx.x; i < v.m; i += 1024) {
        const float r = w[i] - a * vc[i] - bprev * vp[i];
        w[i] = r;
        local = fmaf(r, r, local);
    }
    const float b = sqrtf(cond_block_sum(local, red));
    const float inv = b > 0.0f ? 1.0f / b : 0.0f;
    for (int i = threadIdx.x; i < v.m; i += 1024) {          // (each thread touches only the entries it wrote)
        vp[i] = vc[i];
        vc[i] = w[i] * inv;
    }
    if (threadIdx.x == 0) { alpha[step] = a; beta[step] = b; }
}

// w = sum of `slabs` slab partials: kCondParts threads per entry take every kCondParts-th slab each, then their sums are
// added in order.  The CTA that finishes last for an operator goes on with the recurrence.
__global__ void __launch_bounds__(kCondChunkCols * kCondParts) cond_reduce_kernel(CondViews v, int slabs, int step)
{
    chain_next();
    chain_wait();
    static_assert(kCondChunkCols * kCondParts == 1024, "cond_lanczos counts on 1024 threads");
    __shared__ float part[kCondParts][kCondChunkCols];
    __shared__ float red[32];
    __shared__ int last;
    const int z = blockIdx.y;
    const int c = threadIdx.x % kCondChunkCols, q = threadIdx.x / kCondChunkCols;
    const int i = blockIdx.x * kCondChunkCols + c;           // < mpad, a multiple of kCondChunkCols
    const float* p = v.partial + (size_t)z * v.slabs * v.mpad + i;
    float s = 0.0f;
#pragma unroll 8
    for (int k = q; k < slabs; k += kCondParts) s += p[(size_t)k * v.mpad];
    part[q][c] = s;
    __syncthreads();
    if (q == 0 && i < v.m) {
#pragma unroll
        for (int t = 1; t < kCondParts; ++t) s += part[t][c];
        v.w[(size_t)z * v.mpad + i] = s;
    }
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) {
        last = atomicAdd(v.done + z, 1u) + 1 == gridDim.x;
        if (last) v.done[z] = 0;
    }
    __syncthreads();
    if (!last) return;
    __threadfence();
    cond_lanczos(v, z, step, red);
}

// Largest eigenvalue of the symmetric tridiagonal matrix (alpha[0..k-1]; beta[0..k-2]), found by one warp that cuts the
// interval from 0 to the Gershgorin bound into 33 at a time by the number of
// eigenvalues below each point (Sturm sequence).  A breakdown (beta = 0) only decouples the matrix: the count stays valid.
struct TopEigenvalue {
    static constexpr int k = kLanczosSteps;
    double a[k], b2[k], lo, hi;                              // it lies between lo and hi
    bool bounded;

    __device__ __forceinline__ TopEigenvalue(const float* alpha, const float* beta) : lo(0.0), hi(0.0), bounded(true)
    {
#pragma unroll
        for (int i = 0; i < k; ++i) {
            a[i] = alpha[i];
            const double bl = i > 0 ? fabs((double)beta[i - 1]) : 0.0, br = i + 1 < k ? fabs((double)beta[i]) : 0.0;
            b2[i] = bl * bl;
            const double reach = fabs(a[i]) + bl + br;
            // (matrices with NaN or infinite entries have no bound: fmax would drop a NaN)
            if (bounded && !(reach <= DBL_MAX)) { bounded = false; lo = hi = reach; }
            if (bounded) hi = fmax(hi, reach);
        }
    }
    __device__ __forceinline__ void narrow(int rounds)
    {
        if (!bounded) return;
        const int lane = threadIdx.x & 31;
#pragma unroll 1
        for (int round = 0; round < rounds; ++round) {
            const double step = (hi - lo) * (1.0 / 33.0), x = lo + (lane + 1) * step;
            bool all_below = true;                           // all k eigenvalues lie below x
            double q = 1.0;
#pragma unroll
            for (int i = 0; i < k; ++i) {
                q = a[i] - x - (i > 0 ? b2[i] / q : 0.0);
                if (q == 0.0) q = -1e-300;
                all_below = all_below && q < 0.0;
            }
            const uint32_t mask = __ballot_sync(0xffffffffu, all_below);
            const int first = mask ? __ffs(mask) - 1 : 32;   // the first point with everything below it
            const double h = first < 32 ? lo + (first + 1) * step : hi;
            lo = lo + first * step;
            hi = h;
        }
    }
};

// One warp per operator.  Twelve rounds leave 2^-60 of the bound.  After seven (2^-35) both ends of the intervals nearly always give
// the same float, which then is that of twelve; only where they do not are the other five done.
__global__ void __launch_bounds__(64) cond_verdict_kernel(CondViews v, float bound, float* cond_out, int* status, int deferred)
{
    chain_next();
    chain_wait();
    __shared__ double lo[2], hi[2];
    const int z = threadIdx.x >> 5;
    TopEigenvalue top(v.tri + z * 2 * kLanczosSteps, v.tri + z * 2 * kLanczosSteps + kLanczosSteps);
    auto publish = [&]() {
        if ((threadIdx.x & 31) == 0) { lo[z] = top.lo; hi[z] = top.hi; }
        __syncthreads();
    };
    top.narrow(7);
    publish();
    const bool settled = (float)(sqrt(lo[0]) * sqrt(lo[1])) == (float)(sqrt(hi[0]) * sqrt(hi[1]));
    __syncthreads();
    if (!settled) {
        top.narrow(5);
        publish();
    }
    if (threadIdx.x != 0) return;
    // lambda_max(Op^T Op) = sigma_max^2
    const float c = (float)(sqrt(0.5 * (lo[0] + hi[0])) * sqrt(0.5 * (lo[1] + hi[1])));
    if (cond_out) cond_out[0] = c;
    const int ok = (c * 1.2f <= bound && c == c) ? 1 : 0;   // the estimate is a lower one (tests: >= 0.85 of the true value)
    status[1] = ok;
    // nobody reads the verdict between attempts in deferred mode: a miss becomes a sticky error
    if (deferred && !ok) atomicCAS(status, 0, (int)GELO_ERR_COND);
}

// Eight consecutive elements of a stored row, widened to fp32 (rows start 16-byte aligned, ld is a multiple of 8).
__device__ __forceinline__ void load8(const float* p, float (&a)[8])
{
    const float4 lo = *reinterpret_cast<const float4*>(p), hi = *reinterpret_cast<const float4*>(p + 4);
    a[0] = lo.x; a[1] = lo.y; a[2] = lo.z; a[3] = lo.w; a[4] = hi.x; a[5] = hi.y; a[6] = hi.z; a[7] = hi.w;
}
__device__ __forceinline__ void load8(const __nv_bfloat16* p, float (&a)[8])
{
    const uint4 raw = *reinterpret_cast<const uint4*>(p);
    const uint32_t w[4] = {raw.x, raw.y, raw.z, raw.w};
#pragma unroll
    for (int t = 0; t < 4; ++t) {
        a[2 * t] = __uint_as_float(w[t] << 16);
        a[2 * t + 1] = __uint_as_float(w[t] & 0xffff0000u);
    }
}

__device__ __forceinline__ void load8(const __half* p, float (&a)[8])
{
    const uint4 raw = *reinterpret_cast<const uint4*>(p);
    const __half2* h = reinterpret_cast<const __half2*>(&raw);
#pragma unroll
    for (int t = 0; t < 4; ++t) {
        const float2 f = __half22float2(h[t]);
        a[2 * t] = f.x; a[2 * t + 1] = f.y;
    }
}

// One application Op^T (Op v) in a single pass over the operator: CTA (slab, z) first forms y_r =
// Op[r, :] . v for its rows (two rows per warp at a time, so that a vector load of v serves both), then accumulates
// sum_r y_r Op[r, :] for every column; the second read of the slab comes from L1 or L2.  partial[z][slab][:] receives the
// slab's contribution.
template <typename T>
__global__ void __launch_bounds__(256) cond_step_kernel(CondViews v)
{
    chain_next();
    chain_wait();
    extern __shared__ float ys[];
    const int z = blockIdx.y, slab = blockIdx.x;
    const int r0 = slab * v.rows_per;
    const int r1 = min(v.m, r0 + v.rows_per);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const T* op = static_cast<const T*>(v.op[z]);
    const float* x = v.v + (size_t)z * v.mpad;
    const int full = v.m >> 3, groups = (v.m + 7) >> 3;
    for (int r = r0 + 2 * warp; r < r1; r += 16) {
        const T* a0 = op + (size_t)r * v.ld;
        const T* a1 = (r + 1 < r1) ? a0 + v.ld : a0;         // (an odd last row is read twice and counted once)
        float s0 = 0.0f, s1 = 0.0f;
#pragma unroll 4
        for (int g = lane; g < full; g += 32) {
            float e0[8], e1[8], xv[8];
            load8(a0 + 8 * g, e0);
            load8(a1 + 8 * g, e1);
            load8(x + 8 * g, xv);
#pragma unroll
            for (int t = 0; t < 8; ++t) { s0 = fmaf(e0[t], xv[t], s0); s1 = fmaf(e1[t], xv[t], s1); }
        }
        if (full < groups && lane == (full & 31)) {          // the columns past a multiple of 8
            float e0[8], e1[8];
            load8(a0 + 8 * full, e0);
            load8(a1 + 8 * full, e1);
#pragma unroll
            for (int t = 0; t < 8; ++t)
                if (8 * full + t < v.m) { s0 = fmaf(e0[t], x[8 * full + t], s0); s1 = fmaf(e1[t], x[8 * full + t], s1); }
        }
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) {
            s0 += __shfl_xor_sync(0xffffffffu, s0, off);
            s1 += __shfl_xor_sync(0xffffffffu, s1, off);
        }
        if (lane == 0) {
            ys[r - r0] = s0;
            if (r + 1 < r1) ys[r + 1 - r0] = s1;
        }
    }
    __syncthreads();
    float* out = v.partial + ((size_t)z * v.slabs + slab) * v.mpad;
    for (int g = threadIdx.x; g < groups; g += 256) {
        float acc[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
        const T* a = op + (size_t)r0 * v.ld + 8 * g;
        int r = 0;
        for (; r + 8 <= r1 - r0; r += 8) {                   // rows ascend: the sum keeps its fixed order
            float e[8][8];
#pragma unroll
            for (int u = 0; u < 8; ++u) load8(a + (size_t)(r + u) * v.ld, e[u]);
#pragma unroll
            for (int u = 0; u < 8; ++u) {
                const float y = ys[r + u];
#pragma unroll
                for (int t = 0; t < 8; ++t) acc[t] = fmaf(e[u][t], y, acc[t]);
            }
        }
        for (; r < r1 - r0; ++r) {
            float e[8];
            load8(a + (size_t)r * v.ld, e);
            const float y = ys[r];
#pragma unroll
            for (int t = 0; t < 8; ++t) acc[t] = fmaf(e[t], y, acc[t]);
        }
#pragma unroll
        for (int t = 0; t < 8; ++t)
            if (8 * g + t >= v.m) acc[t] = 0.0f;             // (what stands past the last column is no data)
        float4* o = reinterpret_cast<float4*>(out + 8 * g);
        o[0] = make_float4(acc[0], acc[1], acc[2], acc[3]);
        o[1] = make_float4(acc[4], acc[5], acc[6], acc[7]);
    }
}

// All steps in one launch for a matrix whose rows fit the shared memory of eight CTAs (16 bits: up to 920 rows, fp32: 656).  A cluster per
// operator; each CTA keeps its rows on chip, forms its part of Op^T (Op v), and after one barrier of the cluster every CTA adds the eight
// parts up in the same order and does the recurrence for itself, so the vector never travels.  Bound by latency, 2 us a step; as
// launches of their own the steps take 8 us each.  With the verdict,
// fp32: 64 rows 56 -> 19 us, 350 rows 63 -> 33, 512 rows 64 -> 44, 650 rows 75 -> 62.  Batches gain too, though the two clusters need sixteen
// SMs of their own: calls with d = 1024 and a non-orthogonal A, the general route -> this, us: bf16, 8 x 315 rows on 8 lanes 589 -> 539, 32 x 350 on
// 32 lanes 1156 -> 1090, 32 x 900 on 32 lanes 3570 -> 3348; fp32, 8 x 64 on 8 lanes 414 -> 409, 32 x 300 on 32 lanes 3760 -> 3744, 32 x 512 5594 -> 5559;
// only 32 x 130 in fp32 on 16 or 32 lanes lose, 2590 -> 2610 (waited for 2795 -> 2771).
constexpr int kSmallCtas = 8, kSmallThreads = 1024;
struct CondSmallPlan { int rows, lds; size_t slab, bytes; };
CondSmallPlan cond_small_plan(int m, int es)
{
    CondSmallPlan p;
    p.rows = ceil_div(m, kSmallCtas);
    p.lds = (m + 7) & ~7;
    p.slab = (3 * (size_t)p.lds + 2 * kSmallThreads + ((p.rows + 3) & ~3) + 32) * sizeof(float);     // what stands before the rows
    p.slab = (p.slab + 15) & ~size_t(15);
    p.bytes = p.slab + (size_t)p.rows * p.lds * es;
    return p;
}
bool cond_small_supports(int m, int es) { return m <= kSmallThreads && cond_small_plan(m, es).bytes <= 227 * 1024; }

template <typename T>
__global__ void __cluster_dims__(kSmallCtas, 1, 1) __launch_bounds__(kSmallThreads, 1)
cond_small_kernel(CondViews v, uint64_t seed, uint32_t attempt, int rows_per, int lds, int slab_offset)
{
    chain_next();
    chain_wait();
    extern __shared__ __align__(16) uint8_t cs_smem[];
    float* vs = reinterpret_cast<float*>(cs_smem);           // the Lanczos vector
    float* part = vs + lds;                                  // [2][lds] this CTA's part of w, in turn
    float* sums = part + 2 * lds;                            // [2 kSmallThreads]
    float* ys = sums + 2 * kSmallThreads;
    float* red = ys + ((rows_per + 3) & ~3);
    T* slab = reinterpret_cast<T*>(cs_smem + slab_offset);
    const int z = blockIdx.y, rank = blockIdx.x, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, m = v.m;
    const int r0 = rank * rows_per, rows = max(0, min(rows_per, m - r0)), groups = lds >> 3;
    const T* op = static_cast<const T*>(v.op[z]);
    constexpr int kVec = 16 / (int)sizeof(T);
    for (int e = tid; e < rows * (lds / kVec); e += kSmallThreads) {             // (rows of the operator are whole groups of eight)
        const int r = e / (lds / kVec), c = (e - r * (lds / kVec)) * kVec;
        __align__(16) T t[kVec];
        *reinterpret_cast<uint4*>(t) = *reinterpret_cast<const uint4*>(op + (size_t)(r0 + r) * v.ld + c);
#pragma unroll
        for (int j = 0; j < kVec; ++j)
            if (c + j >= m) t[j] = T(0.0f);                   // (what stands past the last column is no data)
        *reinterpret_cast<uint4*>(slab + (size_t)r * lds + c) = *reinterpret_cast<const uint4*>(t);
    }
    float vi = 0.0f, vp = 0.0f, bprev = 0.0f;                // entry tid of the vector and of the one before; every CTA has them all
    if (4 * tid < lds) {
        float g[4];
        gaussian_block(seed, ((uint64_t)z * v.mpad + 4 * tid) >> 2, GELO_STREAM_POWER, attempt, g);
#pragma unroll
        for (int j = 0; j < 4; ++j) vs[4 * tid + j] = 4 * tid + j < m ? g[j] : 0.0f;
    }
    __syncthreads();
    if (tid < m) vi = vs[tid];
    {
        const float nrm = sqrtf(cond_block_sum(vi * vi, red)), inv = nrm > 0.0f ? 1.0f / nrm : 0.0f;
        vi *= inv;
        if (tid < m) vs[tid] = vi;
    }
    const int pairs = lds >> 1, parts = min(8, kSmallThreads / pairs), my_q = tid / pairs, my_c = 2 * (tid - my_q * pairs);
    for (int step = 0; step < kLanczosSteps; ++step) {
        __syncthreads();                                     // vs
        for (int r = warp; r < rows; r += kSmallThreads / 32) {
            float s = 0.0f;
#pragma unroll 4
            for (int g = lane; g < groups; g += 32) {
                float e[8], x[8];
                load8(slab + (size_t)r * lds + 8 * g, e);
                load8(vs + 8 * g, x);
#pragma unroll
                for (int j = 0; j < 8; ++j) s = fmaf(e[j], x[j], s);
            }
#pragma unroll
            for (int off = 16; off > 0; off >>= 1) s += __shfl_xor_sync(0xffffffffu, s, off);
            if (lane == 0) ys[r] = s;
        }
        __syncthreads();
        if (my_q < parts) {                                  // rows q, q + parts, ... of two columns
            const int q = my_q, c = my_c;
            float a = 0.0f, b = 0.0f;
#pragma unroll 8
            for (int r = q; r < rows; r += parts) {
                const T* t = slab + (size_t)r * lds + c;
                a = fmaf((float)t[0], ys[r], a);
                b = fmaf((float)t[1], ys[r], b);
            }
            sums[q * lds + c] = a;
            sums[q * lds + c + 1] = b;
        }
        __syncthreads();
        float* mine = part + (step & 1) * lds;
        if (tid < lds) {
            float s = sums[tid];
            for (int q = 1; q < parts; ++q) s += sums[q * lds + tid];
            mine[tid] = s;
        }
        // (a part is written again two steps later, after the barrier at which everybody has read it)
        asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
        asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
        float w = 0.0f;
        if (tid < m) {
            float t[kSmallCtas];
#pragma unroll
            for (int k = 0; k < kSmallCtas; ++k)             // all on their way before the first is added
                asm volatile("ld.shared::cluster.f32 %0, [%1];" : "=f"(t[k]) : "r"(tcx::map_rank(tcx::smem_u32(mine + tid), k)));
#pragma unroll
            for (int k = 0; k < kSmallCtas; ++k) w += t[k];
        }
        const float a = cond_block_sum(vi * w, red);
        w = w - a * vi - bprev * vp;
        const float b = sqrtf(cond_block_sum(w * w, red)), inv = b > 0.0f ? 1.0f / b : 0.0f;
        vp = vi;
        vi = w * inv;
        bprev = b;
        if (tid < m) vs[tid] = vi;
        if (rank == 0 && tid == 0) {
            v.tri[z * 2 * kLanczosSteps + step] = a;
            v.tri[z * 2 * kLanczosSteps + kLanczosSteps + step] = b;
        }
    }
    asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");        // nobody's shared memory goes while others read it
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}

template <typename T>
int launch_cond_small(gelo_ctx* ctx, const CondViews& v, cudaStream_t st)
{
    static bool done[64] = {};
    if (ctx->device >= 0 && ctx->device < 64 && !done[ctx->device]) {
        GELO_CUDA_OK(cudaFuncSetAttribute(cond_small_kernel<T>, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024));
        done[ctx->device] = true;
    }
    const CondSmallPlan p = cond_small_plan(v.m, (int)sizeof(T));
    GELO_TRY(launch_chained(ctx, cond_small_kernel<T>, dim3(kSmallCtas, 2), kSmallThreads, p.bytes, st, v, 0x5eedull, 0u, p.rows, p.lds, (int)p.slab));
    return after_launch(ctx);
}

int cond_slabs(int m) { return ceil_div(m, kCondRows) < kCondSlabsMax ? ceil_div(m, kCondRows) : kCondSlabsMax; }

}  // namespace

CondScratch carve_cond(Arena& a, int m)
{
    CondScratch s;
    const size_t mpad = (size_t)((m + 63) / 64) * 64;
    s.vec = static_cast<float*>(a.take((6 + 2 * (size_t)cond_slabs(m)) * mpad * sizeof(float)));
    s.scal = static_cast<float*>(a.take((16 + 4 * kLanczosSteps) * sizeof(float)));
    return s;
}

int run_cond_estimate(gelo_ctx* ctx, int m, const void* A, const void* Ainv, int ld, int dtype, float bound,
                      float* cond_out, const CondScratch& s, cudaStream_t st, bool deferred)
{
    if ((ld % 8) || (reinterpret_cast<uintptr_t>(A) & 15u) || (reinterpret_cast<uintptr_t>(Ainv) & 15u)) return GELO_ERR_INVALID;
    CondViews v;
    v.op[0] = A; v.op[1] = Ainv; v.ld = ld; v.m = m; v.mpad = ((m + 63) / 64) * 64;
    v.slabs = cond_slabs(m);
    v.rows_per = ceil_div(m, v.slabs);
    v.v = s.vec;
    v.vprev = s.vec + 2 * (size_t)v.mpad;
    v.w = s.vec + 4 * (size_t)v.mpad;
    v.partial = s.vec + 6 * (size_t)v.mpad;
    v.tri = s.scal + 16;
    v.done = reinterpret_cast<unsigned*>(s.scal);
    const size_t ys_bytes = (size_t)v.rows_per * sizeof(float);
    if (ys_bytes > 48 * 1024) return GELO_ERR_UNSUPPORTED;
    if (cond_small_supports(m, (int)elem_size(dtype))) {
        if (dtype == GELO_BF16) GELO_TRY(launch_cond_small<__nv_bfloat16>(ctx, v, st));
        else if (dtype == GELO_F16) GELO_TRY(launch_cond_small<__half>(ctx, v, st));
        else GELO_TRY(launch_cond_small<float>(ctx, v, st));
        GELO_TRY(launch_chained(ctx, cond_verdict_kernel, 1, 64, 0, st, v, bound, cond_out, ctx->status_dev, deferred ? 1 : 0));
        return after_launch(ctx);
    }
    dim3 gi(ceil_div(v.mpad, 4 * 256), 2);
    GELO_TRY(launch_chained(ctx, cond_init_kernel, gi, 256, 0, st, v, 0x5eedull, 0u));
    GELO_TRY(after_launch(ctx));
    const dim3 gr(v.mpad / kCondChunkCols, 2), gs(ceil_div(m, v.rows_per), 2);
    for (int step = -1; step < kLanczosSteps; ++step) {
        if (step >= 0) {
            if (dtype == GELO_BF16) GELO_TRY(launch_chained(ctx, cond_step_kernel<__nv_bfloat16>, gs, 256, ys_bytes, st, v));
            else if (dtype == GELO_F16) GELO_TRY(launch_chained(ctx, cond_step_kernel<__half>, gs, 256, ys_bytes, st, v));
            else GELO_TRY(launch_chained(ctx, cond_step_kernel<float>, gs, 256, ys_bytes, st, v));
            GELO_TRY(after_launch(ctx));
        }
        GELO_TRY(launch_chained(ctx, cond_reduce_kernel, gr, kCondChunkCols * kCondParts, 0, st, v, step < 0 ? 1 : (int)gs.x,
                               step));
        GELO_TRY(after_launch(ctx));
    }
    GELO_TRY(launch_chained(ctx, cond_verdict_kernel, 1, 64, 0, st, v, bound, cond_out, ctx->status_dev, deferred ? 1 : 0));
    return after_launch(ctx);
}

}  // namespace gelo

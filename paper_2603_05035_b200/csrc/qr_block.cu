// Householder QR of a Gaussian matrix in blocks of 128 columns, without a column-by-column panel
// (paper Section 3.2 step 1.2: A = Q of the QR of a Gaussian; Table 3 "A-gen (QR)").
//
// A block column P (r x b, r >= 2 b) of a Gaussian matrix, or of what earlier reflectors leave of one, is well
// conditioned (kappa below 6), so its triangular factor can be taken from the Gram matrix: P^T P = R^T R (Cholesky).
// The block reflector that maps P to [-R; 0] is then known in closed form.  With E the first b columns of the identity,
//     V = P + E R,      B = (first b rows of P) + R,      T = R^-1 B^-T,      H = I - V T V^T,      H^T P = -E R
// (the compact WY form of Schreiber and Van Loan for the reflection that exchanges the orthonormal basis P R^-1 with -E;
// T^-1 + T^-T = V^T V holds because B^T R = P^T P + (first b rows of P)^T R).  V differs from P in its top b x b block
// only, so the reflectors stay where the panel was and no pass over the panel forms them.  What is serial in a block is
// a 128 x 128 Cholesky factorisation and a 128 x 128 inverse in one CTA (block_factor_kernel); everything else is a
// product.  The update of columns C right of the block needs W' = T^T V^T C = T^T (P^T C) + D^T C1, D = R T = B^-T,
// C1 = the first b rows of C: P^T C comes out of the same product as P^T P.
// The last block, which would be square, is factorised by the one-launch Householder kernel.
//
// Against 32-column Householder panels in registers (70 us per 32 columns of serial column steps, and rank-32 updates
// between them), which the sampler used before: 2048 + 102 rows, orthogonal, calls back to back 2.80 -> 1.21 ms; the 32-layer
// sweep at 4300 rows 126 -> 114 ms.
#include "common.cuh"
#include "tc_ptx.cuh"

namespace gelo {

namespace {

constexpr int FB = kOuter;                     // block width
constexpr int FS = FB + 4;                     // shared-memory row stride (16-byte rows, conflict-free column walks)
// Two groups of 256 threads eliminate a 128 x 128 matrix each; thread (g, l) of a group (g = 0 .. 15, l = 0 .. 15) holds rows
// g + 16 i and columns l + 16 q (i, q = 0 .. 7).  Step k then always finds its pivot row and column in registers of index
// k / 16, a compile-time constant in a loop over the 16 steps that share it (the loops stay small enough for the
// instruction cache), and the rows that are still to be eliminated are spread evenly over the warps.
constexpr int kFactThreads = 512;
constexpr int kRing = 16;                      // pivot rows in flight: one slot per step that shares a register index
struct FactShared {
    float A[FB][FS];                           // R^-T (lower triangular)
    float X[FB][FS];                           // R while B is eliminated, then D = B^-T
    float row[2][kRing][FB + 4];               // pivot rows of the two groups; [FB]: reciprocal of the pivot
    uint64_t full[2][kRing];                   // row slot published
    uint64_t rready[8];                        // 16 rows of R complete
};
constexpr int kFactSmemBytes = (int)sizeof(FactShared);

__device__ __forceinline__ float fast_rcp(float x)
{
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}

// Bounded wait for a phase of a barrier of this CTA (a block that runs out of patience sets the status word and goes on:
// nothing it does afterwards can hang).
__device__ __forceinline__ void fact_wait(const uint64_t* bar, uint32_t parity, int* status)
{
    const uint32_t addr = tcx::smem_u32(bar);
#pragma unroll 1
    for (int spin = 0; spin < (1 << 22); ++spin)
        if (tcx::mbar_try(addr, parity)) return;
    atomicCAS(status, 0, (int)GELO_ERR_TIMEOUT);
}

// Half warp g publishes its row of register index J: lane l the values of its columns as two float4.
template <int J>
__device__ __forceinline__ void publish_row(const float (&a)[8][8], float* slot, uint64_t* bar, int t, int g, int l)
{
    if (g == t) {
        *reinterpret_cast<float4*>(slot + 4 * l) = make_float4(a[J][0], a[J][1], a[J][2], a[J][3]);
        *reinterpret_cast<float4*>(slot + 64 + 4 * l) = make_float4(a[J][4], a[J][5], a[J][6], a[J][7]);
        if (l == t) slot[FB] = fast_rcp(a[J][J]);
    }
    __syncwarp();
    if (g == t && l == 0) tcx::mbar_arrive(tcx::smem_u32(bar));
}

// Sixteen elimination steps with pivots k = 16 J + t:
//     a_ij -= a_ik a_kj / a_kk   (j != k),      a_ik <- -a_ik / a_kk,
// i.e. the inverse of the eliminating factor grows in the columns that are cleared.  kJordan: all rows i != k are
// eliminated and row k becomes a_kj / a_kk, a_kk <- 1 / a_kk (the full inverse in the end); otherwise only the rows below k.
// The special column and row ride along in the same multiply-adds: a_ik - a_ik (1 + 1 / a_kk) = -a_ik / a_kk and
// a_kj - (a_kk - 1) (a_kj / a_kk) = a_kj / a_kk, exact enough because the caller scales the matrix to pivots around 1.
// There is no barrier of all warps: a step waits for its pivot row only, and the owner of the next one updates and
// publishes it before its other rows, so the latency from row to row is hidden behind the multiply-adds.  (A slot is
// written again 16 steps later; every warp publishes twice in 16 steps and reads a step's row before it publishes the
// next one, so by then all of them have read it.)
template <int J, bool kJordan>
__device__ __forceinline__ void sixteen_steps(float (&a)[8][8], float (*ring)[FB + 4], uint64_t* full, int g, int l, int* status)
{
    const int half = threadIdx.x & 16;
    if (g < 2) publish_row<J>(a, ring[0], full, 0, g, l);
#pragma unroll 1
    for (int t = 0; t < 16; ++t) {
        float c[8];
#pragma unroll
        for (int i = kJordan ? 0 : J; i < 8; ++i) c[i] = __shfl_sync(0xffffffffu, a[i][J], half + t);
        if (kJordan) c[J] -= (g == t) ? 1.0f : 0.0f;
        else c[J] = (g <= t) ? 0.0f : c[J];
        fact_wait(full + t, J & 1, status);
        const float* slot = ring[t];
        const float4 ra = *reinterpret_cast<const float4*>(slot + 4 * l), rb = *reinterpret_cast<const float4*>(slot + 64 + 4 * l);
        const float rp = slot[FB];
        float u[8] = {ra.x * rp, ra.y * rp, ra.z * rp, ra.w * rp, rb.x * rp, rb.y * rp, rb.z * rp, rb.w * rp};
        if (l == t) u[J] = 1.0f + rp;
#pragma unroll
        for (int q = 0; q < 8; ++q) a[J][q] = fmaf(-c[J], u[q], a[J][q]);
        if (t < 15 && (g >> 1) == ((t + 1) >> 1)) publish_row<J>(a, ring[t + 1], full + t + 1, t + 1, g, l);
#pragma unroll
        for (int i = kJordan ? 0 : J + 1; i < 8; ++i)
            if (i != J) {
#pragma unroll
                for (int q = 0; q < 8; ++q) a[i][q] = fmaf(-c[i], u[q], a[i][q]);
            }
    }
}

// The Gram group: elimination of G = L Delta L^T, then row 16 J + g of R = Delta^-1/2 (Delta L^T) and of R^-T = Delta^-1/2
// L^-1, which are final after these steps.
template <int J>
__device__ __forceinline__ void gram_steps(float (&a)[8][8], FactShared& s, float* P1, int ld, int ob, float scale, int g, int l,
                                           int* status)
{
    sixteen_steps<J, false>(a, s.row[0], s.full[0], g, l, status);
    const float d = __shfl_sync(0xffffffffu, a[J][J], (threadIdx.x & 16) + g);   // the row's diagonal entry: column l = g
    const float rs = rsqrtf(d);
    if (!(d > 0.0f)) atomicCAS(status, 0, (int)GELO_ERR_COND);                   // a Gaussian block never gets here
    const int r = 16 * J + g;
#pragma unroll
    for (int q = 0; q < 8; ++q) {
        const int c = l + 16 * q;
        const float v = a[J][q] * rs;
        s.A[r][c] = (c < r) ? v : ((c == r) ? rs : 0.0f);
        s.X[r][c] = (c >= r) ? v : 0.0f;
    }
    __syncwarp();
    if ((threadIdx.x & 31) == 0) tcx::mbar_arrive(tcx::smem_u32(&s.rready[J]));
#pragma unroll
    for (int q = J; q < 8; ++q) {                                                // B = P1 + R, the top block of V
        const int c = l + 16 * q;
        if (c >= r && c < ob) P1[(size_t)r * ld + c] += scale * (a[J][q] * rs);
    }
}

// The other group: Gauss-Jordan inverse of B = P1 + R.  Rows of R are added when their steps begin; they add nothing to the
// columns that earlier steps read.
template <int J>
__device__ __forceinline__ void inverse_steps(float (&b)[8][8], FactShared& s, int g, int l, int* status)
{
    fact_wait(&s.rready[J], 0, status);
#pragma unroll
    for (int q = J; q < 8; ++q) b[J][q] += s.X[16 * J + g][l + 16 * q];
    sixteen_steps<J, true>(b, s.row[1], s.full[1], g, l, status);
}

// One CTA.  Z (ob x ob, stride ldz): the Gram matrix P^T P.  P1: the first ob rows of the panel (stride ld), overwritten
// with B = P1 + R.  T (stride ldt) = R^-1 B^-T and D (stride ldd) = dscale * B^-T, both rounded to tf32 if `round`.
// ob <= 128, a multiple of 4; the kernel works on 128 x 128 with an identity in the part past ob.  `scale` is a power of
// two close to the norm of a panel column.
__global__ void __launch_bounds__(kFactThreads, 1)
block_factor_kernel(const float* __restrict__ Z, int ldz, float* P1, int ld, int ob, float* __restrict__ T,
                    int ldt, float* __restrict__ D, int ldd, float scale, float dscale, int round, int* __restrict__ status)
{
    extern __shared__ __align__(16) uint8_t fsm[];
    FactShared& s = *reinterpret_cast<FactShared*>(fsm);
    const int tid = threadIdx.x, g = (tid & 255) >> 4, l = tid & 15;
    const float s1 = 1.0f / scale, s2 = s1 * s1;

    if (tid == 0) {
        for (int i = 0; i < kRing; ++i) { tcx::mbar_init(tcx::smem_u32(&s.full[0][i]), 1); tcx::mbar_init(tcx::smem_u32(&s.full[1][i]), 1); }
        for (int i = 0; i < 8; ++i) tcx::mbar_init(tcx::smem_u32(&s.rready[i]), 8);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    float a[8][8];
    {
        const float* src = tid < 256 ? Z : P1;
        const int lds = tid < 256 ? ldz : ld;
        const float f = tid < 256 ? s2 : s1, one = tid < 256 ? 1.0f : 0.0f;
#pragma unroll
        for (int i = 0; i < 8; ++i)
#pragma unroll
            for (int q = 0; q < 8; ++q) {
                const int r = g + 16 * i, c = l + 16 * q;
                a[i][q] = (r < ob && c < ob) ? f * src[(size_t)r * lds + c] : (r == c ? one : 0.0f);
            }
    }
    __syncthreads();
    if (tid < 256) {
        gram_steps<0>(a, s, P1, ld, ob, scale, g, l, status);
        gram_steps<1>(a, s, P1, ld, ob, scale, g, l, status);
        gram_steps<2>(a, s, P1, ld, ob, scale, g, l, status);
        gram_steps<3>(a, s, P1, ld, ob, scale, g, l, status);
        gram_steps<4>(a, s, P1, ld, ob, scale, g, l, status);
        gram_steps<5>(a, s, P1, ld, ob, scale, g, l, status);
        gram_steps<6>(a, s, P1, ld, ob, scale, g, l, status);
        gram_steps<7>(a, s, P1, ld, ob, scale, g, l, status);
        __syncthreads();
    } else {
        inverse_steps<0>(a, s, g, l, status);
        inverse_steps<1>(a, s, g, l, status);
        inverse_steps<2>(a, s, g, l, status);
        inverse_steps<3>(a, s, g, l, status);
        inverse_steps<4>(a, s, g, l, status);
        inverse_steps<5>(a, s, g, l, status);
        inverse_steps<6>(a, s, g, l, status);
        inverse_steps<7>(a, s, g, l, status);
        __syncthreads();                                                         // R has been read by everybody
#pragma unroll
        for (int i = 0; i < 8; ++i)
#pragma unroll
            for (int q = 0; q < 8; ++q) s.X[l + 16 * q][g + 16 * i] = a[i][q];
    }
    __syncthreads();
    auto out_val = [&](float v) { return round ? tcx::round_tf32(v) : v; };
    const float ds = dscale * s1;
    for (int idx = tid; idx < FB * FB / 4; idx += kFactThreads) {
        const int r = idx >> 5, c = (idx & 31) * 4;
        if (r < ob && c < ob) {
            const float4 v = *reinterpret_cast<const float4*>(&s.X[r][c]);
            *reinterpret_cast<float4*>(D + (size_t)r * ldd + c) =
                make_float4(out_val(ds * v.x), out_val(ds * v.y), out_val(ds * v.z), out_val(ds * v.w));
        }
    }
    // ---- T = R^-1 D = (R^-T)^T D: 8 rows per warp, 4 columns per lane; a row block from row r0 on only meets rows
    //      k >= r0, so short and long blocks are dealt evenly to the SM's four schedulers ----
    const int warp = tid >> 5, n0 = 4 * (tid & 31);
    const int r0 = 8 * ((warp & 4) ? (warp ^ 3) : warp);
    float x[8][4];
#pragma unroll
    for (int i = 0; i < 8; ++i)
#pragma unroll
        for (int q = 0; q < 4; ++q) x[i][q] = 0.0f;
#pragma unroll 4
    for (int k = r0; k < FB; ++k) {
        const float4 u = *reinterpret_cast<const float4*>(&s.A[k][r0]), v = *reinterpret_cast<const float4*>(&s.A[k][r0 + 4]);
        const float4 y = *reinterpret_cast<const float4*>(&s.X[k][n0]);
        const float uu[8] = {u.x, u.y, u.z, u.w, v.x, v.y, v.z, v.w};
        const float yy[4] = {y.x, y.y, y.z, y.w};
#pragma unroll
        for (int i = 0; i < 8; ++i)
#pragma unroll
            for (int q = 0; q < 4; ++q) x[i][q] = fmaf(uu[i], yy[q], x[i][q]);
    }
#pragma unroll
    for (int i = 0; i < 8; ++i)
        if (r0 + i < ob && n0 < ob)
            *reinterpret_cast<float4*>(T + (size_t)(r0 + i) * ldt + n0) =
                make_float4(out_val(s2 * x[i][0]), out_val(s2 * x[i][1]), out_val(s2 * x[i][2]), out_val(s2 * x[i][3]));
}

// Z = scale * (sum of the K slices of P^T [P | C]), in slice order; the first ob columns (the Gram matrix) stay fp32, the
// others are rounded to tf32 (they feed the next product).  Also clears the rows above the block (z_rows x ob) where the
// superblock's reflectors are zero.
__global__ void __launch_bounds__(256)
block_sum_kernel(const float* __restrict__ planes, size_t plane, int parts, int ldp, int rows, int cols, int ob, float scale,
                 float* __restrict__ Z, int ldz, float* __restrict__ zero, int z_rows, int ld)
{
    const int idx = blockIdx.x * 256 + threadIdx.x;
    const int c4n = cols >> 2, o4n = ob >> 2;
    if (idx < rows * c4n) {
        const int r = idx / c4n, c = (idx - r * c4n) * 4;
        float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll 4
        for (int q = 0; q < parts; ++q) {
            const float4 t = *reinterpret_cast<const float4*>(planes + q * plane + (size_t)r * ldp + c);
            acc.x += t.x; acc.y += t.y; acc.z += t.z; acc.w += t.w;
        }
        acc.x *= scale; acc.y *= scale; acc.z *= scale; acc.w *= scale;
        if (c >= ob) {
            acc.x = tcx::round_tf32(acc.x); acc.y = tcx::round_tf32(acc.y);
            acc.z = tcx::round_tf32(acc.z); acc.w = tcx::round_tf32(acc.w);
        }
        *reinterpret_cast<float4*>(Z + (size_t)r * ldz + c) = acc;
    } else if (idx - rows * c4n < z_rows * o4n) {
        const int e = idx - rows * c4n;
        const int r = e / o4n, c = (e - r * o4n) * 4;
        *reinterpret_cast<float4*>(zero + (size_t)r * ld + c) = make_float4(0.f, 0.f, 0.f, 0.f);
    }
}

// Q <- diag(-I, Q_f S): the columns of the blocks start as -e_j (their R has a negative diagonal, and A takes the
// factor whose R is positive), the last f columns as the Householder factor Qf (f x f at its place in Q) with the
// columns flipped where its R (diagonal of Rf) is negative.  Everything else is cleared.
__global__ void __launch_bounds__(256)
start_q_kernel(float* __restrict__ Q, int ld, int m, int bf, const float* __restrict__ R)
{
    const int r = blockIdx.y;
    const int c = (blockIdx.x * 256 + threadIdx.x) * 4;
    if (c >= ld) return;
    float v[4];
    float* p = Q + (size_t)r * ld + c;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        const int cc = c + j;
        v[j] = (cc == r) ? -1.0f : 0.0f;
        if (cc >= bf) {
            v[j] = 0.0f;
            if (r >= bf && cc < m) v[j] = (R[(size_t)cc * ld + cc] < 0.0f) ? -p[j] : p[j];
        }
    }
    *reinterpret_cast<float4*>(p) = make_float4(v[0], v[1], v[2], v[3]);
}

}  // namespace

bool gaussian_qr_supports(int m) { return m > FB; }

int run_gaussian_qr(gelo_ctx* ctx, int m, float* G, int ld, float* Q, const TcScratch& tc, cudaStream_t st)
{
    static bool attr_done[64] = {};
    if (ctx->device >= 0 && ctx->device < 64 && !attr_done[ctx->device]) {
        GELO_CUDA_OK(cudaFuncSetAttribute(block_factor_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kFactSmemBytes));
        attr_done[ctx->device] = true;
    }
    const float loss1 = 1.0f + kTf32TruncLoss, loss2 = loss1 * loss1;
    const int width = ctx->tc_update_ctas > 0 ? ctx->tc_update_ctas : ctx->sm_count;   // CTAs one launch may use

    // V^T C with few output tiles: the rows are cut into slices whose partial products are summed in a fixed order
    auto slices = [&](int M, int N, int most) {
        const int tiles = ceil_div(M, 128) * ceil_div(N, 256);
        int want = (2 * tiles >= width) ? 1 : ceil_div(2 * width, tiles);
        return want > most ? most : want;
    };
    // C (rows from r0) <- (I - V op(T) V^T) C for the merged reflectors of a superblock (kv columns from c0)
    auto apply = [&](int c0, int kv, const float* T, float* C, int nc, bool transpose_t) -> int {
        const int nr = m - c0;
        const int nc8 = (nc + 7) & ~7;
        const float* V = G + (size_t)c0 * ld + c0;
        const int want = slices(kv, nc8, kSuperKSplit);
        if (want <= 1) {
            GELO_TRY(launch_gemm_tf32(ctx, kv, nc8, nr, V, ld, true, C, ld, false, tc.w32[0], ld, true, loss2, 1, 0, nullptr, st));
        } else {
            int used = 0;
            const size_t plane = (size_t)kv * ld;
            GELO_TRY(launch_gemm_tf32(ctx, kv, nc8, nr, V, ld, true, C, ld, false, tc.wf32, ld, false, 1.0f, want, plane, &used, st));
            GELO_TRY(launch_sum_planes(ctx, tc.wf32, plane, used, ld, kv, nc8, loss2, tc.w32[0], ld, st));
        }
        // (the factor loss1 makes up for the truncation of V in the last product)
        GELO_TRY(launch_gemm_tf32(ctx, kv, nc8, kv, T, kSuper, transpose_t, tc.w32[0], ld, false, tc.w32[1], ld, true, loss1, 1, 0,
                                  nullptr, st));
        return launch_gemm_tf32(ctx, nr, nc, kv, V, ld, false, tc.w32[1], ld, true, C, ld, false, 1.0f, 1, 0, nullptr, st);
    };

    // block columns: 128 wide while at least twice as many rows are left, then one that leaves a square of at most 128
    std::vector<int> start;
    int bf = 0;                                              // first column of the square that is left for Householder
    while (m - bf > FB) {
        start.push_back(bf);
        bf += (m - bf >= 2 * FB) ? FB : ((m - bf - FB + 3) & ~3);
    }
    start.push_back(bf);
    const int nblocks = (int)start.size() - 1;
    const int per = kSuper / FB;
    // ---- factorisation ----
    for (int s = 0; s < nblocks; s += per) {
        const int e = (s + per < nblocks) ? s + per : nblocks;
        const int s0 = start[s], send = start[e];
        float* Ts = tc.tsuper + (size_t)(s / per) * kSuper * kSuper;
        GELO_CUDA_OK(cudaMemsetAsync(Ts, 0, (size_t)kSuper * kSuper * sizeof(float), st));
        for (int b = s; b < e; ++b) {
            const int b0 = start[b], ob = start[b + 1] - b0, bend = b0 + ob;
            const int nr = m - b0, r = b0 - s0;
            const int ncs = (send - b0 + 7) & ~7;            // the block and the superblock's columns right of it
            float* P = G + (size_t)b0 * ld + b0;
            int used = 0;
            const size_t plane = (size_t)FB * ld;
            GELO_TRY(launch_gemm_tf32(ctx, ob, ncs, nr, P, ld, true, P, ld, false, tc.wf32, ld, false, 1.0f,
                                      slices(ob, ncs, kMaxKSplit), plane, &used, st));
            const int work = ob * (ncs >> 2) + r * (ob >> 2);
            block_sum_kernel<<<ceil_div(work, 256), 256, 0, st>>>(tc.wf32, plane, used, ld, ob, ncs, ob, loss2, tc.w32[0], ld,
                                                                 G + (size_t)s0 * ld + b0, r, ld);
            GELO_TRY(after_launch(ctx));
            float* Tb = Ts + (size_t)r * kSuper + r;
            float scale = 1.0f;                              // a power of two with scale^2 about nr
            while (2.0f * scale * scale < (float)nr) scale *= 2.0f;
            block_factor_kernel<<<1, kFactThreads, kFactSmemBytes, st>>>(tc.w32[0], ld, P, ld, ob, Tb, kSuper, tc.t128, FB,
                                                                        scale, loss1, 1, ctx->status_dev);
            GELO_TRY(after_launch(ctx));
            if (send > bend) {
                // W' = T^T (P^T C) + D^T C1, then C -= V W'
                const int nc = send - bend, nc8 = (nc + 7) & ~7;
                GELO_TRY(launch_gemm_tf32_dual(ctx, ob, nc8, ob, Tb, kSuper, tc.w32[0] + ob, ld, tc.t128, FB, P + ob, ld, tc.w32[1], ld,
                                               loss1, st));
                GELO_TRY(launch_gemm_tf32(ctx, nr, nc, ob, P, ld, false, tc.w32[1], ld, true, P + ob, ld, false, 1.0f, 1, 0, nullptr,
                                          st));
            }
            if (r > 0) {
                // merge into the superblock's factor: T[0:r, r:r+ob] = -T[0:r, 0:r] (V_<^T V_b) T_b
                const float* Vl = G + (size_t)b0 * ld + s0;
                GELO_TRY(launch_gemm_tf32(ctx, r, (ob + 7) & ~7, nr, Vl, ld, true, P, ld, false, tc.wf32, FB, false, 1.0f,
                                          slices(r, ob, kMaxKSplit), (size_t)r * FB, &used, st));
                GELO_TRY(launch_sum_planes(ctx, tc.wf32, (size_t)r * FB, used, FB, r, ob, loss2, tc.sx, FB, st));
                GELO_TRY(launch_gemm_tf32(ctx, r, (ob + 7) & ~7, ob, tc.sx, FB, false, Tb, kSuper, false, tc.xb, FB, true, 1.0f, 1, 0,
                                          nullptr, st));
                GELO_TRY(launch_gemm_tf32(ctx, r, (ob + 7) & ~7, r, Ts, kSuper, false, tc.xb, FB, false, Ts + r, kSuper, true, -1.0f,
                                          1, 0, nullptr, st));
            }
        }
        GELO_TRY(apply(s0, send - s0, Ts, G + (size_t)s0 * ld + send, m - send, true));
    }
    // ---- the square that is left, and Q accumulated backwards, one superblock at a time ----
    GELO_TRY(launch_qr_small(ctx, m - bf, G + (size_t)bf * ld + bf, ld, Q + (size_t)bf * ld + bf, st));
    start_q_kernel<<<dim3(ceil_div(ld, 1024), m), 256, 0, st>>>(Q, ld, m, bf, G);
    GELO_TRY(after_launch(ctx));
    for (int s = (nblocks - 1) / per * per; s >= 0; s -= per) {
        const int e = (s + per < nblocks) ? s + per : nblocks;
        const int s0 = start[s];
        GELO_TRY(apply(s0, start[e] - s0, tc.tsuper + (size_t)(s / per) * kSuper * kSuper, Q + (size_t)s0 * ld + s0, m - s0, false));
    }
    return GELO_OK;
}

}  // namespace gelo

// Blocked Householder QR (compact WY) that turns an m x m Gaussian matrix into the
// orthogonal mixing matrix of the offload: A = Q diag(sign R_jj), A^-1 = A^T
// (paper Section 3.2 step 1.2; "If A is orthogonal, A^-1 = A^T").
//
//   for each panel of kPanel columns:
//       panel kernel   : Householder vectors V (unit diagonal), tau, and the
//                        triangular factor T with  H_1 ... H_b = I - V T V^T
//       trailing update: C <- (I - V T^T V^T) C   as three GEMMs
//   Q is then accumulated backwards, panel by panel, from the identity:
//       Q[j0:, j0:] <- (I - V T V^T) Q[j0:, j0:]
//
// The panel kernel is one CTA: lane = panel column, warps stripe over rows, so each
// row of the panel is one coalesced 128-byte access; column norms and the products
// v^T C of all remaining columns come from ONE block-wide reduction per column
// (warp partial sums in registers, cross-warp sums in shared memory).
#include <cooperative_groups.h>

#include "common.cuh"
#include "philox.cuh"

#include <type_traits>

namespace gelo {

namespace {

constexpr int NB = kPanel;          // 32: one lane per panel column
constexpr int kPanelThreads = 1024;
constexpr int kPanelWarps = kPanelThreads / 32;

// R: m x m (stride ld), panel = columns j0 .. j0+jb-1, rows j0 .. m-1 (in place).
// V: m x ld; this panel's reflectors go to columns j0 .. j0+jb-1 (rows < j0 untouched,
//    rows j0.. : zeros above the diagonal, 1 on it, v below).
// T: NB x NB, upper triangular, zero elsewhere.
__global__ void __launch_bounds__(kPanelThreads)
qr_panel_kernel(float* __restrict__ R, int ld, int m, int j0, int jb,
                float* __restrict__ V, float* __restrict__ T)
{
    __shared__ float red[kPanelWarps][NB + 1];
    __shared__ float dsum[NB];
    __shared__ float rowj[NB];
    __shared__ float tau_s[NB];
    __shared__ float gram[NB][NB + 1];
    __shared__ float t_s[NB][NB + 1];

    const int lane = threadIdx.x & 31;
    const int warp = threadIdx.x >> 5;
    const bool col_ok = lane < jb;
    const unsigned full = 0xffffffffu;

    for (int c = 0; c < jb; ++c) {
        const int j = j0 + c;
        // ---- d[c'] = sum_{r > j} R[r, j] * R[r, j0 + c'] ------------------------------
        float acc = 0.0f;
        for (int r = j + 1 + warp; r < m; r += kPanelWarps) {
            const float y = col_ok ? R[(size_t)r * ld + j0 + lane] : 0.0f;
            const float x = __shfl_sync(full, y, c);
            acc = fmaf(x, y, acc);
        }
        red[warp][lane] = acc;
        __syncthreads();
        if (warp == 0) {
            float s = 0.0f;
#pragma unroll 8
            for (int w = 0; w < kPanelWarps; ++w) s += red[w][lane];
            dsum[lane] = s;
            rowj[lane] = col_ok ? R[(size_t)j * ld + j0 + lane] : 0.0f;
        }
        __syncthreads();
        // ---- reflector scalars (every thread, same values) --------------------------------
        const float alpha = rowj[c];
        const float sigma = dsum[c];
        float beta = alpha, tau = 0.0f, scale = 0.0f;
        if (sigma > 0.0f) {
            beta = -copysignf(sqrtf(fmaf(alpha, alpha, sigma)), alpha);
            tau = (beta - alpha) / beta;
            scale = 1.0f / (alpha - beta);
        }
        // w[c'] = v^T R[j:, c'] = R[j, c'] + scale * d[c']   (v = [1; scale * x])
        const float wv = (lane > c && col_ok) ? fmaf(scale, dsum[lane], rowj[lane]) : 0.0f;
        const float tw = tau * wv;
        // ---- apply H_c to the rest of the panel and store v ---------------------------------
        if (warp == 0) {
            // row j itself
            if (col_ok) {
                float y = rowj[lane];
                if (lane > c) y -= tw;
                else if (lane == c) y = beta;
                R[(size_t)j * ld + j0 + lane] = y;
                V[(size_t)j * ld + j0 + lane] = (lane == c) ? 1.0f : ((lane > c) ? 0.0f : V[(size_t)j * ld + j0 + lane]);
            }
            if (lane == 0) tau_s[c] = tau;
        }
        for (int r = j + 1 + warp; r < m; r += kPanelWarps) {
            float y = col_ok ? R[(size_t)r * ld + j0 + lane] : 0.0f;
            const float x = __shfl_sync(full, y, c);
            const float v = x * scale;
            if (col_ok) {
                if (lane > c) {
                    y = fmaf(-tw, v, y);
                    R[(size_t)r * ld + j0 + lane] = y;
                } else if (lane == c) {
                    R[(size_t)r * ld + j0 + lane] = 0.0f;     // below-diagonal part of R
                    V[(size_t)r * ld + j0 + lane] = v;
                }
            }
        }
        __syncthreads();
    }

    // ---- zero V above the diagonal of this panel (rows j0..j0+jb-1 were written column by
    //      column; entries with row < column inside the panel block must be zero) ----------
    for (int idx = threadIdx.x; idx < jb * NB; idx += kPanelThreads) {
        const int r = idx / NB, cc = idx % NB;
        if (cc < jb && r < cc) V[(size_t)(j0 + r) * ld + j0 + cc] = 0.0f;
    }
    __syncthreads();

    // ---- Gram matrix of the reflectors: gram[a][b] = sum_r V[r, a] V[r, b] ----------------
    for (int idx = threadIdx.x; idx < NB * (NB + 1); idx += kPanelThreads) (&gram[0][0])[idx] = 0.0f;
    __syncthreads();
    {
        float g[NB];
#pragma unroll
        for (int a = 0; a < NB; ++a) g[a] = 0.0f;
        for (int r = j0 + warp; r < m; r += kPanelWarps) {
            const float y = col_ok ? V[(size_t)r * ld + j0 + lane] : 0.0f;
#pragma unroll
            for (int a = 0; a < NB; ++a) g[a] = fmaf(__shfl_sync(full, y, a), y, g[a]);
        }
        // fixed summation order (warp 0, 1, ...) keeps the factor bit-reproducible
        for (int w = 0; w < kPanelWarps; ++w) {
            if (warp == w) {
#pragma unroll
                for (int a = 0; a < NB; ++a) gram[a][lane] += g[a];
            }
            __syncthreads();
        }
    }

    // ---- T (forward, columnwise): T[c][c] = tau_c, T[0:c, c] = -tau_c T[0:c, 0:c] gram[0:c, c]
    if (warp == 0) {
        for (int a = 0; a < NB; ++a) t_s[a][lane] = 0.0f;
        __syncwarp();
        for (int c = 0; c < jb; ++c) {
            const float tc = tau_s[c];
            float s = 0.0f;
            if (lane < c) {
                for (int b = lane; b < c; ++b) s = fmaf(t_s[lane][b], gram[b][c], s);
            }
            __syncwarp();
            if (lane < c) t_s[lane][c] = -tc * s;
            else if (lane == c) t_s[c][c] = tc;
            __syncwarp();
        }
        for (int a = 0; a < NB; ++a) T[a * NB + lane] = t_s[a][lane];
    }
}

// ---- register-resident panel on a thread-block cluster -----------------------------------
//
// The same Householder panel, but the whole panel lives in registers spread over a cluster of
// CS CTAs (CS * 32 warps; global warp g holds rows j0 + g + i * CS * 32, i = 0 .. RPT-1; lane =
// panel column).  Per column there is ONE reduction: warp partial sums -> shared memory -> one
// vector per CTA, which every CTA stores into every other CTA's shared memory (distributed
// shared memory) followed by one cluster barrier.  Only the first row of a warp can lie on or
// above the pivot row, so all other rows run branch-free.  The lanes that are idle in the
// reduction (columns already factorised) carry V^T v for the triangular factor T, gathered
// during the previous column's update, so no separate Gram pass is needed.  All sums run in a
// fixed order: results are bit-reproducible.
constexpr int kClusterMax = 8;
constexpr int kMaxRowsPerThread = 28;                      // rows a thread can hold in registers (64 each at 1024 threads)
constexpr int kClusterPanelMaxRows = kClusterMax * kPanelWarps * kMaxRowsPerThread;   // 7168

template <int RPT>
__global__ void __launch_bounds__(kPanelThreads, 1)
qr_panel_cluster_kernel(float* __restrict__ R, int ld, int m, int j0, int jb,
                        float* __restrict__ V, float* __restrict__ T)
{
    namespace cg = cooperative_groups;
    cg::cluster_group cluster = cg::this_cluster();
    const int CS = (int)cluster.num_blocks();
    const int rank = (int)cluster.block_rank();

    __shared__ float red[kPanelWarps][NB + 1];
    __shared__ float slot[2][kClusterMax][NB];
    __shared__ float rowbuf[2][NB];
    __shared__ float gram[NB][NB + 1];
    __shared__ float tau_s[NB];
    __shared__ float t_s[NB][NB + 1];
    __shared__ float coef_s[NB];
    __shared__ float tw_s[NB];
    __shared__ float scal_s[2];

    const int lane = threadIdx.x & 31;
    const int warp = threadIdx.x >> 5;
    const int gw = rank * kPanelWarps + warp;
    const int stride = CS * kPanelWarps;
    const bool col_ok = lane < jb;
    const unsigned full = 0xffffffffu;

    float x[RPT];
#pragma unroll
    for (int i = 0; i < RPT; ++i) {
        const int row = j0 + i * stride + gw;
        x[i] = (row < m && col_ok) ? R[(size_t)row * ld + j0 + lane] : 0.0f;
    }
    for (int idx = threadIdx.x; idx < NB * (NB + 1); idx += kPanelThreads) (&gram[0][0])[idx] = 0.0f;
    if (CS > 1) cluster.sync(); else __syncthreads();     // every CTA of the cluster is running before remote stores

    float g = 0.0f;                                        // v_{c-1}^T v_lane, gathered during the previous update
    for (int c = 0; c <= jb; ++c) {
        const int par = c & 1;
        const int csrc = c & 31;
        // ---- lanes >= c: x_c^T x_lane over the rows below the pivot row j = j0 + c ----
        // (column c of a row is fetched from lane c again in the update below rather than kept: registers decide how
        // many rows a thread can hold, and with them how few SMs a panel occupies)
        float acc = 0.0f;
#pragma unroll
        for (int i = 1; i < RPT; ++i) acc = fmaf(__shfl_sync(full, x[i], csrc), x[i], acc);
        if (gw > c) acc = fmaf(__shfl_sync(full, x[0], csrc), x[0], acc);   // a warp's first row is below row j only past warp c
        red[warp][lane] = (lane >= c) ? acc : ((lane < c - 1) ? g : 0.0f);
        __syncthreads();
        {
            // warp w sums entry w over the 32 warps (butterfly: fixed order) and lane r ships it to CTA r
            float s = red[lane][warp];
#pragma unroll
            for (int off = 16; off > 0; off >>= 1) s += __shfl_xor_sync(full, s, off);
            if (lane < CS) cluster.map_shared_rank(&slot[par][rank][warp], lane)[0] = s;
        }
        if (c < jb && rank == 0 && warp == c) {            // the warp whose first row is row j
            for (int r = 0; r < CS; ++r) cluster.map_shared_rank(&rowbuf[par][lane], r)[0] = x[0];
        }
        if (CS > 1) cluster.sync(); else __syncthreads();

        // ---- warp 0 turns the sums into this column's reflector; everybody else only reads the result ----
        if (warp == 0) {
            float d_own = 0.0f;
            for (int r = 0; r < CS; ++r) d_own += slot[par][r][lane];
            if (c > 0 && lane < c - 1) gram[lane][c - 1] = d_own;
            if (c < jb) {
                const float sigma = __shfl_sync(full, d_own, c);
                const float alpha = rowbuf[par][c];
                const float rj = rowbuf[par][lane];
                float beta = alpha, tau = 0.0f, scale = 0.0f;
                if (sigma > 0.0f) {
                    beta = -copysignf(sqrtf(fmaf(alpha, alpha, sigma)), alpha);
                    tau = (beta - alpha) / beta;
                    scale = 1.0f / (alpha - beta);
                }
                const float wv = (lane > c && col_ok) ? fmaf(scale, d_own, rj) : 0.0f;
                const float tw = tau * wv;
                tw_s[lane] = tw;
                // x <- coef * x_c + (lane == c ? 0 : x):  -tw v for later columns, v itself in column c, nothing before
                coef_s[lane] = (lane > c) ? -tw * scale : ((lane == c) ? scale : 0.0f);
                if (lane == 0) { scal_s[0] = scale; scal_s[1] = beta; tau_s[c] = tau; }
            }
        }
        if (c == jb) break;
        __syncthreads();
        const float coef = coef_s[lane];
        const float scale = scal_s[0];
        // ---- apply H_c; every lane also gathers x_c^T x_lane (only lanes < c use it: v_c^T v_lane for T) ----
        float graw = 0.0f;
#pragma unroll
        for (int i = 1; i < RPT; ++i) {
            const float xci = __shfl_sync(full, x[i], csrc);
            graw = fmaf(xci, x[i], graw);
            x[i] = fmaf(coef, xci, (lane == c) ? 0.0f : x[i]);
        }
        g = 0.0f;
        const float xc0 = __shfl_sync(full, x[0], csrc);
        if (gw > c) {
            graw = fmaf(xc0, x[0], graw);
            x[0] = fmaf(coef, xc0, (lane == c) ? 0.0f : x[0]);
        } else if (gw == c) {                               // row j itself: v_c(j) = 1
            g = x[0];
            if (lane > c) x[0] -= tw_s[lane];
            else if (lane == c) x[0] = scal_s[1];
        }
        g = fmaf(scale, graw, g);
    }

    // ---- write back: R above / on the diagonal, reflectors below it ----
#pragma unroll
    for (int i = 0; i < RPT; ++i) {
        const int row = j0 + i * stride + gw;
        if (row < m && col_ok) {
            const int diag = j0 + lane;
            R[(size_t)row * ld + j0 + lane] = (row <= diag) ? x[i] : 0.0f;
            V[(size_t)row * ld + j0 + lane] = (row > diag) ? x[i] : ((row == diag) ? 1.0f : 0.0f);
        }
    }
    // ---- T on CTA 0, warp 0 (it wrote gram and tau_s itself) ----
    if (rank == 0 && warp == 0) {
        for (int a = 0; a < NB; ++a) t_s[a][lane] = 0.0f;
        __syncwarp();
        for (int c = 0; c < jb; ++c) {
            const float tc = tau_s[c];
            float s = 0.0f;
            if (lane < c) {
                for (int b = lane; b < c; ++b) s = fmaf(t_s[lane][b], gram[b][c], s);
            }
            __syncwarp();
            if (lane < c) t_s[lane][c] = -tc * s;
            else if (lane == c) t_s[c][c] = tc;
            __syncwarp();
        }
        for (int a = 0; a < NB; ++a) T[a * NB + lane] = t_s[a][lane];
    }
}

template <int RPT>
cudaError_t launch_cluster_panel(int cs, cudaStream_t st, float* R, int ld, int m, int j0, int jb, float* V, float* T)
{
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(cs, 1, 1);
    cfg.blockDim = dim3(kPanelThreads, 1, 1);
    cfg.dynamicSmemBytes = 0;
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = cs; attr[0].val.clusterDim.y = 1; attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, qr_panel_cluster_kernel<RPT>, R, ld, m, j0, jb, V, T);
}

// Launches the panel on the cluster / rows-per-thread combination that wastes the fewest row slots.
int launch_qr_panel(gelo_ctx* ctx, float* R, int ld, int m, int j0, int jb, float* V, float* T, cudaStream_t st)
{
    const int rows = m - j0;
    if (rows > kClusterPanelMaxRows) {
        qr_panel_kernel<<<1, kPanelThreads, 0, st>>>(R, ld, m, j0, jb, V, T);
        return after_launch(ctx);
    }
    // Alone on the GPU a panel spreads over as many SMs as give every thread at least two rows (shortest column
    // step); in a batch with many sampling lanes it packs up to 28 rows per thread and occupies as few SMs as
    // possible, since every SM it holds is one that the other lanes' kernels cannot use.
    const int rows_per_thread = ctx->tc_update_ctas > 0 ? kMaxRowsPerThread : 2;
    // (a cluster may have any size up to eight: five CTAs where four are too few, not eight)
    int cs = ceil_div(rows, kPanelWarps * rows_per_thread);
    if (cs > kClusterMax) cs = kClusterMax;
    const int rpt = ceil_div(rows, cs * kPanelWarps);
    ProfScope ps(ctx, PROF_QR_PANEL, 2.0 * rows * (double)jb * jb, st);   // flops of the column dots and updates
    cudaError_t e;
    if (rpt <= 2) e = launch_cluster_panel<2>(cs, st, R, ld, m, j0, jb, V, T);
    else if (rpt <= 3) e = launch_cluster_panel<3>(cs, st, R, ld, m, j0, jb, V, T);
    else if (rpt <= 5) e = launch_cluster_panel<5>(cs, st, R, ld, m, j0, jb, V, T);
    else if (rpt <= 7) e = launch_cluster_panel<7>(cs, st, R, ld, m, j0, jb, V, T);
    else if (rpt <= 9) e = launch_cluster_panel<9>(cs, st, R, ld, m, j0, jb, V, T);
    else if (rpt <= 11) e = launch_cluster_panel<11>(cs, st, R, ld, m, j0, jb, V, T);
    else if (rpt <= 13) e = launch_cluster_panel<13>(cs, st, R, ld, m, j0, jb, V, T);
    else if (rpt <= 15) e = launch_cluster_panel<15>(cs, st, R, ld, m, j0, jb, V, T);
    else if (rpt <= 17) e = launch_cluster_panel<17>(cs, st, R, ld, m, j0, jb, V, T);
    else if (rpt <= 20) e = launch_cluster_panel<20>(cs, st, R, ld, m, j0, jb, V, T);
    else if (rpt <= 24) e = launch_cluster_panel<24>(cs, st, R, ld, m, j0, jb, V, T);
    else e = launch_cluster_panel<28>(cs, st, R, ld, m, j0, jb, V, T);
    if (e != cudaSuccess) return GELO_ERR_CUDA;
    return after_launch(ctx);
}

__global__ void set_diagonal_kernel(float* __restrict__ Q, int ld, int m)
{
    const int r = blockIdx.x * blockDim.x + threadIdx.x;
    if (r < m) Q[(size_t)r * ld + r] = 1.0f;
}

// Q = I: a memset at copy speed, then the ones.
int set_identity(gelo_ctx* ctx, float* Q, int ld, int m, cudaStream_t st)
{
    GELO_CUDA_OK(cudaMemsetAsync(Q, 0, (size_t)m * ld * sizeof(float), st));
    set_diagonal_kernel<<<ceil_div(m, 256), 256, 0, st>>>(Q, ld, m);
    return after_launch(ctx);
}


// Gram matrix of an outer block's reflectors, S = V^T V (V: nr x ob, ob <= 128), as per-slab partial sums:
// CTA s accumulates rows [s * kGramRows, ...) in 32-row chunks staged in shared memory (256 threads, 8 x 8
// outputs each) and writes its 128 x 128 partial to part[s].
constexpr int kGramRows = 256;

__global__ void __launch_bounds__(256)
gram128_kernel(const float* __restrict__ V, int ld, int nr, int ob, float* __restrict__ part)
{
    __shared__ __align__(16) float vs[32][128 + 4];
    const int tid = threadIdx.x;
    const int ty = tid >> 4, tx = tid & 15;
    const int r0 = blockIdx.x * kGramRows;
    const int r1 = min(nr, r0 + kGramRows);
    float acc[8][8];
#pragma unroll
    for (int i = 0; i < 8; ++i)
#pragma unroll
        for (int j = 0; j < 8; ++j) acc[i][j] = 0.0f;
    for (int rb = r0; rb < r1; rb += 32) {
        // 32 rows x 128 columns: thread loads 4 float4 (row = tid / 32 + 8 i, column group = tid % 32)
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const int rr = (tid >> 5) + 8 * i, c4 = (tid & 31) * 4;
            const int row = rb + rr;
            float4 t = make_float4(0.f, 0.f, 0.f, 0.f);
            if (row < r1) {
                const float* p = V + (size_t)row * ld + c4;
                if (c4 + 3 < ob) t = *reinterpret_cast<const float4*>(p);
                else {
                    if (c4 + 0 < ob) t.x = p[0];
                    if (c4 + 1 < ob) t.y = p[1];
                    if (c4 + 2 < ob) t.z = p[2];
                }
            }
            *reinterpret_cast<float4*>(&vs[rr][c4]) = t;
        }
        __syncthreads();
#pragma unroll 8
        for (int k = 0; k < 32; ++k) {
            const float4 a0 = *reinterpret_cast<const float4*>(&vs[k][ty * 4]);
            const float4 a1 = *reinterpret_cast<const float4*>(&vs[k][ty * 4 + 64]);
            const float4 b0 = *reinterpret_cast<const float4*>(&vs[k][tx * 4]);
            const float4 b1 = *reinterpret_cast<const float4*>(&vs[k][tx * 4 + 64]);
            const float a[8] = {a0.x, a0.y, a0.z, a0.w, a1.x, a1.y, a1.z, a1.w};
            const float b[8] = {b0.x, b0.y, b0.z, b0.w, b1.x, b1.y, b1.z, b1.w};
#pragma unroll
            for (int i = 0; i < 8; ++i)
#pragma unroll
                for (int j = 0; j < 8; ++j) acc[i][j] = fmaf(a[i], b[j], acc[i][j]);
        }
        __syncthreads();
    }
    float* out = part + (size_t)blockIdx.x * 128 * 128;
#pragma unroll
    for (int i = 0; i < 8; ++i) {
        const int r = ty * 4 + (i >> 2) * 64 + (i & 3);
#pragma unroll
        for (int h = 0; h < 2; ++h)
            *reinterpret_cast<float4*>(out + (size_t)r * 128 + tx * 4 + h * 64) =
                make_float4(acc[i][4 * h + 0], acc[i][4 * h + 1], acc[i][4 * h + 2], acc[i][4 * h + 3]);
    }
}

// Triangular factor of an outer block from the factors of its 32-column panels:
//   (I - V1 T1 V1^T)(I - V2 T2 V2^T) = I - [V1 V2] [[T1, -T1 (V1^T V2) T2], [0, T2]] [V1 V2]^T,
// applied panel after panel.  part: `slabs` partial Gram matrices of 128 rows with row stride ldp (summed here in
// slab order); T32: the panels' factors.  One CTA, everything in shared memory.
constexpr int kMergeSmemBytes = (2 * 128 * 129 + 96 * 33 + 32 * 33) * 4;

__global__ void __launch_bounds__(1024)
t_merge_kernel(const float* __restrict__ part, int slabs, int ldp, const float* __restrict__ T32, int ob, float* __restrict__ T128)
{
    extern __shared__ float msm[];
    float (*S)[129] = reinterpret_cast<float (*)[129]>(msm);
    float (*Tm)[129] = reinterpret_cast<float (*)[129]>(msm + 128 * 129);
    float (*x_s)[33] = reinterpret_cast<float (*)[33]>(msm + 2 * 128 * 129);
    float (*tk_s)[33] = reinterpret_cast<float (*)[33]>(msm + 2 * 128 * 129 + 96 * 33);
    const int tid = threadIdx.x;
    for (int idx = tid; idx < 128 * 128; idx += 1024) {
        float acc = 0.0f;
        for (int q = 0; q < slabs; ++q) acc += part[((size_t)q * 128 + (idx >> 7)) * ldp + (idx & 127)];
        S[idx >> 7][idx & 127] = acc;
        Tm[idx >> 7][idx & 127] = 0.0f;
    }
    __syncthreads();
    const int nsub = (ob + NB - 1) / NB;
    for (int k = 0; k < nsub; ++k) {
        {
            const int a = tid >> 5, b = tid & 31;                   // 1024 threads = one 32 x 32 factor
            const float t = T32[(size_t)k * NB * NB + tid];
            tk_s[a][b] = t;
            Tm[k * NB + a][k * NB + b] = t;
        }
        __syncthreads();
        const int rows = k * NB;                                    // rows of the already merged part
        // X = S[0:rows, k*32 : k*32+32] * T_k
        for (int idx = tid; idx < rows * NB; idx += 1024) {
            const int r = idx >> 5, cc = idx & 31;
            float acc = 0.0f;
            for (int b = 0; b <= cc; ++b) acc = fmaf(S[r][k * NB + b], tk_s[b][cc], acc);
            x_s[r][cc] = acc;
        }
        __syncthreads();
        // T[0:rows, k*32 : k*32+32] = -T[0:rows, 0:rows] * X   (upper triangular left factor)
        for (int idx = tid; idx < rows * NB; idx += 1024) {
            const int r = idx >> 5, cc = idx & 31;
            float acc = 0.0f;
            for (int q = r; q < rows; ++q) acc = fmaf(Tm[r][q], x_s[q][cc], acc);
            Tm[r][k * NB + cc] = -acc;
        }
        __syncthreads();
    }
    for (int idx = tid; idx < 128 * 128; idx += 1024) T128[idx] = Tm[idx >> 7][idx & 127];
}

// ---- the whole factorisation of a small matrix (m <= 128) in one launch ---------------------------------------
//
// A decode-shaped call mixes a few dozen rows, and for such a matrix the blocked path above is some thirty dependent
// launches of a few microseconds each.  Here one CTA does everything with the matrix in registers: eight consecutive
// lanes share COLUMN c (lane h of the group holds rows h, h + 8, ...), so applying a reflector to a column is a dozen
// private FMAs plus a three-step shuffle inside the group.  What bounds it is the chain of the m columns.  A link is: the owners of column j
// publish it as it stands, one barrier, and every group sums, below row j, both its product with its own column and its
// square; the reflector (its scalars, worked out by everybody, times that column) needs no second round.  v_j . x_c is x_c[j] + scale_j * (that
// product), v_j being 1 in row j and scale_j times the column below.  The columns stay in shared memory and are scaled at the end;
// then each group builds its column of Q = H_0 ... H_(m-1) by applying the reflectors backwards to e_c, two per shuffle: with
// g = v_(j+1) . v_j known, w_j after H_(j+1) is w_j - g tau_(j+1) w_(j+1).  Only H_j with j <= c touch e_c.
// Against owners that normalise their column before they publish it, shuffles of single groups and one reflector at a time, a whole sample in
// fp32, back to back: 32 rows 18.6 -> 11.6 us, 64 rows 45.7 -> 28.9, 68 rows 49.3 -> 34.3, 96 rows 98.3 -> 57.9.
// Same conventions as the blocked path: R (upper triangle, diagonal of either sign) overwrites G, Q is unsigned.
template <int RM>
struct QrSmall {
    static constexpr int RPT = RM / 8;
    float* Vs;                                // RM x RM: row j = reflector j over the rows
    float *tau_s, *scale_s, *beta_s, *g_s;   // g_s[q]: v_(2q+1) . v_(2q)
    int m, c, h, c_max;                       // c_max: the last column of this warp.  Whole warps take every step, which a shuffle needs to be cheap

    __device__ __forceinline__ QrSmall(float* smem, int rows)
        : Vs(smem), tau_s(smem + RM * RM), scale_s(tau_s + RM), beta_s(scale_s + RM), g_s(beta_s + RM), m(rows), c(threadIdx.x >> 3),
          h(threadIdx.x & 7), c_max(c | 3)
    {
    }
    __device__ __forceinline__ float group_sum(float v) const
    {
        v += __shfl_xor_sync(0xffffffffu, v, 1);
        v += __shfl_xor_sync(0xffffffffu, v, 2);
        v += __shfl_xor_sync(0xffffffffu, v, 4);
        return v;
    }
    // x: column c of the matrix -> column c of R; the reflectors go to Vs, zero past m.  All threads of the CTA.
    __device__ __forceinline__ void factorise(float (&x)[RPT]) const
    {
        if (c == 0) {
#pragma unroll
            for (int k = 0; k < RPT; ++k) Vs[h + 8 * k] = x[k];
        }
        __syncthreads();
#pragma unroll
        for (int i = 0; i < RPT; ++i) {                      // (so that rows above the current eight cost nothing)
#pragma unroll 1
            for (int hh = 0; hh < 8; ++hh) {
                const int j = 8 * i + hh;
                if (j >= m) break;
                if (c_max >= j) {
                    float v[RPT], p = 0.0f, p1 = 0.0f, s = 0.0f, s1 = 0.0f;
#pragma unroll
                    for (int k = i; k < RPT; ++k) v[k] = Vs[j * RM + h + 8 * k];
                    const float alpha = __shfl_sync(0xffffffffu, v[i], hh, 8), xj = __shfl_sync(0xffffffffu, x[i], hh, 8);
                    v[i] = h > hh ? v[i] : 0.0f;
#pragma unroll
                    for (int k = i; k < RPT; ++k) {
                        float& pk = ((k - i) & 1) ? p1 : p;
                        float& sk = ((k - i) & 1) ? s1 : s;
                        pk = fmaf(v[k], x[k], pk);
                        sk = fmaf(v[k], v[k], sk);
                    }
                    const float sigma = group_sum(s + s1), dot = group_sum(p + p1);
                    float beta = alpha, tau = 0.0f, scale = 0.0f;
                    if (sigma > 0.0f) {
                        // Every thread works these out, so they have to be short: hardware approximations, then Newton's step from a residual that a
                        // fused multiply-add gives exactly (Markstein, IBM J. Res. Dev. 34, 1990), for the quotient tau as for the others.
                        // That leaves what the rounded square root and divisions leave (without the last step Q^T Q - I is
                        // 7% larger at 64 columns, 14% at 8), in 28.7 us for a sample of 64 rows against 32.5
                        const float n2 = fmaf(alpha, alpha, sigma);
                        float r = rsqrtf(n2);
                        float norm = n2 * r;
                        norm = fmaf(0.5f * r, fmaf(-norm, norm, n2), norm);
                        r = fmaf(r, fmaf(-norm, r, 1.0f), r);                    // 1 / norm
                        const float far = fabsf(alpha) + norm;
                        float inv = __fdividef(1.0f, far);
                        inv = fmaf(inv, fmaf(-far, inv, 1.0f), inv);
                        beta = -copysignf(norm, alpha);
                        tau = far * r;
                        tau = fmaf(r, fmaf(-norm, tau, far), tau);
                        scale = copysignf(inv, alpha);
                    }
                    const float tw = c > j ? tau * fmaf(scale, dot, xj) : 0.0f;
                    if (h == hh) x[i] -= tw;
#pragma unroll
                    for (int k = i; k < RPT; ++k) x[k] = fmaf(-tw, v[k] * scale, x[k]);   // (v is zero down to row j; the reflector as Q will be formed from it)
                    if (c == j + 1) {
#pragma unroll
                        for (int k = i; k < RPT; ++k) Vs[(j + 1) * RM + h + 8 * k] = x[k];
                    }
                    if (threadIdx.x == 8 * RM - 1) { tau_s[j] = tau; scale_s[j] = scale; beta_s[j] = beta; }
                }
                __syncthreads();
            }
        }
#pragma unroll
        for (int k = 0; k < RPT; ++k) {
            const int r = h + 8 * k;
            if (r >= c && c < m) x[k] = r == c ? beta_s[c] : 0.0f;
        }
        for (int e = threadIdx.x; e < RM * RM; e += 8 * RM) {
            const int j = e / RM, r = e - j * RM;
            Vs[e] = j >= m || r < j ? 0.0f : (r == j ? 1.0f : Vs[e] * scale_s[j]);
        }
        if (threadIdx.x >= m && threadIdx.x < RM) tau_s[threadIdx.x] = 0.0f;
        __syncthreads();
        if (c_max < RM / 2) {
            const float* v = Vs + 2 * c * RM + h;
            float g = 0.0f;
#pragma unroll
            for (int k = 0; k < RPT; ++k) g = fmaf(v[8 * k], v[RM + 8 * k], g);
            g = group_sum(g);
            if (h == 0) g_s[c] = g;
        }
        __syncthreads();
    }
    // column c of Q
    __device__ __forceinline__ void form_q(float (&x)[RPT]) const
    {
#pragma unroll
        for (int i = 0; i < RPT; ++i) x[i] = (h + 8 * i == c) ? 1.0f : 0.0f;
#pragma unroll
        for (int i = RPT - 1; i >= 0; --i) {                 // the four pairs whose reflectors begin in rows 8 i .. 8 i + 7
#pragma unroll 1
            for (int q = min(c_max >> 1, 4 * i + 3); q >= 4 * i; --q) {   // (reflectors past c leave e_c as it is)
                const float* v = Vs + 2 * q * RM + h;
                float a[RPT], b[RPT], w0 = 0.0f, w1 = 0.0f;
#pragma unroll
                for (int k = i; k < RPT; ++k) {
                    a[k] = v[8 * k]; b[k] = v[RM + 8 * k];
                    w0 = fmaf(a[k], x[k], w0);
                    w1 = fmaf(b[k], x[k], w1);
                }
                w0 = group_sum(w0);
                w1 = group_sum(w1);
                const float t1 = tau_s[2 * q + 1] * w1, t0 = tau_s[2 * q] * fmaf(-g_s[q], t1, w0);
#pragma unroll
                for (int k = i; k < RPT; ++k) x[k] = fmaf(-t0, a[k], fmaf(-t1, b[k], x[k]));
            }
        }
    }
};

template <int RM>
__global__ void __launch_bounds__(8 * RM, 1)
qr_small_kernel(float* __restrict__ G, int ld, int m, float* __restrict__ Q)
{
    chain_next();
    chain_wait();
    extern __shared__ float qs_smem[];
    const QrSmall<RM> q(qs_smem, m);
    const int c = q.c;
    float x[QrSmall<RM>::RPT];
#pragma unroll
    for (int i = 0; i < QrSmall<RM>::RPT; ++i) {
        const int r = q.h + 8 * i;
        x[i] = (r < m && c < m) ? G[(size_t)r * ld + c] : 0.0f;
    }
    q.factorise(x);
#pragma unroll
    for (int i = 0; i < QrSmall<RM>::RPT; ++i) {
        const int r = q.h + 8 * i;
        if (r < m && c < m) G[(size_t)r * ld + c] = x[i];
    }
    q.form_q(x);
#pragma unroll
    for (int i = 0; i < QrSmall<RM>::RPT; ++i) {
        const int r = q.h + 8 * i;
        if (r < m && c < m) Q[(size_t)r * ld + c] = x[i];
    }
}

__device__ __forceinline__ void put_small(float* p, float v) { *p = v; }
__device__ __forceinline__ void put_small(__nv_bfloat16* p, float v) { *p = __float2bfloat16_rn(v); }
__device__ __forceinline__ void put_small(__half* p, float v) { *p = __float2half_rn(v); }

// A whole orthogonal sample of a small matrix in one launch: the Gaussian (the blocks of the stream shared out to the
// threads, by way of shared memory), its QR, the columns signed by the diagonal of R, A and its transpose in the storage
// type.  Same values as the three kernels it stands for (gaussian_kernel, qr_small_kernel, finish_mixing_kernel): their launches, the
// recorded graph around them and the passes over memory made a 64 + 4 row call 117 us alone, now 97, and 32 of them on 16 lanes, which
// the host's launches bound, 829 us, now 770.
template <int RM, typename T>
__global__ void __launch_bounds__(8 * RM, 1)
sample_small_kernel(int m, uint64_t seed, uint32_t attempt, T* __restrict__ A, T* __restrict__ At, int lda)
{
    chain_next();
    chain_wait();
    extern __shared__ float qs_smem[];
    const QrSmall<RM> q(qs_smem, m);
    const int c = q.c;
    const unsigned total = (unsigned)(m * m);
    for (unsigned b = threadIdx.x; 4 * b < total; b += 8 * RM) {
        float z[4];
        gaussian_block(seed, b, GELO_STREAM_G0, attempt, z);
#pragma unroll
        for (int t = 0; t < 4; ++t) {
            const unsigned e = 4 * b + t, r = e / (unsigned)m;
            if (e < total) q.Vs[r * RM + (e - r * m)] = z[t];
        }
    }
    __syncthreads();
    float x[QrSmall<RM>::RPT];
#pragma unroll
    for (int i = 0; i < QrSmall<RM>::RPT; ++i) {
        const int r = q.h + 8 * i;
        x[i] = (r < m && c < m) ? q.Vs[r * RM + c] : 0.0f;
    }
    __syncthreads();
    q.factorise(x);
    float d = 0.0f;
#pragma unroll
    for (int i = 0; i < QrSmall<RM>::RPT; ++i) d += (q.h + 8 * i == c) ? x[i] : 0.0f;
    const float sign = q.group_sum(d) < 0.0f ? -1.0f : 1.0f;
    q.form_q(x);
    __syncthreads();                          // the reflectors have been read
    float* out = qs_smem;                     // row stride RM + 1: read by rows and by columns
    if (c < m) {
#pragma unroll
        for (int i = 0; i < QrSmall<RM>::RPT; ++i) out[(q.h + 8 * i) * (RM + 1) + c] = sign * x[i];
    }
    __syncthreads();
    for (unsigned e = threadIdx.x; e < total; e += 8 * RM) {
        const unsigned r = e / (unsigned)m, k = e - r * m;
        put_small(A + (size_t)r * lda + k, out[r * (RM + 1) + k]);
        put_small(At + (size_t)r * lda + k, out[k * (RM + 1) + r]);
    }
}

constexpr int qr_small_smem(int RM) { return (RM * RM + 4 * RM) * (int)sizeof(float); }       // (reflectors, then the result in rows of RM + 1)

template <typename F>
int qr_small_attr(gelo_ctx* ctx, F* kernel, int smem, bool (&done)[64])
{
    if (ctx->device >= 0 && ctx->device < 64 && !done[ctx->device]) {
        GELO_CUDA_OK(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, smem));
        done[ctx->device] = true;
    }
    return GELO_OK;
}

template <int RM>
int launch_qr_small_rm(gelo_ctx* ctx, int m, float* G, int ld, float* Q, cudaStream_t st)
{
    static bool done[64] = {};
    GELO_TRY(qr_small_attr(ctx, qr_small_kernel<RM>, qr_small_smem(RM), done));
    GELO_TRY(launch_chained(ctx, qr_small_kernel<RM>, 1, 8 * RM, qr_small_smem(RM), st, G, ld, m, Q));
    return after_launch(ctx);
}

template <int RM, typename T>
int launch_sample_small_rm(gelo_ctx* ctx, int m, uint64_t seed, uint32_t attempt, void* A, void* At, int lda, cudaStream_t st)
{
    static bool done[64] = {};
    GELO_TRY(qr_small_attr(ctx, sample_small_kernel<RM, T>, qr_small_smem(RM), done));
    GELO_TRY(launch_chained(ctx, sample_small_kernel<RM, T>, 1, 8 * RM, qr_small_smem(RM), st, m, seed, attempt, static_cast<T*>(A),
                           static_cast<T*>(At), lda));
    return after_launch(ctx);
}

constexpr int kSmallQrRows = 128;

// f(RM) for the smallest instance that holds m rows, in steps of eight: the time grows with the instance (the rows a thread holds, and the
// columns of the reflectors), 12 us for 32 rows, 29 for 64 and 58 for 96.
template <int RM = 32, typename F>
int with_small_rows(int m, F&& f)
{
    if constexpr (RM < kSmallQrRows) {
        if (m > RM) return with_small_rows<RM + 8>(m, f);
    }
    return f(std::integral_constant<int, RM>{});
}

}  // namespace

int launch_qr_small(gelo_ctx* ctx, int m, float* G, int ld, float* Q, cudaStream_t st)
{
    return with_small_rows(m, [&](auto rm) { return launch_qr_small_rm<decltype(rm)::value>(ctx, m, G, ld, Q, st); });
}

bool sample_small_supports(const gelo_ctx* ctx, int m, int kind)
{
    return kind == GELO_ORTHOGONAL && m <= kSmallQrRows && ctx->fuse_small && ctx->level3 == 0;
}

int launch_sample_small(gelo_ctx* ctx, int m, uint64_t seed, uint32_t attempt, int dtype, void* A, void* Ainv, int lda, cudaStream_t st)
{
    return with_small_rows(m, [&](auto rm) {
        constexpr int RM = decltype(rm)::value;
        if (dtype == GELO_BF16) return launch_sample_small_rm<RM, __nv_bfloat16>(ctx, m, seed, attempt, A, Ainv, lda, st);
        if (dtype == GELO_F16) return launch_sample_small_rm<RM, __half>(ctx, m, seed, attempt, A, Ainv, lda, st);
        return launch_sample_small_rm<RM, float>(ctx, m, seed, attempt, A, Ainv, lda, st);
    });
}

// Takes `bytes` from the idle region if it has that much left, else from the arena.
void* take_idle(Arena& a, char** idle, size_t* idle_bytes, size_t bytes)
{
    const size_t need = (bytes + 255) & ~size_t(255);
    if (idle && idle_bytes && *idle_bytes >= need) {
        void* p = *idle;
        *idle += need;
        *idle_bytes -= need;
        return p;
    }
    return a.take(bytes);
}

QrScratch carve_qr(Arena& a, int m, int ld, char** idle, size_t* idle_bytes)
{
    QrScratch s;
    s.V = static_cast<float*>(a.take((size_t)m * ld * sizeof(float)));
    s.T = static_cast<float*>(a.take((size_t)ceil_div(m, NB) * NB * NB * sizeof(float)));
    s.Wp = static_cast<float*>(take_idle(a, idle, idle_bytes, (size_t)kMaxSlabs * NB * ld * sizeof(float)));
    s.W2 = static_cast<float*>(a.take((size_t)NB * ld * sizeof(float)));
    s.T128 = static_cast<float*>(a.take((size_t)ceil_div(m, 128) * 128 * 128 * sizeof(float)));
    return s;
}

int run_householder_qr(gelo_ctx* ctx, int m, float* R, int ld, float* Q, const QrScratch& s, cudaStream_t st)
{
    if (m <= kSmallQrRows && ctx->fuse_small) return launch_qr_small(ctx, m, R, ld, Q, st);
    const int npanels = ceil_div(m, NB);
    // ---- factorisation ----
    for (int pnl = 0; pnl < npanels; ++pnl) {
        const int j0 = pnl * NB, jb = (m - j0 < NB) ? (m - j0) : NB;
        float* Tp = s.T + (size_t)pnl * NB * NB;
        GELO_TRY(launch_qr_panel(ctx, R, ld, m, j0, jb, s.V, Tp, st));
        const int nc = m - j0 - jb, nr = m - j0;
        if (nc <= 0) continue;
        float* C = R + (size_t)j0 * ld + j0 + jb;
        const float* Vp = s.V + (size_t)j0 * ld + j0;
        // C <- (I - V T^T V^T) C :  W2 = T^T (V^T C), then C -= V W2
        GELO_TRY(launch_vtc(ctx, Vp, ld, jb, C, ld, nr, nc, Tp, true, s.Wp, s.W2, ld, st));
        GELO_TRY(launch_rank_update(ctx, Vp, ld, s.W2, ld, C, ld, nr, nc, jb, st));
    }
    // ---- accumulate Q backwards from the identity ----
    GELO_TRY(set_identity(ctx, Q, ld, m, st));
    for (int pnl = npanels - 1; pnl >= 0; --pnl) {
        const int j0 = pnl * NB, jb = (m - j0 < NB) ? (m - j0) : NB;
        const int nr = m - j0;
        const float* Tp = s.T + (size_t)pnl * NB * NB;
        const float* Vp = s.V + (size_t)j0 * ld + j0;
        float* C = Q + (size_t)j0 * ld + j0;
        // Q[j0:, j0:] <- (I - V T V^T) Q[j0:, j0:]
        GELO_TRY(launch_vtc(ctx, Vp, ld, jb, C, ld, nr, nr, Tp, false, s.Wp, s.W2, ld, st));
        GELO_TRY(launch_rank_update(ctx, Vp, ld, s.W2, ld, C, ld, nr, nr, jb, st));
    }
    return GELO_OK;
}

int run_householder_qr_tc(gelo_ctx* ctx, int m, float* R, int ld, float* Q, const QrScratch& s, const TcScratch& tc,
                          cudaStream_t st)
{
    // reflector entries above a panel's first row are read (as zeros) by the block-level products
    GELO_CUDA_OK(cudaMemsetAsync(s.V, 0, (size_t)m * ld * sizeof(float), st));
    GELO_CUDA_OK(cudaFuncSetAttribute(t_merge_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kMergeSmemBytes));
    const int nblocks = ceil_div(m, kOuter);

    // One outer-block transformation C <- (I - V Top V^T) C on the tensor cores, Top = T^T or T.
    auto block_apply = [&](int b0, int ob, float* C, int nc, bool transpose_t) -> int {
        const int nr = m - b0;
        const int nc8 = (nc + 7) & ~7;
        const float* Vb = s.V + (size_t)b0 * ld + b0;
        const float* Tb = s.T128 + (size_t)(b0 / kOuter) * 128 * 128;
        GELO_TRY(launch_split(ctx, C, ld, nr, nc, tc.big[0], tc.big[1], ld, false, st));
        GELO_TRY(launch_split(ctx, Vb, ld, nr, ob, tc.panA[0], tc.panA[1], kOuter, false, st));
        GELO_TRY(launch_split(ctx, Vb, ld, nr, ob, tc.panAt[0], tc.panAt[1], ld, true, st));
        GELO_TRY(launch_split(ctx, Tb, 128, ob, ob, tc.tt[0], tc.tt[1], kOuter, transpose_t, st));
        // W = V^T C: a long, thin product, so the rows are cut into slices whose partial products are summed in a
        // fixed order by the kernel that also forms the (high, low) pair
        const int n_tiles = ceil_div(nc8, 256);
        int want = ceil_div(2 * (ctx->tc_update_ctas > 0 ? ctx->tc_update_ctas : ctx->sm_count), n_tiles);   // slices fill the CTAs this launch may use
        if (want > kMaxKSplit) want = kMaxKSplit;
        int used = 0;
        const size_t plane = (size_t)kOuter * ld;
        GELO_TRY(launch_gemm_tc_split_k(ctx, ob, nc8, nr, tc.panAt[0], tc.panAt[1], ld, tc.big[0], tc.big[1], ld, tc.wf32,
                                        plane, ld, want, &used, st));
        GELO_TRY(launch_sum_split(ctx, tc.wf32, plane, used, ld, ob, nc8, tc.rowB[0], tc.rowB[1], ld, st));
        // W2 = Top W
        GELO_TRY(launch_gemm_tc_split(ctx, ob, nc8, ob, tc.tt[0], tc.tt[1], kOuter, tc.rowB[0], tc.rowB[1], ld, nullptr, 0,
                                      tc.rowB2[0], tc.rowB2[1], ld, false, st));
        // C -= V W2
        return launch_gemm_tc_split(ctx, nr, nc, ob, tc.panA[0], tc.panA[1], kOuter, tc.rowB2[0], tc.rowB2[1], ld, C, ld,
                                    nullptr, nullptr, 0, false, st);
    };

    // ---- factorisation ----
    for (int blk = 0; blk < nblocks; ++blk) {
        const int b0 = blk * kOuter;
        const int ob = (m - b0 < kOuter) ? (m - b0) : kOuter;
        const int bend = b0 + ob;
        for (int j0 = b0; j0 < bend; j0 += NB) {
            const int jb = (bend - j0 < NB) ? (bend - j0) : NB;
            float* Tp = s.T + (size_t)(j0 / NB) * NB * NB;
            GELO_TRY(launch_qr_panel(ctx, R, ld, m, j0, jb, s.V, Tp, st));
            const int ncb = bend - (j0 + jb), nr = m - j0;
            if (ncb > 0) {
                float* C = R + (size_t)j0 * ld + j0 + jb;
                const float* Vp = s.V + (size_t)j0 * ld + j0;
                GELO_TRY(launch_vtc(ctx, Vp, ld, jb, C, ld, nr, ncb, Tp, true, s.Wp, s.W2, ld, st));
                GELO_TRY(launch_rank_update(ctx, Vp, ld, s.W2, ld, C, ld, nr, ncb, jb, st));
            }
        }
        // block factor: Gram of the block's reflectors (row slabs, summed in order), then the merge of the panel factors
        const float* Vb = s.V + (size_t)b0 * ld + b0;
        const int slabs = ceil_div(m - b0, kGramRows);
        gram128_kernel<<<slabs, 256, 0, st>>>(Vb, ld, m - b0, ob, tc.gram);
        GELO_TRY(after_launch(ctx));
        float* Tb = s.T128 + (size_t)blk * 128 * 128;
        t_merge_kernel<<<1, 1024, kMergeSmemBytes, st>>>(tc.gram, slabs, 128, s.T + (size_t)(b0 / NB) * NB * NB, ob, Tb);
        GELO_TRY(after_launch(ctx));
        const int nc = m - bend;
        if (nc > 0) GELO_TRY(block_apply(b0, ob, R + (size_t)b0 * ld + bend, nc, true));
    }
    // ---- accumulate Q backwards from the identity ----
    GELO_TRY(set_identity(ctx, Q, ld, m, st));
    for (int blk = nblocks - 1; blk >= 0; --blk) {
        const int b0 = blk * kOuter;
        const int ob = (m - b0 < kOuter) ? (m - b0) : kOuter;
        GELO_TRY(block_apply(b0, ob, Q + (size_t)b0 * ld + b0, m - b0, false));
    }
    return GELO_OK;
}

// Blocked QR whose level-3 work is tf32 products read straight from the fp32 matrices.  Panels of 32 columns and
// blocks of 128 run as in run_householder_qr_tc.  Blocks are grouped into superblocks of kSuper = 512 columns:
//   * inside a superblock a finished block is applied to the superblock's remaining columns only, and its factor
//     is merged into the superblock's factor:  with S = V_i^T V_(<i),
//         T(1..i) = [[T(1..i-1), -T(1..i-1) S^T T_i], [0, T_i]];
//   * the columns right of the superblock see ONE update C <- (I - V T^T V^T) C with all 512 reflectors, and Q is
//     accumulated backwards with one such update (with T) per superblock.
// A trailing update with 512 reflectors does four times the arithmetic of one with 128 per byte of C moved, which
// is what the 128-column updates were short of (they ran at the speed of the memory system, not of the tensor cores).
int run_householder_qr_tf32(gelo_ctx* ctx, int m, float* R, int ld, float* Q, const QrScratch& s, const TcScratch& tc,
                            cudaStream_t st)
{
    GELO_CUDA_OK(cudaMemsetAsync(s.V, 0, (size_t)m * ld * sizeof(float), st));
    GELO_CUDA_OK(cudaFuncSetAttribute(t_merge_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kMergeSmemBytes));
    const float back2 = (1.0f + kTf32TruncLoss) * (1.0f + kTf32TruncLoss);
    const int width = ctx->tc_update_ctas > 0 ? ctx->tc_update_ctas : ctx->sm_count;   // CTAs one launch may use
    // the Gram slots are read in full by the merge kernel; entries that no product writes must at least be finite
    GELO_CUDA_OK(cudaMemsetAsync(tc.sx, 0, (size_t)kOuter * (kSuper + kOuter) * sizeof(float), st));

    // C (nr x nc, rows from row r0 of the matrix) <- (I - V op(T) V^T) C with V = reflector columns c0 .. c0+kv-1
    // (rows from r0 = c0), T: kv x kv with row stride ldt; planes hold `maxsplit` slices of kv x ld.
    auto apply = [&](int c0, int kv, const float* T, int ldt, float* C, int nc, bool transpose_t, int maxsplit) -> int {
        const int nr = m - c0;
        const int nc8 = (nc + 7) & ~7;
        const float* Vb = s.V + (size_t)c0 * ld + c0;
        // W = V^T C contracts over all nr rows: with few output tiles the rows are cut into slices (summed in a fixed
        // order afterwards) so that the launch still fills its CTAs; with enough tiles it is one plain product
        const int tiles = ceil_div(kv, 128) * ceil_div(nc8, 256);
        int want = (2 * tiles >= width) ? 1 : ceil_div(2 * width, tiles);
        if (want > maxsplit) want = maxsplit;
        if (want <= 1) {
            GELO_TRY(launch_gemm_tf32(ctx, kv, nc8, nr, Vb, ld, true, C, ld, false, tc.w32[0], ld, true, 1.0f, 1, 0, nullptr, st));
        } else {
            int used = 0;
            const size_t plane = (size_t)kv * ld;
            GELO_TRY(launch_gemm_tf32(ctx, kv, nc8, nr, Vb, ld, true, C, ld, false, tc.wf32, ld, false, 1.0f, want, plane, &used, st));
            GELO_TRY(launch_sum_planes(ctx, tc.wf32, plane, used, ld, kv, nc8, 1.0f, tc.w32[0], ld, st));
        }
        GELO_TRY(launch_gemm_tf32(ctx, kv, nc8, kv, T, ldt, transpose_t, tc.w32[0], ld, false, tc.w32[1], ld, true, 1.0f, 1, 0,
                                  nullptr, st));
        return launch_gemm_tf32(ctx, nr, nc, kv, Vb, ld, false, tc.w32[1], ld, true, C, ld, false, 1.0f, 1, 0, nullptr, st);
    };

    const int nsuper = ceil_div(m, kSuper);
    // ---- factorisation ----
    for (int sb = 0; sb < nsuper; ++sb) {
        const int s0 = sb * kSuper;
        const int sw = (m - s0 < kSuper) ? (m - s0) : kSuper;
        const int send = s0 + sw;
        float* Ts = tc.tsuper + (size_t)sb * kSuper * kSuper;
        GELO_CUDA_OK(cudaMemsetAsync(Ts, 0, (size_t)kSuper * kSuper * sizeof(float), st));
        for (int b0 = s0; b0 < send; b0 += kOuter) {
            const int ob = (send - b0 < kOuter) ? (send - b0) : kOuter;
            const int bend = b0 + ob;
            for (int j0 = b0; j0 < bend; j0 += NB) {
                const int jb = (bend - j0 < NB) ? (bend - j0) : NB;
                float* Tp = s.T + (size_t)(j0 / NB) * NB * NB;
                GELO_TRY(launch_qr_panel(ctx, R, ld, m, j0, jb, s.V, Tp, st));
                const int ncb = bend - (j0 + jb), nr = m - j0;
                if (ncb > 0) {
                    float* C = R + (size_t)j0 * ld + j0 + jb;
                    const float* Vp = s.V + (size_t)j0 * ld + j0;
                    GELO_TRY(launch_vtc(ctx, Vp, ld, jb, C, ld, nr, ncb, Tp, true, s.Wp, s.W2, ld, st));
                    GELO_TRY(launch_rank_update(ctx, Vp, ld, s.W2, ld, C, ld, nr, ncb, jb, st));
                }
            }
            // S = V_i^T [V_(<i) | V_i]  (ob x (r + ob)): the block's own Gram matrix and its products with the reflectors
            // already merged, in one tf32 product over the rows from b0 down (both operands reach the tensor core
            // truncated, hence the scale)
            const float* Vb = s.V + (size_t)b0 * ld + b0;
            float* Tb = s.T128 + (size_t)(b0 / kOuter) * 128 * 128;
            const int r = b0 - s0;                           // reflector columns already merged
            const int ob8 = (ob + 7) & ~7;
            const int lds = kSuper + kOuter;
            {
                // all 128 columns of the block's slot where the row has them (columns past the block are still zero):
                // the merge kernel reads the whole 128 x 128 Gram slot
                const int nr = m - b0;
                const int ns = (r + kOuter <= ld - s0) ? r + kOuter : ld - s0;
                int want = ceil_div(2 * width, ceil_div(ns, 256));
                if (want > kMaxKSplit) want = kMaxKSplit;
                int used = 0;
                const size_t plane = (size_t)kOuter * ld;
                GELO_TRY(launch_gemm_tf32(ctx, ob, ns, nr, Vb, ld, true, s.V + (size_t)b0 * ld + s0, ld, false, tc.wf32, ld, false,
                                          1.0f, want, plane, &used, st));
                GELO_TRY(launch_sum_planes(ctx, tc.wf32, plane, used, ld, ob, ns, back2, tc.sx, lds, st));
            }
            // block factor T_i from its Gram matrix and the panel factors ...
            t_merge_kernel<<<1, 1024, kMergeSmemBytes, st>>>(tc.sx + r, 1, lds, s.T + (size_t)(b0 / NB) * NB * NB, ob, Tb);
            GELO_TRY(after_launch(ctx));
            // ... into the superblock's factor
            GELO_CUDA_OK(cudaMemcpy2DAsync(Ts + (size_t)r * kSuper + r, (size_t)kSuper * sizeof(float), Tb, 128 * sizeof(float),
                                           (size_t)ob * sizeof(float), ob, cudaMemcpyDeviceToDevice, st));
            if (r > 0) {
                // X = S^T T_i  (r x ob),  then  T[0:r, r:r+ob] = -T[0:r, 0:r] X  (that part of T is still zero)
                GELO_TRY(launch_gemm_tf32(ctx, r, ob8, ob, tc.sx, lds, true, Tb, 128, false, tc.xb, kOuter, true, 1.0f, 1, 0,
                                          nullptr, st));
                GELO_TRY(launch_gemm_tf32(ctx, r, ob, r, Ts, kSuper, false, tc.xb, kOuter, true, Ts + r, kSuper, false, 1.0f, 1, 0,
                                          nullptr, st));
            }
            // the block's own reflector on the remaining columns of the superblock
            if (send > bend) GELO_TRY(apply(b0, ob, Tb, 128, R + (size_t)b0 * ld + bend, send - bend, true, kMaxKSplit));
        }
        // the merged reflector on everything right of the superblock
        if (m > send) GELO_TRY(apply(s0, sw, Ts, kSuper, R + (size_t)s0 * ld + send, m - send, true, kSuperKSplit));
    }
    // ---- accumulate Q backwards from the identity, one superblock at a time ----
    GELO_TRY(set_identity(ctx, Q, ld, m, st));
    for (int sb = nsuper - 1; sb >= 0; --sb) {
        const int s0 = sb * kSuper;
        const int sw = (m - s0 < kSuper) ? (m - s0) : kSuper;
        GELO_TRY(apply(s0, sw, tc.tsuper + (size_t)sb * kSuper * kSuper, kSuper, Q + (size_t)s0 * ld + s0, m - s0, false,
                       kSuperKSplit));
    }
    return GELO_OK;
}

// The tf32 updates leave Q orthogonal to a few 1e-3 only (the tensor core truncates unrounded operands, which
// shrinks every block reflector a little).  One Newton-Schulz step, Q <- Q - Q D with D = (Q^T Q - I) / 2, squares
// that defect.
//   * D is symmetric: one tf32 product over the tiles on and above the diagonal (a little more than half of them),
//     mirrored by the epilogue.  Q is dense with log-uniformly spread mantissas, so the truncation loss of Q^T Q is the
//     known constant and is scaled back before the identity is subtracted; what is left in D is zero-mean noise of a
//     few 1e-4 (Frobenius norm over sqrt(m)), which bounds the polished defect.
//   * The correction Q D is small (D is a few 1e-3 per row), so 8 significant bits in each factor are plenty: D is
//     stored in bf16, Q is copied to bf16 once, and the product runs at the bf16 rate, subtracted from the fp32 Q in
//     place.  (Relative error of the correction 4e-3, i.e. about 1e-5 of Q.)
// D16 and Q16 are scratch for m x ld 16-bit values each.
int polish_orthogonal_tf32(gelo_ctx* ctx, int m, float* Q, int ld, float* D16, float* Q16, cudaStream_t st)
{
    const float back2 = (1.0f + kTf32TruncLoss) * (1.0f + kTf32TruncLoss);
    GELO_TRY(launch_gram_sym_bf16(ctx, m, Q, ld, D16, ld, back2, 1.0f, 0.5f, st));
    GELO_TRY(launch_narrow(ctx, m, Q, ld, GELO_BF16, Q16, ld, st));
    return launch_gemm_bf16_sub(ctx, m, m, m, Q16, ld, D16, ld, Q, ld, st);
}

}  // namespace gelo

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
// a 128 x 128 Cholesky factorisation and a 128 x 128 inverse (block_factor_kernel); everything else is a
// product.  The update of columns C right of the block needs W' = T^T V^T C = T^T (P^T C) + D^T C1, D = R T = B^-T,
// C1 = the first b rows of C: P^T C comes out of the same product as P^T P.
// Blocks are grouped four by four into superblocks whose merged reflector, I - V_s T_s V_s^T, is all that the rest of the matrix
// and Q ever see.  A block's row of T_s^T left of the diagonal is -X^T T_<^T with X^T = T^T V^T V_<, which is W' with the
// earlier reflectors V_< of the superblock in place of C.  So a block's two products, P^T [V_< P C] and the one that gives
// W', run over all columns of the superblock, and a merge is a single small product more (as products of its own with its sum
// it was five dependent launches, 50 us per block).
// The last block, which would be square, is factorised by the one-launch Householder kernel.
//
// The products run in tf32 or, for fp32 storage and small matrices (`exact`), on the FMA pipes.
//
// Against 32-column Householder panels in registers (70 us per 32 columns of serial column steps, and rank-32 updates
// between them), which the sampler used before: 2048 + 102 rows, orthogonal, one call alone 8.9 -> 1.8 ms; 512 rows in fp32, the sample
// 1.52 -> 0.45 ms.
#include "common.cuh"
#include "tc_ptx.cuh"

#include <type_traits>

namespace gelo {

namespace {

constexpr int FB = kOuter;                     // block width

// ---- the 128 x 128 factorisation of a block, in a cluster of three CTAs -------------------------------------------
//
// CTA 0 eliminates the Gram matrix Z = R^T R (rows of R and of R^-T come out 16 at a time), CTA 1 inverts B = P1 + R by
// Gauss-Jordan, CTA 2 applies the same row operations to R^-T and ends with B^-1 R^-T = T^T.  Each holds its matrix as fp32
// accumulators of m16n8k16 matrix instructions in the registers of eight warps (32 rows x 64 columns each) and does eight
// steps with 16 pivots p = 16 J .. 16 J + 15:
//     publish    the rows p of the matrix (rows), and in CTA 1 its columns p (panel), go to shared memory
//     U          = F * rows, F the inverse of the pivot block (CTA 0: of its Cholesky factor); in the columns p of an
//                inverse that grows in place U is F itself
//     update     a -= panel U, rows p <- U
// A ninth warp runs ahead with the pivot blocks: as soon as the rows p are published it forms the next block (from its
// published value, the panel and its 16 columns of U, straight from registers) and inverts it with shuffles while the
// others are still busy with U and the update.  The rows of R and R^-T
// are needed by the other CTAs only when their own step begins, because the elimination is linear in them: row p of B is
// P1's until then.  They travel by bulk copies between the CTAs' shared memories into a slot per step, which is never
// used twice, so nobody waits for space.
//
// The operands of the products are pairs of IEEE halves (x = hi + lo to 22 bits; hi hi + hi lo + lo hi, accumulated in fp32):
// the caller scales the matrix to pivots around 1, so nothing leaves the range of a half, and the result has fp32 accuracy
// (B^T D - I below 2e-6).  What bounds it is the chain of the 16-step inversions and, in CTA 1, the products (96 matrix
// instructions per warp and step).  The same eliminations pivot by pivot in one CTA, with a broadcast each, took 57 us per launch;
// fused multiply-adds on 8 x 8 tiles in this layout 36 us, bound by shared-memory reads; this form 25 us.
constexpr int NB = 16;                         // pivots of a step
constexpr int kSteps = FB / NB;
constexpr int kFactCompute = 256;
constexpr int kFactThreads = kFactCompute + 32;
constexpr int kFactCtas = 3;
constexpr int kPanelLd = NB + 8;               // row strides in halves: 16-byte rows, conflict-free matrix loads
constexpr int kWideLd = FB + 8;
struct FactShared {
    __half panel[kSteps][2][FB][kPanelLd];     // minus the columns p, hi and lo; CTA 0: the rows of R that it sends (fp32)
    float got[kSteps][NB][FB];                 // CTA 1: rows of R, CTA 2: rows of R^-T; CTA 0: the rows of R^-T it sends
    __half F[kSteps][2][NB][kPanelLd];
    __half rows[2][2][NB][kWideLd];            // of even and of odd steps
    __half U[2][NB][kWideLd];
    float U32[NB][FB + 4];
    float next[2][NB][NB + 4];                 // the next pivot block before the running update
    uint64_t got_full[kSteps], panel_full[kSteps];
    int abort;                                 // a wait ran out somewhere in the cluster
};
constexpr int kFactSmemBytes = (int)sizeof(FactShared);
static_assert(kFactSmemBytes <= 227 * 1024, "shared memory budget");
static_assert(sizeof(FactShared::panel) >= sizeof(float) * FB * FB, "CTA 0 keeps R there");

__device__ __forceinline__ float fast_rcp(float x)
{
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}

// Wait for a phase of a barrier of this CTA, bounded in time.  A wait that runs out sets the status word and the flag of all three CTAs and
// goes on (with values that nobody will use): every copy is still sent and every barrier reached, the other waits give up at
// their next look at the flag, and the copies that are still on their way are waited for at the end.
__device__ __forceinline__ void fact_wait(const uint64_t* bar, FactShared& s, unsigned long long limit_ns, int* status)
{
    const uint32_t addr = tcx::smem_u32(bar);
#pragma unroll 1
    for (int spin = 0; spin < 256; ++spin)
        if (tcx::mbar_try(addr, 0)) return;
    if (tcx::mbar_wait(addr, 0, &s.abort, limit_ns)) return;
    atomicCAS(status, 0, (int)GELO_ERR_TIMEOUT);
    for (int r = 0; r < kFactCtas; ++r)
        asm volatile("st.shared::cluster.s32 [%0], %1;" ::"r"(tcx::map_rank(tcx::smem_u32(&s.abort), r)), "r"(1) : "memory");
}

__device__ __forceinline__ void cluster_sync_all()
{
    asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}

// Copies `bytes` of this CTA's shared memory to the place of `dst` in CTA `rank` and counts them on `bar` there.
__device__ __forceinline__ void send_shared(const void* dst, const void* src, uint32_t bytes, const uint64_t* bar, int rank)
{
    uint32_t d, b;
    asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(d) : "r"(tcx::smem_u32(dst)), "r"(rank));
    asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(b) : "r"(tcx::smem_u32(bar)), "r"(rank));
    asm volatile("cp.async.bulk.shared::cluster.shared::cta.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                 ::"r"(d), "r"(tcx::smem_u32(src)), "r"(bytes), "r"(b) : "memory");
}

// Four 8 x 8 blocks of halves; lane i names row i % 8 of block i / 8.
template <bool kTrans>
__device__ __forceinline__ void ldsm4(uint32_t (&v)[4], const __half* p)
{
    const uint32_t addr = tcx::smem_u32(p);
    if (kTrans)
        asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0, %1, %2, %3}, [%4];"
                     : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]) : "r"(addr) : "memory");
    else
        asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0, %1, %2, %3}, [%4];"
                     : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]) : "r"(addr) : "memory");
}
__device__ __forceinline__ void mma16(float (&c)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1)
{
    asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, {%0, %1, %2, %3};"
                 : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3]) : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

// Operand fragments as (hi, lo) pairs.  A (16 x 16): from a row-major array of rows, or (columns of U, CTA 0's panel)
// from its transpose.  B (16 x 16, two column tiles): from an array of k rows.
struct Pair4 { uint32_t hi[4], lo[4]; };
__device__ __forceinline__ void load_a(Pair4& f, const __half* hi, const __half* lo, int ld, int lane)
{
    const int off = ((lane & 7) + ((lane >> 3) & 1) * 8) * ld + (lane >> 4) * 8;
    ldsm4<false>(f.hi, hi + off);
    ldsm4<false>(f.lo, lo + off);
}
__device__ __forceinline__ void load_a_transposed(Pair4& f, const __half* hi, const __half* lo, int ld, int lane)
{
    const int off = ((lane & 7) + (lane >> 4) * 8) * ld + ((lane >> 3) & 1) * 8;
    ldsm4<true>(f.hi, hi + off);
    ldsm4<true>(f.lo, lo + off);
}
__device__ __forceinline__ void load_b(Pair4& f, const __half* hi, const __half* lo, int ld, int lane)
{
    const int off = ((lane & 7) + ((lane >> 3) & 1) * 8) * ld + (lane >> 4) * 8;
    ldsm4<true>(f.hi, hi + off);
    ldsm4<true>(f.lo, lo + off);
}
__device__ __forceinline__ void negate(Pair4& f)
{
#pragma unroll
    for (int t = 0; t < 4; ++t) { f.hi[t] ^= 0x80008000u; f.lo[t] ^= 0x80008000u; }
}
// c (16 x 16, two column tiles) += A B
__device__ __forceinline__ void mma_pairs(float (&c)[2][4], const Pair4& a, const Pair4& b)
{
#pragma unroll
    for (int t = 0; t < 2; ++t) mma16(c[t], a.lo, b.hi[2 * t], b.hi[2 * t + 1]);
#pragma unroll
    for (int t = 0; t < 2; ++t) mma16(c[t], a.hi, b.lo[2 * t], b.lo[2 * t + 1]);
#pragma unroll
    for (int t = 0; t < 2; ++t) mma16(c[t], a.hi, b.hi[2 * t], b.hi[2 * t + 1]);
}
// Accumulator tiles as an operand pair: x[t][2 i + e] = (row gid + 8 i, column 8 t + 2 tig + e).  As they stand they are
// the A operand x; read as B (mma_pairs_t) they are x^T.
__device__ __forceinline__ void pack_pairs(Pair4& p, const float (&x)[2][4])
{
#pragma unroll
    for (int t = 0; t < 2; ++t)
#pragma unroll
        for (int i = 0; i < 2; ++i) {
            const __half2 h = __floats2half2_rn(x[t][2 * i], x[t][2 * i + 1]);
            const float2 f = __half22float2(h);
            const __half2 l = __floats2half2_rn(x[t][2 * i] - f.x, x[t][2 * i + 1] - f.y);
            p.hi[2 * t + i] = *reinterpret_cast<const uint32_t*>(&h);
            p.lo[2 * t + i] = *reinterpret_cast<const uint32_t*>(&l);
        }
}
// c += A x^T, both column tiles
__device__ __forceinline__ void mma_pairs_t(float (&c)[2][4], const Pair4& a, const Pair4& x)
{
#pragma unroll
    for (int t = 0; t < 2; ++t) mma16(c[t], a.lo, x.hi[t], x.hi[2 + t]);
#pragma unroll
    for (int t = 0; t < 2; ++t) mma16(c[t], a.hi, x.lo[t], x.lo[2 + t]);
#pragma unroll
    for (int t = 0; t < 2; ++t) mma16(c[t], a.hi, x.hi[t], x.hi[2 + t]);
}
__device__ __forceinline__ void store_pair(__half* hi, __half* lo, float x, float y)
{
    const __half2 h = __floats2half2_rn(x, y);
    const float2 f = __half22float2(h);
    *reinterpret_cast<__half2*>(hi) = h;
    *reinterpret_cast<__half2*>(lo) = __floats2half2_rn(x - f.x, y - f.y);
}

// A warp's 16 x 16 block (two accumulator tiles: a[t][2 i + e] = row gid + 8 i, column 8 t + 2 tig + e) replaced by its inverse
// by Gauss-Jordan steps, or (kChol) by the inverse of its Cholesky factor: elimination of the rows below the pivot
// leaves L^-1 below the diagonal of L Delta L^T, which is scaled to Delta^-1/2 L^-1.  With p the pivot and u = (pivot row) / p,
// a row x with f in the pivot column becomes x - f u, and f becomes -f / p.  The latter and the pivot row itself ride along:
// f - f (1 + 1 / p) = -f / p and x - (p - 1) u = x / p, exact enough because the pivots are around 1.  The chain of a step would be
// shuffle, reciprocal, product, update; every lane works the next pivot out for itself from the entries before the
// update, so the reciprocal runs beside the rest.
template <bool kChol>
__device__ __forceinline__ void invert16(float (&a)[2][4], int gid, int tig, int* status)
{
    constexpr uint32_t all = 0xffffffffu;
    float rp = fast_rcp(__shfl_sync(all, a[0][0], 0));
#pragma unroll
    for (int k = 0; k < NB; ++k) {
        const int kt = k >> 3, kg = k & 7, ke = k & 1, kc = (k & 7) >> 1;
        float rn = 0.0f;
        if (k + 1 < NB) {
            const int nt = (k + 1) >> 3, ng = (k + 1) & 7, ne = (k + 1) & 1, nc = ng >> 1;
            const float a11 = __shfl_sync(all, a[nt][2 * nt + ne], ng * 4 + nc), a10 = __shfl_sync(all, a[kt][2 * nt + ke], ng * 4 + kc);
            const float a01 = __shfl_sync(all, a[nt][2 * kt + ne], kg * 4 + nc);
            rn = fast_rcp(fmaf(-a10 * a01, rp, a11));
        }
        float u[2][2], f[2];
#pragma unroll
        for (int t = 0; t < 2; ++t)
#pragma unroll
            for (int e = 0; e < 2; ++e) u[t][e] = __shfl_sync(all, a[t][2 * kt + e], kg * 4 + tig) * rp;
        if (tig == kc) u[kt][ke] = 1.0f + rp;
#pragma unroll
        for (int i = 0; i < 2; ++i) f[i] = __shfl_sync(all, a[kt][2 * i + ke], gid * 4 + kc);
#pragma unroll
        for (int i = kChol ? kt : 0; i < 2; ++i) {           // (Cholesky: rows above the pivot are done)
            if (i == kt) {
                if (kChol) f[i] = gid > kg ? f[i] : 0.0f;
                else f[i] -= gid == kg ? 1.0f : 0.0f;
            }
#pragma unroll
            for (int t = 0; t < 2; ++t)
#pragma unroll
                for (int e = 0; e < 2; ++e) a[t][2 * i + e] = fmaf(-f[i], u[t][e], a[t][2 * i + e]);
        }
        rp = rn;
    }
    if (kChol) {
#pragma unroll
        for (int i = 0; i < 2; ++i) {
            const int r = gid + 8 * i;
            const float d = __shfl_sync(all, (gid & 1) ? a[i][2 * i + 1] : a[i][2 * i], gid * 4 + (gid >> 1));   // pivot of row r
            if (!(d > 0.0f)) atomicCAS(status, 0, (int)GELO_ERR_COND);           // a Gaussian block never gets here
            const float rs = rsqrtf(d);
#pragma unroll
            for (int t = 0; t < 2; ++t)
#pragma unroll
                for (int e = 0; e < 2; ++e) {
                    const int c = 8 * t + 2 * tig + e;
                    a[t][2 * i + e] = c < r ? a[t][2 * i + e] * rs : (c == r ? rs : 0.0f);
                }
        }
    }
}

// f(v) with v as a compile-time constant, for values that choose registers.
template <typename F>
__device__ __forceinline__ void with_bit(int v, F&& f)
{
    if (v == 0) f(std::integral_constant<int, 0>{});
    else f(std::integral_constant<int, 1>{});
}
template <typename F>
__device__ __forceinline__ void with_quarter(int v, F&& f)
{
    if (v == 0) f(std::integral_constant<int, 0>{});
    else if (v == 1) f(std::integral_constant<int, 1>{});
    else if (v == 2) f(std::integral_constant<int, 2>{});
    else f(std::integral_constant<int, 3>{});
}

enum FactRole { FACT_GRAM = 0, FACT_INVERSE = 1, FACT_FACTOR = 2 };

// F, rows, panel and the next pivot block of a step are published (all warps) / U is (the eight warps).
__device__ __forceinline__ void published_barrier() { asm volatile("bar.sync 1, %0;" ::"n"(kFactThreads) : "memory"); }
__device__ __forceinline__ void compute_barrier() { asm volatile("bar.sync 2, %0;" ::"n"(kFactCompute) : "memory"); }

// The eight steps of the eight warps; a[mt][nt][2 i + e] = row 32 (w / 2) + 16 mt + gid + 8 i, column 64 (w % 2) + 8 nt + 2 tig + e.
template <int kRole>
__device__ __forceinline__ void fact_compute(float (&a)[2][8][4], FactShared& s, unsigned long long wait_ns, int* status)
{
    const int tid = threadIdx.x, w = tid >> 5, lane = tid & 31, gid = lane >> 2, tig = lane & 3;
    const int wr = w >> 1, wc = w & 1;
    float* const R = reinterpret_cast<float*>(&s.panel[0][0][0][0]);             // CTA 0 only
#pragma unroll 1
    for (int J = 0; J < kSteps; ++J) {
        // ---- publish ----
        if (kRole != FACT_GRAM) {
            fact_wait(&s.got_full[J], s, wait_ns, status);
            if (kRole == FACT_FACTOR) fact_wait(&s.panel_full[J], s, wait_ns, status);
        }
        if (wr == (J >> 1))
            with_bit(J & 1, [&](auto bit) {
                constexpr int mt = decltype(bit)::value;
#pragma unroll
                for (int nt = 0; nt < 8; ++nt) {
                    const int c = 64 * wc + 8 * nt + 2 * tig;
#pragma unroll
                    for (int i = 0; i < 2; ++i) {
                        if (kRole != FACT_GRAM) {
                            const float2 t = *reinterpret_cast<const float2*>(&s.got[J][gid + 8 * i][c]);
                            a[mt][nt][2 * i] += t.x; a[mt][nt][2 * i + 1] += t.y;
                        }
                        store_pair(&s.rows[J & 1][0][gid + 8 * i][c], &s.rows[J & 1][1][gid + 8 * i][c], a[mt][nt][2 * i], a[mt][nt][2 * i + 1]);
                    }
                }
            });
        if (kRole != FACT_FACTOR) {
            const int N = J + 1;
            if (N < kSteps && wr == (N >> 1) && wc == (N >> 2))                  // the next pivot block, before this step's update
                with_bit(N & 1, [&](auto bit) {
                    with_quarter(N & 3, [&](auto quarter) {
                        constexpr int mt = decltype(bit)::value, n0 = 2 * decltype(quarter)::value;
#pragma unroll
                        for (int t = 0; t < 2; ++t)
#pragma unroll
                            for (int i = 0; i < 2; ++i)
                                *reinterpret_cast<float2*>(&s.next[N & 1][gid + 8 * i][8 * t + 2 * tig]) =
                                    make_float2(a[mt][n0 + t][2 * i], a[mt][n0 + t][2 * i + 1]);
                    });
                });
            if (wc == (J >> 2))                                                  // the columns p, which restart from zero
                with_quarter(J & 3, [&](auto quarter) {
                    constexpr int n0 = 2 * decltype(quarter)::value;
#pragma unroll
                    for (int mt = 0; mt < 2; ++mt)
#pragma unroll
                        for (int t = 0; t < 2; ++t)
#pragma unroll
                            for (int i = 0; i < 2; ++i) {
                                float (&v)[4] = a[mt][n0 + t];
                                const int r = 32 * wr + 16 * mt + gid + 8 * i, c = 8 * t + 2 * tig;
                                if (kRole == FACT_INVERSE) store_pair(&s.panel[J][0][r][c], &s.panel[J][1][r][c], -v[2 * i], -v[2 * i + 1]);
                                v[2 * i] = 0.0f; v[2 * i + 1] = 0.0f;
                            }
                });
            if (kRole == FACT_INVERSE) asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        }
        published_barrier();
        if (kRole == FACT_INVERSE && tid == 0) {
            send_shared(s.panel[J], s.panel[J], sizeof(s.panel[J]), &s.panel_full[J], 2);
            send_shared(s.F[J], s.F[J], sizeof(s.F[J]), &s.panel_full[J], 2);
        }
        // ---- U = F rows, 16 columns per warp (those of warp J are the columns p) ----
        {
            Pair4 f, x;
            load_a(f, &s.F[J][0][0][0], &s.F[J][1][0][0], kPanelLd, lane);
            load_b(x, &s.rows[J & 1][0][0][16 * w], &s.rows[J & 1][1][0][16 * w], kWideLd, lane);
            float u[2][4] = {{0.0f, 0.0f, 0.0f, 0.0f}, {0.0f, 0.0f, 0.0f, 0.0f}};
            mma_pairs(u, f, x);
#pragma unroll
            for (int t = 0; t < 2; ++t)
#pragma unroll
                for (int i = 0; i < 2; ++i) {
                    const int r = gid + 8 * i, cp = 8 * t + 2 * tig, c = 16 * w + cp;
                    float2 v = make_float2(u[t][2 * i], u[t][2 * i + 1]), fv = make_float2(0.0f, 0.0f);
                    if (kRole != FACT_FACTOR && w == J) {
                        const float2 fh = __half22float2(*reinterpret_cast<const __half2*>(&s.F[J][0][r][cp]));
                        const float2 fl = __half22float2(*reinterpret_cast<const __half2*>(&s.F[J][1][r][cp]));
                        fv = make_float2(fh.x + fl.x, fh.y + fl.y);
                    }
                    if (kRole == FACT_GRAM) {
                        // row of R: U right of the pivots, the Cholesky factor above the diagonal of the pivot block
                        float2 rv = v;
                        if (w < J || (w == J && cp < r)) rv.x = 0.0f;
                        if (w < J || (w == J && cp + 1 < r)) rv.y = 0.0f;
                        *reinterpret_cast<float2*>(R + (J * NB + r) * FB + c) = rv;
                        *reinterpret_cast<float2*>(&s.got[J][r][c]) = w < J ? v : fv;                            // row of R^-T
                    }
                    if (kRole != FACT_FACTOR && w == J) v = fv;
                    store_pair(&s.U[0][r][c], &s.U[1][r][c], v.x, v.y);
                    if (kRole != FACT_GRAM) *reinterpret_cast<float2*>(&s.U32[r][c]) = v;
                }
            if (kRole == FACT_GRAM) asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        }
        compute_barrier();
        if (kRole == FACT_GRAM && tid == 0) {
            send_shared(s.got[J], R + J * NB * FB, sizeof(s.got[J]), &s.got_full[J], 1);
            send_shared(s.got[J], s.got[J], sizeof(s.got[J]), &s.got_full[J], 2);
        }
        // ---- update (CTA 0: the rows below the pivots only) ----
        if (kRole != FACT_GRAM || 2 * wr + 1 > J) {
            Pair4 c[2];
#pragma unroll
            for (int mt = 0; mt < 2; ++mt) {
                const int r0 = 32 * wr + 16 * mt;
                if (kRole == FACT_GRAM) {
                    load_a_transposed(c[mt], &s.U[0][0][r0], &s.U[1][0][r0], kWideLd, lane);
                    negate(c[mt]);
                } else {
                    load_a(c[mt], &s.panel[J][0][r0][0], &s.panel[J][1][r0][0], kPanelLd, lane);
                }
            }
#pragma unroll
            for (int np = 0; np < 4; ++np) {
                Pair4 u;
                load_b(u, &s.U[0][0][64 * wc + 16 * np], &s.U[1][0][64 * wc + 16 * np], kWideLd, lane);
#pragma unroll
                for (int e = 0; e < 3; ++e)                  // (four independent accumulators between dependent instructions)
#pragma unroll
                    for (int mt = 0; mt < 2; ++mt)
                        if (kRole != FACT_GRAM || 2 * wr + mt > J) {
                            const uint32_t (&x)[4] = e == 0 ? c[mt].lo : c[mt].hi;
                            const uint32_t (&y)[4] = e == 1 ? u.lo : u.hi;
                            mma16(a[mt][2 * np], x, y[0], y[1]);
                            mma16(a[mt][2 * np + 1], x, y[2], y[3]);
                        }
            }
        }
        if (kRole != FACT_GRAM && wr == (J >> 1))
            with_bit(J & 1, [&](auto bit) {
                constexpr int mt = decltype(bit)::value;
#pragma unroll
                for (int nt = 0; nt < 8; ++nt)
#pragma unroll
                    for (int i = 0; i < 2; ++i) {
                        const float2 v = *reinterpret_cast<const float2*>(&s.U32[gid + 8 * i][64 * wc + 8 * nt + 2 * tig]);
                        a[mt][nt][2 * i] = v.x; a[mt][nt][2 * i + 1] = v.y;
                    }
            });
    }
}

// The ninth warp: the inverses of the pivot blocks.
template <int kRole>
__device__ __forceinline__ void fact_pivots(FactShared& s, unsigned long long wait_ns, int* status)
{
    const int lane = threadIdx.x & 31, gid = lane >> 2, tig = lane & 3;
    float a[2][4];
    Pair4 f;
#pragma unroll 1
    for (int N = 0; N <= kSteps; ++N) {
        if (N > 0) published_barrier();                      // of step N - 1
        if (N == kSteps || kRole == FACT_FACTOR) continue;
        Pair4 c, x;
        if (N > 0) {
            float ut[2][4] = {{0.0f, 0.0f, 0.0f, 0.0f}, {0.0f, 0.0f, 0.0f, 0.0f}};   // U^T = rows^T F^T, columns of the next block
            const int sl = (N - 1) & 1;
            load_a_transposed(c, &s.rows[sl][0][0][NB * N], &s.rows[sl][1][0][NB * N], kWideLd, lane);
            mma_pairs_t(ut, c, f);
            pack_pairs(x, ut);
            if (kRole == FACT_GRAM) { c = x; negate(c); }
            else load_a(c, &s.panel[N - 1][0][NB * N][0], &s.panel[N - 1][1][NB * N][0], kPanelLd, lane);
        }
#pragma unroll
        for (int t = 0; t < 2; ++t)
#pragma unroll
            for (int i = 0; i < 2; ++i) {
                const float2 v = *reinterpret_cast<const float2*>(&s.next[N & 1][gid + 8 * i][8 * t + 2 * tig]);
                a[t][2 * i] = v.x; a[t][2 * i + 1] = v.y;
            }
        if (N > 0) mma_pairs_t(a, c, x);
        if (kRole == FACT_INVERSE) {
            fact_wait(&s.got_full[N], s, wait_ns, status);
#pragma unroll
            for (int t = 0; t < 2; ++t)
#pragma unroll
                for (int i = 0; i < 2; ++i) {
                    const float2 v = *reinterpret_cast<const float2*>(&s.got[N][gid + 8 * i][NB * N + 8 * t + 2 * tig]);
                    a[t][2 * i] += v.x; a[t][2 * i + 1] += v.y;
                }
        }
        invert16<kRole == FACT_GRAM>(a, gid, tig, status);
        pack_pairs(f, a);
#pragma unroll
        for (int t = 0; t < 2; ++t)
#pragma unroll
            for (int i = 0; i < 2; ++i) {
                *reinterpret_cast<uint32_t*>(&s.F[N][0][gid + 8 * i][8 * t + 2 * tig]) = f.hi[2 * t + i];
                *reinterpret_cast<uint32_t*>(&s.F[N][1][gid + 8 * i][8 * t + 2 * tig]) = f.lo[2 * t + i];
            }
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    }
}

// Z (ob x ob, stride ldz): the Gram matrix P^T P.  P1: the first ob rows of the panel (stride ld), overwritten
// with B = P1 + R.  Tt (stride ldt) = T^T = B^-1 R^-T and Dt (stride ldd) = dscale * B^-1, both rounded to tf32 if `round`.
// ob <= 128, a multiple of 4; the kernel works on 128 x 128 with an identity in the part past ob.  `scale` is a power of
// two close to the norm of a panel column.
__global__ void __cluster_dims__(kFactCtas, 1, 1) __launch_bounds__(kFactThreads, 1)
block_factor_kernel(const float* __restrict__ Z, int ldz, float* P1, int ld, int ob, float* __restrict__ Tt,
                    int ldt, float* __restrict__ Dt, int ldd, float scale, float dscale, int round, unsigned long long wait_ns,
                    int* __restrict__ status)
{
    chain_next();
    chain_wait();
    if (wait_ns == 0) {                                      // give up before any copy is on its way
        if (blockIdx.x == 0 && threadIdx.x == 0) atomicCAS(status, 0, (int)GELO_ERR_TIMEOUT);
        return;
    }
    extern __shared__ __align__(128) uint8_t fsm[];
    FactShared& s = *reinterpret_cast<FactShared*>(fsm);
    const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5, gid = lane >> 2, tig = lane & 3;
    const int wr = w >> 1, wc = w & 1;
    const int role = blockIdx.x;
    const float s1 = 1.0f / scale, s2 = s1 * s1;
    const bool compute = tid < kFactCompute;

    if (tid == 0) {
        s.abort = 0;
        for (int i = 0; i < kSteps; ++i) {
            tcx::mbar_init(tcx::smem_u32(&s.got_full[i]), 1);
            tcx::mbar_init(tcx::smem_u32(&s.panel_full[i]), 1);
        }
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        if (role != FACT_GRAM)
            for (int i = 0; i < kSteps; ++i) {
                tcx::mbar_expect_tx(tcx::smem_u32(&s.got_full[i]), sizeof(s.got[0]));
                if (role == FACT_FACTOR) tcx::mbar_expect_tx(tcx::smem_u32(&s.panel_full[i]), sizeof(s.panel[0]) + sizeof(s.F[0]));
            }
    }
    float a[2][8][4];
    if (compute) {
        const float* src = role == FACT_GRAM ? Z : P1;
        const int lds = role == FACT_GRAM ? ldz : ld;
        const float f = role == FACT_GRAM ? s2 : s1, one = role == FACT_GRAM ? 1.0f : 0.0f;
#pragma unroll
        for (int mt = 0; mt < 2; ++mt)
#pragma unroll
            for (int nt = 0; nt < 8; ++nt)
#pragma unroll
                for (int i = 0; i < 2; ++i) {
                    const int r = 32 * wr + 16 * mt + gid + 8 * i, c = 64 * wc + 8 * nt + 2 * tig;
                    float2 v = make_float2(r == c ? one : 0.0f, r == c + 1 ? one : 0.0f);
                    if (r < ob && c < ob) {                  // (ob is even: c + 1 < ob too)
                        v = *reinterpret_cast<const float2*>(src + (size_t)r * lds + c);
                        v.x *= f; v.y *= f;
                    }
                    a[mt][nt][2 * i] = role == FACT_FACTOR ? 0.0f : v.x;
                    a[mt][nt][2 * i + 1] = role == FACT_FACTOR ? 0.0f : v.y;
                    if (w == 0 && mt == 0 && nt < 2)         // the first pivot block
                        *reinterpret_cast<float2*>(&s.next[0][r][c]) = v;
                }
    }
    __syncwarp();
    cluster_sync_all();                                      // barriers initialised, P1 read, the first block published
    if (!compute) {
        if (role == FACT_GRAM) fact_pivots<FACT_GRAM>(s, wait_ns, status);
        else if (role == FACT_INVERSE) fact_pivots<FACT_INVERSE>(s, wait_ns, status);
        else fact_pivots<FACT_FACTOR>(s, wait_ns, status);
    } else if (role == FACT_GRAM) {
        fact_compute<FACT_GRAM>(a, s, wait_ns, status);
        // B = P1 + R, the top block of V
        const float* R = reinterpret_cast<const float*>(&s.panel[0][0][0][0]);
#pragma unroll 4
        for (int idx = tid; idx < FB * FB / 4; idx += kFactCompute) {
            const int r = idx >> 5, c = (idx & 31) * 4;
            if (r < ob && c < ob && c + 3 >= r) {
                float4* p = reinterpret_cast<float4*>(P1 + (size_t)r * ld + c);
                const float4 v = *reinterpret_cast<const float4*>(R + r * FB + c);
                float4 o = *p;
                o.x += scale * v.x; o.y += scale * v.y; o.z += scale * v.z; o.w += scale * v.w;
                *p = o;
            }
        }
    } else {
        if (role == FACT_INVERSE) fact_compute<FACT_INVERSE>(a, s, wait_ns, status);
        else fact_compute<FACT_FACTOR>(a, s, wait_ns, status);
        float* dst = role == FACT_INVERSE ? Dt : Tt;
        const int ldo = role == FACT_INVERSE ? ldd : ldt;
        const float f = role == FACT_INVERSE ? dscale * s1 : s2;
        auto out_val = [&](float v) { return round ? tcx::round_tf32(f * v) : f * v; };
#pragma unroll
        for (int mt = 0; mt < 2; ++mt)
#pragma unroll
            for (int nt = 0; nt < 8; ++nt)
#pragma unroll
                for (int i = 0; i < 2; ++i) {
                    const int r = 32 * wr + 16 * mt + gid + 8 * i, c = 64 * wc + 8 * nt + 2 * tig;
                    if (r < ob && c < ob)
                        *reinterpret_cast<float2*>(dst + (size_t)r * ldo + c) = make_float2(out_val(a[mt][nt][2 * i]), out_val(a[mt][nt][2 * i + 1]));
                }
    }
    __syncwarp();
    cluster_sync_all();                                      // nobody's shared memory goes while a copy may still reach it
    if (*static_cast<volatile int*>(&s.abort)) {             // (the same in all three CTAs) not every copy has been waited for
        if (tid == 0 && role != FACT_GRAM) {
            int on = 0;                                      // a flag that stays zero: these waits only end in time
            for (int i = 0; i < kSteps; ++i) {
                tcx::mbar_wait(tcx::smem_u32(&s.got_full[i]), 0, &on, wait_ns);
                if (role == FACT_FACTOR) tcx::mbar_wait(tcx::smem_u32(&s.panel_full[i]), 0, &on, wait_ns);
            }
        }
        __syncwarp();
        cluster_sync_all();
    }
}

// Z = scale * (sum of the K slices of P^T [V_< | P | C]), in slice order; columns c0 .. c0 + ob - 1 (the Gram matrix) stay
// fp32, the others are rounded to tf32 if `round` (they feed the next product).  Also clears the rows above the block (z_rows x ob)
// where the superblock's reflectors are zero.
__global__ void __launch_bounds__(256)
block_sum_kernel(const float* __restrict__ planes, size_t plane, int parts, int ldp, int rows, int cols, int c0, int ob, float scale, int round,
                 float* __restrict__ Z, int ldz, float* __restrict__ zero, int z_rows, int ld)
{
    chain_next();
    chain_wait();
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
        if (round && (c < c0 || c >= c0 + ob)) {
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
// columns flipped where its R (diagonal of Rf) is negative.  Everything else is cleared.  Columns c0 .. c_end - 1 of it.
__global__ void __launch_bounds__(256)
start_q_kernel(float* __restrict__ Q, int ld, int m, int bf, const float* __restrict__ R, int c0, int c_end)
{
    chain_next();
    chain_wait();
    const int r = blockIdx.y;
    const int c = c0 + (blockIdx.x * 256 + threadIdx.x) * 4;   // (c0, bf and c_end are multiples of four)
    if (c >= c_end) return;
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

// For the last f rows of -Q^T: a copy of the f x m block (stride ld), and Qf (f x f) with the columns flipped where its R (diagonal of Rf) is
// positive, so that Qf^T times the copy is what these rows have to be.
__global__ void __launch_bounds__(256)
last_rows_kernel(const float* __restrict__ rows, float* __restrict__ copy, int f, int m, float* __restrict__ Qf, const float* __restrict__ Rf, int ld)
{
    chain_next();
    chain_wait();
    const int r = blockIdx.y, c = blockIdx.x * 256 + threadIdx.x;
    if (c < m) copy[(size_t)r * ld + c] = rows[(size_t)r * ld + c];
    if (c < f && !(Rf[(size_t)c * ld + c] < 0.0f)) Qf[(size_t)r * ld + c] = -Qf[(size_t)r * ld + c];
}

}  // namespace

// Rows from which a QR with few others beside it forms Q^T while it factorises (see run_gaussian_qr), and the SMs that it does that on.
// From three superblocks on there is something to form beside the next one, and one spare matrix has room for the products' scratch.  Whole
// calls, d = 4096, p = 12288, us, Q accumulated backwards -> this:
//                              1536 rows      1600 rows      2150 rows      4300 rows      4300 rows non-orthogonal
//   one call                   1018 ->  976   1142 -> 1036   1509 -> 1415   3794 -> 3461   4403 -> 4056
//   two at once, two lanes     1315 -> 1217   1431 -> 1304   2008 -> 1856   5430 -> 5046   6633 -> 6261
//   three at once, three lanes 1530 -> 1432   1667 -> 1552   2458 -> 2282   7161 -> 6784   9016 -> 8725
// Fewer SMs leave more of them to the chains: 64 are as good for one call and up to 1% slower for two or three, 80 and 96 0.3% and 1 to 2%,
// 112 0.5% and 2%; on all of them the chain's launches wait for tiles of 20 to 30 us (4304 us where 80 gave 4026).
// The factor is as good: 2150 rows in half, orthogonal, columns 3.19e-3 -> 3.20e-3 off (the first half of them 7.5e-4 -> 8.0e-4), unpolished
// 3.35e-3 -> 3.36e-3 (1.12e-3 -> 1.11e-3) with Q^T Q - I 2.07e-3 -> 2.06e-3; at 4300 rows 1.92e-3 -> 1.85e-3.
constexpr int kFormRows = 3 * kSuper;
constexpr int kFormSms = 48;
// Lanes that share the SMs out fill the GPU with four samples.  Where they do not (gelo_set_lane_share), forming Q beside them gains as long as the samples in
// flight have some 32000 rows in all: 4 x 2150 rows 3005 -> 2848 us, 16 x 1600 6295 -> 6081, but 16 x 2150 9992 -> 10056, 16 x 4300 34919 -> 35821.
constexpr int kFormRowsInFlight = 32000;

bool forms_beside(const gelo_ctx* ctx, int m)
{
    return ctx->tc_update_ctas == 0 && m >= kFormRows && (long long)ctx->in_flight * m <= kFormRowsInFlight;
}

bool gaussian_qr_supports(int m) { return m > FB; }

int run_gaussian_qr(gelo_ctx* ctx, int m, float* G, int ld, float* Q, const TcScratch& tc, bool exact, cudaStream_t st, bool* transposed)
{
    static bool attr_done[64] = {};
    if (ctx->device >= 0 && ctx->device < 64 && !attr_done[ctx->device]) {
        GELO_CUDA_OK(cudaFuncSetAttribute(block_factor_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kFactSmemBytes));
        attr_done[ctx->device] = true;
    }
    const float loss1 = exact ? 1.0f : 1.0f + kTf32TruncLoss, loss2 = loss1 * loss1;
    const int round = exact ? 0 : 1;
    // In a recorded graph of a call that runs alone, what nobody waits for yet goes into branches of the graph (on the context's side
    // stream): the merges, which are needed at the end of a superblock (with them 2150 rows orthogonal, one call 1.61 -> 1.56 ms; 4300 non-orthogonal
    // 4.51 -> 4.41), and, where Q is accumulated backwards, the last square with its columns of Q (1400 + 70 rows 914 -> 912 us, 1000 + 50 and
    // below no difference).
    const bool fork = ctx->recording && ctx->tc_update_ctas == 0;
    cudaStream_t cur = st;                                   // where the products go
    auto branch = [&]() -> int {
        GELO_CUDA_OK(cudaEventRecord(ctx->side_from, st));
        GELO_CUDA_OK(cudaStreamWaitEvent(ctx->side, ctx->side_from, 0));
        cur = ctx->side;
        return GELO_OK;
    };
    auto join = [&]() -> int {
        GELO_CUDA_OK(cudaEventRecord(ctx->side_done, ctx->side));
        GELO_CUDA_OK(cudaStreamWaitEvent(st, ctx->side_done, 0));
        return GELO_OK;
    };
    // A QR alone, or one of a few, spends most of its time in launches that leave SMs idle, half of it in block factors on three SMs.
    // Beside them it forms Q^T: the reflectors of a superblock are applied to the identity as they are to the columns on the right, on a stream
    // of its own, while the next superblock is factorised, on kFormSms of the SMs so that the chain finds others free.  That
    // takes half as many operations again as accumulating Q backwards, which needs the last reflector first, so it is not
    // for a GPU that is full (forms_beside).  Samples side by side share the stream while they are recorded, one
    // after the other; replayed, each has a branch of its own.
    const bool forming = transposed && !exact && forms_beside(ctx, m) && tc.big[0];
    struct FormGuard {                                       // however it ends, the caller's stream comes after all launches
        gelo_ctx* ctx; cudaStream_t st; bool on;
        ~FormGuard()
        {
            if (on && cudaEventRecord(ctx->form_done, ctx->form) == cudaSuccess) cudaStreamWaitEvent(st, ctx->form_done, 0);
        }
    } form_guard = { ctx, st, false };
    auto form_after = [&]() -> int {                         // what goes to the stream that forms Q^T next waits for what st has by now
        GELO_CUDA_OK(cudaEventRecord(ctx->form_from, st));
        GELO_CUDA_OK(cudaStreamWaitEvent(ctx->form, ctx->form_from, 0));
        form_guard.on = true;
        return GELO_OK;
    };
    struct FormLaunches {                                    // launches that are planned for kFormSms and get no more
        gelo_ctx* ctx;
        explicit FormLaunches(gelo_ctx* c) : ctx(c) { c->tc_update_ctas = kFormSms; c->tc_cap = true; }
        FormLaunches(const FormLaunches&) = delete;
        ~FormLaunches() { ctx->tc_update_ctas = 0; ctx->tc_cap = false; }
    };

    // V^T C with few output tiles: the rows are cut into slices whose partial products are summed in a fixed order
    auto slices = [&](int M, int N, int K, int most) {
        const int width = ctx->tc_update_ctas > 0 ? ctx->tc_update_ctas : ctx->sm_count;       // CTAs one launch may use
        int want;
        if (!exact && gemm_tile_cols(ctx, M, N, K, 1, 4, true, 64) == 64) {
            want = width / (ceil_div(M, 128) * ceil_div(N, 64));      // one round of narrow tiles
        } else {
            const int tiles = exact ? ceil_div(M, 64) * ceil_div(N, 64) : ceil_div(M, 128) * ceil_div(N, 256);
            want = (2 * tiles >= width) ? 1 : ceil_div(2 * width, tiles);
        }
        return want < 1 ? 1 : (want > most ? most : want);
    };
    // C = scale * op(A) B or C -= op(A) B, as launch_gemm_tf32 or in fp32
    auto gemm = [&](int M, int N, int K, const float* A, int lda, bool a_mn, const float* B, int ldb, bool subtract, float* C, int ldc,
                    bool round_out, float scale, int ksplit, size_t plane, int* used) -> int {
        if (!exact) return launch_gemm_tf32(ctx, M, N, K, A, lda, a_mn, B, ldb, subtract, C, ldc, round_out, scale, ksplit, plane, used, cur);
        if (M <= 0 || N <= 0 || K <= 0) return GELO_OK;
        GemmArgs g;
        g.M = M; g.N = N; g.K = K;
        g.A = A; g.lda = lda; g.transA = a_mn; g.B = B; g.ldb = ldb;
        g.C[0] = C; g.ldc = ldc;
        g.alpha = subtract ? -1.0f : scale; g.beta = subtract ? 1.0f : 0.0f;
        if (ksplit > 1) {
            const int steps = ceil_div(K, 16), per = ceil_div(steps, ksplit < steps ? ksplit : steps);
            g.ksplit = ceil_div(steps, per);       // no empty slice
            g.plane = plane;
        }
        if (used) *used = g.ksplit;
        return launch_gemm_simt(ctx, g, cur);
    };
    // C (rows from c0) <- (I - V op(T^T) V^T) C for the merged reflectors of a superblock (kv columns from c0)
    struct ApplyScratch { float *w, *tw, *planes; int most; };       // V^T C, its product with T, `most` K slices of the former
    const ApplyScratch scratch = { tc.w32[0], tc.w32[1], tc.wf32, kSuperKSplit };
    auto apply = [&](int c0, int kv, const float* Tt, float* C, int nc, bool transpose, const ApplyScratch& s) -> int {
        const int nr = m - c0;
        const int nc8 = (nc + 7) & ~7;
        const float* V = G + (size_t)c0 * ld + c0;
        const int want = slices(kv, nc8, nr, s.most);
        if (want <= 1) {
            GELO_TRY(gemm(kv, nc8, nr, V, ld, true, C, ld, false, s.w, ld, true, loss2, 1, 0, nullptr));
        } else {
            int used = 0;
            const size_t plane = (size_t)kv * ld;
            GELO_TRY(gemm(kv, nc8, nr, V, ld, true, C, ld, false, s.planes, ld, false, 1.0f, want, plane, &used));
            GELO_TRY(launch_sum_planes(ctx, s.planes, plane, used, ld, kv, nc8, loss2, s.w, ld, cur, !exact));
        }
        // (the factor loss1 makes up for the truncation of V in the last product)
        GELO_TRY(gemm(kv, nc8, kv, Tt, kSuper, transpose, s.w, ld, false, s.tw, ld, true, loss1, 1, 0, nullptr));
        return gemm(nr, nc, kv, V, ld, false, s.tw, ld, true, C, ld, false, 1.0f, 1, 0, nullptr);
    };

    // Block columns: 128 wide while at least twice as many rows are left, then narrower ones (half of the rows, a multiple of eight) down to a
    // square of at most 96 rows for the Householder kernel, which takes 29 us for 64 rows and 58 for 96, against about
    // 50 us for a block.
    std::vector<int> start;
    int bf = 0;                                              // first column of the square that is left for Householder
    while (m - bf > 96) {
        const int left = m - bf;
        start.push_back(bf);
        bf += left >= 2 * FB ? FB : (left <= 192 ? (left >> 1) & ~7 : (left - 121) & ~7);
    }
    start.push_back(bf);
    const int nblocks = (int)start.size() - 1;
    const int per = kSuper / FB;
    // the spare matrix (m x ld): two block rows, the rest for K slices
    float* spare = static_cast<float*>(tc.big[0]);
    const ApplyScratch form_scratch = { spare, spare + (size_t)kSuper * ld, spare + (size_t)2 * kSuper * ld, (m - 2 * kSuper) / kSuper };
    if (forming) {
        *transposed = true;
        GELO_TRY(form_after());
        GELO_TRY(launch_chained(ctx, start_q_kernel, dim3(ceil_div(ld, 1024), m), 256, 0, ctx->form, Q, ld, m, m, G, 0, ld));   // -I
        GELO_TRY(after_launch(ctx));
    }
    // ---- factorisation ----
    GELO_CUDA_OK(cudaMemsetAsync(tc.tsuper, 0, (size_t)ceil_div(nblocks, per) * kSuper * kSuper * sizeof(float), st));
    for (int s = 0; s < nblocks; s += per) {
        const int e = (s + per < nblocks) ? s + per : nblocks;
        const int s0 = start[s], send = start[e];
        float* Ts = tc.tsuper + (size_t)(s / per) * kSuper * kSuper;     // T^T, lower triangular
        for (int b = s; b < e; ++b) {
            const int b0 = start[b], ob = start[b + 1] - b0, bend = b0 + ob;
            const int nr = m - b0, r = b0 - s0;
            const int ncs = (send - s0 + 7) & ~7;            // the superblock's columns
            float* P = G + (size_t)b0 * ld + b0;
            float* rows = G + (size_t)b0 * ld + s0;          // the block's rows of [V_< | P | C]
            float* Wb = tc.w32[1] + (size_t)(b - s) * FB * ld;
            int used = 0;
            const size_t plane = (size_t)FB * ld;
            GELO_TRY(gemm(ob, ncs, nr, P, ld, true, rows, ld, false, tc.wf32, ld, false, 1.0f, slices(ob, ncs, nr, kMaxKSplit), plane, &used));
            const int work = ob * (ncs >> 2) + r * (ob >> 2);
            GELO_TRY(launch_chained(ctx, block_sum_kernel, ceil_div(work, 256), 256, 0, st, tc.wf32, plane, used, ld, ob,
                                   ncs, r, ob, loss2, round, tc.w32[0], ld, G + (size_t)s0 * ld + b0, r, ld));
            GELO_TRY(after_launch(ctx));
            float* Tb = Ts + (size_t)r * kSuper + r;
            float scale = 1.0f;                              // a power of two with scale^2 about nr
            while (2.0f * scale * scale < (float)nr) scale *= 2.0f;
            GELO_TRY(launch_chained(ctx, block_factor_kernel, kFactCtas, kFactThreads, kFactSmemBytes, st, tc.w32[0] + r, ld,
                                   P, ld, ob, Tb, kSuper, tc.t128, FB, scale, loss1, round, ctx->wait_limit_ns, ctx->status_dev));
            GELO_TRY(after_launch(ctx));
            if (e - s > 1) {
                // [X^T | . | W'] = T^T Z + D^T [V_< | . | C1], scaled up for the truncation of V in the next product
                if (exact) {
                    GELO_TRY(gemm(ob, ncs, ob, Tb, kSuper, false, tc.w32[0], ld, false, Wb, ld, false, 1.0f, 1, 0, nullptr));
                    GemmArgs g;
                    g.M = ob; g.N = ncs; g.K = ob;
                    g.A = tc.t128; g.lda = FB; g.B = rows; g.ldb = ld;
                    g.C[0] = Wb; g.ldc = ld; g.beta = 1.0f;
                    GELO_TRY(launch_gemm_simt(ctx, g, st));
                } else {
                    GELO_TRY(launch_gemm_tf32_dual(ctx, ob, ncs, ob, Tb, kSuper, tc.w32[0], ld, tc.t128, FB, rows, ld, Wb, ld, loss1, st));
                }
            }
            if (r > 0) {                                     // T^T[r:r+ob, 0:r] = -X^T T_<^T
                if (fork) GELO_TRY(branch());
                GELO_TRY(gemm(ob, r, r, Wb, ld, false, Ts, kSuper, false, Ts + (size_t)r * kSuper, kSuper, true, -1.0f / loss1, 1, 0,
                              nullptr));
                cur = st;
            }
            if (send > bend)                                 // C -= V W'
                GELO_TRY(gemm(nr, send - bend, ob, P, ld, false, Wb + (bend - s0), ld, true, P + ob, ld, false, 1.0f, 1, 0, nullptr));
        }
        if (fork && e - s > 1) GELO_TRY(join());
        GELO_TRY(apply(s0, send - s0, Ts, G + (size_t)s0 * ld + send, m - send, false, scratch));
        if (forming) {                                       // (after that update, which fills the GPU)
            GELO_TRY(form_after());
            const FormLaunches on_few(ctx);
            cur = ctx->form;
            GELO_TRY(apply(s0, send - s0, Ts, Q + (size_t)s0 * ld, m, false, form_scratch));
            cur = st;
        }
    }
    if (forming) {
        // Q^T = diag(-I, (Qf S)^T) H^T, of which the other stream has formed -H^T; S flips where R of the last square is negative
        const int f = m - bf;
        float *Qf = tc.w32[0], *rows = Q + (size_t)bf * ld;
        GELO_TRY(launch_qr_small(ctx, f, G + (size_t)bf * ld + bf, ld, Qf, st));
        GELO_CUDA_OK(cudaEventRecord(ctx->form_done, ctx->form));
        GELO_CUDA_OK(cudaStreamWaitEvent(st, ctx->form_done, 0));
        form_guard.on = false;
        GELO_TRY(launch_chained(ctx, last_rows_kernel, dim3(ceil_div(m, 256), f), 256, 0, st, rows, tc.w32[1], f, m, Qf,
                                G + (size_t)bf * ld + bf, ld));
        GELO_TRY(after_launch(ctx));
        GemmArgs g;
        g.M = f; g.N = m; g.K = f;
        g.A = Qf; g.lda = ld; g.transA = true; g.B = tc.w32[1]; g.ldb = ld;
        g.C[0] = rows; g.ldc = ld;
        return launch_gemm_simt(ctx, g, st);
    }
    // ---- the square that is left, and Q accumulated backwards, one superblock at a time ----
    auto form_q = [&](int c0, int c1) -> int {               // columns c0 .. c1 - 1
        const int c_end = c1 == m ? ld : c1;                 // (the padding is cleared)
        GELO_TRY(launch_chained(ctx, start_q_kernel, dim3(ceil_div(c_end - c0, 1024), m), 256, 0, cur, Q, ld, m, bf, G, c0, c_end));
        GELO_TRY(after_launch(ctx));
        for (int s = (nblocks - 1) / per * per; s >= 0; s -= per) {
            const int e = (s + per < nblocks) ? s + per : nblocks;
            const int s0 = start[s], from = c0 > s0 ? c0 : s0;
            GELO_TRY(apply(s0, start[e] - s0, tc.tsuper + (size_t)(s / per) * kSuper * kSuper, Q + (size_t)s0 * ld + from, c1 - from, true,
                           { tc.w32[0] + c0, tc.w32[1] + c0, tc.wf32 + c0, kSuperKSplit }));
        }
        return GELO_OK;
    };
    float* Gf = G + (size_t)bf * ld + bf;
    float* Qf = Q + (size_t)bf * ld + bf;
    if (!fork) {
        GELO_TRY(launch_qr_small(ctx, m - bf, Gf, ld, Qf, st));
        return form_q(0, m);
    }
    // (the columns of the square only have it in common with the others that the reflectors come next: c1 - from <= bf in the
    // first call, so the second's scratch, from column bf on, is its own)
    GELO_TRY(branch());
    GELO_TRY(launch_qr_small(ctx, m - bf, Gf, ld, Qf, cur));
    GELO_TRY(form_q(bf, m));
    cur = st;
    GELO_TRY(form_q(0, bf));
    GELO_TRY(join());
    return GELO_OK;
}

}  // namespace gelo

// bf16 tensor-core GEMM on sm_100a: tcgen05.mma with the accumulator in tensor memory, operands
// staged in shared memory by TMA, fp32 accumulation.  It serves
//   * the three products of the offload (Eq. 1-3): C = A B with bf16 operands and bf16 output,
//     the B operand optionally the stack [H; S] of Eq. 8, the output optionally split Q | K | V;
//   * the level-3 updates of the blocked QR / LU behind the sampling of A: fp32 matrices are held
//     as a bf16 (high, low) pair and the product is accumulated as hi*hi + hi*lo + lo*hi in fp32,
//     with an epilogue that either subtracts the result from an fp32 matrix in place or writes it
//     as a new (high, low) pair;
//   * the same level-3 updates in one product of kind::tf32 straight from the fp32 matrices (no operand
//     conversion passes at all): the A operand is either K-major (a row-major M x K matrix) or MN-major
//     (the transpose of a row-major K x M matrix, which is how V^T C reads the reflectors).
//
//   C (M x N)  (+)=  sum over segments s of  A_s (M x K_s, row-major)  *  B_s (K_s x N, row-major)
//
// * A tiles (128 rows x 64 k) land K-major, B tiles (64 k x BN columns, as 64-column boxes) land
//   N-major; both use the 128-byte swizzle that TMA writes and the MMA reads.
// * A segment names one A tensor map, one B tensor map and a starting k for each; the stacked
//   operand of the mixing product is two segments, a split-precision product is three.  TMA's
//   out-of-bounds zero fill handles every ragged edge (including a seam inside a k-block).
// * CTAs (one per SM, in pairs on 256 x 256 tiles where use_pair() says so) that take tile after tile from the hardware's queue
//   (cluster launch control), so that one which starts late because another stream's kernel held its SM finds less
//   left to do instead of a fixed share: the 32-layer sweep 87 -> 81.5 ms, 32 fp32 calls at 1075 rows on 16 lanes 99 -> 54 ms (one
//   call alone at 4300 rows 5.70 -> 5.75 ms); warp-specialised: warp 0 issues TMA, warp 1 issues MMA and owns
//   the tensor-memory allocation, warps 2-9 drain the accumulator (two warps per TMEM lane
//   quarter, half of the columns each).  Two accumulator stages let the epilogue of one tile
//   overlap the main loop of the next.
// * Every wait on an mbarrier is bounded in time (the context's wait limit, two seconds by default,
//   measured on the GPU's global timer); on expiry the CTA records GELO_ERR_TIMEOUT in the
//   context's status word, stops issuing work, lets what is in flight arrive, releases tensor memory and returns.
#include <cuda.h>

#include <algorithm>

#include "common.cuh"
#include "tc_ptx.cuh"

namespace gelo {

namespace {

using namespace tcx;

constexpr int BM = 128;
constexpr int BK = 64;
constexpr int kAccStages = 2;
constexpr int kEpiWarps = 8;
constexpr int kThreads = 64 + 32 * kEpiWarps;
constexpr uint32_t kABytes = BM * BK * 2;            // 16 KiB
constexpr uint32_t kTmemCols = 512;
constexpr uint32_t kBarBytes = 640;                  // barriers and the ring of tiles
constexpr int kRing = 16;                            // tiles the roles of a CTA may be apart, see next_tile()

enum TcMode { TC_STORE_BF16 = 0, TC_STORE_F32 = 1, TC_SUB_F32 = 2, TC_EMIT_SPLIT = 3, TC_STORE_SYM16 = 4, TC_AFFINE16 = 5 };

struct TcSegment { int a_sel, b_sel, a_k0, b_row0, kb; };

struct TcParams {
    int M, N;
    int nseg;
    TcSegment seg[3];
    int mode;
    void* C0; void* C1; void* C2;   // STORE_*: column-split outputs; SUB_F32: C0 fp32, C1/C2 optional hi/lo; EMIT_SPLIT: C0 hi, C1 lo
    int ldc, csplit, lde;           // lde: row stride of the hi/lo matrices written next to an fp32 C
    int ksplit, kb_per_split;       // K slices (TC_STORE_F32 only): slice q covers k-blocks [q*kb_per_split, ...) of every segment
    long long plane;                // and writes plane q of C0 (stride in elements)
    int round_tf32;                 // TC_STORE_F32: round the stored values to tf32 (they feed a later tf32 product)
    float out_scale;                // TC_STORE_F32 with round_tf32: factor applied before the rounding
    float diag_sub;                 // TC_STORE_F32 with round_tf32: subtracted from the scaled diagonal entries
    float post_scale;               //   ... and the factor applied after that: out = post_scale * (out_scale * acc - diag_sub [row == col])
    int a3d, b3d;                   // the MN-major A tile / the B tile arrives as ONE three-dimensional box (see make_map_nmajor)
    int out_f16;                    // TC_STORE_BF16: operands and output are IEEE half instead of bfloat16
    const float* scale_a;           // TC_STORE_BF16 with 8-bit operands: the per-tensor scales (device scalars); the
    const float* scale_b;           //   accumulator is multiplied by their product before it is rounded
    const void* add; int ldadd;     // TC_AFFINE16: out = out_scale * acc + diag_sub on the diagonal + post_scale * the entry of `add` (optional)
    int tri, tri_tiles;             // TC_STORE_SYM16: the result is symmetric; only the tri_tiles tiles that reach the diagonal or lie
                                    // above it are computed, and what lies below them is filled in by mirroring
    int tiles, stride;              // kShare: all tiles, and how many CTAs (pairs) share them
    uint32_t idesc;                 // instruction descriptor (filled in by the launcher)
    unsigned long long wait_ns;     // limit of every mbarrier wait, nanoseconds (filled in by the launcher from the context)
    int* status;
};

// Epilogue staging for the in-place subtraction: every epilogue warp owns two 32 x 32 fp32 boxes (4 KiB each)
// that TMA reduces into global memory.
constexpr uint32_t kStageBoxBytes = 32 * 32 * 4;
constexpr uint32_t kStagingBytes = kEpiWarps * 2 * kStageBoxBytes;

// Store epilogue staging: 32 rows of 128 bytes per epilogue warp.
constexpr uint32_t kStoreBytes = kEpiWarps * 32 * 128;

// A stage holds 128 bytes of k per A row (64 bf16 or 32 tf32 values) and the matching B rows, so both kinds share
// the shared-memory geometry: kTf32 only changes the element count per k-block, the box width of the N-major B tile
// (128 bytes = 64 bf16 or 32 fp32 columns) and the instruction.  kAMn (tf32 only): the A tile arrives as four
// boxes of 32 m-columns x 32 k-rows, i.e. laid out exactly like a 128-column B tile.
// kPair: a cluster of two CTAs works on one 256-row tile (cta_group::2).  Each holds its 128 rows of A and one half of
// the columns of B, and accumulates its 128 rows over all columns; CTA 0 issues the instructions for both.
template <int BN, bool kStaging, bool kTf32 = false, bool kAMn = false, bool kF8 = false, bool kPair = false>
struct TcCfg {
    static constexpr int kCols = kPair ? BN / 2 : BN;                      // columns of B that one CTA holds
    static constexpr int kTileRows = kPair ? 2 * BM : BM;
    static constexpr uint32_t kStagingUsed = kStaging ? kStagingBytes : kStoreBytes;
    static constexpr int kBKE = kF8 ? 128 : (kTf32 ? 32 : 64);             // elements of k per stage
    static constexpr int kBoxCols = kF8 ? 128 : (kTf32 ? 32 : 64);         // columns of one N-major box (128 bytes)
    static constexpr uint32_t kBoxBytes = (uint32_t)kBKE * 128u;           // one N-major box: kBKE rows of 128 bytes
    static constexpr uint32_t kBBytes = (kCols / kBoxCols) * kBoxBytes;
    static constexpr uint32_t kStageBytes = kABytes + kBBytes;
    // as many stages as fit, six at most: 4 (3 with staging for the in-place subtraction) alone, 6 (5) in a pair
    static constexpr int kFit = (int)((227u * 1024u - 1024u - kBarBytes - kStagingUsed) / kStageBytes);
    static constexpr int kStages = kFit > 6 ? 6 : kFit;
    static constexpr uint32_t kSmemBytes = kStages * kStageBytes + kStagingUsed + 1024 /*alignment slack*/ + kBarBytes;
    // k advance per instruction inside an N-major (or MN-major A) tile: 16 bf16 rows or 8 tf32 rows of 128 bytes
    static constexpr uint32_t kMnStep = kF8 ? 4096u : (kTf32 ? 1024u : 2048u);   // 32 e4m3 rows, 16 bf16 rows or 8 tf32 rows
    // N-major tiles: bf16 in the 16-byte-chunk swizzle (atoms of 8 k-rows, 1024 bytes), fp32 in the 32-byte-chunk
    // swizzle (atoms of 4 k-rows, 512 bytes)
    static constexpr uint32_t kMnLayout = kTf32 ? 1u : 2u;
    static constexpr uint32_t kMnSbo = kTf32 ? 512u : 1024u;
    // Instruction descriptor: fp32 accumulate, operand formats (1 = bf16, 2 = tf32), A K-major or MN-major,
    // B N-major, M = 128 (256 in a pair), N = BN.
    static constexpr uint32_t kFmt = kF8 ? 0u : (kTf32 ? 2u : 1u);         // kind::f8f6f4: 0 = E4M3
    static constexpr uint32_t kInstrDesc = (1u << 4) | (kFmt << 7) | (kFmt << 10) | ((kAMn ? 1u : 0u) << 15) | (1u << 16) |
                                           ((uint32_t)(BN >> 3) << 17) | ((uint32_t)(kTileRows >> 4) << 24);
    static_assert(!kAMn || kTf32, "MN-major A is only wired up for the tf32 kind");
    static_assert(!(kF8 && kTf32), "one operand kind per instance");
    static_assert(kCols % kBoxCols == 0, "a CTA's share of B is whole boxes");
};

// x = hi + lo with hi = bf16(x), lo = bf16(x - hi)
__device__ __forceinline__ void split2(float a, float b, uint32_t& hi, uint32_t& lo)
{
    const __nv_bfloat162 h = __floats2bfloat162_rn(a, b);
    const float2 hf = __bfloat1622float2(h);
    const __nv_bfloat162 l = __floats2bfloat162_rn(a - hf.x, b - hf.y);
    hi = *reinterpret_cast<const uint32_t*>(&h);
    lo = *reinterpret_cast<const uint32_t*>(&l);
}

// Row-tile and column-tile index of work item `tile`.  Ordinary products: row tiles fastest, then column tiles, then K
// slices.  Symmetric products (prm.tri, 256 columns per tile): column tile nt owns the row tiles whose first row is not
// below its last column, mt <= 2 nt + 1 (of 128 rows) or mt <= nt (of 256); they are enumerated column tile after column tile.
template <bool kPair>
__device__ __forceinline__ void tile_coords(const TcParams& prm, int tile, int m_tiles, int mn_tiles, int& mt, int& nt, int& slice)
{
    if (prm.tri) {
        int t = tile;
        nt = 0;
        for (;;) {
            const int cnt = min(m_tiles, kPair ? nt + 1 : 2 * nt + 2);
            if (t < cnt) break;
            t -= cnt; ++nt;
        }
        mt = t; slice = 0;
        return;
    }
    const int mn = tile % mn_tiles;
    slice = tile / mn_tiles;
    mt = mn % m_tiles;
    nt = mn / m_tiles;
}

// ---- the storing epilogue -----------------------------------------------------------------------------
// A warp holds 32 rows of the tile, a lane one row each.  Written from there, every 16-byte store instruction would touch
// 32 lines; so 128 bytes of every row at a time (64 columns of a 16-bit result, 32 of an fp32 one) go through 4 KiB of
// shared memory (16-byte chunks swizzled by the row) and leave as whole lines: eight lanes per row, four rows per instruction.

__device__ __forceinline__ uint32_t stage_addr(uint32_t buf, int row, int chunk) { return buf + row * 128 + ((chunk ^ (row & 7)) << 4); }
__device__ __forceinline__ void stage_put(uint32_t buf, int row, int chunk, uint4 v)
{
    asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(stage_addr(buf, row, chunk)), "r"(v.x), "r"(v.y), "r"(v.z), "r"(v.w) : "memory");
}
__device__ __forceinline__ uint4 stage_get(uint32_t buf, int row, int chunk)
{
    uint4 v;
    asm volatile("ld.shared.v4.b32 {%0, %1, %2, %3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "r"(stage_addr(buf, row, chunk)) : "memory");
    return v;
}

// The staged rows (first one m0) to C, 128 bytes per row from column gn on; elements of kBytes bytes.
template <int kBytes>
__device__ __forceinline__ void write_staged(const TcParams& prm, uint32_t buf, int m0, int gn, int lane, long long offset)
{
    constexpr int kPer = 16 / kBytes;                         // elements per chunk
    const int c = lane & 7, n = gn + kPer * c;
    const int part = n / prm.csplit;                          // column block -> C0 / C1 / C2 (0 unless the output is split)
    char* base = static_cast<char*>(part == 0 ? prm.C0 : (part == 1 ? prm.C1 : prm.C2));
    char* dst = base + (offset + (long long)(m0 + (lane >> 3)) * prm.ldc + (n - part * prm.csplit)) * kBytes;
    const size_t step = (size_t)4 * prm.ldc * kBytes;
    if (n < prm.N) {
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            const int r = 4 * i + (lane >> 3);
            if (m0 + r < prm.M) *reinterpret_cast<uint4*>(dst + i * step) = stage_get(buf, r, c);
        }
    }
}

// Accumulator columns [c, c + 64) of the tile as 64 16-bit values per row: product times the two scales (TC_STORE_BF16),
// or out_scale * product + diag on the diagonal + post_scale * the entry of `add` (TC_AFFINE16).
__device__ __forceinline__ void store_tile16(const TcParams& prm, uint32_t taddr, uint32_t buf, int m0, int gn, int lane)
{
    const bool affine = prm.mode == TC_AFFINE16;
    const int gm = m0 + lane;
    const float sc = affine ? prm.out_scale : (prm.scale_a ? prm.scale_a[0] * prm.scale_b[0] : 1.0f);
    if (affine && prm.add) {
        const int n = gn + 8 * (lane & 7);
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            const int r = 4 * i + (lane >> 3);
            uint4 v = make_uint4(0u, 0u, 0u, 0u);
            if (n < prm.N && m0 + r < prm.M)
                v = *reinterpret_cast<const uint4*>(static_cast<const __nv_bfloat16*>(prm.add) + (size_t)(m0 + r) * prm.ldadd + n);
            stage_put(buf, r, lane & 7, v);
        }
        __syncwarp();
    }
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        uint32_t v[32];
        tc_ld_32cols(taddr + 32 * h, v);
        tc_ld_wait();
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            float f[8];
#pragma unroll
            for (int j = 0; j < 8; ++j) {
                f[j] = sc * __uint_as_float(v[8 * q + j]);
                if (affine && gm == gn + 32 * h + 8 * q + j) f[j] += prm.diag_sub;
            }
            if (affine && prm.add) {
                const uint4 raw = stage_get(buf, lane, 4 * h + q);
                const uint32_t w2[4] = {raw.x, raw.y, raw.z, raw.w};
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    const float2 t = prm.out_f16 ? __half22float2(*reinterpret_cast<const __half2*>(&w2[j]))
                                                 : __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&w2[j]));
                    f[2 * j] = fmaf(prm.post_scale, t.x, f[2 * j]); f[2 * j + 1] = fmaf(prm.post_scale, t.y, f[2 * j + 1]);
                }
            }
            uint32_t o[4];
#pragma unroll
            for (int j = 0; j < 4; ++j)
                o[j] = prm.out_f16 ? pack_f16(__float_as_uint(f[2 * j]), __float_as_uint(f[2 * j + 1]))
                                   : pack_bf16(__float_as_uint(f[2 * j]), __float_as_uint(f[2 * j + 1]));
            stage_put(buf, lane, 4 * h + q, make_uint4(o[0], o[1], o[2], o[3]));
        }
    }
    __syncwarp();
    write_staged<2>(prm, buf, m0, gn, lane, 0);
    __syncwarp();
}

// 32 accumulator columns as fp32, plain or (round_tf32) scaled, shifted on the diagonal and rounded; K slice `slice` of
// the output.
__device__ __forceinline__ void store_tile32(const TcParams& prm, const uint32_t (&v)[32], uint32_t buf, int m0, int gn, int lane, int slice)
{
    const int gm = m0 + lane;
#pragma unroll
    for (int q = 0; q < 8; ++q) {
        float f[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const float a = __uint_as_float(v[4 * q + j]);
            f[j] = prm.round_tf32 ? round_tf32(prm.post_scale * (prm.out_scale * a - ((gm == gn + 4 * q + j) ? prm.diag_sub : 0.0f))) : a;
        }
        stage_put(buf, lane, q, make_uint4(__float_as_uint(f[0]), __float_as_uint(f[1]), __float_as_uint(f[2]), __float_as_uint(f[3])));
    }
    __syncwarp();
    write_staged<4>(prm, buf, m0, gn, lane, (long long)slice * prm.plane);
    __syncwarp();
}

// 16 fp32 columns of 32 rows (a lane holds one row) from column gn on, through 2 KiB of shared memory: four lanes per row.
__device__ __forceinline__ void store_cols16(const TcParams& prm, const float* f, uint32_t buf, int m0, int gn, int lane, long long offset)
{
#pragma unroll
    for (int q = 0; q < 4; ++q)
        asm volatile("st.shared.v4.f32 [%0], {%1, %2, %3, %4};"
                     ::"r"(buf + lane * 64 + ((q ^ ((lane >> 1) & 3)) << 4)), "f"(f[4 * q]), "f"(f[4 * q + 1]), "f"(f[4 * q + 2]), "f"(f[4 * q + 3]) : "memory");
    __syncwarp();
    const int c = lane & 3, n = gn + 4 * c;
    const int part = n / prm.csplit;
    float* base = static_cast<float*>(part == 0 ? prm.C0 : (part == 1 ? prm.C1 : prm.C2));
    float* dst = base + offset + (long long)(m0 + (lane >> 2)) * prm.ldc + (n - part * prm.csplit);
    if (n < prm.N) {
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const int r = 8 * i + (lane >> 2);
            float4 v;
            asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "r"(buf + r * 64 + ((c ^ ((r >> 1) & 3)) << 4)) : "memory");
            if (m0 + r < prm.M) *reinterpret_cast<float4*>(dst + (size_t)(8 * i) * prm.ldc) = v;
        }
    }
    __syncwarp();
}

// The product as a (hi, lo) bf16 pair, eight columns from gn on.
template <int G>
__device__ __forceinline__ void emit_split(const TcParams& prm, int gm, int gn, const uint32_t (&w)[32])
{
    if (gn >= prm.N) return;
    uint4 hi, lo;
    split2(__uint_as_float(w[G * 8 + 0]), __uint_as_float(w[G * 8 + 1]), hi.x, lo.x);
    split2(__uint_as_float(w[G * 8 + 2]), __uint_as_float(w[G * 8 + 3]), hi.y, lo.y);
    split2(__uint_as_float(w[G * 8 + 4]), __uint_as_float(w[G * 8 + 5]), hi.z, lo.z);
    split2(__uint_as_float(w[G * 8 + 6]), __uint_as_float(w[G * 8 + 7]), hi.w, lo.w);
    const size_t off = (size_t)gm * prm.ldc + gn;
    *reinterpret_cast<uint4*>(static_cast<__nv_bfloat16*>(prm.C0) + off) = hi;
    *reinterpret_cast<uint4*>(static_cast<__nv_bfloat16*>(prm.C1) + off) = lo;
}

// Symmetric result (TC_STORE_SYM16): 32 consecutive entries of row gm from column gn on, as
// post_scale * (out_scale * acc - diag_sub [on the diagonal]) in bf16.  Entries above the diagonal whose mirror image
// lies in a tile that is not computed (see tile_coords) are also written there; consecutive lanes hold consecutive
// rows, so those transposed stores are contiguous across the warp.
__device__ __forceinline__ void store_symmetric(const TcParams& prm, int gm, int gn, const uint32_t (&v)[32])
{
    __nv_bfloat16* D = static_cast<__nv_bfloat16*>(prm.C0);
    __align__(16) __nv_bfloat16 h[32];
#pragma unroll
    for (int j = 0; j < 32; ++j)
        h[j] = __float2bfloat16_rn(prm.post_scale * (prm.out_scale * __uint_as_float(v[j]) - ((gm == gn + j) ? prm.diag_sub : 0.0f)));
#pragma unroll
    for (int g = 0; g < 4; ++g)
        if (gn + 8 * g < prm.N)
            *reinterpret_cast<uint4*>(D + (size_t)gm * prm.ldc + gn + 8 * g) = *reinterpret_cast<const uint4*>(&h[8 * g]);
    const int my_pair = gm >> 8;                              // column tile of the mirrored entry
#pragma unroll
    for (int j = 0; j < 32; ++j) {
        const int c = gn + j;
        if (c > gm && c < prm.M && (c >> 7) > 2 * my_pair + 1) D[(size_t)c * prm.ldc + gm] = h[j];
    }
}

// kShare: prm.stride CTAs (pairs) share the tiles in turn instead of taking them from the queue.  Instances of their own: looked at by every one of
// them, the stride cost E4M3 at 2150 x 12288 x 4096 92.6 instead of 90.9 us and a tf32 update of 512 x 4096 x 512 12.5 instead of 12.2.
template <int BN, bool kStaging, bool kTf32, bool kAMn, bool kF8, bool kPair, bool kShare>
__global__ void __launch_bounds__(kThreads, 1)
gemm_tc_kernel(const __grid_constant__ CUtensorMap map_a0, const __grid_constant__ CUtensorMap map_a1,
               const __grid_constant__ CUtensorMap map_b0, const __grid_constant__ CUtensorMap map_b1,
               const __grid_constant__ CUtensorMap map_c, const TcParams prm)
{
    using Cfg = TcCfg<BN, kStaging, kTf32, kAMn, kF8, kPair>;
    constexpr int kStages = Cfg::kStages;
    extern __shared__ uint8_t smem_raw[];
    const uint32_t raw = smem_u32(smem_raw);
    const uint32_t tiles_base = (raw + 1023u) & ~1023u;                 // swizzle atoms need 1024-byte alignment
    uint8_t* gen_base = smem_raw + (tiles_base - raw);
    const uint32_t staging_base = tiles_base + kStages * Cfg::kStageBytes;      // 1024-byte aligned
    const uint32_t bar_base = staging_base + Cfg::kStagingUsed;
    uint8_t* bar_gen = gen_base + kStages * Cfg::kStageBytes + Cfg::kStagingUsed;
    // barrier layout (8 bytes each): full[kStages], empty[kStages], acc_full[2], acc_empty[2]; then tmem slot, abort
    auto full_bar = [&](int s) { return bar_base + 8u * s; };
    auto empty_bar = [&](int s) { return bar_base + 8u * (kStages + s); };
    auto acc_full_bar = [&](int a) { return bar_base + 8u * (2 * kStages + a); };
    auto acc_empty_bar = [&](int a) { return bar_base + 8u * (2 * kStages + kAccStages + a); };
    constexpr uint32_t kMisc = 8 * (2 * kStages + 2 * kAccStages);
    volatile uint32_t* tmem_slot = reinterpret_cast<volatile uint32_t*>(bar_gen + kMisc);
    volatile int* abort_flag = reinterpret_cast<volatile int*>(bar_gen + kMisc + 8);
    const uint32_t clc_bar = bar_base + kMisc + 16, clc_slot = bar_base + ((kMisc + 24 + 15) & ~15u);
    const uint32_t ring_off = ((kMisc + 24 + 15) & ~15u) + 16;
    auto tile_bar = [&](int i) { return bar_base + ring_off + 8u * i; };
    const uint32_t ring_base = bar_base + ring_off + 8u * kRing;
    static_assert(kMisc + 24 + 15 + 16 + 12 * kRing <= kBarBytes, "barriers and ring fit");

    const int warp = threadIdx.x >> 5;
    const int lane = threadIdx.x & 31;

    const int rank = kPair ? (int)cluster_rank() : 0;         // CTA 0 of a pair leads
    const int first_tile = kPair ? blockIdx.x >> 1 : blockIdx.x;
    const int m_tiles = (prm.M + Cfg::kTileRows - 1) / Cfg::kTileRows;
    const int n_tiles = (prm.N + BN - 1) / BN;
    const int mn_tiles = m_tiles * n_tiles;

    chain_next();
    if (threadIdx.x == 0) {
        for (int s = 0; s < kStages; ++s) { mbar_init(full_bar(s), 1); mbar_init(empty_bar(s), 1); }
        for (int a = 0; a < kAccStages; ++a) { mbar_init(acc_full_bar(a), 1); mbar_init(acc_empty_bar(a), kPair ? 2 * kEpiWarps : kEpiWarps); }
        mbar_init(clc_bar, 1);
        for (int i = 0; i < kRing; ++i) mbar_init(tile_bar(i), 1);
        *abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    }
    if (warp == 1) {
        if (kPair) {
            asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;"
                         ::"r"(smem_u32((const void*)tmem_slot)), "r"(kTmemCols) : "memory");
            asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
        } else {
            asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;"
                         ::"r"(smem_u32((const void*)tmem_slot)), "r"(kTmemCols) : "memory");
            asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
        }
    }
    tc_fence_before();
    __syncwarp();
    if (kPair) cluster_sync(); else __syncthreads();
    tc_fence_after();
    const uint32_t tmem_base = *tmem_slot;
    chain_wait();

    // The tiles of a CTA (pair): the one it was launched for, then whatever the leader's producer gets from the hardware's
    // queue of CTAs not yet launched.  It hands each on through a ring; -1 ends.  The roles are at most kStages + 3 tiles apart (a tile
    // has at least one stage of operands, and two accumulators), so a ring of kRing never overruns.
    auto next_tile = [&](uint32_t it, bool& ok) -> int {
        const int i = it % kRing;
        const uint32_t parity = (it / kRing) & 1u;
        if (!(kPair ? mbar_wait_cluster(tile_bar(i), parity, abort_flag, prm.wait_ns) : mbar_wait(tile_bar(i), parity, abort_flag, prm.wait_ns))) {
            ok = false;
            return -1;
        }
        int t;
        asm volatile("ld.shared.s32 %0, [%1];" : "=r"(t) : "r"(ring_base + 4u * i) : "memory");
        return t;
    };

    if (warp == 0) {
        // ================= TMA producer =================
        if (lane == 0) {
            uint32_t it = 0, tile_it = 0;
            bool ok = true, asked = false;
            for (int tile = first_tile; tile >= 0 && ok; ++tile_it) {
                int mt, nt, slice;
                tile_coords<kPair>(prm, tile, m_tiles, mn_tiles, mt, nt, slice);
                const int m0 = mt * Cfg::kTileRows + rank * BM, n0 = nt * BN + rank * Cfg::kCols;
#pragma unroll
                for (int sg = 0; sg < 3; ++sg) {              // constant indices keep the parameters out of local memory
                    if (sg >= prm.nseg || !ok) break;
                    const TcSegment seg = prm.seg[sg];
                    const CUtensorMap* ma = seg.a_sel ? &map_a1 : &map_a0;
                    const CUtensorMap* mb = seg.b_sel ? &map_b1 : &map_b0;
                    const int kb_lo = slice * prm.kb_per_split;
                    const int kb_hi = min(seg.kb, kb_lo + prm.kb_per_split);
                    for (int kb = kb_lo; kb < kb_hi; ++kb, ++it) {
                        const int s = it % kStages;
                        const uint32_t ph = (it / kStages) & 1u;
                        if (!mbar_wait(empty_bar(s), ph ^ 1u, abort_flag, prm.wait_ns)) { ok = false; break; }
                        const uint32_t sa = tiles_base + s * Cfg::kStageBytes;
                        const uint32_t sb = sa + kABytes;
                        // in a pair the copies of both CTAs count on the leader's barrier
                        if (rank == 0) mbar_expect_tx(full_bar(s), kPair ? 2 * Cfg::kStageBytes : Cfg::kStageBytes);
                        const uint32_t bar = kPair ? map_rank(full_bar(s), 0) : full_bar(s);
                        auto load_2d = [&](uint32_t dst, const CUtensorMap* map, int x, int y) {
                            if (kPair) tma_load_2d_pair(dst, map, x, y, bar); else tma_load_2d(dst, map, x, y, bar);
                        };
                        auto load_3d = [&](uint32_t dst, const CUtensorMap* map, int x, int y, int z) {
                            if (kPair) tma_load_3d_pair(dst, map, x, y, z, bar); else tma_load_3d(dst, map, x, y, z, bar);
                        };
                        if (kAMn) {
                            if (prm.a3d) {
                                load_3d(sa, ma, 0, seg.a_k0 + kb * Cfg::kBKE, m0 / Cfg::kBoxCols);
                            } else {
#pragma unroll
                                for (int j = 0; j < BM / Cfg::kBoxCols; ++j)
                                    load_2d(sa + j * Cfg::kBoxBytes, ma, m0 + j * Cfg::kBoxCols, seg.a_k0 + kb * Cfg::kBKE);
                            }
                        } else {
                            load_2d(sa, ma, seg.a_k0 + kb * Cfg::kBKE, m0);
                        }
                        if (prm.b3d) {
                            load_3d(sb, mb, 0, seg.b_row0 + kb * Cfg::kBKE, n0 / Cfg::kBoxCols);
                        } else {
#pragma unroll
                            for (int j = 0; j < Cfg::kCols / Cfg::kBoxCols; ++j)
                                load_2d(sb + j * Cfg::kBoxBytes, mb, n0 + j * Cfg::kBoxCols, seg.b_row0 + kb * Cfg::kBKE);
                        }
                        if (!kShare && rank == 0 && !asked) {     // the next tile, while this one's operands come in
                            mbar_expect_tx(clc_bar, 16);
                            clc_try_cancel(clc_slot, clc_bar);
                            asked = true;
                        }
                    }
                }
                if (rank == 0) {
                    if (asked && !mbar_wait(clc_bar, tile_it & 1u, abort_flag, prm.wait_ns)) ok = false;
                    if (!ok) break;
                    asked = false;
                    if (kShare) {
                        tile = tile + prm.stride < prm.tiles ? tile + prm.stride : -1;
                    } else {
                        const int x = clc_answer(clc_slot);
                        tile = kPair && x >= 0 ? x >> 1 : x;
                    }
                    const uint32_t slot = ring_base + 4u * (tile_it % kRing), bar = tile_bar(tile_it % kRing);
                    asm volatile("st.shared.s32 [%0], %1;" ::"r"(slot), "r"(tile) : "memory");
                    if (kPair) {
                        asm volatile("st.shared::cluster.s32 [%0], %1;" ::"r"(map_rank(slot, 1)), "r"(tile) : "memory");
                        mbar_arrive_cluster(map_rank(bar, 1));
                    }
                    mbar_arrive(bar);
                } else {
                    tile = next_tile(tile_it, ok);
                }
            }
            if (!ok) { *abort_flag = 1; atomicCAS(prm.status, 0, (int)GELO_ERR_TIMEOUT); }
        }
    } else if (warp == 1) {
        // ================= MMA issuer (in a pair: of the leader) =================
        if (lane == 0 && rank == 0) {
            uint32_t acc_it = 0;
            uint32_t s = 0, ph = 0;                   // operand stage and the parity of its "full" phase
            bool ready = false;                       // stage s is already known to be full (tested ahead, see tc_mma4_*_try)
            bool ok = true;
            // k advance per instruction in sixteen-byte units of the descriptors' start address
            constexpr uint64_t kAStep = kAMn ? (Cfg::kMnStep >> 4) : 2, kBStep = Cfg::kMnStep >> 4;
            for (int tile = first_tile; tile >= 0 && ok; tile = next_tile(acc_it, ok), ++acc_it) {
                const int slice = prm.tri ? 0 : tile / mn_tiles;
                int kb_total = 0;
#pragma unroll
                for (int sg = 0; sg < 3; ++sg)
                    if (sg < prm.nseg) {
                        const int kb_lo = slice * prm.kb_per_split;
                        const int kb_hi = min(prm.seg[sg].kb, kb_lo + prm.kb_per_split);
                        kb_total += max(0, kb_hi - kb_lo);
                    }
                const int a = acc_it % kAccStages;
                const uint32_t aph = (acc_it / kAccStages) & 1u;
                if (!mbar_wait(acc_empty_bar(a), aph ^ 1u, abort_flag, prm.wait_ns)) { ok = false; break; }
                tc_fence_after();
                const uint32_t tmem_d = tmem_base + (uint32_t)(a * BN);
                for (int kb = 0; kb < kb_total; ++kb) {
                    if (!ready && !mbar_wait(full_bar(s), ph, abort_flag, prm.wait_ns)) { ok = false; break; }
                    const uint32_t sa = tiles_base + s * Cfg::kStageBytes;
                    const uint32_t sb = sa + kABytes;
                    // A K-major: 8-row groups 1024 bytes apart, 32 bytes per k step.  A MN-major: like B.
                    const uint64_t da = kAMn ? smem_desc(sa, Cfg::kBoxBytes, Cfg::kMnSbo, Cfg::kMnLayout) : smem_desc(sa, 16, 1024);
                    // B: N-major, 128-byte-wide boxes kBoxBytes apart, k-row atoms kMnSbo bytes apart
                    const uint64_t db = smem_desc(sb, Cfg::kBoxBytes, Cfg::kMnSbo, Cfg::kMnLayout);
                    const uint32_t ns = (s + 1 == kStages) ? 0u : s + 1;
                    const uint32_t nph = (ns == 0u) ? (ph ^ 1u) : ph;
                    // four instructions of 32 bytes of k (16 bf16 / 8 tf32) per stage
                    ready = tc_mma4_try<kF8 ? 2 : (kTf32 ? 1 : 0), kPair>(tmem_d, da, db, kAStep, kBStep, prm.idesc, kb != 0 ? 1u : 0u,
                                                                          full_bar(ns), nph);
                    if (kPair) tc_commit_pair(empty_bar(s)); else tc_commit(empty_bar(s));   // frees the stage once these MMAs have read it
                    s = ns; ph = nph;
                }
                if (!ok) break;
                if (kPair) tc_commit_pair(acc_full_bar(a)); else tc_commit(acc_full_bar(a));   // accumulator complete
            }
            if (!ok) { *abort_flag = 1; atomicCAS(prm.status, 0, (int)GELO_ERR_TIMEOUT); }
        }
    } else {
        // ================= epilogue (warps 2..9) =================
        const int quarter = warp & 3;                 // the TMEM lane quarter this warp may read
        const int half = (warp - 2) >> 2;             // which half of the tile's columns
        constexpr int kHalfCols = BN / 2;
        uint32_t acc_it = 0, box_it = 0;
        bool ok = true;
        for (int tile = first_tile; tile >= 0 && ok; tile = next_tile(acc_it, ok), ++acc_it) {
            const int a = acc_it % kAccStages;
            const uint32_t aph = (acc_it / kAccStages) & 1u;
            int mt, nt, slice;
            tile_coords<kPair>(prm, tile, m_tiles, mn_tiles, mt, nt, slice);
            const int m0 = mt * Cfg::kTileRows + rank * BM, n0 = nt * BN;
            const int gm = m0 + quarter * 32 + lane;
            const bool row_ok = gm < prm.M;
            if (kStaging && prm.mode == TC_SUB_F32) {
                // C -= acc without reading C: the negated accumulator goes through a swizzled shared-memory box and
                // a TMA reduce-add into global memory (the addition happens at the L2); TMA clips at the matrix edge
                if (!mbar_wait(acc_full_bar(a), aph, abort_flag, prm.wait_ns)) { ok = false; break; }
                tc_fence_after();
                const uint32_t taddr = tmem_base + ((uint32_t)(quarter * 32) << 16) + (uint32_t)(a * BN);
                const uint32_t my_staging = staging_base + (uint32_t)(warp - 2) * 2u * kStageBoxBytes;
#pragma unroll 1
                for (int c = half * kHalfCols; c < (half + 1) * kHalfCols; c += 32, ++box_it) {
                    const uint32_t buf = my_staging + (box_it & 1u) * kStageBoxBytes;
                    if (lane == 0) asm volatile("cp.async.bulk.wait_group.read 1;" ::: "memory");   // box of two chunks ago is free
                    __syncwarp();
                    uint32_t v[32];
                    tc_ld_32cols(taddr + c, v);
                    tc_ld_wait();
#pragma unroll
                    for (int j4 = 0; j4 < 8; ++j4) {
                        const uint32_t dst = buf + (uint32_t)lane * 128u + (uint32_t)((j4 ^ (lane & 7)) << 4);
                        asm volatile("st.shared.v4.f32 [%0], {%1, %2, %3, %4};"
                                     ::"r"(dst), "f"(-__uint_as_float(v[4 * j4 + 0])), "f"(-__uint_as_float(v[4 * j4 + 1])),
                                       "f"(-__uint_as_float(v[4 * j4 + 2])), "f"(-__uint_as_float(v[4 * j4 + 3])) : "memory");
                    }
                    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                    __syncwarp();
                    if (lane == 0 && n0 + c < prm.N && m0 + quarter * 32 < prm.M) {
                        asm volatile(
                            "cp.reduce.async.bulk.tensor.2d.global.shared::cta.add.tile.bulk_group [%0, {%1, %2}], [%3];"
                            ::"l"(&map_c), "r"(n0 + c), "r"(m0 + quarter * 32), "r"(buf) : "memory");
                    }
                    if (lane == 0) asm volatile("cp.async.bulk.commit_group;" ::: "memory");
                }
            } else {
                if (!mbar_wait(acc_full_bar(a), aph, abort_flag, prm.wait_ns)) { ok = false; break; }
                tc_fence_after();
                const uint32_t taddr = tmem_base + ((uint32_t)(quarter * 32) << 16) + (uint32_t)(a * BN);
                const int c_end = min((half + 1) * kHalfCols, prm.N - n0);
                const uint32_t buf = staging_base + (uint32_t)(warp - 2) * 4096u;
                if (kHalfCols % 64 == 0 && (prm.mode == TC_STORE_BF16 || prm.mode == TC_AFFINE16)) {
#pragma unroll 1
                    for (int c = half * kHalfCols; c < c_end; c += 64) store_tile16(prm, taddr + c, buf, m0 + quarter * 32, n0 + c, lane);
                } else {
#pragma unroll 1
                    for (int c = half * kHalfCols; c < c_end; c += 32) {
                        uint32_t v[32];
                        tc_ld_32cols(taddr + c, v);
                        tc_ld_wait();
                        if (prm.mode == TC_STORE_SYM16) {
                            if (row_ok) store_symmetric(prm, gm, n0 + c, v);
                        } else if (prm.mode == TC_STORE_F32) {
                            store_tile32(prm, v, buf, m0 + quarter * 32, n0 + c, lane, slice);
                        } else if (row_ok) {                  // TC_EMIT_SPLIT
                            const int gn = n0 + c;
                            emit_split<0>(prm, gm, gn, v);
                            emit_split<1>(prm, gm, gn + 8, v);
                            emit_split<2>(prm, gm, gn + 16, v);
                            emit_split<3>(prm, gm, gn + 24, v);
                        }
                    }
                }
            }
            tc_fence_before();
            __syncwarp();
            if (lane == 0) {
                if (kPair) mbar_arrive_cluster(map_rank(acc_empty_bar(a), 0)); else mbar_arrive(acc_empty_bar(a));
            }
        }
        if (lane == 0) asm volatile("cp.async.bulk.wait_group 0;" ::: "memory");   // staged boxes fully written out
        if (!ok && lane == 0) { *abort_flag = 1; atomicCAS(prm.status, 0, (int)GELO_ERR_TIMEOUT); }
    }

    tc_fence_before();
    __syncwarp();
    if (kPair) cluster_sync(); else __syncthreads();
    if (warp == 1) {
        if (*abort_flag) settle(prm.wait_ns);                 // (the CTA's memory is its own until its last warp returns)
        __syncwarp();
        tc_fence_after();
        if (kPair) asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(kTmemCols) : "memory");
        else asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(kTmemCols) : "memory");
    }
}

// ---- fp32 products: three tf32 products of operand pairs that are made on the way ------------------------------------
//
// C = A B in fp32 with fp32-grade accuracy: x = hi + lo, both parts rounded to tf32; lo hi + hi lo + hi hi in fp32.  lo is 2^-11 of x at
// most and of either sign, so lo lo, which is dropped, is 2^-22 of a term at most and cancels (with hi = x as the tensor core reads it, its 13 low
// bits cut off, it is up to 2^-20 and always of the term's sign: products of positive entries came out 8.2e-7 low instead of 4.2e-7).
// A stage holds the fp32 tiles as TMA brings them, which four warps round in place, and beside them their lo parts (element by element at the
// same place, so the swizzle does not matter).  The tensor core adds into its accumulator with truncation, 2^-25 of the running sum per
// instruction and coherent, so an accumulator only takes kX3Slice k-blocks (24 instructions); the epilogue warps add it to sums in
// registers, rounded to nearest, while the other accumulator fills.  Relative error against 64 bits: K = 504 3.7e-7 (hi cut off 4.5e-7; pairs
// written to memory, K in eight slices 7.0e-7), K = 4096 4.0e-7 (4.8e-7, 5.3e-6); with 48 instructions twice that.
//
// Tiles of 256 x 192 on a pair of CTAs; a pair takes one unit (a tile, or a K slice of one) after the other from the hardware's queue, and the epilogue warps
// store one unit's sums while the next one's products run.  192 columns instead of 256 for the registers that the sums take.
// Bound by shared memory: per k-block and SM 28 KB come in, are read and written twice by the converters and read by twelve matrix instructions (84 KB, or
// 120 with the half of B that comes from the other SM), 1530 to 1810 cycles at 128 bytes each, against 1180 cycles of tf32 arithmetic; a k-block
// takes 1960.  Two groups of two warps work on a stage each, so that one's waits and fence pass beside the other's arithmetic (one group of four
// with one unit per pair of CTAs took 2250), and the low parts have three places of their own beside four for the tiles.
// Microseconds, one unit per pair -> this; in brackets the route before either, pairs written to memory, a product that reads them and a sum over eight planes:
//   512 x 12288 x 4096  303 -> 277 (350)    1075 x 12288 x 4096  710 -> 642 (670)    800 x 4096 x 4096  223 -> 193 (187)
//   257 x 12288 x 256  32.6 -> 27.9 (21.7)  768 x 12288 x 256   49.3 -> 38.9 (33.9)  512 x 12288 x 512  49.6 -> 44.0 (124)
// What is left of the last route's lead lies where K is at most some 450 and 256 x 192 tiles fill a round badly; its error was larger everywhere.
constexpr int kX3N = 192, kX3Cols = kX3N / 2, kX3Slice = 2;
constexpr int kX3Stages = 4, kX3LoStages = 3;                 // fp32 tiles on their way, being worked on or read; their low parts
constexpr int kX3ConvWarps = 4, kX3Groups = 2;
constexpr int kX3Threads = kThreads + 32 * kX3ConvWarps;
constexpr uint32_t kX3BBytes = kX3Cols / 32 * 4096u;
constexpr uint32_t kX3Raw = kABytes + kX3BBytes;              // one stage of fp32 tiles; as much again for their low parts
constexpr uint32_t kX3StoreBytes = kEpiWarps * 32 * 64;       // 32 rows of 64 bytes per epilogue warp
constexpr uint32_t kX3BarBytes = 384;
constexpr uint32_t kX3Smem = (kX3Stages + kX3LoStages) * kX3Raw + kX3StoreBytes + 1024 + kX3BarBytes;
static_assert(kX3Smem <= 227 * 1024, "shared memory budget");
static_assert(kX3Raw % 1024 == 0, "tiles start on swizzle atoms");
static_assert(kX3LoStages < kX3Stages, "see the converters' wait for a free place");
constexpr uint32_t kX3Idesc = (1u << 4) | (2u << 7) | (2u << 10) | (1u << 16) | ((uint32_t)(kX3N >> 3) << 17) | ((uint32_t)(2 * BM >> 4) << 24);

struct X3Params {
    TcParams out;                   // M, N, C0..C2, ldc, csplit, plane; wait_ns, status
    int kb, kb0, per;               // k-blocks of 32 in all, of the first B, per K slice
    int a_k1, b_row1;               // where the blocks of the second B start in A's columns and in its rows
    int b3d;
};

// The pair of an fp32 value as bits: hi rounded to tf32 (half a unit added to the magnitude, what is below dropped), lo the rest, which the
// tensor core rounds the same way by dropping what is below half a unit more.  `bad` becomes NaN where that cannot be: the value or its hi is not finite.
__device__ __forceinline__ void x3_pair(float x, uint32_t& hi, uint32_t& lo, float& bad)
{
    hi = (__float_as_uint(x) + 0x1000u) & 0xffffe000u;
    const float rest = x - __uint_as_float(hi);
    bad = fmaf(rest, 0.0f, bad);
    lo = __float_as_uint(rest) + 0x1000u;
}
// ... for those: a NaN stays one, infinities give NaN, and what would round up to infinity is cut off instead
__device__ __forceinline__ void x3_pair_any(float x, uint32_t& hi, uint32_t& lo)
{
    const uint32_t u = __float_as_uint(x);
    if (!(fabsf(x) <= 3.402823466e38f)) {
        hi = lo = 0x7fc00000u;
        return;
    }
    hi = (u + 0x1000u) & 0xffffe000u;
    if ((hi & 0x7f800000u) == 0x7f800000u) hi = u & 0xffffe000u;
    lo = __float_as_uint(x - __uint_as_float(hi)) + 0x1000u;
}

__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(kX3Threads, 1)
gemm_x3_kernel(const __grid_constant__ CUtensorMap map_a, const __grid_constant__ CUtensorMap map_b0, const __grid_constant__ CUtensorMap map_b1,
               const X3Params prm)
{
    extern __shared__ uint8_t smem_raw[];
    const uint32_t raw = smem_u32(smem_raw);
    const uint32_t base = (raw + 1023u) & ~1023u;
    const uint32_t lo_base = base + kX3Stages * kX3Raw, staging = lo_base + kX3LoStages * kX3Raw;
    const uint32_t bars = staging + kX3StoreBytes;
    uint8_t* bars_gen = smem_raw + (bars - raw);
    auto full_bar = [&](int s) { return bars + 8u * s; };                        // this CTA's tiles are there
    auto conv_bar = [&](int s) { return bars + 8u * (kX3Stages + s); };          // leader: so are the pairs in both CTAs
    auto empty_bar = [&](int s) { return bars + 8u * (2 * kX3Stages + s); };
    auto acc_full_bar = [&](int a) { return bars + 8u * (3 * kX3Stages + a); };
    auto acc_empty_bar = [&](int a) { return bars + 8u * (3 * kX3Stages + 2 + a); };
    constexpr uint32_t kMisc = 8 * (3 * kX3Stages + 4);
    volatile uint32_t* tmem_slot = reinterpret_cast<volatile uint32_t*>(bars_gen + kMisc);
    volatile int* abort_flag = reinterpret_cast<volatile int*>(bars_gen + kMisc + 8);
    constexpr uint32_t kClc = (kMisc + 24 + 15) & ~15u;
    const uint32_t clc_bar = bars + kMisc + 16, clc_slot = bars + kClc;
    auto tile_bar = [&](int i) { return bars + kClc + 16u + 8u * i; };
    const uint32_t ring_base = bars + kClc + 16u + 8u * kRing;
    static_assert(kClc + 16 + 12 * kRing <= kX3BarBytes, "barriers and ring fit");

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int rank = (int)cluster_rank();
    const TcParams& out = prm.out;
    const int m_tiles = ceil_div(out.M, 2 * BM), mn_tiles = m_tiles * ceil_div(out.N, kX3N);
    const int first_tile = blockIdx.x >> 1;

    chain_next();
    if (threadIdx.x == 0) {
        for (int s = 0; s < kX3Stages; ++s) { mbar_init(full_bar(s), 1); mbar_init(conv_bar(s), 2 * kX3ConvWarps / kX3Groups); mbar_init(empty_bar(s), 1); }
        for (int a = 0; a < 2; ++a) { mbar_init(acc_full_bar(a), 1); mbar_init(acc_empty_bar(a), 2 * kEpiWarps); }
        mbar_init(clc_bar, 1);
        for (int i = 0; i < kRing; ++i) mbar_init(tile_bar(i), 1);
        *abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    }
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32((const void*)tmem_slot)), "r"(kTmemCols) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncwarp();
    cluster_sync();
    tc_fence_after();
    const uint32_t tmem_base = *tmem_slot;
    chain_wait();
    bool ok = true;

    // The units of a pair (a tile, or a K slice of one): the one that it was launched for, then what the leader's producer gets from the hardware's queue,
    // handed on through a ring as in gemm_tc_kernel.  The roles are at most kX3Stages + 3 units apart.
    auto next_tile = [&](uint32_t it) -> int {
        const int i = it % kRing;
        if (!mbar_wait_cluster(tile_bar(i), (it / kRing) & 1u, abort_flag, out.wait_ns)) { ok = false; return -1; }
        int t;
        asm volatile("ld.shared.s32 %0, [%1];" : "=r"(t) : "r"(ring_base + 4u * i) : "memory");
        return t;
    };
    auto blocks_of = [&](int tile) { return min(prm.kb - tile / mn_tiles * prm.per, prm.per); };

    if (warp == 0) {
        if (lane == 0) {
            uint32_t it = 0;
            bool asked = false;
            int tile = first_tile;
            for (uint32_t unit = 0; tile >= 0; ++unit) {
                const int mn = tile % mn_tiles, kb_lo = tile / mn_tiles * prm.per, blocks = blocks_of(tile);
                const int m0 = mn % m_tiles * 2 * BM + rank * BM, n0 = mn / m_tiles * kX3N + rank * kX3Cols;
                for (int b = 0; b < blocks; ++b, ++it) {
                    const int s = it % kX3Stages;
                    if (!mbar_wait(empty_bar(s), ((it / kX3Stages) & 1u) ^ 1u, abort_flag, out.wait_ns)) { ok = false; break; }
                    const uint32_t sa = base + s * kX3Raw, sb = sa + kABytes;
                    const int kb = kb_lo + b;
                    const bool second = kb >= prm.kb0;
                    const CUtensorMap* mb = second ? &map_b1 : &map_b0;
                    const int k = second ? prm.a_k1 + 32 * (kb - prm.kb0) : 32 * kb, row = second ? prm.b_row1 + 32 * (kb - prm.kb0) : 32 * kb;
                    mbar_expect_tx(full_bar(s), kX3Raw);
                    tma_load_2d(sa, &map_a, k, m0, full_bar(s));
                    if (prm.b3d) {
                        tma_load_3d(sb, mb, 0, row, n0 / 32, full_bar(s));
                    } else {
#pragma unroll
                        for (int j = 0; j < kX3Cols / 32; ++j) tma_load_2d(sb + j * 4096u, mb, n0 + 32 * j, row, full_bar(s));
                    }
                    // The next unit, while the last of this one's operands come in.  Asked for at once, it would be taken from a pair of SMs
                    // that is about to be free: 300 x 4096 x 504 25.9 -> 27.4 us, 32 calls of 512 rows on 32 lanes 3.74 -> 3.98 ms
                    if (rank == 0 && b == blocks - 1) {
                        mbar_expect_tx(clc_bar, 16);
                        clc_try_cancel(clc_slot, clc_bar);
                        asked = true;
                    }
                }
                if (rank == 0) {
                    if (asked && !mbar_wait(clc_bar, unit & 1u, abort_flag, out.wait_ns)) ok = false;
                    if (!ok) break;
                    asked = false;
                    const int x = clc_answer(clc_slot);
                    tile = x >= 0 ? x >> 1 : -1;
                    const uint32_t slot = ring_base + 4u * (unit % kRing), bar = tile_bar(unit % kRing);
                    asm volatile("st.shared.s32 [%0], %1;" ::"r"(slot), "r"(tile) : "memory");
                    asm volatile("st.shared::cluster.s32 [%0], %1;" ::"r"(map_rank(slot, 1)), "r"(tile) : "memory");
                    mbar_arrive_cluster(map_rank(bar, 1));
                    mbar_arrive(bar);
                } else {
                    if (!ok) break;
                    tile = next_tile(unit);
                }
            }
        }
    } else if (warp == 1) {
        if (lane == 0 && rank == 0) {
            uint32_t it = 0, run = 0;                         // stages, and runs of kX3Slice of them
            for (int tile = first_tile, unit = 0; tile >= 0 && ok; tile = ok ? next_tile(unit) : -1, ++unit) {
                const int blocks = blocks_of(tile);
                for (int b = 0; b < blocks; ++b, ++it) {
                    const int s = it % kX3Stages, a = run & 1;
                    if (b % kX3Slice == 0) {
                        if (!mbar_wait_cluster(acc_empty_bar(a), ((run >> 1) & 1u) ^ 1u, abort_flag, out.wait_ns)) { ok = false; break; }
                        tc_fence_after();
                    }
                    if (!mbar_wait_cluster(conv_bar(s), (it / kX3Stages) & 1u, abort_flag, out.wait_ns)) { ok = false; break; }
                    const uint32_t sa = base + s * kX3Raw, sl = lo_base + it % kX3LoStages * kX3Raw, d = tmem_base + 256u * a;
                    const uint64_t a_hi = smem_desc(sa, 16, 1024), a_lo = smem_desc(sl, 16, 1024);
                    const uint64_t b_hi = smem_desc(sa + kABytes, 4096, 512, 1), b_lo = smem_desc(sl + kABytes, 4096, 512, 1);
                    tc_mma4_tf32_pair(d, a_lo, b_hi, 2, 64, kX3Idesc, b % kX3Slice != 0);
                    tc_mma4_tf32_pair(d, a_hi, b_lo, 2, 64, kX3Idesc, 1);
                    tc_mma4_tf32_pair(d, a_hi, b_hi, 2, 64, kX3Idesc, 1);
                    tc_commit_pair(empty_bar(s));
                    if (b % kX3Slice == kX3Slice - 1 || b == blocks - 1) { tc_commit_pair(acc_full_bar(a)); ++run; }
                }
            }
        }
    } else if (warp < 2 + kEpiWarps) {
        const int quarter = warp & 3, half = (warp - 2) >> 2;
        const uint32_t buf = staging + (uint32_t)(warp - 2) * 2048u;
        uint32_t run = 0;
        for (int tile = first_tile, unit = 0; tile >= 0 && ok; tile = ok ? next_tile(unit) : -1, ++unit) {
            float sum[kX3Cols];
#pragma unroll
            for (int j = 0; j < kX3Cols; ++j) sum[j] = 0.0f;
            const int runs = ceil_div(blocks_of(tile), kX3Slice);
#pragma unroll 1
            for (int r = 0; r < runs; ++r, ++run) {
                const int a = run & 1;
                if (!mbar_wait(acc_full_bar(a), (run >> 1) & 1u, abort_flag, out.wait_ns)) { ok = false; break; }
                tc_fence_after();
                const uint32_t taddr = tmem_base + ((uint32_t)(quarter * 32) << 16) + 256u * a + (uint32_t)(half * kX3Cols);
#pragma unroll
                for (int c = 0; c < kX3Cols; c += 16) {
                    uint32_t v[16];
                    tc_ld_16cols(taddr + c, v);
                    tc_ld_wait();
#pragma unroll
                    for (int j = 0; j < 16; ++j) sum[c + j] += __uint_as_float(v[j]);
                }
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive_cluster(map_rank(acc_empty_bar(a), 0));
            }
            if (ok) {
                const int mn = tile % mn_tiles;
                const int m0 = mn % m_tiles * 2 * BM + rank * BM + quarter * 32, n0 = mn / m_tiles * kX3N + half * kX3Cols;
#pragma unroll
                for (int c = 0; c < kX3Cols; c += 16)
                    if (n0 + c < out.N) store_cols16(out, sum + c, buf, m0, n0 + c, lane, (long long)(tile / mn_tiles) * out.plane);
            }
        }
    } else {
        // converters: two warps per stage, two stages at a time, so that one's waits and fence pass beside the other's arithmetic
        const int group = (warp - 2 - kEpiWarps) / (kX3ConvWarps / kX3Groups);
        constexpr int kGroupThreads = 32 * kX3ConvWarps / kX3Groups, kEach = 14;
        constexpr int kRounds = kX3Raw / (16 * kGroupThreads * kEach);
        static_assert(kX3Raw % (16 * kGroupThreads * kEach) == 0, "whole rounds");
        const uint32_t t = 16u * ((threadIdx.x - kThreads) % kGroupThreads);
        uint32_t it = 0;
        for (int tile = first_tile, unit = 0; tile >= 0 && ok; tile = ok ? next_tile(unit) : -1, ++unit) {
            const int blocks = blocks_of(tile);
            for (int b = 0; b < blocks; ++b, ++it) {
                if (it % kX3Groups != group) continue;
                const int s = it % kX3Stages;
                if (!mbar_wait(full_bar(s), (it / kX3Stages) & 1u, abort_flag, out.wait_ns)) { ok = false; break; }
                if (it >= kX3LoStages) {
                    // the place of the low parts was last that of stage it - kX3LoStages; its barrier is at most one phase further, since the
                    // next one that it counts comes after this stage
                    const uint32_t old = it - kX3LoStages;
                    if (!mbar_wait(empty_bar(old % kX3Stages), (old / kX3Stages) & 1u, abort_flag, out.wait_ns)) { ok = false; break; }
                }
                const uint32_t hi_at = base + s * kX3Raw + t, lo_at = lo_base + it % kX3LoStages * kX3Raw + t;
#pragma unroll 1
                for (int r = 0; r < kRounds; ++r) {
                    const uint32_t off = r * (16u * kGroupThreads * kEach);
                    float x[kEach][4], bad = 0.0f;
#pragma unroll
                    for (int i = 0; i < kEach; ++i)           // all loads before the first store
                        asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(x[i][0]), "=f"(x[i][1]), "=f"(x[i][2]), "=f"(x[i][3])
                                     : "r"(hi_at + off + 16u * kGroupThreads * i) : "memory");
#pragma unroll
                    for (int i = 0; i < kEach; ++i) {
                        uint32_t h[4], l[4];
#pragma unroll
                        for (int j = 0; j < 4; ++j) x3_pair(x[i][j], h[j], l[j], bad);
                        asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(hi_at + off + 16u * kGroupThreads * i), "r"(h[0]), "r"(h[1]), "r"(h[2]), "r"(h[3]) : "memory");
                        asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(lo_at + off + 16u * kGroupThreads * i), "r"(l[0]), "r"(l[1]), "r"(l[2]), "r"(l[3]) : "memory");
                    }
                    if (bad != 0.0f) {
#pragma unroll
                        for (int i = 0; i < kEach; ++i) {
                            uint32_t h[4], l[4];
#pragma unroll
                            for (int j = 0; j < 4; ++j) x3_pair_any(x[i][j], h[j], l[j]);
                            asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(hi_at + off + 16u * kGroupThreads * i), "r"(h[0]), "r"(h[1]), "r"(h[2]), "r"(h[3]) : "memory");
                            asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(lo_at + off + 16u * kGroupThreads * i), "r"(l[0]), "r"(l[1]), "r"(l[2]), "r"(l[3]) : "memory");
                        }
                    }
                }
                asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                __syncwarp();
                if (lane == 0) mbar_arrive_cluster(map_rank(conv_bar(s), 0));
            }
        }
    }
    if (!ok) { *abort_flag = 1; atomicCAS(out.status, 0, (int)GELO_ERR_TIMEOUT); }

    tc_fence_before();
    __syncwarp();
    cluster_sync();
    if (warp == 1) {
        if (*abort_flag) settle(out.wait_ns);
        __syncwarp();
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(kTmemCols) : "memory");
    }
}

// ---- host side ----------------------------------------------------------------------------------

typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                  const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

// 2-D bf16 tensor map over a row-major matrix: `cols` contiguous elements per row, `rows` rows,
// row stride `ld` elements; box = box_cols x box_rows; 128-byte swizzle; zero fill out of bounds.
bool make_map(gelo_ctx* ctx, CUtensorMap* map, const void* ptr, uint64_t cols, uint64_t rows, uint64_t ld,
              uint32_t box_cols, uint32_t box_rows)
{
    EncodeTiledFn enc = reinterpret_cast<EncodeTiledFn>(ctx->tmap_encode);
    if (!enc) return false;
    const cuuint64_t dims[2] = { cols, rows };
    const cuuint64_t strides[1] = { ld * 2 };
    const cuuint32_t box[2] = { box_cols, box_rows };
    const cuuint32_t estr[2] = { 1, 1 };
    // (the copy engine only needs the element size and a zero fill: the same map serves IEEE half data)
    return enc(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void*>(ptr), dims, strides, box, estr,
               CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
               CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

bool aligned16(const void* p) { return (reinterpret_cast<uintptr_t>(p) & 15u) == 0; }

// Tensor map of an N-major operand tile: `box_rows` rows of k, `tile_cols` columns, held in shared memory as
// tile_cols / box_cols slabs of box_rows x 128 bytes (box_cols = 128 bytes of columns).  Where the rows are long
// enough, the matrix is described as a THREE-dimensional tensor {128 bytes of columns, rows, 128-byte column chunks}
// (strides: one row, 128 bytes), so that one copy instruction brings the whole tile in exactly that slab order; the
// producer thread then issues two copies per stage instead of up to nine (measured: 8% on the tf32 updates, nothing
// on the bf16 products).  In this view the last chunk of a row is read to its end even where it runs past
// `cols`, so it needs ld >= cols rounded up to a chunk (those columns only produce output columns that are never
// stored); otherwise *three_d = false and the map is the plain two-dimensional one (one copy per slab, zero fill
// past `cols`).  Rows past `rows` and chunks past the last one are zero-filled either way.
bool make_map_nmajor(gelo_ctx* ctx, CUtensorMap* map, const void* ptr, int elem_bytes, bool chunk32, uint64_t cols,
                     uint64_t rows, uint64_t ld, uint32_t box_rows, uint32_t tile_cols, bool* three_d)
{
    EncodeTiledFn enc = reinterpret_cast<EncodeTiledFn>(ctx->tmap_encode);
    if (!enc) return false;
    const uint32_t box_cols = 128u / (uint32_t)elem_bytes;
    const CUtensorMapDataType dt = elem_bytes == 4 ? CU_TENSOR_MAP_DATA_TYPE_FLOAT32
                                 : elem_bytes == 1 ? CU_TENSOR_MAP_DATA_TYPE_UINT8 : CU_TENSOR_MAP_DATA_TYPE_BFLOAT16;
    const CUtensorMapSwizzle sw = chunk32 ? CU_TENSOR_MAP_SWIZZLE_128B_ATOM_32B : CU_TENSOR_MAP_SWIZZLE_128B;
    const uint64_t chunks = (cols + box_cols - 1) / box_cols;
    if (ctx->tma_3d && ld >= chunks * box_cols && tile_cols / box_cols > 1) {
        const cuuint64_t dims[3] = { box_cols, rows, chunks };
        const cuuint64_t strides[2] = { ld * (uint64_t)elem_bytes, 128 };
        const cuuint32_t box[3] = { box_cols, box_rows, tile_cols / box_cols };
        const cuuint32_t estr[3] = { 1, 1, 1 };
        if (enc(map, dt, 3, const_cast<void*>(ptr), dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE, sw,
                CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS) {
            *three_d = true;
            return true;
        }
    }
    *three_d = false;
    const cuuint64_t dims[2] = { cols, rows };
    const cuuint64_t strides[1] = { ld * (uint64_t)elem_bytes };
    const cuuint32_t box[2] = { box_cols, box_rows };
    const cuuint32_t estr[2] = { 1, 1 };
    return enc(map, dt, 2, const_cast<void*>(ptr), dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE, sw,
               CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// CTAs that a launch should plan for: all SMs, or a lane's share of them in a batch (no limit: the tiles go wherever an SM is
// free)
int launch_width(const gelo_ctx* ctx, int mode)
{
    return (mode != TC_STORE_BF16 && ctx->tc_update_ctas > 0 && ctx->tc_update_ctas < ctx->sm_count) ? ctx->tc_update_ctas : ctx->sm_count;
}

// Work items of a product: 256 columns, 128 rows (256 in a pair), times the K slices; symmetric products leave out what
// lies below the diagonal.
int tile_count(int M, int N, int slices, bool tri, bool pair)
{
    const int m_tiles = ceil_div(M, pair ? 2 * BM : BM), n_tiles = ceil_div(N, 256);
    if (!tri) return m_tiles * n_tiles * slices;
    int tiles = 0;
    for (int nt = 0; nt < n_tiles; ++nt) {
        const int own = pair ? nt + 1 : 2 * nt + 2;
        tiles += m_tiles < own ? m_tiles : own;
    }
    return tiles;
}

// Whether a product runs on pairs of CTAs.  A 256 x 256 tile of a pair takes its two SMs no longer than a 128 x 256 tile takes
// one (each SM stages half of B, a third less in all, in six stages instead of four), so the pair wins unless the coarser
// tiles need more rounds.  Measured with the staged stores, single -> pair: 4300 x 12288 x 4096 in bf16 323 -> 292 us (1.34 -> 1.48
// PFLOP/s), 2150 rows 196 -> 166 us, E4M3 operands 2.01 -> 2.37 PFLOP/s at 4300 rows; 1050 x 4096 x 1050, where 144 single tiles make
// one round and 80 pair tiles two, stays single (18.5 us).
bool use_pair(const gelo_ctx* ctx, int M, int N, int slices, bool tri, int mode)
{
    const int width = launch_width(ctx, mode);
    if (M <= BM || width < 2) return false;
    return ceil_div(tile_count(M, N, slices, tri, true), width / 2) <= ceil_div(tile_count(M, N, slices, tri, false), width);
}

template <int BN, bool kStaging, bool kTf32, bool kAMn, bool kF8, bool kPair, bool kShare = false>
int launch_tiles_as(gelo_ctx* ctx, const CUtensorMap& a0, const CUtensorMap& a1, const CUtensorMap& b0, const CUtensorMap& b1,
                    const CUtensorMap& c, const TcParams& p, double flops, cudaStream_t st)
{
    using Cfg = TcCfg<BN, kStaging, kTf32, kAMn, kF8, kPair>;
    static_assert(Cfg::kSmemBytes <= 227 * 1024, "shared memory budget");
    auto kernel = gemm_tc_kernel<BN, kStaging, kTf32, kAMn, kF8, kPair, kShare>;
    static bool attr_done[64] = {};
    if (ctx->device >= 0 && ctx->device < 64 && !attr_done[ctx->device]) {
        GELO_CUDA_OK(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)Cfg::kSmemBytes));
        attr_done[ctx->device] = true;
    }
    TcParams q = p;
    if (p.tri) q.tri_tiles = tile_count(p.M, p.N, 1, true, kPair);
    const int tiles = p.tri ? q.tri_tiles : ceil_div(p.M, Cfg::kTileRows) * ceil_div(p.N, BN) * p.ksplit;
    // both operands of a kind::f16 instruction have the same 16-bit format: 1 = bfloat16, 0 = IEEE half
    q.wait_ns = ctx->wait_limit_ns;
    q.idesc = (!kTf32 && !kF8 && p.out_f16) ? (Cfg::kInstrDesc & ~((7u << 7) | (7u << 10))) : Cfg::kInstrDesc;
    {
        ProfScope ps(ctx, PROF_GEMM_TC, flops, st);
        cudaLaunchConfig_t cfg = {};
        q.tiles = tiles;
        q.stride = kShare ? std::min(tiles, ctx->tc_update_ctas / (kPair ? 2 : 1)) : tiles;
        cfg.gridDim = dim3(q.stride * (kPair ? 2 : 1));
        cfg.blockDim = dim3(kThreads);
        cfg.dynamicSmemBytes = Cfg::kSmemBytes;
        cfg.stream = st;
        cudaLaunchAttribute attr[2];
        attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
        attr[0].val.programmaticStreamSerializationAllowed = chain_launches(ctx) ? 1 : 0;
        attr[1].id = cudaLaunchAttributeClusterDimension;
        attr[1].val.clusterDim.x = 2; attr[1].val.clusterDim.y = 1; attr[1].val.clusterDim.z = 1;
        cfg.attrs = attr;
        cfg.numAttrs = kPair ? 2 : 1;
        GELO_CUDA_OK(cudaLaunchKernelEx(&cfg, kernel, a0, a1, b0, b1, c, q));
    }
    return after_launch(ctx);
}

template <int BN, bool kStaging, bool kTf32 = false, bool kAMn = false, bool kF8 = false>
int launch_tiles(gelo_ctx* ctx, bool pair, const CUtensorMap& a0, const CUtensorMap& a1, const CUtensorMap& b0, const CUtensorMap& b1,
                 const CUtensorMap& c, const TcParams& p, double flops, cudaStream_t st)
{
    if constexpr (BN == 256 && kTf32) {                       // (launches that may not have the whole GPU are planned with 256 columns)
        if (ctx->tc_cap)
            return pair ? launch_tiles_as<BN, kStaging, kTf32, kAMn, kF8, true, true>(ctx, a0, a1, b0, b1, c, p, flops, st)
                        : launch_tiles_as<BN, kStaging, kTf32, kAMn, kF8, false, true>(ctx, a0, a1, b0, b1, c, p, flops, st);
    }
    if constexpr (BN == 256) {
        if (pair) return launch_tiles_as<BN, kStaging, kTf32, kAMn, kF8, true>(ctx, a0, a1, b0, b1, c, p, flops, st);
    }
    return launch_tiles_as<BN, kStaging, kTf32, kAMn, kF8, false>(ctx, a0, a1, b0, b1, c, p, flops, st);
}

// tf32 products on tiles of 64, 128 or 256 columns
template <bool kStaging, bool kAMn>
int launch_tf32_cols(gelo_ctx* ctx, int cols, bool pair, const CUtensorMap& a0, const CUtensorMap& a1, const CUtensorMap& b0,
                     const CUtensorMap& b1, const CUtensorMap& c, const TcParams& p, double flops, cudaStream_t st)
{
    if (cols == 64) return launch_tiles<64, kStaging, true, kAMn>(ctx, false, a0, a1, b0, b1, c, p, flops, st);
    if (cols == 128) return launch_tiles<128, kStaging, true, kAMn>(ctx, false, a0, a1, b0, b1, c, p, flops, st);
    return launch_tiles<256, kStaging, true, kAMn>(ctx, pair, a0, a1, b0, b1, c, p, flops, st);
}

// fp32 tensor map of the matrix that the subtracting epilogue reduces into: 32 x 32 boxes, 128-byte swizzle.
bool make_map_f32_box(gelo_ctx* ctx, CUtensorMap* map, const void* ptr, uint64_t cols, uint64_t rows, uint64_t ld,
                      uint32_t box_rows = 32, bool chunk32 = false)
{
    EncodeTiledFn enc = reinterpret_cast<EncodeTiledFn>(ctx->tmap_encode);
    if (!enc) return false;
    const cuuint64_t dims[2] = { cols, rows };
    const cuuint64_t strides[1] = { ld * 4 };
    const cuuint32_t box[2] = { 32, box_rows };
    const cuuint32_t estr[2] = { 1, 1 };
    // chunk32: the 128-byte swizzle that moves 32-byte chunks, which the MMA wants for fp32 tiles that are not K-major
    return enc(map, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 2, const_cast<void*>(ptr), dims, strides, box, estr,
               CU_TENSOR_MAP_INTERLEAVE_NONE, chunk32 ? CU_TENSOR_MAP_SWIZZLE_128B_ATOM_32B : CU_TENSOR_MAP_SWIZZLE_128B,
               CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
               CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

}  // namespace

// Columns of a tile of an M x N x K product of elements of `bytes` bytes.  A product that fills no more than a part of the GPU is
// bound by what one tile takes from its first copy to its last store, and most of that goes with the columns: 128 x 512 x (2 x 128)
// in tf32 takes 11.4 us on 256 columns per tile and 7.7 us on 64.  So the narrowest tiles that still run in one round are
// taken, as long as what all of them read, which narrow tiles multiply, does not become the bound (512 x 1638 x 2150 reads 170 MB on
// 64 columns: 27 us, against 17 us on 256 with the depth in four slices).  In the lanes of a batch SM time counts, and 256 columns
// use it best.
int gemm_tile_cols(const gelo_ctx* ctx, int M, int N, int K, int slices, int bytes, bool lanes_share, int least)
{
    if (ctx->tc_update_ctas > 0 && lanes_share) return 256;
    for (int cols = least; cols < 256; cols *= 2) {
        const long tiles = (long)ceil_div(M, BM) * ceil_div(N, cols);
        if (tiles * slices <= ctx->sm_count && (double)tiles * K * (BM + cols) * bytes <= 48e6) return cols;
    }
    return 256;
}

bool gemm_tc_supports(const GemmArgs& g)
{
    if (g.dtype == GELO_F32 || g.transA || g.transB || g.alpha != 1.0f || g.beta != 0.0f) return false;
    if (g.M <= 0 || g.N <= 0 || g.K <= 0) return false;
    if ((g.lda % 8) || (g.ldb % 8) || (g.ldc % 8) || (g.N % 8)) return false;
    if (g.nsplit < 1 || g.nsplit > 3 || g.N % g.nsplit || ((g.N / g.nsplit) % 8)) return false;
    if (!aligned16(g.A) || !aligned16(g.B) || (g.B2 && !aligned16(g.B2))) return false;
    for (int i = 0; i < g.nsplit; ++i)
        if (!g.C[i] || !aligned16(g.C[i])) return false;
    if (g.B2 && (g.b_split <= 0 || g.b_split >= g.K)) return false;
    return true;
}

int launch_gemm_tc(gelo_ctx* ctx, const GemmArgs& g, cudaStream_t st)
{
    if (!gemm_tc_supports(g)) return GELO_ERR_UNSUPPORTED;
    if (!ctx->tmap_encode) return GELO_ERR_CUDA;
    constexpr int BN = 256;
    const int rows_first = g.B2 ? g.b_split : g.K;
    const int wide = gemm_tile_cols(ctx, g.M, g.N, g.K, 1, 2, false, 128);
    const bool pair = wide == BN && use_pair(ctx, g.M, g.N, 1, false, TC_STORE_BF16);
    const uint32_t cols = pair ? BN / 2 : wide;               // columns of B per CTA
    CUtensorMap ma, mb, mb2;
    if (!make_map(ctx, &ma, g.A, (uint64_t)g.K, (uint64_t)g.M, (uint64_t)g.lda, BK, BM)) return GELO_ERR_CUDA;
    bool b3d = false, b3d2 = false;
    if (!make_map_nmajor(ctx, &mb, g.B, 2, false, (uint64_t)g.N, (uint64_t)rows_first, (uint64_t)g.ldb, BK, cols, &b3d)) return GELO_ERR_CUDA;
    if (g.B2) {
        if (!make_map_nmajor(ctx, &mb2, g.B2, 2, false, (uint64_t)g.N, (uint64_t)(g.K - g.b_split), (uint64_t)g.ldb, BK, cols, &b3d2))
            return GELO_ERR_CUDA;
        if (b3d2 != b3d) return GELO_ERR_CUDA;                // same width and stride: the same decision
    } else {
        mb2 = mb;
    }
    TcParams p = {};
    p.M = g.M; p.N = g.N;
    p.nseg = 1;
    p.seg[0] = TcSegment{0, 0, 0, 0, ceil_div(rows_first, BK)};
    if (g.B2) {
        const int a_k0 = g.b_split & ~7;                      // TMA needs a 16-byte aligned inner coordinate
        p.nseg = 2;
        p.seg[1] = TcSegment{0, 1, a_k0, a_k0 - g.b_split /* <= 0: rows above S read as zero */,
                             ceil_div(g.K - a_k0, BK)};
    }
    p.ksplit = 1; p.kb_per_split = 1 << 30; p.plane = 0;
    p.mode = TC_STORE_BF16;
    p.b3d = b3d ? 1 : 0;
    p.out_f16 = g.dtype == GELO_F16 ? 1 : 0;
    p.C0 = g.C[0]; p.C1 = g.C[g.nsplit > 1 ? 1 : 0]; p.C2 = g.C[g.nsplit > 2 ? 2 : 0];
    p.ldc = g.ldc; p.csplit = g.N / g.nsplit; p.lde = 0;
    p.status = ctx->status_dev;
    if (wide == 128) return launch_tiles<128, false>(ctx, false, ma, ma, mb, mb2, ma, p, 2.0 * g.M * (double)g.N * g.K, st);
    return launch_tiles<BN, false>(ctx, pair, ma, ma, mb, mb2, ma, p, 2.0 * g.M * (double)g.N * g.K, st);
}

// Split-precision product for the factorisations.  A = Ahi + Alo (M x K, stride lda), B = Bhi + Blo
// (K x N, stride ldb), all bf16; the tensor cores accumulate Ahi Bhi + Ahi Blo + Alo Bhi in fp32.
//   sub_from != nullptr : sub_from (fp32, stride ldc) -= product, and if emit_hi != nullptr the updated
//                         values are also written as a (hi, lo) pair with stride lde
//   sub_from == nullptr : the product itself is written as the pair (emit_hi, emit_lo), stride lde
int launch_gemm_tc_split(gelo_ctx* ctx, int M, int N, int K, const void* Ahi, const void* Alo, int lda,
                         const void* Bhi, const void* Blo, int ldb, float* sub_from, int ldc, void* emit_hi,
                         void* emit_lo, int lde, bool narrow_tiles, cudaStream_t st)
{
    if (M <= 0 || N <= 0 || K <= 0) return GELO_OK;
    if (!ctx->tmap_encode) return GELO_ERR_CUDA;
    if ((lda % 8) || (ldb % 8) || (!sub_from && (N % 8)) || !aligned16(Ahi) || !aligned16(Alo) || !aligned16(Bhi) || !aligned16(Blo))
        return GELO_ERR_INVALID;
    if (sub_from && ((ldc % 4) || !aligned16(sub_from))) return GELO_ERR_INVALID;
    if (emit_hi && ((lde % 8) || !aligned16(emit_hi) || !aligned16(emit_lo))) return GELO_ERR_INVALID;
    if (!sub_from && !emit_hi) return GELO_ERR_INVALID;
    CUtensorMap a0, a1, b0, b1;
    const bool pair = (sub_from || !narrow_tiles) && use_pair(ctx, M, N, 1, false, TC_SUB_F32);
    const uint32_t tile_cols = (!sub_from && narrow_tiles) ? 64 : (pair ? 128 : 256);
    bool b3d = false, b3d1 = false;
    if (!make_map(ctx, &a0, Ahi, (uint64_t)K, (uint64_t)M, (uint64_t)lda, BK, BM) ||
        !make_map(ctx, &a1, Alo, (uint64_t)K, (uint64_t)M, (uint64_t)lda, BK, BM) ||
        !make_map_nmajor(ctx, &b0, Bhi, 2, false, (uint64_t)N, (uint64_t)K, (uint64_t)ldb, BK, tile_cols, &b3d) ||
        !make_map_nmajor(ctx, &b1, Blo, 2, false, (uint64_t)N, (uint64_t)K, (uint64_t)ldb, BK, tile_cols, &b3d1) || b3d != b3d1)
        return GELO_ERR_CUDA;
    TcParams p = {};
    p.M = M; p.N = N;
    const int kb = ceil_div(K, BK);
    p.nseg = 3;
    p.seg[0] = TcSegment{0, 0, 0, 0, kb};
    p.seg[1] = TcSegment{0, 1, 0, 0, kb};
    p.seg[2] = TcSegment{1, 0, 0, 0, kb};
    p.status = ctx->status_dev;
    p.csplit = N;
    p.b3d = b3d ? 1 : 0;
    p.ksplit = 1; p.kb_per_split = 1 << 30; p.plane = 0;
    CUtensorMap mc = a0;
    if (sub_from) {
        if (emit_hi) return GELO_ERR_UNSUPPORTED;
        if (!make_map_f32_box(ctx, &mc, sub_from, (uint64_t)N, (uint64_t)M, (uint64_t)ldc)) return GELO_ERR_CUDA;
        p.mode = TC_SUB_F32;
        p.C0 = sub_from; p.ldc = ldc;
    } else {
        p.mode = TC_EMIT_SPLIT;
        p.C0 = emit_hi; p.C1 = emit_lo; p.ldc = lde; p.lde = lde;
    }
    const double flops = 6.0 * M * (double)N * K;
    if (sub_from) return launch_tiles<256, true>(ctx, pair, a0, a1, b0, b1, mc, p, flops, st);
    if (narrow_tiles) return launch_tiles<64, false>(ctx, pair, a0, a1, b0, b1, mc, p, flops, st);
    return launch_tiles<256, false>(ctx, pair, a0, a1, b0, b1, mc, p, flops, st);
}


int launch_gemm_tc_split_k(gelo_ctx* ctx, int M, int N, int K, const void* Ahi, const void* Alo, int lda, const void* Bhi,
                           const void* Blo, int ldb, float* planes, size_t plane, int ldp, int ksplit, int* used,
                           cudaStream_t st)
{
    if (used) *used = 0;
    if (M <= 0 || N <= 0 || K <= 0) return GELO_OK;
    if (!ctx->tmap_encode) return GELO_ERR_CUDA;
    if ((lda % 8) || (ldb % 8) || (N % 8) || (ldp % 4) || !aligned16(Ahi) || !aligned16(Alo) || !aligned16(Bhi) ||
        !aligned16(Blo) || !aligned16(planes) || (plane % 4) || ksplit < 1)
        return GELO_ERR_INVALID;
    const int kb = ceil_div(K, BK);
    if (ksplit > kb) ksplit = kb;
    const int per = ceil_div(kb, ksplit);
    ksplit = ceil_div(kb, per);                    // no empty slice
    const bool pair = use_pair(ctx, M, N, ksplit, false, TC_STORE_F32);
    const uint32_t cols = pair ? 128 : 256;
    CUtensorMap a0, a1, b0, b1;
    bool b3d = false, b3d1 = false;
    if (!make_map(ctx, &a0, Ahi, (uint64_t)K, (uint64_t)M, (uint64_t)lda, BK, BM) ||
        !make_map(ctx, &a1, Alo, (uint64_t)K, (uint64_t)M, (uint64_t)lda, BK, BM) ||
        !make_map_nmajor(ctx, &b0, Bhi, 2, false, (uint64_t)N, (uint64_t)K, (uint64_t)ldb, BK, cols, &b3d) ||
        !make_map_nmajor(ctx, &b1, Blo, 2, false, (uint64_t)N, (uint64_t)K, (uint64_t)ldb, BK, cols, &b3d1) || b3d != b3d1)
        return GELO_ERR_CUDA;
    TcParams p = {};
    p.M = M; p.N = N;
    p.nseg = 3;
    p.seg[0] = TcSegment{0, 0, 0, 0, kb};
    p.seg[1] = TcSegment{0, 1, 0, 0, kb};
    p.seg[2] = TcSegment{1, 0, 0, 0, kb};
    p.status = ctx->status_dev;
    p.csplit = N;
    p.b3d = b3d ? 1 : 0;
    p.mode = TC_STORE_F32;
    p.C0 = planes; p.ldc = ldp; p.lde = 0;
    p.ksplit = ksplit; p.kb_per_split = per; p.plane = (long long)plane;
    if (used) *used = ksplit;
    return launch_tiles<256, false>(ctx, pair, a0, a1, b0, b1, a0, p, 6.0 * M * (double)N * K, st);
}

// One-product tf32 GEMM on fp32 matrices, fp32 accumulation:  P = op(A) (M x K) * B (K x N, row-major, stride ldb).
//   a_mn = false : A is row-major M x K (stride lda);  a_mn = true : A points at a row-major K x M matrix (stride lda)
//                  and the product uses its transpose.
//   mode TC_SUB_F32   : C (fp32, stride ldc) -= P, in place, by TMA reduce-add
//   mode TC_STORE_F32 : C = P, or with round_out C = post_scale * (out_scale * P - diag_sub * I) rounded to tf32, or
//                       with ksplit > 1 the partial products of the K slices
//                       go to consecutive planes of C (plane stride in elements); *used = slices written
int launch_gemm_tf32(gelo_ctx* ctx, int M, int N, int K, const float* A, int lda, bool a_mn, const float* B, int ldb,
                     bool subtract, float* C, int ldc, bool round_out, float out_scale, int ksplit, size_t plane, int* used,
                     cudaStream_t st, float diag_sub, float post_scale)
{
    if (used) *used = 0;
    if (M <= 0 || N <= 0 || K <= 0) return GELO_OK;
    if (!ctx->tmap_encode) return GELO_ERR_CUDA;
    if ((lda % 4) || (ldb % 4) || (ldc % 4) || !aligned16(A) || !aligned16(B) || !aligned16(C) || !C) return GELO_ERR_INVALID;
    if (!subtract && (N % 8)) return GELO_ERR_INVALID;
    if (subtract && ksplit > 1) return GELO_ERR_INVALID;
    const int kb = ceil_div(K, 32);
    int per = kb;
    if (ksplit > 1) {
        if (ksplit > kb) ksplit = kb;
        per = ceil_div(kb, ksplit);
        ksplit = ceil_div(kb, per);                // no empty slice
    } else {
        ksplit = 1;
    }
    const int wide = gemm_tile_cols(ctx, M, N, K, ksplit, 4, true, 64);
    const bool pair = wide == 256 && use_pair(ctx, M, N, ksplit, false, subtract ? TC_SUB_F32 : TC_STORE_F32);
    const uint32_t cols = pair ? 128 : wide;
    CUtensorMap ma, mb, mc;
    bool a3d = false, b3d = false;
    const bool a_ok = a_mn ? make_map_nmajor(ctx, &ma, A, 4, true, (uint64_t)M, (uint64_t)K, (uint64_t)lda, 32, BM, &a3d)
                           : make_map_f32_box(ctx, &ma, A, (uint64_t)K, (uint64_t)M, (uint64_t)lda, BM);
    if (!a_ok || !make_map_nmajor(ctx, &mb, B, 4, true, (uint64_t)N, (uint64_t)K, (uint64_t)ldb, 32, cols, &b3d)) return GELO_ERR_CUDA;
    mc = ma;
    TcParams p = {};
    p.M = M; p.N = N;
    p.nseg = 1;
    p.seg[0] = TcSegment{0, 0, 0, 0, kb};
    p.status = ctx->status_dev;
    p.csplit = N;
    p.ksplit = 1; p.kb_per_split = 1 << 30; p.plane = 0;
    p.a3d = a3d ? 1 : 0; p.b3d = b3d ? 1 : 0;
    p.round_tf32 = round_out ? 1 : 0;
    p.out_scale = out_scale; p.diag_sub = diag_sub; p.post_scale = post_scale;
    p.C0 = C; p.ldc = ldc;
    const double flops = 2.0 * M * (double)N * K;
    if (subtract) {
        if (!make_map_f32_box(ctx, &mc, C, (uint64_t)N, (uint64_t)M, (uint64_t)ldc, 32)) return GELO_ERR_CUDA;
        p.mode = TC_SUB_F32;
        return a_mn ? launch_tf32_cols<true, true>(ctx, wide, pair, ma, ma, mb, mb, mc, p, flops, st)
                    : launch_tf32_cols<true, false>(ctx, wide, pair, ma, ma, mb, mb, mc, p, flops, st);
    }
    p.mode = TC_STORE_F32;
    if (ksplit > 1) { p.ksplit = ksplit; p.kb_per_split = per; p.plane = (long long)plane; }
    if (used) *used = p.ksplit;
    return a_mn ? launch_tf32_cols<false, true>(ctx, wide, pair, ma, ma, mb, mb, mc, p, flops, st)
                : launch_tf32_cols<false, false>(ctx, wide, pair, ma, ma, mb, mb, mc, p, flops, st);
}

// C = out_scale * (A0 B0 + A1 B1) rounded to tf32: two products of the same sizes in one accumulator.
int launch_gemm_tf32_dual(gelo_ctx* ctx, int M, int N, int K, const float* A0, int lda0, const float* B0, int ldb0, const float* A1,
                          int lda1, const float* B1, int ldb1, float* C, int ldc, float out_scale, cudaStream_t st)
{
    if (M <= 0 || N <= 0 || K <= 0) return GELO_OK;
    if (!ctx->tmap_encode) return GELO_ERR_CUDA;
    if ((lda0 % 4) || (lda1 % 4) || (ldb0 % 4) || (ldb1 % 4) || (ldc % 4) || (N % 8) || !aligned16(A0) || !aligned16(A1) ||
        !aligned16(B0) || !aligned16(B1) || !aligned16(C))
        return GELO_ERR_INVALID;
    const int wide = gemm_tile_cols(ctx, M, N, 2 * K, 1, 4, true, 64);
    const bool pair = wide == 256 && use_pair(ctx, M, N, 1, false, TC_STORE_F32);
    const uint32_t cols = pair ? 128 : wide;
    CUtensorMap a0, a1, b0, b1;
    bool b3d = false, b3d1 = false;
    if (!make_map_f32_box(ctx, &a0, A0, (uint64_t)K, (uint64_t)M, (uint64_t)lda0, BM) ||
        !make_map_f32_box(ctx, &a1, A1, (uint64_t)K, (uint64_t)M, (uint64_t)lda1, BM) ||
        !make_map_nmajor(ctx, &b0, B0, 4, true, (uint64_t)N, (uint64_t)K, (uint64_t)ldb0, 32, cols, &b3d) ||
        !make_map_nmajor(ctx, &b1, B1, 4, true, (uint64_t)N, (uint64_t)K, (uint64_t)ldb1, 32, cols, &b3d1) || b3d != b3d1)
        return GELO_ERR_CUDA;
    TcParams p = {};
    p.M = M; p.N = N;
    const int kb = ceil_div(K, 32);
    p.nseg = 2;
    p.seg[0] = TcSegment{0, 0, 0, 0, kb};
    p.seg[1] = TcSegment{1, 1, 0, 0, kb};
    p.status = ctx->status_dev;
    p.csplit = N;
    p.ksplit = 1; p.kb_per_split = 1 << 30; p.plane = 0;
    p.b3d = b3d ? 1 : 0;
    p.round_tf32 = 1;
    p.out_scale = out_scale; p.post_scale = 1.0f;
    p.C0 = C; p.ldc = ldc;
    p.mode = TC_STORE_F32;
    return launch_tf32_cols<false, false>(ctx, wide, pair, a0, a1, b0, b1, a0, p, 4.0 * M * (double)N * K, st);
}

// D (m x m bf16, stride ldd) = post_scale * (out_scale * Q^T Q - diag_sub I) for a row-major fp32 Q (stride ld): one
// tf32 product in which only the tiles on and above the diagonal are computed (Q^T Q is symmetric) and the rest is
// mirrored by the epilogue.  ldd >= m rounded up to 8.
int launch_gram_sym_bf16(gelo_ctx* ctx, int m, const float* Q, int ld, void* D, int ldd, float out_scale, float diag_sub,
                         float post_scale, cudaStream_t st)
{
    if (m <= 0) return GELO_OK;
    if (!ctx->tmap_encode) return GELO_ERR_CUDA;
    const int m8 = (m + 7) & ~7;
    if ((ld % 4) || ld < m8 || (ldd % 8) || ldd < m8 || !aligned16(Q) || !aligned16(D)) return GELO_ERR_INVALID;
    const bool pair = use_pair(ctx, m, m8, 1, true, TC_STORE_SYM16);
    const uint32_t cols = pair ? 128 : 256;
    CUtensorMap ma, mb;
    bool a3d = false, b3d = false;
    if (!make_map_nmajor(ctx, &ma, Q, 4, true, (uint64_t)m, (uint64_t)m, (uint64_t)ld, 32, BM, &a3d) ||
        !make_map_nmajor(ctx, &mb, Q, 4, true, (uint64_t)m8, (uint64_t)m, (uint64_t)ld, 32, cols, &b3d))
        return GELO_ERR_CUDA;
    TcParams p = {};
    p.M = m; p.N = m8;
    p.nseg = 1;
    p.seg[0] = TcSegment{0, 0, 0, 0, ceil_div(m, 32)};
    p.status = ctx->status_dev;
    p.csplit = m8;
    p.ksplit = 1; p.kb_per_split = 1 << 30; p.plane = 0;
    p.a3d = a3d ? 1 : 0; p.b3d = b3d ? 1 : 0;
    p.out_scale = out_scale; p.diag_sub = diag_sub; p.post_scale = post_scale;
    p.C0 = D; p.ldc = ldd;
    p.mode = TC_STORE_SYM16;
    p.tri = 1;
    return launch_tiles<256, false, true, true>(ctx, pair, ma, ma, mb, mb, ma, p, 2.0 * m * (double)m * m, st);
}

// C (M x N fp32, stride ldc) -= A (M x K bf16, stride lda) * B (K x N bf16, stride ldb), in place by TMA reduce-add.
int launch_gemm_bf16_sub(gelo_ctx* ctx, int M, int N, int K, const void* A, int lda, const void* B, int ldb, float* C, int ldc,
                         cudaStream_t st)
{
    if (M <= 0 || N <= 0 || K <= 0) return GELO_OK;
    if (!ctx->tmap_encode) return GELO_ERR_CUDA;
    if ((lda % 8) || (ldb % 8) || (ldc % 4) || !aligned16(A) || !aligned16(B) || !aligned16(C)) return GELO_ERR_INVALID;
    const bool pair = use_pair(ctx, M, N, 1, false, TC_SUB_F32);
    const uint32_t cols = pair ? 128 : 256;
    CUtensorMap ma, mb, mc;
    bool b3d = false;
    if (!make_map(ctx, &ma, A, (uint64_t)K, (uint64_t)M, (uint64_t)lda, BK, BM) ||
        !make_map_nmajor(ctx, &mb, B, 2, false, (uint64_t)N, (uint64_t)K, (uint64_t)ldb, BK, cols, &b3d) ||
        !make_map_f32_box(ctx, &mc, C, (uint64_t)N, (uint64_t)M, (uint64_t)ldc))
        return GELO_ERR_CUDA;
    TcParams p = {};
    p.M = M; p.N = N;
    p.nseg = 1;
    p.seg[0] = TcSegment{0, 0, 0, 0, ceil_div(K, BK)};
    p.status = ctx->status_dev;
    p.csplit = N;
    p.b3d = b3d ? 1 : 0;
    p.ksplit = 1; p.kb_per_split = 1 << 30; p.plane = 0;
    p.mode = TC_SUB_F32;
    p.C0 = C; p.ldc = ldc;
    return launch_tiles<256, true>(ctx, pair, ma, ma, mb, mb, mc, p, 2.0 * M * (double)N * K, st);
}

// C (M x N, 16-bit type of the operands) = sign * A (M x K) B (K x N) + diag I + add_scale * add (optional, M x N)
int launch_gemm_affine16(gelo_ctx* ctx, int dtype, int M, int N, int K, const void* A, int lda, const void* B, int ldb, float sign,
                         float diag, const void* add, int ldadd, float add_scale, void* C, int ldc, cudaStream_t st)
{
    if (M <= 0 || N <= 0 || K <= 0) return GELO_OK;
    if (!ctx->tmap_encode) return GELO_ERR_CUDA;
    if ((lda % 8) || (ldb % 8) || (ldc % 8) || (N % 8) || (ldadd % 8) || !aligned16(A) || !aligned16(B) || !aligned16(C) ||
        !aligned16(add))
        return GELO_ERR_INVALID;
    const int wide = gemm_tile_cols(ctx, M, N, K, 1, 2, true, 128);
    const bool pair = wide == 256 && use_pair(ctx, M, N, 1, false, TC_AFFINE16);
    const uint32_t cols = pair ? 128 : wide;
    CUtensorMap ma, mb;
    bool b3d = false;
    if (!make_map(ctx, &ma, A, (uint64_t)K, (uint64_t)M, (uint64_t)lda, BK, BM) ||
        !make_map_nmajor(ctx, &mb, B, 2, false, (uint64_t)N, (uint64_t)K, (uint64_t)ldb, BK, cols, &b3d))
        return GELO_ERR_CUDA;
    TcParams p = {};
    p.M = M; p.N = N;
    p.nseg = 1;
    p.seg[0] = TcSegment{0, 0, 0, 0, ceil_div(K, BK)};
    p.ksplit = 1; p.kb_per_split = 1 << 30; p.plane = 0;
    p.mode = TC_AFFINE16;
    p.b3d = b3d ? 1 : 0;
    p.out_f16 = dtype == GELO_F16 ? 1 : 0;
    p.out_scale = sign; p.diag_sub = diag; p.post_scale = add_scale;
    p.add = add; p.ldadd = ldadd;
    p.C0 = C; p.ldc = ldc; p.csplit = N;
    p.status = ctx->status_dev;
    if (wide == 128) return launch_tiles<128, false>(ctx, false, ma, ma, mb, mb, ma, p, 2.0 * M * (double)N * K, st);
    return launch_tiles<256, false>(ctx, pair, ma, ma, mb, mb, ma, p, 2.0 * M * (double)N * K, st);
}

// Y (M x N, bf16) = (sa sb) A8 (M x K, E4M3, row stride lda bytes) * B8 (K x N, E4M3, row stride ldb bytes): the offloaded
// product on 8-bit operands (kind::f8f6f4, fp32 accumulation), sa and sb device scalars.  A stage holds 128 bytes of
// k per A row, i.e. 128 values, and the matching 128 rows of B in boxes of 128 columns.
int launch_gemm_e4m3(gelo_ctx* ctx, int M, int N, int K, const void* A8, int lda, const void* B8, int ldb, const float* sa,
                     const float* sb, void* C, int ldc, cudaStream_t st)
{
    if (M <= 0 || N <= 0 || K <= 0) return GELO_OK;
    if (!ctx->tmap_encode) return GELO_ERR_CUDA;
    if ((lda % 16) || (ldb % 16) || (ldc % 8) || (N % 8) || !aligned16(A8) || !aligned16(B8) || !aligned16(C) || !sa || !sb)
        return GELO_ERR_INVALID;
    EncodeTiledFn enc = reinterpret_cast<EncodeTiledFn>(ctx->tmap_encode);
    const bool pair = use_pair(ctx, M, N, 1, false, TC_STORE_BF16);
    CUtensorMap ma, mb;
    {
        const cuuint64_t dims[2] = { (cuuint64_t)K, (cuuint64_t)M };
        const cuuint64_t strides[1] = { (cuuint64_t)lda };
        const cuuint32_t box[2] = { 128, BM };
        const cuuint32_t estr[2] = { 1, 1 };
        if (enc(&ma, CU_TENSOR_MAP_DATA_TYPE_UINT8, 2, const_cast<void*>(A8), dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
                CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
            return GELO_ERR_CUDA;
    }
    bool b3d = false;
    if (!make_map_nmajor(ctx, &mb, B8, 1, false, (uint64_t)N, (uint64_t)K, (uint64_t)ldb, 128, pair ? 128 : 256, &b3d)) return GELO_ERR_CUDA;
    TcParams p = {};
    p.M = M; p.N = N;
    p.nseg = 1;
    p.seg[0] = TcSegment{0, 0, 0, 0, ceil_div(K, 128)};
    p.ksplit = 1; p.kb_per_split = 1 << 30; p.plane = 0;
    p.mode = TC_STORE_BF16;
    p.b3d = b3d ? 1 : 0;
    p.C0 = C; p.C1 = C; p.C2 = C;
    p.ldc = ldc; p.csplit = N;
    p.scale_a = sa; p.scale_b = sb;
    p.status = ctx->status_dev;
    return launch_tiles<256, false, false, false, true>(ctx, pair, ma, ma, mb, mb, ma, p, 2.0 * M * (double)N * K, st);
}

int launch_gemm_tf32x3(gelo_ctx* ctx, int M, int N, int K, const float* A, int lda, const float* B, const float* B2, int b_split, int ldb,
                       float* const C[3], int ldc, int nsplit, float* planes, cudaStream_t st)
{
    if (M <= 0 || N <= 0 || K <= 0) return GELO_OK;
    if (!ctx->tmap_encode) return GELO_ERR_CUDA;
    if (nsplit < 1 || nsplit > 3 || (N % nsplit) || ((N / nsplit) % 8) || (lda % 4) || (ldb % 4) || (ldc % 4) || !aligned16(A) || !aligned16(B) ||
        (B2 && (!aligned16(B2) || b_split <= 0 || b_split >= K)))
        return GELO_ERR_INVALID;
    for (int q = 0; q < nsplit; ++q)
        if (!C[q] || !aligned16(C[q])) return GELO_ERR_INVALID;
    const int rows = B2 ? b_split : K;
    CUtensorMap ma, b0, b1;
    bool b3d = false, b3d1 = false;
    if (!make_map_f32_box(ctx, &ma, A, (uint64_t)K, (uint64_t)M, (uint64_t)lda, BM) ||
        !make_map_nmajor(ctx, &b0, B, 4, true, (uint64_t)N, (uint64_t)rows, (uint64_t)ldb, 32, kX3Cols, &b3d))
        return GELO_ERR_CUDA;
    b1 = b0;
    X3Params p = {};
    p.kb0 = p.kb = ceil_div(rows, 32);
    if (B2) {
        if (!make_map_nmajor(ctx, &b1, B2, 4, true, (uint64_t)N, (uint64_t)(K - b_split), (uint64_t)ldb, 32, kX3Cols, &b3d1) || b3d1 != b3d)
            return GELO_ERR_CUDA;
        p.a_k1 = b_split & ~3;                                // (16-byte aligned; the rows of B2 above its first read as zero)
        p.b_row1 = p.a_k1 - b_split;
        p.kb += ceil_div(K - p.a_k1, 32);
    }
    p.b3d = b3d ? 1 : 0;
    const int tiles = ceil_div(M, 2 * BM) * ceil_div(N, kX3N);
    // K slices where they fill the rounds better than whole tiles and that is worth their planes, which are written and read: microseconds,
    // with 1.06 per k-block, 2 per unit for what is not hidden of its seams, 6 TB/s for the planes and 5 for the launch that sums them.  1075 x 3072
    // x 1024 76 -> 67, 257 x 12288 x 4096 276 -> 264; 512 x 12288 x 4096 stays whole (277).
    int slices = 1;
    double best = 0.0;
    for (int t = 1; t <= kTf32x3Slices && (t == 1 || (planes && aligned16(planes) && p.kb >= 8 * t)); ++t) {
        const double us = ceil_div(tiles * t, ctx->sm_count / 2) * (1.06 * ceil_div(p.kb, t) + 2.0) + (t > 1 ? 5.0 + 8e-6 * t * (double)M * N / 6.0 : 0.0);
        if (t == 1 || us < best) { best = us; slices = t; }
    }
    p.per = ceil_div(p.kb, slices);
    slices = ceil_div(p.kb, p.per);                           // no empty slice
    TcParams& o = p.out;
    o.M = M; o.N = N;
    o.status = ctx->status_dev; o.wait_ns = ctx->wait_limit_ns;
    float* const Cq[3] = { C[0], C[nsplit > 1 ? 1 : 0], C[nsplit > 2 ? 2 : 0] };
    o.C0 = Cq[0]; o.C1 = Cq[1]; o.C2 = Cq[2]; o.ldc = ldc; o.csplit = N / nsplit;
    if (slices > 1) {                                         // (N is a multiple of 8, so the planes' rows are whole chunks)
        o.C0 = o.C1 = o.C2 = planes; o.ldc = N; o.csplit = N; o.plane = (long long)M * N;
    }
    static bool attr_done[64] = {};
    if (ctx->device >= 0 && ctx->device < 64 && !attr_done[ctx->device]) {
        GELO_CUDA_OK(cudaFuncSetAttribute(gemm_x3_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kX3Smem));
        attr_done[ctx->device] = true;
    }
    {
        ProfScope ps(ctx, PROF_GEMM_TC, 6.0 * M * (double)N * K, st);
        GELO_TRY(launch_chained(ctx, gemm_x3_kernel, 2 * tiles * slices, kX3Threads, kX3Smem, st, ma, b0, b1, p));
    }
    GELO_TRY(after_launch(ctx));
    return slices > 1 ? launch_sum_planes_routed(ctx, planes, (size_t)M * N, slices, M, N, Cq, ldc, N / nsplit, st) : GELO_OK;
}

}  // namespace gelo

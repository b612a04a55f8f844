// Inverse of the non-orthogonal mixing matrix by Newton's iteration (paper Mitigation 1: "The TEE must compute A^-1 per
// batch").
//
// The sampler's A = Q0 + gamma G1 / sqrt(m) comes with a good first guess of its inverse: with X0 = Q0^T the residual
// I - A X0 = -gamma G1 Q0^T / sqrt(m) is a Gaussian matrix whose eigenvalues fill the disc of radius gamma (the circular
// law), so its 2^k-th power, which k steps of
//     X <- X (2 I - A X)
// leave, has Frobenius norm gamma^(2^k) sqrt(m): 0.4% of the identity's after three steps at gamma = 1/2.  Every step is two
// products of 16-bit operands, and a step corrects the rounding of the one before, because it starts from A and the stored
// X.  The last step keeps what is left of the residual small instead of adding it to the identity before it is rounded,
//     R = I - A X,   A^-1 = X + X R   (rounded once, to the storage type),
// and ends at gamma^16 = 1.5e-5 and 2^-9 |R| = 2e-5 (bfloat16), below what the storage type resolves.
//
// Eight products at the 16-bit rate of the tensor cores replace the pivoted LU and its two triangular solves, which were bound
// by some 1000 dependent launches: 4300 rows, one call alone 30.4 -> 8.6 ms, the 32-layer sweep (16 of them) 114 -> 98.5 ms, and
// A^-1 A - I falls from 1.3e-3 to what rounding A^-1 leaves (half: 2.7e-4).
#include "common.cuh"

namespace gelo {

// gamma: beyond 0.55 the fourth step no longer reaches 1e-4 (0.55^16 = 7e-5), and from 1 on the iteration diverges.
// m: smaller matrices take the fp32 iteration.
bool newton_inverse_supports(int m, int dtype, float gamma) { return dtype != GELO_F32 && m >= 256 && gamma <= 0.55f; }

int run_newton_inverse(gelo_ctx* ctx, int m, int dtype, const void* A, int lda, void* X0, void* X1, void* Y, int ld, void* Ainv, int ldi,
                       cudaStream_t st)
{
    const int m8 = (m + 7) & ~7;
    for (int step = 0; step < 3; ++step) {
        GELO_TRY(launch_gemm_affine16(ctx, dtype, m, m8, m, A, lda, X0, ld, -1.0f, 2.0f, nullptr, 0, Y, ld, st));
        GELO_TRY(launch_gemm_affine16(ctx, dtype, m, m8, m, X0, ld, Y, ld, 1.0f, 0.0f, nullptr, 0, X1, ld, st));
        void* t = X0; X0 = X1; X1 = t;
    }
    GELO_TRY(launch_gemm_affine16(ctx, dtype, m, m8, m, A, lda, X0, ld, -1.0f, 1.0f, nullptr, 0, Y, ld, st));
    return launch_gemm_affine16(ctx, dtype, m, m8, m, X0, ld, Y, ld, 1.0f, 0.0f, X0, ld, Ainv, ldi, st);
}

// fp32: five steps (gamma^32 = 2e-10) of products on the FMA pipes.
int run_newton_inverse_f32(gelo_ctx* ctx, int m, const float* A, int lda, float* X0, float* X1, float* Y, int ld, float* Ainv, int ldi,
                           cudaStream_t st)
{
    auto product = [&](const float* a, int la, const float* b, int lb, float alpha, float diag, float* c, int lc) -> int {
        GemmArgs g;
        g.M = m; g.N = m; g.K = m;
        g.A = a; g.lda = la; g.B = b; g.ldb = lb;
        g.C[0] = c; g.ldc = lc; g.alpha = alpha; g.diag = diag;
        return launch_gemm_simt(ctx, g, st);
    };
    for (int step = 0; step < 5; ++step) {
        GELO_TRY(product(A, lda, X0, ld, -1.0f, 2.0f, Y, ld));
        if (step == 4) return product(X0, ld, Y, ld, 1.0f, 0.0f, Ainv, ldi);
        GELO_TRY(product(X0, ld, Y, ld, 1.0f, 0.0f, X1, ld));
        float* t = X0; X0 = X1; X1 = t;
    }
    return GELO_OK;
}

}  // namespace gelo

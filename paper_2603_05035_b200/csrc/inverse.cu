// Inverse of the non-orthogonal mixing matrix by Newton's iteration (paper Mitigation 1: "The TEE must compute A^-1 per
// batch").
//
// The sampler's A = Q0 + gamma G1 / sqrt(m) comes with a good first guess of its inverse: with X0 = Q0^T the residual
// R = I - A X0 = -gamma G1 Q0^T / sqrt(m) is a Gaussian matrix whose eigenvalues fill the disc of radius gamma (the circular
// law), and A^-1 = X0 (I + R + R^2 + ...).  The k-th power of such a matrix has Frobenius norm gamma^k sqrt(m).
//
// Products of 16-bit operands, in two parts.  First X = X0 (I + R + R^2 + R^3 + R^4) in four products, the polynomial by
// completing squares: with S = R + I/4 and N = S^2 + 5/16 I it is N^2 + 5/8 S + 45/64 I.  What is missing, R^5, and all rounding so
// far is then the residual of the stored X, which a last part computes and corrects:
//     R = I - A X,   A^-1 = X + X R                   (two products, ends at gamma^10),
//     R = I - A X,   Z = R^2 + R,   A^-1 = X + X Z    (three, gamma^15),
// with R or Z kept small instead of added to the identity before it is rounded, and A^-1 rounded once.  The second leaves
// 3e-5 at gamma = 1/2, nothing beside the rounding of A^-1 (bfloat16 1.66e-3, half 2.1e-4).  The first leaves 2^-10, with the rounding 1.93e-3 in
// bfloat16 at every m.  It serves bfloat16 from 4096 rows up, where a product costs 0.11 ms: that is where the pivoted LU's error, which
// grows with m, reached the same (1.83e-3 at 3000 rows, 1.94e-3 at 4096, 1.95e-3 at 4300, 2.17e-3 at 6000), so that no size lost precision.
//
// Six or seven products at the 16-bit rate of the tensor cores replace the pivoted LU and its two triangular solves, which were
// bound by some 1000 dependent launches: 4300 rows, one call alone 30.4 -> 8.6 ms (with eight products, four Newton steps from
// X0), the 32-layer sweep (16 of them) 114 -> 98.5 ms; six products instead of eight: 81.5 -> 78 ms later.
#include "common.cuh"

namespace gelo {

// gamma: beyond 0.55 even two corrections leave more than rounding does, and from 1 on the series diverges.
// m: smaller matrices take the fp32 iteration.
bool newton_inverse_supports(int m, int dtype, float gamma) { return dtype != GELO_F32 && m >= 256 && gamma <= 0.55f; }

int run_newton_inverse(gelo_ctx* ctx, int m, int dtype, float gamma, const void* A, int lda, void* X0, void* T1, void* T2, void* X, int ld,
                       void* Ainv, int ldi, cudaStream_t st)
{
    const int m8 = (m + 7) & ~7;
    auto product = [&](const void* a, int la, const void* b, float sign, float diag, const void* add, float add_scale, void* c, int lc) -> int {
        return launch_gemm_affine16(ctx, dtype, m, m8, m, a, la, b, ld, sign, diag, add, ld, add_scale, c, lc, st);
    };
    GELO_TRY(product(A, lda, X0, -1.0f, 1.25f, nullptr, 0.0f, T1, ld));                       // S
    GELO_TRY(product(T1, ld, T1, 1.0f, 0.3125f, nullptr, 0.0f, T2, ld));                      // N
    GELO_TRY(product(T2, ld, T2, 1.0f, 0.703125f, T1, 0.625f, X, ld));                        // the polynomial
    GELO_TRY(product(X0, ld, X, 1.0f, 0.0f, nullptr, 0.0f, T1, ld));
    void* x = T1;
    void* r = T2;
    if (gamma > 0.5f) {                                                                       // gamma^10 first, then its square
        GELO_TRY(product(A, lda, x, -1.0f, 1.0f, nullptr, 0.0f, r, ld));
        GELO_TRY(product(x, ld, r, 1.0f, 0.0f, x, 1.0f, X0, ld));
        x = X0;
    }
    GELO_TRY(product(A, lda, x, -1.0f, 1.0f, nullptr, 0.0f, r, ld));
    if (gamma <= 0.5f && !(dtype == GELO_BF16 && m >= 4096)) {
        GELO_TRY(product(r, ld, r, 1.0f, 0.0f, r, 1.0f, X, ld));
        r = X;
    }
    return product(x, ld, r, 1.0f, 0.0f, x, 1.0f, Ainv, ldi);
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

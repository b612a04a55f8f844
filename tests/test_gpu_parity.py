"""GPU parity: every stage of the offload path, through the C ABI, against the fp64 oracle.

Tolerances (relative Frobenius error against the oracle on the same stored inputs):
fp32 path 1e-4, bf16 path 2e-2.  Integer work (the Philox word stream) is bit-exact.
"""
import numpy as np
import pytest
import torch

from paper_2603_05035_b200 import binding, inputs
from paper_2603_05035_b200.binding import BF16, F32, NONORTHOGONAL, ORTHOGONAL

from gpu_util import dev, f64, make_ctx, padded, sample_rows

pytestmark = pytest.mark.gpu

# f16: the same path with an 11-bit significand instead of bf16's 8.  Storage roundings are 8 times finer; what the tf32 products of the
# sampler leave in A^T A does not shrink with them, so the bound is a quarter of the bf16 one (measured at the benchmark size: 1.3e-3
# orthogonal, 1.1e-3 non-orthogonal)
TOL = {"f32": 1e-4, "bf16": 2e-2, "f16": 5e-3}
TDT = {"f32": torch.float32, "bf16": torch.bfloat16, "f16": torch.float16}


@pytest.fixture(scope="module")
def ctx():
    c = make_ctx(4096, 204, 4096, 12288, "bf16")
    yield c
    assert c.last_status() == binding.OK
    c.close()


# ------------------------------------------------------------------------- sampling

@pytest.mark.parametrize("seed,stream,attempt,first,count", [
    (0, 0, 0, 0, 4096), (0xDEADBEEFCAFEF00D, 1, 3, 5, 1001), (7, 2, 0, (1 << 34) - 3, 64), (1, 3, 1, 2, 1)])
def test_philox_words_bit_exact(ctx, oracle, seed, stream, attempt, first, count):
    out = torch.zeros(count, dtype=torch.int32, device="cuda")
    ctx.philox_words(seed, stream, attempt, first, count, out)
    got = out.cpu().numpy().view(np.uint32)
    assert np.array_equal(got, oracle.philox_words(seed, stream, attempt, first, count))


@pytest.mark.parametrize("rows,cols,ld", [(64, 64, 64), (7, 13, 16), (130, 130, 192), (3, 4096, 4096), (1, 1, 8)])
def test_gaussian_matches_oracle(ctx, oracle, rows, cols, ld):
    out = padded(rows, ld, torch.float32)
    ctx.sample_gaussian(rows, cols, ld, 42, 1, 2, 0.5, out)
    got = out.cpu().numpy()[:, :cols].astype(np.float64)
    ref = 0.5 * oracle.gaussian(42, 1, 2, rows, cols)
    # single-precision log / sqrt / sincospi on exactly representable uniforms: a few ulp at |z| < 5.8
    assert np.max(np.abs(got - ref)) <= 2e-6
    if ld > cols:
        assert torch.isnan(out[:, cols:]).all()      # padding columns are never written


def test_gaussian_refuses_more_than_a_grid(ctx):
    # 2^42 elements are 2^32 thread blocks, more than one launch can have
    out = torch.zeros(64, device="cuda")
    with pytest.raises(binding.GeloError) as e:
        ctx.sample_gaussian(1 << 21, 1 << 21, 1 << 21, 1, 0, 0, 1.0, out)
    assert e.value.status == binding.ERR_INVALID and (out == 0).all()


def test_gaussian_statistics(ctx):
    out = torch.empty((2048, 2048), device="cuda", dtype=torch.float32)
    ctx.sample_gaussian(2048, 2048, 2048, 5, 0, 0, 1.0, out)
    z = out.double()
    n = z.numel()
    assert abs(z.mean().item()) < 5 / np.sqrt(n)
    assert abs(z.var().item() - 1.0) < 5 * np.sqrt(2.0 / n)
    assert abs((z ** 4).mean().item() - 3.0) < 5 * np.sqrt(96.0 / n)


# ------------------------------------------------------------------------- QR

@pytest.mark.parametrize("m", [1, 2, 3, 31, 32, 33, 64, 68, 130, 257, 512])
def test_householder_qr_stage(ctx, oracle, m):
    ld = ctx.mixing_ld(m)
    G64 = oracle.gaussian(100 + m, 0, 0, m, m).astype(np.float32).astype(np.float64)
    G = padded(m, ld, torch.float32)
    G[:, :m] = dev(G64)
    Q = padded(m, ld, torch.float32)
    Qt = padded(m, ld, torch.float32)
    ctx.qr_orthogonal(m, G, ld, Q, Qt)
    q = f64(Q[:, :m]); qt = f64(Qt[:, :m]); r = np.triu(f64(G[:, :m]))
    assert np.array_equal(qt, q.T)
    assert np.linalg.norm(q.T @ q - np.eye(m)) / np.sqrt(m) <= 1e-5
    s = np.where(np.diag(r) < 0, -1.0, 1.0)
    r_pos = (r.T * s).T                                   # diag > 0 after the column signing of Q
    assert np.linalg.norm(q @ r_pos - G64) / np.linalg.norm(G64) <= 1e-5
    # against the oracle's factor of the same matrix: Q is unique once diag(R) > 0, but its
    # trailing columns are conditioned like kappa(G), so compare by column alignment
    q_ref, _ = oracle.householder_qr(G64)
    cosines = np.abs(np.sum(q * q_ref, axis=0))
    assert np.all(np.sum(q * q_ref, axis=0)[: max(1, m // 2)] > 1 - 1e-3)
    assert np.median(cosines) > 1 - 1e-5


# ------------------------------------------------------------------------- LU inverse / cond

@pytest.mark.parametrize("m", [1, 2, 5, 32, 33, 68, 130, 257, 512])
def test_lu_inverse_stage(ctx, oracle, m):
    ld = ctx.mixing_ld(m)
    A64, _ = oracle.sample_mixing(m, 1, seed=200 + m)
    A64 = A64.astype(np.float32).astype(np.float64)
    A = padded(m, ld, torch.float32); A[:, :m] = dev(A64)
    X = padded(m, ld, torch.float32)
    ctx.lu_inverse(m, A, ld, X)
    x = f64(X[:, :m])
    assert np.array_equal(f64(A[:, :m]), A64)             # input preserved
    assert oracle.rel_fro(x, oracle.lu_inverse(A64)) <= 2e-5
    assert np.linalg.norm(A64 @ x - np.eye(m)) / np.sqrt(m) <= 2e-5


def test_lu_inverse_needs_pivoting(ctx, oracle):
    m, ld = 96, 128
    rng = np.random.default_rng(3)
    P = np.eye(m)[rng.permutation(m)]
    A64 = (3.0 * P + 0.05 * rng.standard_normal((m, m))).astype(np.float32).astype(np.float64)
    A = padded(m, ld, torch.float32); A[:, :m] = dev(A64)
    X = padded(m, ld, torch.float32)
    ctx.lu_inverse(m, A, ld, X)
    assert oracle.rel_fro(f64(X[:, :m]), oracle.lu_inverse(A64)) <= 2e-5


@pytest.mark.parametrize("m,gamma", [(64, 0.5), (257, 0.5), (512, 0.5), (96, 3.0)])
def test_cond_estimate(ctx, oracle, m, gamma):
    ld = ctx.mixing_ld(m)
    A64, X64 = oracle.sample_mixing(m, 1, seed=300 + m, gamma=gamma)
    A = padded(m, ld, torch.float32); A[:, :m] = dev(A64)
    X = padded(m, ld, torch.float32); X[:, :m] = dev(X64)
    c = torch.zeros(1, device="cuda")
    ctx.cond_estimate(m, A, X, ld, c)
    ref = oracle.cond2(A64)
    est = c.item()
    assert 0.88 * ref <= est <= 1.001 * ref               # a Ritz value of a few Lanczos steps: a lower estimate within ~10%


@pytest.mark.parametrize("bad", [float("nan"), float("inf")])
def test_cond_estimate_of_broken_matrices_is_no_number(ctx, bad):
    """The verdict is `estimate * 1.2 <= bound`: an entry that is not finite must not come out as a small estimate."""
    m, ld = 200, 256
    A = torch.zeros((m, ld), device="cuda"); A[:, :m] = torch.eye(m, device="cuda")
    B = A.clone(); B[100, 50] = bad
    c = torch.zeros(1, device="cuda")
    for pair in ((A, B), (B, A), (B, B)):
        ctx.cond_estimate(m, *pair, ld, c)
        assert not c.item() <= 1e30
    ctx.cond_estimate(m, A, A, ld, c)
    assert abs(c.item() - 1) <= 1e-4


# ------------------------------------------------------------------------- sample_mixing

def _sample(ctx, m, kind, seed, dt):
    ld = ctx.mixing_ld(m)
    A = padded(m, ld, TDT[dt]); X = padded(m, ld, TDT[dt])
    c = torch.zeros(1, device="cuda")
    ctx.sample_mixing(m, kind, seed, dt, A, X, ld, c)
    torch.cuda.synchronize()
    return A, X, c.item()


@pytest.mark.parametrize("dt", ["f32", "bf16"])
@pytest.mark.parametrize("m", [1, 64, 68, 130, 512])
def test_sample_mixing_orthogonal(ctx, oracle, m, dt):
    A, X, c = _sample(ctx, m, ORTHOGONAL, 11, dt)
    a = f64(A[:, :m]); x = f64(X[:, :m])
    assert c == 1.0
    assert np.array_equal(x, a.T)                          # A^-1 = A^T, bytewise
    defect = np.linalg.norm(a.T @ a - np.eye(m)) / np.sqrt(m)
    assert defect <= (1e-5 if dt == "f32" else 4e-3)
    a_ref, _ = oracle.sample_mixing(m, 0, seed=11)
    tol = 2e-3 if dt == "f32" else 6e-3
    half = max(1, m // 2)
    assert np.max(np.abs(a[:, :half] - a_ref[:, :half])) <= tol
    assert np.median(np.abs(np.sum(a * a_ref, axis=0))) > 1 - 1e-3
    # same seed, same bytes; another seed, another matrix
    A2, _, _ = _sample(ctx, m, ORTHOGONAL, 11, dt)
    assert torch.equal(A[:, :m], A2[:, :m])
    if m > 1:
        A3, _, _ = _sample(ctx, m, ORTHOGONAL, 12, dt)
        assert not torch.equal(A[:, :m], A3[:, :m])


@pytest.mark.parametrize("dt", ["f32", "bf16"])
@pytest.mark.parametrize("m", [64, 130, 512])
def test_sample_mixing_nonorthogonal(ctx, oracle, m, dt):
    A, X, c = _sample(ctx, m, NONORTHOGONAL, 21, dt)
    a = f64(A[:, :m]); x = f64(X[:, :m])
    true_cond = np.linalg.cond(a)
    assert true_cond <= 100.0 and 0.85 * true_cond <= c <= 1.01 * true_cond
    assert np.linalg.norm(a.T @ a - np.eye(m)) / np.sqrt(m) > 0.3        # Mitigation 1: Gram masked
    inv_defect = np.linalg.norm(a @ x - np.eye(m)) / np.sqrt(m)
    assert inv_defect <= (2e-5 if dt == "f32" else 8e-3)
    a_ref, _ = oracle.sample_mixing(m, 1, seed=21, gamma=0.5)
    half = max(1, m // 2)
    assert np.max(np.abs(a[:, :half] - a_ref[:, :half])) <= (2e-3 if dt == "f32" else 8e-3)
    A2, X2, _ = _sample(ctx, m, NONORTHOGONAL, 21, dt)
    assert torch.equal(A[:, :m], A2[:, :m]) and torch.equal(X[:, :m], X2[:, :m])


def test_condition_bound_resampling(oracle):
    """With a large gamma the Gaussian part dominates: first attempts often miss kappa <= 100."""
    c = make_ctx(64, 0, 64, 96, "f32")
    c.set_nonorthogonal(gamma=40.0, cond_bound=100.0, max_attempts=8)
    m, ld = 48, 64
    outcomes = 0
    for seed in range(12):
        conds = [oracle.cond2(oracle.sample_mixing(m, 1, seed, a, 40.0)[0]) for a in range(8)]
        if any(80.0 < x < 118.0 for x in conds):
            continue                                       # borderline for an estimate: skip the seed
        expect = next((a for a, x in enumerate(conds) if x <= 100.0), None)
        A = padded(m, ld, torch.float32); X = padded(m, ld, torch.float32)
        cd = torch.zeros(1, device="cuda")
        try:
            c.sample_mixing(m, NONORTHOGONAL, seed, "f32", A, X, ld, cd)
            assert expect is not None
            a_ref, _ = oracle.sample_mixing(m, 1, seed, expect, 40.0)
            assert np.max(np.abs(f64(A[:, :m]) - a_ref)) <= 0.05 * np.abs(a_ref).max()
            assert np.linalg.cond(f64(A[:, :m])) <= 100.0
        except binding.GeloError as e:
            assert e.status == binding.ERR_COND and expect is None
        outcomes += 1
    assert outcomes >= 3
    c.last_status()
    c.close()

def test_results_only_from_accepted_pairs():
    """A rejected pair writes nothing to the caller's buffers, and a redraw starts from the caller's H even where the results go there:
    sizes with the fused projection and with products of their own."""
    for n, k, d, dt in ((64, 4, 256, "bf16"), (300, 15, 256, "bf16"), (200, 0, 128, "f32")):
        m, p = n + k, d
        c = binding.Context(0)
        c.ensure_workspace(n, k, d, p, dt)
        H = inputs.make_hidden(n, d, dt, 3, True, "cuda")
        W = inputs.make_weight(d, p, dt, 3, "cuda")
        Y = torch.full((n, p), 7.0, device="cuda", dtype=TDT[dt])
        c.set_nonorthogonal(0.5, 1.0, 3)                        # kappa_2 is about 4.7: no attempt can pass
        with pytest.raises(binding.GeloError) as e:
            c.qkv_offload(H, W, n, k, d, p, NONORTHOGONAL, 5, 10.0, dt, Y)
        assert e.value.status == binding.ERR_COND
        torch.cuda.synchronize()
        assert (Y == 7.0).all()
        # a seed whose first estimate is above its second, and a bound between the two (times the 1.2 that the check applies)
        ld = c.mixing_ld(m)
        A = padded(m, ld, TDT[dt]); X = padded(m, ld, TDT[dt]); cond = torch.zeros(1, device="cuda")
        for seed in range(20):
            c.set_nonorthogonal(0.5, 100.0, 1)
            c.sample_mixing(m, NONORTHOGONAL, seed, dt, A, X, ld, cond)
            first = cond.item()
            c.set_nonorthogonal(0.5, 1.2 * first * 0.995, 2)
            try:
                c.sample_mixing(m, NONORTHOGONAL, seed, dt, A, X, ld, cond)
                break
            except binding.GeloError:
                continue
        ref = H.double() @ W.double()
        c.qkv_offload(H, W, n, k, d, p, NONORTHOGONAL, seed, 10.0, dt, H)        # (p = d: the result replaces H)
        torch.cuda.synchronize()
        assert cond.item() < 0.995 * first and c.last_status() == binding.OK
        assert ((H.double() - ref).norm() / ref.norm()).item() <= TOL[dt]
        c.close()


# ------------------------------------------------------------------------- shields

@pytest.mark.parametrize("dt", ["f32", "bf16"])
@pytest.mark.parametrize("n,d,k", [(64, 4096, 4), (2048, 4096, 102), (7, 64, 3), (1, 8, 1), (10, 256, 1)])
def test_shield_rows(ctx, oracle, n, d, k, dt):
    H = inputs.make_hidden(n, d, dt, seed=9, rms_norm=(n % 2 == 0), device="cuda")
    if n == 7:
        H = (H.float() * torch.linspace(0.5, 4.0, n, device="cuda")[:, None]).to(TDT[dt]).contiguous()
    S = torch.full((k, d), float("nan"), device="cuda", dtype=TDT[dt])
    ctx.shield_rows(H, n, d, k, 10.0, 77, dt, S)
    ref = oracle.shield_rows(f64(H), k, 10.0, 77)
    assert oracle.rel_fro(f64(S), ref) <= (2e-6 if dt == "f32" else 4e-3)
    ctx.shield_rows(H, n, d, 0, 10.0, 77, dt, None)       # k = 0 is a no-op


# ------------------------------------------------------------------------- the three products

def _random_mixing(oracle, m, kind, seed, dt):
    a, x = oracle.sample_mixing(m, kind, seed)
    A = dev(a, TDT[dt]); X = dev(x, TDT[dt])
    return A, X


@pytest.mark.parametrize("dt", ["f32", "bf16"])
@pytest.mark.parametrize("n,d,k,nu", [(64, 4096, 4, 5), (2048, 1024, 102, 3), (300, 256, 7, 10), (7, 64, 3, 63)])
def test_student_t_shield_rows(ctx, oracle, n, d, k, nu, dt):
    """Student-t shield rows (both the one-launch and the three-kernel route) against the oracle."""
    ctx.ensure_workspace(n, k, d, 3 * d, dt)
    H = inputs.make_hidden(n, d, dt, 11, False, "cuda")
    S = torch.full((k, d), float("nan"), device="cuda", dtype=TDT[dt])
    ctx.shield_rows_t(H, n, d, k, 10.0, 321, nu, dt, S)
    torch.cuda.synchronize()
    ref = oracle.shield_rows_t(f64(H), k, 10.0, 321, nu)
    # fp32 normals agree with the oracle's to 2e-6 absolute; the ratio g_0 / sqrt(mean g^2) keeps that as a relative error
    # of about 1e-5 of the largest entries; bf16 adds its rounding
    tol = 2e-5 if dt == "f32" else 4e-3
    assert oracle.rel_fro(f64(S), ref) <= tol
    assert np.max(np.abs(f64(S) - ref)) <= 10 * tol * np.sqrt(np.mean(ref * ref)) * (1 + np.max(np.abs(ref)) / np.sqrt(np.mean(ref * ref)))


def test_whole_call_with_student_t_shields(oracle):
    """The result is H W whatever the shield rows are (Eq. 4); the call must stay inside the tolerance with the
    heavier-tailed kind too."""
    c = make_ctx(600, 30, 512, 1536, "bf16")
    c.set_shield_student_t(5)
    n, k, d, p = 600, 30, 512, 1536
    H = inputs.make_hidden(n, d, "bf16", 12, True, "cuda")
    W = inputs.make_weight(d, p, "bf16", 12, "cuda")
    Q = torch.empty((n, d), device="cuda", dtype=torch.bfloat16); K = torch.empty_like(Q); V = torch.empty_like(Q)
    c.qkv_offload(H, W, n, k, d, p, ORTHOGONAL, 5, 10.0, "bf16", Q, K, V)
    torch.cuda.synchronize()
    y = np.hstack([f64(Q), f64(K), f64(V)])
    assert oracle.rel_fro(y, oracle.direct(f64(H), f64(W))) <= TOL["bf16"]
    with pytest.raises(binding.GeloError):
        c.set_shield_student_t(2)
    c.close()


@pytest.mark.parametrize("dt", ["f32", "bf16"])
@pytest.mark.parametrize("n,k,d,p", [(64, 0, 256, 768), (64, 4, 256, 768), (130, 7, 264, 264 * 3),
                                      (1, 0, 8, 24), (200, 10, 512, 1536), (256, 0, 128, 384)])
def test_products_stage_parity(ctx, oracle, n, k, d, p, dt):
    m = n + k
    ld = ctx.mixing_ld(m)
    A = padded(m, ld, TDT[dt]); X = padded(m, ld, TDT[dt])
    a64, x64 = oracle.sample_mixing(m, 1, seed=31)
    A[:, :m] = dev(a64, TDT[dt]); X[:, :m] = dev(x64, TDT[dt])
    H = inputs.make_hidden(n, d, dt, 5, True, "cuda")
    W = inputs.make_weight(d, p, dt, 5, "cuda")
    S = (10.0 * torch.randn((k, d), device="cuda")).to(TDT[dt]) if k else None
    U = torch.full((m, d), float("nan"), device="cuda", dtype=TDT[dt])
    Yp = torch.full((m, p), float("nan"), device="cuda", dtype=TDT[dt])
    Q = torch.full((n, p // 3), float("nan"), device="cuda", dtype=TDT[dt]); K = Q.clone(); V = Q.clone()
    Yfull = torch.full((n, p), float("nan"), device="cuda", dtype=TDT[dt])
    ctx.mix(A, ld, H, S, n, k, d, dt, U)
    ctx.project(U, W, m, d, p, dt, Yp)
    ctx.unmix(X, ld, Yp, n, k, p, dt, Q, K, V)
    ctx.unmix(X, ld, Yp, n, k, p, dt, Yfull)
    tol = 2e-6 if dt == "f32" else 4e-3                    # one rounding of the output per stage
    Hf = f64(H) if S is None else np.vstack([f64(H), f64(S)])
    assert oracle.rel_fro(f64(U), oracle.matmul(f64(A[:, :m]), Hf)) <= tol
    assert oracle.rel_fro(f64(Yp), oracle.matmul(f64(U), f64(W))) <= tol
    y_ref = oracle.matmul(f64(X[:n, :m]), f64(Yp))
    y = np.hstack([f64(Q), f64(K), f64(V)])
    assert oracle.rel_fro(y, y_ref) <= tol
    assert np.array_equal(f64(Yfull), y)                   # split and unsplit outputs carry the same values
    # whole chain against Eq. 4's right-hand side
    assert oracle.rel_fro(y, oracle.direct(f64(H), f64(W))) <= TOL[dt]


def test_mix_full_size_seam_inside_a_k_block(ctx, oracle):
    """The mixing product alone at full size with the H / S seam in the middle of a 64-row k-block (n = 4000 is 32
    past a multiple of 64), the operand pipeline at full depth: sampled rows of U against the oracle's product."""
    n, k, d = 4000, 200, 4096
    m = n + k
    ld = ctx.mixing_ld(m)
    g = torch.Generator(device="cuda"); g.manual_seed(77)
    A = padded(m, ld, torch.bfloat16)
    A[:, :m] = (torch.randn((m, m), device="cuda", generator=g) / np.sqrt(m)).to(torch.bfloat16)
    H = inputs.make_hidden(n, d, "bf16", 78, True, "cuda")
    S = (10.0 * torch.randn((k, d), device="cuda", generator=g)).to(torch.bfloat16)
    U = torch.full((m, d), float("nan"), device="cuda", dtype=torch.bfloat16)
    ctx.mix(A, ld, H, S, n, k, d, "bf16", U)
    torch.cuda.synchronize()
    assert torch.isfinite(U).all()
    rows = sample_rows(m, 64, seed=5, extra=(n - 1, n, n + 1))
    ref = oracle.matmul(f64(A[rows][:, :m]), np.vstack([f64(H), f64(S)]))
    u = f64(U[rows])
    assert oracle.rel_fro(u, ref) <= 4e-3                  # one bf16 rounding of the output
    assert np.max(np.abs(u - ref)) <= 8 * 4e-3 * np.sqrt(np.mean(ref * ref))
    # a seam that is not even a multiple of 8 rows (the second segment then starts at the 16-byte boundary below it)
    n2 = 3997
    U2 = torch.full((n2 + k, d), float("nan"), device="cuda", dtype=torch.bfloat16)
    ld2 = ctx.mixing_ld(n2 + k)
    A2 = padded(n2 + k, ld2, torch.bfloat16); A2[:, :n2 + k] = A[:n2 + k, :n2 + k]
    ctx.mix(A2, ld2, H[:n2].contiguous(), S, n2, k, d, "bf16", U2)
    torch.cuda.synchronize()
    rows2 = np.array([0, 1, 127, 128, 2047, 2048, n2 - 1, n2, n2 + 1, n2 + k - 1], dtype=np.int64)
    ref2 = oracle.matmul(f64(A2[rows2][:, :n2 + k]), np.vstack([f64(H[:n2]), f64(S)]))
    assert oracle.rel_fro(f64(U2[rows2]), ref2) <= 4e-3


@pytest.mark.parametrize("dt", ["bf16", "f16"])
@pytest.mark.parametrize("n,k,d,p,split", [(64, 4, 4096, 12288, True), (64, 0, 256, 768, True), (100, 28, 520, 1536, True),
                                           (1, 0, 8, 192, False), (7, 3, 72, 11008, False), (33, 0, 64, 4736, False)])
def test_project_unmix_one_kernel(ctx, oracle, n, k, d, p, split, dt):
    """Eq. 2 and Eq. 3 in one kernel for a small batch: against the oracle's two products (with Y' rounded to the
    storage type in between, as the stand-alone projection stores it) and against the two stand-alone launches."""
    m = n + k
    ld = ctx.mixing_ld(m)
    ctx.ensure_workspace(n, k, d, p, dt)
    X = padded(m, ld, TDT[dt])
    _, x64 = oracle.sample_mixing(m, 1, seed=32)
    X[:, :m] = dev(x64, TDT[dt])
    g = torch.Generator(device="cuda"); g.manual_seed(91)
    U = (3.0 * torch.randn((m, d), device="cuda", generator=g)).to(TDT[dt])
    W = inputs.make_weight(d, p, dt, 7, "cuda")
    outs = [torch.full((n, p // 3 if split else p), float("nan"), device="cuda", dtype=TDT[dt]) for _ in range(3 if split else 1)]
    ctx.project_unmix(U, W, X, ld, n, k, d, p, dt, *outs)
    torch.cuda.synchronize()
    assert ctx.last_status() == binding.OK
    y = np.hstack([f64(o) for o in outs])
    assert np.isfinite(y).all()
    yp = torch.as_tensor(oracle.matmul(f64(U), f64(W))).to(TDT[dt])           # Y' as stored
    ref = oracle.matmul(f64(X[:n, :m]), f64(yp))
    assert oracle.rel_fro(y, ref) <= 4e-3 * (1.0 if dt == "bf16" else 0.25)      # one rounding of the output
    # the two stand-alone launches give the same values up to the summation order inside the tensor core
    Yp = torch.empty((m, p), device="cuda", dtype=TDT[dt])
    outs2 = [torch.empty_like(o) for o in outs]
    ctx.project(U, W, m, d, p, dt, Yp)
    ctx.unmix(X, ld, Yp, n, k, p, dt, *outs2)
    torch.cuda.synchronize()
    y2 = np.hstack([f64(o) for o in outs2])
    assert oracle.rel_fro(y, y2) <= 1e-3 * (1.0 if dt == "bf16" else 0.25)


def test_project_unmix_rejects_what_it_cannot_serve(ctx):
    L = binding.load_library()
    st = torch.cuda.current_stream().cuda_stream
    t = torch.zeros((256, 256), device="cuda", dtype=torch.bfloat16)
    q = torch.zeros((256, 8192), device="cuda", dtype=torch.bfloat16)
    a = (ctx._h, t.data_ptr(), t.data_ptr(), t.data_ptr())
    assert L.gelo_project_unmix(*a, 256, 129, 0, 256, 192, BF16, q.data_ptr(), None, None, st) == binding.ERR_UNSUPPORTED  # m > 128
    assert L.gelo_project_unmix(*a, 128, 64, 0, 256, 96, BF16, q.data_ptr(), None, None, st) == binding.ERR_UNSUPPORTED    # p % 64
    assert L.gelo_project_unmix(*a, 128, 64, 0, 256, 192, F32, q.data_ptr(), None, None, st) == binding.ERR_UNSUPPORTED
    assert L.gelo_project_unmix(*a, 64, 64, 4, 256, 192, BF16, q.data_ptr(), None, None, st) == binding.ERR_INVALID        # lda < m
    assert L.gelo_project_unmix(*a, 128, 64, 0, 256, 192, BF16, None, None, None, st) == binding.ERR_INVALID


# ------------------------------------------------------------------------- whole call

def _run_offload(ctx, w, call, host=False):
    H, W, seed = inputs.make_call_inputs(w, call, "cuda")
    n, k, d, p = w.n, w.k, w.d, w.p
    ctx.ensure_workspace(n, k, d, p, w.dtype)
    if host:
        Hh = H.cpu().pin_memory()
        out = [torch.empty((n, p // 3), dtype=TDT[w.dtype]).pin_memory() for _ in range(3)]
        ctx.qkv_offload_host(Hh, W, n, k, d, p, w.kind(call), seed, w.shield_scale, w.dtype, *out)
        Q, K, V = out
    else:
        Q = torch.full((n, p // 3), float("nan"), device="cuda", dtype=TDT[w.dtype]); K = Q.clone(); V = Q.clone()
        ctx.qkv_offload(H, W, n, k, d, p, w.kind(call), seed, w.shield_scale, w.dtype, Q, K, V)
        torch.cuda.synchronize()
    return H, W, np.hstack([f64(Q), f64(K), f64(V)])


@pytest.mark.parametrize("name", ["tiny_f32", "decode_bf16"])
def test_offload_small_workloads_full_oracle(ctx, oracle, name):
    w = inputs.WORKLOADS[name]
    for call in range(2):
        H, W, y = _run_offload(ctx, w, call)
        assert oracle.rel_fro(y, oracle.direct(f64(H), f64(W))) <= TOL[w.dtype]
    H, W, y_host = _run_offload(ctx, w, 0, host=True)
    assert oracle.rel_fro(y_host, oracle.direct(f64(H), f64(W))) <= TOL[w.dtype]


@pytest.mark.parametrize("name,calls", [("layer_f32", (0,)), ("shield_bf16", (0,)), ("prefill_bf16", (0, 1))])
def test_offload_full_size_sampled_rows(ctx, oracle, name, calls):
    """Full-size workloads in the benchmark's launch configuration; the oracle computes a row
    sample of H W (every output row has the same error law)."""
    w = inputs.WORKLOADS[name]
    for call in calls:
        H, W, y = _run_offload(ctx, w, call)
        assert np.isfinite(y).all()
        rows = sample_rows(w.n, 96, seed=call, extra=(w.n - w.k - 1, w.n - w.k))
        ref = oracle.rows_times_w(f64(H), f64(W), rows)
        assert oracle.rel_fro(y[rows], ref) <= TOL[w.dtype]
        # no single entry far off either: an error at the tolerance has an rms of TOL * rms(ref) per entry
        assert np.max(np.abs(y[rows] - ref)) <= 8 * TOL[w.dtype] * np.sqrt(np.mean(ref * ref))
        # property that holds at any size: column sums of Y equal (1^T H) W
        colsum_ref = (f64(H).sum(axis=0)[None, :] @ f64(W)).ravel()
        scale = np.linalg.norm(y, axis=0).mean() * np.sqrt(w.n)
        assert np.max(np.abs(y.sum(axis=0) - colsum_ref)) <= 5 * TOL[w.dtype] * scale


def test_offload_is_deterministic(ctx):
    w = inputs.WORKLOADS["decode_bf16"]
    _, _, y1 = _run_offload(ctx, w, 3)
    _, _, y2 = _run_offload(ctx, w, 3)
    assert np.array_equal(y1, y2)


# ------------------------------------------------------------------------- host-side checks

def test_argument_errors(ctx):
    n, d, p = 16, 64, 192
    H = torch.zeros((n, d), device="cuda"); W = torch.zeros((d, p), device="cuda")
    Q = torch.zeros((n, p // 3), device="cuda"); K = Q.clone(); V = Q.clone()
    L = binding.load_library()
    h = ctx._h
    st = torch.cuda.current_stream().cuda_stream
    bad = L.gelo_qkv_offload
    assert bad(h, None, W.data_ptr(), n, 0, d, p, 0, 0, 0.0, 0, Q.data_ptr(), K.data_ptr(), V.data_ptr(), st) == binding.ERR_INVALID
    assert bad(h, H.data_ptr(), W.data_ptr(), n, -1, d, p, 0, 0, 0.0, 0, Q.data_ptr(), K.data_ptr(), V.data_ptr(), st) == binding.ERR_INVALID
    assert bad(h, H.data_ptr(), W.data_ptr(), n, 0, d, p, 5, 0, 0.0, 0, Q.data_ptr(), K.data_ptr(), V.data_ptr(), st) == binding.ERR_INVALID
    assert bad(h, H.data_ptr(), W.data_ptr(), n, 0, d, p, 0, 0, 0.0, 9, Q.data_ptr(), K.data_ptr(), V.data_ptr(), st) == binding.ERR_INVALID
    assert bad(h, H.data_ptr(), W.data_ptr(), n, 0, d, p, 0, 0, 0.0, 0, Q.data_ptr(), K.data_ptr(), None, st) == binding.ERR_INVALID
    # p not divisible by 3 with a split requested
    assert bad(h, H.data_ptr(), W.data_ptr(), n, 0, d, 200, 0, 0, 0.0, 0, Q.data_ptr(), K.data_ptr(), V.data_ptr(), st) == binding.ERR_UNSUPPORTED
    # stride of A too small / not a multiple of 8
    A = torch.zeros((n, 64), device="cuda")
    assert L.gelo_mix(h, A.data_ptr(), 12, H.data_ptr(), None, n, 0, d, 0, H.data_ptr(), st) == binding.ERR_INVALID
    assert L.gelo_mix(h, A.data_ptr(), 20, H.data_ptr(), None, n, 0, d, 0, H.data_ptr(), st) == binding.ERR_INVALID
    # shields announced without a pointer
    assert L.gelo_mix(h, A.data_ptr(), 64, H.data_ptr(), None, n, 2, d, 0, H.data_ptr(), st) == binding.ERR_INVALID


def test_workspace_errors():
    c = binding.Context(0)
    n, d, p = 16, 64, 192
    H = torch.zeros((n, d), device="cuda"); W = torch.zeros((d, p), device="cuda")
    Q = torch.zeros((n, p), device="cuda")
    with pytest.raises(binding.GeloError) as e:
        c.qkv_offload(H, W, n, 0, d, p, 0, 0, 0.0, "f32", Q)
    assert e.value.status == binding.ERR_WORKSPACE
    c.set_workspace(torch.empty(1024, dtype=torch.uint8, device="cuda"))
    with pytest.raises(binding.GeloError) as e:
        c.qkv_offload(H, W, n, 0, d, p, 0, 0, 0.0, "f32", Q)
    assert e.value.status == binding.ERR_WORKSPACE
    c.ensure_workspace(n, 0, d, p, "f32")
    c.qkv_offload(H, W, n, 0, d, p, 0, 0, 0.0, "f32", Q)
    torch.cuda.synchronize()
    assert c.launch_count() > 0 and c.last_status() == binding.OK
    c.close()


# ------------------------------------------------------------------------- batched calls

@pytest.mark.parametrize("name,calls,lanes", [("tiny_f32", 6, 4), ("decode_bf16", 5, 2), ("decode_bf16", 3, 8)])
def test_batched_offload_matches_single_calls(oracle, name, calls, lanes):
    """Concurrent sampling lanes must not change any result: same bytes as one call at a time."""
    w = inputs.WORKLOADS[name]
    n, k, d, p = w.n, w.k, w.d, w.p
    c = binding.Context(0)
    c.set_lanes(lanes)
    c.ensure_batch_workspace(n, k, d, p, w.dtype, lanes)
    kinds = [ORTHOGONAL if i % 2 == 0 else NONORTHOGONAL for i in range(calls)]
    Hs, Ws, seeds = [], [], []
    for i in range(calls):
        H, W, seed = inputs.make_call_inputs(w, i, "cuda")
        Hs.append(H); Ws.append(W); seeds.append(seed)
    td = TDT[w.dtype]
    mk = lambda: [torch.full((n, p // 3), float("nan"), device="cuda", dtype=td) for _ in range(calls)]
    Qb, Kb, Vb = mk(), mk(), mk()
    c.qkv_offload_batch(Hs, Ws, n, k, d, p, kinds, seeds, w.shield_scale, w.dtype, Qb, Kb, Vb)
    torch.cuda.synchronize()
    assert c.last_status() == binding.OK
    for i in range(calls):
        Q = torch.empty((n, p // 3), device="cuda", dtype=td); K = torch.empty_like(Q); V = torch.empty_like(Q)
        c.qkv_offload(Hs[i], Ws[i], n, k, d, p, kinds[i], seeds[i], w.shield_scale, w.dtype, Q, K, V)
        torch.cuda.synchronize()
        assert torch.equal(Q, Qb[i]) and torch.equal(K, Kb[i]) and torch.equal(V, Vb[i])
        y = np.hstack([f64(Qb[i]), f64(Kb[i]), f64(Vb[i])])
        assert oracle.rel_fro(y, oracle.direct(f64(Hs[i]), f64(Ws[i]))) <= TOL[w.dtype]
    # host variant
    Hh = [h.cpu().pin_memory() for h in Hs]
    mkh = lambda: [torch.empty((n, p // 3), dtype=td).pin_memory() for _ in range(calls)]
    Qh, Kh, Vh = mkh(), mkh(), mkh()
    c.qkv_offload_batch_host(Hh, Ws, n, k, d, p, kinds, seeds, w.shield_scale, w.dtype, Qh, Kh, Vh)
    for i in range(calls):
        assert torch.equal(Qh[i], Qb[i].cpu()) and torch.equal(Vh[i], Vb[i].cpu())
    # the variant that does not wait: two batches back to back, results valid after the stream is synchronised
    Qa, Ka, Va = mkh(), mkh(), mkh()
    Q2, K2, V2 = mkh(), mkh(), mkh()
    c.qkv_offload_batch_host_async(Hh, Ws, n, k, d, p, kinds, seeds, w.shield_scale, w.dtype, Qa, Ka, Va)
    c.qkv_offload_batch_host_async(Hh, Ws, n, k, d, p, kinds, seeds, w.shield_scale, w.dtype, Q2, K2, V2)
    torch.cuda.synchronize()
    for i in range(calls):
        assert torch.equal(Qa[i], Qh[i]) and torch.equal(Ka[i], Kh[i]) and torch.equal(Va[i], Vh[i])
        assert torch.equal(Q2[i], Qh[i]) and torch.equal(V2[i], Vh[i])
    assert c.last_status() == binding.OK
    c.close()


def test_small_batches_back_to_back_follow_the_callers_stream(oracle):
    """Small batches run whole calls on the lanes.  A second batch whose inputs are produced on the caller's stream
    AFTER the first batch (from the first batch's outputs) must see them, and the lanes that run on across the seam
    must not overwrite outputs that the caller's stream still reads."""
    w = inputs.WORKLOADS["decode_bf16"]
    n, k, d, p = w.n, w.k, w.d, w.p
    calls, lanes = 12, 4
    c = binding.Context(0)
    c.set_lanes(lanes)
    c.ensure_batch_workspace(n, k, d, p, w.dtype, lanes)
    kinds = [ORTHOGONAL if i % 3 else NONORTHOGONAL for i in range(calls)]
    Hs, Ws, seeds = [], [], []
    for i in range(calls):
        H, W, seed = inputs.make_call_inputs(w, i, "cuda")
        Hs.append(H); Ws.append(W); seeds.append(seed)
    mk = lambda: [torch.full((n, p // 3), float("nan"), device="cuda", dtype=torch.bfloat16) for _ in range(calls)]
    Q1, K1, V1 = mk(), mk(), mk()
    Q2, K2, V2 = mk(), mk(), mk()
    torch.cuda.synchronize()
    c.qkv_offload_batch(Hs, Ws, n, k, d, p, kinds, seeds, w.shield_scale, w.dtype, Q1, K1, V1)
    # next layer's activations from this layer's outputs, on the caller's stream (d = p / 3 here)
    H2 = [(0.5 * (Q1[i] + V1[i]) + Hs[i]).contiguous() for i in range(calls)]
    seeds2 = [s_ + 999 for s_ in seeds]
    c.qkv_offload_batch(H2, Ws, n, k, d, p, kinds, seeds2, w.shield_scale, w.dtype, Q2, K2, V2)
    # the first batch's outputs are consumed after the second batch was enqueued
    sums = [Q1[i].float().sum() + K1[i].float().sum() for i in range(calls)]
    torch.cuda.synchronize()
    assert c.last_status() == binding.OK
    for i in range(calls):
        Q = torch.empty((n, p // 3), device="cuda", dtype=torch.bfloat16); K = torch.empty_like(Q); V = torch.empty_like(Q)
        c.qkv_offload(Hs[i], Ws[i], n, k, d, p, kinds[i], seeds[i], w.shield_scale, w.dtype, Q, K, V)
        torch.cuda.synchronize()
        assert torch.equal(Q, Q1[i]) and torch.equal(K, K1[i]) and torch.equal(V, V1[i])
        assert float(sums[i]) == float(Q.float().sum() + K.float().sum())
        h2 = (0.5 * (Q + V) + Hs[i]).contiguous()
        assert torch.equal(h2, H2[i])
        c.qkv_offload(h2, Ws[i], n, k, d, p, kinds[i], seeds2[i], w.shield_scale, w.dtype, Q, K, V)
        torch.cuda.synchronize()
        assert torch.equal(Q, Q2[i]) and torch.equal(K, K2[i]) and torch.equal(V, V2[i])
        if i in (0, 5, 11):
            y = np.hstack([f64(Q2[i]), f64(K2[i]), f64(V2[i])])
            assert oracle.rel_fro(y, oracle.direct(f64(h2), f64(Ws[i]))) <= TOL["bf16"]
    c.close()


@pytest.mark.parametrize("dtype,n,k,d,p", [("f16", 48, 5, 1024, 3072), ("bf16", 100, 0, 2048, 1536), ("bf16", 17, 3, 512, 768)])
def test_small_batches_other_shapes_and_types(oracle, dtype, n, k, d, p):
    """Whole calls on the lanes for IEEE-half storage, for a call without shield rows and for a ragged row count:
    same bytes as single calls, and H W within the 16-bit tolerance."""
    w = inputs.Workload("small", n, k, d, p, dtype, (ORTHOGONAL, NONORTHOGONAL), 10.0, True, 77, 1)
    calls, lanes = 7, 3
    c = binding.Context(0)
    c.set_lanes(lanes)
    c.ensure_batch_workspace(n, k, d, p, dtype, lanes)
    kinds = [w.kind(i) for i in range(calls)]
    Hs, Ws, seeds = [], [], []
    for i in range(calls):
        H, W, seed = inputs.make_call_inputs(w, i, "cuda")
        Hs.append(H); Ws.append(W); seeds.append(seed)
    td = TDT[dtype]
    mk = lambda: [torch.full((n, p // 3), float("nan"), device="cuda", dtype=td) for _ in range(calls)]
    Qb, Kb, Vb = mk(), mk(), mk()
    for rep in range(2):                                   # the second batch chains onto the first
        c.qkv_offload_batch(Hs, Ws, n, k, d, p, kinds, seeds, w.shield_scale, dtype, Qb, Kb, Vb)
    torch.cuda.synchronize()
    assert c.last_status() == binding.OK
    for i in range(calls):
        Q = torch.empty((n, p // 3), device="cuda", dtype=td); K = torch.empty_like(Q); V = torch.empty_like(Q)
        c.qkv_offload(Hs[i], Ws[i], n, k, d, p, kinds[i], seeds[i], w.shield_scale, dtype, Q, K, V)
        torch.cuda.synchronize()
        assert torch.equal(Q, Qb[i]) and torch.equal(K, Kb[i]) and torch.equal(V, Vb[i])
        y = np.hstack([f64(Qb[i]), f64(Kb[i]), f64(Vb[i])])
        assert oracle.rel_fro(y, oracle.direct(f64(Hs[i]), f64(Ws[i]))) <= TOL[dtype]
    c.close()


def test_small_batch_with_shared_outputs_keeps_call_order():
    """Calls of a batch may share their output buffers and are then written in call order, also for the small
    batches whose calls would otherwise run concurrently on the lanes."""
    w = inputs.WORKLOADS["decode_bf16"]
    n, k, d, p = w.n, w.k, w.d, w.p
    calls, lanes = 9, 4
    c = binding.Context(0)
    c.set_lanes(lanes)
    c.ensure_batch_workspace(n, k, d, p, w.dtype, lanes)
    Hs, Ws, seeds = [], [], []
    for i in range(calls):
        H, W, seed = inputs.make_call_inputs(w, i, "cuda")
        Hs.append(H); Ws.append(W); seeds.append(seed)
    kinds = [ORTHOGONAL] * calls
    Q = torch.full((n, p // 3), float("nan"), device="cuda", dtype=torch.bfloat16); K = Q.clone(); V = Q.clone()
    for rep in range(3):
        c.qkv_offload_batch(Hs, Ws, n, k, d, p, kinds, seeds, w.shield_scale, w.dtype, [Q] * calls, [K] * calls, [V] * calls)
    torch.cuda.synchronize()
    Ql = torch.empty_like(Q); Kl = torch.empty_like(Q); Vl = torch.empty_like(Q)
    c.qkv_offload(Hs[-1], Ws[-1], n, k, d, p, kinds[-1], seeds[-1], w.shield_scale, w.dtype, Ql, Kl, Vl)
    torch.cuda.synchronize()
    assert torch.equal(Q, Ql) and torch.equal(K, Kl) and torch.equal(V, Vl)
    # partially overlapping outputs count as shared too
    big = torch.full((2 * n, p // 3), float("nan"), device="cuda", dtype=torch.bfloat16)
    Qo = [big[: n], big[n // 2: n // 2 + n]]
    Ko = [torch.empty_like(Q) for _ in range(2)]; Vo = [torch.empty_like(Q) for _ in range(2)]
    c.qkv_offload_batch(Hs[:2], Ws[:2], n, k, d, p, kinds[:2], seeds[:2], w.shield_scale, w.dtype, Qo, Ko, Vo)
    torch.cuda.synchronize()
    c.qkv_offload(Hs[1], Ws[1], n, k, d, p, kinds[1], seeds[1], w.shield_scale, w.dtype, Ql, Kl, Vl)
    c.qkv_offload(Hs[0], Ws[0], n, k, d, p, kinds[0], seeds[0], w.shield_scale, w.dtype, Q, K, V)
    torch.cuda.synchronize()
    assert torch.equal(Qo[1], Ql) and torch.equal(big[: n // 2], Q[: n // 2])
    assert c.last_status() == binding.OK
    c.close()


# two and three lanes: projections that fit beside each other are set up under their predecessors, others are not (12, 48 and 64 CTAs per
# projection); the same bytes as call by call
@pytest.mark.parametrize("lanes,p", [(3, 768), (2, 3072), (3, 3072), (2, 4096)])
def test_small_batches_on_few_lanes_match_single_calls(lanes, p):
    n, k, d, dt, calls = 100, 5, 512, "bf16", 7
    c = binding.Context(0)
    c.set_lanes(lanes)
    c.ensure_batch_workspace(n, k, d, p, dt, lanes)
    H = [inputs.make_hidden(n, d, dt, 40 + i, True, "cuda") for i in range(calls)]
    W = [inputs.make_weight(d, p, dt, 90 + i, "cuda") for i in range(calls)]
    kinds = [(ORTHOGONAL, NONORTHOGONAL)[i % 2] for i in range(calls)]
    Y = torch.zeros((2, calls, n, p), dtype=torch.bfloat16, device="cuda")
    for _ in range(2):
        c.qkv_offload_batch(H, W, n, k, d, p, kinds, list(range(calls)), 10.0, dt, list(Y[0]))
    for i in range(calls):
        c.qkv_offload(H[i], W[i], n, k, d, p, kinds[i], i, 10.0, dt, Y[1, i])
    torch.cuda.synchronize()
    assert c.last_status() == binding.OK and torch.equal(Y[0], Y[1])
    c.close()


# a call that reads the result of the one before it, on the sizes whose calls run on their lanes (fused, and with products of their own)
# and on one that never does
@pytest.mark.parametrize("n,k", [(64, 4), (300, 15), (2300, 20)])
def test_batched_calls_that_read_earlier_results_run_in_call_order(n, k):
    d, dt, calls = 256, "bf16", 7
    c = binding.Context(0)
    c.set_lanes(6)
    c.ensure_batch_workspace(n, k, d, d, dt, 6)
    W = [inputs.make_weight(d, d, dt, 90 + i, "cuda") * 3.0 for i in range(calls)]       # (keeps the scale of the rows)
    chain = torch.zeros((calls + 1, n, d), dtype=torch.bfloat16, device="cuda")
    for _ in range(2):
        chain.zero_()
        chain[0] = inputs.make_hidden(n, d, dt, 40, True, "cuda")
        rows = [chain[i] for i in range(calls + 1)]
        torch.cuda._sleep(20_000_000)                # every call is enqueued before the first one starts
        c.qkv_offload_batch(rows[:-1], W, n, k, d, d, [ORTHOGONAL] * calls, [500 + i for i in range(calls)], 10.0, dt, rows[1:])
        torch.cuda.synchronize()
        assert c.last_status() == binding.OK
        for i in range(calls):
            ref = chain[i].double() @ W[i].double()
            assert ref.norm() > 0 and ((chain[i + 1].double() - ref).norm() / ref.norm()).item() <= TOL[dt]
    c.close()


def test_batched_calls_in_place_stay_independent():
    """A result that replaces the call's own H concerns no other call: the same bytes as with buffers of their own."""
    for n, k in ((64, 4), (300, 15)):
        d, dt, calls = 256, "bf16", 7
        c = binding.Context(0)
        c.set_lanes(6)
        c.ensure_batch_workspace(n, k, d, d, dt, 6)
        H = torch.stack([inputs.make_hidden(n, d, dt, 40 + i, True, "cuda") for i in range(calls)])
        W = [inputs.make_weight(d, d, dt, 90 + i, "cuda") for i in range(calls)]
        kinds = [(ORTHOGONAL, NONORTHOGONAL)[i % 2] for i in range(calls)]
        Y = torch.zeros_like(H)
        for out in (Y, H):
            c.qkv_offload_batch(list(H), W, n, k, d, d, kinds, [500 + i for i in range(calls)], 10.0, dt, list(out))
        torch.cuda.synchronize()
        assert c.last_status() == binding.OK and torch.equal(H, Y) and Y.abs().sum() > 0
        c.close()



def test_batched_offload_full_size(oracle):
    w = inputs.WORKLOADS["prefill_bf16"]
    n, k, d, p = w.n, w.k, w.d, w.p
    calls = 20                      # the benchmark's configuration: 16 lanes, a quarter of the SMs per level-3 update
    c = binding.Context(0)
    c.set_lanes(16)
    c.ensure_batch_workspace(n, k, d, p, w.dtype, 16)
    Hs, Ws, seeds = [], [], []
    for i in range(calls):
        H, W, seed = inputs.make_call_inputs(w, i, "cuda")
        Hs.append(H); Ws.append(W); seeds.append(seed)
    kinds = [w.kind(i) for i in range(calls)]
    outs = [[torch.empty((n, p // 3), device="cuda", dtype=torch.bfloat16) for _ in range(calls)] for _ in range(3)]
    c.qkv_offload_batch(Hs, Ws, n, k, d, p, kinds, seeds, w.shield_scale, w.dtype, *outs)
    torch.cuda.synchronize()
    assert c.last_status() == binding.OK
    for i in (0, 7, 19):
        y = np.hstack([f64(outs[0][i]), f64(outs[1][i]), f64(outs[2][i])])
        rows = sample_rows(n, 48, seed=i, extra=(n - k - 1, n - k))
        ref = oracle.rows_times_w(f64(Hs[i]), f64(Ws[i]), rows)
        assert oracle.rel_fro(y[rows], ref) <= TOL["bf16"]
        assert np.max(np.abs(y[rows] - ref)) <= 8 * TOL["bf16"] * np.sqrt(np.mean(ref * ref))
    c.close()


# ------------------------------------------------------------------------- split-precision tensor-core update

@pytest.mark.parametrize("M,N,K", [(128, 256, 128), (300, 520, 128), (1000, 777, 96), (4300, 4172, 128), (64, 8, 32),
                                    (130, 1, 5)])
def test_tensor_core_update_f32(ctx, oracle, M, N, K):
    rng = np.random.default_rng(M + N + K)
    A = dev(rng.standard_normal((M, K)).astype(np.float32))
    B = dev(rng.standard_normal((K, N)).astype(np.float32))
    ldc = ((N + 63) // 64) * 64
    C = torch.zeros((M, ldc), device="cuda", dtype=torch.float32)
    C0 = rng.standard_normal((M, N)).astype(np.float32)
    C[:, :N] = dev(C0)
    ctx.update_f32(M, N, K, A, K, B, N, C, ldc)
    ref = C0.astype(np.float64) - (oracle.matmul(f64(A), f64(B)) if M * N * K < 3e8 else f64(A) @ f64(B))
    got = f64(C[:, :N])
    # bf16 (high, low) pairs carry 16 significand bits: products are good to about 2^-16
    assert np.linalg.norm(got - ref) / np.linalg.norm(ref) <= 2e-5
    assert np.max(np.abs(got - ref)) <= 4e-4 * np.sqrt(K)


@pytest.mark.parametrize("m", [130, 257, 512, 1000])
def test_lu_inverse_tensor_core_blocks(oracle, m):
    c = make_ctx(m, 0, 8, 24, "f32")
    c.set_level3(2)
    ld = c.mixing_ld(m)
    A64, _ = oracle.sample_mixing(m, 1, seed=400 + m)
    A64 = A64.astype(np.float32).astype(np.float64)
    A = padded(m, ld, torch.float32); A[:, :m] = dev(A64)
    X = padded(m, ld, torch.float32)
    c.lu_inverse(m, A, ld, X)
    x = f64(X[:, :m])
    # operands carried as bf16 (high, low) pairs have 16 significand bits (2^-17 each); the two triangular
    # solves amplify that by the conditioning of L and U: a few 1e-4 at kappa(A) ~ 5, far inside the bf16
    # path's budget (A^-1 is rounded to bf16, 4e-3, right afterwards)
    assert oracle.rel_fro(x, oracle.lu_inverse(A64)) <= 1e-3
    assert np.linalg.norm(A64 @ x - np.eye(m)) / np.sqrt(m) <= 1e-3
    assert c.last_status() == binding.OK
    c.close()


@pytest.mark.parametrize("m", [100, 130, 257, 512, 1000])
def test_householder_qr_tensor_core_blocks(oracle, m):
    c = make_ctx(m, 0, 8, 24, "f32")
    c.set_level3(2)
    ld = c.mixing_ld(m)
    G64 = oracle.gaussian(500 + m, 0, 0, m, m).astype(np.float32).astype(np.float64)
    G = padded(m, ld, torch.float32); G[:, :m] = dev(G64)
    Q = padded(m, ld, torch.float32)
    c.qr_orthogonal(m, G, ld, Q)
    q = f64(Q[:, :m]); r = np.triu(f64(G[:, :m]))
    s = np.where(np.diag(r) < 0, -1.0, 1.0)
    # split-precision products (16 significand bits per operand): defects of a few 1e-5, against 1.6e-3 from
    # rounding A to bf16 afterwards
    assert np.linalg.norm(q.T @ q - np.eye(m)) / np.sqrt(m) <= 2e-4
    assert np.linalg.norm(q @ (r.T * s).T - G64) / np.linalg.norm(G64) <= 2e-4
    q_ref, _ = oracle.householder_qr(G64)
    assert np.all(np.sum(q * q_ref, axis=0)[: max(1, m // 2)] > 1 - 2e-3)
    assert c.last_status() == binding.OK
    c.close()


# ------------------------------------------------------------------------- tf32 tensor-core updates

@pytest.mark.parametrize("M,N,K", [(128, 256, 128), (300, 520, 128), (1000, 776, 96), (4300, 4172, 128), (64, 8, 32),
                                    (130, 4, 8)])
def test_tensor_core_update_tf32(ctx, oracle, M, N, K):
    """C -= A B as one tf32 product straight from the fp32 operands (no operand conversion passes)."""
    rng = np.random.default_rng(M + N + K)
    lda = (K + 3) // 4 * 4
    ldb = (N + 63) // 64 * 64
    A0 = rng.standard_normal((M, K)).astype(np.float32)
    B0 = rng.standard_normal((K, N)).astype(np.float32)
    C0 = rng.standard_normal((M, N)).astype(np.float32)
    A = torch.zeros((M, lda), device="cuda"); A[:, :K] = dev(A0)
    B = padded(K, ldb, torch.float32); B[:, :N] = dev(B0)
    C = padded(M, ldb, torch.float32); C[:, :N] = dev(C0)
    ctx.set_level3(3)
    try:
        ctx.update_f32(M, N, K, A, lda, B, ldb, C, ldb)
    finally:
        ctx.set_level3(0)
    a64, b64 = A0.astype(np.float64), B0.astype(np.float64)
    prod = oracle.matmul(a64, b64) if M * N * K < 3e8 else a64 @ b64
    got = f64(C[:, :N])
    err = got - (C0.astype(np.float64) - prod)
    # the tensor core keeps 10 fraction bits of each operand and drops the rest: every term loses up to 2^-10 per
    # operand, 2^-11 / (2 ln 2) on average for log-uniformly spread mantissas, i.e. 7.0e-4 for the product
    assert np.linalg.norm(err) / np.linalg.norm(prod) <= 1.2e-3
    loss = np.sum(err * prod) / np.sum(prod * prod)          # C - (1 - loss) A B against C - A B
    if M * N >= 128 * 256:
        assert abs(loss - 2 * 3.5224e-4) <= 5e-5
    assert torch.isnan(C[:, N:]).all()                     # padding columns are never written


@pytest.mark.parametrize("m", [100, 130, 257, 512, 1000, 2300, 2700])
def test_householder_qr_tf32_blocks(oracle, m):
    """QR with tf32 level-3 updates and the Newton-Schulz polish, as the bf16 path runs it (2300 and 2700 rows: five and six
    superblocks, the last one partial)."""
    c = make_ctx(m, 0, 8, 24, "f32")
    c.set_level3(3)
    ld = c.mixing_ld(m)
    G64 = oracle.gaussian(500 + m, 0, 0, m, m).astype(np.float32).astype(np.float64)
    G = padded(m, ld, torch.float32); G[:, :m] = dev(G64)
    Q = padded(m, ld, torch.float32)
    c.qr_orthogonal(m, G, ld, Q)
    q = f64(Q[:, :m]); r = np.triu(f64(G[:, :m]))
    s = np.where(np.diag(r) < 0, -1.0, 1.0)
    d = q.T @ q - np.eye(m)
    # polished: what is left is the zero-mean tf32 noise of Q^T Q (about 3e-4), far below the 1.6e-3 that rounding A
    # to bf16 adds afterwards; the trace shows that no coherent shrinkage survives
    assert np.linalg.norm(d) / np.sqrt(m) <= 6e-4
    assert abs(np.trace(d)) / m <= 1e-4
    # the factorisation itself is tf32-grade
    assert np.linalg.norm(q @ (r.T * s).T - G64) / np.linalg.norm(G64) <= 5e-3
    q_ref, _ = oracle.householder_qr(G64)
    assert np.all(np.sum(q * q_ref, axis=0)[: max(1, m // 2)] > 1 - 5e-3)
    assert c.last_status() == binding.OK
    c.close()


def test_orthogonal_sample_bf16_benchmark_size(ctx):
    """Orthogonal A at the benchmark size on the default (tf32 + polish) route: A^T A = I up to bf16 rounding."""
    m = 4300
    lda = ctx.mixing_ld(m)
    A = padded(m, lda, torch.bfloat16); X = padded(m, lda, torch.bfloat16)
    ctx.sample_mixing(m, ORTHOGONAL, 31337, "bf16", A, X, lda)
    a = A[:, :m].double()
    assert torch.equal(X[:, :m], A[:, :m].t())
    d = a.t() @ a - torch.eye(m, device="cuda", dtype=torch.float64)
    # bf16 rounding alone: relative errors uniform in +-2^-9 on both factors of every term, 2^-9 sqrt(2/3) = 1.6e-3
    # per off-diagonal entry pair and twice that on the diagonal, 2.35e-3 in this norm; the polished Q adds 3e-4
    assert d.norm().item() / np.sqrt(m) <= 2.6e-3
    assert abs(torch.trace(d).item()) / m <= 2e-4
    # bit-reproducible at this size too (nine superblocks, split-K sums in fixed order), for both kinds
    A2 = padded(m, lda, torch.bfloat16); X2 = padded(m, lda, torch.bfloat16)
    ctx.sample_mixing(m, ORTHOGONAL, 31337, "bf16", A2, X2, lda)
    assert torch.equal(A2[:, :m], A[:, :m])
    ctx.sample_mixing(m, NONORTHOGONAL, 31337, "bf16", A, X, lda)
    ctx.sample_mixing(m, NONORTHOGONAL, 31337, "bf16", A2, X2, lda)
    assert torch.equal(A2[:, :m], A[:, :m]) and torch.equal(X2[:, :m], X[:, :m])
    r = X[:, :m].double() @ A[:, :m].double() - torch.eye(m, device="cuda", dtype=torch.float64)
    assert r.norm().item() / np.sqrt(m) <= 4e-3            # measured 2.5e-3: bf16 rounding of A^-1 plus the LU's 1.3e-3


# ------------------------------------------------------------------------- attention output projection

@pytest.mark.parametrize("dt", ["f32", "bf16"])
@pytest.mark.parametrize("kind", [ORTHOGONAL, NONORTHOGONAL])
def test_output_projection_unsplit(ctx, oracle, dt, kind):
    """The same procedure on the attention output projection O: a d x d weight, one unsplit result."""
    n, k, d = 320, 16, 512
    p = d
    ctx.ensure_workspace(n, k, d, p, dt)
    H = inputs.make_hidden(n, d, dt, 41, True, "cuda")
    W = inputs.make_weight(d, p, dt, 41, "cuda")
    Y = torch.full((n, p), float("nan"), device="cuda", dtype=TDT[dt])
    ctx.qkv_offload(H, W, n, k, d, p, kind, 4242, 10.0, dt, Y)
    torch.cuda.synchronize()
    assert oracle.rel_fro(f64(Y), oracle.direct(f64(H), f64(W))) <= TOL[dt]


@pytest.mark.parametrize("p,kind", [(4096, ORTHOGONAL), (11008, NONORTHOGONAL)])
def test_unsplit_projections_full_size(ctx, oracle, p, kind):
    """The attention output projection (p = d) and an MLP up-projection (p = 11008, not a multiple of the 256-column
    tiles) at n = 4096, d = 4096 with 204 shield rows: sampled rows against the oracle's H W."""
    n, k, d = 4096, 204, 4096
    ctx.ensure_workspace(n, k, d, p, "bf16")
    H = inputs.make_hidden(n, d, "bf16", 51, True, "cuda")
    W = inputs.make_weight(d, p, "bf16", 51, "cuda")
    Y = torch.full((n, p), float("nan"), device="cuda", dtype=torch.bfloat16)
    ctx.qkv_offload(H, W, n, k, d, p, kind, 5151, 10.0, "bf16", Y)
    torch.cuda.synchronize()
    assert ctx.last_status() == binding.OK
    assert torch.isfinite(Y).all()
    rows = sample_rows(n, 64, seed=p)
    ref = oracle.rows_times_w(f64(H), f64(W), rows)
    y = f64(Y[rows])
    assert oracle.rel_fro(y, ref) <= TOL["bf16"]
    assert np.max(np.abs(y - ref)) <= 8 * TOL["bf16"] * np.sqrt(np.mean(ref * ref))


# ------------------------------------------------------------------------- block-diagonal variant

@pytest.mark.parametrize("dt,n,k,d,block,split", [("bf16", 1024, 52, 512, 256, True), ("f32", 300, 20, 256, 128, True),
                                                   ("bf16", 700, 0, 512, 192, False), ("bf16", 4096, 204, 4096, 512, True)])
def test_block_diagonal_variant(oracle, dt, n, k, d, block, split):
    """Block-diagonal orthogonal A: every group mixes its share of shield rows with its data rows, and the result
    is H W whatever the grouping (Eq. 4 holds for any invertible A)."""
    p = 3 * d if split else d
    calls = 3
    c = binding.Context(0)
    c.set_lanes(16)
    c.ensure_blockdiag_workspace(n, k, d, p, dt, block, 16)
    Hs = [inputs.make_hidden(n, d, dt, 60 + i, True, "cuda") for i in range(calls)]
    Ws = [inputs.make_weight(d, p, dt, 60 + i, "cuda") for i in range(calls)]
    mk = lambda cols: [torch.full((n, cols), float("nan"), device="cuda", dtype=TDT[dt]) for _ in range(calls)]
    if split:
        Q, K, V = mk(p // 3), mk(p // 3), mk(p // 3)
        c.qkv_offload_blockdiag_batch(Hs, Ws, n, k, d, p, block, [500 + i for i in range(calls)], 10.0, dt, Q, K, V)
    else:
        Q = mk(p)
        c.qkv_offload_blockdiag_batch(Hs, Ws, n, k, d, p, block, [500 + i for i in range(calls)], 10.0, dt, Q)
    torch.cuda.synchronize()
    assert c.last_status() == binding.OK
    for i in range(calls):
        y = np.hstack([f64(Q[i]), f64(K[i]), f64(V[i])]) if split else f64(Q[i])
        if n * d * p < 2e9:
            assert oracle.rel_fro(y, oracle.direct(f64(Hs[i]), f64(Ws[i]))) <= TOL[dt]
        else:
            rows = sample_rows(n, 48, seed=i, extra=[n * j // 9 + e for j in range(1, 9) for e in (-1, 0)])
            assert oracle.rel_fro(y[rows], oracle.rows_times_w(f64(Hs[i]), f64(Ws[i]), rows)) <= TOL[dt]
    # a different seed draws different A_j and still lands on the same product
    Q2, K2, V2 = mk(p // 3 if split else p), mk(p // 3), mk(p // 3)
    if split:
        c.qkv_offload_blockdiag_batch(Hs[:1], Ws[:1], n, k, d, p, block, [99], 10.0, dt, Q2[:1], K2[:1], V2[:1])
    else:
        c.qkv_offload_blockdiag_batch(Hs[:1], Ws[:1], n, k, d, p, block, [99], 10.0, dt, Q2[:1])
    torch.cuda.synchronize()
    assert oracle.rel_fro(f64(Q2[0]), f64(Q[0])) <= 2 * TOL[dt]
    if dt == "bf16":
        assert not torch.equal(Q2[0], Q[0])                   # rounding differs with A: the mixing really changed
    # unsupported groupings are refused before any launch
    L = binding.load_library()
    assert L.gelo_blockdiag_workspace_bytes(n, k, d, p, binding.dtype_code(dt), 100, 16) == 0       # not a multiple of 64
    assert L.gelo_blockdiag_workspace_bytes(4096, 0, d, p, binding.dtype_code(dt), 64, 16) == 0     # 64 groups > 32 lanes
    c.close()


@pytest.mark.parametrize("d,p", [(512, 1376), (1376, 512)])
def test_mlp_shaped_projections(ctx, oracle, d, p):
    """The same procedure on MLP-shaped weights (up: d -> 2.6875 d, down: back), one unsplit result, widths that are
    not multiples of the 256-column tiles."""
    n, k = 320, 16
    ctx.ensure_workspace(n, k, d, p, "bf16")
    H = inputs.make_hidden(n, d, "bf16", 43, True, "cuda")
    W = inputs.make_weight(d, p, "bf16", 43, "cuda")
    for kind in (ORTHOGONAL, NONORTHOGONAL):
        Y = torch.full((n, p), float("nan"), device="cuda", dtype=torch.bfloat16)
        ctx.qkv_offload(H, W, n, k, d, p, kind, 4343, 10.0, "bf16", Y)
        torch.cuda.synchronize()
        assert oracle.rel_fro(f64(Y), oracle.direct(f64(H), f64(W))) <= TOL["bf16"]


# ------------------------------------------------------------------------- IEEE half storage

@pytest.mark.parametrize("kind", [ORTHOGONAL, NONORTHOGONAL])
@pytest.mark.parametrize("n,k,d", [(64, 4, 256), (600, 30, 512), (2048, 102, 1024)])
def test_half_precision_path(ctx, oracle, kind, n, k, d):
    """fp16 operands (the third precision of the paper's functional-equality table): whole path and stages."""
    p = 3 * d
    m = n + k
    ctx.ensure_workspace(n, k, d, p, "f16")
    H = inputs.make_hidden(n, d, "f16", 71, True, "cuda")
    W = inputs.make_weight(d, p, "f16", 71, "cuda")
    Q = torch.full((n, d), float("nan"), device="cuda", dtype=torch.float16); K = Q.clone(); V = Q.clone()
    ctx.qkv_offload(H, W, n, k, d, p, kind, 7171, 10.0, "f16", Q, K, V)
    torch.cuda.synchronize()
    y = np.hstack([f64(Q), f64(K), f64(V)])
    assert oracle.rel_fro(y, oracle.direct(f64(H), f64(W))) <= TOL["f16"]
    # stages on their own: stored A against its stored inverse, shield rows against the oracle, one product
    lda = ctx.mixing_ld(m)
    A = padded(m, lda, torch.float16); X = padded(m, lda, torch.float16)
    ctx.sample_mixing(m, kind, 99, "f16", A, X, lda)
    a, x = f64(A[:, :m]), f64(X[:, :m])
    assert np.linalg.norm(x @ a - np.eye(m)) / np.sqrt(m) <= (1e-3 if kind == ORTHOGONAL else 3e-3)
    if kind == ORTHOGONAL:
        assert np.array_equal(x, a.T)
    S = torch.full((k, d), float("nan"), device="cuda", dtype=torch.float16)
    ctx.shield_rows(H, n, d, k, 10.0, 5, "f16", S)
    assert oracle.rel_fro(f64(S), oracle.shield_rows(f64(H), k, 10.0, 5)) <= 6e-4
    U = torch.full((m, d), float("nan"), device="cuda", dtype=torch.float16)
    ctx.mix(A, lda, H, S, n, k, d, "f16", U)
    ref = oracle.matmul(a, np.vstack([f64(H), f64(S)])) if m * m * d < 3e8 else a @ np.vstack([f64(H), f64(S)])
    assert oracle.rel_fro(f64(U), ref) <= 6e-4


def test_batch_of_zero_calls_and_bad_batches():
    c = binding.Context(0)
    c.ensure_batch_workspace(64, 0, 64, 192, "f32", 2)
    c.qkv_offload_batch([], [], 64, 0, 64, 192, [], [], 0.0, "f32", [], [], [])       # nothing to do
    H = torch.zeros((64, 64), device="cuda"); W = torch.zeros((64, 192), device="cuda")
    Q = torch.zeros((64, 64), device="cuda")
    with pytest.raises(binding.GeloError) as e:                                        # unknown mixing kind
        c.qkv_offload_batch([H], [W], 64, 0, 64, 192, [7], [0], 0.0, "f32", [Q], [Q], [Q])
    assert e.value.status == binding.ERR_INVALID
    with pytest.raises(binding.GeloError) as e:                                        # K given, V missing
        c.qkv_offload_batch([H], [W], 64, 0, 64, 192, [0], [0], 0.0, "f32", [Q], [Q], [None])
    assert e.value.status == binding.ERR_INVALID
    c.set_workspace(torch.empty(4096, dtype=torch.uint8, device="cuda"))
    with pytest.raises(binding.GeloError) as e:
        c.qkv_offload_batch([H], [W], 64, 0, 64, 192, [0], [0], 0.0, "f32", [Q], [Q], [Q])
    assert e.value.status == binding.ERR_WORKSPACE
    c.close()


@pytest.mark.parametrize("kind", [ORTHOGONAL, NONORTHOGONAL])
def test_offload_beyond_the_register_resident_panels(oracle, kind):
    """m = 4400 rows exceed what a cluster's registers hold (4352): the first panels fall back to the
    one-CTA kernels that work out of L2, the rest use the cluster kernels."""
    n, k, d, p = 4400, 0, 64, 192
    c = binding.Context(0)
    c.ensure_workspace(n, k, d, p, "bf16")
    H = inputs.make_hidden(n, d, "bf16", 77, True, "cuda")
    W = inputs.make_weight(d, p, "bf16", 77, "cuda")
    Q = torch.empty((n, p // 3), device="cuda", dtype=torch.bfloat16); K = torch.empty_like(Q); V = torch.empty_like(Q)
    c.qkv_offload(H, W, n, k, d, p, kind, 9, 0.0, "bf16", Q, K, V)
    torch.cuda.synchronize()
    assert c.last_status() == binding.OK
    y = np.hstack([f64(Q), f64(K), f64(V)])
    assert oracle.rel_fro(y, oracle.direct(f64(H), f64(W))) <= TOL["bf16"]
    c.close()


def test_profile_counts_launches(ctx):
    w = inputs.WORKLOADS["decode_bf16"]
    H, W, seed = inputs.make_call_inputs(w, 0, "cuda")
    ctx.ensure_workspace(w.n, w.k, w.d, w.p, w.dtype)
    Q = torch.empty((w.n, w.p // 3), device="cuda", dtype=torch.bfloat16); K = torch.empty_like(Q); V = torch.empty_like(Q)
    ctx.profile_start()
    ctx.qkv_offload(H, W, w.n, w.k, w.d, w.p, ORTHOGONAL, seed, 10.0, w.dtype, Q, K, V)
    prof = ctx.profile_stop()
    assert prof["gemm_tc"]["launches"] == 1 and prof["gemm_tc"]["ms"] > 0          # project + unmix in one tensor-core kernel
    assert prof["qr_panel"]["launches"] == 0                                        # m = 68: the one-launch factorisation, no panels
    assert prof["gemm_tc"]["work"] == pytest.approx(2.0 * (68 * 4096 * 12288 + 64 * 68 * 12288))     # (the mix runs on the FMA pipes)


# ------------------------------------------------------------------------- bounded waits

def test_zero_wait_limit_reports_timeout_and_context_stays_usable(oracle):
    """With a wait limit of zero every tensor-core CTA gives up before it issues a copy or an MMA (nothing is in flight
    when it returns); the status word then says TIMEOUT, and after the limit is restored the same call is correct."""
    c = binding.Context(0)
    n, d, p = 128, 256, 768
    H = inputs.make_hidden(n, d, "bf16", 3, True, "cuda")
    W = inputs.make_weight(d, p, "bf16", 3, "cuda")
    Y = torch.full((n, p), float("nan"), device="cuda", dtype=torch.bfloat16)
    c.set_wait_limit_ns(0)
    c.project(H, W, n, d, p, "bf16", Y)
    torch.cuda.synchronize()
    assert c.last_status() == binding.ERR_TIMEOUT
    assert torch.isnan(Y).all()                            # nothing was computed, nothing was written
    assert c.last_status() == binding.OK                   # reading the status cleared it
    c.set_wait_limit_ns(2_000_000_000)
    c.project(H, W, n, d, p, "bf16", Y)
    torch.cuda.synchronize()
    assert c.last_status() == binding.OK
    assert oracle.rel_fro(f64(Y), oracle.direct(f64(H), f64(W))) <= 4e-3
    c.close()


# ------------------------------------------------------------------------- ordering of the host variants

def test_async_host_batches_of_different_shapes_back_to_back(oracle):
    """Two enqueue-only host batches of different shapes on one lane (so that both stage into the same workspace
    region), and a device call before a host batch, with no synchronisation in between: the copy streams of the
    later call must wait for the earlier call's kernels.  Results against the device-resident variant, bytewise."""
    c = binding.Context(0)
    c.set_lanes(1)
    shapes = [(192, 8, 256), (128, 4, 512)]
    need = max(int(c._lib.gelo_batch_workspace_bytes(n, k, d, 3 * d, BF16, 1)) for n, k, d in shapes)
    c.set_workspace(torch.empty(need, dtype=torch.uint8, device="cuda"))
    calls = 3
    data = []
    for (n, k, d) in shapes:
        p = 3 * d
        Hs = [inputs.make_hidden(n, d, "bf16", 60 + i, True, "cuda") for i in range(calls)]
        Ws = [inputs.make_weight(d, p, "bf16", 60 + i, "cuda") for i in range(calls)]
        Hh = [h.cpu().pin_memory() for h in Hs]
        out_h = [[torch.zeros((n, d), dtype=torch.bfloat16).pin_memory() for _ in range(calls)] for _ in range(3)]
        out_d = [[torch.empty((n, d), device="cuda", dtype=torch.bfloat16) for _ in range(calls)] for _ in range(3)]
        data.append((n, k, d, p, Hs, Ws, Hh, out_h, out_d))
    kinds = [ORTHOGONAL, NONORTHOGONAL, ORTHOGONAL]
    seeds = [900, 901, 902]
    for rep in range(3):                                   # several rounds: the race, if any, is a matter of timing
        # a single device call first (it uses the same workspace), then the two host batches, no sync in between
        n0, k0, d0, p0, Hs0, Ws0, _, _, out_d0 = data[0]
        c.qkv_offload(Hs0[0], Ws0[0], n0, k0, d0, p0, NONORTHOGONAL, 77, 10.0, "bf16", out_d0[0][0], out_d0[1][0], out_d0[2][0])
        for (n, k, d, p, Hs, Ws, Hh, out_h, out_d) in data:
            c.qkv_offload_batch_host_async(Hh, Ws, n, k, d, p, kinds, seeds, 10.0, "bf16", *out_h)
        torch.cuda.synchronize()
        assert c.last_status() == binding.OK
        for (n, k, d, p, Hs, Ws, Hh, out_h, out_d) in data:
            c.qkv_offload_batch(Hs, Ws, n, k, d, p, kinds, seeds, 10.0, "bf16", *out_d)
            torch.cuda.synchronize()
            for j in range(3):
                for i in range(calls):
                    assert torch.equal(out_h[j][i], out_d[j][i].cpu()), (rep, n, j, i)
                    out_h[j][i].zero_()
    y = np.hstack([f64(data[1][8][j][1]) for j in range(3)])
    assert oracle.rel_fro(y, oracle.direct(f64(data[1][4][1]), f64(data[1][5][1]))) <= TOL["bf16"]
    c.close()


# ------------------------------------------------------------------------- E4M3 operands for the offloaded product

@pytest.mark.parametrize("dt", ["bf16", "f32"])
@pytest.mark.parametrize("rows,cols", [(68, 4096), (300, 528), (1, 16), (4300, 1024)])
def test_e4m3_quantiser_is_bit_exact(ctx, oracle, rows, cols, dt):
    """Per-tensor E4M3 quantiser: scale and every code against the oracle's (same binary32 division, same rounding)."""
    g = torch.Generator(device="cuda"); g.manual_seed(rows + cols)
    X = (torch.randn((rows, cols), device="cuda", generator=g) * torch.rand((rows, 1), device="cuda", generator=g) * 7).to(TDT[dt])
    codes = torch.full((rows, cols), 0xAA, device="cuda", dtype=torch.uint8)
    scale = torch.zeros(2, device="cuda", dtype=torch.float32)
    ctx.quantize_e4m3(X, rows, cols, dt, codes, scale)
    torch.cuda.synchronize()
    ref_codes, ref_scale = oracle.quantize_e4m3(f64(X).astype(np.float32))
    assert np.float32(scale[0].item()) == ref_scale
    got = oracle.e4m3_decode(codes.cpu().numpy())
    assert np.array_equal(got, oracle.e4m3_decode(ref_codes))          # (compares values: +0 and -0 are the same number)
    Z = torch.zeros((8, 32), device="cuda", dtype=TDT[dt])
    zc = torch.full((8, 32), 0xAA, device="cuda", dtype=torch.uint8)
    ctx.quantize_e4m3(Z, 8, 32, dt, zc, scale)
    torch.cuda.synchronize()
    assert scale[0].item() == 1.0 and not zc.any()


@pytest.mark.parametrize("m,d,p", [(200, 1024, 768), (130, 208, 272), (68, 4096, 12288), (1, 16, 16)])
def test_e4m3_projection_stage(ctx, oracle, m, d, p):
    """Eq. 2 on E4M3 operands: the device product against the oracle's product of the SAME stored codes (what is left
    is the bf16 rounding of the output), and against the unquantised product (FP8-grade: a few percent)."""
    U = (3.0 * torch.randn((m, d), device="cuda")).to(torch.bfloat16)
    W = inputs.make_weight(d, p, "bf16", 21, "cuda")
    U8 = torch.empty((m, d), device="cuda", dtype=torch.uint8); W8 = torch.empty((d, p), device="cuda", dtype=torch.uint8)
    su = torch.zeros(2, device="cuda"); sw = torch.zeros(2, device="cuda")
    ctx.quantize_e4m3(U, m, d, "bf16", U8, su)
    ctx.quantize_e4m3(W, d, p, "bf16", W8, sw)
    Y = torch.full((m, p), float("nan"), device="cuda", dtype=torch.bfloat16)
    ctx.project_e4m3(U8, su, W8, sw, m, d, p, Y)
    torch.cuda.synchronize()
    assert ctx.last_status() == binding.OK
    ref = oracle.project_e4m3(U8.cpu().numpy(), su[0].item(), W8.cpu().numpy(), sw[0].item())
    assert oracle.rel_fro(f64(Y), ref) <= 4e-3
    if d >= 208:
        assert oracle.rel_fro(f64(Y), oracle.matmul(f64(U), f64(W))) <= 0.08


def test_e4m3_projection_full_size_and_chain(ctx, oracle):
    """The benchmark shape (m = 4300 mixed rows with 10x shield rows, d = 4096, p = 12288) on sampled rows, and what the
    FP8 product does to the whole call: bf16 mix, E4M3 projection, bf16 unmix."""
    n, k, d, p = 4096, 204, 4096, 12288
    m = n + k
    ld = ctx.mixing_ld(m)
    ctx.ensure_workspace(n, k, d, p, "bf16")
    H = inputs.make_hidden(n, d, "bf16", 61, True, "cuda")
    W = inputs.make_weight(d, p, "bf16", 61, "cuda")
    A = padded(m, ld, torch.bfloat16); X = padded(m, ld, torch.bfloat16)
    S = torch.empty((k, d), device="cuda", dtype=torch.bfloat16)
    U = torch.empty((m, d), device="cuda", dtype=torch.bfloat16)
    ctx.sample_mixing(m, ORTHOGONAL, 6161, "bf16", A, X, ld)
    ctx.shield_rows(H, n, d, k, 10.0, 6161, "bf16", S)
    ctx.mix(A, ld, H, S, n, k, d, "bf16", U)
    U8 = torch.empty((m, d), device="cuda", dtype=torch.uint8); W8 = torch.empty((d, p), device="cuda", dtype=torch.uint8)
    su = torch.zeros(2, device="cuda"); sw = torch.zeros(2, device="cuda")
    ctx.quantize_e4m3(U, m, d, "bf16", U8, su)
    ctx.quantize_e4m3(W, d, p, "bf16", W8, sw)
    Yp = torch.full((m, p), float("nan"), device="cuda", dtype=torch.bfloat16)
    ctx.project_e4m3(U8, su, W8, sw, m, d, p, Yp)
    Q = torch.empty((n, d), device="cuda", dtype=torch.bfloat16); K = torch.empty_like(Q); V = torch.empty_like(Q)
    ctx.unmix(X, ld, Yp, n, k, p, "bf16", Q, K, V)
    torch.cuda.synchronize()
    assert ctx.last_status() == binding.OK and torch.isfinite(Yp).all()
    rows = sample_rows(m, 48, seed=3, extra=(n - 1, n))
    u_dec = oracle.e4m3_decode(U8[rows].cpu().numpy()) * su[0].item()
    w_dec = oracle.e4m3_decode(W8.cpu().numpy()) * sw[0].item()
    ref = oracle.matmul(u_dec, w_dec)
    assert oracle.rel_fro(f64(Yp[rows]), ref) <= 4e-3
    # the whole call: 3 mantissa bits per operand give about 5% on Y', and the shield rows' 6x energy brings the data
    # rows to about 12% after unmixing (the bound derived for this path: 0.2)
    y = np.hstack([f64(Q), f64(K), f64(V)])
    drows = sample_rows(n, 32, seed=4)
    err = oracle.rel_fro(y[drows], oracle.rows_times_w(f64(H), f64(W), drows))
    assert 0.02 < err <= 0.2


@pytest.mark.parametrize("n,k,kind", [(255, 12, 0), (300, 1, 1)])
def test_fp32_products_of_any_depth(ctx, oracle, n, k, kind):
    """Shield rows and a K that is no multiple of four on the tf32 pairs (products above 1 GFLOP); 300 + 1 rows end a quad after one."""
    d, p = 2048, 6144
    H = inputs.make_hidden(n, d, "f32", 5, True, "cuda"); W = inputs.make_weight(d, p, "f32", 6, "cuda")
    ctx.ensure_workspace(n, k, d, p, "f32")
    Q = torch.empty((n, p), device="cuda")
    ctx.qkv_offload(H, W, n, k, d, p, kind, 77, 10.0, "f32", Q, None, None)
    torch.cuda.synchronize()
    ref = H.double() @ W.double()
    # the fp32 path's tolerance
    assert ((Q.double() - ref).norm() / ref.norm()).item() <= TOL["f32"]


# The tensor-core kernel of the large ones by itself: tiles of 256 x 192 with one row, a few columns (not whole boxes of 32) or a few k over, K from two
# k-blocks to many, whole tiles and K slices
@pytest.mark.parametrize("m,d,p", [(129, 4104, 1000), (257, 2056, 1992), (512, 40, 24600), (300, 504, 4096), (1075, 4096, 1536)])
def test_fp32_products_on_the_tensor_cores(m, d, p):
    c = binding.Context(0)
    c.ensure_workspace(m, 0, d, p, "f32")
    g = torch.Generator(device="cuda")
    g.manual_seed(m)
    U = torch.randn((m, d), generator=g, device="cuda")
    W = torch.randn((d, p), generator=g, device="cuda")
    Y = torch.full((m, p), float("nan"), device="cuda")
    c.project(U, W, m, d, p, "f32", Y)
    assert c.last_status() == binding.OK
    ref = U.double() @ W.double()
    # 24 truncated additions of 2^-25 each, half of that on the average, beside which the dropped lo lo (2^-22 of a term at most, of either sign) and the
    # sums' own rounding are small
    assert ((Y.double() - ref).norm() / ref.norm()).item() <= 8e-7
    assert (Y.double() - ref).abs().max().item() <= 1e-5 * d ** 0.5
    c.close()


# Many units per pair of CTAs, so that copies, converters, products and stores are in different ones: of a single k-block, of three (an accumulator run cut
# short), and K slices of several tiles that are not all of one length (1075 x 3072 x 1032: 33 k-blocks in slices of 9 and less)
@pytest.mark.parametrize("m,d,p", [(512, 32, 33000), (300, 96, 24600), (1075, 1032, 3072), (641, 72, 12288)])
def test_fp32_products_of_many_units(m, d, p):
    c = binding.Context(0)
    c.ensure_workspace(m, 0, d, p, "f32")
    g = torch.Generator(device="cuda"); g.manual_seed(m)
    W = torch.randn((d, p), generator=g, device="cuda")
    for i in range(3):
        U = torch.randn((m, d), generator=g, device="cuda")
        Y = torch.full((m, p), float("nan"), device="cuda")
        c.project(U, W, m, d, p, "f32", Y)
        ref = U.double() @ W.double()
        assert ((Y.double() - ref).norm() / ref.norm()).item() <= 8e-7
        assert (Y.double() - ref).abs().max().item() <= 1e-5 * d ** 0.5      # (as above)
    assert c.last_status() == binding.OK
    c.close()


# The operand pairs by themselves: U is diagonal, so every result is one product of two entries and there is nothing to add up.  With both parts rounded to
# nearest lo is half a unit of tf32 at most, 2^-11 of the entry, its own rounding 2^-23, the dropped lo lo 2^-22, and three truncated additions take up to
# 2^-23 each: 3.5 x 2^-22 in all.  Entries of 1 + 2^-10 - 2^-23 have parts of 1 + 2^-10 and -2^-23, of which only the additions lose anything; cut off
# instead of rounded, lo would be nearly 2^-10 and the dropped lo lo nearly 2^-20
@pytest.mark.parametrize("dist,bound", [("uniform", 3.5 * 2.0 ** -22), ("adverse", 1.5 * 2.0 ** -22)])
def test_fp32_operand_pairs(dist, bound):
    n, p = 512, 2048
    c = binding.Context(0)
    c.ensure_workspace(n, 0, n, p, "f32")
    g = torch.Generator(device="cuda"); g.manual_seed(5)
    W = torch.rand((n, p), generator=g, device="cuda") + 1
    u = torch.rand(n, generator=g, device="cuda") + 1
    if dist == "adverse":
        W.fill_(1 + 2.0 ** -10 - 2.0 ** -23); u.fill_(1 + 2.0 ** -10 - 2.0 ** -23)
    Y = torch.empty((n, p), device="cuda")
    c.project(torch.diag(u).contiguous(), W, n, n, p, "f32", Y)
    assert c.last_status() == binding.OK
    ref = u.double()[:, None] * W.double()
    assert ((Y.double() - ref).abs() / ref).max().item() <= bound
    c.close()


# A NaN, whatever its bits, and an infinity reach every result that their row of U or column of W takes part in, as something that is not finite, and no other;
# the largest finite values are not taken for infinities
@pytest.mark.parametrize("bits", [0x7f800001, 0xff801fff, 0x7fc00000, 0x7fffffff, 0x7f800000, 0xff800000])
def test_fp32_products_carry_what_is_not_finite(bits):
    m, d, p = 300, 512, 4096
    c = binding.Context(0)
    c.ensure_workspace(m, 0, d, p, "f32")
    g = torch.Generator(device="cuda"); g.manual_seed(9)
    U = torch.randn((m, d), generator=g, device="cuda"); W = torch.randn((d, p), generator=g, device="cuda")
    U[290, :] = 0; U[290, 7] = 3.4028e38                      # rounds up to infinity in tf32
    W[7, :] = W[7, :].clamp(-0.9, 0.9)
    ref = U.double() @ W.double()
    signed = bits - (1 << 32) if bits >= 1 << 31 else bits
    U.view(torch.int32)[17, 33] = signed
    W.view(torch.int32)[400, 1234] = signed
    Y = torch.empty((m, p), device="cuda")
    c.project(U, W, m, d, p, "f32", Y)
    assert c.last_status() == binding.OK
    hit = torch.zeros((m, p), dtype=torch.bool, device="cuda"); hit[17, :] = True; hit[:, 1234] = True
    assert not torch.isfinite(Y[hit]).any()
    if bits & 0x7fffff:
        assert torch.isnan(Y[hit]).all()
    assert torch.isfinite(Y[~hit]).all()
    assert ((Y.double() - ref)[~hit].abs() <= 1e-5 * (U.double().nan_to_num().abs() @ W.double().nan_to_num().abs())[~hit]).all()
    c.close()


# The kernel of the large fp32 products with a wait limit of zero: every role gives up before the first copy, nothing is written
def test_zero_wait_limit_reaches_the_fp32_products():
    m, d, p = 256, 256, 8192                                  # (too short for K slices, whose sum is a launch of its own)
    c = binding.Context(0)
    c.ensure_workspace(m, 0, d, p, "f32")
    g = torch.Generator(device="cuda"); g.manual_seed(2)
    U = torch.randn((m, d), generator=g, device="cuda"); W = torch.randn((d, p), generator=g, device="cuda")
    Y = torch.full((m, p), float("nan"), device="cuda")
    c.set_wait_limit_ns(0)
    c.project(U, W, m, d, p, "f32", Y)
    assert c.last_status() == binding.ERR_TIMEOUT
    assert torch.isnan(Y).all()
    c.set_wait_limit_ns(2_000_000_000)
    c.project(U, W, m, d, p, "f32", Y)
    assert c.last_status() == binding.OK
    ref = U.double() @ W.double()
    assert ((Y.double() - ref).norm() / ref.norm()).item() <= 8e-7
    c.close()


# fp32 products on either side of the lines between the two FMA kernels: 148 tiles of 64 x 64 and one more where the last stage of k is short,
# 296 and one more where it is full, with a last tile of eight columns and a K that ends a quad after two
@pytest.mark.parametrize("m,d,p", [(33, 72, 9472), (33, 72, 9480), (32, 64, 18944), (32, 64, 18952), (65, 64, 9472), (1, 8, 8)])
def test_fp32_products_on_both_fma_kernels(ctx, m, d, p):
    g = torch.Generator(device="cuda"); g.manual_seed(m + p)
    U = torch.randn((m, d), generator=g, device="cuda"); W = torch.randn((d, p), generator=g, device="cuda")
    Y = torch.full((m, p), float("nan"), device="cuda")
    ctx.project(U, W, m, d, p, "f32", Y)
    ref = U.double() @ W.double()
    # sums of 72 products in fp32
    assert ((Y.double() - ref).norm() / ref.norm()).item() <= 2e-6


# whole calls on the lanes: one over the small path, the last size that takes it and the first that does not; fewer calls than
# lanes, a second round per lane, results in one buffer that every call overwrites (call order is promised)
@pytest.mark.parametrize("n,k,calls,shared", [(120, 9, 6, False), (2200, 104, 5, False), (2201, 104, 5, False), (300, 15, 13, False), (300, 15, 7, True)])
def test_medium_batches_match_single_calls(n, k, calls, shared):
    d, p, dt = 256, 384, "bf16"
    c = binding.Context(0)
    c.set_lanes(6)
    c.ensure_batch_workspace(n, k, d, p, dt, 6)
    H = [inputs.make_hidden(n, d, dt, 40 + i, True, "cuda") for i in range(calls)]
    W = [inputs.make_weight(d, p, dt, 90 + i, "cuda") for i in range(calls)]
    out = torch.zeros((1 if shared else calls, 3, n, p // 3), dtype=torch.bfloat16, device="cuda")
    pick = lambda j: [out[0 if shared else i, j] for i in range(calls)]
    kinds = [(ORTHOGONAL, NONORTHOGONAL)[i % 2] for i in range(calls)]
    seeds = [500 + i for i in range(calls)]
    for _ in range(2):                                            # the second batch chains onto the first
        c.qkv_offload_batch(H, W, n, k, d, p, kinds, seeds, 10.0, dt, pick(0), pick(1), pick(2))
    torch.cuda.synchronize()
    assert c.last_status() == binding.OK
    for i in ([calls - 1] if shared else range(calls)):
        ref = H[i].double() @ W[i].double()
        got = torch.cat([out[0 if shared else i, j] for j in range(3)], dim=1).double()
        assert ((got - ref).norm() / ref.norm()).item() <= TOL[dt]
        if n > 1000:
            continue                                              # (sums are cut into other slices on the lanes; see the next test)
        one = torch.zeros((3, n, p // 3), dtype=torch.bfloat16, device="cuda")
        c.qkv_offload(H[i], W[i], n, k, d, p, kinds[i], seeds[i], 10.0, dt, *one)
        torch.cuda.synchronize()
        assert torch.equal(one, out[0 if shared else i])
    c.close()


def test_lanes_use_the_seeds_of_their_calls():
    """Where sums are cut differently on the lanes, results differ from those of single calls by the entries of A that round the other way
    (half of what another seed makes of the same H and W, whose roundings are all its own)."""
    n, k, d, p, dt, calls = 1000, 50, 256, 384, "bf16", 8
    c = binding.Context(0)
    c.set_lanes(6)
    c.ensure_batch_workspace(n, k, d, p, dt, 6)
    H = [inputs.make_hidden(n, d, dt, 40, True, "cuda")] * calls
    W = [inputs.make_weight(d, p, dt, 90, "cuda")] * calls
    kinds = [(ORTHOGONAL, NONORTHOGONAL)[i % 2] for i in range(calls)]
    Y = torch.zeros((2, calls, n, p), dtype=torch.bfloat16, device="cuda")
    for _ in range(2):
        c.qkv_offload_batch(H, W, n, k, d, p, kinds, [500 + i for i in range(calls)], 10.0, dt, list(Y[0]))
    for i in range(calls):
        c.qkv_offload(H[i], W[i], n, k, d, p, kinds[i], 500 + i, 10.0, dt, Y[1, i])
    torch.cuda.synchronize()
    assert c.last_status() == binding.OK
    y = Y.double()
    for i in range(calls):
        assert (y[0, i] - y[1, i]).norm() <= 0.7 * (y[0, i] - y[1, (i + 2) % calls]).norm()
    c.close()


# the median of the norms: the first size past the one-launch path, one value past a round of the CTA, more rounds, norms over six orders
# of magnitude, all norms equal, half of them equal on either side of the middle
@pytest.mark.parametrize("n,shape", [(257, "spread"), (1025, "spread"), (4096, "equal"), (3000, "half"), (2999, "half"), (5001, "spread")])
def test_shield_scale_is_the_median(ctx, oracle, n, shape):
    d, k = 16, 3
    g = torch.Generator(device="cuda"); g.manual_seed(n)
    H = torch.randn((n, d), generator=g, device="cuda")
    if shape == "spread":
        H = H * torch.exp(14.0 * torch.rand((n, 1), generator=g, device="cuda") - 7.0)
    elif shape == "equal":
        H = H[:1].repeat(n, 1)
    else:
        H[: n // 2] = H[0] * 3.0
        H[n // 2:] = H[n // 2] * 5.0
    H = H.contiguous()
    ctx.ensure_workspace(n, k, d, 48, "f32")
    S = torch.empty((k, d), device="cuda")
    ctx.shield_rows(H, n, d, k, 10.0, 91, "f32", S)
    ref = oracle.shield_rows(f64(H), k, 10.0, 91)
    assert np.max(np.abs(f64(S) - ref)) <= 2e-5 * np.max(np.abs(ref))     # an fp32 norm and one product, as in test_shield_rows

"""The sampler's own factorisation routes on the GPU (block QR of a Gaussian) against the oracle's factor."""
import numpy as np
import pytest
import torch

from paper_2603_05035_b200 import binding, inputs
from gpu_util import f64, padded

pytestmark = pytest.mark.gpu

ORTHOGONAL, NONORTHOGONAL = binding.ORTHOGONAL, binding.NONORTHOGONAL
TDT = {"f32": torch.float32, "bf16": torch.bfloat16, "f16": torch.float16}


def _sample(m, kind, seed, dt):
    c = binding.Context(0)
    c.ensure_workspace(m, 0, 8, 24, dt)
    ld = c.mixing_ld(m)
    A = padded(m, ld, TDT[dt]); X = padded(m, ld, TDT[dt])
    c.sample_mixing(m, kind, seed, dt, A, X, ld)
    assert c.last_status() == binding.OK
    c.close()
    return f64(A[:, :m]), f64(X[:, :m])


# 256: the first size of the route, blocks of 128 and 64 columns and a square of 64; 257: a square of an odd size; 383 .. 385: three
# blocks whose middle one is as wide as it gets, full, or full with an odd square; 513, 641: a second group of blocks begins
@pytest.mark.parametrize("m", [256, 257, 383, 384, 385, 513, 641])
def test_block_qr_of_a_gaussian(oracle, m):
    a, x = _sample(m, ORTHOGONAL, 900 + m, "f16")
    assert np.array_equal(x, a.T)
    # rounding A to half: 2^-12 sqrt(2/3) per off-diagonal pair and twice that on the diagonal, 2.9e-4 in this norm, beside
    # the 3.1e-4 of zero-mean tf32 noise that the polishing step leaves
    d = a.T @ a - np.eye(m)
    assert np.linalg.norm(d) / np.sqrt(m) <= 6e-4
    assert abs(np.trace(d)) / m <= 1e-4
    # the factor itself: tf32 products err by 2^-11 sqrt(2/3) = 4e-4 per block.  Four blocks at a time act as one merged reflector,
    # in which the blocks right of a column cancel only as well as those products do, so a column of the first half
    # meets the errors of all m / 128 blocks, beside those of its own triangular factor and of Q; the last columns are conditioned like
    # the Gaussian itself, so they are only aligned
    G64 = oracle.gaussian(900 + m, 0, 0, m, m).astype(np.float32).astype(np.float64)
    q_ref, _ = oracle.householder_qr(G64)
    h = m // 2
    assert np.linalg.norm(a[:, :h] - q_ref[:, :h]) / np.sqrt(h) <= 4e-4 * (2 + m / 128)
    assert np.median(np.sum(a * q_ref, axis=0)) > 1 - 1e-4


# A sample alone forms Q^T while it factorises from 1536 rows on: the last size of the other route and the first of this one, an odd one, a
# last superblock of few columns
@pytest.mark.parametrize("m", [1535, 1536, 1547, 2131, 2560])
def test_factor_formed_beside_the_factorisation(oracle, m):
    a, x = _sample(m, ORTHOGONAL, 900 + m, "f16")
    assert np.array_equal(x, a.T)
    d = a.T @ a - np.eye(m)
    assert np.linalg.norm(d) / np.sqrt(m) <= 6e-4             # as in the test above
    q_ref, r = np.linalg.qr(oracle.gaussian(900 + m, 0, 0, m, m).astype(np.float32).astype(np.float64))
    q_ref *= np.sign(np.diag(r))
    h = m // 2
    assert np.linalg.norm(a[:, :h] - q_ref[:, :h]) / np.sqrt(h) <= 4e-4 * (2 + m / 128)
    # a wrong sign or a row of the last square that has not been turned shows in single columns
    along = np.sum(a * q_ref, axis=0)
    assert along[: m - 128].min() > 0.9 and np.median(along[-64:]) > 0.9
    # every column of the last square among them: the last ones are conditioned like the Gaussian, but for these seeds none is off by more than 0.01
    assert along[m - 128:].min() > 0.5
    # non-orthogonal: b = Q + G1 / (2 sqrt(m)), Q without the polish, which took the noise of the tf32 products out of a
    b, y = _sample(m, NONORTHOGONAL, 900 + m, "f16")
    assert np.linalg.norm(b @ y - np.eye(m)) / np.sqrt(m) <= 1.2e-3       # rounding of A^-1, 2.1e-4 relative, times |A| <= 1.5 and |A^-1| <= 3.3
    q = b - 0.5 / np.sqrt(m) * oracle.gaussian(900 + m, 1, 0, m, m)
    assert np.linalg.norm(q[:, :h] - q_ref[:, :h]) / np.sqrt(h) <= 2 * 4e-4 * (2 + m / 128)


# Two and three calls at once form their factors beside their factorisations too, on branches of their recordings that were captured through the same
# stream of the context: recorded, replayed, and against calls one by one
@pytest.mark.parametrize("calls,n,k", [(2, 1500, 47), (3, 1500, 47), (3, 1536, 0)])
def test_factors_formed_in_small_batches(calls, n, k):
    d, p, dt = 256, 768, "bf16"
    c = binding.Context(0)
    c.set_lanes(calls)
    c.ensure_batch_workspace(n, k, d, p, dt, calls)
    H = [inputs.make_hidden(n, d, dt, 30 + i, True, "cuda") for i in range(calls)]
    W = [inputs.make_weight(d, p, dt, 60 + i, "cuda") for i in range(calls)]
    kinds = [(ORTHOGONAL, NONORTHOGONAL)[i % 2] for i in range(calls)]
    out = torch.zeros((3, calls, n, p), dtype=TDT[dt], device="cuda")
    for run in range(2):
        c.qkv_offload_batch(H, W, n, k, d, p, kinds, [80 + i for i in range(calls)], 10.0, dt, list(out[run]))
    for i in range(calls):
        c.qkv_offload(H[i], W[i], n, k, d, p, kinds[i], 80 + i, 10.0, dt, out[2, i])
    assert c.last_status() == binding.OK
    assert torch.equal(out[0], out[1])
    for i in range(calls):
        ref = H[i].double() @ W[i].double()
        for run in (0, 2):
            assert ((out[run, i].double() - ref).norm() / ref.norm()).item() <= 2e-2        # the bf16 path's tolerance
        assert ((out[0, i].double() - out[2, i].double()).norm() / ref.norm()).item() <= 2e-2
    c.close()


# Factors are formed beside their factorisations only while the samples in flight do not fill the GPU (32000 rows in all), also where lanes do not share
# the SMs out (share 1): beyond, another number of launches per call
def test_factors_are_formed_for_few_samples_only():
    n, d, p, dt = 1536, 64, 64, "bf16"
    W = inputs.make_weight(d, p, dt, 1, "cuda")
    H = [inputs.make_hidden(n, d, dt, 1, True, "cuda")] * 24
    launches = {}
    for calls in (1, 4, 24):
        c = binding.Context(0)
        c.set_lanes(calls)
        c.set_lane_share(1)
        c.ensure_batch_workspace(n, 0, d, p, dt, calls)
        Y = torch.zeros((calls, n, p), dtype=TDT[dt], device="cuda")
        for run in range(2):
            c.launch_count(reset=True)
            c.qkv_offload_batch(H[:calls], [W] * calls, n, 0, d, p, [ORTHOGONAL] * calls, list(range(calls)), 10.0, dt, list(Y))
            launches[calls] = c.launch_count() / calls
        assert c.last_status() == binding.OK
        ref = H[0].double() @ W.double()
        assert all(((y.double() - ref).norm() / ref.norm()).item() <= 2e-2 for y in Y)       # the bf16 path's tolerance
        c.close()
    assert launches[4] == launches[1] and launches[24] != launches[1]


# 256: the first size of the iteration, a single pair of tile rows; 257 and 300: ragged tiles; gamma 0.55 is the last it takes,
# 0.6 goes to the LU
@pytest.mark.parametrize("m,gamma,dt", [(256, 0.5, "f16"), (257, 0.5, "bf16"), (300, 0.55, "f16"), (700, 0.5, "f16"), (300, 0.6, "f16")])
def test_inverse_of_the_nonorthogonal_sample(m, gamma, dt):
    c = binding.Context(0)
    c.ensure_workspace(m, 0, 8, 24, dt)
    c.set_nonorthogonal(gamma)
    ld = c.mixing_ld(m)
    A = padded(m, ld, TDT[dt]); X = padded(m, ld, TDT[dt]); cond = torch.zeros(1, device="cuda")
    c.sample_mixing(m, NONORTHOGONAL, 70 + m, dt, A, X, ld, cond)
    assert c.last_status() == binding.OK
    c.close()
    a, x = f64(A[:, :m]), f64(X[:, :m])
    ref = np.linalg.inv(a)
    assert abs(cond.item() / np.linalg.cond(a) - 1) <= 0.12          # a lower estimate, see the estimator's own test
    # what is left is one rounding of A^-1 to the storage type, half an ulp at most and 1/sqrt(3) of that in the mean over
    # a binade: 2^-9 / sqrt(3) * 1.5 = 1.7e-3 (bf16), 2.1e-4 (half); the LU adds up to 1.3e-3
    bound = {"bf16": 2.0e-3, "f16": 2.5e-4}[dt] + (1.3e-3 if gamma > 0.55 else 0.0)
    assert np.linalg.norm(x - ref) / np.linalg.norm(ref) <= bound


# bfloat16 at the last size with all corrections and the first two with one product less, against A^-1 in 64 bits.  Rounding alone is 1.66e-3 (2^-9 / sqrt(3)
# over a binade); the shorter iteration leaves gamma^10 = 9.8e-4 beside it, 1.93e-3 together, which is what the pivoted LU came to
# at 4096 rows (1.94e-3; 1.95e-3 at 4300, 2.17e-3 at 6000)
@pytest.mark.parametrize("m,bound", [(4095, 1.75e-3), (4096, 2.0e-3), (4300, 2.0e-3)])
def test_inverse_of_large_samples(m, bound):
    c = binding.Context(0)
    c.ensure_workspace(m, 0, 8, 24, "bf16")
    ld = c.mixing_ld(m)
    A = padded(m, ld, torch.bfloat16); X = padded(m, ld, torch.bfloat16)
    c.sample_mixing(m, NONORTHOGONAL, 70 + m, "bf16", A, X, ld)
    assert c.last_status() == binding.OK
    c.close()
    ref = torch.linalg.inv(A[:, :m].double())
    assert ((X[:, :m].double() - ref).norm() / ref.norm()).item() <= bound


# fp32 above the sizes of the iteration: the block QR, its polish and the LU of what follows, up to the last size of the route and one past it
@pytest.mark.parametrize("m", [769, 1075, 3072, 3073])
def test_large_fp32_samples(m):
    c = binding.Context(0)
    c.ensure_workspace(m, 0, 8, 24, "f32")
    ld = c.mixing_ld(m)
    A = padded(m, ld, torch.float32); X = padded(m, ld, torch.float32)
    eye = torch.eye(m, device="cuda", dtype=torch.float64)
    c.sample_mixing(m, ORTHOGONAL, 300 + m, "f32", A, X, ld)
    a = A[:, :m].double()
    assert torch.equal(X[:, :m], A[:, :m].T)
    # sums of m products: sqrt(m) 2^-24 = 3.3e-6 at 3072 rows (1.4e-6 measured with the panels)
    assert ((a.T @ a - eye).norm() / m ** 0.5).item() <= m ** 0.5 * 2.0 ** -24
    c.sample_mixing(m, NONORTHOGONAL, 300 + m, "f32", A, X, ld)
    # the eliminations of m columns amplify 2^-24 by a growth that goes with m: 2.3e-5 at 900 rows, 6.6e-5 at 2000
    assert ((X[:, :m].double() @ A[:, :m].double() - eye).norm() / m ** 0.5).item() <= m * 2.0 ** -24
    assert c.last_status() == binding.OK
    c.close()


# the fp32 route: 129: its first size, one block of 64; 250: an odd split; 700: two groups of blocks; 768: the last size of the iteration; half at
# 200 rows takes it too
@pytest.mark.parametrize("m,dt", [(129, "f32"), (250, "f32"), (700, "f32"), (768, "f32"), (200, "f16")])
def test_exact_block_route(oracle, m, dt):
    a, x = _sample(m, ORTHOGONAL, 300 + m, dt)
    assert np.array_equal(x, a.T)
    # fp32: sums of m products with eps = 2^-24 each leave sqrt(m) eps = 1.6e-6 at most in an entry of A^T A; half: its own rounding
    bound = 2.0e-6 if dt == "f32" else 4e-4
    assert np.linalg.norm(a.T @ a - np.eye(m)) / np.sqrt(m) <= bound
    G64 = oracle.gaussian(300 + m, 0, 0, m, m).astype(np.float32).astype(np.float64)
    q_ref, _ = oracle.householder_qr(G64)
    h = m // 2
    # 2e-6 per block from its factor (the Gram matrix squares a condition of at most 6), times at most m / 100 blocks
    assert np.linalg.norm(a[:, :h] - q_ref[:, :h]) / np.sqrt(h) <= (2e-6 * (2 + m / 100) if dt == "f32" else 4e-4)
    a, x = _sample(m, NONORTHOGONAL, 300 + m, dt)
    assert np.linalg.norm(x @ a - np.eye(m)) / np.sqrt(m) <= (3e-6 if dt == "f32" else 5e-4)


# The buffers of a call lie elsewhere where n and k split the same m differently, or where the rows are a group of a block-diagonal call.
# 330 rows: the size at which the first three differ; every call after the first finds recordings of the others in the context.
@pytest.mark.parametrize("kind", [ORTHOGONAL, NONORTHOGONAL])
@pytest.mark.parametrize("entry", ["call", "batch"])
def test_calls_of_equal_m_in_one_context(entry, kind):
    d, p, dt, calls = 256, 768, "bf16", 6 if entry == "batch" else 1
    c = binding.Context(0)
    c.set_lanes(6)
    c.ensure_blockdiag_workspace(660, 0, d, p, dt, 384, 6)
    c.ensure_batch_workspace(330, 60, d, p, dt, 6)
    out = torch.zeros((calls, 3, 660, p // 3), dtype=TDT[dt], device="cuda")
    for n, k, block in ((300, 30, 0), (330, 0, 0), (660, 0, 384), (300, 30, 0), (330, 0, 0), (270, 60, 0)):
        H = [inputs.make_hidden(n, d, dt, n + i, True, "cuda") for i in range(calls)]
        W = [inputs.make_weight(d, p, dt, n + i, "cuda") for i in range(calls)]
        o = [[out[i, j, :n] for i in range(calls)] for j in range(3)]
        seeds = [7 + i for i in range(calls)]
        if block:
            c.qkv_offload_blockdiag_batch(H, W, n, k, d, p, block, seeds, 10.0, dt, *o)
        elif entry == "batch":
            c.qkv_offload_batch(H, W, n, k, d, p, [kind] * calls, seeds, 10.0, dt, *o)
        else:
            c.qkv_offload(H[0], W[0], n, k, d, p, kind, seeds[0], 10.0, dt, o[0][0], o[1][0], o[2][0])
        torch.cuda.synchronize()
        assert c.last_status() == binding.OK
        for i in range(calls):
            ref = H[i].double() @ W[i].double()
            got = torch.cat([out[i, j, :n] for j in range(3)], dim=1).double()
            assert ((got - ref).norm() / ref.norm()).item() <= 2e-2, (n, k, block, i)        # the bf16 path's tolerance
        out.zero_()
    c.close()


# The block factor's copies between CTAs are waited for as long as the context says: with a limit of zero it gives up before it sends any, which
# the fp32 route (no tensor-core kernel in it) reports by itself.
def test_zero_wait_limit_reaches_the_block_factor():
    m, dt = 300, "f32"
    c = binding.Context(0)
    c.ensure_workspace(m, 0, 8, 24, dt)
    ld = c.mixing_ld(m)
    A = padded(m, ld, TDT[dt]); X = padded(m, ld, TDT[dt])
    c.set_wait_limit_ns(0)
    c.sample_mixing(m, ORTHOGONAL, 5, dt, A, X, ld)
    assert c.last_status() == binding.ERR_TIMEOUT
    c.set_wait_limit_ns(2_000_000_000)
    c.sample_mixing(m, ORTHOGONAL, 5, dt, A, X, ld)
    assert c.last_status() == binding.OK
    a = f64(A[:, :m])
    assert np.linalg.norm(a.T @ a - np.eye(m)) / np.sqrt(m) <= 2e-6
    c.close()


# A call by itself launches its sample the first time a size is met, records it the second time and replays it from then on: the same bytes
# each time.  The recordings are bounded: past the bound, more sizes take no more memory.
def test_sampling_graphs_are_bounded():
    d, dt = 64, "bf16"
    c = binding.Context(0)
    c.ensure_workspace(480, 0, d, d, dt)
    W = inputs.make_weight(d, d, dt, 3, "cuda")
    H = inputs.make_hidden(480, d, dt, 3, True, "cuda")
    Y = torch.zeros((3, 480, d), dtype=TDT[dt], device="cuda")
    free = {}
    for m in range(130, 480):
        for kind in (ORTHOGONAL, NONORTHOGONAL):
            for i in range(3 if m % 50 == 0 else 2):
                c.qkv_offload(H, W, m, 0, d, d, kind, m, 10.0, dt, Y[i])
            torch.cuda.synchronize()
            if m % 50 == 0:
                assert torch.equal(Y[0, :m], Y[1, :m]) and torch.equal(Y[0, :m], Y[2, :m])
        free[m] = torch.cuda.mem_get_info()[0]
    assert c.last_status() == binding.OK
    # 512 recordings, two for every size, are reached at 385 rows; one of them takes 0.36 MB and more, 57 MB for the 79 sizes from 400 on
    assert free[400] - free[479] <= 24 << 20
    c.close()


# fp32 batches: the samples of few lanes run in blocks, those of many in panels beside each other (768 rows: from sixteen orthogonal or
# non-orthogonal ones on, alternating kinds from more); either way H W comes out
@pytest.mark.parametrize("n,lanes,kinds,panels", [(768, 8, (0,), False), (768, 16, (0,), True), (768, 16, (1,), True), (768, 16, (0, 1), False),
                                                  (1000, 16, (0, 1), True), (129, 32, (0,), False)])
def test_fp32_batches_choose_the_route_by_what_is_in_flight(n, lanes, kinds, panels):
    d, p = 64, 64
    c = binding.Context(0)
    c.set_lanes(lanes)
    c.ensure_batch_workspace(n, 0, d, p, "f32", lanes)
    H = [inputs.make_hidden(n, d, "f32", 40 + i, True, "cuda") for i in range(lanes)]
    W = [inputs.make_weight(d, p, "f32", 90, "cuda")] * lanes
    Y = torch.zeros((lanes, n, p), device="cuda")
    call = lambda: c.qkv_offload_batch(H, W, n, 0, d, p, [kinds[i % len(kinds)] for i in range(lanes)], list(range(lanes)), 10.0, "f32", list(Y))
    c.profile_start()
    call()
    assert (c.profile_stop()["qr_panel"]["launches"] > 0) == panels
    Y.zero_()
    call()
    torch.cuda.synchronize()
    assert c.last_status() == binding.OK
    for i in range(lanes):
        ref = H[i].double() @ W[i].double()
        assert ((Y[i].double() - ref).norm() / ref.norm()).item() <= 1e-4           # the fp32 path's tolerance
    c.close()


# the one-launch samples hold their rows in steps of eight: both sides of a few steps, the first and the last size
@pytest.mark.parametrize("m", [7, 32, 33, 40, 41, 73, 80, 81, 104, 105, 121, 128])
def test_one_launch_samples(oracle, m):
    a, x = _sample(m, ORTHOGONAL, 60 + m, "f32")
    assert np.array_equal(x, a.T)
    assert np.linalg.norm(a.T @ a - np.eye(m)) / np.sqrt(m) <= 1e-6           # m reflections, 2^-24 each
    q_ref, _ = oracle.householder_qr(oracle.gaussian(60 + m, 0, 0, m, m).astype(np.float32).astype(np.float64))
    h = (m + 1) // 2
    assert np.linalg.norm(a[:, :h] - q_ref[:, :h]) / np.sqrt(h) <= 2e-5       # columns conditioned below 6 times what R loses


# The general route's verdict on matrices that are not finite (the one-launch route's is with the estimator's own tests): 657 rows are its first size in fp32
@pytest.mark.parametrize("m", [657, 1000])
@pytest.mark.parametrize("bad", [float("nan"), float("inf")])
def test_condition_estimate_of_large_broken_matrices(bad, m):
    c = binding.Context(0)
    c.ensure_workspace(m, 0, 8, 24, "f32")
    ld = c.mixing_ld(m)
    A = torch.zeros((m, ld), device="cuda"); A[:, :m] = torch.eye(m, device="cuda")
    B = A.clone(); B[100, 50] = bad
    est = torch.zeros(1, device="cuda")
    for pair in ((A, B), (B, A), (B, B)):
        c.cond_estimate(m, *pair, ld, est)
        assert not est.item() <= 1e30
    c.cond_estimate(m, A, A, ld, est)
    assert abs(est.item() - 1) <= 1e-4
    c.close()


# The estimate of kappa_2 in one launch: one row per CTA and less, ragged rows and columns, its last fp32 size and the first of the general route; in
# bfloat16 its last size and the next through a sample
@pytest.mark.parametrize("m,dt", [(2, "f32"), (9, "f32"), (135, "f32"), (656, "f32"), (657, "f32"), (920, "bf16"), (921, "bf16")])
def test_condition_estimate_on_both_routes(m, dt):
    c = binding.Context(0)
    c.ensure_workspace(m, 0, 8, 24, dt)
    ld = c.mixing_ld(m)
    A = padded(m, ld, TDT[dt]); X = padded(m, ld, TDT[dt])
    est = torch.zeros(1, device="cuda")
    if dt == "f32":
        g = torch.Generator().manual_seed(m)
        a = torch.eye(m, dtype=torch.float64) + 0.5 * torch.randn((m, m), generator=g, dtype=torch.float64) / m ** 0.5
        A[:, :m] = a.float(); X[:, :m] = torch.linalg.inv(A[:, :m].double()).float()
        A[:, m:] = float("inf"); X[:, m:] = float("nan")          # the padding is never read as data
        c.cond_estimate(m, A, X, ld, est)
    else:
        c.sample_mixing(m, NONORTHOGONAL, 3, dt, A, X, ld, est)
    assert c.last_status() == binding.OK
    s = torch.linalg.svdvals(A[:, :m].double())
    ref = (s[0] / s[-1]).item()
    assert 0.85 * ref <= est.item() <= 1.01 * ref                # a lower estimate; of A and of A^-1 as stored
    c.close()


# The eigenvalue search is carried to the last bit of the float it returns.  1 x 1 operators have the square of their entry, rounded once, as the only
# entry of their Lanczos matrix; these are pairs whose result lies so close to the middle of two floats that the bracket of the first seven rounds,
# 33^-7 wide and with its upper end on the eigenvalue, has its own middle on the other side
def test_condition_estimate_to_the_last_bit():
    rng = np.random.default_rng(7)
    a = rng.uniform(0.5, 2.0, 1 << 20).astype(np.float32)
    x = rng.uniform(0.5, 2.0, 1 << 20).astype(np.float32)
    lam = [(t * t).astype(np.float64) for t in (a, x)]
    est = (np.sqrt(lam[0]) * np.sqrt(lam[1])).astype(np.float32)
    short = (np.sqrt(lam[0] * (1 - 0.5 * 33.0 ** -7)) * np.sqrt(lam[1] * (1 - 0.5 * 33.0 ** -7))).astype(np.float32)
    pick = np.flatnonzero(est != short)[:16]
    assert len(pick) == 16
    c = binding.Context(0)
    c.ensure_workspace(1, 0, 8, 24, "f32")
    A = torch.zeros((1, 8), device="cuda"); X = torch.zeros((1, 8), device="cuda"); out = torch.zeros(16, device="cuda")
    for i, j in enumerate(pick):
        A[0, 0] = float(a[j]); X[0, 0] = float(x[j])
        c.cond_estimate(1, A, X, 8, out[i:])
    assert c.last_status() == binding.OK
    assert np.array_equal(out.cpu().numpy(), est[pick])
    c.close()


# The scalars of a reflector are as good as the rounded square root and divisions: Q of a 2 x 2 matrix is one reflector, whose few operations are repeated here in
# binary32.  An approximation that is off by a unit now and then shows in one of its four entries
def test_reflector_scalars_of_the_one_launch_sample():
    c = binding.Context(0)
    c.ensure_workspace(2, 0, 8, 24, "f32")
    A = torch.zeros((400, 2, 64), device="cuda"); X = torch.zeros((2, 64), device="cuda"); G = torch.zeros((400, 2, 2), device="cuda")
    for s in range(400):
        c.sample_gaussian(2, 2, 2, 4000 + s, 0, 0, 1.0, G[s])
        c.sample_mixing(2, ORTHOGONAL, 4000 + s, "f32", A[s], X, 64)
    assert c.last_status() == binding.OK
    f = lambda v: np.asarray(v, dtype=np.float32)
    g = G.cpu().numpy()
    a, b = g[:, 0, 0], g[:, 1, 0]
    fma = lambda x, y, z: f(x.astype(np.float64) * y + z)          # (48 bits of product and a term of like size: rounded once, but for rare ties)
    beta = -np.copysign(np.sqrt(fma(a, a, b * b)), a)
    tau, v = (beta - a) / beta, b * (f(1) / (a - beta))
    t = tau * v
    q = np.stack([np.stack([f(1) - tau, -t], 1), np.stack([-t, fma(-t, v, f(1))], 1)], 1)          # q[:, row, column]
    # columns signed by the diagonal of R
    x0, x1 = g[:, 0, 1], g[:, 1, 1]
    tw = tau * fma(f(1) / (a - beta), b * x1, x0)
    r = np.stack([beta, fma(-tw, v, x1)], 1)
    q *= np.where(r < 0, f(-1), f(1))[:, None, :]
    same = (A[:, :, :2].cpu().numpy() == q).all(axis=(1, 2))
    assert same.mean() >= 0.98
    c.close()

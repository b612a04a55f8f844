"""Performance cases of the obfuscated projection offload: the work that a user has the library do.

Every case goes through the public binding (`paper_2603_05035_b200.binding.Context`) as a serving program would: a context, its
workspace and the weights are set up once, then calls are made on the current stream.  Sizes are the workloads of
`paper_2603_05035_b200.inputs` (Llama-2-7B projections: d = 4096, p = 3 d = 12288) and generic ones around them.

`path` names the entry point:
  call       one whole call (sample A, shield rows, mix, project, unmix)
  batch      several independent calls at once, sampling on `lanes` streams (the layers of one forward pass)
  host       the same with activations and results in pinned host memory
  blockdiag  the structured variant with a block-diagonal A
  staged     the five stages called one by one, as a trusted side does that hands U to an accelerator and gets Y' back
  fp8        the accelerator's side with E4M3 operands: quantise the U that arrived, multiply by the resident codes of W
"""
import math
import os

import torch

# the lanes of the batched calls are streams: give each a hardware work queue (only has an effect before CUDA starts)
os.environ.setdefault("CUDA_DEVICE_MAX_CONNECTIONS", "32")

from paper_2603_05035_b200 import binding, inputs  # noqa: E402

KINDS = {"orthogonal": (binding.ORTHOGONAL,), "nonorthogonal": (binding.NONORTHOGONAL,),
         "alternating": (binding.ORTHOGONAL, binding.NONORTHOGONAL)}
SHIELD_SCALE = 10.0          # shield rows at ten times the median row norm, as every workload with shields has them
LARGEST_COST = 32 * (4300.0 ** 3 * 5.4 + 2.0 * 4300 * 4096 * 12288 * 2)      # bound on what draw() gives, see _cost()


def _case(name, path, n, k, d, p, dtype, kind="orthogonal", split=True, calls=1, lanes=1, block=0):
    return {"name": name, "path": path, "n": n, "k": k, "d": d, "p": p, "dtype": dtype, "kind": kind, "split": split,
            "calls": calls, "lanes": lanes, "block": block}


def listed():
    return [
        # the smallest call anybody makes: a correctness-sized fp32 layer, all latency and launches
        _case("tiny_fp32_call", "call", 64, 0, 256, 768, "f32"),
        # one new token for 64 sequences, one layer at a time: the latency of a decode step's projection
        _case("decode_call", "call", 64, 4, 4096, 12288, "bf16"),
        # the same for all 32 layers at once: seeds are known ahead, so the layers' calls go in as one batch
        _case("decode_step_32_layers", "batch", 64, 4, 4096, 12288, "bf16", calls=32, lanes=16),
        # a short prompt with an odd number of rows on a narrower model in IEEE half, the trusted side's steps one by one
        _case("short_prompt_f16_staged", "staged", 333, 17, 2048, 6144, "f16", kind="nonorthogonal"),
        # one full-width layer in fp32 with a non-orthogonal A
        _case("layer_fp32_call", "call", 512, 0, 4096, 12288, "f32", kind="nonorthogonal"),
        # a medium prompt, orthogonal A, five per cent shield rows
        _case("medium_prompt_call", "call", 2048, 102, 4096, 12288, "bf16"),
        # four prompts of 1024 tokens through one layer, waited for: the latency of a prefill call
        _case("prefill_call", "call", 4096, 204, 4096, 12288, "bf16", kind="nonorthogonal"),
        # the same through all 32 layers, kinds alternating: the throughput workload
        _case("prefill_sweep_32_layers", "batch", 4096, 204, 4096, 12288, "bf16", kind="alternating", calls=32, lanes=32),
        # the output projection (one square weight, unsplit result) of eight layers for a ragged number of rows
        _case("output_projection_8_layers", "batch", 1000, 50, 4096, 4096, "bf16", kind="alternating", split=False, calls=8, lanes=8),
        # eight layers whose activations live in host memory
        _case("host_prompt_8_layers", "host", 1024, 51, 4096, 12288, "bf16", calls=8, lanes=8),
        # prefill with the structured A, four layers
        _case("blockdiag_prefill_4_layers", "blockdiag", 4096, 204, 4096, 12288, "bf16", calls=4, lanes=32, block=512),
        # the accelerator's product on E4M3 operands for a medium prompt
        _case("fp8_projection", "fp8", 2048, 102, 4096, 12288, "bf16"),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _cost(c):
    m = c["n"] + c["k"]
    sampling = 0.0 if c["path"] == "fp8" else (5.4 * m * m * min(m, c["block"] or m))
    return c["calls"] * (sampling + 4.0 * m * c["d"] * c["p"])


def draw(rng):
    """One more case of the same ranges: rows from 7 to 4096 (decode and prefill), widths from 256 to 4096."""
    while True:
        path = rng.choice(["call", "call", "call", "batch", "batch", "host", "staged", "blockdiag", "fp8"])
        dtype = rng.choice(["bf16", "bf16", "bf16", "f16", "f32"])
        kind = rng.choice(["orthogonal", "orthogonal", "nonorthogonal"])
        n = _log_int(rng, 7, 4096)
        d = 16 * _log_int(rng, 16, 256)
        split = rng.random() < 0.7
        p = 3 * d if split else (d if rng.random() < 0.5 else 16 * _log_int(rng, 16, 688))
        k = 0 if rng.random() < 0.2 else max(1, round(0.05 * n))
        calls, lanes, block = 1, 1, 0
        if dtype == "f32":
            n, k = min(n, 1024), min(k, 51)
        if path in ("batch", "host"):
            calls = rng.choice([2, 3, 5, 8, 16, 32])
            lanes = rng.choice([4, 8, 16, 32])
            if path == "host":                                   # pinned memory is slow to set up: keep it below a gigabyte
                n, k, calls = min(n, 1024), min(k, 51), min(calls, 8)
            if kind == "nonorthogonal":
                kind = "alternating"
        if path == "blockdiag":
            if n < 300 or dtype == "f32":
                continue
            kind, calls, lanes, block = "orthogonal", rng.choice([1, 2, 4, 8]), 32, rng.choice([256, 512, 1024])
        if path == "fp8":
            dtype, split, kind = "bf16", False, "orthogonal"
        if path == "staged" and n > 512:
            continue
        c = _case("", path, n, k, d, p, dtype, kind, split, calls, lanes, block)
        del c["name"]
        if _cost(c) <= LARGEST_COST:
            return c


def _outputs(case, device):
    """One buffer for all results of a case: [calls, 3, n, p / 3] or [calls, 1, n, p], and the pieces a call writes."""
    parts = 3 if case["split"] else 1
    td = inputs.torch_dtype(case["dtype"])
    out = torch.zeros((case["calls"], parts, case["n"], case["p"] // parts), dtype=td, device=device)
    if case["path"] == "host":
        out = out.pin_memory()
    return out, [[out[i, j] for i in range(case["calls"])] if j < parts else None for j in range(3)]


def prepare(case, seed):
    n, k, d, p, dtype = case["n"], case["k"], case["d"], case["p"], case["dtype"]
    calls = case["calls"]
    ctx = binding.Context(torch.cuda.current_device())
    s = {"case": case, "ctx": ctx}
    s["seeds"] = [(seed * 1000003 + 17 * i + 1) & (2 ** 63 - 1) for i in range(calls)]
    s["W"] = [inputs.make_weight(d, p, dtype, (seed << 8) + i, "cuda") for i in range(calls)]
    s["H"] = [inputs.make_hidden(n, d, dtype, (seed << 8) + i, True, "cuda") for i in range(calls)]
    kinds = KINDS[case["kind"]]
    s["kinds"] = [kinds[i % len(kinds)] for i in range(calls)]
    td = inputs.torch_dtype(dtype)
    m = n + k
    if case["path"] == "fp8":
        # what the accelerator holds: the codes of W; what arrives: U = A [H; S], a rotation of unit-variance rows and of shield
        # rows at SHIELD_SCALE times their norm, so every entry is close to Gaussian with the mean energy of both
        W = s.pop("W")[0]
        s["W8"] = torch.empty((d, p), dtype=torch.uint8, device="cuda")
        s["w_scale"] = torch.empty(2, dtype=torch.float32, device="cuda")
        ctx.quantize_e4m3(W, d, p, dtype, s["W8"], s["w_scale"])
        g = torch.Generator(device="cuda")
        g.manual_seed(seed)
        std = math.sqrt((n + SHIELD_SCALE ** 2 * k) / m)
        s["U"] = (torch.randn((m, d), generator=g, device="cuda") * std).to(td)
        del s["H"]
        s["U8"] = torch.empty((m, d), dtype=torch.uint8, device="cuda")
        s["u_scale"] = torch.empty(2, dtype=torch.float32, device="cuda")
        s["Y"] = torch.empty((m, p), dtype=torch.bfloat16, device="cuda")
        return s
    ctx.set_lanes(case["lanes"])
    s["out"], s["QKV"] = _outputs(case, "cpu" if case["path"] == "host" else "cuda")
    if case["path"] == "host":
        s["H"] = [h.cpu().pin_memory() for h in s["H"]]
    if case["path"] == "blockdiag":
        ctx.ensure_blockdiag_workspace(n, k, d, p, dtype, case["block"], case["lanes"])
    elif case["path"] in ("batch", "host"):
        ctx.ensure_batch_workspace(n, k, d, p, dtype, case["lanes"])
    else:
        ctx.ensure_workspace(n, k, d, p, dtype)
    if case["path"] == "staged":
        ld = ctx.mixing_ld(m)
        s["A"] = torch.zeros((m, ld), dtype=td, device="cuda")
        s["Ainv"] = torch.zeros((m, ld), dtype=td, device="cuda")
        s["S"] = torch.empty((k, d), dtype=td, device="cuda") if k else None
        s["U"] = torch.empty((m, d), dtype=td, device="cuda")
        s["Yp"] = torch.empty((m, p), dtype=td, device="cuda")
    return s


def run(state):
    c, ctx = state["case"], state["ctx"]
    n, k, d, p, dtype = c["n"], c["k"], c["d"], c["p"], c["dtype"]
    m = n + k
    if c["path"] == "fp8":
        ctx.quantize_e4m3(state["U"], m, d, dtype, state["U8"], state["u_scale"])
        ctx.project_e4m3(state["U8"], state["u_scale"], state["W8"], state["w_scale"], m, d, p, state["Y"])
        return state["Y"], state["U8"]
    H, W, (Q, K, V) = state["H"], state["W"], state["QKV"]
    if c["path"] == "staged":
        A, Ainv, S, U, Yp = state["A"], state["Ainv"], state["S"], state["U"], state["Yp"]
        ld = ctx.mixing_ld(m)
        ctx.sample_mixing(m, state["kinds"][0], state["seeds"][0], dtype, A, Ainv, ld)
        if k:
            ctx.shield_rows(H[0], n, d, k, SHIELD_SCALE, state["seeds"][0], dtype, S)
        ctx.mix(A, ld, H[0], S, n, k, d, dtype, U)
        ctx.project(U, W[0], m, d, p, dtype, Yp)
        ctx.unmix(Ainv, ld, Yp, n, k, p, dtype, Q[0], K and K[0], V and V[0])
        return state["out"], U
    if c["path"] == "call":
        ctx.qkv_offload(H[0], W[0], n, k, d, p, state["kinds"][0], state["seeds"][0], SHIELD_SCALE, dtype,
                        Q[0], K and K[0], V and V[0])
    elif c["path"] == "blockdiag":
        ctx.qkv_offload_blockdiag_batch(H, W, n, k, d, p, c["block"], state["seeds"], SHIELD_SCALE, dtype, Q, K, V)
    else:
        call = ctx.qkv_offload_batch_host if c["path"] == "host" else ctx.qkv_offload_batch
        call(H, W, n, k, d, p, state["kinds"], state["seeds"], SHIELD_SCALE, dtype, Q, K, V)
    return state["out"]


def work(case):
    """Inputs read once, results written once; the arithmetic of the method with A dense (or in blocks)."""
    n, k, d, p, calls = case["n"], case["k"], case["d"], case["p"], case["calls"]
    m = n + k
    if case["path"] == "fp8":
        return {"bytes": 3 * m * d + d * p + 2 * m * p, "flops": 2.0 * m * d * p}
    es = 4 if case["dtype"] == "f32" else 2
    b = min(m, case["block"] or m)
    qr = 8.0 / 3.0 * m * b * b                                   # Householder QR and its Q
    lu = 2.0 * m * m * m                                         # elimination and inverse
    share = {"orthogonal": 0.0, "nonorthogonal": 1.0, "alternating": (calls // 2) / calls}[case["kind"]]
    flops = qr + share * lu + 2.0 * m * b * d + 2.0 * m * d * p + 2.0 * n * b * p
    return {"bytes": calls * es * (n * d + d * p + n * p), "flops": calls * flops}


def tolerance(case):
    if case["path"] == "fp8":
        return {"rel": 4e-3, "max": 0.05}          # same codes (exact), the product rounded once to bf16
    if case["path"] == "staged":
        # U = A [H; S] is an output here, and the last columns of A, which carry the shields' energy, are conditioned like the
        # Gaussian they come from: with tf32 products 1.2e-2 .. 1.4e-2 against U from a 64-bit QR of the same Gaussian
        return {"rel": 2e-4 if case["dtype"] == "f32" else 3e-2}
    # against H W in 64 bits: bf16 8e-3 .. 9e-3, half 1e-3 .. 4e-3, fp32 5e-7 .. 7e-5 (rounding of A, U, Y', carried by shield
    # rows at ten times the norm); another A of the same quality differs by as much again
    return {"rel": {"bf16": 2e-2, "f16": 8e-3, "f32": 2e-4}[case["dtype"]]}

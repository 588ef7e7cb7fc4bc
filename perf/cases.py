"""The work that a user of this package has it do, as timed cases.

A case is one pass through the public calls of ``paper_2602_06183_b200.binding``: a training step of the FFN
layer (forward and backward, as a sparse, dense or routed step), or one of the stand-alone passes (2:4 pruning,
SquaredReLU + V:N:M sparsification, the E4M3 product). Buffers that a training loop allocates once (context,
workspace, outputs) are made in ``prepare``; everything that a step does with new values is in ``run``.
Sizes are those of the package's own configurations and tests, or lie between them.
"""
from __future__ import annotations

import math

import torch

from paper_2602_06183_b200 import binding

BF16 = torch.bfloat16
# largest cost of a drawn step, in units of tokens x d_model x d_ffn: a quarter of the largest listed case
MAX_STEP = 16384 * 8192 * 28672 // 4


def listed():
    return [
        # The parity-size layer: a handful of tiles per product, so launches and latency are all of it.
        {"name": "step_small", "kind": "sparse", "T": 1024, "D": 256, "F": 1024, "V": 64, "M": 8, "mode": 0, "flags": 0},
        # The smaller model of the paper's table (d_model 2048) with its weight sparsifier, soft-thresholding, and
        # 128-token blocks, on a micro-batch of 4096 tokens.
        {"name": "step_d2048_soft_v128", "kind": "sparse", "T": 4096, "D": 2048, "F": 8192, "V": 128, "M": 8, "mode": 1, "flags": 0},
        # The d_model 4096 layer: the benchmark's workload.
        {"name": "step_d4096", "kind": "sparse", "T": 8192, "D": 4096, "F": 16384, "V": 64, "M": 8, "mode": 0, "flags": 0},
        # The largest configuration (d_model 8192).
        {"name": "step_d8192", "kind": "sparse", "T": 16384, "D": 8192, "F": 28672, "V": 64, "M": 8, "mode": 0, "flags": 0},
        # Sizes that are no powers of two (odd multiples of 128: half-empty last tiles in every product), groups of
        # four (plain 2:4 activations), W2 held as [d_ffn, d_model].
        {"name": "step_ragged_m4", "kind": "sparse", "T": 1920, "D": 1408, "F": 5504, "V": 64, "M": 4, "mode": 0, "flags": 16},
        # 87.5 % sparse activations: the condensed products that gather the kept weight rows.
        {"name": "step_d4096_m16", "kind": "sparse", "T": 8192, "D": 4096, "F": 16384, "V": 128, "M": 16, "mode": 0, "flags": 0},
        # The dense steps before and after the sparse phase of a run's schedule.
        {"name": "dense_step_d2048", "kind": "dense", "T": 4096, "D": 2048, "F": 8192, "V": 64, "M": 8, "mode": 0, "flags": 0},
        # The routed step (neuron-level experts) on the d_model 4096 layer.
        {"name": "routed_d4096_e4", "kind": "routed", "T": 8192, "D": 4096, "F": 16384, "E": 4, "mode": 0},
        # Stand-alone pruning of a weight matrix after an optimiser step: the smallest of the sweep, and a larger
        # one whose groups run down the columns, with the soft threshold.
        {"name": "prune_4096", "kind": "prune", "rows": 4096, "cols": 4096, "dim": 1, "mode": 0},
        {"name": "prune_strided_soft", "kind": "prune", "rows": 4096, "cols": 16384, "dim": 0, "mode": 1},
        # Stand-alone activation sparsification at the size of the activation sweep.
        {"name": "act_16384", "kind": "act", "T": 16384, "F": 16384, "V": 64, "M": 8},
        # A linear layer on E4M3 operands: weights pruned and quantised in one pass, tokens quantised, 2:4 product
        # (the shape of the paper's product micro-benchmark).
        {"name": "fp8_4096_16384", "kind": "fp8", "Mr": 4096, "Nc": 16384, "K": 4096},
    ]


def _size(rng, lo, hi, multiple):
    """A multiple of `multiple` between lo and hi, even over the logarithm."""
    v = math.exp(rng.uniform(math.log(lo), math.log(hi)))
    return max(-(-lo // multiple), min(hi // multiple, round(v / multiple))) * multiple


def draw(rng):
    kind = rng.choice(["sparse", "sparse", "sparse", "sparse", "dense", "routed", "routed", "prune", "prune", "act", "fp8"])
    if kind in ("sparse", "dense"):
        M = rng.choice([4, 8, 8, 8, 16, 32]) if kind == "sparse" else 8
        q, qf = (128, 128) if M < 16 else (256, 32 * M if M > 8 else 128)
        while True:
            c = {"kind": kind, "T": _size(rng, 256, 16384, q), "D": _size(rng, 256, 8192, q),
                 "F": _size(rng, 1024, 28672, qf), "V": rng.choice([64, 64, 128]), "M": M, "mode": rng.choice([0, 0, 1]),
                 "flags": rng.choice([0, 0, 0, 16])}
            if c["T"] * c["D"] * c["F"] <= MAX_STEP:
                return c
    if kind == "routed":
        E = rng.choice([2, 4, 8, 16])
        while True:
            c = {"kind": kind, "T": _size(rng, 512, 16384, 256), "D": _size(rng, 256, 8192, 256),
                 "F": _size(rng, 4096, 28672, 256 * E), "E": E, "mode": rng.choice([0, 0, 1])}
            if c["T"] * c["D"] * c["F"] <= MAX_STEP:
                return c
    if kind == "prune":
        dim = rng.choice([0, 1])
        rows = _size(rng, 512, 28672, 16) if dim == 0 else int(_size(rng, 512, 28672, 1))
        return {"kind": kind, "rows": rows, "cols": _size(rng, 1024, 16384, 8 if dim == 0 else 16), "dim": dim,
                "mode": rng.choice([0, 1])}
    if kind == "act":
        M, V = rng.choice([8, 8, 16, 32]), rng.choice([64, 64, 128])
        return {"kind": kind, "T": _size(rng, 1024, 16384, V), "F": _size(rng, 1024, 16384, 128), "V": V, "M": M}
    return {"kind": "fp8", "Mr": _size(rng, 512, 16384, 256), "Nc": _size(rng, 512, 16384, 256), "K": _size(rng, 512, 8192, 256)}


def _normal(shape, std, gen):
    t = torch.randn(shape, generator=gen, device="cuda", dtype=torch.float32)
    return t.mul_(std).to(BF16)


def prepare(case, seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))
    kind = case["kind"]
    if kind in ("sparse", "dense", "routed"):
        T, D, F = case["T"], case["D"], case["F"]
        s = {"kind": kind, "X": _normal((T, D), 1.0, g), "dY": _normal((T, D), 1.0, g)}
        s["W1"] = _normal((F, D), 0.02, g)
        s["W2"] = _normal((F, D) if case.get("flags", 0) & binding.SF_FFN_W2_FD else (D, F), 0.02, g)
        if kind == "routed":
            s["desc"] = binding.make_router_desc(T, D, F, case["E"], prune_mode=case["mode"])
            s["means"] = _normal((case["E"], D), 1.0, g)
            ctx, ws = binding.sf_routed_ffn_workspace_size(s["desc"])
            s["ctx"] = torch.zeros((ctx,), dtype=torch.uint8, device="cuda")
            s["ws"] = torch.zeros((ws,), dtype=torch.uint8, device="cuda")
        else:
            s["desc"] = binding.make_desc(T, D, F, case["V"], case["M"], prune_mode=case["mode"], flags=case["flags"])
            s["ctx"], s["ws"] = binding.alloc_ffn_buffers(s["desc"])
        s["Y"], s["dX"] = torch.empty_like(s["X"]), torch.empty_like(s["X"])
        s["dW1"], s["dW2"] = torch.empty_like(s["W1"]), torch.empty_like(s["W2"])
        return s
    if kind == "prune":
        W = _normal((case["rows"], case["cols"]), 0.02, g)
        # exact ties of magnitude in some groups, as in the package's own pruning sweep
        tie = torch.rand((case["rows"] // 4, case["cols"] // 4), generator=g, device="cuda") < 0.05
        r, c = tie.nonzero(as_tuple=True)
        if case["dim"] == 1:
            W[4 * r, 4 * c + 2] = -W[4 * r, 4 * c]
        else:
            W[4 * r + 2, 4 * c] = -W[4 * r, 4 * c]
        s = {"kind": kind, "W": W, "dim": case["dim"], "mode": case["mode"]}
        s["out"] = binding.sf_prune24_compress(W, s["dim"], s["mode"])
        return s
    if kind == "act":
        # about 90 % of the pre-activations are negative, as in a trained model
        P = _normal((case["T"], case["F"]), 1.0, g).sub_(1.3)
        s = {"kind": kind, "P": P, "V": case["V"], "M": case["M"]}
        s["out"] = binding.sf_vnm_sparsify_act(P, s["V"], s["M"])
        return s
    Mr, Nc, K = case["Mr"], case["Nc"], case["K"]
    s = {"kind": kind, "W": _normal((Mr, K), 0.02, g), "X": _normal((Nc, K), 1.0, g), "sw": 2048.0, "sx": 64.0}
    s["packed"] = binding.sf_prune24_compress_fp8(s["W"], 0, s["sw"])
    s["Xq"] = torch.empty((Nc, K), dtype=torch.uint8, device="cuda")
    s["C"] = torch.empty((Mr, Nc), dtype=BF16, device="cuda")
    s["ws"] = torch.zeros((binding.sf_gemm_fp8_workspace_size(Mr, K),), dtype=torch.uint8, device="cuda")
    return s


def run(s):
    kind = s["kind"]
    if kind == "sparse":
        binding.sf_sparse_ffn_fwd(s["desc"], s["X"], s["W1"], s["W2"], s["Y"], s["ctx"], s["ws"])
        binding.sf_sparse_ffn_bwd(s["desc"], s["dY"], s["X"], s["W1"], s["W2"], s["ctx"], s["dX"], s["dW1"], s["dW2"], s["ws"])
        return {k: s[k] for k in ("Y", "dX", "dW1", "dW2")}
    if kind == "dense":
        binding.sf_dense_ffn_fwd(s["desc"], s["X"], s["W1"], s["W2"], s["Y"], s["ctx"], s["ws"])
        binding.sf_dense_ffn_bwd(s["desc"], s["dY"], s["X"], s["W1"], s["W2"], s["ctx"], s["dX"], s["dW1"], s["dW2"], s["ws"])
        return {k: s[k] for k in ("Y", "dX", "dW1", "dW2")}
    if kind == "routed":
        binding.sf_routed_ffn_fwd(s["desc"], s["X"], s["W1"], s["W2"], s["means"], s["Y"], s["ctx"], s["ws"])
        binding.sf_routed_ffn_bwd(s["desc"], s["dY"], s["X"], s["W1"], s["W2"], s["ctx"], s["dX"], s["dW1"], s["dW2"], s["ws"])
        return {k: s[k] for k in ("Y", "dX", "dW1", "dW2")}
    if kind == "prune":
        vals, meta, _ = binding.sf_prune24_compress(s["W"], s["dim"], s["mode"], out=s["out"])
        return {"vals": vals, "meta": meta}
    if kind == "act":
        vals, meta, colidx, relu, _ = binding.sf_vnm_sparsify_act(s["P"], s["V"], s["M"], out=s["out"])
        return {"vals": vals, "meta": meta, "colidx": colidx, "relu": relu}
    vals, meta, _ = binding.sf_prune24_compress_fp8(s["W"], 0, s["sw"], out=s["packed"])
    binding.sf_fp8_quantize(s["X"], s["sx"], out=s["Xq"])
    binding.sf_gemm_fp8_sparse24(vals, meta, s["Xq"], 1.0 / (s["sw"] * s["sx"]), C_out=s["C"], workspace=s["ws"])
    return {"vals": vals, "meta": meta, "Xq": s["Xq"], "C": s["C"]}


def work(case):
    """Inputs read once and outputs written once; multiply-adds on the stored operands (a 2:4 operand has half of
    the dense product's, V:N:M activations 2 / M of it; the weight gradients reduce over tokens, along which
    neither format is structured, and count as dense)."""
    kind = case["kind"]
    if kind in ("sparse", "dense", "routed"):
        T, D, F = case["T"], case["D"], case["F"]
        product = 2.0 * T * D * F
        if kind == "sparse":
            units = 2 * 0.5 + 2 * 2.0 / case["M"] + 2
        elif kind == "dense":
            units = 6.0
        else:
            units = (4 * 0.5 + 2) / case["E"]
        # X, dY, W1, W2 in; Y, dX, dW1, dW2 out
        return {"bytes": 2.0 * (4 * T * D + 4 * D * F), "flops": units * product}
    if kind == "prune":
        return {"bytes": 3.125 * case["rows"] * case["cols"], "flops": 0.0}
    if kind == "act":
        T, F, M = case["T"], case["F"], case["M"]
        return {"bytes": T * F * (2 + 8.5 / M) + (T // case["V"]) * (F // M) * 4.0, "flops": 0.0}
    Mr, Nc, K = case["Mr"], case["Nc"], case["K"]
    # W and X read; codes, metadata and the product written
    return {"bytes": 2.625 * Mr * K + 3.0 * Nc * K + 2.0 * Mr * Nc, "flops": 1.0 * Mr * Nc * K}


def tolerance(case):
    """About four times what these calls differ by from themselves when the reductions run in another order (tokens,
    d_model and d_ffn permuted in blocks, results permuted back; 2-norm of the difference over that of the result):
      sparse   2.8e-3 (3e-5 at the smallest size): a pre-activation that rounds the other way can change which of two
               equal magnitudes is kept, so single elements move by up to the result's root mean square (0.91 of it)
      routed   6e-4, single elements 0.12; a token whose two best logits nearly tie would change expert
      dense    5e-4, single elements one bf16 step (8.6e-3)
      fp8      7.5e-6, single elements one bf16 step: products of codes are exact in float32 and nearly so are their sums
    Selections of the stand-alone passes are exact: they depend on stored bytes and one stated order of additions."""
    kind = case["kind"]
    if kind in ("prune", "act"):
        return "exact"
    if kind == "sparse":
        return {"rel": 1e-2, "max": 0.99}
    if kind == "routed":
        return {"rel": 2.5e-3, "max": 0.5}
    if kind == "dense":
        return {"rel": 2e-3, "max": 0.035}
    return {"rel": 3e-5, "max": 0.035}

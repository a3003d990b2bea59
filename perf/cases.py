"""What is measured: the calls that programs make of this library, over the sizes they make them at.

Six kinds of pass, all through the package's public entry points, written as the README writes them:

``quantize``   ``abs_quantize`` of a bf16 matrix: the training recipe's options included, no decode
``roundtrip``  ``abs_quantize`` followed by ``abs_dequantize`` (storage: weights, activations, format sweeps)
``serve``      a linear layer at inference: the weights were quantized when the model was loaded, each pass
               quantizes the activations and multiplies (bf16 output; optionally with the tensor scale that the next
               layer's quantizer needs)
``forward``    ``linear.forward_tc``: the training forward pass, both operands quantized in the pass
``backward``   ``linear.backward_tc``: both gradient products of the layer with Hadamard, stochastic rounding and 17/16
``emulated``   ``linear.forward`` and ``linear.backward``: the paper's experiments, one-pass emulation and bf16 GEMMs
"""
import math

import torch

from paper_2603_28765_b200 import binding as B
from paper_2603_28765_b200 import linear

SIGN_MASK = 0x5A3C


def listed():
    return [
        # one token of a decoder step through a square projection: latency and launches are all there is
        {"name": "serve_if4_1_token", "kind": "serve", "fmt": "if4", "tokens": 1, "d_in": 4096, "d_out": 4096, "chained": False},
        # a decoder step of a small batch through the wide projection of a feed-forward block, chained to the next layer
        {"name": "serve_if4_24_tokens", "kind": "serve", "fmt": "if4", "tokens": 24, "d_in": 4096, "d_out": 14336, "chained": True},
        # prompt processing with an odd number of tokens, plain NVFP4
        {"name": "serve_nvfp4_1000_tokens", "kind": "serve", "fmt": "nvfp4", "tokens": 1000, "d_in": 4096, "d_out": 14336, "chained": True},
        # the training layer of the report and the README, forward and backward
        {"name": "forward_if4_8192", "kind": "forward", "fmt": "if4", "tokens": 8192, "d_in": 4096, "d_out": 14336},
        {"name": "backward_if4_8192", "kind": "backward", "fmt": "if4", "tokens": 8192, "d_in": 4096, "d_out": 14336},
        # a smaller training layer in the format without integer groups
        {"name": "backward_nvfp4_2048", "kind": "backward", "fmt": "nvfp4", "tokens": 2048, "d_in": 4096, "d_out": 4096},
        # the paper's experiments as they were run, on a square layer
        {"name": "emulated_if4_4096", "kind": "emulated", "fmt": "if4", "tokens": 4096, "d_in": 4096, "d_out": 4096},
        # the benchmark's tensor: activations with outlier columns
        {"name": "roundtrip_if4_8192x4096", "kind": "roundtrip", "fmt": "if4", "rows": 8192, "cols": 4096, "data": "activation", "option": "none"},
        # an odd, small activation matrix in a block-size-8 format
        {"name": "roundtrip_if4_bs8_333x2064", "kind": "roundtrip", "fmt": "if4_bs8", "rows": 333, "cols": 2064, "data": "activation", "option": "none"},
        # the two other element widths: a weight matrix, and the format sweep's large tensor
        {"name": "roundtrip_if3_4096x14336", "kind": "roundtrip", "fmt": "if3", "rows": 4096, "cols": 14336, "data": "weight", "option": "none"},
        {"name": "roundtrip_if6_16384x8192", "kind": "roundtrip", "fmt": "if6_e2m3", "rows": 16384, "cols": 8192, "data": "mixture", "option": "none"},
        # the gradient tensor of the training recipe: Hadamard, stochastic rounding and the 17/16 factor
        {"name": "gradient_if4_16384x8192", "kind": "quantize", "fmt": "if4", "rows": 16384, "cols": 8192, "data": "gradient", "option": "hadamard_stochastic"},
    ]


# ----------------------------------------------------------------------------- more of the same ranges


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def _multiple(rng, lo, hi, of):
    return max(of, int(round(_log(rng, lo, hi) / of)) * of)


def draw(rng):
    kind = rng.choice(["serve", "serve", "forward", "backward", "emulated", "roundtrip", "roundtrip", "roundtrip", "quantize", "quantize"])
    if kind in ("roundtrip", "quantize"):
        case = {"kind": kind}
        cols = _multiple(rng, 208, 14336, 16)
        rows = max(1, int(_log(rng, 1, min(16384, 16384 * 8192 // cols))))
        if kind == "roundtrip":
            case["fmt"] = rng.choice(["if4", "if4", "nvfp4", "if3", "if6_e2m3", "if6_e3m2", "if4_bs8", "nvfp4_bs8", "if3_bs8"])
            case["option"] = rng.choice(["none", "none", "tiled_scales"]) if case["fmt"] in ("if4", "nvfp4") else "none"
        else:
            case["fmt"] = rng.choice(["if4", "if4", "nvfp4"])
            case["option"] = rng.choice(["hadamard", "stochastic", "hadamard_stochastic", "columns", "columns_hadamard_stochastic"])
            if case["option"].startswith("columns"):
                rows = (rows + 15) // 16 * 16
        case.update(rows=rows, cols=cols, data=rng.choice(["activation", "weight", "gradient", "mixture"]))
        return case
    fmt = rng.choice(["if4", "if4", "nvfp4"])
    if kind == "serve":
        return {"kind": kind, "fmt": fmt, "tokens": int(_log(rng, 1, 2048)), "d_in": _multiple(rng, 1024, 14336, 256),
                "d_out": _multiple(rng, 1024, 14336, 128), "chained": rng.random() < 0.5}
    return {"kind": kind, "fmt": fmt, "tokens": _multiple(rng, 512, 8192, 256), "d_in": _multiple(rng, 1024, 4096, 256),
            "d_out": _multiple(rng, 1024, 14336, 256)}


# ----------------------------------------------------------------------------- inputs


def _data(kind, rows, cols, gen):
    """bf16 matrix with the values of the configuration of that name (``inputs.py``), drawn on the device."""
    def normal(*shape):
        return torch.randn(shape, generator=gen, device="cuda")

    if kind == "activation":            # 0.5 * Student-t(3), 0.5 % of the columns times 50
        x = normal(rows, cols)
        x *= 0.5 * (sum(normal(rows, cols).square_() for _ in range(3)) / 3.0).rsqrt_()
        columns = torch.randperm(cols, generator=gen, device="cuda")[: max(1, cols // 200)]
        x[:, columns] *= 50.0
    elif kind == "weight":
        x = normal(rows, cols) * 0.02
    elif kind == "gradient":            # magnitudes that span four decades over the rows
        x = normal(rows, cols) * 1e-3 * (10.0 ** (4.0 * torch.rand((rows, 1), generator=gen, device="cuda") - 2.0))
    else:                               # 0.7 N(0,1) + 0.3 Laplace(0,1), 0.1 % of the entries times 100
        u = torch.rand((rows, cols), generator=gen, device="cuda") - 0.5
        laplace = -u.sign() * torch.log1p(-2.0 * u.abs().clamp_max(0.4999999))
        x = torch.where(torch.rand((rows, cols), generator=gen, device="cuda") < 0.7, normal(rows, cols), laplace)
        x = torch.where(torch.rand((rows, cols), generator=gen, device="cuda") < 0.001, 100.0 * x, x)
    return x.bfloat16()


_OPTIONS = {
    "none": 0,
    "tiled_scales": B.ABS_F_SCALES_SWIZZLED,
    "hadamard": B.ABS_F_HADAMARD16,
    "stochastic": B.ABS_F_STOCHASTIC | B.ABS_F_SR_SCALE_17_16,
    "hadamard_stochastic": B.ABS_F_HADAMARD16 | B.ABS_F_STOCHASTIC | B.ABS_F_SR_SCALE_17_16,
    "columns": 0,
    "columns_hadamard_stochastic": B.ABS_F_HADAMARD16 | B.ABS_F_STOCHASTIC | B.ABS_F_SR_SCALE_17_16,
}


def prepare(case, seed):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    state = {"case": case, "fmt": B.FMT_NAMES[case["fmt"]], "seed": seed}
    kind = case["kind"]
    if kind in ("roundtrip", "quantize"):
        flags = _OPTIONS[case["option"]]
        state["opts"] = B.make_opts(flags, SIGN_MASK, seed) if flags else None
        state["x"] = _data(case["data"], case["rows"], case["cols"], gen)
        return state
    state["x"] = _data("activation", case["tokens"], case["d_in"], gen)
    w = _data("weight", case["d_out"], case["d_in"], gen)
    if kind == "serve":
        state["qw"] = B.abs_quantize(state["fmt"], w)
    else:
        state["w"] = w
    if kind in ("backward", "emulated"):
        state["dy"] = _data("gradient", case["tokens"], case["d_out"], gen)
    return state


# ----------------------------------------------------------------------------- one pass


def run(state):
    case, fmt, x = state["case"], state["fmt"], state["x"]
    kind = case["kind"]
    if kind == "quantize":
        call = B.abs_quantize_transposed if case["option"].startswith("columns") else B.abs_quantize
        return call(fmt, x, opts=state["opts"])
    if kind == "roundtrip":
        codes, scales, alpha = B.abs_quantize(fmt, x, opts=state["opts"])
        return codes, scales, alpha, B.abs_dequantize(fmt, codes, scales, alpha, *x.shape, opts=state["opts"])
    if kind == "serve":
        qx = B.abs_quantize(fmt, x)
        return B.abs_matmul(fmt, qx, state["qw"], case["tokens"], case["d_out"], case["d_in"], bf16=True,
                            next_fmt=fmt if case["chained"] else None)
    if kind == "forward":
        return linear.forward_tc(x, state["w"], fmt)
    if kind == "backward":
        return linear.backward_tc(x, state["w"], state["dy"], fmt, sign_mask=SIGN_MASK, seed=state["seed"])
    y = linear.forward(x, state["w"], fmt)
    return (y, *linear.backward(x, state["w"], state["dy"], fmt, sign_mask=SIGN_MASK, seed=state["seed"]))


# ----------------------------------------------------------------------------- what a pass cannot do without


def work(case):
    kind, fmt = case["kind"], B.FMT_NAMES[case["fmt"]]
    per_value = B.FMT_BITS[fmt] / 8 + 1 / B.FMT_GROUP[fmt]            # bytes of codes and scales
    if kind in ("roundtrip", "quantize"):
        n = case["rows"] * case["cols"]
        return {"bytes": n * (2 + per_value) * (2 if kind == "roundtrip" else 1), "flops": 0}
    t, k, n = case["tokens"], case["d_in"], case["d_out"]
    if kind == "serve":
        return {"bytes": 2 * t * k + per_value * n * k + 2 * t * n, "flops": 2 * t * k * n}
    if kind == "forward":
        return {"bytes": 2 * t * k + 2 * n * k + 4 * t * n, "flops": 2 * t * k * n}
    if kind == "backward":
        return {"bytes": 2 * (t * k + n * k + t * n) + 4 * (t * k + n * k), "flops": 4 * t * k * n}
    return {"bytes": 2 * (t * k + n * k + t * n) + 2 * (t * n + t * k + n * k), "flops": 6 * t * k * n}


def tolerance(case):
    kind = case["kind"]
    if kind in ("roundtrip", "quantize"):
        return "exact"                  # codes, scales, alpha and decoded values are defined bit for bit
    if kind in ("forward", "backward"):
        # float32 outputs of exact products summed in float32: 6e-8 against float64, 5e-8 against a sum in another order
        # inside the tensor cores; a plain float32 chain over the groups of K adds the square root of its length
        return {"rel": 1e-6}
    if kind == "serve" and case["chained"]:
        return {"rel": 5e-3}            # the tensor scale is one bf16 value: one rounding of it the other way is 2^-8
    return {"rel": 6e-4}                # bf16 outputs: 1.6e-4 for a library GEMM against float64, 1e-5 for this kernel

"""The workloads this library is timed on, as an optimiser that trains a decoder calls it.

Five kinds of case, all through the package's public functions:

  root       one matrix through fp4_root_ns (clip, normalise, Newton-Schulz iterations)
  stack      the projections of a decoder stack through one fp4_root_ns_batched call
  optimizer  the whole Root step of a decoder stack: momentum in the 5-bit state with stochastic
             rounding, its clip histograms handed to the batched call, weights updated by it
  quantize   fp4_quantize of one tensor
  adamw      fp4_adamw_update of one flat parameter tensor

Sizes come from workloads.py (the benchmark's stack, the four-block timing shapes), from the sweep
and from bench.py; the ragged ones are generic: multiples of 16 (the block length) that are
multiples of neither 128 nor 256.  `option` selects what a caller may choose: "base" (plain NVFP4
rounding), "paper" (random Hadamard transform and adaptive 4/6 scaling) and, for matrices, "bf16"
(BF16 storage of the high-precision copies).
"""
from __future__ import annotations

import math

import torch

import paper_2607_04422_b200 as fp4
from paper_2607_04422_b200 import workloads

STEPS = 5           # Newton-Schulz iterations of the method
MU = 0.95           # momentum
LR, WEIGHT_DECAY = 0.02, 0.1
FLAGS = {"base": 0, "paper": fp4.FP4_FLAG_RHT | fp4.FP4_FLAG_FOUR_SIX, "bf16": fp4.FP4_FLAG_STORE_BF16}
SIGNS = 0xA53C      # sign mask of fp4_quantize with the transform


def listed():
    return [
        # the smallest matrix of the configurations: bound by launches and latency
        {"name": "root 256x512", "kind": "root", "rows": 256, "cols": 512, "option": "base", "input": "gaussian"},
        # one attention projection of a 1-2 B model on its own, low-rank with outliers for the clip
        {"name": "root 2048 square", "kind": "root", "rows": 2048, "cols": 2048, "option": "base", "input": "lowrank"},
        # an MLP down projection (tall: worked on transposed), memory-saving storage
        {"name": "root 8192x2048 bf16", "kind": "root", "rows": 8192, "cols": 2048, "option": "bf16", "input": "rows"},
        # one matrix of a shape that is a multiple of 16 only, with the paper's quantiser
        {"name": "root 1040x2896 paper", "kind": "root", "rows": 1040, "cols": 2896, "option": "paper",
         "input": "gradient"},
        # the largest matrix of the sweep
        {"name": "root 16384 square", "kind": "root", "rows": 16384, "cols": 16384, "option": "base",
         "input": "gaussian"},
        # the benchmark: four blocks of a 3 B decoder in one call
        {"name": "stack 3B", "kind": "stack", "hidden": 3072, "kv": 3072, "ffn": 8192, "blocks": 4, "option": "base"},
        # one block of the d = 4096 timing shapes (grouped-query attention) with the paper's quantiser
        {"name": "stack 4096 gqa paper", "kind": "stack", "hidden": 4096, "kv": 1024, "ffn": 11008, "blocks": 1,
         "option": "paper"},
        # two blocks of a small decoder whose sizes fit no tile
        {"name": "stack 1600 ragged", "kind": "stack", "hidden": 1600, "kv": 400, "ffn": 4304, "blocks": 2,
         "option": "base"},
        # a whole optimiser step on one block of the 3 B decoder
        {"name": "optimizer 3B block", "kind": "optimizer", "hidden": 3072, "kv": 3072, "ffn": 8192, "blocks": 1,
         "option": "base"},
        # a large weight or activation tensor, and a small one with the paper's quantiser
        {"name": "quantize 8192", "kind": "quantize", "rows": 8192, "cols": 8192, "option": "base"},
        {"name": "quantize 1152x2688 paper", "kind": "quantize", "rows": 1152, "cols": 2688, "option": "paper"},
        # the parameters outside Root's matrices: embeddings and the like
        {"name": "adamw 64M", "kind": "adamw", "n": 1 << 26, "sr": False},
    ]


def _size(rng, lo, hi, unit=16):
    """A multiple of `unit` in [lo, hi], spread over its logarithm; half of the time a round one."""
    v = math.exp(rng.uniform(math.log(lo), math.log(hi)))
    if rng.random() < 0.5:
        unit = max(unit, 256 if v >= 512 else 128)
    return max(lo, min(hi, int(round(v / unit)) * unit))


def draw(rng):
    kind = rng.choice(["root", "root", "root", "stack", "optimizer", "quantize", "adamw"])
    # BF16 storage is for shapes whose dimensions are multiples of 256: elsewhere it saves nothing
    if kind == "root":
        option = rng.choice(["base", "paper", "bf16"])
        lo, unit = (256, 256) if option == "bf16" else (128, 16)
        return {"kind": kind, "rows": _size(rng, lo, 8192, unit), "cols": _size(rng, lo, 8192, unit),
                "option": option, "input": rng.choice(["gaussian", "lowrank", "rows", "gradient"])}
    if kind in ("stack", "optimizer"):
        option = rng.choice(["base", "base", "paper", "bf16"])
        unit = 256 if option == "bf16" else 16
        hidden = _size(rng, 512, 4096 if kind == "stack" else 2560, unit)
        kv = max(unit, hidden // rng.choice([1, 4, 8]) // unit * unit)
        ffn = int(hidden * rng.uniform(2.0, 4.0)) // unit * unit
        return {"kind": kind, "hidden": hidden, "kv": kv, "ffn": ffn, "blocks": rng.choice([1, 2]), "option": option}
    if kind == "quantize":
        return {"kind": kind, "rows": _size(rng, 128, 16384, 128), "cols": _size(rng, 128, 8192, 128),
                "option": rng.choice(["base", "paper"])}
    return {"kind": "adamw", "n": 256 * int(math.exp(rng.uniform(math.log(1 << 8), math.log(1 << 18)))),
            "sr": rng.random() < 0.5}


def _shapes(case):
    """(m, n) of every matrix of a case."""
    if case["kind"] in ("stack", "optimizer"):
        return [(m, n) for _, m, n in workloads.gqa_stack_shapes(case["hidden"], case["ffn"], case["kv"],
                                                                  case["blocks"])]
    return [(case["rows"], case["cols"])]


def _matrix(m, n, kind, gen):
    """An update matrix as workloads.py draws it, made on the GPU."""
    def randn(*shape):
        return torch.randn(shape, device="cuda", generator=gen)

    def mask(frac):
        return torch.rand((m, n), device="cuda", generator=gen) < frac
    if kind == "gaussian":
        return randn(m, n)
    if kind == "rows":                       # rows of log-normal magnitude
        return randn(m, n) * torch.exp(randn(m, 1))
    if kind == "lowrank":                    # rank 64 plus noise, 0.1 % heavy-tailed outliers (Student-t, nu = 3)
        x = randn(m, 64) @ randn(n, 64).T / 8.0 + 0.1 * randn(m, n)
        t = randn(m, n) / torch.sqrt((randn(m, n) ** 2 + randn(m, n) ** 2 + randn(m, n) ** 2) / 3.0)
        return torch.where(mask(1e-3), 20.0 * t, x)
    x = randn(m, n) + randn(m, 32) @ randn(n, 32).T / math.sqrt(32.0)   # gradient-like: rank 32 plus noise
    return torch.where(mask(5e-4), 20.0 * x, x)


def _bytes(n):
    return torch.empty(n, dtype=torch.uint8, device="cuda")


def prepare(case, seed):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(int(seed))
    kind, st = case["kind"], {"kind": case["kind"]}
    if kind == "root":
        m, n = case["rows"], case["cols"]
        flags = FLAGS[case["option"]]
        st["G"] = _matrix(m, n, case["input"], gen)
        st["out"] = torch.empty_like(st["G"])
        st["params"] = fp4.NsParams.make(flags=flags, seed=7) if flags else None
        st["ws"] = _bytes(fp4.fp4_root_ns_workspace_bytes(m, n, STEPS, flags))
    elif kind == "stack":
        shapes, flags = _shapes(case), FLAGS[case["option"]]
        st["G"] = [_matrix(m, n, "gradient", gen) for m, n in shapes]
        st["out"] = [torch.empty_like(g) for g in st["G"]]
        st["params"] = fp4.NsParams.make(flags=flags, seed=7) if flags else None
        st["ws"] = _bytes(fp4.fp4_root_ns_batched_workspace_bytes(shapes, STEPS, flags))
    elif kind == "optimizer":
        shapes, flags = _shapes(case), FLAGS[case["option"]] | fp4.FP4_FLAG_NO_OUT
        st["G"] = [_matrix(m, n, "gradient", gen) for m, n in shapes]
        st["M"] = [torch.empty_like(g) for g in st["G"]]
        st["out"] = [torch.empty_like(g) for g in st["G"]]
        st["W"] = [(torch.randn((m, n), device="cuda", generator=gen) * 0.05).to(torch.bfloat16) for m, n in shapes]
        st["codes"] = [torch.zeros((m, n // 2), dtype=torch.uint8, device="cuda") for m, n in shapes]
        st["scales"] = [torch.zeros((m, n // 16), dtype=torch.int16, device="cuda") for m, n in shapes]
        st["hist"] = torch.zeros((len(shapes), 8192), dtype=torch.int32, device="cuda")
        st["params"] = fp4.NsParams.make(flags=flags, seed=7, top_hist=list(st["hist"]), weights=st["W"], lr=LR,
                                         weight_decay=WEIGHT_DECAY)
        st["ws"] = _bytes(fp4.fp4_root_ns_batched_workspace_bytes(shapes, STEPS, flags))
        st["t"] = 1
        # a run under way: the state holds the momentum of an earlier gradient
        for i, (m, n) in enumerate(shapes):
            fp4.fp4_momentum_update(_matrix(m, n, "gradient", gen), st["codes"][i], st["scales"][i], None, None, MU)
    elif kind == "quantize":
        m, n = case["rows"], case["cols"]
        st["x"] = _matrix(m, n, "rows", gen)
        st["codes"] = torch.empty((m, n // 2), dtype=torch.uint8, device="cuda")
        st["scales"] = _bytes(fp4.fp4_scale_bytes(m, n))
        st["tensor_scale"] = torch.empty(1, device="cuda")
        st["flags"] = FLAGS[case["option"]] | (SIGNS << 16 if case["option"] == "paper" else 0)
    else:
        n = case["n"]
        st["W"] = (torch.randn(n, device="cuda", generator=gen) * 0.05).to(torch.bfloat16)
        scale = torch.exp(torch.randn((n // 256, 1), device="cuda", generator=gen)) * 1e-2

        def gradient():
            return (torch.randn((n // 256, 256), device="cuda", generator=gen) * scale).reshape(n).to(torch.bfloat16)
        st["m_codes"], st["v_codes"] = (torch.zeros(n // 2, dtype=torch.uint8, device="cuda") for _ in range(2))
        st["m_scales"], st["v_scales"] = (torch.zeros(n // 16, dtype=torch.int16, device="cuda") for _ in range(2))
        st["v_means"] = torch.zeros(n // 256, dtype=torch.int16, device="cuda")
        st["flags"] = fp4.FP4_MOM_FLAG_SR if case["sr"] else 0
        st["t"] = 1
        st["G"] = gradient()
        _adamw(st)                           # a run under way: both moments hold an earlier gradient
        st["G"] = gradient()
    return st


def _adamw(st):
    fp4.fp4_adamw_update(st["W"], st["G"], st["m_codes"], st["m_scales"], st["v_codes"], st["v_scales"], st["v_means"],
                         lr=1e-3, step=st["t"], flags=st["flags"], seed=st["t"])
    st["t"] += 1


def run(state):
    kind = state["kind"]
    if kind == "root":
        fp4.fp4_root_ns(state["G"], state["out"], STEPS, state["params"], state["ws"])
        return state["out"]
    if kind == "stack":
        fp4.fp4_root_ns_batched(state["G"], state["out"], STEPS, state["params"], state["ws"])
        return state["out"]
    if kind == "optimizer":
        t = state["t"]
        state["t"] = t + 1
        for i, g in enumerate(state["G"]):
            fp4.fp4_momentum_update(g, state["codes"][i], state["scales"][i], state["M"][i], state["hist"][i], MU,
                                    flags=fp4.FP4_MOM_FLAG_SR, seed=t)
        fp4.fp4_root_ns_batched(state["M"], state["out"], STEPS, state["params"], state["ws"])
        return [state["W"], state["codes"], state["scales"], state["M"]]
    if kind == "quantize":
        fp4.fp4_quantize(state["x"], state["codes"], state["scales"], state["tensor_scale"], state["flags"])
        return [state["codes"], state["scales"], state["tensor_scale"]]
    _adamw(state)
    return [state[k] for k in ("W", "m_codes", "m_scales", "v_codes", "v_scales", "v_means")]


def work(case):
    kind = case["kind"]
    if kind == "quantize":                   # FP32 in; 4-bit codes and a scale byte per 16 out
        n = case["rows"] * case["cols"]
        return {"bytes": n * (4 + 0.5625), "flops": 4.0 * n}
    if kind == "adamw":                      # W in and out, G in, the 5-bit and the 5.0625-bit state in and out
        return {"bytes": case["n"] * 8.515625, "flops": 100.0 * case["n"]}
    elements = flops = 0.0
    for m, n in _shapes(case):
        s, l = min(m, n), max(m, n)
        elements += m * n
        flops += STEPS * (3.0 * s * s * l + 1.0 * s ** 3)   # the two symmetric products: upper triangle only
    # root: FP32 in and out.  optimizer: G in, M out, W in and out, the momentum state in and out
    per = 8.0 if kind != "optimizer" else 4 + 4 + 4 + 2 * 0.625
    return {"bytes": elements * per, "flops": flops}


def tolerance(case):
    # Codes, scales and BF16 weights of the quantiser and of AdamW are defined bit for bit, and so are the
    # momentum and its state.
    if case["kind"] in ("quantize", "adamw"):
        return "exact"
    # The iterations against the CPU oracle, whose products are summed in FP64 (12 shapes up to 2048 x 2048, four
    # kinds of input): a sum that falls on the other side of a rounding boundary changes one code, which
    # the following iterations spread.  Seen: 2.1e-5 (largest element 2.4e-3) with plain rounding, either
    # storage; 1.05e-2 (0.32) with the paper's quantiser, where a near-tie of the two encodings changes a whole block.
    return {"rel": 3e-2, "max": 0.95} if case["option"] == "paper" else {"rel": 1e-4, "max": 1e-2}

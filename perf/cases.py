"""The calls users of this library make, as cases to time: shapes and options, inputs, one pass, what it cannot do
without, and how far another correct implementation may be off.

Every case goes through the public functions of `paper_2411_09909_b200.amx` with their defaults (outputs and scratch
come from the call).  Kinds of cases:

  linear     one fully quantized linear layer, `quant_gemm`: bf16 activation cast in the call, the weight quantized
             ahead or cast in the call too; group size 32 and the ablation's 16, 64 and 128
  decode     one token step: a few rows through all linear layers of one decoder block, canonical weights
  prepared   prefill with a weight prepared once: `quantize_prepared` + `gemm_prepared`, or the NVFP4 pair
  attention  `attention_heads`: all heads of one layer, grouped queries, causal or not
  cast       one direct cast of a tensor: `quantize`, `fake_quantize` (the paper's emulation) or `dequantize`
  report     one line of the error report: `quantize`, then `quant_error`

Layer shapes are those of `inputs.LINEAR_CONFIGS`; activations have channel outliers and offsets (or the SiLU skew),
weights are normal, as `inputs` draws them.
"""
from __future__ import annotations

import torch

from paper_2411_09909_b200 import amx
from paper_2411_09909_b200.inputs import LINEAR_CONFIGS

FORMATS = {"amxfp4": amx.FMT_AMXFP4, "sym_fp8": amx.FMT_SYM_FP8, "mxfp4": amx.FMT_MXFP4, "amxfp4_pot": amx.FMT_AMXFP4_POT,
           "mxfp4_round": amx.FMT_MXFP4_POT_ROUND, "amxfp4_round": amx.FMT_AMXFP4_POT_ROUND}


def listed():
    return [
        # a small layer, batch of 128 tokens (config 1): launches and host work decide
        {"name": "linear_128x1024x1024", "kind": "linear", "M": 128, "N": 1024, "K": 1024, "gs": 32, "weight": "quantized"},
        # one user's next token through the four linears of a 7B decoder block
        {"name": "decode_7b_1row", "kind": "decode", "config": 2, "M": 1},
        # a served batch of 24 sequences, the 8B block
        {"name": "decode_8b_24rows", "kind": "decode", "config": 3, "M": 24},
        # a prompt of odd length through the 7B up projection, weight quantized ahead
        {"name": "linear_1000x11008x4096", "kind": "linear", "M": 1000, "N": 11008, "K": 4096, "gs": 32, "weight": "quantized"},
        # the paper's direct-cast setting: both operands bf16, both cast per call (config 2, QKV)
        {"name": "linear_both_2048x12288x4096", "kind": "linear", "M": 2048, "N": 12288, "K": 4096, "gs": 32, "weight": "bf16"},
        # group-size ablation: the same layer with groups of 128 (tests and the error report use 16, 64 and 128 as well)
        {"name": "linear_gs128_1024x4096x4096", "kind": "linear", "M": 1024, "N": 4096, "K": 4096, "gs": 128, "weight": "quantized"},
        # 70B prefill, 16384 tokens, weight prepared once (config 4, QKV): the benchmark's own layer
        {"name": "prefill_70b_qkv", "kind": "prepared", "M": 16384, "N": 10240, "K": 8192, "fmt": "amxfp4", "out": "f32"},
        # the symmetric format the paper compares with, 8B gate projection, result for a bf16 consumer
        {"name": "prefill_8b_gate_mxfp4", "kind": "prepared", "M": 8192, "N": 14336, "K": 4096, "fmt": "mxfp4", "out": "bf16"},
        # long-context attention of one layer (config 5)
        {"name": "attention_32x8192", "kind": "attention", "heads": 32, "kv_heads": 32, "L": 8192, "d": 128, "causal": False},
        # an ordinary prompt, ragged length, grouped queries, causal
        {"name": "attention_32over8_1056_causal", "kind": "attention", "heads": 32, "kv_heads": 8, "L": 1056, "d": 128, "causal": True},
        # casting an activation (or a weight, once) of the largest layer
        {"name": "quantize_16384x8192", "kind": "cast", "op": "quantize", "rows": 16384, "K": 8192, "gs": 32, "fmt": "amxfp4"},
        # one line of the error report, group 16
        {"name": "report_4096x11008_gs16", "kind": "report", "rows": 4096, "K": 11008, "gs": 16, "fmt": "amxfp4"},
    ]


def _log(rng, lo, hi):
    return int(round(lo * (hi / lo) ** rng.random()))


def draw(rng):
    kind = rng.choice(("linear", "linear", "decode", "prepared", "prepared", "attention", "attention", "cast", "report"))
    if kind == "linear":
        gs = rng.choice((32, 32, 32, 16, 64, 128))
        return {"kind": kind, "M": _log(rng, 1, 4096 if gs == 32 else 1024), "N": _log(rng, 512, 14336 if gs == 32 else 4096),
                "K": max(1, _log(rng, 512, 8192 if gs == 32 else 4096) // 128) * 128, "gs": gs,
                "weight": rng.choice(("quantized", "quantized", "bf16"))}
    if kind == "decode":
        return {"kind": kind, "config": rng.choice((2, 3)), "M": _log(rng, 1, 64)}
    if kind == "prepared":
        K, N = rng.choice([s for c in (2, 3) for s in LINEAR_CONFIGS[c]["layers"]] + [LINEAR_CONFIGS[4]["layers"][0]])
        fmt = rng.choice(("amxfp4", "amxfp4", "sym_fp8", "mxfp4", "nvfp4", "anvfp4"))
        return {"kind": kind, "M": _log(rng, 256, 16384), "N": N, "K": K, "fmt": fmt,
                "out": "f32" if "nv" in fmt else rng.choice(("f32", "bf16"))}
    if kind == "attention":
        heads = rng.choice((8, 16, 32))
        return {"kind": kind, "heads": heads, "kv_heads": heads // rng.choice((1, 4, 8)), "L": _log(rng, 4, 256) * 32,
                "d": rng.choice((64, 128, 128)), "causal": rng.choice((True, False))}
    rows, K, gs = _log(rng, 64, 16384), _log(rng, 8, 64) * 128, rng.choice((32, 32, 16, 64, 128))
    if kind == "cast":
        return {"kind": kind, "op": rng.choice(("quantize", "fake_quantize", "dequantize")), "rows": rows, "K": K, "gs": gs,
                "fmt": rng.choice(tuple(FORMATS))}
    return {"kind": kind, "rows": rows, "K": K, "gs": gs, "fmt": rng.choice(tuple(FORMATS))}


def _layers(case):
    """(N, K) of the layers one pass of a decode case goes through."""
    return [(N, K) for K, N in LINEAR_CONFIGS[case["config"]]["layers"]]


def _activation(g, rows, K, skewed=False):
    x = torch.randn(rows, K, device="cuda", generator=g)
    if skewed:
        return torch.nn.functional.silu(1.5 * x).to(torch.bfloat16)
    x += 0.3 * torch.randn(K, device="cuda", generator=g)
    x[:, torch.randperm(K, device="cuda", generator=g)[:max(1, K // 200)]] *= 60.0
    return x.to(torch.bfloat16)


def _weight(g, N, K):
    return (0.02 * torch.randn(N, K, device="cuda", generator=g)).to(torch.bfloat16)


def prepare(case, seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    s = dict(case)
    if case["kind"] == "linear":
        s["x"], w = _activation(g, case["M"], case["K"]), _weight(g, case["N"], case["K"])
        if case["weight"] == "bf16":
            s["w"] = w
        else:
            s["codes"], s["scales"] = amx.quantize(w, case["gs"])
    elif case["kind"] == "decode":
        skewed = case["config"] == 3
        s["layers"] = [(_activation(g, case["M"], K, skewed), *amx.quantize(_weight(g, N, K))) for N, K in _layers(case)]
    elif case["kind"] == "prepared":
        s["x"], w = _activation(g, case["M"], case["K"], skewed=case["fmt"] == "mxfp4"), _weight(g, case["N"], case["K"])
        if "nv" in case["fmt"]:
            s["w"] = amx.quantize_nvfp4(w, case["fmt"] == "anvfp4", prepared_as="w")[3]
        else:
            s["w"] = amx.quantize_prepared(w, True, fmt=FORMATS[case["fmt"]], want_codes=False)[2]
    elif case["kind"] == "attention":
        for t, heads in (("q", case["heads"]), ("k", case["kv_heads"]), ("v", case["kv_heads"])):
            x = torch.randn(heads, case["L"], case["d"], device="cuda", generator=g)
            x[:, :, torch.randperm(case["d"], device="cuda", generator=g)[:2]] *= 20.0
            s[t] = x.to(torch.bfloat16)
    else:
        s["x"] = _activation(g, case["rows"], case["K"])
        if case.get("op") == "dequantize":
            s["codes"], s["scales"] = amx.quantize(s["x"], case["gs"], FORMATS[case["fmt"]])
    return s


def run(s):
    if s["kind"] == "linear":
        if s["weight"] == "bf16":
            return amx.quant_gemm(s["x"], group_size=s["gs"], w_bf16=s["w"])
        return amx.quant_gemm(s["x"], s["codes"], s["scales"], s["gs"])
    if s["kind"] == "decode":
        return [amx.quant_gemm(x, codes, scales) for x, codes, scales in s["layers"]]
    if s["kind"] == "prepared":
        M, N, K, fmt = s["M"], s["N"], s["K"], s["fmt"]
        if "nv" in fmt:
            _, scales, tensor_scale, a = amx.quantize_nvfp4(s["x"], fmt == "anvfp4", prepared_as="a")
            return [scales, tensor_scale, amx.gemm_nvfp4(a, s["w"], M, N, K, sym=fmt == "nvfp4")]
        _, scales, a = amx.quantize_prepared(s["x"], False, fmt=FORMATS[fmt], want_codes=False)
        return [scales, amx.gemm_prepared(a, s["w"], M, N, K, sym=fmt != "amxfp4",
                                          out_dtype=torch.bfloat16 if s["out"] == "bf16" else torch.float32)]
    if s["kind"] == "attention":
        return amx.attention_heads(s["q"], s["k"], s["v"], amx.ATTN_CAUSAL if s["causal"] else amx.GEMM_AUTO)
    fmt = FORMATS[s["fmt"]]
    if s["kind"] == "report":
        codes, scales = amx.quantize(s["x"], s["gs"], fmt)
        return [codes, scales, amx.quant_error(s["x"], codes, scales, s["gs"])]
    if s["op"] == "quantize":
        return amx.quantize(s["x"], s["gs"], fmt)
    if s["op"] == "fake_quantize":
        return amx.fake_quantize(s["x"], s["gs"], fmt)
    return amx.dequantize(s["codes"], s["scales"], s["gs"])


def work(case):
    """Inputs read once, outputs written once; useful operations of the products only."""
    kind = case["kind"]
    if kind in ("linear", "decode", "prepared"):
        M, nbytes, flops = case["M"], 0.0, 0.0
        for N, K in _layers(case) if kind == "decode" else [(case["N"], case["K"])]:
            gs = 16 if "nv" in case.get("fmt", "") else case.get("gs", 32)
            weight = 2.0 if case.get("weight") == "bf16" else 0.5 + 2.0 / gs
            nbytes += 2.0 * M * K + weight * N * K + (2.0 if case.get("out") == "bf16" else 4.0) * M * N
            nbytes += 2.0 * M * K / gs if kind == "prepared" else 0.0          # the canonical scales come back too
            flops += 2.0 * M * N * K
        return {"bytes": nbytes, "flops": flops}
    if kind == "attention":
        H, KV, L, d = case["heads"], case["kv_heads"], case["L"], case["d"]
        return {"bytes": 2.0 * L * d * (H + 2 * KV) + 4.0 * L * d * H, "flops": 4.0 * L * L * d * H / (2 if case["causal"] else 1)}
    per = {"quantize": 2.5, "report": 2.5, "fake_quantize": 4.0, "dequantize": 2.5}[case.get("op", "report")]
    return {"bytes": (per + (0.0 if per == 4.0 else 2.0 / case["gs"])) * case["rows"] * case["K"], "flops": 0.0}


def tolerance(case):
    kind = case["kind"]
    if kind == "cast":
        return "exact"                               # codes, scales and decoded values are determined bit for bit
    if kind == "report":
        return {"rel": 2e-6}                         # the sums only; the codes are whole numbers and stay the same
    if kind == "attention":
        # fp32 softmax rounded to bf16 and cast to FP4: a last-bit difference of one probability can move a code
        return {"rel": 5e-3, "max": 0.5}
    return {"rel": 4e-3 if case.get("out") == "bf16" else 1e-5}   # fp32 accumulation in another order

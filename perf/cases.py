"""The work this library is used for, as cases that can be timed and compared.

Every case is one call, or the two calls that belong together, of ``paper_2104_08378_b200.binding`` on tensors that
are already on the GPU: the forward product of a 2:4-pruned linear layer over prompts (many tokens) and in token-by-
token decoding (few tokens), the INT8 deployment with its dequantising epilogue, a pruned 3x3 convolution, the
pruning-and-compression of a weight matrix, and the re-imposition of the pattern after a weight update.

``listed`` holds the workloads of the repository's configurations and benchmark and a few generic sizes between them;
``draw`` spreads the same kinds over the whole range of sizes, ragged ones among them.
"""
import math

import torch

from paper_2104_08378_b200 import binding as sp

MAX_PRODUCT = 49152 * 8192 * 12288   # M * N * K of the largest listed product
MAX_WEIGHT = 49152 * 12288


def _linear(name, ab, M, N, K, **more):
    """One product: weights M x K (compressed), N tokens.  cd: result type; tokens_out: result as [tokens, M] instead
    of [M, tokens]; beta: C is added; b_rows: activations stored K x N; pad: row padding of activations and result in
    elements (a slice of a wider buffer)."""
    case = {"name": name, "kind": "linear", "ab": ab, "cd": ab, "M": M, "N": N, "K": K, "tokens_out": False,
            "beta": 0.0, "b_rows": False, "pad": 0}
    case.update(more)
    return case


def listed():
    return [
        # the smallest call: a projection of a small model, one short prompt; launch latency is what counts
        _linear("tiny_f16", "f16", 256, 256, 512),
        # token-by-token decoding of 32 sequences through the largest layer: streams the whole compressed weight
        _linear("decode_large_bf16", "bf16", 49152, 32, 12288, tokens_out=True),
        # the same in the INT8 deployment with a mid-sized layer and 32 sequences: a short call
        {"name": "decode_int8", "kind": "dequant", "M": 4096, "N": 32, "K": 4096, "cd": "bf16", "tokens_out": True,
         "bias": True, "relu": False},
        # BERT-base feed-forward up-projection, 32 sequences of 128 tokens
        _linear("bert_ffn_bf16", "bf16", 3072, 4096, 768),
        # a ragged product with an addend, activations stored K x N, padded rows: what a fused graph with odd sizes calls
        _linear("ragged_f16", "f16", 1184, 736, 1008, beta=-1.5, b_rows=True, pad=16),
        # INT8 linear layer, raw INT32 results
        _linear("int8_linear", "i8", 4096, 8192, 4096, cd="i32"),
        # INT8 deployment of the BERT layer: per-row scales, bias and ReLU, INT8 activations [tokens, features] out
        {"name": "int8_ffn_requant", "kind": "dequant", "M": 3072, "N": 4096, "K": 768, "cd": "i8", "tokens_out": True,
         "bias": True, "relu": True},
        # TF32 layer (the 1:2 pattern), 8192 tokens
        _linear("tf32_linear", "f32", 4096, 8192, 4096),
        # 8-bit floating-point prompt processing, [tokens, features] in and out
        _linear("fp8_prefill", "e4m3", 16384, 8192, 8192, cd="bf16", tokens_out=True),
        # ResNet-50-style 3x3 convolution, NHWC in and out, batch 256
        {"name": "resnet_conv_f16", "kind": "conv", "ab": "f16", "Nb": 256, "H": 14, "W": 14, "Cin": 256, "M": 256},
        # sparse retraining of one layer: the pattern is imposed on the updated weights, which are compressed again
        {"name": "retrain_bf16", "kind": "retrain", "ab": "bf16", "M": 12288, "K": 3072},
        # the largest work: prune + compress of a GPT-3-sized feed-forward weight, then its product with 8192 tokens
        {"name": "gpt3_step_bf16", "kind": "step", "ab": "bf16", "M": 49152, "N": 8192, "K": 12288},
    ]


def _log(rng, lo, hi, multiple):
    """A multiple of `multiple` between lo and hi, even over the logarithm."""
    v = math.exp(rng.uniform(math.log(lo), math.log(hi)))
    return min(hi // multiple * multiple, max(multiple, round(v / multiple) * multiple))


def draw(rng):
    kind = rng.choice(["decode", "decode", "linear", "linear", "linear", "int8", "dequant", "conv", "retrain", "step"])
    if kind == "conv":
        h, w = rng.choice([(7, 7), (14, 14), (28, 28), (56, 56), (rng.randint(8, 40), rng.randint(8, 40))])
        unit = 16 // math.gcd(h * w, 16)                       # N * H * W has to be a multiple of 16
        nb = max(unit, _log(rng, 2, 256, unit))
        cin = rng.choice([128, 256, 384, 512])
        while nb > unit and nb * h * w * cin > 256 * 28 * 28 * 256:
            nb = max(unit, nb // 2 // unit * unit)
        while nb * h * w * cin * 2 < 131072:                   # the entry point's smallest activation
            nb += unit
        return {"kind": "conv", "ab": rng.choice(["f16", "bf16"]), "Nb": nb, "H": h, "W": w, "Cin": cin,
                "M": _log(rng, 64, 512, 16)}
    if kind == "retrain":
        M, K = _log(rng, 256, 49152, 1), _log(rng, 256, 12288, rng.choice([16, 64, 256]))
        return {"kind": "retrain", "ab": rng.choice(["bf16", "f16", "i8"]), "M": M, "K": K}
    M, K = _log(rng, 256, 49152, 16), _log(rng, 256, 12288, 16)
    if kind == "step":
        N = _log(rng, 256, 8192, 16)
        return {"kind": "step", "ab": rng.choice(["bf16", "f16"]), "M": M, "N": N, "K": K}
    if kind == "decode":
        N = rng.choice([16, 32, 48, 64, 96, 128])
        ab = rng.choice(["bf16", "f16", "e4m3", "i8"])
        if ab in ("e4m3", "i8"):
            M, N, K = (max(32, v // 32 * 32) for v in (M, N, K))
        if ab == "i8":
            return {"kind": "dequant", "M": M, "N": N, "K": K, "cd": "bf16", "tokens_out": True,
                    "bias": rng.random() < 0.5, "relu": rng.random() < 0.5}
        case = _linear("", ab, M, N, K, tokens_out=rng.random() < 0.75, cd="bf16" if ab == "e4m3" else ab)
    else:
        M, N, K = _log(rng, 256, 16384, 32), _log(rng, 192, 16384, 32), _log(rng, 256, 12288, 32)
        if kind == "dequant":
            return {"kind": "dequant", "M": M, "N": N, "K": K, "cd": rng.choice(["i8", "bf16"]),
                    "tokens_out": rng.random() < 0.75, "bias": True, "relu": rng.random() < 0.5}
        if kind == "int8":
            return _drop_name(_linear("", "i8", M, N, K, cd="i32", beta=rng.choice([0.0, 0.0, 1.0])))
        ab = rng.choice(["bf16", "bf16", "f16", "f32", "e4m3"])
        b_rows = rng.random() < 0.15
        case = _linear("", ab, M, N, K, cd="bf16" if ab == "e4m3" else ab, beta=rng.choice([0.0, 0.0, 1.0, -1.5]),
                       tokens_out=rng.random() < 0.5, b_rows=b_rows, pad=rng.choice([0, 0, 16]))
    return _drop_name(case)


def _drop_name(case):
    return {k: v for k, v in case.items() if k != "name"}


# ---- inputs ----------------------------------------------------------------------------------------------------------
def _values(g, shape, dt, sigma, pad=0):
    """Random values of type dt (N(0, sigma), or uniform int8); with pad, a view of rows that are `pad` longer."""
    full = (shape[0], shape[1] + pad) if pad else shape
    if dt == "i8":
        t = torch.randint(-127, 128, full, dtype=torch.int8, device="cuda", generator=g)
    elif dt == "i32":
        t = torch.randint(-1 << 20, 1 << 20, full, dtype=torch.int32, device="cuda", generator=g)
    elif dt == "f32":
        t = torch.randn(full, device="cuda", generator=g).mul_(sigma)
    elif dt in ("e4m3", "e5m2"):
        t = torch.randn(full, dtype=torch.bfloat16, device="cuda", generator=g).mul_(sigma).to(sp.TORCH_DTYPE[dt])
    else:
        t = torch.randn(full, dtype=sp.TORCH_DTYPE[dt], device="cuda", generator=g).mul_(sigma)
    return t[:, :shape[1]] if pad else t


def prepare(case, seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    kind = case["kind"]
    state = {"case": case}
    if kind in ("retrain", "step"):
        w = _values(g, (case["M"], case["K"]), case["ab"], 0.02)
        if kind == "retrain":
            # the pattern comes from the weights before the update
            _, state["meta"], _ = sp.compress(w)
            if case["ab"] == "i8":
                step = torch.randint(-8, 9, w.shape, dtype=torch.int8, device="cuda", generator=g)
                w = (w // 2).add_(step)
            else:
                w.add_(torch.randn(w.shape, dtype=w.dtype, device="cuda", generator=g), alpha=0.002)
            state["w"], state["masked"] = w, torch.empty_like(w)
            return state
        state.update(w=w, pruned=torch.empty_like(w), vals=torch.empty((case["M"], case["K"] // 2), dtype=w.dtype, device="cuda"),
                     meta=torch.empty(sp.meta_bytes(case["ab"], case["M"], case["K"]), dtype=torch.uint8, device="cuda"),
                     x=_values(g, (case["N"], case["K"]), case["ab"], 1.0), c=_values(g, (case["M"], case["N"]), case["ab"], 1.0),
                     out=torch.empty((case["M"], case["N"]), dtype=w.dtype, device="cuda"))
        return state
    if kind == "conv":
        K = 9 * case["Cin"]
        w = _values(g, (case["M"], K), case["ab"], math.sqrt(2.0 / K))
        state["x"] = _values(g, (case["Nb"] * case["H"] * case["W"], case["Cin"]), case["ab"], 1.0).relu_().view(
            case["Nb"], case["H"], case["W"], case["Cin"])
        state["vals"], state["meta"], _ = sp.compress(w)
        return state
    M, N, K = case["M"], case["N"], case["K"]
    ab = case.get("ab", "i8")
    state["vals"], state["meta"], _ = sp.compress(_values(g, (M, K), ab, 1.0 if ab == "e4m3" else 0.02))
    pad = case.get("pad", 0)
    state["x"] = _values(g, (K, N) if case.get("b_rows") else (N, K), ab, 1.0, pad)
    if kind == "dequant":
        # INT8 codes of about +-127 over K products: scales that bring the results to about +-1
        state["scale"] = torch.rand(M, device="cuda", generator=g).add_(0.5).mul_(1.0 / (5400.0 * math.sqrt(K)))
        state["bias"] = torch.randn(M, device="cuda", generator=g).mul_(0.1) if case["bias"] else None
        return state
    if case["beta"] != 0.0:
        state["c"] = _values(g, (N, M) if case["tokens_out"] else (M, N), case["cd"], 1.0, pad)
    if pad:
        rows, cols = (N, M) if case["tokens_out"] else (M, N)
        state["out"] = torch.empty((rows, cols + pad), dtype=sp.TORCH_DTYPE[case["cd"]], device="cuda")[:, :cols]
    return state


# ---- one pass --------------------------------------------------------------------------------------------------------
def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "linear":
        return sp.gemm(state["vals"], state["meta"], state["x"], beta=case["beta"], C=state.get("c"), out=state.get("out"),
                       cd=case["cd"], b_row_major=case["b_rows"], cd_col_major=case["tokens_out"])
    if kind == "dequant":
        return sp.gemm_i8_dequant(state["vals"], state["meta"], state["x"], state["scale"], bias=state["bias"],
                                  relu=case["relu"], out_scale=0.03, cd=case["cd"], cd_col_major=case["tokens_out"])
    if kind == "conv":
        return sp.conv3x3_nhwc(state["vals"], state["meta"], state["x"], nhwc_out=True)
    if kind == "retrain":
        masked = sp.apply_mask(state["w"], state["meta"], out=state["masked"])
        vals, meta, _ = sp.compress(masked)
        return [masked, vals, meta]
    sp.prune_compress(state["w"], pruned=state["pruned"], vals=state["vals"], meta=state["meta"])
    sp.gemm(state["vals"], state["meta"], state["x"], beta=1.0, C=state["c"], out=state["out"])
    return [state["pruned"], state["vals"], state["meta"], state["out"]]


# ---- what a pass cannot do without -----------------------------------------------------------------------------------
_BYTES = {"f16": 2, "bf16": 2, "f32": 4, "i8": 1, "i32": 4, "e4m3": 1, "e5m2": 1}


def _compressed_bytes(ab, M, K):
    """Kept values and 2 bits of position each (one nibble per pair in the 1:2 pattern)."""
    return M * K // 2 * _BYTES[ab] + (M * K // 4 if ab == "f32" else M * K // 8)


def work(case):
    """flops: the M * N * K / 2 multiply-adds of the kept values, so that the sparse tensor rate in these units is the
    dense rate of the same type."""
    kind = case["kind"]
    if kind == "retrain":
        M, K, ab = case["M"], case["K"], case["ab"]
        return {"bytes": 2 * M * K * _BYTES[ab] + M * K // 8 + _compressed_bytes(ab, M, K), "flops": 0.0}
    if kind == "conv":
        pixels, K = case["Nb"] * case["H"] * case["W"], 9 * case["Cin"]
        return {"bytes": 2 * pixels * (case["Cin"] + case["M"]) + _compressed_bytes(case["ab"], case["M"], K),
                "flops": float(case["M"]) * pixels * K}
    M, N, K = case["M"], case["N"], case["K"]
    if kind == "step":
        # weight in, pruned weight and compressed form out (the product reads the compressed form as it is made), C, D, x
        return {"bytes": 2 * (2 * M * K + 2 * M * N + N * K) + _compressed_bytes(case["ab"], M, K), "flops": float(M) * N * K}
    ab = case.get("ab", "i8")
    outs = M * N * _BYTES[case["cd"]] * (2 if case.get("beta") else 1)
    extra = 4 * M * (2 if case.get("bias") else 1) if kind == "dequant" else 0
    return {"bytes": _compressed_bytes(ab, M, K) + N * K * _BYTES[ab] + outs + extra, "flops": float(M) * N * K}


def tolerance(case):
    """INT8 products and everything that selects, moves or codes values is defined bit for bit (the dequantising
    epilogue has one fixed order of FP32 operations).  Floating products: about four times the distance of the result
    from a product in 64 bits: 1.66e-3 for BF16 and 2.07e-4 for FP16 results whatever K (the rounding of the result),
    4.8e-6 at K = 4096 for FP32 results (the running sum in the tensor cores)."""
    kind = case["kind"]
    if kind in ("retrain", "dequant"):
        return "exact"
    cd = case.get("cd", case.get("ab"))
    if cd == "i32":
        return "exact"
    if cd == "f32":
        return {"rel": max(1e-5, 5e-9 * case["K"])}
    return {"rel": 6.6e-3} if cd == "bf16" else {"rel": 9e-4}

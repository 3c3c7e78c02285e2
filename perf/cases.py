"""The work that users of this library have it do, as cases that can be timed and compared.

A case is one pass through the public binding: a linear layer, the four linear layers of a transformer
block, a patch embedding, or the offline preparation of a block's weights.  Sizes are those of the
workload configurations of ``inputs.py`` (DeiT, Swin, ViT) and of the ranges around them; inputs are
drawn on the GPU with the distributions described there.

kind "layer" / "block": activations [m, h] in, outputs out.  The attention between qkv and proj and
the LayerNorm and residual between proj and fc1 are not part of this library, so those layers get
activations of their own; fc2 reads what fc1 wrote.  mode says which model runs:
  computed  INT8 2:4 layers, every activation scale computed from the tensor
  supplied  the deployed INT8 model: supplied scales, fc1 writes the INT8 codes that fc2 reads
  absmax    INT8 with computed scales, fc2's derived from the maximum that fc1's epilogue reports
  int4      4-bit weights and activations on the INT8 path, computed scales
  f16       the FP16 2:4 model, no quantise node
kind "patch": image batch -> quantised patch rows -> embeddings, "computed" or "supplied" scale.
kind "weights": FP32 weights of a block -> packed operands, mode "int8", "f16" or "int4" (stored form
and its expansion).
"""
import math

import torch

from paper_2305_10727_b200 import binding as B

# Largest activation tensor of a drawn block, in elements: that of the largest listed one.
_MAX_MH = 65792 * 1280


def listed():
    return [
        # one MLP layer of the smallest model at batch 8: a call of two launches, where latency counts
        {"name": "layer_deit_tiny_b8", "kind": "layer", "mode": "computed", "m": 8 * 197, "h": 192, "n": 768,
         "gelu": True, "out": "f16", "dist": "normal"},
        # a large model answering one image: launches, and a token count that fills no tile
        {"name": "block_vit_huge_b1", "kind": "block", "mode": "computed", "m": 257, "h": 1280, "mlp": 5120,
         "dist": "normal"},
        # an odd, small batch of the 4-bit model
        {"name": "block_deit_base_b5_int4", "kind": "block", "mode": "int4", "m": 5 * 197, "h": 768, "mlp": 3072,
         "dist": "normal"},
        # the headline workload: DeiT-Base at the batch of an inference server
        {"name": "block_deit_base_b64", "kind": "block", "mode": "computed", "m": 64 * 197, "h": 768, "mlp": 3072,
         "dist": "normal"},
        # the sparse FP16 model that the INT8 one is made from, same batch
        {"name": "block_deit_base_b64_f16", "kind": "block", "mode": "f16", "m": 64 * 197, "h": 768, "mlp": 3072,
         "dist": "normal"},
        # the deployed form of a larger model
        {"name": "block_vit_large_b128_supplied", "kind": "block", "mode": "supplied", "m": 128 * 197, "h": 1024,
         "mlp": 4096, "dist": "normal"},
        # short rows, heavy-tailed activations, scales taken from the producing layer
        {"name": "block_swin_base_s3_b256_absmax", "kind": "block", "mode": "absmax", "m": 256 * 196, "h": 512,
         "mlp": 2048, "dist": "student_t4"},
        # many tokens, widths that fill no 128-feature tile
        {"name": "block_swin_tiny_s1_b32_supplied", "kind": "block", "mode": "supplied", "m": 32 * 3136, "h": 96,
         "mlp": 384, "dist": "student_t4"},
        # offline throughput: the largest model at the largest batch
        {"name": "block_vit_huge_b256", "kind": "block", "mode": "computed", "m": 256 * 257, "h": 1280, "mlp": 5120,
         "dist": "normal"},
        # the first layer of a model
        {"name": "patch_deit_base_p16_b64", "kind": "patch", "mode": "computed", "b": 64, "side": 224, "p": 16,
         "n": 768},
        # making a model's INT8 weights, and the 4-bit ones (stored form, then what the GEMM reads)
        {"name": "weights_vit_large_int8", "kind": "weights", "mode": "int8", "h": 1024, "mlp": 4096},
        {"name": "weights_deit_base_int4", "kind": "weights", "mode": "int4", "h": 768, "mlp": 3072},
    ]


def _log_uniform(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def _width(rng):
    """Model width: one of the configurations', or any multiple of 16 in their range."""
    if rng.random() < 0.5:
        return rng.choice([96, 192, 512, 768, 1024, 1280])
    return 16 * round(_log_uniform(rng, 96, 1280) / 16)


def _tokens(rng, h):
    """Tokens of a batch: whole images, or any count (images of mixed sizes, dropped tokens)."""
    per = rng.choice([49, 196, 197, 257, 3136])
    most = min(32 * 3136, _MAX_MH // h)
    m = _log_uniform(rng, 49, most)
    return int(m) if rng.random() < 0.4 else max(1, round(m / per)) * per if round(m / per) * per <= most else int(m)


def draw(rng):
    kind = rng.choices(["block", "layer", "patch", "weights"], [6, 3, 1, 2])[0]
    if kind == "weights":
        h = _width(rng)
        return {"kind": kind, "mode": rng.choice(["int8", "f16", "int4"]), "h": h, "mlp": 4 * h}
    if kind == "patch":
        p = rng.choice([4, 8, 14, 16])
        return {"kind": kind, "mode": rng.choice(["computed", "supplied"]), "b": int(_log_uniform(rng, 1, 129)),
                "side": p * rng.choice([112 // p, 224 // p, 384 // p]), "p": p, "n": _width(rng)}
    mode = rng.choices(["computed", "supplied", "absmax", "int4", "f16"], [4, 4, 2, 2, 3])[0]
    h = _width(rng)
    case = {"kind": kind, "mode": mode, "m": _tokens(rng, h), "h": h, "dist": rng.choice(["normal", "student_t4"])}
    if kind == "block":
        case["mlp"] = 4 * h
    else:
        if mode == "absmax":
            case["mode"] = "computed"
        case["n"] = _width(rng)
        case["gelu"] = rng.random() < 0.5
        case["out"] = "i8" if case["mode"] == "supplied" and rng.random() < 0.5 else "f16"
    return case


def _layers(case):
    """[(name, K, N, gelu)]"""
    h = case["h"]
    if case["kind"] == "layer":
        return [("layer", h, case["n"], case["gelu"])]
    return [("qkv", h, 3 * h, False), ("proj", h, h, False), ("fc1", h, case["mlp"], True),
            ("fc2", case["mlp"], h, False)]


# ---- inputs ----

def _normal(gen, *shape):
    return torch.randn(shape, generator=gen, device="cuda")


def _weight(gen, n, k):
    return _normal(gen, n, k).mul_(0.02)


def _activation(gen, m, k, dist):
    x = _normal(gen, m, k)
    if dist == "student_t4":
        # normal / sqrt(chi2_4 / 4) / sqrt(2); a chi-square of four degrees is -2 ln(u1 u2)
        u = torch.rand((m, k), generator=gen, device="cuda").mul_(torch.rand((m, k), generator=gen, device="cuda"))
        x.div_(u.clamp_min_(1e-12).log_().mul_(-1.0).sqrt_())
    return x.half()


def _make_weights(mode, W):
    """Packed operand and per-channel scale (None for the FP16 model) of one layer, and the stored form for int4."""
    if mode == "f16":
        vals, meta = B.compress24_f16(B.prune24(W))
        return B.pack24_f16(vals, meta), None, None
    if mode == "int4":
        Wq, w_scale = B.quant_weight4(B.prune48(W))
        stored = B.compress48(Wq)
        return B.pack24(*B.expand48(*stored)), w_scale, stored
    Wq, w_scale = B.quant_weight(B.prune24(W))
    return B.pack24(*B.compress24(Wq)), w_scale, None


def _scalar(v):
    return torch.full((1,), v, dtype=torch.float32, device="cuda")


def prepare(case, seed):
    gen = torch.Generator(device="cuda").manual_seed(seed)
    mode = case["mode"]
    st = {"kind": case["kind"], "mode": mode}
    if case["kind"] == "weights":
        st["W"] = [_weight(gen, n, k) for _, k, n, _ in _layers(case)]
        return st
    i8 = lambda m, k: torch.empty((m, k), dtype=torch.int8, device="cuda")  # noqa: E731
    if case["kind"] == "patch":
        b, side, p, n = case["b"], case["side"], case["p"], case["n"]
        mean = torch.tensor([0.485, 0.456, 0.406], device="cuda").view(1, 3, 1, 1)
        std = torch.tensor([0.229, 0.224, 0.225], device="cuda").view(1, 3, 1, 1)
        st["img"] = torch.rand((b, 3, side, side), generator=gen, device="cuda").sub_(mean).div_(std).half()
        Wf = B.flatten_conv_weight(_weight(gen, n, 3 * p * p).view(n, 3, p, p))
        st["Wp"], st["w_scale"], _ = _make_weights("int8", Wf)
        st["bias"] = _normal(gen, n).mul_(0.01)
        st["p"], st["n"] = p, n
        tokens, kp = b * (side // p) ** 2, Wf.shape[1]
        st["Xq"], st["Y"] = i8(tokens, kp), torch.empty((tokens, n), dtype=torch.float16, device="cuda")
        st["x_scale"] = _scalar(2.64 / 127)          # the whitest pixel, normalised
        st["workspace"] = torch.zeros(B.quant_act_workspace(tokens, kp), dtype=torch.uint8, device="cuda")
        st["status"] = torch.zeros(4, dtype=torch.int32, device="cuda")
        return st
    m = case["m"]
    st["layers"] = []
    for name, k, n, gelu in _layers(case):
        Wp, w_scale, _ = _make_weights(mode if mode in ("f16", "int4") else "int8", _weight(gen, n, k))
        L = {"name": name, "N": n, "act": B.ACT_GELU if gelu else B.ACT_NONE, "Wp": Wp, "w_scale": w_scale,
             "bias": _normal(gen, n).mul_(0.01), "status": torch.zeros(4, dtype=torch.int32, device="cuda"),
             "out_type": B.OUT_F16, "out_scale": None}
        L["X"] = None if name == "fc2" else _activation(gen, m, k, case["dist"])
        if mode == "supplied" and (name == "fc1" or case.get("out") == "i8"):
            # a calibrated output scale: what this layer's outputs reach (2:4 weights keep ~0.86 of sigma^2)
            sigma = 0.02 * math.sqrt(0.86 * k)
            L["out_type"], L["out_scale"] = B.OUT_I8, _scalar(4.5 * sigma / 127)
        if mode != "f16":
            L["Xq"] = None if mode == "supplied" and name == "fc2" else i8(m, k)
            # a learned scale clamps the tails of its tensor
            L["x_scale"] = _scalar((4.5 if case["dist"] == "normal" else 8.0) / 127)
            L["workspace"] = torch.zeros(B.quant_act_workspace(m, k), dtype=torch.uint8, device="cuda")
        L["Y"] = torch.empty((m, n), dtype=torch.int8 if L["out_type"] == B.OUT_I8 else torch.float16, device="cuda")
        if mode == "absmax" and name == "fc1":
            L["amax"] = _scalar(0.0)
        st["layers"].append(L)
    return st


# ---- one pass ----

def _run_weights(st):
    out = []
    for W in st["W"]:
        packed, w_scale, stored = _make_weights(st["mode"], W)
        out.append([t for t in (packed, w_scale, *(stored or ())) if t is not None])
    return out


def _run_patch(st):
    given = st["mode"] == "supplied"
    Xq, xs = B.patch_quant(st["img"], st["p"], Xq=st["Xq"], x_scale=st["x_scale"],
                           scale_mode=B.SCALE_GIVEN if given else B.SCALE_COMPUTE, workspace=st["workspace"])
    Y = B.spgemm_i8(Xq, st["Wp"], st["n"], st["w_scale"], xs, st["bias"], Y=st["Y"], status_buf=st["status"])
    return [Y, xs]


def run(st):
    if st["kind"] == "weights":
        return _run_weights(st)
    if st["kind"] == "patch":
        return _run_patch(st)
    mode, out, prev = st["mode"], [], None
    for L in st["layers"]:
        X = prev["Y"] if L["X"] is None else L["X"]
        if mode == "f16":
            out.append(B.spgemm_f16(X, L["Wp"], L["N"], L["bias"], L["act"], Y=L["Y"], status_buf=L["status"]))
            prev = L
            continue
        if X.dtype == torch.int8:                      # fc2 of the deployed model: fc1 wrote its codes
            Xq, xs = X, prev["out_scale"]
        elif mode == "supplied":
            Xq, xs = B.quant_act(X, L["Xq"], L["x_scale"], B.SCALE_GIVEN)
        elif mode == "int4":
            Xq, xs = B.quant_act4(X, L["Xq"], L["x_scale"], workspace=L["workspace"])
        elif mode == "absmax" and prev is not None and "amax" in prev:
            Xq, xs = B.quant_act_absmax(X, prev["amax"], L["Xq"], L["x_scale"])
        else:
            Xq, xs = B.quant_act(X, L["Xq"], L["x_scale"], workspace=L["workspace"])
        if "amax" in L:
            Y, _ = B.spgemm_i8_absmax(Xq, L["Wp"], L["N"], L["w_scale"], xs, L["bias"], L["act"], L["Y"],
                                      L["amax"].zero_(), L["status"])
        else:
            Y = B.spgemm_i8(Xq, L["Wp"], L["N"], L["w_scale"], xs, L["bias"], L["act"], L["out_type"],
                            L["out_scale"], L["Y"], L["status"])
        out += [Y] if xs is L.get("out_scale") or mode == "supplied" else [Y, xs]
        prev = L
    return out


# ---- what a pass cannot do without ----

def work(case):
    mode = case["mode"]
    if case["kind"] == "weights":
        # FP32 in; packed operand and scale out (stored 4-bit form as well)
        per = {"int8": 4 + 0.625, "f16": 4 + 1.125, "int4": 4 + 0.3125 + 0.625}[mode]
        return {"bytes": sum(per * n * k + 4 * n for _, k, n, _ in _layers(case)), "flops": 0}
    if case["kind"] == "patch":
        tokens, k, n = case["b"] * (case["side"] // case["p"]) ** 2, 3 * case["p"] ** 2, case["n"]
        return {"bytes": 2 * tokens * k + 0.625 * n * k + 8 * n + 2 * tokens * n, "flops": tokens * n * k}
    m, bytes_, flops = case["m"], 0, 0
    for name, k, n, _ in _layers(case):
        one_byte_out = mode == "supplied" and (name == "fc1" or case.get("out") == "i8")
        bytes_ += (0 if name == "fc2" else 2 * m * k) + m * n * (1 if one_byte_out else 2)
        bytes_ += (1.125 if mode == "f16" else 0.625) * n * k + 8 * n
        flops += m * n * k                             # two of every four weights: half of 2 m n k
    return {"bytes": bytes_, "flops": flops}


def tolerance(case):
    if case["kind"] == "weights":
        return "exact"                                 # codes, positions, scales: integers and single IEEE operations
    # Against the same layers in binary64: binary16 outputs are 2.1e-4 of the 2-norm off (their rounding), at
    # most 5e-4 in one value, more (5e-3) where a code of fc2's input lies on a rounding tie; INT8 outputs
    # behind a GELU differ in 1.5e-5 of the codes, which lie on such ties.
    return {"rel": 8e-4, "max": 1e-2, "differ": 1e-4}

"""The work whose speed is measured: DN forwards and the layers they are made of.

Every case goes through the public entry points of the Python binding
(`ElasticModel.forward` and the `elasto_op_*` calls). Sizes are those of the
workloads in `paper_2609_10018_gb300.synth`: elastic ViT-B/16, ViT-S/16 and the
tiny fp32 ViT, and the elastic ResNet-50, in their full and pruned modes, at
serving batches from one image to the largest.

Kinds of case (the "kind" entry):
  vit, resnet   one whole forward of one mode, logits returned;
  gemm          one projection / 1x1 convolution with its fused epilogue;
  attention     multi-head attention over the kept heads of one layer;
  conv          one k x k convolution over the kept channels.
"""
import math

import numpy as np
import torch
import torch.nn.functional as F

from paper_2609_10018_gb300 import binding, synth

DEVICE = "cuda"

# gemm "role" -> (epilogue, 16-bit operand type)
ROLES = {
    "bias": (binding.EPI_BIAS_BF16, torch.bfloat16),                    # QKV projection
    "gelu": (binding.EPI_BIAS_GELU_BF16, torch.bfloat16),               # FC1
    "residual": (binding.EPI_BIAS_RESID_F32, torch.bfloat16),           # out-projection, FC2: x += ...
    "relu_f16": (binding.EPI_BIAS_RELU_F16, torch.float16),             # 1x1 conv + folded BN
    "shortcut_f16": (binding.EPI_BIAS_F16, torch.float16),              # shortcut projection
    "block_out_f16": (binding.EPI_BIAS_RESID_RELU_F16, torch.float16),  # last 1x1 conv of a block
}


def listed():
    return [
        # offline / throughput serving: the full ViT-B/16 mode at its largest batch
        {"name": "vit_b_256", "kind": "vit", "model": "vit_b16", "mode": 0, "batch": 256},
        # interactive serving: one image, the paper's latency protocol
        {"name": "vit_b_1", "kind": "vit", "model": "vit_b16", "mode": 0, "batch": 1},
        # fp32-stored weights and images, a few small images
        {"name": "vit_tiny_8", "kind": "vit", "model": "tiny", "mode": 0, "batch": 8},
        # the CNN: ResNet-50 at its throughput batch
        {"name": "resnet50_128", "kind": "resnet", "mode": 0, "batch": 128},
        # QKV projection of the largest batch (256 x 197 tokens, 12 heads)
        {"name": "qkv_256", "kind": "gemm", "role": "bias", "M": 50432, "N": 2304, "K": 768},
        # MLP up-projection + GELU at a middling batch (32 x 197 tokens)
        {"name": "fc1_32", "kind": "gemm", "role": "gelu", "M": 6304, "N": 3072, "K": 768},
        # MLP down-projection of the 50 % mode into the fp32 residual stream
        {"name": "fc2_half_256", "kind": "gemm", "role": "residual", "M": 50432, "N": 768, "K": 1536},
        # last 1x1 convolution of a stage-1 block with its shortcut, 128 images of 56 x 56
        {"name": "conv3_stage1_128", "kind": "gemm", "role": "block_out_f16", "M": 401408, "N": 256, "K": 64},
        # attention of one ViT-B layer at the largest batch
        {"name": "attention_256", "kind": "attention", "batch": 256, "tokens": 197, "heads": 12},
        # the smallest call: attention of the tiny ViT's pruned mode
        {"name": "attention_tiny", "kind": "attention", "batch": 8, "tokens": 65, "heads": 2},
        # 3x3 convolution of stage 1, all 64 channels, 128 images of 56 x 56
        {"name": "conv2_stage1_128", "kind": "conv", "batch": 128, "size": 56, "C": 64, "N": 64, "k": 3, "stride": 1},
        # strided 3x3 convolution into stage 3 of the 75 % mode, a ragged serving batch
        {"name": "conv2_stage3_100", "kind": "conv", "batch": 100, "size": 28, "C": 192, "N": 192, "k": 3, "stride": 2},
    ]


def _log_uniform(rng, lo, hi):
    return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(["vit", "resnet", "gemm", "gemm", "attention", "conv"])
    if kind == "vit":
        model = rng.choice(["vit_b16", "vit_s16", "tiny"])
        return {"kind": kind, "model": model, "mode": rng.randrange(synth.VIT_CONFIGS[model].n_modes),
                "batch": _log_uniform(rng, 1, 256)}
    if kind == "resnet":
        return {"kind": kind, "mode": rng.randrange(synth.RESNET50.n_modes), "batch": _log_uniform(rng, 1, 128)}
    if kind == "attention":
        return {"kind": kind, "batch": _log_uniform(rng, 1, 256), "tokens": rng.randrange(17, 257),
                "heads": rng.randrange(1, 13)}
    if kind == "conv":
        size = rng.choice([7, 13, 14, 28, 31, 56])
        width = {7: 512, 13: 256, 14: 256, 28: 128, 31: 128, 56: 64}[size]
        channels = [c for c in range(8, width + 1, 8)]
        k = rng.choice([1, 3, 3])
        return {"kind": kind, "batch": _log_uniform(rng, 1, 128), "size": size, "C": rng.choice(channels),
                "N": rng.choice(channels), "k": k, "stride": rng.choice([1, 1, 2])}
    role = rng.choice(sorted(ROLES))
    if role.endswith("f16"):  # images x pixels of a stage, kept widths of its blocks
        side, wide = rng.choice([(56, 256), (28, 512), (14, 1024), (7, 2048)])
        m = _log_uniform(rng, 1, 128) * side * side
        inner = 8 * rng.randrange(1, wide // 32 + 1)
        n, k = (inner, wide) if role == "relu_f16" else (wide, inner)
        return {"kind": kind, "role": role, "M": m, "N": n, "K": k}
    m, dim = _log_uniform(rng, 197, 50432), rng.choice([192, 384, 768])
    inner = 8 * rng.randrange(8, dim // 2 + 1)
    n, k = (dim, inner) if role == "residual" else (inner, dim)
    return {"kind": kind, "role": role, "M": m, "N": n, "K": k}


# ---------------------------------------------------------------- inputs

def _generator(seed):
    return torch.Generator(device=DEVICE).manual_seed(int(seed))


def _normal(shape, g, std=1.0):
    return torch.randn(shape, generator=g, device=DEVICE) * std


def _vit_config(case):
    return synth.VIT_CONFIGS[case["model"]]


def _vit_weights(cfg, g):
    """N(0, 0.02) tensors and LayerNorm gains around 1, in the model's storage type, on the GPU."""
    out = {}
    for name, shape in synth.vit_weight_shapes(cfg).items():
        w = _normal(shape, g, 0.02)
        if name.endswith(("ln1_w", "ln2_w")) or name == "norm_w":
            w += 1.0
        out[name] = w if cfg.dtype == synth.F32 else w.bfloat16()
    return out


def _resnet_weights(cfg, g):
    """He-normal convolutions; BN statistics as a trained network's: small gains on each block's last BN."""
    def uniform(shape, lo, hi):
        return torch.rand(shape, generator=g, device=DEVICE) * (hi - lo) + lo

    out = {}
    for name, shape in synth.resnet_weight_shapes(cfg).items():
        if name.endswith("_w") and len(shape) == 4:
            w = _normal(shape, g, math.sqrt(2.0 / (shape[1] * shape[2] * shape[3])))
        elif name in ("fc_w", "fc_b"):
            w = _normal(shape, g, 0.01)
        elif name.endswith(".g"):
            w = uniform(shape, 0.1, 0.3) if ".bn3." in name else uniform(shape, 0.5, 1.0)
        elif name.endswith(".b"):
            w = _normal(shape, g, 0.05)
        elif name.endswith(".mean"):
            w = _normal(shape, g, 0.1)
        else:
            w = uniform(shape, 0.5, 1.5)
        out[name] = w.bfloat16()
    return out


def _host(w):
    """Host arrays as the library takes them: fp32, or bf16 bit patterns."""
    return {k: (v.cpu().numpy() if v.dtype == torch.float32 else v.view(torch.int16).cpu().numpy().view(np.uint16))
            for k, v in w.items()}


def _model_inputs(case, seed):
    """(config, weights on the GPU, kept tables of all modes, images [B, H, W, C])."""
    g = _generator(seed)
    vit = case["kind"] == "vit"
    cfg = _vit_config(case) if vit else synth.RESNET50
    weights = _vit_weights(cfg, g) if vit else _resnet_weights(cfg, g)
    tables = synth.make_vit_tables(cfg) if vit else synth.make_resnet_tables(cfg)
    images = torch.rand((case["batch"], cfg.img, cfg.img, cfg.chans), generator=g, device=DEVICE)
    return cfg, weights, tables, images if cfg.dtype == synth.F32 else images.bfloat16()


def _layer_inputs(case, seed):
    """The tensors of one layer's call, in the layout that its entry point takes."""
    g = _generator(seed)
    if case["kind"] == "attention":
        # q, k, v of normalised tokens through N(0, 0.02) projections of 64-wide heads
        std = 0.02 * math.sqrt(768)
        return {"qkv": _normal((case["batch"], case["tokens"], 3, case["heads"], 64), g, std).bfloat16()}
    if case["kind"] == "conv":
        b, s, c, n, k = case["batch"], case["size"], case["C"], case["N"], case["k"]
        x = _normal((b, s, s, c), g).relu_().half()  # a ReLU came before
        w = _normal((n, k, k, c), g, math.sqrt(2.0 / (c * k * k))).half()
        return {"x": x, "w": w, "bias": _normal((n,), g, 0.05)}
    m, n, k = case["M"], case["N"], case["K"]
    dtype = ROLES[case["role"]][1]
    a = _normal((m, k), g)
    t = {"bias": _normal((n,), g, 0.05)}
    if dtype == torch.float16:
        a.relu_()
        t["w"] = _normal((n, k), g, math.sqrt(2.0 / k)).half()
    else:
        t["w"] = _normal((n, k), g, 0.02).bfloat16()
    t["a"] = a.to(dtype)
    if case["role"] == "residual":
        t["x"] = _normal((m, n), g)
    elif case["role"] == "block_out_f16":
        t["resid"] = _normal((m, n), g).relu_().half()
    return t


def _packed_filter(w, c):
    """[N, k, k, C] -> the packed layout of elasto_op_conv2d (channels padded to 16, or to a multiple of 64)."""
    cp = 16 if c <= 16 else (c + 63) // 64 * 64
    return F.pad(w, (0, cp - c)).contiguous()


def _conv_out(case):
    return (case["size"] + 2 * (case["k"] // 2) - case["k"]) // case["stride"] + 1


def prepare(case, seed):
    state = {"case": case}
    if case["kind"] in ("vit", "resnet"):
        cfg, weights, tables, images = _model_inputs(case, seed)
        make = binding.ElasticModel.vit if case["kind"] == "vit" else binding.ElasticModel.resnet
        state["model"] = make(cfg, _host(weights), tables, max_batch=case["batch"])
        state["model"].set_mode(case["mode"])
        state["images"] = images
        state["logits"] = torch.empty((case["batch"], cfg.classes), device=DEVICE)
        return state
    state.update(_layer_inputs(case, seed))
    if case["kind"] == "attention":
        state["out"] = torch.empty((case["batch"], case["tokens"], case["heads"] * 64), dtype=torch.bfloat16,
                                   device=DEVICE)
    elif case["kind"] == "conv":
        state["w"] = _packed_filter(state["w"], case["C"])
        o = _conv_out(case)
        state["out"] = torch.empty((case["batch"], o, o, case["N"]), dtype=torch.float16, device=DEVICE)
    elif case["role"] == "residual":
        state["out"] = state.pop("x")  # updated in place, as the residual stream is
    else:
        state["out"] = torch.empty((case["M"], case["N"]), dtype=ROLES[case["role"]][1], device=DEVICE)
    return state


def run(state):
    case = state["case"]
    stream = torch.cuda.current_stream().cuda_stream
    if case["kind"] in ("vit", "resnet"):
        logits = state["logits"]
        state["model"].forward(stream, state["images"].data_ptr(), case["batch"], logits.data_ptr())
        return logits
    out = state["out"]
    if case["kind"] == "attention":
        binding.elasto_op_attention(stream, state["qkv"].data_ptr(), out.data_ptr(), case["batch"], case["tokens"],
                                    case["heads"])
    elif case["kind"] == "conv":
        binding.elasto_op_conv2d(stream, state["x"].data_ptr(), case["batch"], case["size"], case["size"], case["C"],
                                 state["w"].data_ptr(), case["N"], case["k"], case["stride"], case["k"] // 2,
                                 state["bias"].data_ptr(), 1, out.data_ptr())
    else:
        resid = state.get("resid")
        binding.elasto_op_gemm(stream, state["a"].data_ptr(), state["w"].data_ptr(), state["bias"].data_ptr(),
                               out.data_ptr(), None if resid is None else resid.data_ptr(), case["M"], case["N"],
                               case["K"], ROLES[case["role"]][0])
    return out


# ---------------------------------------------------------------- work

def _vit_macs(cfg, mode):
    n, d, w, f = cfg.tokens, cfg.dim, 64 * cfg.mode_heads[mode], cfg.mode_mlp[mode]
    layer = n * d * 3 * w + 2 * n * n * w + n * w * d + 2 * n * d * f
    return cfg.n_patches * d * cfg.patch ** 2 * cfg.chans + cfg.layers * layer + d * cfg.classes


def _vit_weight_values(cfg, mode):
    d, w, f = cfg.dim, 64 * cfg.mode_heads[mode], cfg.mode_mlp[mode]
    return d * cfg.patch ** 2 * cfg.chans + cfg.layers * (4 * d * w + 2 * d * f) + d * cfg.classes


def _resnet_layers(cfg, mode):
    """(output pixels, multiply-adds per pixel, weight values) of every convolution and the classifier."""
    frac = cfg.mode_frac[mode]
    half = lambda s: (s - 1) // 2 + 1  # noqa: E731
    size = half(cfg.img)
    layers = [(size * size, 64 * 147, 64 * 147)]
    size = half(size)
    for cin, width, stride, down in synth.resnet_blocks(cfg):
        kept = int(round(width * frac))
        out = half(size) if stride == 2 else size
        layers += [(size * size, kept * cin, kept * cin), (out * out, 9 * kept * kept, 9 * kept * kept),
                   (out * out, 4 * width * kept, 4 * width * kept)]
        if down:
            layers.append((out * out, 4 * width * cin, 4 * width * cin))
        size = out
    return layers + [(1, 2048 * cfg.classes, 2048 * cfg.classes)]


def work(case):
    kind = case["kind"]
    if kind in ("vit", "resnet"):
        cfg = _vit_config(case) if kind == "vit" else synth.RESNET50
        if kind == "vit":
            macs, values = _vit_macs(cfg, case["mode"]), _vit_weight_values(cfg, case["mode"])
        else:
            layers = _resnet_layers(cfg, case["mode"])
            macs, values = sum(p * m for p, m, _ in layers), sum(v for _, _, v in layers)
        size = 4 if cfg.dtype == synth.F32 else 2
        return {"bytes": size * (values + case["batch"] * cfg.img ** 2 * cfg.chans) + 4 * case["batch"] * cfg.classes,
                "flops": 2 * macs * case["batch"]}
    if kind == "attention":
        b, n, h = case["batch"], case["tokens"], case["heads"]
        return {"bytes": 2 * 4 * b * n * h * 64, "flops": 4 * b * h * n * n * 64}
    if kind == "conv":
        o, taps = _conv_out(case), case["k"] ** 2 * case["C"] * case["N"]
        pixels = case["batch"] * o * o
        return {"bytes": 2 * (case["batch"] * case["size"] ** 2 * case["C"] + taps + pixels * case["N"]),
                "flops": 2 * pixels * taps}
    m, n, k = case["M"], case["N"], case["K"]
    out = {"residual": 8, "block_out_f16": 4}.get(case["role"], 2)  # bytes per output value, the residual's read among them
    return {"bytes": 2 * (m * k + n * k) + out * m * n, "flops": 2 * m * n * k}


def tolerance(case):
    """About four times the measured distance from 64 bits: one rounding of the
    output to its type, and what the layers before a whole model's logits add."""
    if case["kind"] == "vit":
        return {"rel": 0.015, "max": 0.1}  # measured 2.3e-3 to 3.2e-3
    if case["kind"] == "resnet":
        return {"rel": 0.002, "max": 0.01}  # measured 3.4e-4
    if case["kind"] == "attention":
        return {"rel": 0.01, "max": 0.05}  # measured 2.3e-3
    if case["kind"] == "conv" or ROLES[case["role"]][1] == torch.float16:
        return {"rel": 1e-3, "max": 4e-3}  # measured 2.1e-4
    if case["role"] == "residual":
        return {"rel": 1e-5, "max": 1e-4}  # 32-bit sums, measured 1e-6
    return {"rel": 7e-3, "max": 0.04}  # measured 1.7e-3


# ---------------------------------------------------------------- 64 bits

def _exact_vit(cfg, w, table, images):
    w = {k: v.double() for k, v in w.items()}
    b, p, d, g = images.shape[0], cfg.patch, cfg.dim, cfg.img // cfg.patch
    norm = lambda x, s: F.layer_norm(x, (d,), w[s + "_w"], w[s + "_b"], 1e-6)  # noqa: E731
    patches = images.double().view(b, g, p, g, p, cfg.chans).permute(0, 1, 3, 5, 2, 4).reshape(b, g * g, -1)
    x = patches @ w["patch_w"].reshape(d, -1).T + w["patch_b"]
    x = torch.cat([w["cls"].expand(b, 1, d), x], 1) + w["pos"]
    n = x.shape[1]
    for l in range(cfg.layers):
        heads = torch.from_numpy(np.asarray(table["heads"][l], np.int64)).to(DEVICE)
        mlp = torch.from_numpy(np.asarray(table["mlp"][l], np.int64)).to(DEVICE)
        rows = (heads[:, None] * 64 + torch.arange(64, device=DEVICE)).reshape(-1)
        y = norm(x, f"l{l}.ln1")
        q, k, v = ((y @ w[f"l{l}.qkv_w"][i * d + rows].T + w[f"l{l}.qkv_b"][i * d + rows])
                   .view(b, n, -1, 64).transpose(1, 2) for i in range(3))
        o = ((q @ k.transpose(2, 3)) / 8.0).softmax(-1) @ v
        x = x + o.transpose(1, 2).reshape(b, n, -1) @ w[f"l{l}.proj_w"][:, rows].T + w[f"l{l}.proj_b"]
        y = norm(x, f"l{l}.ln2")
        h = F.gelu(y @ w[f"l{l}.fc1_w"][mlp].T + w[f"l{l}.fc1_b"][mlp])
        x = x + h @ w[f"l{l}.fc2_w"][:, mlp].T + w[f"l{l}.fc2_b"]
    return norm(x[:, 0], "norm") @ w["head_w"].T + w["head_b"]


def _exact_conv(x, w, stride, pad):
    """x [B, H, W, C], w [N, k, k, C] in 64 bits -> [B, Ho, Wo, N], a matrix product per tap."""
    k, ho = w.shape[1], (x.shape[1] + 2 * pad - w.shape[1]) // stride + 1
    wo = (x.shape[2] + 2 * pad - k) // stride + 1
    x = F.pad(x, (0, 0, pad, pad, pad, pad))
    out = 0
    for ky in range(k):
        for kx in range(k):
            out = out + x[:, ky:ky + stride * (ho - 1) + 1:stride, kx:kx + stride * (wo - 1) + 1:stride] @ w[:, ky, kx].T
    return out


def _exact_resnet(cfg, w, table, images):
    w = {k: v.double() for k, v in w.items()}

    def conv_bn(x, conv, bn, stride, pad, rows=None, cols=None):
        f = w[conv].permute(0, 2, 3, 1)
        scale = w[bn + ".g"] / torch.sqrt(w[bn + ".var"] + 1e-5)
        shift = w[bn + ".b"] - w[bn + ".mean"] * scale
        if rows is not None:
            f, scale, shift = f[rows], scale[rows], shift[rows]
        if cols is not None:
            f = f[..., cols]
        return _exact_conv(x, f, stride, pad) * scale + shift

    x = conv_bn(images.double(), "stem_w", "stem_bn", 2, 3).relu()
    x = F.max_pool2d(x.permute(0, 3, 1, 2), 3, 2, 1).permute(0, 2, 3, 1)
    for i, (_, _, stride, down) in enumerate(synth.resnet_blocks(cfg)):
        a, b = (torch.from_numpy(np.asarray(table[s][i], np.int64)).to(DEVICE) for s in "ab")
        y = conv_bn(x, f"b{i}.conv1_w", f"b{i}.bn1", 1, 0, a).relu()
        y = conv_bn(y, f"b{i}.conv2_w", f"b{i}.bn2", stride, 1, b, a).relu()
        y = conv_bn(y, f"b{i}.conv3_w", f"b{i}.bn3", 1, 0, None, b)
        x = (y + (conv_bn(x, f"b{i}.down_w", f"b{i}.down_bn", stride, 0) if down else x)).relu()
    return x.mean((1, 2)) @ w["fc_w"].T + w["fc_b"]


def exact(case, seed):
    if case["kind"] in ("vit", "resnet"):
        cfg, w, tables, images = _model_inputs(case, seed)
        forward = _exact_vit if case["kind"] == "vit" else _exact_resnet
        return torch.cat([forward(cfg, w, tables[case["mode"]], part) for part in images.split(64)])
    t = {k: v.double() for k, v in _layer_inputs(case, seed).items()}
    if case["kind"] == "attention":
        q, k, v = (t["qkv"][:, :, i].transpose(1, 2) for i in range(3))
        o = ((q @ k.transpose(2, 3)) / 8.0).softmax(-1) @ v
        return o.transpose(1, 2).reshape(case["batch"], case["tokens"], -1)
    if case["kind"] == "conv":
        return (_exact_conv(t["x"], t["w"], case["stride"], case["k"] // 2) + t["bias"]).relu()
    y = t["a"] @ t["w"].T + t["bias"]
    if case["role"] == "gelu":
        return F.gelu(y)
    if case["role"] == "residual":
        return t["x"] + y
    if case["role"] == "block_out_f16":
        return (y + t["resid"]).relu()
    return y.relu() if case["role"] == "relu_f16" else y

"""The work that users have this library do, as cases that can be timed and compared.

Every case is one call of a public entry point the way an inference program makes it: the attention block of the C ABI,
an encoder layer, a stack of layers, the attention module of the paper's power table, a whole DeiT-shaped model, and a
single integer linear.  The library is forward-only, so there is no backward direction.  Sizes are those of the
repository's configurations, tests and benchmark sweep (ViT-Tiny / Small / Base widths, DeiT-S, 197 / 198 / 577 / 785
tokens), or generic ragged ones.

A program has its weights quantized and its buffers laid out before it sees an input, so prepare() builds the layer (or
module, or model) and the fp32 input of the case; run() is one forward pass.  Values follow the distributions of the
repository's synthetic inputs: N(0, 1) activations (with 1 % outlier channels where a case says so), N(0, 0.02) weights,
N(0, 0.01) biases, LSQ step sizes 2 mean|x| / sqrt(Qp).
"""
import math

import numpy as np
import torch

import paper_2504_18547_b200 as vt
from paper_2504_18547_b200.encoder import DeitModel, EncoderLayer, EncoderStack, NormedAttention

W_STD = 0.02
PATCH_DIM = 16 * 16 * 3


def listed():
    return [
        # one image through a ViT-Tiny attention block: the smallest call a latency-bound user makes (bit-packed codes)
        {"name": "tiny_block_b1", "kind": "block", "batch": 1, "tokens": 197, "heads": 3, "bits": 4, "outliers": False},
        # a ViT-Small attention block at a usual batch, with outlier channels, codes bit-packed throughout
        {"name": "small_block_b64", "kind": "block", "batch": 64, "tokens": 197, "heads": 6, "bits": 4, "outliers": True},
        # twelve ViT-Base layers for one image: interactive classification, where launches and host time count
        {"name": "base_encoder12_b1", "kind": "encoder", "batch": 1, "tokens": 197, "heads": 12, "mlp": 3072, "bits": 4,
         "layers": 12},
        # a ViT-Base layer at a small serving batch, 3-bit codes
        {"name": "base_layer_3bit_b8", "kind": "layer", "batch": 8, "tokens": 197, "heads": 12, "mlp": 3072, "bits": 3,
         "softmax": "exp", "layernorm": "fp32", "wide": True},
        # the benchmark's workload: a ViT-Base layer at batch 128, 4-bit codes
        {"name": "base_layer_b128", "kind": "layer", "batch": 128, "tokens": 197, "heads": 12, "mlp": 3072, "bits": 4,
         "softmax": "exp", "layernorm": "fp32", "wide": True},
        # the same layer with the paper's own quantizers throughout (Eq. 4 softmax, Eq. 5 LayerNorm), offline evaluation
        {"name": "paper_layer_b64", "kind": "layer", "batch": 64, "tokens": 197, "heads": 12, "mlp": 3072, "bits": 4,
         "softmax": "shift", "layernorm": "compare", "wide": True},
        # 8-bit codes: the width a deployment starts from before it goes lower
        {"name": "base_layer_8bit_b32", "kind": "layer", "batch": 32, "tokens": 197, "heads": 12, "mlp": 3072, "bits": 8,
         "softmax": "exp", "layernorm": "fp32", "wide": True},
        # high-resolution input: 28 x 28 patches and a class token
        {"name": "base_layer_t785_b16", "kind": "layer", "batch": 16, "tokens": 785, "heads": 12, "mlp": 3072, "bits": 4,
         "softmax": "exp", "layernorm": "fp32", "wide": True},
        # ragged everywhere: odd batch and tokens, five heads, an MLP width that is no multiple of a tile, 2-bit codes
        {"name": "ragged_layer_2bit_b7", "kind": "layer", "batch": 7, "tokens": 145, "heads": 5, "mlp": 1290, "bits": 2,
         "softmax": "exp", "layernorm": "fp32", "wide": True},
        # the self-attention module of the paper's power table at DeiT-S width, 3-bit
        {"name": "deit_s_attention_b64", "kind": "normed", "batch": 64, "tokens": 198, "heads": 6, "bits": 3},
        # the whole DeiT-S-shaped model the paper evaluates: patches in, logits out
        {"name": "deit_s_model_b128", "kind": "model", "batch": 128, "tokens": 198, "heads": 6, "mlp": 1536, "bits": 4,
         "layers": 12},
        # one integer linear on bit-packed codes (quantize, then the requantizing contraction), the MLP's first shape
        {"name": "linear_packed_3072", "kind": "linear", "rows": 64 * 197, "k": 768, "n": 3072, "bits": 4, "wide": False,
         "epi": "requant"},
    ]


def _cost(c):
    """A rough measure of a case's time, to keep drawn cases no dearer than the largest listed one."""
    w = work(c)
    slow = 4.0 if c.get("layernorm") == "compare" or c.get("softmax") == "shift" or c["bits"] == 8 or c.get("wide") is False else 1.0
    if c["kind"] == "normed" or c.get("tokens", 0) > 256:
        slow = max(slow, 4.0)
    return slow * (w["bytes"] / 3e12 + w["flops"] / 1e15)


def draw(rng):
    def log_int(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    limit = max(_cost(c) for c in listed())
    while True:
        kind = rng.choice(("block", "layer", "layer", "layer", "encoder", "normed", "linear", "model"))
        bits = rng.choice((2, 3, 4, 4))
        heads = rng.randint(1, 16)
        if kind == "linear":
            c = {"kind": kind, "rows": log_int(1, 50432), "k": 16 * log_int(4, 256), "n": log_int(10, 4096), "bits": rng.choice((2, 3, 4, 8)),
                 "wide": rng.random() < 0.6, "epi": rng.choice(("requant", "dequant", "gelu", "acc"))}
        elif kind == "block":
            c = {"kind": kind, "batch": log_int(1, 128), "tokens": log_int(17, 400), "heads": heads, "bits": bits,
                 "outliers": rng.random() < 0.3}
        elif kind == "normed":
            c = {"kind": kind, "batch": log_int(1, 128), "tokens": log_int(17, 400), "heads": heads, "bits": rng.choice((2, 3, 4))}
        elif kind == "encoder":
            c = {"kind": kind, "batch": log_int(1, 64), "tokens": log_int(33, 256), "heads": heads, "mlp": 256 * heads,
                 "bits": bits, "layers": rng.randint(2, 12)}
        elif kind == "model":
            c = {"kind": kind, "batch": log_int(1, 128), "tokens": log_int(50, 256), "heads": heads, "mlp": 256 * heads,
                 "bits": bits, "layers": rng.randint(2, 12)}
        else:
            option = rng.choice(("plain", "plain", "plain", "long", "paper", "bits8", "packed"))
            c = {"kind": kind, "batch": log_int(1, 256), "tokens": log_int(17, 256), "heads": heads,
                 "mlp": rng.choice((256 * heads, 256 * heads, 2 * rng.randint(60, 2000))), "bits": bits, "softmax": "exp",
                 "layernorm": "fp32", "wide": True}
            if option == "long":
                c.update(tokens=rng.randint(257, 1024))
            elif option == "paper":
                c.update(softmax="shift", layernorm="compare")
            elif option == "bits8":
                c.update(bits=8)
            elif option == "packed":
                c.update(wide=False)
        if _cost(c) <= limit:
            return c


# ---- inputs -------------------------------------------------------------------------------------------------------


def _gen(seed, tag):
    g = torch.Generator(device="cuda")
    g.manual_seed(1_000_003 * int(seed) + tag)
    return g


def _normal(g, shape, mean, std):
    return torch.randn(shape, generator=g, device="cuda", dtype=torch.float32).mul_(std).add_(mean)


def _qp(bits, signed):
    return (1 << (bits - 1)) - 1 if signed else (1 << bits) - 1


def _gauss_step(sigma, bits, signed=True):
    return np.float32(2.0 * sigma * math.sqrt(2.0 / math.pi) / math.sqrt(_qp(bits, signed)))


def _row_steps(w, bits):
    return (2.0 / math.sqrt(_qp(bits, True)) * w.double().abs().mean(dim=1)).clamp_min_(1e-8).float()


def _host(t):
    return t.cpu().numpy()


def _layer_params(g, dim, mlp, bits, tokens, x_rms=1.0):
    """Weights, biases and step sizes of one block as host arrays, the form the layer classes take."""
    p = {}

    def linear(name, n, k):
        w = _normal(g, (n, k), 0.0, W_STD)
        p["w_" + name], p["s_w_" + name], p["b_" + name] = _host(w), _host(_row_steps(w, bits)), _host(_normal(g, (n,), 0.0, 0.01))

    linear("qkv", 3 * dim, dim)
    linear("proj", dim, dim)
    sigma = W_STD * math.sqrt(dim) * x_rms
    p["s_x"] = _gauss_step(x_rms, bits)
    p["s_q"] = p["s_k"] = p["s_v"] = _gauss_step(sigma, bits)
    p["s_p"] = np.float32(2.0 / (tokens * math.sqrt(_qp(bits, False))))
    p["s_o"] = _gauss_step(1.2 * sigma / math.sqrt(tokens) + 0.01, bits)
    if mlp:
        for n in ("ln1", "ln2"):
            p[n + "_g"], p[n + "_b"] = _host(_normal(g, (dim,), 1.0, 0.02)), _host(_normal(g, (dim,), 0.0, 0.02))
        linear("fc1", mlp, dim)
        linear("fc2", dim, mlp)
        p["s_ln"] = _gauss_step(1.0, bits)
        y = _normal(g, (65536,), 0.0, W_STD * math.sqrt(dim)).double()
        p["s_g"] = np.float32(2.0 * float(torch.nn.functional.gelu(y).abs().mean()) / math.sqrt(_qp(bits, False)))
    return p


def _activations(g, rows, dim, outliers=False):
    x = _normal(g, (rows, dim), 0.0, 1.0)
    if outliers:
        x[:, torch.randperm(dim, generator=g, device="cuda")[: math.ceil(0.01 * dim)]] *= 10.0
    return x


def _model_ends(g, dim, bits, tokens, classes=10):
    p = {"tokens": _host(_normal(g, (tokens, dim), 0.0, 0.02)), "lnf_g": _host(_normal(g, (dim,), 1.0, 0.02)),
         "lnf_b": _host(_normal(g, (dim,), 0.0, 0.02)), "s_patch": _gauss_step(1.0, bits), "s_lnf": _gauss_step(1.0, bits)}
    for name, n, k in (("pe", dim, PATCH_DIM), ("head", classes, dim), ("head_dist", classes, dim)):
        w = _normal(g, (n, k), 0.0, W_STD)
        p["w_" + name], p["s_w_" + name], p["b_" + name] = _host(w), _host(_row_steps(w, bits)), _host(_normal(g, (n,), 0.0, 0.01))
    return p


# ---- the interface ------------------------------------------------------------------------------------------------


def prepare(case, seed):
    c, g = case, _gen(seed, 1)
    kind, bits = c["kind"], c["bits"]
    s = {"kind": kind, "bits": bits}
    if kind == "linear":
        m, k, n, wide = c["rows"], c["k"], c["n"], c["wide"]
        w = _normal(g, (n, k), 0.0, W_STD)
        steps = _row_steps(w, bits)
        codes = vt.vitint_quantize(w, 0.0, bits, True, row_steps=steps)
        s["w"] = vt.vitint_widen(codes) if wide and bits != 8 else codes
        s["x"], s["step"] = _activations(g, m, k), float(_gauss_step(1.0, bits))
        box = 8 if wide and bits != 8 else 0
        s["xq"] = vt.Codes.empty(m, k, bits, True, container=box)
        bias = _normal(g, (n,), 0.0, 0.01)
        s["w_step"], s["bias"] = steps, bias
        if c["epi"] == "requant":
            out_step = float(_gauss_step(W_STD * math.sqrt(k), bits))
            alpha, beta = vt.fold_requant(s["step"], _host(steps), _host(bias), np.float32(out_step))
            s["epi"] = vt.Epilogue(mode=vt.EPI_REQUANT, alpha=torch.from_numpy(alpha).cuda(), beta=torch.from_numpy(beta).cuda(),
                                   out_bits=bits, out_signed=True, out_container=box)
        elif c["epi"] == "gelu":
            inv = torch.full((n,), 1.0 / float(_gauss_step(0.6 * W_STD * math.sqrt(k), bits, False)), device="cuda")
            s["epi"] = vt.Epilogue(mode=vt.EPI_REQUANT, act=1, inv_out_step=inv, out_bits=bits, out_signed=False, out_container=box)
        elif c["epi"] == "dequant":
            s["epi"] = vt.Epilogue(mode=vt.EPI_DEQUANT_F32)
        else:
            s["epi"] = vt.Epilogue(mode=vt.EPI_ACC_I32)
        if c["epi"] in ("requant", "gelu"):
            s["out"] = vt.Codes.empty(m, n, bits, c["epi"] == "requant", container=box)
        else:
            s["out"] = torch.empty((m, n), dtype=torch.float32 if c["epi"] == "dequant" else torch.int32, device="cuda")
        return s
    dim, tokens = 64 * c["heads"], c["tokens"]
    rows = c["batch"] * tokens
    if kind == "block":
        rms = math.sqrt(1.0 + 99.0 * math.ceil(0.01 * dim) / dim) if c["outliers"] else 1.0
        p = _layer_params(g, dim, 0, bits, tokens, rms)
        dev = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()
        seg = np.repeat(np.array([p["s_q"], p["s_k"], p["s_v"]], np.float32), dim)
        alpha, beta = vt.fold_requant(p["s_x"], p["s_w_qkv"], p["b_qkv"], seg)
        alpha_o, _ = vt.fold_requant(p["s_p"], np.full(dim, p["s_v"], np.float32), None, p["s_o"])
        quant = lambda n: vt.vitint_quantize(dev(p["w_" + n]), 0.0, bits, True, row_steps=dev(p["s_w_" + n]))
        s["block"] = vt.AttentionWeights(
            batch=c["batch"], tokens=tokens, heads=c["heads"], bits=bits, w_qkv=quant("qkv"), alpha_qkv=dev(alpha),
            beta_qkv=dev(beta), q_step=float(p["s_q"]), k_step=float(p["s_k"]), v_step=float(p["s_v"]), p_step=float(p["s_p"]),
            o_step=float(p["s_o"]), p_bits=bits, alpha_o=dev(alpha_o), beta_o=None, w_proj=quant("proj"),
            w_proj_step=dev(p["s_w_proj"]), b_proj=dev(p["b_proj"]), proj_epi=vt.Epilogue(mode=vt.EPI_DEQUANT_F32))
        s["x"], s["step"] = _activations(g, rows, dim, c["outliers"]), float(p["s_x"])
        s["xq"] = vt.Codes.empty(rows, dim, bits, True)
        s["work"] = torch.empty(vt.vitint_attention_block_workspace_bytes(s["block"]), dtype=torch.uint8, device="cuda")
        s["out"] = torch.empty((rows, dim), dtype=torch.float32, device="cuda")
    elif kind == "layer":
        s["layer"] = EncoderLayer(c["batch"], tokens, c["heads"], c["mlp"], bits, _layer_params(g, dim, c["mlp"], bits, tokens),
                                  wide_activations=c["wide"], softmax=c["softmax"], layernorm=c["layernorm"])
        s["x"], s["out"] = _activations(g, rows, dim), torch.empty((rows, dim), dtype=torch.float32, device="cuda")
    elif kind == "encoder":
        s["stack"] = EncoderStack([_layer_params(g, dim, c["mlp"], bits, tokens) for _ in range(c["layers"])], c["batch"], tokens,
                                  c["heads"], c["mlp"], bits)
        s["x"], s["out"] = _activations(g, rows, dim), torch.empty((rows, dim), dtype=torch.float32, device="cuda")
    elif kind == "normed":
        norm = {n + "n_" + k: _host(_normal(g, (64,), 1.0 if k == "g" else 0.0, 0.02)) for n in ("q", "k") for k in ("g", "b")}
        norm["s_qn"] = norm["s_kn"] = _gauss_step(1.0, bits)
        s["module"] = NormedAttention(c["batch"], tokens, c["heads"], bits, _layer_params(g, dim, 0, bits, tokens), norm)
        s["step"] = float(_gauss_step(1.0, bits))
        # the module sits behind a quantizing LayerNorm: its input is codes, one per byte as the layers store them
        s["xq"] = vt.vitint_quantize(_activations(g, rows, dim), s["step"], bits, True,
                                     out=vt.Codes.empty(rows, dim, bits, True, container=8))
    else:
        s["model"] = DeitModel(_model_ends(g, dim, bits, tokens),
                               [_layer_params(g, dim, c["mlp"], bits, tokens) for _ in range(c["layers"])], c["batch"], tokens,
                               c["heads"], c["mlp"], bits)
        x = _activations(g, rows, PATCH_DIM).view(c["batch"], tokens, PATCH_DIM)
        x[:, :2] = 0.0                    # the class and distillation rows carry no patch
        s["x"] = x.view(rows, PATCH_DIM)
    return s


def run(state):
    s = state
    kind = s["kind"]
    if kind == "layer":
        return s["layer"].forward(s["x"], s["out"])
    if kind == "encoder":
        return s["stack"].forward(s["x"], s["out"])
    if kind == "model":
        return s["model"].forward(s["x"])
    if kind == "normed":
        return s["module"].forward(s["xq"], s["step"]).data
    vt.vitint_quantize(s["x"], s["step"], s["bits"], True, out=s["xq"])
    if kind == "block":
        return vt.vitint_attention_block(s["xq"], s["block"], out=s["out"], workspace=s["work"])
    vt.vitint_linear(s["xq"], s["step"], s["w"], s["w_step"], s["bias"], s["epi"], out=s["out"])
    return s["out"].data if isinstance(s["out"], vt.Codes) else s["out"]


def work(case):
    """Integer operations (two per multiply-accumulate), and the bytes of input, output and weights (at their bit-packed
    width) once."""
    c = case
    packed = {2: 2, 3: 4, 4: 4, 8: 8}[c["bits"]] / 8.0
    if c["kind"] == "linear":
        m, k, n = c["rows"], c["k"], c["n"]
        out = 4.0 if c["epi"] in ("dequant", "acc") else 1.0 if c["wide"] else packed
        return {"bytes": 4.0 * m * k + packed * n * k + out * m * n, "flops": 2.0 * m * n * k}
    dim, t = 64 * c["heads"], c["tokens"]
    rows = c["batch"] * t
    attention = 2.0 * 2 * c["batch"] * c["heads"] * t * t * 64
    if c["kind"] == "normed":
        return {"bytes": rows * dim * (1.0 + packed) + packed * 3 * dim * dim, "flops": attention + 2.0 * rows * dim * 3 * dim}
    if c["kind"] == "block":
        return {"bytes": 8.0 * rows * dim + packed * 4 * dim * dim, "flops": attention + 2.0 * rows * dim * 4 * dim}
    layers = c.get("layers", 1)
    weights = 4 * dim * dim + 2 * dim * c["mlp"]
    flops = layers * (attention + 2.0 * rows * weights)
    if c["kind"] == "model":
        return {"bytes": 4.0 * rows * PATCH_DIM + packed * (layers * weights + PATCH_DIM * dim),
                "flops": flops + 2.0 * rows * PATCH_DIM * dim}
    return {"bytes": 8.0 * rows * dim + packed * layers * weights, "flops": flops}


def tolerance(case):
    """Four times the largest difference seen between this path and the same path evaluated in fp64 (LayerNorm, softmax and
    GELU in fp64, contractions exact), over the listed cases and thirty drawn ones.  What differs is a code that lies on a
    rounding boundary: about one in 10^6 after a LayerNorm or softmax, one in 2 * 10^6 after a GELU, none where no
    floating-point stage precedes the quantizer."""
    c = case
    if c["kind"] == "normed":
        return "exact"                                      # integer and single-rounding operations only
    if c["kind"] == "linear":
        if c["epi"] == "gelu":
            return {"rel": 0.0, "differ": 2e-6}             # seen: 5.2e-7 of the codes at 8 bits
        return {"rel": 1e-6, "max": 1e-6} if c["epi"] == "dequant" else "exact"
    if c["kind"] == "block":
        return {"rel": 1e-3, "max": 0.3}                    # seen: 2.6e-8; one code of P on a boundary gives about 3e-4
    if c["kind"] == "layer":
        if c["layernorm"] == "compare":
            return {"rel": 1e-3, "max": 0.1}                # seen: 2.8e-5, max 0.007, from the GELU codes alone
        return {"rel": 0.015, "max": 0.9}                   # seen: 4.2e-3, max 0.3
    # Several layers: a flipped code changes its row and, through the attention, its image, and each layer multiplies such
    # changes (seen: 0.2 after four to twelve layers when a code flips early, 1e-7 when none does).  No more is allowed here
    # than a few flips in the last layers would give.
    return {"rel": 0.03, "max": 0.9}

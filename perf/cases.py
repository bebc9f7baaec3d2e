"""The workloads this library's speed is judged by: what a user of the PWL forward pass runs, through the public
calls of the Python binding, from a single request to a full batch.

An encoder case is one call of Context.encoder_stack (fp32, bf16 or int8), a CNN case one call of
Context.resnet50_forward, "attention_i8" one call of the int8 attention operator, and "rows" one call of each
memory-bound operator (LayerNorm, element-wise GELU table, int8 quantisation) on the same activations.  Shapes are
the BERT-base / BERT-large / ResNet shapes of nm_inputs.py and nm_inputs_cnn.py, their width and depth variants and
the tests' sizes; inputs and weights follow the same distributions (N(0, 1) activations, N(0, 0.02) weights,
He-normal convolutions, U(0, 1) images), drawn on the device.
"""
import math

import torch

import paper_2305_14405_b200 as nm
from nm_inputs_cnn import resnet_conv_specs

DEVICE = 0
NM_DTYPE = {"f32": nm.F32, "bf16": nm.BF16, "f16": nm.F16, "i8": nm.I8}
TORCH_DTYPE = {"f32": torch.float32, "bf16": torch.bfloat16, "f16": torch.float16, "i8": torch.bfloat16}


def listed():
    return [
        # the smallest layer the library is asked for: one fp32 layer on one sequence, launch latency and CUDA cores
        encoder("f32_tiny_layer", "f32", B=1, L=128, H=256, layers=1),
        # the paper's FP32 evaluation of a BERT-base-shaped encoder on a batch of sentence pairs
        encoder("f32_base_b8", "f32", B=8, L=128, H=768, layers=12),
        # one online request: a single short sentence through the whole BERT-base encoder, no padding
        encoder("bf16_base_sentence", "bf16", B=1, L=37, H=768, layers=12),
        # one BERT-base layer on a small batch: the latency-sized building block of other people's graphs
        encoder("bf16_base_layer_b8", "bf16", B=8, L=128, H=768, layers=1),
        # a batch padded to its longest member, which is nobody's power of two
        encoder("bf16_base_ragged", "bf16", B=7, L=333, H=768, layers=12),
        # offline scoring: a full batch of full-length sequences
        encoder("bf16_base_b32_l512", "bf16", B=32, L=512, H=768, layers=12),
        # the paper's INT8 evaluation at BERT-large size: one request ...
        encoder("i8_large_request", "i8", B=1, L=128, H=1024, layers=24),
        # ... and a full batch
        encoder("i8_large_b16_l512", "i8", B=16, L=512, H=1024, layers=24),
        # image classification, one image at a time ...
        resnet("resnet50_b1", "f16", batch=1),
        # ... and a full batch
        resnet("resnet50_b128", "f16", batch=128),
        # the int8 attention operator on its own, as an int8 network's author calls it
        attention_i8("attention_i8_b32_l512", B=32, L=512, heads=12),
        # the memory-bound operators on a tensor far larger than the L2
        rows("rows_bf16_large", "bf16", n=1 << 19, H=768),
    ]


def draw(rng):
    kind = rng.choice(["bf16", "bf16", "bf16", "i8", "i8", "f32", "f32", "resnet", "resnet", "attention_i8", "rows"])
    if kind in ("bf16", "i8", "f32"):
        top_tokens = {"bf16": 16384, "i8": 8192, "f32": 1024}[kind]
        H = rng.choice({"bf16": [256, 512, 768, 768, 1024], "i8": [512, 768, 1024, 1024], "f32": [256, 512, 768]}[kind])
        layers = log_int(rng, 1, {"bf16": 12, "i8": 24, "f32": 12}[kind])
        L = log_int(rng, 16, min(512, top_tokens))
        if rng.random() < 0.4:   # padded to a round length, as a tokenizer does
            L = max(16, L // 16 * 16)
        B = log_int(rng, 1, min({"bf16": 32, "i8": 16, "f32": 8}[kind], top_tokens // L))
        if H > 768 and kind == "bf16":   # no more work than the largest listed case
            layers = min(layers, 6)
        return encoder(None, kind, B, L, H, layers, segments=rng.choice([16, 64, 64, 256]))
    if kind == "resnet":
        blocks = rng.choice([(2, 2, 2, 2), (3, 4, 6, 3), (3, 4, 6, 3), (3, 4, 23, 3)])
        width = rng.choice([32, 64, 64, 64, 128])
        top = 128
        if blocks[2] > 6:
            top //= 2
        if width > 64:
            top //= 4
        return resnet(None, rng.choice(["f16", "bf16"]), log_int(rng, 1, top), blocks, width)
    if kind == "attention_i8":
        L = 128 * log_int(rng, 1, 8)
        heads = rng.choice([4, 12, 16])
        return attention_i8(None, log_int(rng, 1, max(1, min(32, 32 * 12 * 512 * 512 // (heads * L * L)))), L, heads)
    H = 8 * log_int(rng, 16, 512)
    return rows(None, rng.choice(["bf16", "bf16", "f16", "f32"]), log_int(rng, 100, (1 << 28) // H), H)


def log_int(rng, lo, hi):
    """A whole number from lo to hi, its logarithm uniform."""
    return max(lo, min(hi, int(math.exp(rng.uniform(math.log(lo), math.log(hi + 1))))))


def named(name, case):
    return case if name is None else dict(case, name=name)


def encoder(name, dtype, B, L, H, layers, segments=64):
    return named(name, {"kind": "encoder", "dtype": dtype, "B": B, "L": L, "H": H, "layers": layers, "segments": segments})


def resnet(name, dtype, batch, blocks=(3, 4, 6, 3), width=64):
    return named(name, {"kind": "resnet", "dtype": dtype, "batch": batch, "width": width,
                        **{"blocks%d" % i: b for i, b in enumerate(blocks)}})


def attention_i8(name, B, L, heads, segments=64):
    return named(name, {"kind": "attention_i8", "B": B, "L": L, "heads": heads, "segments": segments})


def rows(name, dtype, n, H, segments=64):
    return named(name, {"kind": "rows", "dtype": dtype, "rows": n, "H": H, "segments": segments})


# ---------------------------------------------------------------- preparation


def table_ranges(L):
    return {"gelu": (-4.0, 4.0), "exp": (-8.0, 0.0), "recip": (L / 16.0, float(L)), "rsqrt": (0.25, 4.0)}


def prepare(case, seed):
    gen = torch.Generator(device="cuda:%d" % DEVICE)
    gen.manual_seed(seed)
    return {"encoder": prepare_encoder, "resnet": prepare_resnet, "attention_i8": prepare_attention_i8,
            "rows": prepare_rows}[case["kind"]](case, gen)


def normal(gen, shape, std=1.0, mean=0.0):
    return torch.randn(shape, generator=gen, device=gen.device) * std + mean


def quantize_rows(w):
    """Symmetric int8 per output channel: codes and scales."""
    s = (w.abs().amax(dim=1) / 127.0).clamp_min(1e-12)
    return torch.clamp(torch.round(w / s[:, None]), -127, 127).to(torch.int8), s


def prepare_encoder(case, gen):
    B, L, H, F, dtype = case["B"], case["L"], case["H"], 4 * case["H"], case["dtype"]
    td = TORCH_DTYPE[dtype]
    ctx = nm.Context(DEVICE)
    ctx.load_encoder_tables(case["segments"], table_ranges(L))
    sig_v = 0.02 * math.sqrt(H)
    layers = []
    for _ in range(case["layers"]):
        w = {}
        for name, shape in (("Wqkv", (3 * H, H)), ("Wo", (H, H)), ("W1", (F, H)), ("W2", (H, F))):
            m = normal(gen, shape, 0.02)
            if dtype == "i8":
                w[name], w["s_w" + name[1:].lower()] = quantize_rows(m)
            else:
                w[name] = m.to(td)
        for name, n in (("bqkv", 3 * H), ("bo", H), ("b1", F), ("b2", H)):
            w[name] = normal(gen, (n,), 0.02)
        for i in ("1", "2"):
            w["g" + i] = normal(gen, (H,), 0.1, 1.0)
            w["be" + i] = normal(gen, (H,), 0.1)
        if dtype == "i8":   # static activation scales, from the distributions
            w.update(a_x=5.5 / 127.0, a_attn=6.0 * sig_v / math.sqrt(L) / 127.0, a_x1=5.5 / 127.0, a_g=4.5 * sig_v / 127.0)
        layers.append(w)
    cfg = ctx.encoder_cfg(B, L, H, H // 64, F, NM_DTYPE[dtype])
    x = normal(gen, (B * L, H)).to(td)
    return {"case": case, "ctx": ctx, "cfg": cfg, "layers": layers, "x": x, "y": torch.empty_like(x),
            "array": nm.layer_array([ctx.encoder_weights(w) for w in layers]),
            "workspace": torch.empty(ctx.encoder_workspace_bytes(cfg), dtype=torch.uint8, device=gen.device)}


def resnet_blocks(case):
    return tuple(case["blocks%d" % i] for i in range(4))


def prepare_resnet(case, gen):
    td, batch, blocks, width = TORCH_DTYPE[case["dtype"]], case["batch"], resnet_blocks(case), case["width"]
    ctx = nm.Context(DEVICE)
    ctx.load_function_table(nm.SLOT_RELU, nm.FUNC_RELU, 2, -8.0, 8.0)
    cfg = ctx.resnet50_cfg(batch, NM_DTYPE[case["dtype"]], blocks=blocks, base_width=width)
    specs = resnet_conv_specs(blocks, width)
    array, convs = (nm.ConvParams * len(specs))(), []
    for i, (cin, cout, k, _, _) in enumerate(specs):
        fan_in = cin * k * k
        # the folded BatchNorm's factor; small in the last convolution of a block, so that the sum over a deep
        # network's blocks keeps its range, as training does
        scale = normal(gen, (cout,), 0.1, 1.0) * (0.3 if i > 0 and specs[i - 1][2] == 3 else 1.0)
        w = (normal(gen, (cout, k, k, cin), math.sqrt(2.0 / fan_in)) * scale[:, None, None, None]).to(td)
        b = normal(gen, (cout,), 0.1)
        array[i].w, array[i].bias = w.data_ptr(), b.data_ptr()
        convs.append((w, b))
    x = torch.rand((batch, 224, 224, 3), generator=gen, device=gen.device).to(td)
    return {"case": case, "ctx": ctx, "cfg": cfg, "convs": convs, "array": array, "x": x,
            "fc_w": normal(gen, (1000, 32 * width), math.sqrt(1.0 / (32 * width))).to(td), "fc_b": normal(gen, (1000,), 0.01),
            "logits": torch.empty((batch, 1000), dtype=td, device=gen.device),
            "workspace": torch.empty(ctx.resnet50_workspace_bytes(cfg), dtype=torch.uint8, device=gen.device)}


def prepare_attention_i8(case, gen):
    B, L, H = case["B"], case["L"], case["heads"] * 64
    ctx = nm.Context(DEVICE)
    ctx.load_encoder_tables(case["segments"], table_ranges(L))
    scale = 4.5 * 0.6 / 127.0
    codes = torch.clamp(torch.round(normal(gen, (B * L, 3 * H), 0.6 / scale)), -127, 127).to(torch.int8)
    return {"case": case, "ctx": ctx, "qkv": codes, "scale": scale,
            "out": torch.empty((B * L, H), dtype=torch.bfloat16, device=gen.device)}


def prepare_rows(case, gen):
    n, H, td = case["rows"], case["H"], TORCH_DTYPE[case["dtype"]]
    ctx = nm.Context(DEVICE)
    ctx.load_encoder_tables(case["segments"], table_ranges(512))
    x = torch.empty((n, H), dtype=td, device=gen.device)
    step = max(1, (1 << 26) // H)
    for i in range(0, n, step):
        x[i:i + step] = normal(gen, (min(step, n - i), H)).to(td)
    return {"case": case, "ctx": ctx, "x": x, "gamma": normal(gen, (H,), 0.1, 1.0), "beta": normal(gen, (H,), 0.1),
            "normed": torch.empty_like(x), "gelu": torch.empty_like(x),
            "codes": torch.empty((n, H), dtype=torch.int8, device=gen.device)}


# ---------------------------------------------------------------- one pass


def run(s):
    case, ctx = s["case"], s["ctx"]
    if case["kind"] == "encoder":
        ctx.encoder_stack(s["array"], case["layers"], s["cfg"], s["x"], s["y"], s["workspace"])
        return s["y"]
    if case["kind"] == "resnet":
        ctx.resnet50_forward(s["array"], s["fc_w"], s["fc_b"], s["cfg"], s["x"], s["logits"], s["workspace"])
        return s["logits"]
    if case["kind"] == "attention_i8":
        ctx.attention_pwl_i8(s["qkv"], s["out"], case["B"], case["L"], case["heads"], 64, s["scale"], s["scale"], s["scale"])
        return s["out"]
    ctx.layernorm_pwl(s["x"], s["gamma"], s["beta"], s["normed"])
    ctx.pwl_apply(nm.SLOT_GELU, s["x"], s["gelu"])
    ctx.quantize_i8(s["x"], 127.0 / 5.5, s["codes"])
    return s["normed"], s["gelu"], s["codes"]


# ---------------------------------------------------------------- what a pass cannot do without


def work(case):
    if case["kind"] == "encoder":
        T, L, H, F = case["B"] * case["L"], case["L"], case["H"], 4 * case["H"]
        act = {"f32": 4, "bf16": 2, "i8": 2}[case["dtype"]]
        wt = {"f32": 4, "bf16": 2, "i8": 1}[case["dtype"]]
        vectors = 4 * (13 * H + (9 * H if case["dtype"] == "i8" else 0))   # biases, gammas, betas, weight scales
        return {"bytes": case["layers"] * (wt * (4 * H * H + 2 * H * F) + vectors) + 2 * T * H * act,
                "flops": case["layers"] * (2 * T * (4 * H * H + 2 * H * F) + 4 * T * L * H)}
    if case["kind"] == "resnet":
        blocks, width, N = resnet_blocks(case), case["width"], case["batch"]
        size, flops, weights = 224, 0, 0
        specs = iter(resnet_conv_specs(blocks, width))

        def conv(out_size):
            nonlocal flops, weights
            cin, cout, k, _, _ = next(specs)
            flops += 2 * N * out_size * out_size * cout * cin * k * k
            weights += 2 * cout * cin * k * k + 4 * cout

        conv(112)
        size = 56
        for stage, nb in enumerate(blocks):
            for b in range(nb):
                out_size = size // 2 if b == 0 and stage > 0 else size
                conv(size)
                conv(out_size)
                conv(out_size)
                if b == 0:
                    conv(out_size)
                size = out_size
        feat = 32 * width
        return {"bytes": weights + 2 * 1000 * feat + 4 * 1000 + 2 * N * (224 * 224 * 3 + 1000),
                "flops": flops + 2 * N * feat * (49 + 1000)}
    if case["kind"] == "attention_i8":
        T, H = case["B"] * case["L"], case["heads"] * 64
        return {"bytes": 3 * T * H + 2 * T * H, "flops": 4 * T * case["L"] * H}
    n, es = case["rows"] * case["H"], {"f32": 4, "bf16": 2, "f16": 2}[case["dtype"]]
    return {"bytes": 2 * n * es + 2 * n * es + n * (es + 1) + 8 * case["H"], "flops": 8 * n + 3 * n + 2 * n}


def tolerance(case):
    """About four times what other correct implementations differ by: the library's CUDA-core and resident-score
    kernels and a 64-bit evaluation that rounds where the storage type does.  The differences of independent layers
    add up in quadrature (one bf16 layer 2.7e-3 ... twelve 9.4e-3, 24 int8 layers 5.5e-2, where a last-bit difference
    moves a code to its neighbour; fp32 sums of 768 terms 3.6e-7 per layer)."""
    if case["kind"] == "encoder":
        return {"rel": {"f32": 1.5e-6, "bf16": 1e-2, "i8": 3e-2}[case["dtype"]] * math.sqrt(case["layers"])}
    if case["kind"] == "resnet":   # 5e-4 (fp16) and 3.2e-3 (bf16) at every depth
        return {"rel": 2e-3 if case["dtype"] == "f16" else 1.3e-2}
    if case["kind"] == "attention_i8":
        return "exact"   # every integer exact, every fp32 step one defined rounding
    return {"rel": {"f32": 1e-6, "f16": 3e-4, "bf16": 2e-3}[case["dtype"]]}   # one rounding to the storage type

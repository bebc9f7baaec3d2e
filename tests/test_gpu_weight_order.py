"""Weights that another kernel of the same stream has just written: a chain of kernels fetches weights early, and must still see
what was enqueued before the call."""
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype", ["bf16", "i8"])
def test_layer_after_its_weights_were_written_by_the_stream(nm, dtype):
    ctx = nm.Context(0)
    try:
        B, L, H = 1, 64, 768
        F = 4 * H
        ctx.load_encoder_tables(64, {"gelu": (-4.0, 4.0), "exp": (-8.0, 0.0), "recip": (L / 16.0, float(L)), "rsqrt": (0.25, 4.0)})
        g = torch.Generator(device="cuda").manual_seed(1)
        i8 = dtype == "i8"

        def matrix(n, k):
            if i8:
                return torch.randint(-127, 128, (n, k), generator=g, device="cuda", dtype=torch.int8)
            return (torch.randn((n, k), generator=g, device="cuda") * 0.02).bfloat16()

        names = {"Wqkv": (3 * H, H), "Wo": (H, H), "W1": (F, H), "W2": (H, F)}
        src = {n: matrix(*s) for n, s in names.items()}
        vec = {n: torch.randn(k, generator=g, device="cuda") * 0.02 for n, k in
               (("bqkv", 3 * H), ("bo", H), ("b1", F), ("b2", H), ("be1", H), ("be2", H))}
        vec.update(g1=torch.ones(H, device="cuda"), g2=torch.ones(H, device="cuda"))
        if i8:
            vec.update({"s_w" + n[1:].lower(): torch.full((s[0],), 0.02 / 40, device="cuda") for n, s in names.items()},
                       a_x=0.04, a_attn=0.01, a_x1=0.04, a_g=0.02)
        vec["g1"], vec["g2"] = vec["g1"] + vec["be1"], vec["g2"] + vec["be2"]
        host = {n: t for n, t in vec.items() if not torch.is_tensor(t)}
        src.update({n: t for n, t in vec.items() if torch.is_tensor(t)})     # biases, LayerNorm's vectors, weight scales
        dst = {n: torch.zeros_like(t) for n, t in src.items()}
        cfg = ctx.encoder_cfg(B, L, H, H // 64, F, nm.I8 if i8 else nm.BF16)
        w = [ctx.encoder_weights({**t, **host}) for t in (src, dst)]
        x = torch.randn((B * L, H), generator=g, device="cuda").bfloat16()
        ws = torch.empty(ctx.encoder_workspace_bytes(cfg), dtype=torch.uint8, device="cuda")
        want, y = torch.empty_like(x), torch.empty_like(x)
        arrays = [nm.layer_array([s, s]) for s in w]
        ctx.encoder_stack(arrays[0], 2, cfg, x, want, ws)
        torch.cuda.synchronize()
        A, out = torch.randn((4096, 3072), device="cuda").bfloat16(), torch.empty((4096, 3072), dtype=torch.bfloat16, device="cuda")
        Wf = torch.randn((3072, 3072), device="cuda").bfloat16()
        eye, product = torch.eye(H, device="cuda").bfloat16(), torch.empty((F, H), dtype=torch.bfloat16, device="cuda")
        one = torch.zeros((1, 8), device="cuda")
        one[0, 0] = 1.0
        last = ("W1", "b1", "g1", "be2") if not i8 else ("b1", "g1", "be2", "s_w2")   # one of them a kernel's that lets its successor start early
        column = {n: torch.nn.functional.pad(src[n][:, None], (0, 7)).contiguous() for n in last if n != "W1"}
        for run in range(24):
            for t in dst.values():
                t.zero_()
            ctx.linear_pwl(A, Wf, out)              # keeps the stream busy while the rest is enqueued
            for n, t in dst.items():
                t.copy_(src[n])
            n = last[run % len(last)]
            dst[n].zero_()
            if n == "W1":
                ctx.linear_pwl(src["W1"], eye, dst["W1"])
            else:                                   # 1 x v + 0 ...: the vector itself
                ctx.linear_pwl(one, column[n], dst[n][None])
            ctx.encoder_stack(arrays[1], 2, cfg, x, y, ws)
            torch.cuda.synchronize()
            assert torch.equal(y, want), run
        ctx.check_device_status()
    finally:
        ctx.close()


def test_resnet_after_its_weights_were_written_by_the_stream(nm):
    ctx = nm.Context(0)
    try:
        ctx.load_function_table(nm.SLOT_RELU, nm.FUNC_RELU, 2, -8.0, 8.0)
        g = torch.Generator(device="cuda").manual_seed(2)
        cfg = ctx.resnet50_cfg(1, nm.F16, num_classes=1000, blocks=(1, 1, 1, 1), base_width=64)
        from nm_inputs_cnn import resnet_conv_specs
        specs = resnet_conv_specs((1, 1, 1, 1), 64)
        src = []
        for cin, cout, k, _, _ in specs:
            src.append((torch.randn((cout, k, k, cin), generator=g, device="cuda") * (2.0 / (cin * k * k)) ** 0.5).half())
            src.append(torch.randn(cout, generator=g, device="cuda") * 0.1)
        src.append((torch.randn((1000, 2048), generator=g, device="cuda") * 0.02).half())
        src.append(torch.randn(1000, generator=g, device="cuda"))
        dst = [torch.zeros_like(t) for t in src]
        arrays = []
        for t in (src, dst):
            a = (nm.ConvParams * len(specs))()
            for i in range(len(specs)):
                a[i].w, a[i].bias = t[2 * i].data_ptr(), t[2 * i + 1].data_ptr()
            arrays.append(a)
        x = torch.rand((1, 224, 224, 3), generator=g, device="cuda").half()
        ws = torch.empty(ctx.resnet50_workspace_bytes(cfg), dtype=torch.uint8, device="cuda")
        want, y = [torch.empty((1, 1000), dtype=torch.float16, device="cuda") for _ in range(2)]
        ctx.resnet50_forward(arrays[0], src[-2], src[-1], cfg, x, want, ws)
        torch.cuda.synchronize()
        assert torch.isfinite(want).all() and want.float().std() > 0
        A, out = torch.randn((4096, 3072), device="cuda").half(), torch.empty((4096, 3072), dtype=torch.float16, device="cuda")
        Wf, eye = torch.randn((3072, 3072), device="cuda").half(), torch.eye(64, device="cuda").half()
        conv2 = 2   # the first 1 x 1 convolution behind the stem: 64 x 64
        assert src[conv2].shape == (64, 1, 1, 64)
        for run in range(20):
            for t in dst:
                t.zero_()
            ctx.linear_pwl(A, Wf, out)
            for t, s in zip(dst, src):
                t.copy_(s)
            if run % 2:                             # by a kernel that lets its successor start early
                dst[conv2].zero_()
                ctx.linear_pwl(src[conv2].view(64, 64), eye, dst[conv2].view(64, 64), algo=nm.ALGO_TC)
            ctx.resnet50_forward(arrays[1], dst[-2], dst[-1], cfg, x, y, ws)
            torch.cuda.synchronize()
            assert torch.equal(y, want), run
        ctx.check_device_status()
    finally:
        ctx.close()

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
        dst = {n: torch.zeros_like(t) for n, t in src.items()}
        cfg = ctx.encoder_cfg(B, L, H, H // 64, F, nm.I8 if i8 else nm.BF16)
        w = [ctx.encoder_weights({**t, **vec}) for t in (src, dst)]
        x = torch.randn((B * L, H), generator=g, device="cuda").bfloat16()
        ws = torch.empty(ctx.encoder_workspace_bytes(cfg), dtype=torch.uint8, device="cuda")
        want, y = torch.empty_like(x), torch.empty_like(x)
        arrays = [nm.layer_array([s, s]) for s in w]
        ctx.encoder_stack(arrays[0], 2, cfg, x, want, ws)
        torch.cuda.synchronize()
        A, out = torch.randn((4096, 3072), device="cuda").bfloat16(), torch.empty((4096, 3072), dtype=torch.bfloat16, device="cuda")
        Wf = torch.randn((3072, 3072), device="cuda").bfloat16()
        eye, product = torch.eye(H, device="cuda").bfloat16(), torch.empty((F, H), dtype=torch.bfloat16, device="cuda")
        for run in range(20):
            for t in dst.values():
                t.zero_()
            ctx.linear_pwl(A, Wf, out)              # keeps the stream busy while the rest is enqueued
            for n, t in dst.items():
                t.copy_(src[n])
            if not i8:                              # and one weight by a kernel that lets its successor start early
                dst["W1"].zero_()
                ctx.linear_pwl(src["W1"], eye, dst["W1"])
            ctx.encoder_stack(arrays[1], 2, cfg, x, y, ws)
            torch.cuda.synchronize()
            assert torch.equal(y, want), run
        ctx.check_device_status()
    finally:
        ctx.close()

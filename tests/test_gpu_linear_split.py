"""GPU parity, linear operator on problems of few tiles (K split over a thread-block cluster) and convolutions likewise."""
import numpy as np
import pytest
import torch

import nm_inputs
import oracle
from util import load_tables_both, rms_rel, to_np

pytestmark = pytest.mark.gpu
RANGES = {"gelu": (-4.0, 4.0), "relu": (-3.0, 3.0)}


@pytest.fixture(scope="module")
def ctx(nm):
    c = nm.Context(0)
    yield c
    c.close()


def strided(a, td, pad):
    """The matrix as the left part of a wider one (row pitch larger than the row)."""
    t = torch.full((a.shape[0], a.shape[1] + pad), float("nan") if td.is_floating_point else 77, dtype=td, device="cuda")
    t[:, :a.shape[1]] = torch.from_numpy(np.ascontiguousarray(a)).cuda().to(td)
    return t[:, :a.shape[1]]


# rows: one, a warp's edge, a tile's edge; columns: less than a tile, a tile's edge, no multiple of 8; K: one block, a
# ragged block, every split
SHAPES = [(1, 8, 8), (1, 768, 768), (31, 64, 72), (33, 68, 128), (37, 2304, 768), (64, 60, 520), (127, 132, 200),
          (128, 768, 3072), (129, 320, 1032), (300, 128, 64), (1024, 768, 768), (1500, 1004, 64)]


@pytest.mark.parametrize("dtype", ["bf16", "f16"])
@pytest.mark.parametrize("M,N,K", SHAPES)
@pytest.mark.parametrize("epi", ["plain", "gelu_bias", "bias_res", "relu_res_first"])
def test_16_bit(nm, ctx, dtype, M, N, K, epi, algo=0):
    tabs = load_tables_both(ctx, 64, RANGES)
    td = nm_inputs.torch_dtype(dtype)
    A, W = nm_inputs.matrix((M, K), M + K, dtype, 1.0), nm_inputs.matrix((N, K), N, dtype, 0.05)
    rng = np.random.default_rng(K)
    bias = None if epi == "plain" else (0.1 * rng.standard_normal(N)).astype(np.float32)
    res = nm_inputs.round_to(rng.standard_normal((M, N)).astype(np.float32), dtype) if "res" in epi else None
    slot, tab = {"gelu_bias": (nm.SLOT_GELU, "gelu"), "relu_res_first": (nm.SLOT_RELU, "relu")}.get(epi, (nm.SLOT_NONE, None))
    first = epi == "relu_res_first"
    pad = 8 if (M + N) % 2 else 0
    out = torch.full((M, N + 8 - N % 8 + pad), float("nan"), dtype=td, device="cuda")
    ctx.linear_pwl(strided(A, td, pad + 8 - K % 8), strided(W, td, 8 - K % 8), out[:, :N], slot=slot, res_first=first, algo=algo,
                   bias=None if bias is None else torch.from_numpy(bias).cuda(),
                   residual=None if res is None else strided(res, td, 8 - N % 8 + pad))
    ctx.check_device_status()
    assert torch.isnan(out[:, N:].float()).all()
    if first:
        z = oracle.linear(A, W, bias, res, None)
        ref = np.asarray(z, np.float64)
        s = np.clip(np.floor(np.asarray(z, np.float32) * np.float32(64 / 6.0) + np.float32(32.0)), 0, 63).astype(int)
        ref = tabs["relu"].k.astype(np.float64)[s] * ref + tabs["relu"].b.astype(np.float64)[s]
    else:
        ref = oracle.linear(A, W, bias, res, tabs[tab] if tab else None)
    got = to_np(out[:, :N])
    assert np.all(np.isfinite(got))
    # the storage type's rounding of the result, and fp32 sums of up to 3072 products (1e-5 of the rms allows for both
    # sides of a table's breakpoint)
    half_ulp = {"bf16": 2.0 ** -8, "f16": 2.0 ** -11}[dtype]
    rms = np.sqrt(np.mean(ref * ref))
    assert np.all(np.abs(got - ref) <= half_ulp * 1.01 * np.abs(ref) + 1e-5 * max(rms, 1.0)), np.abs(got - ref).max()


@pytest.mark.parametrize("dtype", ["bf16", "f16"])
@pytest.mark.parametrize("S", [1, 2, 4, 8])
@pytest.mark.parametrize("BN", [32, 64])
@pytest.mark.parametrize("M,N,K,epi", [(1, 36, 520, "bias_res"), (37, 100, 1032, "gelu_bias"), (127, 64, 512, "plain"), (130, 196, 904, "relu_res_first")])
def test_every_form_16_bit(nm, ctx, dtype, S, BN, M, N, K, epi):
    """Every cluster size and width of the kernel: fewer rows than CTAs, a row less than a tile and two more, columns and K ragged."""
    test_16_bit(nm, ctx, dtype, M, N, K, epi, nm.algo_split(S, BN))


@pytest.mark.parametrize("out", ["bf16", "i8", "f32"])
@pytest.mark.parametrize("S", [1, 2, 4, 8])
@pytest.mark.parametrize("BN", [32, 64])
@pytest.mark.parametrize("M,N,K", [(1, 36, 1040), (37, 100, 2000), (127, 64, 1024), (130, 196, 1808)])
def test_every_form_int8(nm, ctx, out, S, BN, M, N, K):
    test_int8_bit_exact(nm, ctx, M, N, K, out, nm.algo_split(S, BN))


@pytest.mark.parametrize("S", [1, 2, 4, 8])
@pytest.mark.parametrize("BN", [32, 64])
@pytest.mark.parametrize("N,H,Cin,Cout,k,stride,pad,res", [(1, 13, 64, 72, 3, 1, 1, True), (3, 9, 64, 200, 3, 2, 1, False), (2, 7, 512, 40, 1, 2, 0, True)])
def test_every_form_convolution(nm, ctx, S, BN, N, H, Cin, Cout, k, stride, pad, res):
    test_convolution(nm, ctx, N, H, Cin, Cout, k, stride, pad, res, nm.algo_split(S, BN))


def test_forced_forms_are_refused_where_they_do_not_fit(nm, ctx):
    A, W = [torch.zeros(s, dtype=torch.bfloat16, device="cuda") for s in ((8, 256), (64, 256))]   # four K-blocks
    out = torch.zeros(8, 64, dtype=torch.bfloat16, device="cuda")
    with pytest.raises(nm.NmError) as ei:
        ctx.linear_pwl(A, W, out, algo=nm.algo_split(8, 64))
    assert ei.value.code == 5
    with pytest.raises(nm.NmError) as ei:
        ctx.linear_pwl(A.float(), W.float(), out.float(), algo=nm.algo_split(1, 64))
    assert ei.value.code == 5


@pytest.mark.parametrize("algo", [0, 2, 3])
@pytest.mark.parametrize("M,N,K", [(40, 8, 64), (130, 12, 72), (300, 60, 64), (300, 68, 128), (513, 132, 136), (700, 260, 64), (9000, 1004, 64)])
def test_rows_that_are_no_multiple_of_16_bytes(nm, ctx, M, N, K, algo):
    """Nothing is written beyond a row (the border holds NaN), by no kernel."""
    test_16_bit(nm, ctx, "bf16", M, N, K, "bias_res", algo)


@pytest.mark.parametrize("algo", [0, 2, 3])
@pytest.mark.parametrize("M,N,K,out", [(300, 68, 128, "i8"), (140, 332, 144, "bf16"), (600, 268, 64, "i8"), (600, 1020, 64, "bf16")])
def test_int8_rows_that_are_no_multiple_of_16_bytes(nm, ctx, M, N, K, out, algo):
    test_int8_bit_exact(nm, ctx, M, N, K, out, algo)


@pytest.mark.parametrize("M,N,K,out", [(1, 8, 16, "f32"), (33, 68, 128, "i8"), (128, 1024, 1024, "bf16"), (128, 4096, 1024, "i8"),
                                       (128, 1024, 4096, "f32"), (200, 328, 144, "bf16")])
def test_int8_bit_exact(nm, ctx, M, N, K, out, algo=0):
    tabs = load_tables_both(ctx, 64, RANGES)
    Aq, Wq = nm_inputs.int8_matrix((M, K), 21), nm_inputs.int8_matrix((N, K), 22)
    rng = np.random.default_rng(23)
    a_scale = np.float32(4.0 / 127)
    ws = (rng.uniform(0.5, 1.5, N) * 0.08 / 127).astype(np.float32)
    bias = (0.1 * rng.standard_normal(N)).astype(np.float32)
    out_scale = np.float32(0.02)
    td = {"bf16": torch.bfloat16, "i8": torch.int8, "f32": torch.float32}[out]
    ldo = (N + 15) // 16 * 16
    o = torch.full((M, ldo), 99, dtype=td, device="cuda")
    acc = torch.full((M, N), -1, dtype=torch.int32, device="cuda")
    idx = torch.full((M, N), -7, dtype=torch.int32, device="cuda")
    ctx.linear_pwl(torch.from_numpy(Aq).cuda(), torch.from_numpy(Wq).cuda(), o[:, :N], bias=torch.from_numpy(bias).cuda(),
                   slot=nm.SLOT_GELU, a_scale=float(a_scale), w_scale=torch.from_numpy(ws).cuda(),
                   inv_out_scale=float(np.float32(1.0) / out_scale), acc_dump=acc, idx_dump=idx, algo=algo)
    ctx.check_device_status()
    assert (o[:, N:] == 99).all()
    r = oracle.linear_i8(Aq, Wq, a_scale, ws, bias, None, tabs["gelu"], out_scale=out_scale)
    assert np.array_equal(acc.cpu().numpy(), r["acc"])
    assert np.array_equal(idx.cpu().numpy(), r["idx"])
    got = o[:, :N].cpu().contiguous()
    if out == "i8":
        assert np.array_equal(got.numpy(), r["q"])
    elif out == "f32":
        assert np.array_equal(got.numpy().view(np.uint32), r["y"].view(np.uint32))
    else:
        assert torch.equal(got, torch.from_numpy(r["y"]).to(torch.bfloat16))


@pytest.mark.parametrize("N,H,Cin,Cout,k,stride,pad,res", [(1, 14, 256, 256, 3, 1, 1, False), (1, 7, 512, 512, 3, 1, 1, False),
                                                           (2, 7, 512, 72, 1, 2, 0, False), (1, 56, 64, 64, 3, 1, 1, True),
                                                           (3, 9, 64, 200, 3, 2, 1, True)])
def test_convolution(nm, ctx, N, H, Cin, Cout, k, stride, pad, res, forced=0):
    """The split kernel's implicit GEMM against the explicit gather on the CUDA cores."""
    ctx.load_function_table(nm.SLOT_RELU, nm.FUNC_RELU, 2, -8.0, 8.0)
    g = torch.Generator(device="cuda").manual_seed(H + Cin)
    x = torch.randn((N, H, H, Cin), generator=g, device="cuda").half()
    w = (torch.randn((Cout, k, k, Cin), generator=g, device="cuda") * (2.0 / (Cin * k * k)) ** 0.5).half()
    b = torch.randn(Cout, generator=g, device="cuda") * 0.1
    Ho = (H + 2 * pad - k) // stride + 1
    r = torch.randn((N, Ho, Ho, Cout), generator=g, device="cuda").half() if res else None
    outs = []
    for algo in (forced, nm.ALGO_SIMT):
        out = torch.full((N, Ho, Ho, Cout), float("nan"), device="cuda").half()
        d = ctx.conv_desc(x, w, out, stride, pad, bias=b, residual=r, slot=nm.SLOT_RELU, res_first=res, algo=algo)
        ctx.conv2d_pwl(d, torch.empty(max(256, ctx.conv2d_workspace_bytes(d)), dtype=torch.uint8, device="cuda"))
        ctx.check_device_status()
        outs.append(to_np(out))
    # fp32 sums in another order, then one rounding each to fp16: at most one unit in the last place apart
    assert np.all(np.abs(outs[0] - outs[1]) <= 2.0 ** -10 * np.abs(outs[1]) + 1e-5), np.abs(outs[0] - outs[1]).max()
    assert rms_rel(outs[0], outs[1]) <= 2.0 ** -11


@pytest.mark.parametrize("M", [1, 3, 7, 37, 127, 130])
@pytest.mark.parametrize("N,K", [(36, 640), (64, 1024), (768, 3072), (1024, 4096)])
def test_rows_of_a_cluster(nm, ctx, M, N, K):
    """Fewer rows than CTAs in a cluster, row counts that do not divide among them."""
    test_16_bit(nm, ctx, "bf16", M, N, K, "bias_res")


@pytest.mark.parametrize("dtype", ["bf16", "f16"])
@pytest.mark.parametrize("M,N,K", [(8, 256, 16), (8, 256, 64), (16, 768, 256), (37, 768, 768), (37, 768, 3072), (48, 1024, 4096), (1, 256, 9000),
                                   (300, 32, 32), (300, 32, 128), (300, 36, 288), (300, 48, 1024)])
def test_sums_of_few_rows_or_columns(nm, ctx, dtype, M, N, K):
    """Their sums are no further from the exact ones than the CUDA cores' chains of fp32 FMAs.  A row's sums are seen before
    they are rounded to 16 bits: the bias takes away the row's exact sums and leaves the error."""
    td = nm_inputs.torch_dtype(dtype)
    g = torch.Generator(device="cuda").manual_seed(K)
    A = torch.randn((M, K), generator=g, device="cuda").to(td)
    W = (torch.randn((N, K), generator=g, device="cuda") * 0.02).to(td)
    exact = A.double() @ W.double().t()
    err = {}
    for algo in (nm.ALGO_AUTO, nm.ALGO_SIMT):
        e = []
        for m in range(0, M, (M + 31) // 32):
            bias = -exact[m].float()
            out = torch.empty((M, N + 8 - N % 8), dtype=td, device="cuda")[:, :N]
            ctx.linear_pwl(A, W, out, bias=bias, algo=algo)
            e.append(out[m].double() - (exact[m] + bias.double()))
        err[algo] = float(torch.cat(e).pow(2).mean().sqrt())
    ctx.check_device_status()
    # (256 and more errors a case: their rms is known to 5 %)
    assert err[nm.ALGO_AUTO] <= 1.05 * err[nm.ALGO_SIMT], err

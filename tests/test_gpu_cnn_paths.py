"""GPU parity of the convolution's and the pool's special forms at their edges: the first layer's row pairs, the halo form of
the 3 x 3 convolution, the packed maximum."""
import numpy as np
import pytest
import torch

from util import rms_rel, to_np

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx(nm):
    c = nm.Context(0)
    c.load_function_table(nm.SLOT_RELU, nm.FUNC_RELU, 2, -8.0, 8.0)
    yield c
    c.close()


def conv_both(nm, ctx, x, w, b, stride, pad, res=None):
    """The chosen kernel and the explicit gather on the CUDA cores."""
    N, H, W, _ = x.shape
    Cout, kh, kw = w.shape[:3]
    Ho, Wo = (H + 2 * pad - kh) // stride + 1, (W + 2 * pad - kw) // stride + 1
    outs = []
    for algo in (nm.ALGO_AUTO, nm.ALGO_SIMT):
        out = torch.full((N, Ho, Wo, Cout), float("nan"), device="cuda").to(x.dtype)
        d = ctx.conv_desc(x, w, out, stride, pad, bias=b, residual=res, slot=nm.SLOT_RELU, res_first=res is not None, algo=algo)
        ctx.conv2d_pwl(d, torch.empty(max(256, ctx.conv2d_workspace_bytes(d)), dtype=torch.uint8, device="cuda"))
        ctx.check_device_status()
        outs.append(to_np(out))
    # fp32 sums in another order, then one rounding each to the storage type: at most one unit in the last place apart
    ulp = 2.0 ** -10 if x.dtype == torch.float16 else 2.0 ** -7
    assert np.all(np.abs(outs[0] - outs[1]) <= ulp * np.abs(outs[1]) + 1e-5), np.abs(outs[0] - outs[1]).max()
    assert rms_rel(outs[0], outs[1]) <= ulp / 2


def operands(N, H, W, Cin, Cout, kh, kw, dtype, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    x = torch.randn((N, H, W, Cin), generator=g, device="cuda").to(dtype)
    w = (torch.randn((Cout, kh, kw, Cin), generator=g, device="cuda") * (2.0 / (Cin * kh * kw)) ** 0.5).to(dtype)
    return x, w, torch.randn(Cout, generator=g, device="cuda") * 0.1, g


@pytest.mark.parametrize("dtype", [torch.float16, torch.bfloat16])
@pytest.mark.parametrize("N,H,W,Cin,Cout,kh,kw,pad", [(2, 64, 48, 3, 64, 7, 7, 3), (1, 33, 29, 3, 24, 7, 7, 3), (3, 17, 40, 1, 8, 5, 3, 1),
                                                      (1, 30, 31, 4, 72, 2, 8, 0), (2, 15, 15, 2, 16, 1, 1, 0), (1, 224, 224, 3, 64, 7, 7, 3)])
def test_first_layer_row_pairs(nm, ctx, dtype, N, H, W, Cin, Cout, kh, kw, pad):
    x, w, b, _ = operands(N, H, W, Cin, Cout, kh, kw, dtype, H + W)
    conv_both(nm, ctx, x, w, b, 2, pad)


@pytest.mark.parametrize("N,H,W,Cin,Cout,kh,kw,pad", [(2, 32, 24, 3, 64, 7, 7, 3), (1, 33, 20, 3, 16, 3, 3, 1), (2, 31, 17, 4, 8, 5, 8, 2),
                                                      (1, 20, 20, 3, 8, 1, 1, 0), (1, 30, 30, 3, 24, 4, 7, 1), (70, 32, 32, 3, 64, 7, 7, 3)])
def test_first_layer_reads_no_row_outside_the_window(nm, ctx, N, H, W, Cin, Cout, kh, kw, pad):
    """Rows of NaN and infinities reach the outputs whose window holds them and no others."""
    x, w, b, _ = operands(N, H, W, Cin, Cout, kh, kw, torch.float16, H)
    Ho, Wo = (H + 2 * pad - kh) // 2 + 1, (W + 2 * pad - kw) // 2 + 1
    for rows in ([H // 2], [H // 2 + 1], [0, H - 1], [3]):
        xr = x.clone()
        xr[:, rows] = float("nan")
        xr[0, rows] = float("inf")
        out = torch.zeros((N, Ho, Wo, Cout), device="cuda").half()
        d = ctx.conv_desc(xr, w, out, 2, pad, bias=b, slot=nm.SLOT_NONE)
        ctx.conv2d_pwl(d, torch.empty(max(256, ctx.conv2d_workspace_bytes(d)), dtype=torch.uint8, device="cuda"))
        ctx.check_device_status()
        holds = [any(2 * oy - pad <= r < 2 * oy - pad + kh for r in rows) for oy in range(Ho)]
        finite = torch.isfinite(out).all(3).all(2).all(0).tolist()
        assert [not f for f in finite] == holds, (rows, finite, holds)


@pytest.mark.parametrize("dtype", [torch.float16, torch.bfloat16])
@pytest.mark.parametrize("N,H,W,Cin,Cout,res", [(30, 56, 56, 64, 64, False), (85, 28, 28, 128, 128, False), (150, 24, 20, 64, 40, True),
                                                (75, 33, 31, 128, 72, True), (41, 50, 40, 192, 128, False), (199, 32, 18, 64, 64, True)])
def test_halo(nm, ctx, dtype, N, H, W, Cin, Cout, res):
    """Whole and cut-off patches in both directions, an odd number of patches, weights resident and in a ring."""
    x, w, b, g = operands(N, H, W, Cin, Cout, 3, 3, dtype, N)
    r = torch.randn((N, H, W, Cout), generator=g, device="cuda").to(dtype) if res else None
    conv_both(nm, ctx, x, w, b, 1, 1, r)


@pytest.mark.parametrize("dtype", [torch.float16, torch.bfloat16])
@pytest.mark.parametrize("N,H,W,C,ks,stride,pad", [(2, 112, 112, 64, 3, 2, 1), (1, 7, 5, 8, 3, 2, 1), (3, 9, 13, 24, 2, 2, 0), (1, 8, 8, 136, 5, 1, 4),
                                                   (2, 6, 6, 16, 1, 1, 0), (1, 3, 300, 8, 3, 3, 2), (65539, 2, 2, 8, 2, 2, 0), (70001, 1, 1, 24, 1, 1, 0),
                                                   (333, 5, 4, 40, 3, 1, 1), (20, 7, 7, 1024, 7, 1, 0), (2, 70000, 2, 8, 1, 1, 0)])
def test_maxpool_is_exact(ctx, dtype, N, H, W, C, ks, stride, pad):
    g = torch.Generator(device="cuda").manual_seed(C)
    x = torch.randn((N, H, W, C), generator=g, device="cuda").to(dtype)
    x[0, 0, 0, 0], x[0, -1, -1, 1], x[0, min(1, H - 1), min(1, W - 1), 2] = float("inf"), float("-inf"), torch.finfo(dtype).min
    Ho, Wo = (H + 2 * pad - ks) // stride + 1, (W + 2 * pad - ks) // stride + 1
    y = torch.full((N, Ho, Wo, C), float("nan"), device="cuda").to(dtype)
    ctx.maxpool2d(x, y, ks, stride, pad)
    ctx.check_device_status()
    p = torch.nn.functional.pad(x.float().permute(0, 3, 1, 2), (pad, pad + ks, pad, pad + ks), value=float("-inf"))
    want = torch.nn.functional.max_pool2d(p, ks, stride)[:, :, :Ho, :Wo].permute(0, 2, 3, 1)
    assert torch.equal(y.float(), want)

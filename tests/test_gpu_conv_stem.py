"""GPU parity of the first convolution's forms: the patch-wise one at its edges, the row pairs where the output is wider."""
import pytest
import torch

import test_gpu_cnn_paths
from test_gpu_cnn_paths import conv_both, ctx, operands  # noqa: F401

pytestmark = pytest.mark.gpu


# one output pixel, a patch of 8 x 16 and one more in each direction, both tile widths, an odd number of patches, eight filter rows,
# padding wider than the filter's half; 136 and 144 columns, nine filter rows: the row pairs
@pytest.mark.parametrize("dtype", [torch.float16, torch.bfloat16])
@pytest.mark.parametrize("N,H,W,Cin,Cout,kh,kw,pad,res", [
    (1, 7, 7, 3, 8, 7, 7, 0, False), (1, 32, 16, 3, 64, 7, 7, 3, True), (1, 34, 18, 4, 128, 8, 8, 4, False), (5, 31, 15, 3, 72, 6, 5, 5, True),
    (3, 33, 50, 2, 40, 3, 3, 1, False), (40, 64, 66, 3, 64, 7, 7, 3, False), (2, 20, 300, 1, 16, 4, 2, 0, True),
    (2, 40, 24, 3, 136, 7, 7, 3, False), (1, 30, 30, 3, 144, 7, 7, 3, True), (2, 31, 30, 3, 64, 9, 7, 4, False)])
def test_first_layer(nm, ctx, dtype, N, H, W, Cin, Cout, kh, kw, pad, res):  # noqa: F811
    x, w, b, g = operands(N, H, W, Cin, Cout, kh, kw, dtype, H + W)
    Ho, Wo = (H + 2 * pad - kh) // 2 + 1, (W + 2 * pad - kw) // 2 + 1
    r = torch.randn((N, Ho, Wo, Cout), generator=g, device="cuda").to(dtype) if res else None
    conv_both(nm, ctx, x, w, b, 2, pad, r)


@pytest.mark.parametrize("dtype", [torch.float16, torch.bfloat16])
@pytest.mark.parametrize("N,H,W,Cin,Cout,kh,kw,pad", [(40, 64, 66, 3, 64, 7, 7, 3), (16, 224, 224, 3, 64, 7, 7, 3), (9, 100, 70, 4, 128, 8, 8, 4),
                                                      (24, 90, 64, 1, 16, 4, 2, 0), (70, 40, 48, 3, 72, 6, 5, 5), (33, 50, 50, 2, 40, 3, 3, 1)])
@pytest.mark.parametrize("inf", [False, True])
def test_the_forms_of_the_first_layer_agree_in_every_bit(nm, ctx, dtype, N, H, W, Cin, Cout, kh, kw, pad, inf):  # noqa: F811
    """Both take the same 16 products per step of the sum, in the same order of steps."""
    x, w, b, _ = operands(N, H, W, Cin, Cout, kh, kw, dtype, H + W)
    if inf:
        x[0, H // 2, W // 2, 0], x[0, H - 1, 0, Cin - 1] = float("inf"), float("-inf")
    outs = []
    for algo in (nm.ALGO_AUTO, nm.ALGO_TC):
        out = torch.full((N, (H + 2 * pad - kh) // 2 + 1, (W + 2 * pad - kw) // 2 + 1, Cout), float("nan"), device="cuda").to(dtype)
        d = ctx.conv_desc(x, w, out, 2, pad, bias=b, slot=nm.SLOT_RELU, algo=algo)
        ctx.conv2d_pwl(d, torch.empty(ctx.conv2d_workspace_bytes(d), dtype=torch.uint8, device="cuda"))
        ctx.check_device_status()
        outs.append(out.nan_to_num(12345.0))
    assert torch.equal(*outs)


@pytest.mark.parametrize("N,H,Cout,patchwise", [(1, 16, 128, True), (64, 18, 128, True), (512, 16, 64, True), (512, 18, 64, False), (512, 24, 64, True),
                                                (512, 24, 128, False), (64, 34, 64, True), (128, 34, 64, False), (128, 18, 128, False), (512, 32, 128, True), (512, 48, 128, False), (64, 66, 64, True),
                                                (64, 66, 128, False), (64, 100, 128, False), (8, 224, 64, True)])
def test_the_form_follows_the_patches(nm, ctx, N, H, Cout, patchwise):  # noqa: F811
    """Outputs that leave much of a fixed patch empty go to the row pairs (three launches instead of two), with the same result."""
    x, w, b, _ = operands(N, H, H, 3, Cout, 7, 7, torch.float16, H)
    outs = []
    for algo, launches in ((nm.ALGO_AUTO, 2 if patchwise else 3), (nm.ALGO_TC, 3)):
        out = torch.full((N, (H - 1) // 2 + 1, (H - 1) // 2 + 1, Cout), float("nan"), device="cuda").half()
        d = ctx.conv_desc(x, w, out, 2, 3, bias=b, slot=nm.SLOT_RELU, algo=algo)
        ctx.launch_count(reset=True)
        ctx.conv2d_pwl(d, torch.empty(ctx.conv2d_workspace_bytes(d), dtype=torch.uint8, device="cuda"))
        assert ctx.launch_count() == launches
        ctx.check_device_status()
        outs.append(out)
    assert torch.equal(*outs) and outs[0].isfinite().all()


# 136 columns; nine filter rows; outputs that leave too much of a patch empty
@pytest.mark.parametrize("N,H,W,Cin,Cout,kh,kw,pad", [(2, 40, 24, 3, 136, 7, 7, 3), (2, 31, 30, 3, 64, 9, 7, 4), (1, 33, 20, 4, 136, 3, 3, 1),
                                                      (128, 34, 34, 3, 64, 7, 7, 3), (200, 18, 18, 3, 128, 5, 5, 2)])
def test_row_pairs_read_no_row_outside_the_window(nm, ctx, N, H, W, Cin, Cout, kh, kw, pad):  # noqa: F811
    test_gpu_cnn_paths.test_first_layer_reads_no_row_outside_the_window(nm, ctx, N, H, W, Cin, Cout, kh, kw, pad)


# 600 patches each: two channel blocks, whose weights stay in shared memory; three, whose weights pass through a ring; one to compare
@pytest.mark.parametrize("dtype", [torch.float16, torch.bfloat16])
@pytest.mark.parametrize("Cin", [64, 128, 192])
@pytest.mark.parametrize("Cout,res", [(64, False), (40, True)])
def test_halo_of_64_columns(nm, ctx, dtype, Cin, Cout, res):  # noqa: F811
    """Few outputs, so that all products of a patch come from one issuing lane."""
    x, w, b, g = operands(40, 48, 40, Cin, Cout, 3, 3, dtype, Cin)
    r = torch.randn((40, 48, 40, Cout), generator=g, device="cuda").to(dtype) if res else None
    conv_both(nm, ctx, x, w, b, 1, 1, r)

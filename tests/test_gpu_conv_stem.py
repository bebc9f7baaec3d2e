"""GPU parity of the first convolution's forms: the patch-wise one at its edges, the row pairs where the output is wider."""
import pytest
import torch

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

"""GPU parity, the fp32 path: the linear operator on the tensor cores (bf16 terms, K split over clusters) and the plain kernel, attention
with terms and with the score block in shared memory."""
import numpy as np
import pytest
import torch

import nm_inputs
import oracle
from util import assert_close_f32, load_tables_both, to_np

pytestmark = pytest.mark.gpu
# fp32 sums of up to 3072 products: rounding errors add up like sqrt(3072) 2^-24 of the rms = 3.3e-6, six sigma and the
# product of two such factors in attention below this
RTOL = 2e-5


@pytest.fixture(scope="module")
def ctx(nm):
    c = nm.Context(0)
    yield c
    c.close()


def strided(a, pad):
    t = torch.full((a.shape[0], a.shape[1] + pad), float("nan"), device="cuda")
    t[:, :a.shape[1]] = torch.from_numpy(np.ascontiguousarray(a, np.float32)).cuda()
    return t[:, :a.shape[1]]


# rows, columns: one, a thread's and a tile's edges, no multiple of 4; K: less than a chunk, a chunk's, a K-block's and
# both groups' edges, every split
@pytest.mark.parametrize("M,N,K", [(1, 4, 1), (2, 64, 3), (37, 60, 31), (128, 64, 32), (129, 68, 33), (64, 128, 64), (65, 132, 65),
                                   (127, 30, 96), (128, 768, 768), (128, 256, 3072), (333, 1536, 100), (700, 768, 260)])
@pytest.mark.parametrize("epi", ["plain", "gelu_bias", "bias_res", "relu_res_first"])
@pytest.mark.parametrize("algo", [0, 1])
def test_linear(nm, ctx, M, N, K, epi, algo):
    tabs = load_tables_both(ctx, 64, {"gelu": (-4.0, 4.0), "relu": (-3.0, 3.0)})
    A, W = nm_inputs.matrix((M, K), M + K, "f32", 1.0), nm_inputs.matrix((N, K), N, "f32", 0.05)
    rng = np.random.default_rng(K)
    bias = None if epi == "plain" else (0.1 * rng.standard_normal(N)).astype(np.float32)
    res = rng.standard_normal((M, N)).astype(np.float32) if "res" in epi else None
    slot, tab = {"gelu_bias": (nm.SLOT_GELU, "gelu"), "relu_res_first": (nm.SLOT_RELU, "relu")}.get(epi, (nm.SLOT_NONE, None))
    first = epi == "relu_res_first"
    kp, np_ = 4 + -K % 4, 4 + -N % 4
    out = torch.full((M, N + np_), float("nan"), device="cuda")
    ctx.linear_pwl(strided(A, kp), strided(W, kp), out[:, :N], slot=slot, res_first=first, algo=algo,
                   bias=None if bias is None else torch.from_numpy(bias).cuda(), residual=None if res is None else strided(res, np_))
    ctx.check_device_status()
    assert torch.isnan(out[:, N:]).all()
    if first:
        z = np.asarray(oracle.linear(A, W, bias, res, None), np.float64)
        s = np.clip(np.floor(z.astype(np.float32) * np.float32(64 / 6.0) + np.float32(32.0)), 0, 63).astype(int)
        ref = tabs["relu"].k.astype(np.float64)[s] * z + tabs["relu"].b.astype(np.float64)[s]
    else:
        ref = oracle.linear(A, W, bias, res, tabs[tab] if tab else None)
    assert_close_f32(to_np(out[:, :N]), ref, "linear f32 %s" % epi, rtol=RTOL)


# the last length's scores do not fit shared memory: the general kernel's
@pytest.mark.parametrize("B,L,h,pad", [(1, 1, 1, 0), (2, 31, 2, 0), (1, 33, 3, 4), (2, 64, 1, 0), (1, 65, 2, 0), (3, 100, 2, 8),
                                       (2, 128, 4, 0), (1, 333, 2, 0), (1, 1300, 1, 0), (1, 1500, 1, 0)])
@pytest.mark.parametrize("n", [16, 256])
@pytest.mark.parametrize("algo", [0, 1])
def test_attention(ctx, B, L, h, pad, n, algo):
    tabs = load_tables_both(ctx, n, {"exp": (-8.0, 0.0), "recip": (max(L / 16.0, 0.5), float(max(L, 2)))})
    H = h * 64
    qkv = nm_inputs.matrix((B * L, 3 * H), L + h, "f32", 1.0)
    qkv[:, :2 * H] *= 0.8
    out = torch.full((B * L + 1, H), float("nan"), device="cuda")
    ctx.attention_pwl(strided(qkv, pad), out, B, L, h, 64, algo=algo)
    ctx.check_device_status()
    assert torch.isnan(out[B * L:]).all()
    ref = oracle.attention(qkv, B, L, h, 64, tabs["exp"], tabs["recip"])
    assert_close_f32(to_np(out[:B * L]), ref, "attention f32 L=%d" % L, rtol=RTOL)


def test_the_plain_kernels_can_be_forced(nm, ctx):
    """algo 1 is another kernel than the one chosen: fp32 sums in another order show in the last bits."""
    load_tables_both(ctx, 64, {"exp": (-8.0, 0.0), "recip": (8.0, 128.0)})
    A, W = [torch.from_numpy(nm_inputs.matrix(s, 3, "f32", 1.0)).cuda() for s in ((128, 768), (256, 768))]
    lin = [torch.empty(128, 256, device="cuda") for _ in range(2)]
    qkv = torch.from_numpy(nm_inputs.matrix((128, 192), 4, "f32", 1.0)).cuda()
    att = [torch.empty(128, 64, device="cuda") for _ in range(2)]
    for algo in (nm.ALGO_AUTO, nm.ALGO_SIMT):
        ctx.linear_pwl(A, W, lin[algo], algo=algo)
        ctx.attention_pwl(qkv, att[algo], 1, 128, 1, 64, algo=algo)
    ctx.check_device_status()
    assert not torch.equal(*lin) and not torch.equal(*att)


def test_first_calls_from_several_threads(nm):
    """The first fp32 products of a context, on a stream per thread."""
    import threading
    ctx = nm.Context(0)
    try:
        A, W = [torch.from_numpy(nm_inputs.matrix(s, 3, "f32", 1.0)).cuda() for s in ((100, 768), (768, 768))]
        outs = [torch.zeros(100, 768, device="cuda") for _ in range(8)]
        streams = [torch.cuda.Stream() for _ in outs]
        torch.cuda.synchronize()
        threads = [threading.Thread(target=lambda o=o, s=s: ctx.linear_pwl(A, W, o, stream=s)) for o, s in zip(outs, streams)]
        for t in threads:
            t.start()
        for t in threads:
            t.join()
        torch.cuda.synchronize()
        assert all(torch.equal(o, outs[0]) for o in outs) and outs[0].abs().sum() > 0
    finally:
        ctx.close()

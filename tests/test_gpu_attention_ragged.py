"""GPU parity, attention at sequence lengths that are not a multiple of 128 (masked last block, probabilities as sums of
16-bit terms)."""
import numpy as np
import pytest
import torch

import nm_inputs
import oracle
from util import load_tables_both, rms_rel, to_np

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx(nm):
    c = nm.Context(0)
    yield c
    c.close()


def run(ctx, dtype, B, L, h, seed, pad=0, n=64, exp_range=(-8.0, 0.0), score_shift=0.0):
    tabs = load_tables_both(ctx, n, {"exp": exp_range, "recip": (max(L / 16.0, 0.5), float(max(L, 2)))})
    H, td = h * 64, nm_inputs.torch_dtype(dtype)
    qkv = nm_inputs.matrix((B * L, 3 * H), seed, dtype, 1.0)
    qkv[:, :2 * H] *= 0.8
    if score_shift:   # every score far below zero: a zero-filled key beyond L would be the row's largest
        qkv[:, :H] += score_shift
        qkv[:, H:2 * H] -= score_shift
    qkv = nm_inputs.round_to(qkv, dtype)
    buf = torch.zeros((B * L, 3 * H + pad), dtype=td, device="cuda")
    buf[:, :3 * H] = torch.from_numpy(qkv).cuda().to(td)
    out = torch.full((B * L + 1, H), float("nan"), dtype=td, device="cuda")
    ctx.attention_pwl(buf[:, :3 * H], out, B, L, h, 64)
    ctx.check_device_status()
    assert torch.isnan(out[B * L:].float()).all()   # nothing is written beyond the last row
    ref = oracle.attention(qkv, B, L, h, 64, tabs["exp"], tabs["recip"])
    return to_np(out[:B * L]), ref


def check(got, ref, dtype):
    """The result's own rounding to the storage type is at most 2^-8 (bf16) or 2^-11 (fp16) of each element, its rms over
    many elements at most 1/sqrt(3) of that; the probabilities add nothing / 2^-22 and the fp32 sums little more."""
    half_ulp = {"bf16": 2.0 ** -8, "f16": 2.0 ** -11}[dtype]
    assert np.all(np.isfinite(got))
    rms = np.sqrt(np.mean(ref * ref))
    assert np.all(np.abs(got - ref) <= half_ulp * 1.01 * np.abs(ref) + 2e-5 * rms + 2.0 ** -25), np.abs(got - ref).max()
    if got.size >= 1024:
        assert rms_rel(got, ref) <= half_ulp / np.sqrt(3.0)


@pytest.mark.parametrize("dtype", ["bf16", "f16"])
@pytest.mark.parametrize("B,L,h,pad", [(1, 1, 1, 0), (2, 7, 2, 0), (1, 37, 12, 0), (3, 63, 1, 8), (1, 64, 2, 0), (2, 65, 3, 0),
                                       (2, 96, 1, 0), (1, 127, 2, 16), (2, 129, 2, 0), (1, 191, 1, 0), (1, 193, 2, 0),
                                       (2, 333, 3, 0), (1, 511, 2, 0), (1, 1000, 1, 0)])
def test_lengths(ctx, dtype, B, L, h, pad):
    check(*run(ctx, dtype, B, L, h, seed=L + h, pad=pad), dtype)


def test_masked_keys_are_not_the_maximum(ctx):
    got, ref = run(ctx, "bf16", 1, 70, 2, seed=5, score_shift=1.0)
    check(got, ref, "bf16")


@pytest.mark.parametrize("n,exp_range", [(16, (-8.0, 0.0)), (256, (-8.0, 0.0)), (64, (-6.0, -0.5))])
def test_tables(ctx, n, exp_range):
    """Small and large tables, and one whose range ends below zero (the upper clamp)."""
    check(*run(ctx, "bf16", 2, 150, 2, seed=n, n=n, exp_range=exp_range), "bf16")


def test_several_tiles_per_cta(ctx):
    """More tiles than resident CTAs (two per SM): barrier phases run on from tile to tile, odd counts per tile."""
    B, L, h = 12, 190, 16
    assert B * h * 2 > 2 * torch.cuda.get_device_properties(0).multi_processor_count
    check(*run(ctx, "bf16", B, L, h, seed=3), "bf16")


def test_forced_streaming_kernel_still_takes_multiples_of_128_only(nm, ctx):
    q = torch.zeros(100, 192, dtype=torch.bfloat16, device="cuda")
    with pytest.raises(nm.NmError) as ei:
        ctx.attention_pwl(q, torch.zeros(100, 64, dtype=torch.bfloat16, device="cuda"), 1, 100, 1, 64, algo=nm.ALGO_TC)
    assert ei.value.code == 5


@pytest.mark.parametrize("dtype", ["bf16", "f16"])
@pytest.mark.parametrize("L", [1, 33, 100, 200, 333])
def test_infinite_values(nm, ctx, dtype, L):
    """An infinite V element gives an infinity in its channel, as on the CUDA cores, wherever no NaN comes in; other channels
    do not see it."""
    load_tables_both(ctx, 64, {"exp": (-8.0, 0.0), "recip": (max(L / 16.0, 0.5), float(max(L, 2)))})
    B, h, td = 2, 2, nm_inputs.torch_dtype(dtype)
    H = 64 * h
    qkv = nm_inputs.matrix((B * L, 3 * H), L, dtype, 1.0)
    qkv[:, :2 * H] *= 0.5
    v = qkv[:, 2 * H:]
    v[0, 3], v[L - 1, 5], v[L // 2, 70], v[L + L // 3, 64], v[L, 9] = np.inf, -np.inf, np.inf, -np.inf, np.nan
    outs = []
    for algo in (nm.ALGO_AUTO, nm.ALGO_SIMT):
        out = torch.zeros((B * L, H), dtype=td, device="cuda")
        ctx.attention_pwl(torch.from_numpy(qkv).cuda().to(td), out, B, L, h, 64, algo=algo)
        ctx.check_device_status()
        outs.append(to_np(out))
    got, want = outs
    assert np.isinf(want[:, [3, 5, 70, 64]]).any() and np.isnan(want[L:, 9]).all()
    assert np.array_equal(np.isnan(got), np.isnan(want))
    inf = np.isinf(want)
    assert np.array_equal(got[inf], want[inf])
    rest = np.isfinite(want)
    assert np.all(np.abs(got[rest] - want[rest]) <= {"bf16": 2.0 ** -7, "f16": 2.0 ** -10}[dtype] * np.abs(want[rest]) + 1e-5)


def test_probabilities_keep_their_bits(nm, ctx):
    """Outputs that are not the correctly rounded float64 result: with probabilities of 16 bits they were 2.4e-3 of all; the
    CUDA-core kernel, whose probabilities are fp32, has 2.6e-4."""
    B, L, h = 4, 333, 12
    ek, eb = ctx.load_function_table(nm.SLOT_EXP, nm.FUNC_EXP, 64, -8.0, 0.0)
    rk, rb = ctx.load_function_table(nm.SLOT_RECIP, nm.FUNC_RECIP, 64, L / 16.0, float(L))
    g = torch.Generator(device="cuda").manual_seed(1)
    qkv = torch.randn((B * L, 3 * 64 * h), generator=g, device="cuda")
    qkv[:, :2 * 64 * h] *= 0.8
    qkv = qkv.bfloat16()
    q, k, v = [t.double().view(B, L, h, 64).transpose(1, 2) for t in qkv.split(64 * h, 1)]

    def pwl(x, lo, hi, kk, bb):
        kk, bb = [torch.tensor(t, device="cuda", dtype=torch.float64) for t in (kk, bb)]
        i = ((x - lo) * (64 / (hi - lo))).floor().clamp(0, 63).long()
        return kk[i] * x + bb[i]

    s = (q @ k.transpose(-1, -2)) * 0.125
    e = pwl(s - s.amax(-1, keepdim=True), -8.0, 0.0, ek, eb)
    o = (e @ v) * pwl(e.sum(-1, keepdim=True), L / 16.0, float(L), rk, rb)
    want = o.transpose(1, 2).reshape(B * L, 64 * h).bfloat16()
    out = torch.empty_like(want)
    ctx.attention_pwl(qkv, out, B, L, h, 64)
    ctx.check_device_status()
    assert (out != want).double().mean() < 4e-4


@pytest.mark.parametrize("dtype", [torch.bfloat16, torch.float16])
@pytest.mark.parametrize("L", [1, 16, 17, 33, 48, 49, 64, 100, 127, 128])
@pytest.mark.parametrize("exp_range", [(-8.0, 0.0), (-6.0, -0.5)])
def test_sequences_do_not_depend_on_the_batch(ctx, dtype, L, exp_range):
    """One or two softmax warps, one or two CTAs per SM: the form follows the number of (batch, head) pairs, every bit stays."""
    h, most = 12, 30   # 12, 144, 156, 288, 300 and 360 pairs on 148 SMs
    load_tables_both(ctx, 64, {"exp": exp_range, "recip": (max(L / 16.0, 0.5), float(max(L, 2)))})
    g = torch.Generator(device="cuda").manual_seed(L)
    x = (torch.randn((most * L, 3 * 64 * h), generator=g, device="cuda") * 0.8).to(dtype)
    outs = []
    for B in (most, 25, 24, 13, 12, 1):
        out = torch.full((most * L, 64 * h), float("nan"), device="cuda").to(dtype)
        ctx.attention_pwl(x, out, B, L, h, 64)
        ctx.check_device_status()
        assert out[:B * L].isfinite().all() and out[B * L:].isnan().all()
        outs.append(out[:B * L])
    assert all(torch.equal(outs[0][:o.shape[0]], o) for o in outs)

"""GPU parity, fp32 products as bf16 terms on the tensor cores: precision, the ends of the exponent range, infinities and NaN."""
import numpy as np
import pytest
import torch

import nm_inputs
from util import load_tables_both

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx(nm):
    c = nm.Context(0)
    yield c
    c.close()


def linear(ctx, A, W, algo=0):
    out = torch.full((A.shape[0], W.shape[0]), float("nan"), device="cuda")
    ctx.linear_pwl(A, W, out, algo=algo)
    ctx.check_device_status()
    return out


# one CTA, both tile widths, splits, remainders of rows, columns and K
@pytest.mark.parametrize("M,N,K", [(5, 8, 40), (128, 64, 64), (129, 196, 132), (300, 512, 2048), (1000, 1600, 768), (128, 768, 3072), (2000, 2304, 260)])
def test_linear_precision(ctx, M, N, K):
    """Four truncated steps of a sum, 4 * 1.55e-8, a chain of K / 64 rounded additions, 7.4e-9 sqrt(K / 64), and the rounding of the
    result, 2.5e-8, all relative to the sums' rms.  They are added up, since the truncations all go towards zero."""
    A, W = [torch.from_numpy(nm_inputs.matrix(s, K, "f32", d)).cuda() for s, d in (((M, K), 1.0), ((N, K), 0.02))]
    ref = A.double() @ W.double().t()
    err = ((linear(ctx, A, W).double() - ref).norm() / ref.norm()).item()
    assert err < 4 * 1.55e-8 + 7.4e-9 * (K / 64) ** 0.5 + 2.5e-8


@pytest.mark.parametrize("M,N", [(64, 256), (1024, 768)])
@pytest.mark.parametrize("K", [16, 64, 768, 3072])
@pytest.mark.parametrize("kind", ["normal", "positive", "uniform"])
def test_linear_is_no_less_accurate_than_a_chain_of_fmas(nm, ctx, M, N, K, kind):
    """Operands of one sign, too, where the truncations do not average out: test_linear_precision's bound, and the plain kernel's error
    (measured: at most 1.2e-7 against 6e-8 at K = 16 to 1e-6 at K = 3072)."""
    A, W = [torch.from_numpy(nm_inputs.matrix(s, K, "f32", d)).cuda() for s, d in (((M, K), 1.0), ((N, K), 0.02))]
    if kind != "normal":
        A, W = A.abs(), W.abs()
    if kind == "uniform":   # the fractional part of a wide normal distribution
        A, W = (50 * A).frac(), (2500 * W).frac()
    ref = A.double() @ W.double().t()
    errs = [((linear(ctx, A, W, algo).double() - ref).norm() / ref.norm()).item() for algo in (nm.ALGO_AUTO, nm.ALGO_SIMT)]
    assert errs[0] < 4 * 1.55e-8 + 7.4e-9 * (K / 64) ** 0.5 + 2.5e-8 and errs[0] < errs[1], errs


@pytest.mark.parametrize("e", [-126, -128, -130, -133, -136])
def test_linear_of_subnormal_operands(ctx, e):
    """The first term of an operand of 2^-126 2^-n has 8 - n bits, so the products that are left out are up to 2^(n - 26) of
    the whole one, at most 2^-18; the operand itself is a multiple of 2^(n - 23) of its size."""
    A, W = [torch.from_numpy(nm_inputs.matrix(s, 7, "f32", 1.0)).cuda() for s in ((72, 200), (68, 200))]
    A = (A.sign().double() * (1 + A.abs().double() % 1) * 2.0 ** e).float()
    ref = A.double() @ W.double().t()
    for got, want in ((linear(ctx, A, W * 2.0 ** 100), ref * 2.0 ** 100), (linear(ctx, W * 2.0 ** 100, A), ref.t() * 2.0 ** 100)):
        assert ((got.double() - want).norm() / want.norm()).item() < 1e-7 + 2.0 ** (min(-126 - e, 8) - 26)


# K that ends in a K-block of 64: within a group of four, at its end, one block and several, one CTA and splits; rows and columns cut off
@pytest.mark.parametrize("K", [1, 2, 3, 4, 5, 15, 63, 65, 66, 127, 130, 199, 1031])
@pytest.mark.parametrize("M,N", [(1, 4), (130, 68), (2000, 1540)])
def test_linear_partial_k_block(nm, ctx, M, N, K):
    """What lies behind a row's end is neither added nor, behind the last row, read (the tensors end there).  Each sum's error is bounded
    by the magnitudes of its products, since single sums, of which there may be few, can be small: four truncations of 2^-23, a chain of K / 64
    roundings, that of the result and what is left out, 2^-24 each."""
    kp = K + -K % 4
    A, W = [torch.full(((r - 1) * kp + K + 1,), float("nan"), device="cuda")[:-1] for r in (M, N)]
    a, w = [torch.as_strided(t, (r, K), (kp, 1)) for t, r in ((A, M), (W, N))]
    a.copy_(torch.from_numpy(nm_inputs.matrix((M, K), K, "f32", 1.0)))
    w.copy_(torch.from_numpy(nm_inputs.matrix((N, K), K + 1, "f32", 0.02)))
    ref = a.double() @ w.double().t()
    size = a.double().abs() @ w.double().abs().t()
    assert ((linear(ctx, a, w).double() - ref).abs() <= (4 * 2.0 ** -23 + (K / 64 + 3) * 2.0 ** -24) * size).all()


@pytest.mark.parametrize("a_exp,w_exp", [(0, 0), (-118, 100), (-122, 100), (100, -122), (-110, 0), (0, -110), (-110, 100), (40, 40), (100, -100)])
def test_linear_exponents(ctx, a_exp, w_exp):
    """The terms' scaling keeps the range of fp32: the same result times a power of two."""
    A, W = [torch.from_numpy(nm_inputs.matrix(s, 7, "f32", 1.0)).cuda() for s in ((70, 200), (68, 200))]
    A, W = A.sign() * (A.abs() + 0.1), W.sign() * (W.abs() + 0.1)
    base = linear(ctx, A, W)
    got = linear(ctx, A * 2.0 ** a_exp, W * 2.0 ** w_exp)
    assert torch.equal(got, base * 2.0 ** (a_exp + w_exp))


@pytest.mark.parametrize("M,N,K", [(37, 60, 100), (200, 132, 320)])
def test_linear_not_finite(nm, ctx, M, N, K):
    A, W = [torch.from_numpy(nm_inputs.matrix(s, 9, "f32", 1.0)).cuda() for s in ((M, K), (N, K))]
    big = torch.finfo(torch.float32).max
    for i, v in enumerate([float("inf"), -float("inf"), float("nan"), big, -big]):
        A[3 * i, (7 * i + 1) % K] = v
        W[2 * i + 1, (11 * i + 5) % K] = v
    W[20, :] = 0
    W[20, 1] = 0.25   # exact in bf16: its lower terms are zero
    got, ref = linear(ctx, A, W), linear(ctx, A, W, nm.ALGO_SIMT)
    assert torch.equal(got.isnan(), ref.isnan()) and torch.equal(got.isinf(), ref.isinf())
    assert torch.equal(got[got.isinf()], ref[got.isinf()]) and ref.isinf().any() and ref.isnan().any()
    f = ref.isfinite()
    assert ((got - ref)[f].abs() <= 1e-5 * ref[f].abs().clamp(min=K ** 0.5)).all()


# every sum of the tile by FMAs: remainders of rows, columns and K (of a row's last three k, too), one CTA and splits, both widths
@pytest.mark.parametrize("M,N,K", [(1, 4, 7), (33, 36, 30), (128, 64, 64), (129, 100, 161), (200, 132, 320), (300, 512, 2048), (1000, 1600, 70)])
def test_linear_of_large_operands(ctx, M, N, K):
    """From 2^112 on a term of an operand is infinite, the product itself is not."""
    A, W = [torch.from_numpy(nm_inputs.matrix(s, K, "f32", 1.0)).cuda() for s in ((M, K + -K % 4), (N, K + -K % 4))]
    A[:, K:], W[:, K:] = float("nan"), float("inf")
    A, W = (A * 2.0 ** 124)[:, :K], (W * 2.0 ** -100)[:, :K]
    got, ref = linear(ctx, A, W), A.double() @ W.double().t()
    # a chain of K rounded sums: 2^-24 of the running sum each, at most 2^-24 sqrt(K) of the rms here
    assert ((got.double() - ref).norm() / ref.norm()).item() < 2.0 ** -24 * K ** 0.5 + 2.0 ** -24


def time_of(call):
    graph, side = torch.cuda.CUDAGraph(), torch.cuda.Stream()
    call()
    side.wait_stream(torch.cuda.current_stream())
    with torch.cuda.graph(graph, stream=side):
        for _ in range(20):
            call()
    times = []
    for _ in range(5):
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        a.record()
        graph.replay()
        b.record()
        torch.cuda.synchronize()
        times.append(a.elapsed_time(b))
    return min(times)


@pytest.mark.parametrize("M,N,K", [(1024, 768, 3072), (37, 768, 3072), (128, 768, 256)])
def test_not_finite_linear_takes_no_longer_than_a_plain_product(ctx, M, N, K):
    """2 to 6 times the finite product with one row, up to 11 with all; element by element it was 50 (one row) to 600 times."""
    A, W = [torch.from_numpy(nm_inputs.matrix(s, 9, "f32", 1.0)).cuda() for s in ((M, K), (N, K))]
    out = torch.empty(M, N, device="cuda")
    finite = time_of(lambda: ctx.linear_pwl(A, W, out))
    for rows, value in ((slice(5, 6), float("nan")), (slice(None), float("nan")), (slice(None), float("inf"))):
        odd = A.clone()
        odd[rows] = value
        assert time_of(lambda: ctx.linear_pwl(odd, W, out)) < 16 * finite


@pytest.mark.parametrize("L", [1, 15, 16, 17, 64, 65, 100, 128])
@pytest.mark.parametrize("n", [2, 64, 256])
@pytest.mark.parametrize("odd", [None, "q", "k", "v", "large_v"])
def test_attention(nm, ctx, L, n, odd):
    """Against the CUDA-core kernel; one head of three has an operand that takes it off the tensor cores."""
    B, h = 2, 3
    load_tables_both(ctx, n, {"exp": (-8.0, 0.0), "recip": (max(L / 16.0, 0.5), float(max(L, 2)))})
    x = torch.from_numpy(nm_inputs.matrix((B * L, 3 * h * 64), L, "f32", 0.8)).cuda()
    if odd:
        col = {"q": 64, "k": 3 * 64 + 64, "v": 6 * 64 + 64, "large_v": 6 * 64 + 64}[odd]
        # (an infinite key's exponential is -inf, the extension of the table's first line; what comes of its infinite sum depends on
        # where the reciprocal is multiplied)
        x[L - 1, col + 5] = {"large_v": 1e30, "k": float("nan")}.get(odd, float("inf"))
    outs = []
    for algo in (nm.ALGO_AUTO, nm.ALGO_SIMT):
        out = torch.full((B * L + 1, h * 64), float("nan"), device="cuda")
        ctx.attention_pwl(x, out, B, L, h, 64, algo=algo)
        ctx.check_device_status()
        assert out[B * L:].isnan().all()
        outs.append(out[:B * L].cpu().numpy().astype(np.float64))
    got, ref = outs
    assert (np.isnan(got) == np.isnan(ref)).all() and (np.isinf(got) == np.isinf(ref)).all()
    assert (got[np.isinf(ref)] == ref[np.isinf(ref)]).all()
    f = np.isfinite(ref)
    # two products of up to 128 terms and a table slope of up to n segments' rounding each; the odd head's own size
    scale = np.maximum(np.abs(ref), np.where(f, 1.0, 0.0) * 0.05)
    with np.errstate(invalid="ignore"):
        row = np.max(np.where(f, np.abs(ref), 0.0), axis=1, keepdims=True)
    assert (np.abs(got - ref)[f] <= (2e-5 * np.maximum(scale, row))[f]).all()


@pytest.mark.parametrize("L", [1, 16, 17, 33, 64, 65, 100, 128, 200])
@pytest.mark.parametrize("positive", [False, True])
@pytest.mark.parametrize("B", [4, 16])
def test_attention_precision(nm, ctx, B, L, positive):
    """Against float64 with the same tables.  B 4: the tensor cores up to L = 128, 0.6e-7 to 1.2e-7 measured (without the products m m', h l', l h' of P V
    it would be 2e-6); the tiled kernel beyond and, with 192 heads, up to 64 keys: 1.0e-7 to 1.9e-7, 2.8e-7 with 200.  The plain kernel has more."""
    h = 12
    tabs = load_tables_both(ctx, 64, {"exp": (-8.0, 0.0), "recip": (max(L / 16.0, 0.5), float(max(L, 2)))})
    x = torch.from_numpy(nm_inputs.matrix((B * L, 3 * h * 64), L, "f32", 0.8)).cuda()
    if positive:
        x[:, 2 * h * 64:].abs_()
    q, k, v = [t.double().view(B, L, h, 64).transpose(1, 2) for t in x.split(h * 64, 1)]

    def pwl(z, name, lo, hi):
        kk, bb = [torch.from_numpy(t).cuda().double() for t in (tabs[name].k, tabs[name].b)]
        i = ((z - lo) * (64 / (hi - lo))).floor().clamp(0, 63).long()
        return kk[i] * z + bb[i]

    s = (q @ k.transpose(-1, -2)) * 0.125
    e = pwl(s - s.amax(-1, keepdim=True), "exp", -8.0, 0.0)
    ref = ((e @ v) * pwl(e.sum(-1, keepdim=True), "recip", max(L / 16.0, 0.5), float(max(L, 2)))).transpose(1, 2).reshape(B * L, h * 64)
    errs = []
    for algo in (nm.ALGO_AUTO, nm.ALGO_SIMT):
        out = torch.full((B * L, h * 64), float("nan"), device="cuda")
        ctx.attention_pwl(x, out, B, L, h, 64, algo=algo)
        ctx.check_device_status()
        errs.append(((out.double() - ref).norm() / ref.norm()).item())
    terms = L <= 128 and (L > 64 or B * h <= 148)
    assert errs[0] < (1.5e-7 if terms else 2.5e-7 if L <= 128 else 3.5e-7) and errs[0] < 1.03 * errs[1], errs


@pytest.mark.parametrize("L", [37, 128, 200])
def test_attention_replay_takes_the_table_of_its_time(ctx, L):
    """A launch captured with a small exp table and replayed with a large one."""
    B, h = 2, 3
    ranges = {"exp": (-8.0, 0.0), "recip": (L / 16.0, float(L))}
    x = torch.from_numpy(nm_inputs.matrix((B * L, 3 * h * 64), L, "f32", 0.8)).cuda()
    out, ref = torch.zeros(B * L, h * 64, device="cuda"), torch.zeros(B * L, h * 64, device="cuda")
    load_tables_both(ctx, 16, ranges)
    ctx.attention_pwl(x, out, B, L, h, 64)
    graph, side = torch.cuda.CUDAGraph(), torch.cuda.Stream()
    side.wait_stream(torch.cuda.current_stream())
    with torch.cuda.graph(graph, stream=side):
        ctx.attention_pwl(x, out, B, L, h, 64)
    torch.cuda.synchronize()
    load_tables_both(ctx, 256, ranges)
    ctx.attention_pwl(x, ref, B, L, h, 64)
    graph.replay()
    torch.cuda.synchronize()
    ctx.check_device_status()
    assert torch.equal(out, ref)


@pytest.mark.parametrize("B,L", [(8, 128), (8, 37)])
def test_not_finite_attention_takes_no_longer_than_a_plain_one(ctx, B, L):
    """Products on the CUDA cores: 2 to 4 times the finite call; with each operand from memory it was 40 times."""
    h = 12
    load_tables_both(ctx, 64, {"exp": (-8.0, 0.0), "recip": (L / 16.0, float(L))})
    x = torch.from_numpy(nm_inputs.matrix((B * L, 3 * h * 64), L, "f32", 0.8)).cuda()
    out = torch.empty(B * L, h * 64, device="cuda")
    finite = time_of(lambda: ctx.attention_pwl(x, out, B, L, h, 64))
    x[:, 5::64] = float("nan")
    assert time_of(lambda: ctx.attention_pwl(x, out, B, L, h, 64)) < 8 * finite


@pytest.mark.parametrize("B,L", [(64, 16), (64, 37), (128, 64), (12, 64), (13, 64), (64, 65)])
def test_short_attention_of_many_heads(nm, ctx, B, L):
    """On both sides of the line between the kernels; the whole tensor of each against the plain kernel."""
    h = 12
    load_tables_both(ctx, 64, {"exp": (-8.0, 0.0), "recip": (L / 16.0, float(L))})
    x = torch.from_numpy(nm_inputs.matrix((B * L, 3 * h * 64), L, "f32", 0.8)).cuda()
    outs = []
    for algo in (nm.ALGO_AUTO, nm.ALGO_SIMT):
        out = torch.full((B * L, h * 64), float("nan"), device="cuda")
        ctx.attention_pwl(x, out, B, L, h, 64, algo=algo)
        ctx.check_device_status()
        outs.append(out.double())
    # both off by less than 3e-7 of the rms against float64
    assert ((outs[0] - outs[1]).norm() / outs[1].norm()).item() < 6e-7


@pytest.mark.parametrize("L", [16, 37, 64])
def test_short_attention_takes_more_heads_in_proportion(ctx, L):
    """1536 (batch, head) pairs take about 5 to 8 times as long as 96, which do not fill the GPU; a CTA per SM for each pair took 10 to 11 times."""
    h = 12
    load_tables_both(ctx, 64, {"exp": (-8.0, 0.0), "recip": (L / 16.0, float(L))})
    x = torch.from_numpy(nm_inputs.matrix((128 * L, 3 * h * 64), L, "f32", 0.8)).cuda()
    out = torch.empty(128 * L, h * 64, device="cuda")
    few, many = [time_of(lambda: ctx.attention_pwl(x, out, B, L, h, 64)) for B in (8, 128)]
    assert many < 9 * few

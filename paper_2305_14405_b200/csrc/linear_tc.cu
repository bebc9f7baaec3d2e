// Host side of the tensor-core linear operator: kernel and tile selection, tensor maps and launch of
// linear_tc_kernel (linear_tc_kernel.cuh) or linear_split_kernel (linear_split_kernel.cuh) for matrices in memory.
#include "linear_split_kernel.cuh"

using namespace nm_tc;

namespace {

void fill_args(nm_ctx* ctx, const nm_linear_desc* d, NmChain chain, TcArgs* a)
{
    memset(a, 0, sizeof(*a));
    a->M = d->M; a->N = d->N; a->K = d->K;
    a->bias = d->bias;
    a->has_res = d->residual ? 1 : 0;
    a->res_first = d->res_first;
    a->tab = d->slot == NM_SLOT_NONE ? nullptr : ctx->d_tables + d->slot;
    a->n_seg = d->slot == NM_SLOT_NONE ? 0 : ctx->h_tables[d->slot].n;
    a->a_scale = d->a_scale; a->w_scale = d->w_scale; a->inv_out_scale = d->inv_out_scale;
    a->acc_dump = d->acc_dump; a->idx_dump = d->idx_dump;
    a->status = ctx->d_status;
    a->weights_ready = chain.weights_ready;
    a->late_trigger = chain.late_trigger;
}

template <typename InT, typename OutT, bool TWO, int BN>
nm_status launch(nm_ctx* ctx, const nm_linear_desc* d, int steps, NmChain chain, cudaStream_t st)
{
    constexpr int B_ROWS = TWO ? BN / 2 : BN;
    constexpr int TILE_M = TWO ? 2 * BM : BM;
    TcArgs a;
    fill_args(ctx, d, chain, &a);
    const int bk = ROW_BYTES / (int)sizeof(InT);
    const int64_t m_tiles = (d->M + TILE_M - 1) / TILE_M;
    a.num_n_tiles = (int)((d->N + BN - 1) / BN);
    if (m_tiles * a.num_n_tiles > 0x7fffffffLL) return NM_ERR_SHAPE;
    a.num_tiles = (int)(m_tiles * a.num_n_tiles);
    a.num_k_blocks = (int)((d->K + bk - 1) / bk);
    a.acc_steps = steps;
    a.accs = steps ? (4 * a.num_k_blocks + steps - 1) / steps : 1;
    // Weights of 2 MB and less stay in L2 from pass to pass unless the stack is very deep, and asking for them then costs up to 1.5 %
    // (7 layers, 432 tokens, H 512: 356 against 361 us; ResNet-50 batch 7: 964 and 977); larger ones do not: 12 layers, 7 x 333
    // tokens, 170 MB of weights: 1008 -> 998 us, int8 24 layers, 128 tokens, 300 MB: 870 -> 859.
    a.prefetch_w = chain.weights_ready && !chain.back_to_back && d->N * d->K * (int64_t)sizeof(InT) > (2 << 20);
    size_t smem = 0;
    if (!plan_smem<InT, TWO, BN>(&a, d->bias || TcIn<InT>::is_int, &smem)) return NM_ERR_UNSUPPORTED;

    CUtensorMap tmA, tmW, tmO, tmR;
    nm_status s = make_tmap(ctx, &tmA, d->A, d->in_dtype, d->M, d->K, d->lda, BM);
    if (s != NM_OK) return s;
    s = make_tmap(ctx, &tmW, d->W, d->in_dtype, d->N, d->K, d->ldw, B_ROWS);
    if (s != NM_OK) return s;
    s = make_tmap(ctx, &tmO, d->out, d->out_dtype, d->M, d->N, d->ldo, 32);
    if (s != NM_OK) return s;
    if (d->residual) s = make_tmap(ctx, &tmR, d->residual, d->out_dtype, d->M, d->N, d->ldr, 32);
    else tmR = tmO;
    if (s != NM_OK) return s;
    return launch_kernel<InT, OutT, TWO, BN, false>(ctx, tmA, tmW, tmO, tmR, a, smem,
                                                    2.0 * (double)d->M * (double)d->N * (double)d->K, st);
}

template <typename InT, typename OutT, int BN>
nm_status launch_split(nm_ctx* ctx, const nm_linear_desc* d, const TileChoice& c, NmChain chain, cudaStream_t st)
{
    const int S = c.S;
    const int bk = ROW_BYTES / (int)sizeof(InT);
    const int64_t k_blocks = (d->K + bk - 1) / bk, n_tiles = (d->N + BN - 1) / BN, tiles = (d->M + BM - 1) / BM * n_tiles;
    SplitArgs s;
    memset(&s, 0, sizeof(s));
    if (tiles > 0x7fffffffLL / S) return NM_ERR_SHAPE;
    s.S = S;
    fill_args(ctx, d, chain, &s.t);
    s.t.acc_steps = c.steps;
    s.t.num_n_tiles = (int)n_tiles;
    s.t.num_tiles = (int)tiles;
    s.t.num_k_blocks = (int)k_blocks;
    s.residual = d->residual; s.ldr = d->ldr;
    s.out = d->out; s.ldo = d->ldo;
    CUtensorMap tmA, tmW;
    nm_status e = make_tmap(ctx, &tmA, d->A, d->in_dtype, d->M, d->K, d->lda, BM);
    if (e != NM_OK) return e;
    e = make_tmap(ctx, &tmW, d->W, d->in_dtype, d->N, d->K, d->ldw, BN);
    if (e != NM_OK) return e;
    return launch_split_kernel<InT, OutT, BN, false>(ctx, tmA, tmW, s, chain.back_to_back, 2.0 * (double)d->M * (double)d->N * (double)d->K, st);
}

// Kernel and tile for d: the cheapest by the model (like_fma: with accumulators as good as a chain of fp32 FMAs), or a forced one, with algo 2 and 3 the persistent kernel with a tile by the width
// alone; algo 3 asks for one CTA per tile, otherwise CTA pairs from one 256-row tile on.
template <typename InT, typename OutT>
TileChoice choose(nm_ctx* ctx, const nm_linear_desc* d, bool like_fma, NmChain chain)
{
    constexpr bool NARROW = !TcIn<InT>::is_int;   // tiles of 64 and 128 columns are built for the 16-bit types
    const bool whole_chunks = d->N * sizeof(OutT) % 16 == 0;
    const int bk = ROW_BYTES / (int)sizeof(InT);
    if (nm_algo_is_split(d->algo)) return forced_split(d->algo, (d->K + bk - 1) / bk);
    if (nm_algo_forced(d->algo) && whole_chunks)
        return {0, NARROW && d->N <= 64 ? 64 : (NARROW && d->N <= 128 ? 128 : 256), d->algo != 3 && d->M >= 256, 0.0, 0};
    const EpiNeeds epi = {d->slot == NM_SLOT_NONE ? 0 : ctx->h_tables[d->slot].n, d->residual != nullptr, d->bias != nullptr || TcIn<InT>::is_int};
    return choose_tile(d->M, (d->M + BM - 1) / BM, d->N, (d->K + bk - 1) / bk, NARROW, epi, false, whole_chunks, like_fma ? (d->K + 15) / 16 : 0, chain,
                       ctx->sm_count);
}

template <typename InT, typename OutT>
nm_status launch_choice(nm_ctx* ctx, const nm_linear_desc* d, const TileChoice& c, NmChain chain, cudaStream_t st)
{
    if (c.S) return c.BN == 32 ? launch_split<InT, OutT, 32>(ctx, d, c, chain, st) : launch_split<InT, OutT, 64>(ctx, d, c, chain, st);
    if constexpr (!TcIn<InT>::is_int) {
        if (c.BN == 64) return c.two ? launch<InT, OutT, true, 64>(ctx, d, c.steps, chain, st) : launch<InT, OutT, false, 64>(ctx, d, c.steps, chain, st);
        if (c.BN == 128) return c.two ? launch<InT, OutT, true, 128>(ctx, d, c.steps, chain, st) : launch<InT, OutT, false, 128>(ctx, d, c.steps, chain, st);
    }
    return c.two ? launch<InT, OutT, true, 256>(ctx, d, c.steps, chain, st) : launch<InT, OutT, false, 256>(ctx, d, c.steps, chain, st);
}

template <typename InT, typename OutT>
nm_status launch_sel(nm_ctx* ctx, const nm_linear_desc* d, NmChain chain, cudaStream_t st)
{
    constexpr int64_t CHUNK = 16 / sizeof(OutT);
    // Few rows or columns had the CUDA cores' fp32 FMA chains before the split kernel took them: no sum of theirs gets worse.
    const bool like_fma = !TcIn<InT>::is_int && !nm_algo_forced(d->algo) && (d->M < 64 || d->N < 64);
    const TileChoice c = choose<InT, OutT>(ctx, d, like_fma, chain);
    const int64_t main_n = d->N / CHUNK * CHUNK;
    if (c.S < 0) return NM_ERR_UNSUPPORTED;
    if (like_fma || nm_algo_is_split(d->algo) || main_n == d->N || main_n < 8 || d->acc_dump || d->idx_dump) return launch_choice<InT, OutT>(ctx, d, c, chain, st);
    // A row that is no multiple of 16 bytes: all of it by the split kernel, or the last 4 to 12 columns by the split kernel and the
    // others by themselves, whichever the model finds cheaper (16384 x 1004 x 1024: 58.4 us and 38.5); with dumps, whose
    // row is N, the former.
    nm_linear_desc m = *d, r = *d;
    m.N = main_n;
    r.N = d->N - main_n;
    r.W = (const uint8_t*)d->W + main_n * d->ldw * sizeof(InT);
    r.out = (uint8_t*)d->out + main_n * sizeof(OutT);
    if (d->residual) r.residual = (const uint8_t*)d->residual + main_n * sizeof(OutT);
    if (d->bias) r.bias = d->bias + main_n;
    if (d->w_scale) r.w_scale = d->w_scale + main_n;
    const TileChoice cm = choose<InT, OutT>(ctx, &m, false, chain), cr = choose<InT, OutT>(ctx, &r, false, chain);
    if (!nm_algo_forced(d->algo) && c.us <= cm.us + cr.us) return launch_choice<InT, OutT>(ctx, d, c, chain, st);
    const nm_status e = launch_choice<InT, OutT>(ctx, &m, cm, chain, st);
    if (e != NM_OK) return e;
    return launch_choice<InT, OutT>(ctx, &r, cr, chain, st);
}

}  // namespace

bool nm_linear_tc_supported(const nm_linear_desc* d)
{
    if (d->in_dtype == NM_F32) return false;
    const size_t es = nm_dtype_size(d->in_dtype);
    if (d->M < 1 || d->N < 8 || d->K < 1) return false;
    if ((d->K * es) % 16 != 0) return false;  // TMA: global extents and pitches in 16-byte units
    if (d->N % 4 != 0) return false;          // vector loads of bias / scales, vector dumps
    if (d->in_dtype == NM_I8) return d->out_dtype == NM_BF16 || d->out_dtype == NM_F32 || d->out_dtype == NM_I8;
    return d->out_dtype == d->in_dtype;
}

nm_status nm_launch_linear_tc(nm_ctx* ctx, const nm_linear_desc* d, cudaStream_t st, NmChain chain)
{
    if (!nm_linear_tc_supported(d)) return NM_ERR_UNSUPPORTED;
    switch (d->in_dtype) {
    case NM_BF16: return launch_sel<__nv_bfloat16, __nv_bfloat16>(ctx, d, chain, st);
    case NM_F16: return launch_sel<__half, __half>(ctx, d, chain, st);
    case NM_I8:
        if (d->out_dtype == NM_BF16) return launch_sel<int8_t, __nv_bfloat16>(ctx, d, chain, st);
        if (d->out_dtype == NM_F32) return launch_sel<int8_t, float>(ctx, d, chain, st);
        return launch_sel<int8_t, int8_t>(ctx, d, chain, st);
    default: return NM_ERR_UNSUPPORTED;
    }
}

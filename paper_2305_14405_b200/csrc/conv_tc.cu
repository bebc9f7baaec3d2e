// Host side of the implicit-GEMM convolution: chooses the patch of output pixels a tile covers,
// encodes the 4-D tensor maps over the NHWC tensors themselves and launches linear_tc_kernel
// (linear_tc_kernel.cuh) or linear_split_kernel (linear_split_kernel.cuh) in its CONV form.  Section 3.1: a convolution is a matrix product whose dimensions
// follow from width, height and channels; here the matrix is never written to memory.
#include "linear_split_kernel.cuh"

using namespace nm_tc;

namespace {

nm_status make_tmap4(nm_ctx* ctx, CUtensorMap* m, const void* base, nm_dtype dt, const uint64_t dim[4],
                     const uint64_t stride_bytes[3], const uint32_t box[4], const uint32_t estr[4],
                     CUtensorMapSwizzle swizzle = CU_TENSOR_MAP_SWIZZLE_128B)
{
    cuuint64_t gdim[4] = {dim[0], dim[1], dim[2], dim[3]};
    cuuint64_t gstr[3] = {stride_bytes[0], stride_bytes[1], stride_bytes[2]};
    cuuint32_t b[4] = {box[0], box[1], box[2], box[3]};
    cuuint32_t e[4] = {estr[0], estr[1], estr[2], estr[3]};
    CUresult r = ((EncodeTiledFn)ctx->encode_tiled)(m, tmap_type(dt), 4, const_cast<void*>(base), gdim, gstr, b, e,
                                                    CU_TENSOR_MAP_INTERLEAVE_NONE, swizzle,
                                                    CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                                                    CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    return r == CUDA_SUCCESS ? NM_OK : NM_ERR_CUDA;
}

int ceil_div(int a, int b) { return (a + b - 1) / b; }

// The patch TW x TH x NB (powers of two, product 128, TW <= 32) that wastes the fewest tile rows on
// pixels outside the output; ties go to the wider patch (longer contiguous runs per TMA row).
void choose_patch(int Wo, int Ho, int N, int* TW, int* TH, int* NB)
{
    double best = -1.0;
    for (int tw = 32; tw >= 1; tw >>= 1) {
        for (int th = 128 / tw; th >= 1; th >>= 1) {
            const int nb = 128 / (tw * th);
            const double covered = (double)ceil_div(Wo, tw) * tw * ceil_div(Ho, th) * th * ceil_div(N, nb) * nb;
            const double eff = (double)Wo * Ho * N / covered;
            if (eff > best + 1e-9) { best = eff; *TW = tw; *TH = th; *NB = nb; }
        }
    }
}

int64_t count_patches(int Wo, int Ho, int N)
{
    int tw, th, nb;
    choose_patch(Wo, Ho, N, &tw, &th, &nb);
    return (int64_t)ceil_div(Wo, tw) * ceil_div(Ho, th) * ceil_div(N, nb);
}

// Patch geometry and epilogue operands common to both kernels; returns the number of patches.
int64_t fill_args(nm_ctx* ctx, const NmConvTc* c, NmChain chain, TcArgs* a)
{
    memset(a, 0, sizeof(*a));
    ConvDev& cv = a->cv;
    choose_patch(c->Wo, c->Ho, c->N, &cv.TW, &cv.TH, &cv.NB);
    cv.tiles_x = ceil_div(c->Wo, cv.TW);
    cv.tiles_y = ceil_div(c->Ho, cv.TH);
    cv.sw = c->sw; cv.sh = c->sh; cv.pw = c->pw; cv.ph = c->ph;
    cv.kw_eff = c->taps_x; cv.cblocks = c->cblocks;
    cv.ky_last = c->taps_y - 1; cv.ky_jump = c->last_row_jump;
    cv.Ho = c->Ho; cv.Nimg = c->N;
    cv.dw = c->depthwise;
    cv.stem_kh = c->stem_kh;
    a->M = (int64_t)c->N * c->Ho * c->Wo; a->N = c->Cout; a->K = c->Ktot;
    a->bias = c->bias;
    a->has_res = c->residual ? 1 : 0;
    a->res_first = c->res_first;
    a->tab = c->slot == NM_SLOT_NONE ? nullptr : ctx->d_tables + c->slot;
    a->n_seg = c->slot == NM_SLOT_NONE ? 0 : ctx->h_tables[c->slot].n;
    a->status = ctx->d_status;
    a->weights_ready = chain.weights_ready && !c->depthwise;
    a->late_trigger = chain.late_trigger;
    a->num_k_blocks = c->taps_y * c->taps_x * c->cblocks;
    a->accs = 1;
    return (int64_t)cv.tiles_x * cv.tiles_y * ceil_div(c->N, cv.NB);
}

// A: one box per filter tap, strided like the convolution
nm_status make_tmap_a(nm_ctx* ctx, CUtensorMap* m, const NmConvTc* c, const ConvDev& cv)
{
    const uint32_t abox[4] = {64u, (uint32_t)((cv.TW - 1) * cv.sw + 1), (uint32_t)((cv.TH - 1) * cv.sh + 1), (uint32_t)cv.NB};
    const uint32_t aestr[4] = {1u, (uint32_t)cv.sw, (uint32_t)cv.sh, 1u};
    if (abox[1] > 256 || abox[2] > 256) return NM_ERR_UNSUPPORTED;
    return make_tmap4(ctx, m, c->a_base, c->dtype, c->a_dim, c->a_stride, abox, aestr);
}

// output / residual: the 32 tile rows of an epilogue warp are a sub-box of the patch
nm_status make_tmaps_out(nm_ctx* ctx, CUtensorMap* tmO, CUtensorMap* tmR, const NmConvTc* c, const ConvDev& cv)
{
    const int bh = cv.TH < 32 / cv.TW ? cv.TH : 32 / cv.TW;
    const int bn = 32 / (cv.TW * bh);
    const uint64_t odim[4] = {(uint64_t)c->Cout, (uint64_t)c->Wo, (uint64_t)c->Ho, (uint64_t)c->N};
    const uint64_t ostr[3] = {(uint64_t)c->Cout * 2, (uint64_t)c->Wo * c->Cout * 2, (uint64_t)c->Ho * c->Wo * c->Cout * 2};
    const uint32_t obox[4] = {64u, (uint32_t)cv.TW, (uint32_t)bh, (uint32_t)bn};
    const uint32_t one[4] = {1u, 1u, 1u, 1u};
    nm_status s = make_tmap4(ctx, tmO, c->out, c->dtype, odim, ostr, obox, one);
    if (s != NM_OK) return s;
    if (!c->residual) {
        *tmR = *tmO;
        return NM_OK;
    }
    return make_tmap4(ctx, tmR, c->residual, c->dtype, odim, ostr, obox, one);
}

// Is the halo form (linear_tc_kernel.cuh) the faster one?  3 x 3, stride 1, padding 1, at least two rounds of CTA pairs, and less
// time by the bytes a tile takes from L2 (50 a clock) and the tensor core's cycles, although its fixed 8 x 16 patch wastes rows
// that the free patch does not: 128 images, 56 x 56, 64 -> 64: 35 us against 77; 28 x 28, 128 -> 128: 39.2 against
// 44.8.  Wider outputs are bound by the tensor core in either form.
bool use_halo(const NmConvTc* c, int64_t free_patches, int sms)
{
    if (c->algo != 0 || c->taps_x != 3 || c->taps_y != 3 || c->sw != 1 || c->sh != 1 || c->pw != 1 || c->ph != 1 || c->depthwise ||
        c->Cout > 128 || c->Cout <= 32)
        return false;
    const int64_t halo_patches = (int64_t)ceil_div(c->Wo, 8) * ceil_div(c->Ho, 16) * c->N;
    if (halo_patches < 2LL * 2 * sms) return false;
    const int bn = c->Cout <= 64 ? 64 : 128;
    const double b_bytes = bn / 2 * ROW_BYTES, taps = 9.0 * c->cblocks, mma = bn == 64 ? 160.0 : 256.0;
    const double w_stream = bn == 64 && c->cblocks <= 2 ? 0.0 : taps * b_bytes;   // (up to 18 weight tiles stay in shared memory)
    const double feed_free = taps * (A_BYTES + b_bytes) / 50, feed_halo = (c->cblocks * (double)HALO_BYTES + w_stream) / 50;
    const double t_free = (double)free_patches * (feed_free > taps * mma ? feed_free : taps * mma);
    const double t_halo = (double)halo_patches * (feed_halo > taps * mma ? feed_halo : taps * mma);
    return t_halo < 0.9 * t_free;
}

// The forms that load a patch of 8 x 16 output pixels' input once: HALO3X3 and STEM.
template <typename T, int BN, int FORM>
nm_status launch_halo(nm_ctx* ctx, const NmConvTc* c, NmChain chain, cudaStream_t st)
{
    TcArgs a;
    fill_args(ctx, c, chain, &a);
    ConvDev& cv = a.cv;
    cv.TW = 8; cv.TH = 16; cv.NB = 1;
    cv.tiles_x = ceil_div(c->Wo, cv.TW);
    cv.tiles_y = ceil_div(c->Ho, cv.TH);
    const int64_t patches = (int64_t)cv.tiles_x * cv.tiles_y * c->N;
    a.num_n_tiles = 1;
    if (patches / 2 > 0x7ffffffeLL) return NM_ERR_UNSUPPORTED;
    a.num_tiles = (int)((patches + 1) / 2);
    size_t smem = 0;
    if (!plan_smem_halo<T, BN, FORM>(&a, c->bias != nullptr, &smem)) return NM_ERR_UNSUPPORTED;
    CUtensorMap tmA, tmW, tmO, tmR;
    const uint32_t halo[4] = {64u, HALO_W, HALO_H, 1u}, stem[4] = {STEM_PITCH / 2, (uint32_t)(30 + c->stem_kh), 1u, 1u}, one[4] = {1u, 1u, 1u, 1u};
    nm_status s = make_tmap4(ctx, &tmA, c->a_base, c->dtype, c->a_dim, c->a_stride, FORM == STEM ? stem : halo, one,
                             FORM == STEM ? CU_TENSOR_MAP_SWIZZLE_NONE : CU_TENSOR_MAP_SWIZZLE_128B);
    if (s != NM_OK) return s;
    s = make_tmap(ctx, &tmW, c->w, c->dtype, c->Cout, c->Ktot, c->ldw, BN / 2);
    if (s != NM_OK) return s;
    s = make_tmaps_out(ctx, &tmO, &tmR, c, cv);
    if (s != NM_OK) return s;
    if constexpr (FORM == HALO3X3 && BN == 64) {
        if (a.w_resident) return launch_kernel<T, T, true, BN, true, HALO_RESIDENT>(ctx, tmA, tmW, tmO, tmR, a, smem, c->flops, st);
    }
    return launch_kernel<T, T, true, BN, true, FORM>(ctx, tmA, tmW, tmO, tmR, a, smem, c->flops, st);
}

template <typename T, int BN>
nm_status launch_split(nm_ctx* ctx, const NmConvTc* c, int S, NmChain chain, cudaStream_t st)
{
    SplitArgs s;
    memset(&s, 0, sizeof(s));
    const int64_t patches = fill_args(ctx, c, chain, &s.t);
    s.t.num_n_tiles = ceil_div(c->Cout, BN);
    const int64_t tiles = patches * s.t.num_n_tiles;
    if (tiles > 0x7fffffffLL / S) return NM_ERR_SHAPE;
    s.S = S;
    s.t.num_tiles = (int)tiles;
    s.residual = c->residual; s.ldr = c->Cout;
    s.out = c->out; s.ldo = c->Cout;
    s.Wo = c->Wo;
    CUtensorMap tmA, tmW;
    nm_status e = make_tmap_a(ctx, &tmA, c, s.t.cv);
    if (e != NM_OK) return e;
    e = make_tmap(ctx, &tmW, c->w, c->dtype, c->depthwise ? 64 : c->Cout, c->Ktot, c->ldw, BN);
    if (e != NM_OK) return e;
    return launch_split_kernel<T, T, BN, true>(ctx, tmA, tmW, s, chain.back_to_back, c->flops, st);
}

template <typename T, bool TWO, int BN>
nm_status launch(nm_ctx* ctx, const NmConvTc* c, NmChain chain, cudaStream_t st)
{
    constexpr int B_ROWS = TWO ? BN / 2 : BN;
    TcArgs a;
    const int64_t patches = fill_args(ctx, c, chain, &a);
    const ConvDev& cv = a.cv;
    const int64_t m_tiles = TWO ? (patches + 1) / 2 : patches;
    a.num_n_tiles = ceil_div(c->Cout, BN);
    if (m_tiles * a.num_n_tiles > 0x7fffffffLL) return NM_ERR_SHAPE;
    a.num_tiles = (int)(m_tiles * a.num_n_tiles);
    size_t smem = 0;
    if (!plan_smem<T, TWO, BN>(&a, c->bias != nullptr, &smem)) return NM_ERR_UNSUPPORTED;

    CUtensorMap tmA, tmW, tmO, tmR;
    nm_status s = make_tmap_a(ctx, &tmA, c, cv);
    if (s != NM_OK) return s;
    // (depthwise form: W is the one 64 x 64 matrix, whatever the number of output channels)
    s = make_tmap(ctx, &tmW, c->w, c->dtype, c->depthwise ? 64 : c->Cout, c->Ktot, c->ldw, B_ROWS);
    if (s != NM_OK) return s;
    s = make_tmaps_out(ctx, &tmO, &tmR, c, cv);
    if (s != NM_OK) return s;
    return launch_kernel<T, T, TWO, BN, true>(ctx, tmA, tmW, tmO, tmR, a, smem, c->flops, st);
}

template <typename T>
nm_status launch_sel(nm_ctx* ctx, const NmConvTc* c, NmChain chain, cudaStream_t st)
{
    if (c->stem_kh) return c->Cout <= 64 ? launch_halo<T, 64, STEM>(ctx, c, chain, st) : launch_halo<T, 128, STEM>(ctx, c, chain, st);
    TileChoice t;
    if (c->algo == 0) {
        const int64_t patches = count_patches(c->Wo, c->Ho, c->N);
        if (use_halo(c, patches, ctx->sm_count)) {
            const nm_status e = c->Cout <= 64 ? launch_halo<T, 64, HALO3X3>(ctx, c, chain, st) : launch_halo<T, 128, HALO3X3>(ctx, c, chain, st);
            if (e != NM_ERR_UNSUPPORTED) return e;
        }
        t = choose_tile((int64_t)c->N * c->Ho * c->Wo, patches, c->Cout, (int64_t)c->taps_y * c->taps_x * c->cblocks, true,
                        EpiNeeds{c->slot == NM_SLOT_NONE ? 0 : ctx->h_tables[c->slot].n, c->residual != nullptr, c->bias != nullptr},
                        c->depthwise != 0, true, 0, chain, ctx->sm_count);
    } else if (nm_algo_is_split(c->algo)) {
        t = forced_split(c->algo, (int64_t)c->taps_y * c->taps_x * c->cblocks);
        if (t.S < 0) return NM_ERR_UNSUPPORTED;
    } else {
        t.S = 0;
        t.BN = c->Cout <= 64 || c->depthwise ? 64 : (c->Cout <= 128 ? 128 : 256);
        t.two = c->algo != 3 && (int64_t)c->N * c->Ho * c->Wo >= 256;
    }
    if (t.S) return t.BN == 32 ? launch_split<T, 32>(ctx, c, t.S, chain, st) : launch_split<T, 64>(ctx, c, t.S, chain, st);
    if (t.BN == 64) return t.two ? launch<T, true, 64>(ctx, c, chain, st) : launch<T, false, 64>(ctx, c, chain, st);
    if (t.BN == 128) return t.two ? launch<T, true, 128>(ctx, c, chain, st) : launch<T, false, 128>(ctx, c, chain, st);
    return t.two ? launch<T, true, 256>(ctx, c, chain, st) : launch<T, false, 256>(ctx, c, chain, st);
}

}  // namespace

// Is the patch-wise form of a first layer (STEM) faster than the row pairs'?  Its patch is 8 x 16 pixels of one image, theirs leaves as few
// rows empty as it can and may hold several images.  Few patches, up to four a SM with 64 columns and one with 128: it is (0.73 to 1.00
// of the time and 0.91 to 1.03).  Beyond, by patches over patches of the row pairs, its time over theirs with the copies, 64 to 2048 images:
// 64 columns 1.0: 0.65 to 0.86, 1.43: 0.90 to 0.93, 1.7: 0.97 to 1.01, 2.0 (8 x 8 outputs): 0.75 to 0.89, 2.66 (17 x 17): 1.14 to 1.25, 3.16 (9 x 9): 0.98
// to 1.10; 128 columns 1.0: 0.78 to 0.92, 1.33: 1.00 to 1.04, 1.43: 1.11, 1.78: 1.01 to 1.26, 2.66: 1.37 to 1.61, 3.16: 1.10 to 1.50.
bool nm_conv_stem_pays(int Wo, int Ho, int N, int Cout)
{
    const int64_t patches = (int64_t)ceil_div(Wo, 8) * ceil_div(Ho, 16) * N;
    return patches <= (Cout <= 64 ? 4 : 1) * 148 || (double)patches <= (Cout <= 64 ? 2.0 : 1.3) * (double)count_patches(Wo, Ho, N);
}

nm_status nm_launch_conv_tc(nm_ctx* ctx, const NmConvTc* c, cudaStream_t st, NmChain chain)
{
    if (c->dtype == NM_F16) return launch_sel<__half>(ctx, c, chain, st);
    if (c->dtype == NM_BF16) return launch_sel<__nv_bfloat16>(ctx, c, chain, st);
    return NM_ERR_UNSUPPORTED;
}

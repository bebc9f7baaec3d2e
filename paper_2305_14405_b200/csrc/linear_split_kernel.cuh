// The linear operator for problems whose tiles do not fill the GPU (a single request, a late convolution
// stage): one 128 x BN output tile (BN = 64 or 32) per thread-block cluster, the K dimension split over the
// cluster's CTAs.
//
//   out[m][j] = PWL( sum_c A[m][c]*W[j][c] * scale_j + bias[j] ) + residual[m][j]
//
// Such a launch is bound by latency: with the persistent kernel's 256-column tiles a BERT-base layer on 128
// tokens keeps 3 to 12 SMs busy, each walking through the whole of K on its own.  Here every CTA multiplies
// its share of the K-blocks (TMA ring, tcgen05.mma into tensor memory) and finishes every S-th row of the tile.
// It sends its fp32 or int32 partial rows straight from registers to the CTAs that own them (st.async over
// distributed shared memory, counted on the owner's mbarrier), waits for the rows sent to it, adds the S
// partial rows in rank order (the sum does not depend on timing), applies scale, bias, table and residual and
// stores whole row segments.  Nobody reads another CTA's memory and no CTA waits for a cluster barrier: with
// the partial tiles left where they were made, the barrier before the remote reads, the reads and the barrier
// before the exit took 1300 + 1300 to 3000 + 1300 cycles of a launch of 8 to 12 thousand (12 layers, 37 tokens: 470 us
// then, 417 so).  S is a template parameter: a launch runs its code once, from a cold instruction cache, and what it does not
// need is in its way (37 tokens: 403 -> 391 us, ResNet-50 batch 1: 373 -> 357).
//
// CONV = true: the A operand is the NHWC activation, as in linear_tc_kernel (a tile's 128 rows are a patch of
// output pixels and a K-block is one 4-D TMA box).
#pragma once
#include "linear_tc_kernel.cuh"

namespace nm_tc {

constexpr int SPLIT_THREADS = 256;
constexpr int SPLIT_MAX_STAGES = 6;

struct SplitArgs {
    TcArgs t;               // num_tiles, num_n_tiles, num_k_blocks, stages and the epilogue's operands
    int S;                  // CTAs per cluster
    const void* residual;
    int64_t ldr, ldo;
    void* out;
    int Wo;                 // CONV: output pixels per row
};

// Words per row of a partial tile: 16-byte row stores and loads without bank conflicts.
constexpr int part_pitch(int bn) { return bn + 4; }

template <typename OutT> struct Quad;
template <> struct Quad<float> {
    using Raw = float4;
    static __device__ __forceinline__ Raw fetch(const float* p) { return *reinterpret_cast<const float4*>(p); }
    static __device__ __forceinline__ float4 widen(const Raw& w) { return w; }
    static __device__ __forceinline__ void store(float* p, const float4& v, float) { *reinterpret_cast<float4*>(p) = v; }
};
template <> struct Quad<__nv_bfloat16> {
    using Raw = uint2;
    static __device__ __forceinline__ Raw fetch(const __nv_bfloat16* p) { return *reinterpret_cast<const uint2*>(p); }
    static __device__ __forceinline__ float4 widen(const Raw& w)
    {
        const float2 a = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&w.x));
        const float2 b = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&w.y));
        return make_float4(a.x, a.y, b.x, b.y);
    }
    static __device__ __forceinline__ void store(__nv_bfloat16* p, const float4& v, float)
    {
        const __nv_bfloat162 a = __floats2bfloat162_rn(v.x, v.y), b = __floats2bfloat162_rn(v.z, v.w);
        *reinterpret_cast<uint2*>(p) = make_uint2(*reinterpret_cast<const uint32_t*>(&a), *reinterpret_cast<const uint32_t*>(&b));
    }
};
template <> struct Quad<__half> {
    using Raw = uint2;
    static __device__ __forceinline__ Raw fetch(const __half* p) { return *reinterpret_cast<const uint2*>(p); }
    static __device__ __forceinline__ float4 widen(const Raw& w)
    {
        const float2 a = __half22float2(*reinterpret_cast<const __half2*>(&w.x));
        const float2 b = __half22float2(*reinterpret_cast<const __half2*>(&w.y));
        return make_float4(a.x, a.y, b.x, b.y);
    }
    static __device__ __forceinline__ void store(__half* p, const float4& v, float)
    {
        const __half2 a = __floats2half2_rn(v.x, v.y), b = __floats2half2_rn(v.z, v.w);
        *reinterpret_cast<uint2*>(p) = make_uint2(*reinterpret_cast<const uint32_t*>(&a), *reinterpret_cast<const uint32_t*>(&b));
    }
};
template <> struct Quad<int8_t> {
    using Raw = uint32_t;   // there is no int8 residual
    static __device__ __forceinline__ Raw fetch(const int8_t*) { return 0u; }
    static __device__ __forceinline__ float4 widen(const Raw&) { return make_float4(0.f, 0.f, 0.f, 0.f); }
    static __device__ __forceinline__ void store(int8_t* p, const float4& v, float inv)
    {
        *reinterpret_cast<uint32_t*>(p) = nm_quant_i8x4(v.x, v.y, v.z, v.w, inv);
    }
};

// 16 bytes into the shared memory of a CTA of the cluster, counted on that CTA's mbarrier
__device__ __forceinline__ void st_async_v4(uint32_t cluster_addr, uint32_t a, uint32_t b, uint32_t c, uint32_t d, uint32_t cluster_bar)
{
    asm volatile("st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.v4.b32 [%0], {%1,%2,%3,%4}, [%5];" ::"r"(cluster_addr),
                 "r"(a), "r"(b), "r"(c), "r"(d), "r"(cluster_bar)
                 : "memory");
}
__device__ __forceinline__ uint4 ld_cluster_v4(uint32_t cluster_addr)
{
    uint4 v;
    asm volatile("ld.shared::cluster.v4.b32 {%0,%1,%2,%3}, [%4];"
                 : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w)
                 : "r"(cluster_addr));
    return v;
}

// Final sum and epilogue of a cluster's tile: this CTA takes rows rank, rank + S, ... of the `rows` that exist and adds
// the S partial rows in rank order, part_pitch(BN) words per row.  PUSHED: they are in this CTA's shared memory, row r of
// CTA k at row k * (BM / S) + r / S of `part`; otherwise in each CTA's own, row r at row r of its `part`.  Four columns
// per thread, whole row segments per group of BN / 4 threads.  Rows go in batches of up to FIN_U per thread, all loads
// of a batch in flight together, and the vectors and the first batch's residual are fetched before the product is even
// started: a row at a time cost a memory latency per row.  CTAS: S, or 0 where it is not known at compile time.
constexpr int FIN_U = 4;

template <bool INT, typename OutT, int BN, bool CONV, int THREADS, bool PUSHED, int CTAS = 0>
struct Finisher {
    static constexpr int PITCH = part_pitch(BN);
    static constexpr int QPR = BN / 4;            // 4-column groups per row
    static constexpr int RPP = THREADS / QPR;     // rows per pass
    const SplitArgs& s;
    const int rank, mt, nt, rows;
    const Patch pt;
    const int qc;          // this thread's 4-column group in every pass
    const int64_t col;
    const bool col_ok;     // N is a multiple of 4
    float4 bias, sc;
    typename Quad<OutT>::Raw res[FIN_U];

    __device__ __forceinline__ Finisher(const SplitArgs& s_, int rank_, int mt_, int nt_, int rows_, const Patch& pt_)
        : s(s_), rank(rank_), mt(mt_), nt(nt_), rows(rows_), pt(pt_), qc((int)threadIdx.x % QPR),
          col((int64_t)nt_ * BN + qc * 4), col_ok(col < s_.t.N)
    {
    }
    // row of the output matrix that row r of the tile is, or -1
    __device__ __forceinline__ int64_t out_row(int r) const
    {
        if (r >= rows) return -1;
        if constexpr (CONV) {
            const ConvDev& cv = s.t.cv;
            const int ox = pt.ox0 + r % cv.TW, oy = pt.oy0 + (r / cv.TW) % cv.TH, img = pt.img0 + r / (cv.TW * cv.TH);
            if (ox >= s.Wo || oy >= cv.Ho || img >= cv.Nimg) return -1;
            return ((int64_t)img * cv.Ho + oy) * s.Wo + ox;
        } else {
            return (int64_t)mt * BM + r;
        }
    }
    __device__ __forceinline__ int tile_row(int i) const { return ((int)threadIdx.x / QPR + i * RPP) * ctas() + rank; }
    __device__ __forceinline__ int ctas() const { return CTAS ? CTAS : s.S; }
    __device__ __forceinline__ void load_res(int i0)
    {
        if (!s.residual || !col_ok) return;
#pragma unroll
        for (int u = 0; u < FIN_U; ++u) {
            const int64_t g = out_row(tile_row(i0 + u));
            if (g >= 0) res[u] = Quad<OutT>::fetch(reinterpret_cast<const OutT*>(s.residual) + g * s.ldr + col);
        }
    }
    __device__ __forceinline__ void prefetch_vectors()
    {
        bias = make_float4(0.f, 0.f, 0.f, 0.f);
        sc = bias;
        if (col_ok) {
            if (s.t.bias) bias = __ldg(reinterpret_cast<const float4*>(s.t.bias + col));
            if constexpr (INT) {
                const float4 ws = __ldg(reinterpret_cast<const float4*>(s.t.w_scale + col));
                const float as = s.t.a_scale;
                sc = make_float4(as * ws.x, as * ws.y, as * ws.z, as * ws.w);
            }
        }
    }
    __device__ __forceinline__ void run(const uint32_t* part, const float2* tab)
    {
        const int per_thread = (rows + ctas() * RPP - 1) / (ctas() * RPP);
        if (per_thread <= 1) batches<1>(part, tab);
        else if (per_thread <= 2) batches<2>(part, tab);
        else batches<FIN_U>(part, tab);
    }
    template <int U>
    __device__ __forceinline__ void batches(const uint32_t* part, const float2* tab)
    {
        const TcArgs& a = s.t;
        const int S = ctas();
        const bool has_tab = a.tab != nullptr;
        const float inv_h = has_tab ? a.tab->inv_h : 0.f, off = has_tab ? a.tab->off : 0.f, nm1 = (float)(a.n_seg - 1);
        const uint32_t part_u = nm_smem_u32(part);
        const int slot = PUSHED ? BM / S : 0, lg = 31 - __clz(S);   // slot: rows between the partial rows of two CTAs; S is 1, 2, 4, 8
        auto partial = [&](int r, int k) {
            if constexpr (PUSHED) return *reinterpret_cast<const uint4*>(part + (k * slot + (r >> lg)) * PITCH + qc * 4);
            else return S == 1 ? *reinterpret_cast<const uint4*>(part + (size_t)r * PITCH + qc * 4)
                               : ld_cluster_v4(nm_mapa(part_u + (uint32_t)(r * PITCH + qc * 4) * 4u, (uint32_t)k));
        };
        for (int i0 = 0; tile_row(i0) < rows; i0 += U) {
            if (i0 > 0) load_res(i0);
            uint32_t acc[U][4];
#pragma unroll
            for (int u = 0; u < U; ++u) {
                // (a row beyond the tile's last is read from the last and not used)
                const uint4 p = partial(min(tile_row(i0 + u), BM - 1), 0);
                acc[u][0] = p.x; acc[u][1] = p.y; acc[u][2] = p.z; acc[u][3] = p.w;
            }
#pragma unroll 2
            for (int k = 1; k < S; ++k) {
                uint4 o[U];
#pragma unroll
                for (int u = 0; u < U; ++u) o[u] = partial(min(tile_row(i0 + u), BM - 1), k);
#pragma unroll
                for (int u = 0; u < U; ++u) {
                    const uint32_t w[4] = {o[u].x, o[u].y, o[u].z, o[u].w};
#pragma unroll
                    for (int i = 0; i < 4; ++i) {
                        if constexpr (INT) acc[u][i] += w[i];
                        else acc[u][i] = __float_as_uint(__uint_as_float(acc[u][i]) + __uint_as_float(w[i]));
                    }
                }
            }
#pragma unroll
            for (int u = 0; u < U; ++u) {
                const int64_t grow = out_row(tile_row(i0 + u));
                if (grow < 0 || !col_ok) continue;
                float x[4];
                const float bv[4] = {bias.x, bias.y, bias.z, bias.w}, sv[4] = {sc.x, sc.y, sc.z, sc.w};
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    if constexpr (INT) x[i] = __fmaf_rn((float)(int)acc[u][i], sv[i], bv[i]);
                    else x[i] = __uint_as_float(acc[u][i]) + bv[i];
                }
                if constexpr (INT) {
                    if (a.acc_dump)
                        *reinterpret_cast<int4*>(a.acc_dump + grow * a.N + col) =
                            make_int4((int)acc[u][0], (int)acc[u][1], (int)acc[u][2], (int)acc[u][3]);
                }
                float4 rv = make_float4(0.f, 0.f, 0.f, 0.f);
                if (s.residual) rv = Quad<OutT>::widen(res[u]);
                if (s.residual && a.res_first) { x[0] += rv.x; x[1] += rv.y; x[2] += rv.z; x[3] += rv.w; }
                int seg[4] = {-1, -1, -1, -1};
                if (has_tab) {
#pragma unroll
                    for (int i = 0; i < 4; ++i) {
                        seg[i] = nm_pwl_index(x[i], inv_h, off, nm1);
                        const float2 t = tab[seg[i]];
                        x[i] = __fmaf_rn(t.x, x[i], t.y);
                    }
                }
                if (a.idx_dump) *reinterpret_cast<int4*>(a.idx_dump + grow * a.N + col) = make_int4(seg[0], seg[1], seg[2], seg[3]);
                if (s.residual && !a.res_first) { x[0] += rv.x; x[1] += rv.y; x[2] += rv.z; x[3] += rv.w; }
                Quad<OutT>::store(reinterpret_cast<OutT*>(s.out) + grow * s.ldo + col, make_float4(x[0], x[1], x[2], x[3]), a.inv_out_scale);
            }
        }
    }
};

template <typename InT, typename OutT, int BN, bool CONV, int S>
__global__ void __launch_bounds__(SPLIT_THREADS, 2)
linear_split_kernel(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmW, const SplitArgs s)
{
    const TcArgs& a = s.t;
    constexpr bool INT = TcIn<InT>::is_int;
    constexpr int B_BYTES = BN * ROW_BYTES;
    constexpr int STAGE_BYTES = A_BYTES + B_BYTES;
    constexpr int BK_ELEMS = ROW_BYTES / (int)sizeof(InT);
    constexpr uint32_t IDESC = nm_idesc(TcIn<InT>::c_fmt, TcIn<InT>::ab_fmt, 0, 0, BM, BN);
    constexpr int PITCH = part_pitch(BN);

    extern __shared__ uint8_t smem_raw[];
    __shared__ uint64_t bar_full[SPLIT_MAX_STAGES], bar_empty[SPLIT_MAX_STAGES], bar_acc, bar_part;
    __shared__ uint32_t tmem_slot;
    __shared__ int abort_flag;
    __shared__ float2 s_tab[NM_MAX_SEGMENTS];

    const int rank = S > 1 ? (int)nm_cluster_ctarank() : 0;
    const int tile = (int)blockIdx.x / S;
    const int mt = tile / a.num_n_tiles, nt = tile % a.num_n_tiles;
    const int kb0 = rank * a.num_k_blocks / S, kb1 = (rank + 1) * a.num_k_blocks / S;
    const int stages = a.stages;
    uint8_t* tiles = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
    // The partial rows: without a split they take the ring's place once K is done; with one they arrive while the ring may
    // still be in use.
    uint32_t* part = reinterpret_cast<uint32_t*>(tiles + (S > 1 ? (size_t)stages * STAGE_BYTES : 0));
    const int rows = CONV ? BM : (int)(a.M - (int64_t)mt * BM < BM ? a.M - (int64_t)mt * BM : BM);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;

    if (threadIdx.x == 0) {
        abort_flag = 0;
        nm_prefetch_tmap(&tmA);
        nm_prefetch_tmap(&tmW);
        for (int i = 0; i < stages; ++i) {
            nm_mbar_init(&bar_full[i], 1);
            nm_mbar_init(&bar_empty[i], 1);
        }
        nm_mbar_init(&bar_acc, 1);
        nm_mbar_init(&bar_part, 1);
        nm_fence_barrier_init();
        // what the others will send: their columns of each of this CTA's rows
        if (S > 1) nm_mbar_expect_tx(&bar_part, (uint32_t)((rows - rank + S - 1) / S) * (uint32_t)(S - 1) * BN * 4u);
    }
    constexpr bool MULTI = !INT && !CONV;   // several accumulators (TcArgs::acc_steps)
    const uint32_t tmem_cols = !MULTI ? BN : a.accs <= 1 ? BN : a.accs <= 2 ? 2 * BN : a.accs <= 4 ? 4 * BN : 8 * BN;
    if (warp == 1) {
        nm_tmem_alloc(&tmem_slot, tmem_cols);
        nm_tmem_relinquish();
    }
    if (a.tab) {
        for (int i = threadIdx.x; i < a.n_seg; i += SPLIT_THREADS) s_tab[i] = a.tab->kb[i];
    }
    nm_tc_fence_before();
    __syncthreads();
    nm_tc_fence_after();
    if (S > 1) asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");   // this CTA's barrier may be sent to
    const uint32_t tmem = tmem_slot;
    volatile int* abortp = &abort_flag;
    if (!a.late_trigger) nm_grid_launch_dependents();
    // Weights that were complete before the previous kernel started need not wait for it: this CTA's share goes into the
    // ring's stages and, beyond those, into L2 while that kernel still runs.
    int early = 0;   // K-blocks whose W tile is on its way
    if (a.weights_ready && warp == 0) {
        early = kb1 - kb0 < stages ? kb1 - kb0 : stages;
        if (nm_elect_one()) {
            for (int i = 0; i < early; ++i) {
                nm_mbar_expect_tx(&bar_full[i], STAGE_BYTES);
                nm_tma_load_2d(tiles + (size_t)i * STAGE_BYTES + A_BYTES, &tmW, (kb0 + i) * BK_ELEMS, nt * BN, &bar_full[i]);
            }
            for (int kb = kb0 + early; kb < kb1 && mt == 0; ++kb) nm_tma_prefetch_2d(&tmW, kb * BK_ELEMS, nt * BN);
        }
        __syncwarp();
    }
    Patch pt = {0, 0, 0};
    if constexpr (CONV) pt = patch_of(a.cv, mt);
    Finisher<INT, OutT, BN, CONV, SPLIT_THREADS, true, S> fin(s, rank, mt, nt, rows, pt);
    // One lane runs the producer's and the issuer's loops for the 16-bit types (12 layers, 37 tokens: 547 -> 537 us); for int8 all
    // lanes do, with one elected to issue (24 layers, 128 tokens: 1215 us against 1230).
    constexpr bool ONE_LANE = !INT;
    auto vote = [](bool done) { return ONE_LANE ? done : __all_sync(0xffffffffu, done) != 0; };
    bool ok = true;
    if (a.weights_ready) fin.prefetch_vectors();
    nm_grid_dependency_wait();
    if (a.late_trigger) nm_grid_launch_dependents();
    if (!a.weights_ready) fin.prefetch_vectors();
    if (warp != 0) fin.load_res(0);
    if (warp == 0) {
        // ------------------------------------------------ TMA producer
        if (!ONE_LANE || nm_elect_one()) {
            int stage = 0;
            uint32_t phase = 0;
            int kx = 0, ky = 0, cb = 0;
            if constexpr (CONV) {
                const int tap = kb0 / a.cv.cblocks;
                cb = kb0 - tap * a.cv.cblocks;
                ky = tap / a.cv.kw_eff;
                kx = tap - ky * a.cv.kw_eff;
            }
            for (int kb = kb0; kb < kb1; ++kb) {
                if (!vote(nm_mbar_wait(&bar_empty[stage], phase ^ 1u, abortp, a.status))) { ok = false; break; }
                uint8_t* sa = tiles + (size_t)stage * STAGE_BYTES;
                int c_c = 0, c_w = 0, c_h = 0, w_k = kb * BK_ELEMS, w_n = nt * BN;
                if constexpr (CONV) {
                    c_c = cb * BK_ELEMS;
                    c_w = pt.ox0 * a.cv.sw - a.cv.pw + kx;
                    c_h = pt.oy0 * a.cv.sh - a.cv.ph + ky + (ky == a.cv.ky_last ? a.cv.ky_jump : 0);
                    if (a.cv.dw) {   // pooling: channel block = column tile, one constant matrix for every tap and tile
                        c_c = nt * BK_ELEMS;
                        w_k = 0;
                        w_n = 0;
                    }
                    if (++cb == a.cv.cblocks) {
                        cb = 0;
                        if (++kx == a.cv.kw_eff) { kx = 0; ++ky; }
                    }
                }
                if (ONE_LANE || nm_elect_one()) {
                    if (kb - kb0 >= early) nm_mbar_expect_tx(&bar_full[stage], STAGE_BYTES);
                    if constexpr (CONV) nm_tma_load_4d(sa, &tmA, c_c, c_w, c_h, pt.img0, &bar_full[stage]);
                    else nm_tma_load_2d(sa, &tmA, kb * BK_ELEMS, mt * BM, &bar_full[stage]);
                    if (kb - kb0 >= early) nm_tma_load_2d(sa + A_BYTES, &tmW, w_k, w_n, &bar_full[stage]);
                }
                if constexpr (!ONE_LANE) __syncwarp();
                if (++stage == stages) { stage = 0; phase ^= 1u; }
            }
            if (!ok) {
                long long t0 = clock64();  // bounded pause: copies in flight land before teardown
                while (clock64() - t0 < 4000000LL) {}
            }
        }
        __syncwarp();
        fin.load_res(0);
    } else if (warp == 1) {
        // ------------------------------------------------ MMA issuer
        if (!ONE_LANE || nm_elect_one()) {
            int stage = 0;
            uint32_t phase = 0;
            bool ready = false;
            [[maybe_unused]] uint32_t acc = tmem;
            [[maybe_unused]] int left = a.acc_steps;   // steps that the accumulator still takes (0: no limit)
            [[maybe_unused]] uint32_t accum_on = 0;
            for (int kb = kb0; kb < kb1; ++kb) {
                if (!ready && !vote(nm_mbar_wait(&bar_full[stage], phase, abortp, a.status))) { ok = false; break; }
                if constexpr (ONE_LANE) {   // look at the next stage while this one's MMAs are issued
                    const int nxt = stage + 1 == stages ? 0 : stage + 1;
                    ready = nm_mbar_test_wait(&bar_full[nxt], nxt == 0 ? phase ^ 1u : phase);
                }
                nm_tc_fence_after();
                const uint32_t sa = nm_smem_u32(tiles + (size_t)stage * STAGE_BYTES);
                const uint64_t adesc = nm_smem_desc_sw128(sa), bdesc = nm_smem_desc_sw128(sa + A_BYTES);
                if (ONE_LANE || nm_elect_one()) {
#pragma unroll
                    for (int k = 0; k < 4; ++k) {  // 4 x 32 bytes of K per 128-byte row
                        const uint32_t accum = MULTI ? accum_on : (kb != kb0 || k != 0) ? 1u : 0u;
                        if constexpr (INT) nm_mma_i8(tmem, adesc + 2 * k, bdesc + 2 * k, IDESC, accum);
                        else nm_mma_f16(MULTI ? acc : tmem, adesc + 2 * k, bdesc + 2 * k, IDESC, accum);
                        if constexpr (MULTI) {
                            accum_on = 1u;
                            if (--left == 0) {
                                acc += BN;
                                left = a.acc_steps;
                                accum_on = 0u;
                            }
                        }
                    }
                    nm_tc_commit(&bar_empty[stage]);
                }
                if constexpr (!ONE_LANE) __syncwarp();
                if (++stage == stages) { stage = 0; phase ^= 1u; }
            }
            // After a timeout the commit still counts the MMAs that were issued, so that the wait below ends with them.
            if (ONE_LANE || nm_elect_one()) nm_tc_commit(&bar_acc);
        }
        __syncwarp();
    }
    // Every warp waits for the accumulator: all MMAs have then read the ring, whose place the partial tile takes.
    if (!nm_mbar_wait_relaxed<20>(&bar_acc, 0, abortp, a.status)) ok = false;
    __syncwarp();
    nm_tc_fence_after();
    __syncthreads();
    ok = ok && !abort_flag;
    if (S > 1) asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");   // (long complete: it was reached before K)
    {   // two warps per tensor-memory lane quarter, each half of the columns
        const int q = warp & 3, c0 = (warp >> 2) * (BN / 2), row = q * 32 + lane, owner = row & (S - 1);
        uint32_t* mine = part + (((rank * BM + row) >> (31 - __clz(S))) * PITCH + c0);   // the row's place, in the owner
        const uint32_t t_addr = tmem + ((uint32_t)(q * 32) << 16) + (uint32_t)c0;
        const uint32_t dst = nm_mapa(nm_smem_u32(mine), (uint32_t)owner), bar = nm_mapa(nm_smem_u32(&bar_part), (uint32_t)owner);
        const int used = MULTI && a.accs > 1 ? (4 * (kb1 - kb0) + a.acc_steps - 1) / a.acc_steps : 1;   // this CTA's accumulators
        if (ok && q * 32 < rows) {
#pragma unroll
            for (int c = 0; c < BN / 2; c += 16) {
                uint32_t r[16];
                nm_tmem_ld16_sync(t_addr + (uint32_t)c, r);
                if constexpr (MULTI) {
                    for (int i = 1; i < used; ++i) {
                        uint32_t o[16];
                        nm_tmem_ld16_sync(t_addr + (uint32_t)(i * BN + c), o);
#pragma unroll
                        for (int j = 0; j < 16; ++j) r[j] = __float_as_uint(__uint_as_float(r[j]) + __uint_as_float(o[j]));
                    }
                }
                if (row >= rows) continue;
                if (owner == rank) {
#pragma unroll
                    for (int i = 0; i < 16; i += 4)
                        *reinterpret_cast<uint4*>(mine + c + i) = make_uint4(r[i], r[i + 1], r[i + 2], r[i + 3]);
                } else {
#pragma unroll
                    for (int i = 0; i < 16; i += 4) st_async_v4(dst + (uint32_t)(c + i) * 4u, r[i], r[i + 1], r[i + 2], r[i + 3], bar);
                }
            }
        }
    }
    // The rows of other CTAs: one thread acquires them, at cluster scope, and hands them on through the block's barrier (256
    // threads that each acquire at cluster scope cost 0.13 us a launch: int8 24 layers, 128 tokens 878 -> 890 us).
    if (S > 1 && ok && threadIdx.x == 0) (void)nm_mbar_wait_cluster(&bar_part, 0, abortp, a.status);
    __syncthreads();
    ok = ok && !abort_flag;

    if (ok) fin.run(part, s_tab);

    // ---------------------------------------------------- teardown (all paths)
    nm_tc_fence_before();
    __syncthreads();
    if (warp == 1) {
        __syncwarp();
        nm_tc_fence_after();
        nm_tmem_dealloc(tmem, tmem_cols);
    }
    // Every row sent to this CTA has arrived before it gets here, unless something timed out: then it stays until the others,
    // who may still be sending, have got as far or are gone.
    if (S > 1 && __syncthreads_or(ok ? 0 : 1)) nm_cluster_sync();
}

// Launch attributes of a kernel in clusters of S CTAs; returns their number.
inline unsigned split_launch_attrs(const nm_ctx* ctx, cudaLaunchAttribute* attr, int S)
{
    unsigned n = 0;
    if (ctx->pdl) {
        attr[n].id = cudaLaunchAttributeProgrammaticStreamSerialization;
        attr[n].val.programmaticStreamSerializationAllowed = 1;
        ++n;
    }
    attr[n].id = cudaLaunchAttributeClusterDimension;
    attr[n].val.clusterDim.x = (unsigned)S;
    attr[n].val.clusterDim.y = 1;
    attr[n].val.clusterDim.z = 1;
    return n + 1;
}

// Which kernel and tile a problem of `rows` rows (`m_tiles` blocks of 128), N columns and `k_blocks` K-blocks gets: the least
// time by a model fitted to measured times in us of chains of equal launches.
//   persistent kernel, 16-bit types: 352 problems, 300 to 16384 rows, N 256 to 4096, K 256 to 4096, with and without a table, each on all six
//     tiles; 3 % off on the average, and the tile it picks 0.5 % behind the best, 9 % at most.  Full rounds of tiles take
//     k_blocks * busy, or their epilogue; a part-filled one between k_blocks * lone and that (counted as a full round, 16384 x
//     1536 x 512 went to a narrower tile: 27.5 us, 21.9 with 256 x 256 pairs); `fill`: what the first tiles and the last
//     epilogue cost more when all SMs run them.  int8: base + every round in full, fitted to 72 problems of up to 4096 rows (the
//     other form picked it too often over the split kernel there, 1024 x 1536 x 512: 5.6 us and 7.9).
//   split kernel, n CTAs: base with the epilogue of the rows that exist + the K-blocks beyond those in flight at once (more when
//     CTAs share an SM) + the exchange.
//   Between kernels that are no matrix products the persistent kernel's longer set-up and tail overlap less, 0.4 us (11 layers, 128
//   tokens: 497 us without it, 437 with), and by how much depends on the tile: fitted to encoders of 300 to 12800 rows with each of
//   their four products on each tile, the picked one is 0.27 us behind the best there, 0.64 without.  A CNN's launches stand back to back and begin while their predecessor drains: there every
//   round counts with its epilogue and narrow tiles do better than alone, so they have a row of parameters of their own (ResNet-50 batch
//   13: 624 us, 657 with the other row; batch 23: 747 and 782).  There, and among the split kernel's widths, the wider tile wins
//   within 3 %: it leaves more SMs to the neighbours.  Elsewhere the split kernel wins within 3 % (37 x 2304 x 768: 4.6 us, 5.4 on
//   persistent tiles).
// E.g. 128 x 768 x 3072: 13.4 us in one round of the best persistent tile, 7.0 split over 8; 1024 x 768 x 768: 5.9 with 128 x 64
// tiles, 9.8 with 256 x 256 pairs.
// `fma_steps`: 0, or the K-steps of 16 of a sum that is to be as good as a chain of FMAs (steps_like_fma; each further
// accumulator costs 0.3 us, 0.9 between other kernels, which wait for its tensor memory).
// `whole_chunks`: a row of the output is a multiple of 16 bytes.  The persistent kernel stores through a tensor map, which
// writes whole 16-byte chunks and would reach beyond a row that is not; the split kernel stores four columns at a time.
struct TileChoice {
    int S;      // CTAs per cluster of the split kernel; 0: the persistent kernel
    int BN;
    bool two;   // persistent kernel: CTA pairs
    double us;  // by the model
    int steps;  // MMA steps per accumulator (TcArgs::acc_steps), 0: all
};

// How many MMA steps of 16 K-elements an accumulator may take if the sum is to be no further from the exact one than a chain of
// fp32 FMAs.  The tensor core truncates the sum at every step: measured against float64, a chain of n steps is off by 1.55e-8 n of
// the sum's rms, a chain of K FMAs by 7.4e-9 sqrt(K) = 3.0e-8 sqrt(steps) (bf16, K 16 to 4096: 2.1e-8, 6.6e-8, 2.4e-7, 7.3e-7, 3.3e-6,
// 4.4e-6 for one accumulator at K 16, 64, 256, 768, 3072, 4096; FMAs 1.9e-8, 5.1e-8, 1.1e-7, 2.1e-7, 5.2e-7, 6.0e-7).
inline int steps_like_fma(int64_t k_steps)
{
    const int n = (int)((k_steps < 32 ? 1.4 : 1.75) * sqrt((double)k_steps) - 0.1);
    return n < 1 ? 1 : n;
}
constexpr int SPLIT_ACC_COLS = 256;   // tensor-memory columns of a CTA: two of them share an SM

// A cluster's CTAs share a GPC, so not every SM is in one: the CTAs, in clusters of S, that certainly find an SM each.
inline bool split_alone(int S, int64_t ctas, int sms) { return ctas <= (S == 8 ? sms * 3 / 4 : sms * 7 / 8); }

// K-blocks in flight per CTA.  One CTA per SM: six stages, or five with 64 columns (12 layers, 37 tokens: 416 us, 436 with the
// shallow ring); more CTAs, or neighbours in the stream of the same kind, whose set-up should overlap: what lets two share an SM
// (ResNet-50 batch 1: 381 us, 430 with the deep ring).  Clusters of 8 fill fewer SMs: 128 CTAs with deep rings ran as two waves
// (48 x 1024 x 4096: 12.4 us against 7.5).
inline int split_stages(int BN, int S, int64_t ctas, int sms, bool back_to_back)
{
    if (S == 1) return 4;
    if (back_to_back) return BN == 64 ? 3 : 4;
    return BN == 64 ? (split_alone(S, ctas, sms) ? 5 : 3) : (split_alone(S, ctas, sms) ? 6 : 4);
}

// The form NM_ALGO_SPLIT asks for; S = -1 if K has too few K-blocks for it.
inline TileChoice forced_split(int32_t algo, int64_t k_blocks)
{
    const int S = algo & 15;
    return {S <= k_blocks ? S : -1, (algo & 0xff0) >> 4, false, 0.0, 0};
}

inline TileChoice choose_tile(int64_t rows, int64_t m_tiles, int64_t N, int64_t k_blocks, bool narrow_tiles, const EpiNeeds& epi, bool only64,
                              bool whole_chunks, int64_t fma_steps, NmChain chain, int sms)
{
    const bool has_table = epi.n_seg > 0;
    struct P { int BN; bool two; double base, lone, busy, round, round_table, table, fill; };
    static const P apart[6] = {{256, true, 5.35, 0.265, 0.358, 1.67, 1.79, 2.36, 0.53}, {256, false, 5.03, 0.272, 0.435, 1.83, 1.35, 2.06, 0.0},
                               {128, true, 3.97, 0.162, 0.240, 1.06, 0.56, 1.42, 0.97}, {128, false, 3.83, 0.161, 0.271, 1.18, 0.48, 1.37, 0.04},
                               {64, true, 3.37, 0.150, 0.208, 0.93, 0.13, 1.42, 1.15},  {64, false, 3.18, 0.165, 0.202, 0.95, 0.05, 1.29, 0.57}};
    struct J { double base, kb, round; };
    static const J int8[2] = {{5.56, 0.420, 4.4}, {4.72, 0.461, 4.8}};
    static const J joined[6] = {{4.9, 0.386, 3.6}, {5.4, 0.43, 3.6}, {4.5, 0.26, 1.8}, {3.9, 0.322, 1.8}, {3.9, 0.26, 0.9}, {3.5, 0.30, 0.9}};
    const bool in_cnn = chain.back_to_back;
    TileChoice best = {1, 64, false, 1e30, 0};   // the split kernel takes anything
    for (int i = 0; i < 6; ++i) {
        const P& p = apart[i];
        if (!whole_chunks || (!narrow_tiles && p.BN != 256) || (only64 && p.BN != 64) || (p.two && m_tiles < 2)) continue;
        if (narrow_tiles && p.BN > 64 && N <= p.BN / 2) continue;   // half the tile would be padding
        if (ring_stages(p.BN, p.two, epi) < 2) continue;            // no room beside a large table
        const int64_t tiles = (p.two ? (m_tiles + 1) / 2 : m_tiles) * ((N + p.BN - 1) / p.BN), slots = p.two ? sms / 2 : sms;
        // (the 64-column tiles have room for up to four accumulators in each of their two buffers)
        const int steps = fma_steps ? steps_like_fma(fma_steps) : 0;
        if (fma_steps && (p.BN != 64 || 4 * k_blocks > 4 * steps)) continue;
        double t;
        if (in_cnn) {
            const J& j = joined[i];
            const double loop = (double)k_blocks * j.kb;
            t = j.base + (double)((tiles + slots - 1) / slots) * (loop < j.round ? j.round : loop) + (has_table ? 1.8 * p.BN / 256 : 0.0);
        } else if (!narrow_tiles) {
            const int64_t rounds = (tiles + slots - 1) / slots;
            const double share = tiles < slots ? (double)tiles / slots : 1.0;
            double loop = (double)k_blocks * int8[i].kb;
            if (rounds > 2 && loop < int8[i].round) loop = int8[i].round;
            t = int8[i].base + (double)rounds * loop + 1.28 * share + (has_table ? 1.5 : 0.0) + (chain.weights_ready ? 0.4 : 0.0);
        } else {
            const double full = (double)(tiles / slots), part = (double)(tiles % slots) / slots, k = (double)k_blocks;
            const double epilogue = p.round + (has_table ? p.round_table : 0.0), busy = k * p.busy, some = k * (p.lone + (p.busy - p.lone) * part);
            t = p.base + full * (busy > epilogue ? busy : epilogue) + (part > 0.0 ? (full > 0.0 && some < epilogue ? epilogue : some) : 0.0) +
                (has_table ? p.table : 0.0) + p.fill * (full > 0.0 ? 1.0 : part);
            if (chain.weights_ready)
                t += 0.8 + (p.BN == 256 ? (has_table ? 1.5 : 0.5) : p.BN == 64 ? (has_table ? -0.8 : -0.4) : has_table || (epi.res && !p.two) ? 0.4 : -0.4);
        }
        if (t < best.us * (in_cnn ? 0.97 : 1.0)) best = {0, p.BN, p.two, t, steps};
    }
    const double tile_rows = (rows < BM ? (double)rows : (double)BM) / BM;
    for (int BN = 64; BN >= (only64 ? 64 : 32); BN /= 2) {
        const int64_t tiles = m_tiles * ((N + BN - 1) / BN);
        for (int S = 1; S <= 8 && S <= k_blocks; S *= 2) {
            const int64_t n = tiles * S;
            if (n > 0x7fffffffLL || (n > 2 * sms && (fma_steps ? best.us < 1e30 : whole_chunks || S > 1))) break;
            int steps = 0;
            if (fma_steps) {
                const int64_t mine = 4 * ((k_blocks + S - 1) / S), most = SPLIT_ACC_COLS / BN;
                steps = steps_like_fma(fma_steps);
                if (mine > steps * most) {
                    // (more than 150 000 K-elements: nothing does, and the last form takes longer chains)
                    if (BN > 32 || best.us < 1e30 || (S < 8 && 2 * S <= k_blocks)) continue;
                    steps = (int)((mine + most - 1) / most);
                }
            }
            const double per = (double)((k_blocks + S - 1) / S), share = (double)n / sms, beyond = per - split_stages(BN, S, n, sms, in_cnn);
            const double t = 4.29 + 0.73 * tile_rows * BN / 64 + 0.038 * per +
                             (BN == 64 ? 0.235 : 0.179) * (beyond > 0 ? beyond : 0) * (share > 1 ? share : 1) +
                             (S == 1 ? 0.0 : S == 2 ? 0.21 : S == 4 ? 0.26 : 0.56) +
                             (0.35 * (share < 1 ? share : 1) + 0.85 * (share > 1 ? share - 1 : 0)) * BN / 32 + (has_table ? 0.42 * BN / 64 : 0.0) +
                             (steps ? (chain.weights_ready ? 0.9 : 0.3) * (double)(int)((4.0 * per - 1.0) / steps) : 0.0);
            if (t < best.us * (in_cnn || best.S ? 0.97 : 1.03)) best = {S, BN, false, t, steps};
        }
    }
    return best;
}

template <typename InT, typename OutT, int BN, bool CONV>
inline nm_status launch_split_kernel(nm_ctx* ctx, const CUtensorMap& tmA, const CUtensorMap& tmW, SplitArgs& s, bool back_to_back,
                                     double work, cudaStream_t st)
{
    constexpr int STAGE_BYTES = A_BYTES + BN * ROW_BYTES;
    constexpr int PART_BYTES = BM * part_pitch(BN) * 4;   // without a split it takes the ring's place and must fit in it
    constexpr int MIN_STAGES = (PART_BYTES + STAGE_BYTES - 1) / STAGE_BYTES;
    static_assert(MIN_STAGES <= 3, "partial tile");
    const int per = (s.t.num_k_blocks + s.S - 1) / s.S, most = split_stages(BN, s.S, (int64_t)s.t.num_tiles * s.S, ctx->sm_count, back_to_back);
    s.t.accs = s.t.acc_steps ? (4 * per + s.t.acc_steps - 1) / s.t.acc_steps : 1;
    s.t.stages = per < MIN_STAGES ? MIN_STAGES : (per > most ? most : per);
    const size_t smem = (size_t)s.t.stages * STAGE_BYTES + (s.S > 1 ? PART_BYTES : 0) + 1024;
    auto kern = s.S == 1   ? linear_split_kernel<InT, OutT, BN, CONV, 1>
                : s.S == 2 ? linear_split_kernel<InT, OutT, BN, CONV, 2>
                : s.S == 4 ? linear_split_kernel<InT, OutT, BN, CONV, 4>
                           : linear_split_kernel<InT, OutT, BN, CONV, 8>;
    if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)(SPLIT_MAX_STAGES * STAGE_BYTES + PART_BYTES + 1024)) !=
        cudaSuccess)
        return NM_ERR_CUDA;
    cudaLaunchConfig_t cfg;
    memset(&cfg, 0, sizeof(cfg));
    cfg.gridDim = dim3((unsigned)(s.t.num_tiles * s.S));
    cfg.blockDim = dim3(SPLIT_THREADS);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute attr[2];
    cfg.attrs = attr;
    cfg.numAttrs = split_launch_attrs(ctx, attr, s.S);
    NmLaunchScope scope(ctx, NM_KERNEL_LINEAR_TC, work, st);
    if (cudaLaunchKernelEx(&cfg, kern, tmA, tmW, s) != cudaSuccess) return NM_ERR_CUDA;
    return cudaGetLastError() == cudaSuccess ? NM_OK : NM_ERR_CUDA;
}

}  // namespace nm_tc

// Fused attention with PWL softmax, streaming variant: several CTAs per SM.
//
// Same function as attention_tc.cu (Section 3.1: attention is a linear operator; Section 3.2.2:
// exp and 1/x as PWL tables), per query row
//     s_j = scale*<q,k_j>;  m = max_j s_j;  e_j = PWL_exp(s_j - m);  sigma = sum_j e_j;
//     o = PWL_recip(sigma) * sum_j e_j v_j
// with m the FINAL row maximum (a PWL exponential is not multiplicative, so there is no
// running-maximum rescaling).  Instead of keeping the whole 128 x L score block in tensor memory,
// this kernel computes Q K^T TWICE: a first sweep over the keys only for the row maximum, a second
// sweep for the exponentials.  The tensor pipe is idle most of the time in this ALU-bound kernel, so
// the second Q K^T is free, and the footprint drops to 128 tensor-memory columns and ~50 KB of
// shared memory (plus Q and the table): three CTAs fit on an SM and one CTA's loads, MMAs and hand-offs
// overlap the others' arithmetic.
//
// CTAs are persistent: one resident wave (three per SM) walks over the (batch, head, 128-query block) tiles.
// Barriers, tensor memory and the replicated table are set up once per CTA; every mbarrier's phase is a running
// count carried from tile to tile; after a tile's last Q K^T the control warp already fetches the next tile's Q
// and first K chunks, after its last P V the next first V chunk, and the next tile's first product starts as
// soon as the softmax warps have read the accumulator out of tensor memory.
//
// The 16-bit P tile never touches shared memory: the softmax warps write it to further tensor-memory columns
// (tcgen05.st) and P V takes its A operand from there; the shared-memory pipe, which the table lookups load most,
// loses the tile's stores and the tensor core's reads of it.
//
// RAGGED form (an L that is not a multiple of 128, otherwise the CUDA-core kernel's): the tensor maps fill rows
// beyond the sequence with zeros, the scores of keys beyond L are masked in the last block only, and warps whose
// 32 queries all lie beyond L keep the barriers' pace without arithmetic.  The CUDA-core kernel holds its
// probabilities in fp32, so this form does not round them to 16 bits: a bf16 P is three terms whose sum is e exactly,
// an fp16 P two terms of 22 bits of e, scaled by a power of two per row; all of a probability's terms have its sign and
// none of them is zero, so that an infinite V gives an infinity and not 0 * inf (ProbTerms).  The tensor core truncates
// its sums, so the second and third terms, 2^-8 and less of the first, are kept out of the first one's sum: they have an
// accumulator of their own, or go first.  Outputs that are not the correctly rounded ones, of all, at L 37 / 333 / 500, with
// one accumulator and two rounded terms, so, and on the CUDA cores: bf16 2.2e-3, 2.4e-3, 2.5e-3 | 1.0e-4, 1.7e-4, 2.2e-4 |
// 1.3e-4, 2.6e-4, 3.1e-4; fp16 0.9e-3, 3.5e-3, 5.0e-3 | 0.9e-3, 1.9e-3, 2.6e-3 | 1.0e-3, 1.7e-3, 2.0e-3.
// The terms of 32 keys at a time, 48 columns, lie behind the second accumulator: 256 columns, two CTAs per SM.
// B 7, L 333, 12 heads: 2368 us on the CUDA cores, 21.7 here (18.7 with two rounded terms); B 32, L 500: 141 (112).
//
// ONE form (L <= 128, a single 128-key chunk): the scores and the accumulator do not share columns (128 | 64, and P behind
// them: 256 columns, two CTAs per SM), so the one Q K^T of sweep 1 serves sweep 2 as well, and nothing is fetched or
// multiplied twice in what is then a latency-bound kernel (B 1, L 128, 16 heads: 6.4 -> 4.9 us).  All of V is fetched at once and P V
// runs once, over all keys.  DUO (launch_one says when): two softmax warps share 32 rows, half of the blocks of 16 keys each; the second one's
// sums go on from the first one's, in the order that one warp would take, so that the forms agree in every bit (int8 24 layers, 128 tokens: 889 -> 849 us; with several chunks per tile, where
// the shared-memory pipe is the bound, two warps per quarter lose: B 32, L 512, 12 heads 70.8 -> 80.1).  RAGGED and ONE: the first two
// terms of a block of 16 keys take the place of its scores, the third goes behind the accumulator, and P V takes the smallest
// terms first, instead of one product per 64 keys (B 32, L 100, 12 heads: 15.0 -> 12.6 us; B 1, L 37: 4.6).
//
//   warp 0            control: TMA loads (K chunks through two stages, V chunks through one) and the tcgen05.mma
//                     for S = Q K_c^T and O += P_c V_c (V as an MN-major operand).  It sleeps in a named barrier
//                     (bar.sync) that the softmax warps signal with bar.arrive, so hand-offs cost no polling.
//   warps 1..4 (DUO: 1..8)  softmax, one (two) per tensor-memory lane quarter: tcgen05.ld, row maximum (sweep 1); PWL exp, row
//                     sum, P tile (sweep 2); PWL reciprocal, scaling, store (optionally as int8 codes for the int8
//                     encoder).
#include <string.h>

#include <type_traits>

#include "nm_common.cuh"

namespace {

constexpr int BQ = 128;    // query rows per CTA
constexpr int HD = 64;     // head dimension
constexpr int CK = 64;     // keys per chunk
constexpr int ROWB = 128;  // bytes per tile row (64 x 16-bit)
constexpr int STAGE = CK * ROWB;      // 8 KB
constexpr int PBUF = BQ * ROWB;       // 16 KB

struct SArgs {
    int B, L, heads;
    float scale;
    const NmTable* t_exp;
    const NmTable* t_rcp;
    void* out;
    int* status;
    int n_exp;
    float e_max;         // RAGGED, fp16: the largest |PWL_exp(x)| for x from the table's lower end to 0
    int8_t* out_q;       // when set: the output goes out as int8 codes (of the value rounded to T) instead
    float q_inv_scale;
};

template <typename T> struct AT;
template <> struct AT<__nv_bfloat16> {
    static constexpr uint32_t fmt = 1;
    static __device__ __forceinline__ float round(float a) { return __bfloat162float(__float2bfloat16_rn(a)); }
    static __device__ __forceinline__ uint32_t pack(float a, float b)
    {
        __nv_bfloat162 h = __floats2bfloat162_rn(a, b);
        return *reinterpret_cast<uint32_t*>(&h);
    }
};
template <> struct AT<__half> {
    static constexpr uint32_t fmt = 0;
    static __device__ __forceinline__ float round(float a) { return __half2float(__float2half_rn(a)); }
    static __device__ __forceinline__ uint32_t pack(float a, float b)
    {
        __half2 h = __floats2half2_rn(a, b);
        return *reinterpret_cast<uint32_t*>(&h);
    }
};

// Two probabilities as 16-bit terms, one packed word per term.  Each term but the last is the remainder so far rounded
// towards zero and, being cut from a value one unit lower (the product with 1 - 2^-24, rounded towards zero), always smaller
// than the remainder: the next term is never zero and has the same sign, and a zero probability has only zero terms.
// bf16, 8 bits a term: after two terms at most 8 bits are left, so the three add up to e exactly.  fp16, 11 bits a term.
template <typename T> struct ProbTerms;
template <> struct ProbTerms<__nv_bfloat16> {
    static constexpr int N = 3;
    static __device__ __forceinline__ void split(float e0, float e1, uint32_t& w0, uint32_t& w1, uint32_t& w2)
    {
        const float below = 0x1.fffffep-1f;   // 1 - 2^-24
        const uint32_t h0 = __float_as_uint(__fmul_rz(e0, below)), h1 = __float_as_uint(__fmul_rz(e1, below));
        const float r0 = e0 - __uint_as_float(h0 & 0xffff0000u), r1 = e1 - __uint_as_float(h1 & 0xffff0000u);
        const uint32_t m0 = __float_as_uint(__fmul_rz(r0, below)), m1 = __float_as_uint(__fmul_rz(r1, below));
        const float l0 = r0 - __uint_as_float(m0 & 0xffff0000u), l1 = r1 - __uint_as_float(m1 & 0xffff0000u);
        w0 = __byte_perm(h0, h1, 0x7632);
        w1 = __byte_perm(m0, m1, 0x7632);
        w2 = __byte_perm(__float_as_uint(l0), __float_as_uint(l1), 0x7632);
    }
};
template <> struct ProbTerms<__half> {
    static constexpr int N = 2;
    static __device__ __forceinline__ void split(float e0, float e1, uint32_t& w0, uint32_t& w1, uint32_t&)
    {
        const float below = 0x1.fffffep-1f;
        asm("cvt.rz.f16x2.f32 %0, %1, %2;" : "=r"(w0) : "f"(__fmul_rz(e1, below)), "f"(__fmul_rz(e0, below)));
        const float2 hi = __half22float2(*reinterpret_cast<const __half2*>(&w0));
        w1 = AT<__half>::pack(e0 - hi.x, e1 - hi.y);
    }
};

__device__ __forceinline__ float max3f(float a, float b, float c)
{
    float d;
    asm("max.f32 %0, %1, %2, %3;" : "=f"(d) : "f"(a), "f"(b), "f"(c));
    return d;
}

// A tile is one (batch, head, 128-query block); tile index = (b * heads + g) * blocks_per_seq + qb.
struct Tile { int qb, g, b; };
struct TileGeom { int blocks_per_seq, heads; };
__device__ __forceinline__ Tile tile_decode(const TileGeom& gm, int t)
{
    Tile r;
    r.qb = t % gm.blocks_per_seq;
    r.g = (t / gm.blocks_per_seq) % gm.heads;
    r.b = t / (gm.blocks_per_seq * gm.heads);
    return r;
}
// What the first loads of a tile need: tensor maps, staging buffers, their barriers.
struct LoadCtx {
    const CUtensorMap *tmQ, *tmK, *tmV;
    uint8_t *q_s, *k_st, *p_s, *v_st;
    uint64_t *bar_q, *bar_k1_full, *bar_v_full;   // bar_k1_full: [2]
    int n128, v_chunks;
};
// Q and the first two 128-key chunks of sweep 1 (stage 0 = the two K stages, stage 1 = the buffer p_s).  One
// thread; the buffers must be free.
__device__ __forceinline__ void load_tile_head(const LoadCtx& c, const Tile& t)
{
    nm_mbar_expect_tx(c.bar_q, BQ * ROWB);
    nm_tma_load_3d(c.q_s, c.tmQ, t.g * HD, t.qb * BQ, t.b, c.bar_q);
#pragma unroll
    for (int st = 0; st < 2; ++st) {
        if (st >= c.n128) break;
        uint8_t* dst = st == 0 ? c.k_st : c.p_s;
        uint64_t* bar = c.bar_k1_full + st;
        nm_mbar_expect_tx(bar, 2 * STAGE);
        nm_tma_load_3d(dst, c.tmK, t.g * HD, st * 2 * CK, t.b, bar);
        nm_tma_load_3d(dst + STAGE, c.tmK, t.g * HD, st * 2 * CK + CK, t.b, bar);
    }
}
// The first V chunk of a tile, or all of its V (one thread; the V stage must be free).
__device__ __forceinline__ void load_first_v(const LoadCtx& c, const Tile& t)
{
    nm_mbar_expect_tx(c.bar_v_full, c.v_chunks * STAGE);
    for (int i = 0; i < c.v_chunks; ++i) nm_tma_load_3d(c.v_st + i * STAGE, c.tmV, t.g * HD, i * CK, t.b, c.bar_v_full);
}

// Forms: several 128-key chunks; ONE: a single one; DUO: a single one, with two softmax warps per lane quarter instead of one.
enum Form { MANY, ONE_CHUNK, DUO_CHUNK };
// Threads of a CTA: the control warp and the softmax warps.
template <Form FORM> constexpr int CTA_THREADS = FORM == DUO_CHUNK ? 288 : 160;

// PER_SM: CTAs that an SM holds, by registers and tensor memory three, with 256 columns two.  RAGGED and DUO: two with 96 registers, of which
// 24 bytes spill, or one with 162.
template <typename T, bool CLAMP_HI, bool RAGGED, Form FORM, int PER_SM>
__global__ void __launch_bounds__(CTA_THREADS<FORM>, PER_SM)
attention_stream_kernel(const __grid_constant__ CUtensorMap tmQ, const __grid_constant__ CUtensorMap tmK,
                        const __grid_constant__ CUtensorMap tmV, const SArgs a)
{
    constexpr bool ONE = FORM != MANY, DUO = FORM == DUO_CHUNK;
    constexpr uint32_t IDESC_QK = nm_idesc(1, AT<T>::fmt, 0, 0, BQ, CK);   // S chunk: 128 x 64
    constexpr uint32_t IDESC_PV = nm_idesc(1, AT<T>::fmt, 0, 1, BQ, HD);   // O: 128 x 64, V MN-major
    constexpr uint32_t IDESC_QK1 = nm_idesc(1, AT<T>::fmt, 0, 0, BQ, 2 * CK);   // sweep 1: 128 x 128
    // S | O, sweep 1 writes 128 keys over [S | O]; ONE: S of 128 keys | O | P
    constexpr uint32_t TMEM_COLS = ONE ? 256 : 128;
    constexpr uint32_t O_OFF = ONE ? 128 : 64;
    // The 16-bit P tile goes through a second allocation of 32 columns (64 keys, two per column) and is the A operand
    // of P V from there; three CTAs hold 3 x (128 + 32) of the SM's 512 columns.  RAGGED: 64 columns for the sum of the
    // lower terms and 64 for the terms of 32 keys, 16 columns each.
    constexpr uint32_t P_COLS = RAGGED ? 128 : 32;
    constexpr int TERMS = RAGGED ? ProbTerms<T>::N : 1;
    constexpr bool SCALED = RAGGED && std::is_same<T, __half>::value;
    constexpr int NT = CTA_THREADS<FORM>;
    constexpr int LD = DUO ? 16 : 32;   // scores that sweep 1 reads at a time

    extern __shared__ uint8_t smem_raw[];
    __shared__ uint64_t bar_q, bar_drain;
    __shared__ uint64_t bar_k_full[2], bar_k1_full[2], bar_v_full, bar_s_full, bar_p_empty;
    __shared__ uint32_t tmem_slot, tmem_slot_p;
    __shared__ int abort_flag;
    // DUO: the two warps' row maxima (SCALED: and minima), and what they pass on to add a row up as one of them would
    __shared__ float s_pair[DUO ? 2 : 1][2][BQ];
    __shared__ float4 s_sum[DUO ? 9 : 1][DUO ? BQ : 1];

    const int L = a.L;
    const int n = RAGGED ? (L + CK - 1) / CK : L / CK;                    // 64-key chunks of sweep 2
    // P V products: one for all keys (ONE), one per 32 keys (RAGGED), otherwise one per chunk
    const int n_pv = ONE ? 1 : !RAGGED ? n : (L + 31) / 32;
    const int n128 = ONE ? 1 : RAGGED ? (L + 2 * CK - 1) / (2 * CK) : L / (2 * CK);   // 128-key chunks of sweep 1
    uint8_t* base = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
    uint8_t* q_s = base;                       // 16 KB
    uint8_t* k_st = q_s + BQ * ROWB;           // 2 x 8 KB
    uint8_t* v_st = k_st + 2 * STAGE;          // 8 KB
    uint8_t* p_s = v_st + STAGE;               // 16 KB: sweep 1's second K stage
    float2* rep = reinterpret_cast<float2*>(p_s + PBUF);   // (n_exp + 1) x 16 copies

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    // A CTA walks over the (batch, head, 128-query block) tiles blockIdx.x, blockIdx.x + gridDim.x, ...: barriers,
    // tensor memory and the replicated table are set up once, and the control warp fetches the next tile's Q,
    // first K chunks and first V chunk while the softmax warps finish the current one.
    const int blocks_per_seq = n128;   // BQ = 2 CK
    const int n_tiles = a.B * a.heads * blocks_per_seq;
    const TileGeom geom = {blocks_per_seq, a.heads};
    auto tile_of = [geom](int t) { return tile_decode(geom, t); };
    LoadCtx lc;
    lc.tmQ = &tmQ; lc.tmK = &tmK; lc.tmV = &tmV;
    lc.q_s = q_s; lc.k_st = k_st; lc.p_s = p_s; lc.v_st = v_st;
    lc.bar_q = &bar_q; lc.bar_k1_full = &bar_k1_full[0]; lc.bar_v_full = &bar_v_full;
    lc.n128 = n128;
    lc.v_chunks = 1;
    if (ONE) {   // all of V in the buffer that sweep 1 of longer sequences takes
        lc.v_st = p_s;
        lc.v_chunks = n;
    }

    if (threadIdx.x == 0) {
        abort_flag = 0;
        nm_prefetch_tmap(&tmQ);
        nm_prefetch_tmap(&tmK);
        nm_prefetch_tmap(&tmV);
        nm_mbar_init(&bar_q, 1);
        nm_mbar_init(&bar_drain, 1);
        nm_mbar_init(&bar_k_full[0], 1);
        nm_mbar_init(&bar_k_full[1], 1);
        nm_mbar_init(&bar_k1_full[0], 1);
        nm_mbar_init(&bar_k1_full[1], 1);
        nm_mbar_init(&bar_v_full, 1);
        nm_mbar_init(&bar_s_full, 1);
        nm_mbar_init(&bar_p_empty, 1);
        nm_fence_barrier_init();
        // The first copies go out before the rest of the set-up (tensor-memory allocation, table
        // replication, block barrier), so that their latency overlaps it: Q, the first two 128-key chunks
        // of sweep 1 and the first V chunk.
        nm_grid_dependency_wait();   // Q, K, V come from the previous kernel
        if ((int)blockIdx.x < n_tiles) {
            const Tile t0 = tile_of((int)blockIdx.x);
            load_tile_head(lc, t0);
            load_first_v(lc, t0);
        }
    }
    if (warp == 0) {
        nm_tmem_alloc(&tmem_slot, TMEM_COLS);
        if constexpr (!ONE) nm_tmem_alloc(&tmem_slot_p, P_COLS);
        nm_tmem_relinquish();
    } else {
        // 16-way replicated exp table: entry s, copy c at rep[s*16 + c].  A 64-bit warp load is served
        // half a warp at a time, so 16 copies already make arbitrary lookups conflict-free.  One extra
        // entry (a copy of the last) lets input 0 of a table whose range ends at 0 go unclamped.
        const int ne = a.n_exp;
        for (int i = threadIdx.x - 32; i < (ne + 1) * 16; i += NT - 32) rep[i] = a.t_exp->kb[min(i >> 4, ne - 1)];
    }
    nm_tc_fence_before();
    __syncthreads();
    nm_tc_fence_after();
    const uint32_t tmem_base = tmem_slot;
    const uint32_t tmem_p = ONE ? tmem_base + 192u : tmem_slot_p;
    const uint32_t tmem_lo = tmem_slot_p, tmem_t = tmem_slot_p + 64u;   // RAGGED, not ONE: sum of the lower terms; the terms
    volatile int* abortp = &abort_flag;
    nm_grid_launch_dependents();   // the next kernel may start its set-up
    nm_grid_dependency_wait();     // Q, K, V come from the previous kernel

    if (warp == 0) {
        // ------------------------------------------------ control warp
        // Runs with all 32 lanes (barrier tests, counters and descriptors stay warp-uniform); one
        // elected lane issues the TMA and tcgen05 instructions.  It sleeps in a named barrier until
        // the four softmax warps have arrived there, so signalling costs no polling:
        //   S-consumed(i): chunk i's scores are in registers -> K stage i & 1 is free (load the chunk
        //                  after next into it) and S is free (issue Q K^T for the next chunk);
        //   P-ready(j):    the P tile of the j-th chunk of sweep 2 is in tensor memory -> O += P V.
        const uint32_t bar_sc = 2, bar_pr = 3, bar_oc = 6;
        auto wait = [&](uint64_t* bar, uint32_t parity) {
            return __all_sync(0xffffffffu, nm_mbar_wait_relaxed<20>(bar, parity, abortp, a.status)) != 0;
        };
        bool ok = true;
        const uint64_t qdesc = nm_smem_desc_sw128(nm_smem_u32(q_s));
        // completions consumed so far on each barrier (they run on from tile to tile)
        uint32_t q_cnt = 0, k1_cnt0 = 0, k1_cnt1 = 0, k_cnt0 = 0, k_cnt1 = 0, v_cnt = 0, pv_cnt = 0;
        for (int tile = (int)blockIdx.x, ti = 0; tile < n_tiles; tile += (int)gridDim.x, ++ti) {
            const Tile t = tile_of(tile);
            const int g = t.g, b = t.b;
            const bool more = tile + (int)gridDim.x < n_tiles;
            if (ok && !wait(&bar_q, q_cnt & 1u)) ok = false;
            ++q_cnt;
            // the previous tile's epilogue has read O out of tensor memory (sweep 1 writes over [S | O])
            if (ti > 0) asm volatile("bar.sync %0, %1;" ::"r"(bar_oc), "n"(NT) : "memory");
            // ---- sweep 1: [S | O] = Q K^T for 128 keys at a time; K stage i & 1 (0: the two K stages
            // taken together, 1: the P tile)
            auto issue_qk1 = [&](int i) {
                const uint32_t par = ((i & 1) ? k1_cnt1 : k1_cnt0) & 1u;
                if (i & 1) ++k1_cnt1; else ++k1_cnt0;
                if (!ok) return;
                if (!wait(&bar_k1_full[i & 1], par)) { ok = false; return; }
                nm_tc_fence_after();
                const uint64_t kdesc = nm_smem_desc_sw128(nm_smem_u32((i & 1) ? p_s : k_st));
                if (nm_elect_one()) {
#pragma unroll
                    for (int k = 0; k < 4; ++k) nm_mma_f16(tmem_base, qdesc + 2 * k, kdesc + 2 * k, IDESC_QK1, k != 0);
                    nm_tc_commit(&bar_s_full);
                }
                __syncwarp();
            };
            if (n128 > 0) issue_qk1(0);
            for (int i = 0; !ONE && i < n128; ++i) {
                asm volatile("bar.sync %0, %1;" ::"r"(bar_sc), "n"(NT) : "memory");   // S-consumed: chunk i is in registers
                if (i + 1 < n128) issue_qk1(i + 1);
                if (ok && i + 2 < n128 && nm_elect_one()) {   // its MMAs are complete: the stage takes the chunk after next
                    uint8_t* dst = (i & 1) ? p_s : k_st;
                    const int key0 = (i + 2) * 2 * CK;
                    nm_mbar_expect_tx(&bar_k1_full[i & 1], 2 * STAGE);
                    nm_tma_load_3d(dst, &tmK, g * HD, key0, b, &bar_k1_full[i & 1]);
                    nm_tma_load_3d(dst + STAGE, &tmK, g * HD, key0 + CK, b, &bar_k1_full[i & 1]);
                }
                __syncwarp();
            }
            // ---- sweep 2: chunk j is 64 keys; K stage j & 1
            auto load_k = [&](int j) {
                if (ok && nm_elect_one()) {
                    nm_mbar_expect_tx(&bar_k_full[j & 1], STAGE);
                    nm_tma_load_3d(k_st + (size_t)(j & 1) * STAGE, &tmK, g * HD, j * CK, b, &bar_k_full[j & 1]);
                }
                __syncwarp();
            };
            auto issue_qk = [&](int j) {   // S = Q K^T
                const uint32_t par = ((j & 1) ? k_cnt1 : k_cnt0) & 1u;
                if (j & 1) ++k_cnt1; else ++k_cnt0;
                if (!ok) return;
                if (!wait(&bar_k_full[j & 1], par)) { ok = false; return; }
                nm_tc_fence_after();
                const uint64_t kdesc = nm_smem_desc_sw128(nm_smem_u32(k_st + (size_t)(j & 1) * STAGE));
                if (nm_elect_one()) {
#pragma unroll
                    for (int k = 0; k < 4; ++k) nm_mma_f16(tmem_base, qdesc + 2 * k, kdesc + 2 * k, IDESC_QK, k != 0);
                    nm_tc_commit(&bar_s_full);
                }
                __syncwarp();
            };
            if constexpr (!ONE) {
                load_k(0);   // every MMA of sweep 1 has completed: the K stages are free
                if (n > 1) load_k(1);
                issue_qk(0);
            }
            for (int u = 0; u < n_pv; ++u) {
                const int j = RAGGED && !ONE ? u >> 1 : u;                              // chunk
                const bool chunk_ends = !RAGGED || ONE || (u & 1) || u + 1 == n_pv;     // (it holds one or two P V products)
                const bool chunk_begins = !RAGGED || ONE || !(u & 1);
                if constexpr (!ONE) {
                    if (chunk_ends) {
                        asm volatile("bar.sync %0, %1;" ::"r"(bar_sc), "n"(NT) : "memory");   // S-consumed(j)
                        if (j + 1 < n) issue_qk(j + 1);
                        if (j + 2 < n) load_k(j + 2);
                    }
                } else if (u + 1 == n_pv && more && ok) {
                    if (!wait(&bar_s_full, (uint32_t)ti & 1u)) ok = false;   // the tile's one product has read Q and K
                }
                // Last product: every Q K^T of the tile has completed, so Q, the K stages and p_s take the next tile's
                // first loads now.
                if (u + 1 == n_pv && more && ok && nm_elect_one()) load_tile_head(lc, tile_of(tile + (int)gridDim.x));
                __syncwarp();
                asm volatile("bar.sync %0, %1;" ::"r"(bar_pr), "n"(NT) : "memory");   // P-ready(u)
                if (chunk_begins) {
                    if (ok && !wait(&bar_v_full, v_cnt & 1u)) ok = false;
                    ++v_cnt;
                }
                if (ok) {
                    nm_tc_fence_after();
                    const uint32_t v_addr = nm_smem_u32(lc.v_st);
                    // V rows (keys) 16 k .. 16 k + 15 of the stage: two groups of 8 rows, 1024 bytes apart
                    auto vdesc = [v_addr](int k) { return nm_smem_desc_sw128(v_addr + (uint32_t)(16 * k * ROWB)); };
                    if (nm_elect_one()) {
                        if constexpr (!RAGGED) {
#pragma unroll
                            for (int k = 0; k < (ONE ? 8 : 4); ++k)
                                nm_mma_f16_a_tmem(tmem_base + O_OFF, tmem_p + (uint32_t)(8 * k), vdesc(k), IDESC_PV, (j | k) != 0);
                        } else if constexpr (ONE) {
                            const int steps = (L + 15) / 16;
#pragma unroll
                            for (int t = TERMS - 1; t >= 0; --t)
                                for (int k = 0; k < steps; ++k)
                                    nm_mma_f16_a_tmem(tmem_base + O_OFF, t == 2 ? tmem_p + (uint32_t)(8 * k) : tmem_base + (uint32_t)(16 * k + 8 * t),
                                                   vdesc(k), IDESC_PV, t != TERMS - 1 || k != 0);
                        } else {
                            const int k0 = 2 * (u & 1);
#pragma unroll
                            for (int t = TERMS - 1; t >= 0; --t)
#pragma unroll
                                for (int k = 0; k < 2; ++k)
                                    nm_mma_f16_a_tmem(t == 0 ? tmem_base + O_OFF : tmem_lo, tmem_t + (uint32_t)(16 * t + 8 * k), vdesc(k0 + k), IDESC_PV,
                                                   u != 0 || k != 0 || (t != 0 && t != TERMS - 1));
                        }
                        nm_tc_commit(&bar_p_empty);
                    }
                    __syncwarp();
                }
                const uint32_t pv_par = pv_cnt & 1u;   // parity of this P V's completion
                ++pv_cnt;
                // the V stage is free once this P V has completed (nothing else to do until then): it takes the
                // next chunk's V, or after the last chunk the next tile's first one
                const bool last = u + 1 == n_pv;
                if (ok && chunk_ends && (!last || more)) {
                    if (!wait(&bar_p_empty, pv_par)) ok = false;
                    if (ok && nm_elect_one()) {
                        if (!last) {
                            nm_mbar_expect_tx(&bar_v_full, STAGE);
                            nm_tma_load_3d(v_st, &tmV, g * HD, (j + 1) * CK, b, &bar_v_full);
                        } else {
                            load_first_v(lc, tile_of(tile + (int)gridDim.x));
                        }
                    }
                    __syncwarp();
                }
            }
        }
        if (!ok) {   // after an abort: let copies land and MMAs retire (bounded) before teardown
            if (nm_elect_one()) {
                nm_tc_commit(&bar_drain);
                long long t0 = clock64();
                while (!nm_mbar_try_wait(&bar_drain, 0) && clock64() - t0 < 200000000LL) {}
                while (clock64() - t0 < 4000000LL) {}
            }
            __syncwarp();
        }
    } else {
        // ------------------------------------------------ softmax warps
        // One row per thread.  A warp never blocks on the others: it signals the control warp with bar.arrive.
        const int q = warp & 3;
        const int row = q * 32 + lane;
        const int part = DUO ? (warp - 1) >> 2 : 0;   // which of the two warps that share 32 rows, half of the blocks of 16 keys each
        const int blocks = RAGGED ? (L + 15) / 16 : 8, first = part * ((blocks + 1) / 2), last = part || !DUO ? blocks : (blocks + 1) / 2;   // ONE: its blocks
        const uint32_t bar_sc = 2, bar_pr = 3, bar_oc = 6;
        // this row's value of the other warp, which takes the same steps
        [[maybe_unused]] auto swap = [&](float (*buf)[BQ], float v) {
            buf[part][row] = v;
            asm volatile("bar.sync %0, 64;" ::"r"(8 + q) : "memory");
            return buf[part ^ 1][row];
        };
        const uint32_t t_row = tmem_base + ((uint32_t)(q * 32) << 16);
        const float inv_h = a.t_exp->inv_h, off = a.t_exp->off, nm1 = (float)(a.n_exp - 1);
        // this lane's copy of the replicated table, with the constant of the index trick folded in:
        // (bits << 7) = 0xA0000000 + s*128 (mod 2^32) for bits = 0x4B400000 + s
        const uint32_t rep_lane = nm_smem_u32(rep) + (uint32_t)(lane & 15) * 8u - 0xA0000000u;
        const uint64_t scale2 = nm_pack2(a.scale, a.scale), inv_h2 = nm_pack2(inv_h, inv_h), off2 = nm_pack2(off, off);
        const uint64_t magic2 = nm_pack2(12582912.0f, 12582912.0f);
        const uint32_t p_row = tmem_p + ((uint32_t)(q * 32) << 16);   // this warp's lane quarter of the P columns
        int ok = 1;
        // All lanes test the barrier; only when it is not yet complete does lane 0 poll (with sleeps).
        auto wait_all = [&](uint64_t* bar, uint32_t par) {
            if (!ok) return;
            const bool done = nm_mbar_try_wait(bar, par);
            if (!__all_sync(0xffffffffu, done)) {
                int w = 1;
                if (lane == 0) w = nm_mbar_wait_relaxed(bar, par, abortp, a.status) ? 1 : 0;
                ok = __shfl_sync(0xffffffffu, w, 0);
                if (ok) (void)nm_mbar_try_wait(bar, par);
            }
        };
        // completions consumed so far: S products, P V products
        uint32_t s_cnt = 0, pv_base = 0;
        float r_inv_h = 0.f, r_off = 0.f, r_nm1 = 0.f;   // fetched early where latency counts and registers do not
        if constexpr (ONE) {
            r_inv_h = a.t_rcp->inv_h;
            r_off = a.t_rcp->off;
            r_nm1 = (float)(a.t_rcp->n - 1);
        }
        for (int tile = (int)blockIdx.x; tile < n_tiles; tile += (int)gridDim.x) {
            const Tile t = tile_of(tile);
            const int qb = t.qb, g = t.g, b = t.b;
            const bool more = tile + (int)gridDim.x < n_tiles;
            // RAGGED: a warp whose 32 queries all lie beyond the sequence waits and signals like the others, but
            // computes nothing (its rows of the accumulator are never stored)
            const bool live = !RAGGED || qb * BQ + q * 32 < L;
            // ---- sweep 1: the final row maximum
            float m = -INFINITY;
            [[maybe_unused]] float lowest = INFINITY;   // SCALED: the smallest score
#pragma unroll 1
            for (int i = 0; i < n128; ++i) {
                wait_all(&bar_s_full, s_cnt & 1u);
                ++s_cnt;
                if (ok && live) {
                    nm_tc_fence_after();
#pragma unroll
                    for (int hh = 0; hh < 4; ++hh) {   // 128 keys: the scores span [S | O]
                        uint32_t r[LD];
                        const int key = DUO ? (first + hh) * 16 : hh * 32;
                        if (DUO ? first + hh >= last : RAGGED && ONE && key >= L) continue;   // no keys there
                        if constexpr (DUO) nm_tmem_ld16_sync(t_row + (uint32_t)key, r);
                        else nm_tmem_ld32_sync(t_row + (uint32_t)key, r);
                        if (!ONE && hh == 3) {   // all of it is in registers: the control warp may overwrite S
                            nm_tc_fence_before();
                            asm volatile("bar.arrive %0, %1;" ::"r"(bar_sc), "n"(NT) : "memory");
                        }
                        if (RAGGED && i == n128 - 1) {   // keys beyond L do not take part
                            const int lim = L - i * 2 * CK - key;
#pragma unroll
                            for (int k = 0; k < LD; ++k) {
                                if (SCALED && k < lim) lowest = fminf(lowest, __uint_as_float(r[k]));
                                if (k >= lim) r[k] = 0xff800000u;   // -inf
                            }
                        } else if (SCALED) {
#pragma unroll
                            for (int k = 0; k < LD; ++k) lowest = fminf(lowest, __uint_as_float(r[k]));
                        }
                        float m0 = -INFINITY, m1 = -INFINITY;
#pragma unroll
                        for (int k = 0; k < LD; k += 4) {
                            m0 = max3f(m0, __uint_as_float(r[k]), __uint_as_float(r[k + 1]));
                            m1 = max3f(m1, __uint_as_float(r[k + 2]), __uint_as_float(r[k + 3]));
                        }
                        m = max3f(m, m0, m1);
                    }
                } else if (!ONE) {
                    asm volatile("bar.arrive %0, %1;" ::"r"(bar_sc), "n"(NT) : "memory");
                }
            }
            if constexpr (DUO) m = fmaxf(m, swap(s_pair[0], m));
            if constexpr (DUO && SCALED) lowest = fminf(lowest, swap(s_pair[1], lowest));
            // RAGGED: the scores are scaled and rounded before the maximum is subtracted, and the segment number is clamped on
            // both sides, as on the CUDA cores.  Otherwise one FMA does both, and its result must not lie above 0, which is what
            // bounds the segment number there: the product is rounded up.  Rounded to nearest, fma(m, scale, -m scale) lies up
            // to half an ulp of m * scale above 0 for a scale that is no power of two, past the table's spare entry from 1e6 on.
            const float neg_ms = RAGGED ? -__fmul_rn(m, a.scale) : -__fmul_ru(m, a.scale);
            const uint64_t neg_ms2 = nm_pack2(neg_ms, neg_ms);
            float sum0 = 0.f, sum1 = 0.f, sum2 = 0.f, sum3 = 0.f;
            [[maybe_unused]] int groups = 0;   // DUO: groups of 8 keys that the second warp has put into s_sum
            // SCALED: the power of two that brings the largest |e| this row can have to 2^14 .. 2^15 (below the table the first
            // segment goes on), and its inverse; an fp16 term then loses nothing to the narrow exponent
            [[maybe_unused]] float up = 1.f, down = 1.f;
            if constexpr (SCALED) {
                const float x = __fadd_rn(__fmul_rn(lowest, a.scale), neg_ms);
                const float2 kb0 = rep[lane & 15];
                const float big = fmaxf(a.e_max, nm_pwl_index(x, inv_h, off, nm1) == 0 ? fabsf(__fmaf_rn(kb0.x, x, kb0.y)) : 0.f);
                const int ex = min(max(14 + 127 - (int)(__float_as_uint(big) >> 23), -100), 100);
                up = __uint_as_float((uint32_t)(127 + ex) << 23);
                down = __uint_as_float((uint32_t)(127 - ex) << 23);
            }
            // ---- sweep 2: e = PWL_exp(s - m), row sum, P tiles.
            // W scores of this thread's row -> exponentials, in groups of 8.  MASKED: keys from `lim` on lie beyond L; they take
            // the maximum as their score (which keeps the table index in range) and the exponential 0.
            constexpr int W = RAGGED || ONE ? 16 : 32;   // (with several terms of P, 32 keys at a time spill)
            auto exponentials = [&](uint32_t* r, int lim, auto masked, auto&& use) {
                constexpr bool MASKED = decltype(masked)::value;
                if constexpr (MASKED) {
#pragma unroll
                    for (int k = 0; k < W; ++k)
                        if (k >= lim) r[k] = __float_as_uint(m);
                }
#pragma unroll
                for (int jj = 0; jj < W / 8; ++jj) {   // 8 keys
                    float e[8];
#pragma unroll
                    for (int k = 0; k < 8; k += 2) {
                        // two scores at a time on the packed fp32 instructions: each half is the same correctly
                        // rounded operation as the scalar form
                        uint64_t x2, u2, b2;
                        const float s0 = __uint_as_float(r[jj * 8 + k]), s1 = __uint_as_float(r[jj * 8 + k + 1]);
                        if constexpr (RAGGED) {   // (the packed mul and add would be contracted into an FMA)
                            x2 = nm_pack2(__fadd_rn(__fmul_rn(s0, a.scale), neg_ms), __fadd_rn(__fmul_rn(s1, a.scale), neg_ms));
                        } else {
                            asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(x2) : "l"(nm_pack2(s0, s1)), "l"(scale2), "l"(neg_ms2));
                        }
                        asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(u2) : "l"(x2), "l"(inv_h2), "l"(off2));
                        float x0, x1, u0, u1;
                        nm_unpack2(x2, x0, x1);
                        nm_unpack2(u2, u0, u1);
                        u0 = fmaxf(u0, 0.0f);
                        u1 = fmaxf(u1, 0.0f);
                        if (CLAMP_HI) {
                            u0 = fminf(u0, nm1);
                            u1 = fminf(u1, nm1);
                        }
                        // floor(u) sits in the low mantissa bits after a round-down add of 1.5 * 2^23
                        asm("add.rm.f32x2 %0, %1, %2;" : "=l"(b2) : "l"(nm_pack2(u0, u1)), "l"(magic2));
                        float f0, f1;
                        nm_unpack2(b2, f0, f1);
                        float k0, c0, k1, c1;
                        asm("ld.shared.v2.f32 {%0, %1}, [%2];" : "=f"(k0), "=f"(c0) : "r"((__float_as_uint(f0) << 7) + rep_lane));
                        asm("ld.shared.v2.f32 {%0, %1}, [%2];" : "=f"(k1), "=f"(c1) : "r"((__float_as_uint(f1) << 7) + rep_lane));
                        e[k] = __fmaf_rn(k0, x0, c0);
                        e[k + 1] = __fmaf_rn(k1, x1, c1);
                        if constexpr (MASKED) {
                            if (jj * 8 + k >= lim) e[k] = 0.f;
                            if (jj * 8 + k + 1 >= lim) e[k + 1] = 0.f;
                        }
                    }
                    if (DUO && part == 1) {   // (to be added up behind the first warp's)
                        s_sum[groups++][row] = make_float4(e[0] + e[4], e[1] + e[5], e[2] + e[6], e[3] + e[7]);
                    } else {
                        sum0 += e[0] + e[4];
                        sum1 += e[1] + e[5];
                        sum2 += e[2] + e[6];
                        sum3 += e[3] + e[7];
                    }
                    use(jj, e);
                }
            };
            if constexpr (!RAGGED && ONE) {
#pragma unroll 1
                for (int k = first; k < last; ++k) {
                    uint32_t r[16], pk[8];
                    if (ok) {
                        nm_tmem_ld16_sync(t_row + (uint32_t)(16 * k), r);
                        exponentials(r, W, std::false_type{}, [&](int jj, const float* e) {
#pragma unroll
                            for (int i = 0; i < 4; ++i) pk[jj * 4 + i] = AT<T>::pack(e[2 * i], e[2 * i + 1]);
                        });
                        nm_tmem_st8(p_row + (uint32_t)(8 * k), pk);
                    }
                }
                nm_tmem_st_wait();
                nm_tc_fence_before();
                asm volatile("bar.arrive %0, %1;" ::"r"(bar_pr), "n"(NT) : "memory");
            } else if constexpr (!RAGGED) {
#pragma unroll 1
                for (int j = 0; j < n; ++j) {
                    wait_all(&bar_s_full, s_cnt & 1u);
                    ++s_cnt;
                    if (ok) nm_tc_fence_after();
#pragma unroll
                    for (int hh = 0; hh < 2; ++hh) {
                        uint32_t r[32];
                        if (ok) nm_tmem_ld32_sync(t_row + (uint32_t)(hh * 32), r);
                        if (hh == 1) {
                            nm_tc_fence_before();
                            asm volatile("bar.arrive %0, %1;" ::"r"(bar_sc), "n"(NT) : "memory");
                        }
                        uint32_t pk[16];   // the half's 32 exponentials, packed to 16 bits
                        if (ok)
                            exponentials(r, W, std::false_type{}, [&](int jj, const float* e) {
#pragma unroll
                                for (int k = 0; k < 4; ++k) pk[jj * 4 + k] = AT<T>::pack(e[2 * k], e[2 * k + 1]);
                            });
                        // The stores wait until P V of the previous chunk has read the tile; that MMA was
                        // issued just before this chunk began, so the first half's arithmetic runs ahead of it.
                        if (hh == 0 && j >= 1) wait_all(&bar_p_empty, (pv_base + (uint32_t)(j - 1)) & 1u);
                        if (ok) {
                            if (hh == 0 && j >= 1) nm_tc_fence_after();   // ordered after the P V that read the columns
                            nm_tmem_st16(p_row + (uint32_t)(hh * 16), pk);   // keys 32 hh .. 32 hh + 31 of this thread's row
                        }
                    }
                    nm_tmem_st_wait();          // the P columns are written
                    nm_tc_fence_before();
                    asm volatile("bar.arrive %0, %1;" ::"r"(bar_pr), "n"(NT) : "memory");
                }
            } else {
                // 16 keys' scores at tensor-memory column `src` -> the terms of their exponentials
                uint32_t term[3][8];
                auto block = [&](uint32_t src, int lim, auto masked, auto&& loaded) {
                    uint32_t r[16];
                    if (ok && live) nm_tmem_ld16_sync(src, r);
                    loaded();
                    if (ok && live)
                        exponentials(r, lim, masked, [&](int jj, const float* e) {
#pragma unroll
                            for (int k = 0; k < 4; ++k)
                                ProbTerms<T>::split(SCALED ? e[2 * k] * up : e[2 * k], SCALED ? e[2 * k + 1] * up : e[2 * k + 1],
                                                    term[0][jj * 4 + k], term[1][jj * 4 + k], term[2][jj * 4 + k]);
                        });
                };
                const uint32_t lanes = (uint32_t)(q * 32) << 16;
                if constexpr (ONE) {
                    auto keys16 = [&](int k, auto masked) {
                        block(t_row + (uint32_t)(16 * k), L - 16 * k, masked, [] {});
                        if (ok && live) {
                            nm_tmem_st8(t_row + (uint32_t)(16 * k), term[0]);
                            nm_tmem_st8(t_row + (uint32_t)(16 * k + 8), term[1]);
                            if constexpr (TERMS == 3) nm_tmem_st8(p_row + (uint32_t)(8 * k), term[2]);
                        }
                    };
#pragma unroll 1
                    for (int k = first; k < (last < blocks ? last : blocks - 1); ++k) keys16(k, std::false_type{});
                    if (first < last && last == blocks) keys16(blocks - 1, std::true_type{});
                    nm_tmem_st_wait();
                    nm_tc_fence_before();
                    asm volatile("bar.arrive %0, %1;" ::"r"(bar_pr), "n"(NT) : "memory");
                } else {
                    auto keys32 = [&](int u, auto masked) {
                        const bool chunk_ends = (u & 1) || u + 1 == n_pv;
                        if (!(u & 1)) {
                            wait_all(&bar_s_full, s_cnt & 1u);
                            ++s_cnt;
                            if (ok) nm_tc_fence_after();
                        }
#pragma unroll
                        for (int hh = 0; hh < 2; ++hh) {
                            block(t_row + (uint32_t)((u & 1) * 32 + hh * 16), L - u * 32 - hh * 16, masked, [&] {
                                if (hh == 1 && chunk_ends) {   // all of the chunk's scores are in registers
                                    nm_tc_fence_before();
                                    asm volatile("bar.arrive %0, %1;" ::"r"(bar_sc), "n"(NT) : "memory");
                                }
                            });
                            // the stores wait until the previous P V has read the columns; 16 keys' arithmetic runs ahead of it
                            if (hh == 0 && u >= 1) wait_all(&bar_p_empty, (pv_base + (uint32_t)(u - 1)) & 1u);
                            if (ok && live) {
                                if (hh == 0 && u >= 1) nm_tc_fence_after();
#pragma unroll
                                for (int t = 0; t < TERMS; ++t) nm_tmem_st8(tmem_t + lanes + (uint32_t)(16 * t + 8 * hh), term[t]);
                            }
                        }
                        nm_tmem_st_wait();
                        nm_tc_fence_before();
                        asm volatile("bar.arrive %0, %1;" ::"r"(bar_pr), "n"(NT) : "memory");
                    };
#pragma unroll 1
                    for (int u = 0; u < n_pv - 1; ++u) keys32(u, std::false_type{});
                    keys32(n_pv - 1, std::true_type{});
                }
            }
            float sum = (sum0 + sum1) + (sum2 + sum3);
            if constexpr (DUO) {
                // Added up in the order that one warp would take, so that the last bit does not depend on the split (an int8
                // network's codes do on that bit): the second warp goes on from the first one's four sums.
                float* const total = &s_pair[0][0][row];   // (the maxima have been read: both warps are at the barrier below)
                if (part == 0) s_sum[8][row] = make_float4(sum0, sum1, sum2, sum3);
                asm volatile("bar.sync %0, 64;" ::"r"(8 + q) : "memory");
                if (part == 1) {
                    float4 c = s_sum[8][row];
                    for (int i = 0; i < groups; ++i) {
                        const float4 v = s_sum[i][row];
                        c.x += v.x; c.y += v.y; c.z += v.z; c.w += v.w;
                    }
                    *total = sum = (c.x + c.y) + (c.z + c.w);
                }
                asm volatile("bar.sync %0, 64;" ::"r"(8 + q) : "memory");
                sum = *total;
            }
            // ---- r = PWL_recip(sigma), then O * r
            const int sr = ONE ? nm_pwl_index(sum, r_inv_h, r_off, r_nm1)
                               : nm_pwl_index(sum, a.t_rcp->inv_h, a.t_rcp->off, (float)(a.t_rcp->n - 1));
            const float2 kbr = a.t_rcp->kb[sr];
            const float rinv = __fmaf_rn(kbr.x, sum, kbr.y);
            wait_all(&bar_p_empty, (pv_base + (uint32_t)(n_pv - 1)) & 1u);   // the last P V has completed
            pv_base += (uint32_t)n_pv;
            if (ok) nm_tc_fence_after();
            const bool store_row = !RAGGED || qb * BQ + row < L;
            T* orow = reinterpret_cast<T*>(a.out) + ((size_t)b * L + (size_t)qb * BQ + row) * ((size_t)a.heads * HD) +
                      (size_t)g * HD;
            const uint32_t o_addr = t_row + O_OFF;
#pragma unroll
            for (int j2 = 0; j2 < (DUO ? HD / 32 : HD / 16); ++j2) {   // 16 channels at a time
                const int jj = DUO ? 2 * part + j2 : j2;
                uint32_t r0[16];
                if (ok && live) {
                    nm_tmem_ld16_sync(o_addr + (uint32_t)(jj * 16), r0);
                    if constexpr (RAGGED && !ONE) {
                        uint32_t r1[16];
                        nm_tmem_ld16_sync(tmem_lo + ((uint32_t)(q * 32) << 16) + (uint32_t)(jj * 16), r1);
#pragma unroll
                        for (int k = 0; k < 16; ++k) r0[k] = __float_as_uint(__uint_as_float(r0[k]) + __uint_as_float(r1[k]));
                    }
                }
                if (j2 == (DUO ? HD / 32 : HD / 16) - 1 && more) {
                    // all of O is in registers: the control warp may start the next tile's sweep 1 over [S | O]
                    nm_tc_fence_before();
                    asm volatile("bar.arrive %0, %1;" ::"r"(bar_oc), "n"(NT) : "memory");
                }
                if (ok && store_row) {
                    float v[16];
#pragma unroll
                    for (int k = 0; k < 16; ++k) v[k] = (SCALED ? __uint_as_float(r0[k]) * down : __uint_as_float(r0[k])) * rinv;
                    if (a.out_q) {
                        int8_t code[16];
#pragma unroll
                        for (int k = 0; k < 16; ++k) code[k] = nm_quant_i8(AT<T>::round(v[k]), a.q_inv_scale);
                        int8_t* qrow = a.out_q + ((size_t)b * L + (size_t)qb * BQ + row) * ((size_t)a.heads * HD) +
                                       (size_t)g * HD;
                        reinterpret_cast<uint4*>(qrow)[jj] = *reinterpret_cast<const uint4*>(code);
                    } else {
                        uint32_t w[8];
#pragma unroll
                        for (int k = 0; k < 8; ++k) w[k] = AT<T>::pack(v[2 * k], v[2 * k + 1]);
                        reinterpret_cast<uint4*>(orow)[2 * jj] = make_uint4(w[0], w[1], w[2], w[3]);
                        reinterpret_cast<uint4*>(orow)[2 * jj + 1] = make_uint4(w[4], w[5], w[6], w[7]);
                    }
                }
            }
        }
    }

    nm_tc_fence_before();
    __syncthreads();
    if (warp == 0) {
        __syncwarp();
        nm_tc_fence_after();
        nm_tmem_dealloc(tmem_base, TMEM_COLS);
        if constexpr (!ONE) nm_tmem_dealloc(tmem_p, P_COLS);
    }
}

typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                  const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

// [B][L][heads*64] view with token pitch stride_t and batch pitch stride_b (elements); box 64 x rows x 1.
nm_status make_map(nm_ctx* ctx, CUtensorMap* m, const void* ptr, nm_dtype dt, const nm_attn_desc* d, int rows)
{
    CUtensorMapDataType t = dt == NM_BF16 ? CU_TENSOR_MAP_DATA_TYPE_BFLOAT16 : CU_TENSOR_MAP_DATA_TYPE_FLOAT16;
    cuuint64_t gdim[3] = {(cuuint64_t)d->heads * HD, (cuuint64_t)d->L, (cuuint64_t)d->B};
    cuuint64_t gstr[2] = {(cuuint64_t)d->stride_t * 2, (cuuint64_t)d->stride_b * 2};
    cuuint32_t box[3] = {HD, (cuuint32_t)rows, 1};
    cuuint32_t estr[3] = {1, 1, 1};
    CUresult r = ((EncodeTiledFn)ctx->encode_tiled)(m, t, 3, const_cast<void*>(ptr), gdim, gstr, box, estr,
                                                    CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
                                                    CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                                                    CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    return r == CUDA_SUCCESS ? NM_OK : NM_ERR_CUDA;
}

template <typename T, bool CLAMP_HI, bool RAGGED, Form FORM, int PER_SM>
nm_status launch(nm_ctx* ctx, const nm_attn_desc* d, cudaStream_t st, int8_t* out_q, float q_inv_scale)
{
    SArgs a;
    a.B = d->B; a.L = d->L; a.heads = d->heads; a.scale = d->scale;
    a.t_exp = ctx->d_tables + d->exp_slot;
    a.t_rcp = ctx->d_tables + d->recip_slot;
    a.out = d->out;
    a.status = ctx->d_status;
    a.n_exp = ctx->h_tables[d->exp_slot].n;
    a.e_max = 0.f;
    if (RAGGED && d->dtype == NM_F16) {
        const NmTable& t = ctx->h_tables[d->exp_slot];
        const double h = ((double)t.x_max - t.x_min) / t.n;
        for (int i = 0; i < t.n; ++i) {   // each segment's ends as far as they are not above 0; the last one goes on to 0
            const double ends[2] = {t.x_min + i * h, i + 1 == t.n && t.x_max < 0.f ? 0.0 : t.x_min + (i + 1) * h};
            for (double x : ends) {
                if (i > 0 && ends[0] > 0.0) continue;
                if (x > 0.0) x = 0.0;
                const double e = fabs((double)t.kb[i].x * x + t.kb[i].y);
                if (e > a.e_max) a.e_max = (float)e;
            }
        }
    }
    a.out_q = out_q;
    a.q_inv_scale = q_inv_scale;
    const size_t smem = (size_t)BQ * ROWB + 3 * (size_t)STAGE + (size_t)PBUF + (size_t)(a.n_exp + 1) * 16 * sizeof(float2) + 1024;
    if (smem > 227 * 1024 - 2048) return NM_ERR_UNSUPPORTED;   // an exp table too large to replicate
    CUtensorMap tmQ, tmK, tmV;
    nm_status s;
    if ((s = make_map(ctx, &tmQ, d->Q, d->dtype, d, BQ)) != NM_OK) return s;
    if ((s = make_map(ctx, &tmK, d->K, d->dtype, d, CK)) != NM_OK) return s;
    if ((s = make_map(ctx, &tmV, d->V, d->dtype, d, CK)) != NM_OK) return s;
    auto kern = attention_stream_kernel<T, CLAMP_HI, RAGGED, FORM, PER_SM>;
    if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) != cudaSuccess)
        return NM_ERR_CUDA;
    const int64_t tiles = (int64_t)d->B * d->heads * ((d->L + BQ - 1) / BQ);
    if (tiles > 0x7fffffffLL) return NM_ERR_SHAPE;
    // persistent: one resident wave of CTAs, each walking over tiles; by the launch bounds (registers), by tensor memory
    // (3 x 160 or 2 x 256 of 512 columns) and, if the exp table makes the shared memory larger, by that (233472 bytes per SM,
    // 1 KB reserved per CTA).
    int64_t per_sm = 233472 / (int64_t)(smem + 1024 + (FORM == DUO_CHUNK ? 22 * 1024 : 1536));
    if (per_sm > PER_SM) per_sm = PER_SM;
    if (per_sm < 1) per_sm = 1;
    int64_t grid = (int64_t)ctx->sm_count * per_sm;
    if (grid > tiles) grid = tiles;
    cudaLaunchConfig_t cfg;
    memset(&cfg, 0, sizeof(cfg));
    cfg.gridDim = dim3((unsigned)grid);
    cfg.blockDim = dim3(CTA_THREADS<FORM>);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = ctx->pdl ? 1 : 0;
    NmLaunchScope scope(ctx, NM_KERNEL_ATTENTION_TC, 4.0 * (double)d->B * d->heads * (double)d->L * d->L * HD, st);
    if (cudaLaunchKernelEx(&cfg, kern, tmQ, tmK, tmV, a) != cudaSuccess) return NM_ERR_CUDA;
    return cudaGetLastError() == cudaSuccess ? NM_OK : NM_ERR_CUDA;
}

// The form for a (batch, head) of one chunk.  Two softmax warps halve the chain of one head, one warp gets more heads through an SM.  us, one
// warp, two with two CTAs per SM, two with one (bf16, 12 heads a sequence):
//   L 37    B 1 5.2, 5.3, 4.6   B 12 5.9, 6.1, 5.3   B 24 7.4, 7.2, 10.1   B 32 8.6, 9.8, 13.0   B 128 21.1, 24.5, 34.2
//   L 100   B 1 6.9, 7.7, 6.4   B 12 7.6, 8.2, 6.8   B 24 9.8, 11.0, 13.1  B 32 12.6, 14.7, 17.1 B 128 35.6, 43.4, 48.4
//   L 24    B 24 7.1, 6.2       L 64   B 16 7.4, 7.7   (two with two, up to 48 keys, as long as one round takes all heads)
//   L 128   B 1 5.3, 5.3        B 12 5.7, 5.5        B 24 8.1, 8.0         B 32 9.5, 9.7         B 128 27.0, 28.0   (unmasked: no spills with two)
template <typename T, bool CLAMP_HI, bool RAGGED>
nm_status launch_one(nm_ctx* ctx, const nm_attn_desc* d, cudaStream_t st, int8_t* out_q, float q_inv_scale)
{
    const int64_t heads = (int64_t)d->B * d->heads;
    if (RAGGED && heads <= ctx->sm_count) return launch<T, CLAMP_HI, RAGGED, DUO_CHUNK, RAGGED ? 1 : 2>(ctx, d, st, out_q, q_inv_scale);
    if (heads <= 2 * ctx->sm_count && (!RAGGED || d->L <= 48)) return launch<T, CLAMP_HI, RAGGED, DUO_CHUNK, 2>(ctx, d, st, out_q, q_inv_scale);
    return launch<T, CLAMP_HI, RAGGED, ONE_CHUNK, 2>(ctx, d, st, out_q, q_inv_scale);
}

}  // namespace

bool nm_attention_stream_supported(const nm_attn_desc* d)
{
    return d->L % 128 == 0 && nm_attention_stream_any_length_supported(d);
}

bool nm_attention_stream_any_length_supported(const nm_attn_desc* d)
{
    if (d->dtype != NM_BF16 && d->dtype != NM_F16) return false;
    if (d->d != HD || d->L < 1) return false;
    if ((d->stride_t * 2) % 16 != 0 || (d->stride_b * 2) % 16 != 0) return false;
    return true;
}

nm_status nm_launch_attention_stream(nm_ctx* ctx, const nm_attn_desc* d, cudaStream_t st, int8_t* out_q,
                                     float q_inv_scale)
{
    if (!nm_attention_stream_any_length_supported(d)) return NM_ERR_UNSUPPORTED;
    // the unmasked forms' softmax input is never above 0: a table whose range reaches 0 needs no upper clamp there
    const bool clamp_hi = ctx->h_tables[d->exp_slot].x_max < 0.0f;
    const bool ragged = d->L % 128 != 0, one = d->L <= 128;
#define NM_ATTN_FORM(T, CH, RG)                                                                                       \
    (one ? launch_one<T, CH, RG>(ctx, d, st, out_q, q_inv_scale) : launch<T, CH, RG, MANY, RG ? 2 : 3>(ctx, d, st, out_q, q_inv_scale))
#define NM_ATTN_CASE(T) (ragged ? NM_ATTN_FORM(T, true, true) : clamp_hi ? NM_ATTN_FORM(T, true, false) : NM_ATTN_FORM(T, false, false))
    if (d->dtype == NM_BF16) return NM_ATTN_CASE(__nv_bfloat16);
    return NM_ATTN_CASE(__half);
#undef NM_ATTN_CASE
#undef NM_ATTN_FORM
}

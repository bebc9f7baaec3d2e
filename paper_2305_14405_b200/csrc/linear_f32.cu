// fp32 linear operator with PWL epilogue on the tensor cores: every fp32 operand is the sum of three bf16 terms
// (f32_terms.cuh: the terms, their six products, and why an accumulator of the first product takes four steps only, one K-block;
// the sum warps add it to their fp32 registers while the other one fills).
//
// A CTA takes a 128 x BN tile (BN = 128 or 64): eight warps fetch the fp32 operands, split them and write the terms into a ring
// of K-major, 128-byte-swizzled operand tiles; one warp issues the products; eight warps add the accumulators up.  Problems of few tiles
// split K over a thread-block cluster, whose partial tiles are added through distributed shared memory.
// A result that is not finite (an infinite or NaN operand, one of 2^112 or more, sums beyond the fp32 range) is
// computed again as a chain of FMAs, so that infinities come out as they do there and not as the difference of two.
//
// Bound by the shared-memory port with 128 columns: per K-block of 64 k the terms' stores take 768 cycles, the products' operand reads
// 1536, the fp32 fetch 1390 beside them; 2700 were measured.  The fetch loop must not spill (beside 200 KB of shared memory the L1 is
// too small to hold a spilled register: 5000 cycles), hence the two chunks at a time, the one walking pointer and the tail apart.
// (By -Xptxas -v 8 bytes spill with 128 columns, none with 64; with a partial last K-block, a kernel of its own, 16 and 12.)
// Relative errors against float64 here and with packed FMAs on the CUDA cores, which this kernel replaced: 1024 x 768 x 768
// 9.0e-8 and 2.5e-7, x 3072 1.2e-7 and 2.5e-7, 128 x 768 x 256 8.1e-8 and 9.7e-8; operands of one sign 8.0e-8 and 1.1e-7, 9.1e-8
// and 6.7e-8, 8.0e-8 and 5.0e-8.  Times: 1024 x 2304 x 768 23.9 us and 84.5, 1024 x 768 x 3072 42.3 and 132.1, 40 x 768 x 3072 12.4
// and 24.0, 128 x 768 x 256 6.9 and 7.6, 200 x 768 x 16 6.4 and 5.9 (the set-up of tensor memory and barriers).
#include "f32_terms.cuh"
#include "linear_split_kernel.cuh"

using namespace nm_tc;

namespace {

constexpr int FBK = 64;           // K-elements of a stage: 128 bytes of bf16 per row and term
constexpr int F_PROD = 256;       // threads that fetch and split: warps 0 to 7; warp 8 issues the products
constexpr int F_SUM_WARPS = 8;    // warps 9 to 16
constexpr int F_THREADS = F_PROD + 32 + 32 * F_SUM_WARPS;
constexpr int FIN_THREADS = 512;  // of them run the final sum

template <int BN> struct F32Tile {
    static constexpr int B_BYTES = BN * ROW_BYTES;
    static constexpr int STAGE_BYTES = 3 * (A_BYTES + B_BYTES);
    static constexpr int STAGES = BN == 128 ? 2 : 3;
    static constexpr int SMEM = STAGES * STAGE_BYTES + 1024;
    static constexpr int CHUNKS = (BM + BN) / 16;      // 16-byte chunks of fp32 per thread and stage
    static constexpr int AHEAD = BN == 128 ? 8 : 12;   // of them in flight, in registers
    static constexpr int GROUP = BN == 128 ? 2 : 1;    // split together
    static_assert((BM * part_pitch(BN) + F_SUM_WARPS * 2 * 64 * (16 + 4)) * 4 <= STAGES * STAGE_BYTES,
                  "the partial tile and the slices of fma_chains take the ring's place");
};

// Sums that are not finite, among those of a warp's 32 rows and COLS columns at `sums`: chains of K FMAs instead.  16 rows and 32 columns
// at a time, those without such a sum passed over; 4 x 4 chains per lane, the operands 16 k at a time through the warp's own CHAIN_WORDS of
// shared memory, one buffer filling while the other is multiplied.  1024 x 768 x 3072, 48 us alone: one row of NaN or infinities 258 to 274 us,
// nothing but NaN 521 (each such sum by its row's thread, from memory: 2240 and 28400); 37 x 768 x 3072, 16 us: 45 and 72.  The finite
// product pays for the code with up to 1 % (8 x 4 chains, which need 40 more registers: with 3 %, and 360 and 369 us).
constexpr int CHAIN_K = 16, CHAIN_PITCH = CHAIN_K + 4, CHAIN_BUF = 64 * CHAIN_PITCH, CHAIN_WORDS = 2 * CHAIN_BUF;

template <int COLS>
__device__ __forceinline__ void fma_chains(const float* A, const float* W, int64_t lda, int64_t ldw, int K, int rows, int cols, float* sums, int pitch, float* slice)
{
    const int lane = threadIdx.x & 31, ry = lane >> 3, cx = lane & 7;   // rows ry + 4 i, columns cx + 8 j
    __syncwarp();
#pragma unroll 1
    for (int cr = 0; cr < COLS / 16; ++cr) {
        const int c = (cr >> 1) * 32, r_lo = (cr & 1) * 16;
        uint32_t odd = 0;   // bit 4 i + j
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const int r = r_lo + ry + 4 * i, n = c + cx + 8 * j;
                if (r < rows && n < cols && !(fabsf(sums[r * pitch + n]) <= 3.402823466e38f)) odd |= 1u << (4 * i + j);
            }
        if (!__any_sync(0xffffffffu, odd != 0)) continue;
        float v[4][4];
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int j = 0; j < 4; ++j) v[i][j] = 0.f;
        // row r of A at row r of a buffer, row c + r of W at 32 + r (for one that does not exist the first one again); zeros beyond K,
        // which leave a chain as it is
        auto fetch = [&](int k0) {
            const int k = k0 + (lane & 3) * 4, left = min(K - k, 4), bytes = left > 0 ? 4 * left : 0;
            const uint32_t dst = nm_smem_u32(slice + ((k0 / CHAIN_K) & 1) * CHAIN_BUF + (lane >> 2) * CHAIN_PITCH + (lane & 3) * 4);
#pragma unroll 1
            for (int i = 0; i < 8; ++i) {
                const int r = (8 * i + (lane >> 2)) & 31;
                const float* p = (i < 4 ? A + (r < rows ? r : 0) * lda : W + (c + r < cols ? c + r : c) * ldw) + (bytes ? k : 0);
                asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst + (uint32_t)(8 * i * CHAIN_PITCH * 4)), "l"(p), "r"(bytes) : "memory");
            }
            asm volatile("cp.async.commit_group;" ::: "memory");
        };
        __syncwarp();
        fetch(0);
#pragma unroll 1
        for (int k0 = 0; k0 < K; k0 += CHAIN_K) {
            if (k0 + CHAIN_K < K) {
                fetch(k0 + CHAIN_K);
                asm volatile("cp.async.wait_group 1;" ::: "memory");
            } else {
                asm volatile("cp.async.wait_group 0;" ::: "memory");
            }
            __syncwarp();
            const float* buf = slice + ((k0 / CHAIN_K) & 1) * CHAIN_BUF;
#pragma unroll 1
            for (int kk = 0; kk < CHAIN_K; kk += 4) {
                float4 w[4];
#pragma unroll
                for (int j = 0; j < 4; ++j) w[j] = *reinterpret_cast<const float4*>(buf + (32 + cx + 8 * j) * CHAIN_PITCH + kk);
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    const float4 x = *reinterpret_cast<const float4*>(buf + (r_lo + ry + 4 * i) * CHAIN_PITCH + kk);
#pragma unroll
                    for (int j = 0; j < 4; ++j)
                        v[i][j] = __fmaf_rn(x.w, w[j].w, __fmaf_rn(x.z, w[j].z, __fmaf_rn(x.y, w[j].y, __fmaf_rn(x.x, w[j].x, v[i][j]))));
                }
            }
            __syncwarp();   // the buffer may be filled again
        }
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int j = 0; j < 4; ++j)
                if (odd & (1u << (4 * i + j))) sums[(r_lo + ry + 4 * i) * pitch + c + cx + 8 * j] = v[i][j];
    }
}

// TAIL: K is no multiple of a K-block.  A kernel of its own, so that the fetch loop over whole K-blocks keeps its registers: with the last
// K-block's loads in flight together in the same kernel 1024 x 768 x 3072 took 45.9 us instead of 42.3.  us with the last K-block's loads
// one after another behind branches, so, and with packed FMAs: 128 x 256 x 200 9.8, 7.6, 8.6; 200 x 768 x 16 8.6, 6.4, 5.9;
// 16384 x 768 x 16 68.7, 52.3, 58.6.  Without a partial K-block 128 x 768 x 256 7.4 -> 6.9, 40 x 768 x 3072 12.8 -> 12.4.
template <int BN, bool TAIL>
__global__ void __launch_bounds__(F_THREADS, 1)
linear_f32_kernel(const float* __restrict__ A, const float* __restrict__ W, int64_t lda, int64_t ldw, const SplitArgs s)
{
    using T = F32Tile<BN>;
    const TcArgs& a = s.t;
    constexpr int PITCH = part_pitch(BN);
    constexpr uint32_t IDESC = nm_idesc(1, 1, 0, 0, BM, BN);
    constexpr uint32_t TMEM_COLS = 4 * BN;   // two accumulators of h h', one of the 2^-16 and one of the 2^-32 products

    extern __shared__ uint8_t smem_raw[];
    __shared__ uint64_t bar_full[T::STAGES], bar_empty[T::STAGES], bar_acc_full[2], bar_acc_empty[2], bar_end;
    __shared__ uint32_t tmem_slot;
    __shared__ int abort_flag;
    __shared__ float2 s_tab[NM_MAX_SEGMENTS];

    uint8_t* ring = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
    float* part = reinterpret_cast<float*>(ring);
    const int S = s.S;
    const int rank = S > 1 ? (int)nm_cluster_ctarank() : 0;
    const int tile = (int)blockIdx.x / S;
    const int mt = tile / a.num_n_tiles, nt = tile % a.num_n_tiles;
    const int kb0 = (int)((int64_t)rank * a.num_k_blocks / S), kb1 = (int)((int64_t)(rank + 1) * a.num_k_blocks / S);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int64_t m0 = (int64_t)mt * BM, n0 = (int64_t)nt * BN;
    const int rows = (int)min((int64_t)BM, a.M - m0), cols = (int)min((int64_t)BN, a.N - n0);

    if (tid == 0) {
        abort_flag = 0;
        for (int i = 0; i < T::STAGES; ++i) {
            nm_mbar_init(&bar_full[i], F_PROD / 32);
            nm_mbar_init(&bar_empty[i], 1);
        }
        for (int i = 0; i < 2; ++i) {
            nm_mbar_init(&bar_acc_full[i], 1);
            nm_mbar_init(&bar_acc_empty[i], F_SUM_WARPS);
        }
        nm_mbar_init(&bar_end, 1);
        nm_fence_barrier_init();
    }
    if (warp == F_PROD / 32) {
        nm_tmem_alloc(&tmem_slot, TMEM_COLS);
        nm_tmem_relinquish();
    }
    if (a.tab) {
        for (int i = tid; i < a.n_seg; i += F_THREADS) s_tab[i] = a.tab->kb[i];
    }
    nm_tc_fence_before();
    __syncthreads();
    nm_tc_fence_after();
    const uint32_t tmem = tmem_slot;
    volatile int* abortp = &abort_flag;
    if (!a.late_trigger) nm_grid_launch_dependents();
    // weights that were complete before the previous kernel started are fetched before the wait for it
    if (!a.weights_ready || warp >= F_PROD / 32) nm_grid_dependency_wait();
    if (a.late_trigger) nm_grid_launch_dependents();
    bool ok = true;

    if (warp < F_PROD / 32) {
        // ------------------------------------------------ operands
        // This thread's: chunk tid % 16 (four k) of rows tid / 16 + 16 i, first of W, then of A.  Rows that do not exist are
        // not read: what their registers hold goes into rows and columns of the product that are not stored.
        const int c4 = (tid & 15) * 4, r0 = tid >> 4;
        uint32_t exists = 0;   // bit i: row i of this thread does
#pragma unroll
        for (int i = 0; i < T::CHUNKS; ++i) {
            if (i < BN / 16 ? 16 * i + r0 < cols : 16 * i - BN + r0 < rows) exists |= 1u << i;
        }
        const int64_t stepA = 16 * lda, stepW = 16 * ldw;
        const float* pA = A + (m0 + r0) * lda + c4 + (int64_t)kb0 * FBK;   // row 0 in the K-block that is fetched next
        const float* pW = W + (n0 + r0) * ldw + c4 + (int64_t)kb0 * FBK;
        const int full = TAIL ? min(kb1, (int)(a.K / FBK)) : kb1;   // K-blocks that are all there end here
        // (one pointer walks along the rows: an address per row would be kept in registers)
        const float* pf = pW;
        uint32_t mask = kb0 < full ? exists : 0u;
        float4 reg[T::AHEAD];
        auto fetch = [&](int i) {
            if (i == 0) pf = pW;
            if (i == BN / 16) pf = pA;
            float4& v = reg[i % T::AHEAD];
            asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.u32 p, %5, 0;\n\t"
                         "@p ld.global.cg.v4.f32 {%0, %1, %2, %3}, [%4];\n\t}"
                         : "+f"(v.x), "+f"(v.y), "+f"(v.z), "+f"(v.w)
                         : "l"(pf), "r"(mask & (1u << i)));
            pf += i < BN / 16 ? stepW : stepA;
        };
        // row r of a term's tile at byte 128 r, its 16-byte chunk j at j ^ (r % 8); this thread's rows all have r % 8 = r0 % 8
        const uint32_t dst0 = nm_smem_u32(ring) + (uint32_t)(r0 * ROW_BYTES + (((c4 >> 3) ^ (r0 & 7)) << 4) + ((c4 & 4) << 1));
        auto put = [&](uint32_t d, uint32_t term, const uint2& h, const uint2& m, const uint2& l) {
            asm volatile("st.shared.v2.b32 [%0], {%1, %2};" ::"r"(d), "r"(h.x), "r"(h.y) : "memory");
            asm volatile("st.shared.v2.b32 [%0], {%1, %2};" ::"r"(d + term), "r"(m.x), "r"(m.y) : "memory");
            asm volatile("st.shared.v2.b32 [%0], {%1, %2};" ::"r"(d + 2 * term), "r"(l.x), "r"(l.y) : "memory");
        };
#pragma unroll
        for (int i = 0; i < T::AHEAD; ++i) {
            if (i == BN / 16 && a.weights_ready) nm_grid_dependency_wait();
            reg[i] = make_float4(0.f, 0.f, 0.f, 0.f);
            fetch(i);
        }
        if (T::AHEAD == BN / 16 && a.weights_ready) nm_grid_dependency_wait();
        // where a thread's row i goes in a stage: the terms of A lie before those of W
        auto place = [](int i) { return (uint32_t)(i < BN / 16 ? 3 * A_BYTES + i * 16 * ROW_BYTES : (i - BN / 16) * 16 * ROW_BYTES); };
        int stage = 0;
        uint32_t phase = 0;
        for (int kb = kb0; kb < kb1; ++kb) {
            if (!nm_mbar_wait(&bar_empty[stage], phase ^ 1u, abortp, a.status)) { ok = false; break; }
            const uint32_t dst = dst0 + (uint32_t)(stage * T::STAGE_BYTES);
            if (!TAIL || kb < full) {
#pragma unroll
                for (int i = 0; i < T::CHUNKS; i += T::GROUP) {
                    uint2 h[T::GROUP], m[T::GROUP], l[T::GROUP];
#pragma unroll
                    for (int j = 0; j < T::GROUP; ++j) nm_f32_terms4(reg[(i + j) % T::AHEAD], h[j], m[j], l[j]);
#pragma unroll
                    for (int j = 0; j < T::GROUP; ++j) {
                        const int n = (i + j + T::AHEAD) % T::CHUNKS;
                        if (n == 0) {
                            pA += FBK;
                            pW += FBK;
                            mask = kb + 1 < full ? exists : 0u;
                        }
                        fetch(n);
                    }
#pragma unroll
                    for (int j = 0; j < T::GROUP; ++j) put(dst + place(i + j), i < BN / 16 ? T::B_BYTES : A_BYTES, h[j], m[j], l[j]);
                }
            } else if constexpr (TAIL) {
                // K ends in this one: zeros beyond it, and the last one to three k of a row, whose end may be the memory's, singly.
                // Predicated loads, as many in flight as the registers hold: behind branches each waits for the one before.
                const int left = (int)a.K - (kb * FBK + c4);
                const uint32_t whole = left >= 4 ? exists : 0u, ends = left > 0 && left < 4 ? exists : 0u;
#pragma unroll
                for (int i = 0; i < T::CHUNKS; i += T::AHEAD) {
#pragma unroll
                    for (int j = 0; j < T::AHEAD; ++j) {
                        if (i + j == 0) pf = pW;   // (both have come to this K-block)
                        if (i + j == BN / 16) pf = pA;
                        float4& v = reg[j];
                        v = make_float4(0.f, 0.f, 0.f, 0.f);
                        asm volatile("{\n\t.reg .pred p, x, y, z;\n\tsetp.ne.u32 p, %5, 0;\n\tsetp.ne.u32 x, %6, 0;\n\tsetp.gt.and.s32 y, %7, 1, x;\n\tsetp.gt.and.s32 z, %7, 2, x;\n\t"
                                     "@p ld.global.cg.v4.f32 {%0, %1, %2, %3}, [%4];\n\t@x ld.global.cg.f32 %0, [%4];\n\t"
                                     "@y ld.global.cg.f32 %1, [%4 + 4];\n\t@z ld.global.cg.f32 %2, [%4 + 8];\n\t}"
                                     : "+f"(v.x), "+f"(v.y), "+f"(v.z), "+f"(v.w)
                                     : "l"(pf), "r"(whole & (1u << (i + j))), "r"(ends & (1u << (i + j))), "r"(left));
                        pf += i + j < BN / 16 ? stepW : stepA;
                    }
#pragma unroll
                    for (int j = 0; j < T::AHEAD; ++j) {
                        uint2 h, m, l;
                        nm_f32_terms4(reg[j], h, m, l);
                        put(dst + place(i + j), i + j < BN / 16 ? T::B_BYTES : A_BYTES, h, m, l);
                    }
                }
            }
            nm_fence_proxy_async();
            __syncwarp();
            if (lane == 0) nm_mbar_arrive(&bar_full[stage]);
            if (++stage == T::STAGES) { stage = 0; phase ^= 1u; }
        }
    } else if (warp == F_PROD / 32) {
        // ------------------------------------------------ products, those of an accumulator together
        int stage = 0;
        uint32_t phase = 0, acc_phase = 0;
        for (int kb = kb0; kb < kb1; ++kb) {
            if (!__all_sync(0xffffffffu, nm_mbar_wait(&bar_full[stage], phase, abortp, a.status))) { ok = false; break; }
            const uint32_t sa = nm_smem_u32(ring + (size_t)stage * T::STAGE_BYTES), sb = sa + 3 * A_BYTES;
            const uint64_t ah = nm_smem_desc_sw128(sa), bh = nm_smem_desc_sw128(sb);
            constexpr uint64_t AT = A_BYTES >> 4, BT = T::B_BYTES >> 4;   // from term to term
            const int buf = (kb - kb0) & 1;
            if (!__all_sync(0xffffffffu, nm_mbar_wait(&bar_acc_empty[buf], acc_phase ^ 1u, abortp, a.status))) { ok = false; break; }
            nm_tc_fence_after();
            if (nm_elect_one()) {
#pragma unroll
                for (int k = 0; k < 4; ++k) nm_mma_f16(tmem + (uint32_t)(buf * BN), ah + 2 * k, bh + 2 * k, IDESC, k != 0);   // 32 bytes of K per row
                nm_tc_commit(&bar_acc_full[buf]);
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    nm_mma_f16(tmem + 2 * BN, ah + 2 * k, bh + BT + 2 * k, IDESC, kb != kb0 || k != 0);
                    nm_mma_f16(tmem + 2 * BN, ah + AT + 2 * k, bh + 2 * k, IDESC, 1u);
                }
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    nm_mma_f16(tmem + 3 * BN, ah + AT + 2 * k, bh + BT + 2 * k, IDESC, kb != kb0 || k != 0);
                    nm_mma_f16(tmem + 3 * BN, ah + 2 * k, bh + 2 * BT + 2 * k, IDESC, 1u);
                    nm_mma_f16(tmem + 3 * BN, ah + 2 * AT + 2 * k, bh + 2 * k, IDESC, 1u);
                }
                nm_tc_commit(&bar_empty[stage]);
            }
            __syncwarp();
            if (++stage == T::STAGES) { stage = 0; phase ^= 1u; }
            acc_phase ^= (uint32_t)buf;
        }
        if (nm_elect_one()) nm_tc_commit(&bar_end);   // (after a timeout it still counts what was issued)
        __syncwarp();
    } else {
        // ------------------------------------------------ sums: 32 rows and half of the columns per warp
        const int c0 = ((warp - F_PROD / 32 - 1) >> 2) * (BN / 2), q = warp & 3, row = q * 32 + lane;
        const uint32_t t_addr = tmem + ((uint32_t)(q * 32) << 16) + (uint32_t)c0;
        uint64_t acc[BN / 4];   // pairs of columns
#pragma unroll
        for (int i = 0; i < BN / 4; ++i) acc[i] = 0ull;
        uint32_t phase = 0;
        for (int kb = kb0; kb < kb1; ++kb) {
            const int buf = (kb - kb0) & 1;
            if (!__all_sync(0xffffffffu, nm_mbar_wait(&bar_acc_full[buf], phase, abortp, a.status))) { ok = false; break; }
            nm_tc_fence_after();
#pragma unroll
            for (int c = 0; c < BN / 2; c += 16) {
                uint32_t r[16];
                nm_tmem_ld16_sync(t_addr + (uint32_t)(buf * BN + c), r);
#pragma unroll
                for (int i = 0; i < 16; i += 2)
                    asm("add.rn.f32x2 %0, %0, %1;" : "+l"(acc[(c + i) / 2]) : "l"(nm_pack2(__uint_as_float(r[i]), __uint_as_float(r[i + 1]))));
            }
            nm_tc_fence_before();
            __syncwarp();
            if (lane == 0) nm_mbar_arrive(&bar_acc_empty[buf]);
            phase ^= (uint32_t)buf;
        }
        // every product is done, and has read the ring, whose place the partial tile takes
        if (!nm_mbar_wait(&bar_end, 0, abortp, a.status)) ok = false;
        __syncwarp();
        nm_tc_fence_after();
        bool odd = false;   // a sum that is not finite
        float* mine = part + row * PITCH + c0;
        if (__all_sync(0xffffffffu, ok && !*abortp)) {
#pragma unroll
            for (int c = 0; c < BN / 2; c += 4) {
                float v[4];
                nm_unpack2(acc[c / 2], v[0], v[1]);
                nm_unpack2(acc[c / 2 + 1], v[2], v[3]);
                *reinterpret_cast<float4*>(mine + c) = make_float4(v[0], v[1], v[2], v[3]);
            }
#pragma unroll 1
            for (int c = 0; c < BN / 2; c += 16) {
                uint32_t mid[16], low[16];
                nm_tmem_ld16_sync(t_addr + (uint32_t)(2 * BN + c), mid);
                nm_tmem_ld16_sync(t_addr + (uint32_t)(3 * BN + c), low);
#pragma unroll
                for (int i = 0; i < 16; i += 4) {
                    float4* p = reinterpret_cast<float4*>(mine + c + i);
                    float4 v = *p;
                    auto add = [&](float& x, int j) {
                        x = nm_f32_sum(x, mid[j], low[j]);
                        odd |= !(fabsf(x) <= 3.402823466e38f);
                    };
                    add(v.x, i);
                    add(v.y, i + 1);
                    add(v.z, i + 2);
                    add(v.w, i + 3);
                    *p = v;
                }
            }
            if (__builtin_expect(__any_sync(0xffffffffu, odd && row < rows), 0)) {
                const int64_t k0 = (int64_t)kb0 * FBK;
                float* slice = part + BM * PITCH + (warp - F_PROD / 32 - 1) * CHAIN_WORDS;
                fma_chains<BN / 2>(A + (m0 + q * 32) * lda + k0, W + (n0 + c0) * ldw + k0, lda, ldw, (int)(min((int64_t)kb1 * FBK, a.K) - k0),
                                   rows - q * 32, cols - c0, part + q * 32 * PITCH + c0, PITCH, slice);
            }
        }
        nm_tc_fence_before();
    }
    Finisher<false, float, BN, false, FIN_THREADS, false> fin(s, rank, mt, nt, rows, Patch{0, 0, 0});
    fin.prefetch_vectors();
    fin.load_res(0);
    if (S > 1) nm_cluster_sync();
    else __syncthreads();
    if (tid < FIN_THREADS && !*abortp) fin.run(reinterpret_cast<const uint32_t*>(part), s_tab);
    if (S > 1) nm_cluster_sync();   // a peer may still be reading this CTA's partial tile
    if (warp == F_PROD / 32) {
        nm_tc_fence_after();
        nm_tmem_dealloc(tmem, TMEM_COLS);
    }
}

struct F32Choice {
    int BN, S;
};

// Columns per tile and CTAs per cluster: the least time by a model of 18 problems of 16 to 1024 rows, N 256 to 3072, K 256 to 3072, each
// with nine forms (6 % off on the average; the form it picks is 0.7 % behind the best, 3 % at most), in us: the launch, the first
// operands and the epilogue, the K-blocks of 64, more when all SMs fetch, the exchange of a split, and what a further round of CTAs costs
// beside its K-blocks.  A round is what the GPU holds of clusters of S, which is less than its SMs for most S (1024 x 768 x 768
// with 128 columns: 22.6, 16.6 and, in two rounds, 30.2 us for S = 1, 2, 3).
F32Choice choose_f32(int64_t M, int64_t N, int k_blocks, const int* resident)
{
    struct P { int BN; double base, kb, busy, split, per_cta, round; };
    static const P forms[2] = {{128, 5.56, 1.34, 0.22, 0.1, 0.46, 8.0}, {64, 3.93, 1.12, 0.0, 1.19, 0.14, 7.1}};
    F32Choice best = {64, 1};
    double best_t = 1e30;
    for (const P& p : forms) {
        const int64_t tiles = ((M + BM - 1) / BM) * ((N + p.BN - 1) / p.BN);
        for (int S = 1; S <= 8 && S <= k_blocks; ++S) {
            if (resident[S] < 1) continue;
            const double rounds = (double)((tiles + resident[S] - 1) / resident[S]);
            const double share = tiles < resident[S] ? (double)tiles / resident[S] : 1.0;
            const double t = p.base + rounds * (p.kb + p.busy * share) * ((k_blocks + S - 1) / S) + (S > 1 ? p.split + p.per_cta * S : 0.0) + p.round * (rounds - 1.0);
            if (t < best_t * 0.98) { best_t = t; best = {p.BN, S}; }
        }
    }
    return best;
}

template <int BN>
nm_status launch_f32(nm_ctx* ctx, const nm_linear_desc* d, SplitArgs& s, cudaLaunchConfig_t& cfg, cudaLaunchAttribute* attr, cudaStream_t st)
{
    auto kern = d->K % FBK == 0 ? linear_f32_kernel<BN, false> : linear_f32_kernel<BN, true>;
    const int64_t n_tiles = (d->N + BN - 1) / BN, tiles = (d->M + BM - 1) / BM * n_tiles;
    s.t.num_n_tiles = (int)n_tiles;
    s.t.num_tiles = (int)tiles;
    if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, F32Tile<BN>::SMEM) != cudaSuccess)
        return NM_ERR_CUDA;
    cfg.dynamicSmemBytes = F32Tile<BN>::SMEM;
    cfg.numAttrs = split_launch_attrs(ctx, attr, s.S);
    cfg.gridDim = dim3((unsigned)(tiles * s.S));
    NmLaunchScope scope(ctx, NM_KERNEL_LINEAR_TC, 2.0 * (double)d->M * (double)d->N * (double)d->K, st);
    if (cudaLaunchKernelEx(&cfg, kern, (const float*)d->A, (const float*)d->W, d->lda, d->ldw, s) != cudaSuccess)
        return NM_ERR_CUDA;
    return cudaGetLastError() == cudaSuccess ? NM_OK : NM_ERR_CUDA;
}

}  // namespace

bool nm_linear_f32_supported(const nm_linear_desc* d)
{
    return d->in_dtype == NM_F32 && d->N % 4 == 0 && d->K <= 0x7fffffffLL;
}

nm_status nm_launch_linear_f32(nm_ctx* ctx, const nm_linear_desc* d, cudaStream_t st, NmChain chain)
{
    if ((d->M + 63) / 64 > 65535 || (d->M + BM - 1) / BM * ((d->N + 63) / 64) > 0x7fffffffLL / 8) return NM_ERR_SHAPE;
    SplitArgs s;
    memset(&s, 0, sizeof(s));
    TcArgs& a = s.t;
    a.M = d->M; a.N = d->N; a.K = d->K;
    a.bias = d->bias;
    a.res_first = d->res_first;
    a.tab = d->slot == NM_SLOT_NONE ? nullptr : ctx->d_tables + d->slot;
    a.n_seg = d->slot == NM_SLOT_NONE ? 0 : ctx->h_tables[d->slot].n;
    a.idx_dump = d->idx_dump;
    a.status = ctx->d_status;
    a.weights_ready = chain.weights_ready;
    a.late_trigger = chain.late_trigger;
    a.num_k_blocks = (int)((d->K + FBK - 1) / FBK);
    s.residual = d->residual; s.ldr = d->ldr;
    s.out = d->out; s.ldo = d->ldo;
    cudaLaunchConfig_t cfg;
    memset(&cfg, 0, sizeof(cfg));
    cfg.blockDim = dim3(F_THREADS);
    cfg.stream = st;
    cudaLaunchAttribute attr[2];
    cfg.attrs = attr;
    // clusters of 1..8 CTAs the device holds (one CTA of either width per SM), asked for once per context (or by several threads,
    // which find the same; the first word is set when the others are, and orders them for a thread that did not ask)
    int* resident = ctx->f32_resident;
    if (__atomic_load_n(&resident[0], __ATOMIC_ACQUIRE) == 0) {
        cfg.dynamicSmemBytes = F32Tile<64>::SMEM;
        if (cudaFuncSetAttribute(linear_f32_kernel<64, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, F32Tile<64>::SMEM) != cudaSuccess)
            return NM_ERR_CUDA;
        for (int S = 1; S <= 8; ++S) {
            int n = 0;
            cfg.numAttrs = split_launch_attrs(ctx, attr, S);
            cfg.gridDim = dim3((unsigned)(S * ctx->sm_count));
            if (cudaOccupancyMaxActiveClusters(&n, linear_f32_kernel<64, false>, &cfg) != cudaSuccess) {
                (void)cudaGetLastError();
                n = S == 1 ? ctx->sm_count : 0;
            }
            __atomic_store_n(&resident[S], n, __ATOMIC_RELAXED);
        }
        __atomic_store_n(&resident[0], 1, __ATOMIC_RELEASE);
    }
    const F32Choice c = choose_f32(d->M, d->N, a.num_k_blocks, resident);
    s.S = c.S;
    return c.BN == 128 ? launch_f32<128>(ctx, d, s, cfg, attr, st) : launch_f32<64>(ctx, d, s, cfg, attr, st);
}

// fp32 attention with PWL softmax on the CUDA cores, heads of 64 channels.
//     s_j = scale*<q,k_j>; m = max s; e_j = PWLexp(s_j - m); sigma = sum e; r = PWLrecip(sigma); o = r * sum_j e_j v_j
// A CTA takes 32 queries of one (batch, head): the scores against all L keys stay in shared memory as fp32, so the
// final row maximum is known before the first exponential and nothing is computed twice.  K and then V pass through
// a two-stage cp.async ring in blocks of 64 keys; each of the 128 threads holds 4 x 4 scores, later 4 x 4 outputs, in
// registers, so an element read from shared memory serves four multiplications (the one-warp-per-row kernel in
// simt_kernels.cu reads K and V from the cache for every multiplication, and is left to other head sizes and to
// sequences whose scores do not fit).  Bound by shared-memory reads, 8 per 64 multiplications of a thread.
// B 8, L 128, 12 heads: 402 us with one warp per row, 18.4 us so.  Up to 128 keys go to the tensor-core kernel below.
#include <string.h>

#include "f32_terms.cuh"

namespace {

constexpr int QB = 32;      // queries per CTA
constexpr int KB = 64;      // keys per block
constexpr int HD = 64;
constexpr int TP = HD + 4;  // words per row of Q, K, V in shared memory
constexpr int THREADS = 128;

struct F32AttnArgs {
    const float *Q, *K, *V;
    float* out;
    int B, L, heads, q_blocks, LP;   // LP: words per score row
    int64_t stride_b, stride_t;
    float scale;
    const NmTable *t_exp, *t_rcp;
    int* status;
};

__device__ __forceinline__ void cp_async16z(uint32_t dst, const void* src, bool valid)
{
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(valid ? 16 : 0) : "memory");
}
#define NM_CP_COMMIT() asm volatile("cp.async.commit_group;" ::: "memory")
#define NM_CP_WAIT(n) asm volatile("cp.async.wait_group %0;" ::"n"(n) : "memory")

__global__ void __launch_bounds__(THREADS) attention_f32_kernel(const F32AttnArgs a)
{
    extern __shared__ __align__(16) float sm[];
    float2* s_tab = reinterpret_cast<float2*>(sm);          // NM_MAX_SEGMENTS
    float* s_q = sm + 2 * NM_MAX_SEGMENTS;                  // QB x TP
    float* s_kv = s_q + QB * TP;                            // 2 x KB x TP
    float* s_s = s_kv + 2 * KB * TP;                        // QB x LP
    __shared__ float s_r[QB];
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int qb = (int)blockIdx.x % a.q_blocks, g = (int)blockIdx.x / a.q_blocks % a.heads, b = (int)blockIdx.x / (a.q_blocks * a.heads);
    const int L = a.L, LP = a.LP, q0 = qb * QB, nb = (L + KB - 1) / KB;
    const int n_exp = a.t_exp->n;
    for (int i = tid; i < n_exp; i += THREADS) s_tab[i] = a.t_exp->kb[i];
    const float inv_h = a.t_exp->inv_h, off = a.t_exp->off, nm1 = (float)(n_exp - 1);
    nm_grid_launch_dependents();
    nm_grid_dependency_wait();

    const float* Qp = a.Q + b * a.stride_b + (int64_t)g * HD;
    const float* Kp = a.K + b * a.stride_b + (int64_t)g * HD;
    const float* Vp = a.V + b * a.stride_b + (int64_t)g * HD;
    const int lr = tid >> 4, lc = (tid & 15) * 4;   // loads: 16 chunks per row, 8 rows per pass
    const uint32_t kv_u = nm_smem_u32(s_kv);
    auto load_block = [&](const float* base, int blk, int st) {
#pragma unroll
        for (int i = 0; i < KB / 8; ++i) {
            const int r = lr + 8 * i, key = blk * KB + r;
            const bool v = key < L;
            cp_async16z(kv_u + (uint32_t)((st * KB + r) * TP + lc) * 4u, base + (int64_t)(v ? key : 0) * a.stride_t + lc, v);
        }
    };
#pragma unroll
    for (int i = 0; i < QB / 8; ++i) {
        const int r = lr + 8 * i;
        const bool v = q0 + r < L;
        cp_async16z(nm_smem_u32(s_q + r * TP + lc), Qp + (int64_t)(v ? q0 + r : 0) * a.stride_t + lc, v);
    }
    load_block(Kp, 0, 0);
    NM_CP_COMMIT();

    const int ty = tid >> 4, tx = tid & 15;   // rows ty + 8 i; keys tx + 16 j, or channels 4 tx ..
    // ---- scores; block nb of the ring's walk is V's block 0
    for (int blk = 0; blk < nb; ++blk) {
        if (blk + 1 < nb) load_block(Kp, blk + 1, (blk + 1) & 1);
        else load_block(Vp, 0, (blk + 1) & 1);
        NM_CP_COMMIT();
        NM_CP_WAIT(1);
        __syncthreads();
        const float* kt = s_kv + (blk & 1) * KB * TP;
        uint64_t acc[4][4];
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int j = 0; j < 4; ++j) acc[i][j] = 0ull;
#pragma unroll 4
        for (int c = 0; c < HD; c += 4) {
            ulonglong2 rq[4];
#pragma unroll
            for (int i = 0; i < 4; ++i) rq[i] = *reinterpret_cast<const ulonglong2*>(s_q + (ty + 8 * i) * TP + c);
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const ulonglong2 rk = *reinterpret_cast<const ulonglong2*>(kt + (tx + 16 * j) * TP + c);
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(acc[i][j]) : "l"(rq[i].x), "l"(rk.x));
                    asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(acc[i][j]) : "l"(rq[i].y), "l"(rk.y));
                }
            }
        }
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                float lo, hi;
                nm_unpack2(acc[i][j], lo, hi);
                s_s[(ty + 8 * i) * LP + blk * KB + tx + 16 * j] = (lo + hi) * a.scale;
            }
        __syncthreads();   // the stage may be loaded again
    }
    // ---- softmax: a warp takes 8 rows, four at a time; the scores become exponentials, 0 beyond L
    for (int rr = 0; rr < 8; rr += 4) {
        float* row[4];
        float m[4], sum[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            row[i] = s_s + (warp * 8 + rr + i) * LP;
            m[i] = -INFINITY;
            sum[i] = 0.f;
        }
        for (int j = lane; j < L; j += 32) {
#pragma unroll
            for (int i = 0; i < 4; ++i) m[i] = fmaxf(m[i], row[i][j]);
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1)
#pragma unroll
            for (int i = 0; i < 4; ++i) m[i] = fmaxf(m[i], __shfl_xor_sync(0xffffffffu, m[i], o));
        for (int j = lane; j < nb * KB; j += 32) {
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const float x = row[i][j] - m[i];
                const float2 kb = s_tab[nm_pwl_index(x, inv_h, off, nm1)];
                const float e = j < L ? __fmaf_rn(kb.x, x, kb.y) : 0.f;
                row[i][j] = e;
                sum[i] += e;
            }
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1)
#pragma unroll
            for (int i = 0; i < 4; ++i) sum[i] += __shfl_xor_sync(0xffffffffu, sum[i], o);
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const float2 kbr = a.t_rcp->kb[nm_pwl_index(sum[i], a.t_rcp->inv_h, a.t_rcp->off, (float)(a.t_rcp->n - 1))];
            if (lane == 0) s_r[warp * 8 + rr + i] = __fmaf_rn(kbr.x, sum[i], kbr.y);
        }
    }
    // ---- O = P V
    float o[4][4];
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int c = 0; c < 4; ++c) o[i][c] = 0.f;
    for (int blk = 0; blk < nb; ++blk) {
        const int st = (nb + blk) & 1;
        if (blk + 1 < nb) load_block(Vp, blk + 1, st ^ 1);
        NM_CP_COMMIT();
        NM_CP_WAIT(1);
        __syncthreads();   // the block has landed (and, the first time, every row of exponentials is written)
        const float* vt = s_kv + st * KB * TP;
#pragma unroll 4
        for (int k = 0; k < KB; k += 4) {
            float4 p[4];
#pragma unroll
            for (int i = 0; i < 4; ++i) p[i] = *reinterpret_cast<const float4*>(s_s + (ty + 8 * i) * LP + blk * KB + k);
#pragma unroll
            for (int kk = 0; kk < 4; ++kk) {
                const float4 v = *reinterpret_cast<const float4*>(vt + (k + kk) * TP + 4 * tx);
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    const float pi = kk == 0 ? p[i].x : kk == 1 ? p[i].y : kk == 2 ? p[i].z : p[i].w;
                    o[i][0] = __fmaf_rn(pi, v.x, o[i][0]);
                    o[i][1] = __fmaf_rn(pi, v.y, o[i][1]);
                    o[i][2] = __fmaf_rn(pi, v.z, o[i][2]);
                    o[i][3] = __fmaf_rn(pi, v.w, o[i][3]);
                }
            }
        }
        __syncthreads();
    }
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const int r = ty + 8 * i;
        if (q0 + r < L) {
            const float rinv = s_r[r];
            *reinterpret_cast<float4*>(a.out + ((int64_t)b * L + q0 + r) * ((int64_t)a.heads * HD) + g * HD + 4 * tx) =
                make_float4(o[i][0] * rinv, o[i][1] * rinv, o[i][2] * rinv, o[i][3] * rinv);
        }
    }
}

// ---- up to 128 keys: both products on the tensor cores, every operand three bf16 terms (f32_terms.cuh) ----
//
// One CTA per (batch, head): all of Q, K and V are fetched once and split, S = Q K^T lies in tensor memory, four threads
// share a row's softmax, the terms of the exponentials take the place of the scores and are the A operand of P V from there.  Bound
// by latency, one chain of load, split, product, softmax, product.  Operands of 2^48 and more, infinities and NaN take
// the products of this CTA to the CUDA cores (a sum of terms would make a NaN of an infinity).
// Times, and relative errors against float64, of this kernel and of the one above it: B 8, L 128, 12 heads 12.5 us, 8.9e-8 and
// 18.4 us, 2.2e-7; B 8, L 37 7.9 and 11.2; B 1, L 16, 4 heads 5.0 and 6.3.  Longer sequences keep the kernel above: their scores fit
// neither tensor memory nor, as terms, shared memory.
constexpr int TC_THREADS = 512;
constexpr int PARTS = TC_THREADS / 128;      // threads that share a row
constexpr int PART_KEYS = 128 / PARTS;
constexpr int LOAD_ROWS = TC_THREADS / 16;   // rows that are fetched at a time
constexpr int LOADS = 128 / LOAD_ROWS;
constexpr int TILE = 128 * 128;   // bytes of one term: 128 rows of 64 bf16
constexpr int E_PITCH = 128 + 4, F_PITCH = HD + 4;   // words per row of scores, and of operands, for the CUDA cores' products
static_assert((128 * E_PITCH + 2 * 128 * F_PITCH) * 4 <= 9 * TILE, "they take the place of the terms");
constexpr float TC_LIMIT = 0x1p48f;   // (a low term is up to 2^15 of its operand: 64 products stay finite)
// room for the largest table: the segments are counted on the device, where a captured launch finds the table of its replay
constexpr int TC_SMEM = 9 * TILE + 1024 + NM_MAX_SEGMENTS * 16 * (int)sizeof(float2);

// The products of a CTA as chains of FMAs, for operands that the terms do not take: the operands in shared memory behind the scores.
// B 8, L 128, 12 heads with a NaN in every head: 58 us, 627 with each operand from memory.  Functions of their own: a launch runs the kernel's
// code once or twice, from a cold instruction cache, and these should not lie in its way (inlined, finite B 8, L 37 8.0 -> 8.2 us).
__device__ __forceinline__ void stage(const float* p, int64_t stride, int L, float* dst)
{
    const int c4 = ((int)threadIdx.x & 15) * 4;
#pragma unroll 1
    for (int r = (int)threadIdx.x >> 4; r < 128; r += LOAD_ROWS)
        *reinterpret_cast<float4*>(dst + r * F_PITCH + c4) = r < L ? __ldcg(reinterpret_cast<const float4*>(p + r * stride + c4)) : make_float4(0.f, 0.f, 0.f, 0.f);
}

__device__ __noinline__ void scores_by_fma(const float* Q, const float* K, int64_t stride, int L, float* s_e)
{
    const int row = (int)threadIdx.x & 127, key0 = ((int)threadIdx.x >> 7) * PART_KEYS, lim = min(L - key0, PART_KEYS);
    float *s_q = s_e + 128 * E_PITCH, *s_k = s_q + 128 * F_PITCH;
    stage(Q, stride, L, s_q);
    stage(K, stride, L, s_k);
    __syncthreads();
#pragma unroll 1
    for (int j = 0; j < lim; j += 8) {
        float s[8];
#pragma unroll
        for (int i = 0; i < 8; ++i) s[i] = 0.f;
#pragma unroll 1
        for (int c = 0; c < HD; c += 4) {
            const float4 x = *reinterpret_cast<const float4*>(s_q + row * F_PITCH + c);
#pragma unroll
            for (int i = 0; i < 8; ++i) {
                const float4 y = *reinterpret_cast<const float4*>(s_k + (key0 + j + i) * F_PITCH + c);
                s[i] = __fmaf_rn(x.w, y.w, __fmaf_rn(x.z, y.z, __fmaf_rn(x.y, y.y, __fmaf_rn(x.x, y.x, s[i]))));
            }
        }
#pragma unroll
        for (int i = 0; i < 8; i += 4) *reinterpret_cast<float4*>(s_e + row * E_PITCH + key0 + j + i) = make_float4(s[i], s[i + 1], s[i + 2], s[i + 3]);
    }
}

// 16 channels of a row: its exponentials, at s_e, times V, times rinv
__device__ __noinline__ void output_by_fma(const float* V, int64_t stride, int L, float* s_e, float rinv, float* out)
{
    const int row = (int)threadIdx.x & 127, c0 = ((int)threadIdx.x >> 7) * 16;
    float* s_v = s_e + 128 * E_PITCH;
    stage(V, stride, L, s_v);
    __syncthreads();
    if (row >= L) return;
    float x[16];
#pragma unroll
    for (int c = 0; c < 16; ++c) x[c] = 0.f;
#pragma unroll 1
    for (int j = 0; j < L; ++j) {
        const float e = s_e[row * E_PITCH + j];
#pragma unroll
        for (int c = 0; c < 16; c += 4) {
            const float4 y = *reinterpret_cast<const float4*>(s_v + j * F_PITCH + c0 + c);
            x[c] = __fmaf_rn(e, y.x, x[c]);
            x[c + 1] = __fmaf_rn(e, y.y, x[c + 1]);
            x[c + 2] = __fmaf_rn(e, y.z, x[c + 2]);
            x[c + 3] = __fmaf_rn(e, y.w, x[c + 3]);
        }
    }
#pragma unroll
    for (int c = 0; c < 16; c += 4) *reinterpret_cast<float4*>(out + c) = make_float4(x[c] * rinv, x[c + 1] * rinv, x[c + 2] * rinv, x[c + 3] * rinv);
}

__global__ void __launch_bounds__(TC_THREADS, 1) attention_f32_tc_kernel(const F32AttnArgs a)
{
    extern __shared__ uint8_t smem_raw[];
    __shared__ uint64_t bar_s, bar_o;
    __shared__ uint32_t tmem_slot;
    __shared__ int abort_flag;
    __shared__ float s_red[PARTS][128];
    uint8_t* tiles = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
    float* s_e = reinterpret_cast<float*>(tiles);   // 128 x E_PITCH in the terms' place, for the CUDA cores' products; their operands behind it
    float2* rep = reinterpret_cast<float2*>(tiles + 9 * TILE);   // the exp table, 16-way replicated
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int g = (int)blockIdx.x % a.heads, b = (int)blockIdx.x / a.heads;
    const int L = a.L, steps = (L + 15) / 16;   // of 16 keys
    const int n_exp = a.t_exp->n;

    if (tid == 0) {
        abort_flag = 0;
        nm_mbar_init(&bar_s, 1);
        nm_mbar_init(&bar_o, 1);
        nm_fence_barrier_init();
    }
    if (warp == 0) {
        nm_tmem_alloc(&tmem_slot, 512);
        nm_tmem_relinquish();
    }
    for (int i = tid; i < n_exp * 16; i += TC_THREADS) rep[i] = a.t_exp->kb[i >> 4];
    const float inv_h = a.t_exp->inv_h, off = a.t_exp->off, nm1 = (float)(n_exp - 1);
    const float r_inv_h = a.t_rcp->inv_h, r_off = a.t_rcp->off, r_nm1 = (float)(a.t_rcp->n - 1);
    // The successor may start only when this CTA has its tensor memory: a successor that took columns first and then waited for this grid
    // would wait for good.
    __syncthreads();
    nm_grid_launch_dependents();
    nm_grid_dependency_wait();

    // ---- operands: chunk tid % 16 (four channels) of rows tid / 16 + 32 i, zeros beyond L
    const float* Qp = a.Q + b * a.stride_b + (int64_t)g * HD;
    const float* Kp = a.K + b * a.stride_b + (int64_t)g * HD;
    const float* Vp = a.V + b * a.stride_b + (int64_t)g * HD;
    const int c4 = (tid & 15) * 4, r0 = tid >> 4;
    const uint32_t dst0 = nm_smem_u32(tiles) + (uint32_t)(r0 * 128 + (((c4 >> 3) ^ (r0 & 7)) << 4) + ((c4 & 4) << 1));
    float4 q[LOADS], k[LOADS], v[LOADS];
    auto fetch = [&](const float* p, float4* x) {
#pragma unroll
        for (int i = 0; i < LOADS; ++i)
            x[i] = r0 + LOAD_ROWS * i < L ? __ldcg(reinterpret_cast<const float4*>(p + (int64_t)(r0 + LOAD_ROWS * i) * a.stride_t + c4)) : make_float4(0.f, 0.f, 0.f, 0.f);
    };
    int odd = 0;
    auto put = [&](int which, const float4* x) {
#pragma unroll
        for (int i = 0; i < LOADS; ++i) {
            if (LOAD_ROWS * i >= steps * 16) break;
            uint2 h, m, l;
            nm_f32_terms4(x[i], h, m, l);
            const uint32_t d = dst0 + (uint32_t)(which * 3 * TILE + i * LOAD_ROWS * 128);
            asm volatile("st.shared.v2.b32 [%0], {%1, %2};" ::"r"(d), "r"(h.x), "r"(h.y) : "memory");
            asm volatile("st.shared.v2.b32 [%0], {%1, %2};" ::"r"(d + TILE), "r"(m.x), "r"(m.y) : "memory");
            asm volatile("st.shared.v2.b32 [%0], {%1, %2};" ::"r"(d + 2 * TILE), "r"(l.x), "r"(l.y) : "memory");
            odd |= !(fmaxf(fmaxf(fabsf(x[i].x), fabsf(x[i].y)), fmaxf(fabsf(x[i].z), fabsf(x[i].w))) < TC_LIMIT) ||
                   !(x[i].x + x[i].y + x[i].z + x[i].w < INFINITY);   // (the maximum passes over a NaN)
        }
    };
    fetch(Qp, q);
    fetch(Kp, k);
    fetch(Vp, v);
    put(0, q);
    put(1, k);
    put(2, v);
    nm_fence_proxy_async();
    nm_tc_fence_before();
    odd = __syncthreads_or(odd);
    nm_tc_fence_after();
    const uint32_t tmem = tmem_slot;
    volatile int* abortp = &abort_flag;
    const uint32_t base = nm_smem_u32(tiles);
    constexpr uint64_t T1 = TILE >> 4;   // from term to term in a descriptor
    // Tensor memory: scores h h', mid, low at 0, 128, 256; then the scores at 0, the terms of P at 128, 192, 256; then O: h h' of keys
    // 0 to 63 and 64 to 127 at 0 and 64, mid at 320, low at 384.
    if (warp == 0 && !odd) {
        const uint32_t idesc = nm_idesc(1, 1, 0, 0, 128, 0) | ((uint32_t)(steps * 2) << 17);   // N = the keys
        const uint64_t qd = nm_smem_desc_sw128(base), kd = nm_smem_desc_sw128(base + 3 * TILE);
        if (nm_elect_one()) {
#pragma unroll
            for (int i = 0; i < 4; ++i) nm_mma_f16(tmem, qd + 2 * i, kd + 2 * i, idesc, i != 0);
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                nm_mma_f16(tmem + 128, qd + 2 * i, kd + T1 + 2 * i, idesc, i != 0);
                nm_mma_f16(tmem + 128, qd + T1 + 2 * i, kd + 2 * i, idesc, 1u);
            }
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                nm_mma_f16(tmem + 256, qd + T1 + 2 * i, kd + T1 + 2 * i, idesc, i != 0);
                nm_mma_f16(tmem + 256, qd + 2 * i, kd + 2 * T1 + 2 * i, idesc, 1u);
                nm_mma_f16(tmem + 256, qd + 2 * T1 + 2 * i, kd + 2 * i, idesc, 1u);
            }
            nm_tc_commit(&bar_s);
        }
        __syncwarp();
    }
    // ---- softmax: row 32 (warp % 4) + lane, 32 keys of it per thread, 16 at a time: loops, since a launch runs this code once or
    // twice, from a cold instruction cache
    const int row = (warp & 3) * 32 + lane, part = warp >> 2, key0 = part * PART_KEYS;
    const int lim = min(L - key0, PART_KEYS);   // keys of this thread that exist, at most 0: none
    const uint32_t t_row = tmem + ((uint32_t)((warp & 3) * 32) << 16);
    bool ok = true;
    if (odd) {
        scores_by_fma(Qp, Kp, a.stride_t, L, s_e);
    } else {
        ok = nm_mbar_wait(&bar_s, 0, abortp, a.status);
    }
    __syncwarp();
    nm_tc_fence_after();
    float m = -INFINITY;
#pragma unroll 1
    for (int c = 0; c < lim; c += 16) {
        uint32_t s[16];
        if (odd) {
#pragma unroll
            for (int j = 0; j < 16; ++j) s[j] = row < L && c + j < lim ? __float_as_uint(s_e[row * E_PITCH + key0 + c + j]) : 0u;
        } else {
            uint32_t mid[16], low[16];
            nm_tmem_ld16_sync(t_row + (uint32_t)(key0 + c), s);
            nm_tmem_ld16_sync(t_row + (uint32_t)(128 + key0 + c), mid);
            nm_tmem_ld16_sync(t_row + (uint32_t)(256 + key0 + c), low);
#pragma unroll
            for (int j = 0; j < 16; ++j) s[j] = __float_as_uint(nm_f32_sum(__uint_as_float(s[j]), mid[j], low[j]));
        }
#pragma unroll
        for (int j = 0; j < 16; ++j) {
            const float x = __uint_as_float(s[j]) * a.scale;
            s[j] = __float_as_uint(x);
            if (c + j < lim) m = fmaxf(m, x);
        }
        nm_tmem_st16(t_row + (uint32_t)(key0 + c), s);
    }
    nm_tmem_st_wait();
    s_red[part][row] = m;
    nm_tc_fence_before();
    __syncthreads();   // and the products have been read everywhere: P may take their place
    nm_tc_fence_after();
    m = fmaxf(fmaxf(s_red[0][row], s_red[1][row]), fmaxf(s_red[2][row], s_red[3][row]));
    float sum = 0.f;
    const float2* my = rep + (lane & 15);
    auto exponentials = [&](int c, float* e) {   // of keys key0 + c and on, 0 beyond L
        uint32_t s[16];
        nm_tmem_ld16_sync(t_row + (uint32_t)(key0 + c), s);
#pragma unroll
        for (int j = 0; j < 16; ++j) {
            const float x = __uint_as_float(s[j]) - m;
            const float2 t = my[nm_pwl_index(x, inv_h, off, nm1) * 16];
            e[j] = c + j < lim ? __fmaf_rn(t.x, x, t.y) : 0.f;
        }
    };
#pragma unroll 1
    for (int c = 0; c < lim; c += 16) {
        float e[16], some = 0.f;
        exponentials(c, e);
        uint32_t h[8], md[8], l[8];
#pragma unroll
        for (int j = 0; j < 16; j += 2) {
            some += e[j] + e[j + 1];
            odd |= row < L && (!(fabsf(e[j]) < TC_LIMIT) || !(fabsf(e[j + 1]) < TC_LIMIT));
            nm_f32_terms2(e[j], e[j + 1], h[j / 2], md[j / 2], l[j / 2]);
        }
        sum += some;
        const uint32_t t = t_row + (uint32_t)(128 + (key0 + c) / 2);
        nm_tmem_st8(t, h);
        nm_tmem_st8(t + 64, md);
        nm_tmem_st8(t + 128, l);
    }
    nm_tmem_st_wait();
    __syncthreads();   // the maxima have been read
    s_red[part][row] = sum;
    nm_tc_fence_before();
    odd = __syncthreads_or(odd);
    nm_tc_fence_after();
    sum = (s_red[0][row] + s_red[1][row]) + (s_red[2][row] + s_red[3][row]);
    const int ri = nm_pwl_index(sum, r_inv_h, r_off, r_nm1);
    const float2 rk = a.t_rcp->kb[ri];
    const float rinv = __fmaf_rn(rk.x, sum, rk.y);
    // ---- O = P V: 16 channels of a row per thread
    if (warp == 0 && !odd) {
        constexpr uint32_t idesc = nm_idesc(1, 1, 0, 1, 128, HD);
        auto vd = [base](int t, int i) { return nm_smem_desc_sw128(base + (uint32_t)((6 + t) * TILE + 16 * i * 128)); };
        auto p = [tmem](int t, int i) { return tmem + (uint32_t)(128 + 64 * t + 8 * i); };
        if (nm_elect_one()) {
            for (int i = 0; i < steps; ++i) nm_mma_f16_a_tmem(tmem + (i < 4 ? 0 : 64), p(0, i), vd(0, i), idesc, i & 3);
            for (int i = 0; i < steps; ++i) {
                nm_mma_f16_a_tmem(tmem + 320, p(0, i), vd(1, i), idesc, i != 0);
                nm_mma_f16_a_tmem(tmem + 320, p(1, i), vd(0, i), idesc, 1u);
            }
            for (int i = 0; i < steps; ++i) {
                nm_mma_f16_a_tmem(tmem + 384, p(1, i), vd(1, i), idesc, i != 0);
                nm_mma_f16_a_tmem(tmem + 384, p(0, i), vd(2, i), idesc, 1u);
                nm_mma_f16_a_tmem(tmem + 384, p(2, i), vd(0, i), idesc, 1u);
            }
            nm_tc_commit(&bar_o);
        }
        __syncwarp();
    }
    float* out = a.out + ((int64_t)b * L + row) * ((int64_t)a.heads * HD) + g * HD + part * 16;
    if (odd) {
#pragma unroll 1
        for (int c = 0; c < lim; c += 16) {
            float e[16];
            exponentials(c, e);
#pragma unroll
            for (int j = 0; j < 16; ++j) s_e[row * E_PITCH + key0 + c + j] = e[j];
        }
        output_by_fma(Vp, a.stride_t, L, s_e, rinv, out);
    } else {
        ok = nm_mbar_wait(&bar_o, 0, abortp, a.status) && ok;
        __syncwarp();
        nm_tc_fence_after();
        uint32_t h0[16], h1[16], mid[16], low[16];
        const uint32_t o = t_row + (uint32_t)(part * 16);
        nm_tmem_ld16_sync(o, h0);
        if (steps > 4) nm_tmem_ld16_sync(o + 64, h1);
        nm_tmem_ld16_sync(o + 320, mid);
        nm_tmem_ld16_sync(o + 384, low);
        float x[16];
#pragma unroll
        for (int j = 0; j < 16; ++j) {
            x[j] = __uint_as_float(h0[j]);
            if (steps > 4) x[j] += __uint_as_float(h1[j]);
            x[j] = nm_f32_sum(x[j], mid[j], low[j]) * rinv;
        }
        if (ok && row < L) {
#pragma unroll
            for (int j = 0; j < 16; j += 4) *reinterpret_cast<float4*>(out + j) = make_float4(x[j], x[j + 1], x[j + 2], x[j + 3]);
        }
    }
    nm_tc_fence_before();
    __syncthreads();
    if (warp == 0) {
        nm_tc_fence_after();
        nm_tmem_dealloc(tmem, 512);
    }
}

int score_pitch(int L) { return (L + KB - 1) / KB * KB + 4; }
size_t smem_bytes(int L) { return sizeof(float) * (2 * (size_t)NM_MAX_SEGMENTS + (QB + 2 * KB) * TP + (size_t)QB * score_pitch(L)); }

// Is the tensor-core kernel the faster one?  It holds one CTA, 128 rows, per SM whatever L is; the other one four, and up to
// 64 keys it needs one or two of 32 rows.  So with 65 to 128 keys always (4 to 1536 (batch, head) pairs: 0.37 to 1.05 of the other's time),
// with less if one round takes all pairs (L 16, 37, 64: 96 pairs 0.71, 0.70, 0.73; 12 pairs 0.80, 1.06, 1.14), not with more rounds
// (192 pairs 1.01, 1.22, 1.29; 1536 pairs 57 us against 31, 86 against 61, 97 against 63).
bool use_tc(const nm_attn_desc* d, int sms)
{
    return d->L <= 128 && (d->L > 64 || (int64_t)d->B * d->heads <= sms);
}

}  // namespace

bool nm_attention_f32_supported(const nm_attn_desc* d)
{
    if (d->dtype != NM_F32 || d->d != HD || d->L > 4096) return false;
    if (d->stride_t % 4 != 0 || d->stride_b % 4 != 0) return false;   // 16-byte loads of the rows
    return smem_bytes(d->L) <= 226 * 1024;
}

nm_status nm_launch_attention_f32(nm_ctx* ctx, const nm_attn_desc* d, cudaStream_t st)
{
    F32AttnArgs a;
    a.Q = (const float*)d->Q; a.K = (const float*)d->K; a.V = (const float*)d->V; a.out = (float*)d->out;
    a.B = d->B; a.L = d->L; a.heads = d->heads;
    a.q_blocks = (d->L + QB - 1) / QB;
    a.LP = score_pitch(d->L);
    a.stride_b = d->stride_b; a.stride_t = d->stride_t; a.scale = d->scale;
    a.t_exp = ctx->d_tables + d->exp_slot; a.t_rcp = ctx->d_tables + d->recip_slot;
    a.status = ctx->d_status;
    const bool tc = use_tc(d, ctx->sm_count);
    const int64_t blocks = (int64_t)(tc ? 1 : a.q_blocks) * d->heads * d->B;
    if (blocks > 0x7fffffffLL) return NM_ERR_UNSUPPORTED;
    auto kern = tc ? attention_f32_tc_kernel : attention_f32_kernel;
    const size_t smem = tc ? TC_SMEM : smem_bytes(d->L);
    if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, tc ? TC_SMEM : 226 * 1024) != cudaSuccess) return NM_ERR_CUDA;
    cudaLaunchConfig_t cfg;
    memset(&cfg, 0, sizeof(cfg));
    cfg.gridDim = dim3((unsigned)blocks);
    cfg.blockDim = dim3(tc ? TC_THREADS : THREADS);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = ctx->pdl ? 1 : 0;
    NmLaunchScope scope(ctx, tc ? NM_KERNEL_ATTENTION_TC : NM_KERNEL_ATTENTION_SIMT, 4.0 * (double)d->B * d->heads * (double)d->L * d->L * d->d, st);
    if (cudaLaunchKernelEx(&cfg, kern, a) != cudaSuccess) return NM_ERR_CUDA;
    return cudaGetLastError() == cudaSuccess ? NM_OK : NM_ERR_CUDA;
}

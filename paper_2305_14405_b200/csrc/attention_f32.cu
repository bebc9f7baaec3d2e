// fp32 attention with PWL softmax on the CUDA cores, heads of 64 channels.
//     s_j = scale*<q,k_j>; m = max s; e_j = PWLexp(s_j - m); sigma = sum e; r = PWLrecip(sigma); o = r * sum_j e_j v_j
// A CTA takes 32 queries of one (batch, head): the scores against all L keys stay in shared memory as fp32, so the
// final row maximum is known before the first exponential and nothing is computed twice.  K and then V pass through
// a two-stage cp.async ring in blocks of 64 keys; each of the 128 threads holds 4 x 4 scores, later 4 x 4 outputs, in
// registers, so an element read from shared memory serves four multiplications (the one-warp-per-row kernel in
// simt_kernels.cu reads K and V from the cache for every multiplication, and is left to other head sizes and to
// sequences whose scores do not fit).  Bound by shared-memory reads, 8 per 64 multiplications of a thread.
// B 8, L 128, 12 heads: 402 us with one warp per row, 18.6 us so.
#include <string.h>

#include "nm_common.cuh"

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

int score_pitch(int L) { return (L + KB - 1) / KB * KB + 4; }
size_t smem_bytes(int L) { return sizeof(float) * (2 * (size_t)NM_MAX_SEGMENTS + (QB + 2 * KB) * TP + (size_t)QB * score_pitch(L)); }

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
    const int64_t blocks = (int64_t)a.q_blocks * d->heads * d->B;
    if (blocks > 0x7fffffffLL) return NM_ERR_UNSUPPORTED;
    const size_t smem = smem_bytes(d->L);
    if (cudaFuncSetAttribute(attention_f32_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, 226 * 1024) != cudaSuccess)
        return NM_ERR_CUDA;
    cudaLaunchConfig_t cfg;
    memset(&cfg, 0, sizeof(cfg));
    cfg.gridDim = dim3((unsigned)blocks);
    cfg.blockDim = dim3(THREADS);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = ctx->pdl ? 1 : 0;
    NmLaunchScope scope(ctx, NM_KERNEL_ATTENTION_SIMT, 4.0 * (double)d->B * d->heads * (double)d->L * d->L * d->d, st);
    if (cudaLaunchKernelEx(&cfg, attention_f32_kernel, a) != cudaSuccess) return NM_ERR_CUDA;
    return cudaGetLastError() == cudaSuccess ? NM_OK : NM_ERR_CUDA;
}

// fp32 linear operator with PWL epilogue on the CUDA cores (the fp32 tolerance rules out tf32, and three-way bf16
// splits lose bits in the tensor cores' accumulation).
//
// Bound by the register file behind the FMA pipe: an 8 x 8 outer product with three distinct operands per instruction
// runs at 49 TFLOP/s as scalar FFMA and at 63 with the packed form (registers only, no loads), so the packed form it is,
// and it runs along K, where both operands lie as they are needed: a thread's accumulator is a PAIR of partial sums
// (even and odd k, added at the end), fma.rn.f32x2 takes two adjacent k of a row of A and of W, and nothing is transposed
// or duplicated.  One CTA per SM (two smaller ones are not placed evenly) computes a 128 x 64 tile with two groups of 128
// threads, 8 x 8 elements per thread; a group takes every other K-block of 32 with a cp.async ring and a named barrier of
// its own, so that the groups drift apart and one's barrier and first fragments hide behind the other's arithmetic
// (against one ring for both: 98 -> 89 us at 1024 x 2304 x 768).  Fragments are double-buffered in registers.  Problems of
// few tiles split K over a thread-block cluster.  1024 x 2304 x 768: 41 TFLOP/s; the 64 x 64-tile kernel before: 16.
#include "linear_split_kernel.cuh"

using namespace nm_tc;

namespace {

constexpr int FBM = BM;       // 128 rows, as Finisher expects
constexpr int FBN = 64;
constexpr int FG = 2;             // thread groups
constexpr int FBK = 32;
constexpr int FPITCH = FBK + 4;   // words per operand row: 8 rows of a warp's loads fall on distinct banks
constexpr int FSTAGES = 3;
constexpr int F_THREADS = 128 * FG;
constexpr int FSTAGE_WORDS = (FBM + FBN) * FPITCH;
constexpr int PART_WORDS = FBM * part_pitch(FBN);

__device__ __forceinline__ void cp_async16(uint32_t dst, const void* src, int bytes)
{
    // bytes < 16: the rest of the 16 are zero-filled and not read
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(bytes) : "memory");
}

__global__ void __launch_bounds__(F_THREADS, 1)
linear_f32_kernel(const float* __restrict__ A, const float* __restrict__ W, int64_t lda, int64_t ldw, const SplitArgs s)
{
    const TcArgs& a = s.t;
    extern __shared__ __align__(16) float fsm[];
    __shared__ float2 s_tab[NM_MAX_SEGMENTS];
    const int S = s.S;
    const int rank = S > 1 ? (int)nm_cluster_ctarank() : 0;
    const int tile = (int)blockIdx.x / S;
    const int mt = tile / a.num_n_tiles, nt = tile % a.num_n_tiles;
    const int kb0 = (int)((int64_t)rank * a.num_k_blocks / S), kb1 = (int)((int64_t)(rank + 1) * a.num_k_blocks / S);
    const int tid = threadIdx.x;
    const int64_t m0 = (int64_t)mt * FBM, n0 = (int64_t)nt * FBN;
    if (a.tab) {
        for (int i = tid; i < a.n_seg; i += F_THREADS) s_tab[i] = a.tab->kb[i];
    }
    nm_grid_launch_dependents();
    nm_grid_dependency_wait();

    // 192 operand rows of 8 chunks per stage, 12 chunks per thread of a group: rows gt/8 + 16 i (i < 8: A, else W)
    const int grp = tid >> 7, gt = tid & 127;
    float* ring = fsm + grp * FSTAGES * FSTAGE_WORDS;
    const int c4 = (gt & 7) * 4;
    const float* srcA = A + (m0 + (gt >> 3)) * lda + c4;
    const float* srcW = W + (n0 + (gt >> 3)) * ldw + c4;
    const int rowsA = (int)min((int64_t)FBM, a.M - m0) - (gt >> 3), rowsW = (int)min((int64_t)FBN, a.N - n0) - (gt >> 3);
    const uint32_t dst = nm_smem_u32(ring) + (uint32_t)((gt >> 3) * FPITCH + c4) * 4u;
    auto load = [&](int kb, int stage) {
        const int64_t left = a.K - ((int64_t)kb * FBK + c4);   // valid elements from this chunk's first k on
        const int bytes = left >= 4 ? 16 : (left > 0 ? (int)left * 4 : 0);
        const uint32_t d = dst + (uint32_t)(stage * FSTAGE_WORDS) * 4u;
        const float* pa = srcA + (int64_t)kb * FBK;
        const float* pw = srcW + (int64_t)kb * FBK;
#pragma unroll
        for (int i = 0; i < FBM / 16; ++i) {
            const int n = 16 * i < rowsA ? bytes : 0;
            cp_async16(d + (uint32_t)(16 * i * FPITCH) * 4u, n ? (const void*)(pa + 16 * i * lda) : (const void*)A, n);
        }
#pragma unroll
        for (int i = 0; i < FBN / 16; ++i) {
            const int n = 16 * i < rowsW ? bytes : 0;
            cp_async16(d + (uint32_t)((FBM + 16 * i) * FPITCH) * 4u, n ? (const void*)(pw + 16 * i * ldw) : (const void*)A, n);
        }
    };
    const int ty = (gt >> 5) * 4 + ((gt & 31) >> 3), tx = gt & 7;   // rows ty + 16 i, columns tx + 8 j
    uint64_t acc[8][8];   // sums over the even and the odd k
#pragma unroll
    for (int i = 0; i < 8; ++i)
#pragma unroll
        for (int j = 0; j < 8; ++j) acc[i][j] = 0ull;

#pragma unroll
    for (int i = 0; i < FSTAGES - 1; ++i) {
        if (kb0 + grp + FG * i < kb1) load(kb0 + grp + FG * i, i);
        asm volatile("cp.async.commit_group;" ::: "memory");
    }
    int stage = 0;
    for (int kb = kb0 + grp; kb < kb1; kb += FG) {
        asm volatile("cp.async.wait_group %0;" ::"n"(FSTAGES - 2) : "memory");
        // this K-block has landed for the whole group, and all of it has left the stage loaded next
        asm volatile("bar.sync %0, %1;" ::"r"(1 + grp), "n"(128) : "memory");
        if (kb + FG * (FSTAGES - 1) < kb1) load(kb + FG * (FSTAGES - 1), stage == 0 ? FSTAGES - 1 : stage - 1);
        asm volatile("cp.async.commit_group;" ::: "memory");
        const float* sa = ring + stage * FSTAGE_WORDS + ty * FPITCH;
        const float* sb = ring + stage * FSTAGE_WORDS + (FBM + tx) * FPITCH;
        uint64_t ra[2][8], rb[2][8];
        auto frag = [&](int b, int k2) {
#pragma unroll
            for (int i = 0; i < 8; ++i) ra[b][i] = *reinterpret_cast<const uint64_t*>(sa + 16 * i * FPITCH + k2);
#pragma unroll
            for (int j = 0; j < 8; ++j) rb[b][j] = *reinterpret_cast<const uint64_t*>(sb + 8 * j * FPITCH + k2);
        };
        frag(0, 0);
#pragma unroll
        for (int k2 = 0; k2 < FBK; k2 += 2) {
            const int b = (k2 >> 1) & 1;
            if (k2 + 2 < FBK) frag(b ^ 1, k2 + 2);
#pragma unroll
            for (int j = 0; j < 8; ++j)
#pragma unroll
                for (int i = 0; i < 8; ++i) asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(acc[i][j]) : "l"(ra[b][i]), "l"(rb[b][j]));
        }
        stage = stage + 1 == FSTAGES ? 0 : stage + 1;
    }
    asm volatile("cp.async.wait_group 0;" ::: "memory");
    __syncthreads();   // everyone is done with the rings: the groups' tiles take their place
    constexpr int PITCH = part_pitch(FBN);
    float* part = fsm;
    {
        float* mine = part + grp * PART_WORDS;
#pragma unroll
        for (int i = 0; i < 8; ++i)
#pragma unroll
            for (int j = 0; j < 8; ++j) {
                float lo, hi;
                nm_unpack2(acc[i][j], lo, hi);
                mine[(ty + 16 * i) * PITCH + tx + 8 * j] = lo + hi;
            }
    }
    __syncthreads();
#pragma unroll
    for (int i = 0; i < FBM * FBN / 4 / F_THREADS; ++i) {   // the groups' sum
        const int u = tid + i * F_THREADS;
        float* p = part + (u / (FBN / 4)) * PITCH + (u % (FBN / 4)) * 4;
        float4 v = *reinterpret_cast<const float4*>(p);
#pragma unroll
        for (int g = 1; g < FG; ++g) {
            const float4 o = *reinterpret_cast<const float4*>(p + g * PART_WORDS);
            v.x += o.x; v.y += o.y; v.z += o.z; v.w += o.w;
        }
        *reinterpret_cast<float4*>(p) = v;
    }
    const int rows = (int)(a.M - m0 < FBM ? a.M - m0 : FBM);
    Finisher<false, float, FBN, false, F_THREADS, false> fin(s, rank, mt, nt, rows, Patch{0, 0, 0});
    fin.prefetch_vectors();
    fin.load_res(0);
    if (S > 1) nm_cluster_sync();
    else __syncthreads();
    fin.run(reinterpret_cast<const uint32_t*>(part), s_tab);
    if (S > 1) nm_cluster_sync();   // a peer may still be reading this CTA's partial tile
}

// CTAs per cluster: the least time by measured figures, in us: 1.65 per K-block of 32, 4.9 per round of CTAs for the
// launch, the ring's fill and the epilogue, 0.7 + 0.25 S for the exchange.  A round is what the GPU holds of clusters of S,
// which is less than its SMs for most S.
int choose_f32_split(int64_t tiles, int k_blocks, const int* resident)
{
    int best = 1;
    double best_t = 1e30;
    for (int S = 1; S <= 8 && S <= k_blocks; ++S) {
        if (resident[S] < 1) continue;
        const double rounds = (double)((tiles + resident[S] - 1) / resident[S]);
        const double t = rounds * (1.65 * ((k_blocks + S - 1) / S) + 4.9 + (S > 1 ? 0.7 + 0.25 * S : 0.0));
        if (t < best_t * 0.98) { best_t = t; best = S; }
    }
    return best;
}

}  // namespace

bool nm_linear_f32_supported(const nm_linear_desc* d)
{
    return d->in_dtype == NM_F32 && d->N % 4 == 0 && d->K <= 0x7fffffffLL;
}

nm_status nm_launch_linear_f32(nm_ctx* ctx, const nm_linear_desc* d, cudaStream_t st)
{
    const int64_t m_tiles = (d->M + FBM - 1) / FBM, n_tiles = (d->N + FBN - 1) / FBN, tiles = m_tiles * n_tiles;
    if ((d->M + 63) / 64 > 65535 || tiles > 0x7fffffffLL / 8) return NM_ERR_SHAPE;
    SplitArgs s;
    memset(&s, 0, sizeof(s));
    TcArgs& a = s.t;
    a.M = d->M; a.N = d->N; a.K = d->K;
    a.bias = d->bias;
    a.res_first = d->res_first;
    a.tab = d->slot == NM_SLOT_NONE ? nullptr : ctx->d_tables + d->slot;
    a.n_seg = d->slot == NM_SLOT_NONE ? 0 : ctx->h_tables[d->slot].n;
    a.idx_dump = d->idx_dump;
    a.num_n_tiles = (int)n_tiles;
    a.num_tiles = (int)tiles;
    a.num_k_blocks = (int)((d->K + FBK - 1) / FBK);
    s.residual = d->residual; s.ldr = d->ldr;
    s.out = d->out; s.ldo = d->ldo;
    constexpr size_t smem = (size_t)FG * FSTAGES * FSTAGE_WORDS * 4;
    static_assert(PART_WORDS <= FSTAGES * FSTAGE_WORDS, "partial tiles");
    if (cudaFuncSetAttribute(linear_f32_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) != cudaSuccess)
        return NM_ERR_CUDA;
    cudaLaunchConfig_t cfg;
    memset(&cfg, 0, sizeof(cfg));
    cfg.blockDim = dim3(F_THREADS);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute attr[2];
    cfg.attrs = attr;
    // clusters of 1..8 CTAs the device holds, asked for once per context (or by several threads, which find the same; the first
    // word is set when the others are, and orders them for a thread that did not ask)
    int* resident = ctx->f32_resident;
    if (__atomic_load_n(&resident[0], __ATOMIC_ACQUIRE) == 0) {
        for (int S = 1; S <= 8; ++S) {
            int n = 0;
            cfg.numAttrs = split_launch_attrs(ctx, attr, S);
            cfg.gridDim = dim3((unsigned)(S * ctx->sm_count));
            if (cudaOccupancyMaxActiveClusters(&n, linear_f32_kernel, &cfg) != cudaSuccess) {
                (void)cudaGetLastError();
                n = S == 1 ? ctx->sm_count : 0;
            }
            __atomic_store_n(&resident[S], n, __ATOMIC_RELAXED);
        }
        __atomic_store_n(&resident[0], 1, __ATOMIC_RELEASE);
    }
    s.S = choose_f32_split(tiles, a.num_k_blocks, resident);
    cfg.numAttrs = split_launch_attrs(ctx, attr, s.S);
    cfg.gridDim = dim3((unsigned)(tiles * s.S));
    NmLaunchScope scope(ctx, NM_KERNEL_LINEAR_SIMT, 2.0 * (double)d->M * (double)d->N * (double)d->K, st);
    if (cudaLaunchKernelEx(&cfg, linear_f32_kernel, (const float*)d->A, (const float*)d->W, d->lda, d->ldw, s) != cudaSuccess)
        return NM_ERR_CUDA;
    return cudaGetLastError() == cudaSuccess ? NM_OK : NM_ERR_CUDA;
}

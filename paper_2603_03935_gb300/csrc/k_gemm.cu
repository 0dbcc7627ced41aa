// D-weighted mask pooling as a tensor-core GEMM (Sec. III-C: each mask's
// embedding is the sum of its patches' features, each weighted by its
// distinctiveness D and its share of the mask).
//
//   E[m][d] = sum_p W[m][p] * F[p][d]      (W: pooling weights, F: tokens)
//
// computed as E^T = F^T W^T so the long token dimension D fills the 128 rows
// of one tcgen05 MMA and the masks (<= 256) form its N dimension:
//   A (128 x 32, K-major) = F^T tile  -- transposed while staged into shared memory
//   B (N   x 32, K-major) = W tile    -- W rows are already K-contiguous
// FP32 precision: the fp32 operands are split as x = hi + lo with hi, lo TF32
// and three kind::tf32 MMAs (hi*hi + hi*lo + lo*hi) accumulate in fp32 in
// TMEM, which keeps the fp32-level accuracy of the product (relative error
// ~1e-6).  BF16 precision: both operands rounded to bf16 (tokens given in
// bf16 are exact), one kind::f16 MMA per 16-wide K step, fp32 accumulation.
// FP8 precision: E4M3 operands with power-of-two scales, token p as
// rn(f_p / 2^a_p) and the weight rows prepared by the weights kernel, one
// kind::f8f6f4 MMA per 32-wide K step; the epilogue multiplies column m by
// its row scale 2^b_m.
//
// The patches (K) fall into up to 8 groups of chunks, by their number alone.
// Each group is accumulated by itself and the groups' sums are added in order,
// so E does not depend on how many CTAs share the work.  A 128-row tile of D
// belongs to a cluster of KS CTAs, each of which takes a KS-th of the groups;
// with KS > 1 the groups' sums meet through distributed shared memory, with
// one CTA they are added on the way.  One elected thread issues the MMAs; a
// two-stage shared-memory ring is recycled through mbarriers that
// tcgen05.commit arrives on.  Every wait is bounded by a global-timer limit
// after which the kernel records DISC_ERR_TIMEOUT and returns.
//
// The contraction reads each token once for ~M/2 flop per byte, so it is bound
// by how many token loads are in flight: 256 threads of 16 loads, one chunk
// ahead, two CTAs per SM.  bf16 tokens stay as loaded until they are staged
// (widened at the load, they made every chunk wait for the next one's: 32
// building frames at BF16 63 us, 55 so).  With 128 threads, one CTA per SM and
// one CTA per tile whatever the batch, a 32-frame Room batch took 95 us (now
// 53) and a single frame (6 CTAs) 59 us (now 15).
#include <cuda_bf16.h>

#include <algorithm>

#include "disc_common.cuh"
#include "kernels.h"

namespace disc {

namespace {

__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ float tf32_rna(float x)
{
    uint32_t r;
    asm("cvt.rna.tf32.f32 %0, %1;" : "=r"(r) : "f"(x));
    return __uint_as_float(r);
}

// Shared-memory matrix descriptor, SWIZZLE_NONE, K-major canonical layout:
// core matrices of 8 rows x 16 bytes stored contiguously (128 B); LBO = byte
// distance between core matrices adjacent along K, SBO = along M/N.
__device__ __forceinline__ uint64_t smem_desc(uint32_t addr, uint32_t lbo, uint32_t sbo)
{
    uint64_t d = 0;
    d |= (uint64_t)((addr >> 4) & 0x3FFFu);
    d |= (uint64_t)((lbo >> 4) & 0x3FFFu) << 16;
    d |= (uint64_t)((sbo >> 4) & 0x3FFFu) << 32;
    d |= (uint64_t)1 << 46;  // descriptor version of the tcgen05 family
    return d;                // base offset 0, absolute LBO mode, no swizzle
}

// Instruction descriptor of kind::tf32: D fp32, A/B tf32, both K-major.
__host__ __device__ constexpr uint32_t idesc_tf32(int M, int N)
{
    return (1u << 4) | (2u << 7) | (2u << 10) | ((uint32_t)(N >> 3) << 17) | ((uint32_t)(M >> 4) << 24);
}

__device__ __forceinline__ void mma_tf32(uint32_t tmem_d, uint64_t a, uint64_t b, uint32_t idesc, uint32_t acc)
{
    asm volatile(
        "{\n.reg .pred p;\nsetp.ne.b32 p, %4, 0;\n"
        "tcgen05.mma.cta_group::1.kind::tf32 [%0], %1, %2, %3, p;\n}\n" ::"r"(tmem_d),
        "l"(a), "l"(b), "r"(idesc), "r"(acc));
}

// Instruction descriptor of kind::f16 with bf16 A/B: D fp32, both K-major.
__host__ __device__ constexpr uint32_t idesc_bf16(int M, int N)
{
    return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(N >> 3) << 17) | ((uint32_t)(M >> 4) << 24);
}

__device__ __forceinline__ void mma_bf16(uint32_t tmem_d, uint64_t a, uint64_t b, uint32_t idesc, uint32_t acc)
{
    asm volatile(
        "{\n.reg .pred p;\nsetp.ne.b32 p, %4, 0;\n"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(tmem_d),
        "l"(a), "l"(b), "r"(idesc), "r"(acc));
}

// Instruction descriptor of kind::f8f6f4 with E4M3 A/B: D fp32, both K-major.
__host__ __device__ constexpr uint32_t idesc_e4m3(int M, int N)
{
    return (1u << 4) | (0u << 7) | (0u << 10) | ((uint32_t)(N >> 3) << 17) | ((uint32_t)(M >> 4) << 24);
}

__device__ __forceinline__ void mma_e4m3(uint32_t tmem_d, uint64_t a, uint64_t b, uint32_t idesc, uint32_t acc)
{
    asm volatile(
        "{\n.reg .pred p;\nsetp.ne.b32 p, %4, 0;\n"
        "tcgen05.mma.cta_group::1.kind::f8f6f4 [%0], %1, %2, %3, p;\n}\n" ::"r"(tmem_d),
        "l"(a), "l"(b), "r"(idesc), "r"(acc));
}

__device__ __forceinline__ uint32_t pack_e4m3(float a, float b, float c, float d)
{
    return (uint32_t)to_e4m3(a) | ((uint32_t)to_e4m3(b) << 8) | ((uint32_t)to_e4m3(c) << 16) |
           ((uint32_t)to_e4m3(d) << 24);
}

__device__ __forceinline__ uint32_t pack_bf16(float lo, float hi)
{
    return (uint32_t)__bfloat16_as_ushort(__float2bfloat16_rn(lo)) |
           ((uint32_t)__bfloat16_as_ushort(__float2bfloat16_rn(hi)) << 16);
}

__device__ __forceinline__ void mma_commit(uint32_t mbar)
{
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(mbar)
                 : "memory");
}

__device__ __forceinline__ uint64_t global_ns()
{
    uint64_t t;
    asm volatile("mov.u64 %0, %globaltimer;" : "=l"(t));
    return t;
}

// bounded wait for the phase with the given parity; false after ~1 s
__device__ __forceinline__ bool mbar_wait(uint32_t mbar, uint32_t parity)
{
    const uint64_t t0 = global_ns();
    while (true) {
        uint32_t ok;
        asm volatile(
            "{\n.reg .pred p;\nmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\nselp.u32 %0, 1, 0, p;\n}\n"
            : "=r"(ok)
            : "r"(mbar), "r"(parity)
            : "memory");
        if (ok) return true;
        if (global_ns() - t0 > 1000000000ull) return false;
    }
}

// 16 accumulator columns of the warp's 32 lanes; the registers hold them after
// tcgen05.wait::ld, and tmem_use keeps their uses behind it
__device__ __forceinline__ void tmem_ld16(uint32_t taddr, uint32_t (&r)[16])
{
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
          "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
        : "r"(taddr));
}
__device__ __forceinline__ void tmem_use(uint32_t (&r)[16])
{
#pragma unroll
    for (int j = 0; j < 16; j++) asm volatile("" : "+r"(r[j]));
}
__device__ __forceinline__ void tmem_st16(uint32_t taddr, const float (&v)[16])
{
    asm volatile(
        "tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16};" ::"r"(
            taddr),
        "f"(v[0]), "f"(v[1]), "f"(v[2]), "f"(v[3]), "f"(v[4]), "f"(v[5]), "f"(v[6]), "f"(v[7]), "f"(v[8]), "f"(v[9]),
        "f"(v[10]), "f"(v[11]), "f"(v[12]), "f"(v[13]), "f"(v[14]), "f"(v[15])
        : "memory");
}

__device__ __forceinline__ void fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }

// a token as it lies in memory (a chunk's loads stay in flight until they are
// widened, where the chunk is staged) and its value
__device__ __forceinline__ float ldtok(const float* F, size_t i) { return __ldg(F + i); }
__device__ __forceinline__ unsigned short ldtok(const __nv_bfloat16* F, size_t i)
{
    return __ldg((const unsigned short*)F + i);
}
__device__ __forceinline__ float tok_f32(float x) { return x; }
__device__ __forceinline__ float tok_f32(unsigned short x) { return __uint_as_float((unsigned)x << 16); }

}  // namespace

constexpr uint32_t A_TILE_BYTES = GEMM_MT * GEMM_KC * 4;  // 16 KB (tf32); bf16 tiles take half, e4m3 a quarter
constexpr uint32_t A_LBO = (GEMM_MT / 8) * 128;           // 2048: next 16-byte K group (4 tf32 / 8 bf16 / 16 e4m3)

constexpr int GEMM_THREADS = 256;
constexpr int GEMM_GROUPS = 8;  // groups of chunks at most

// Tensor memory: registers let two CTAs onto an SM, not three
// (set_gemm_kernel_attrs checks that), and a CTA takes at most half of the SM's
// 512 columns, or all of its shared memory as well. So an allocation never
// waits (a cluster's CTA that waited for columns held by another cluster could
// wait for itself).
constexpr int GEMM_COLS = 256;
constexpr size_t SMEM_MAX = 227 * 1024, GEMM_SMEM = SMEM_MAX - 1024;  // (beside the kernel's static bytes)
__host__ __device__ constexpr uint32_t columns_of(int n)
{
    return n <= 32 ? 32 : n <= 64 ? 64 : n <= 128 ? 128 : n <= 256 ? 256 : 512;
}
// operand bytes of one stage: tf32 A hi | A lo (fp32 tokens only: bf16 ones are exact in tf32) | B hi | B lo, or
// bf16 / e4m3 A | B
__host__ __device__ constexpr uint32_t gemm_stage_bytes(int NT, int precision, bool bf16_tokens)
{
    return precision == DISC_FP8_E4M3 ? A_TILE_BYTES / 4 + (uint32_t)NT * GEMM_KC
           : precision == DISC_BF16   ? A_TILE_BYTES / 2 + (uint32_t)NT * GEMM_KC * 2
                                      : A_TILE_BYTES * (bf16_tokens ? 1 : 2) + (uint32_t)NT * GEMM_KC * 8;
}
// columns of one CTA's accumulators: with a cluster one per group, else one
// and the sum of the groups before
__host__ __device__ constexpr int gemm_columns(int NT, int KS, int groups)
{
    return KS > 1 ? groups / KS * NT : groups > 1 ? 2 * NT : NT;
}
// The bytes of one CTA: two pipeline stages and the barriers; with a cluster
// also room for the partial sums over the stages.
__host__ size_t gemm_smem_bytes(int NT, int precision, bool bf16_tokens, int KS, int groups)
{
    if (gemm_columns(NT, KS, groups) > GEMM_COLS) return GEMM_SMEM;
    size_t b = 2 * (size_t)gemm_stage_bytes(NT, precision, bf16_tokens);
    if (KS > 1) b = std::max(b, (size_t)(groups / KS) * NT * GEMM_MT * 4);
    return b + 128;
}
static_assert(2 * gemm_stage_bytes(MAX_MASKS, DISC_FP32, false) + 128 <= GEMM_SMEM, "the largest stage pair fits an SM");
static_assert((size_t)MAX_MASKS * GEMM_MT * 4 + 128 <= GEMM_SMEM, "so do the partial sums of a group");

// Test hook: when set, the kernel issues no MMA and no commit, so its bounded
// waits run out and the frame fails with DISC_ERR_TIMEOUT (nothing is in
// flight when the tensor memory is freed).
__device__ int g_gemm_stall = 0;

cudaError_t set_gemm_stall(bool on)
{
    const int v = on ? 1 : 0;
    return cudaMemcpyToSymbol(g_gemm_stall, &v, sizeof(v));
}

// PR: the disc_precision of the frames this instance serves
template <typename T, int PR>
__global__ void __launch_bounds__(GEMM_THREADS, 2) k_pool_gemm(const FrameParams* fps, BatchScratch bs, int NT,
                                                               int groups)
{
    extern __shared__ __align__(128) uint8_t smem[];
    __shared__ int s_err;
    const FrameParams& fp = fps[blockIdx.z];
    const Scratch sc = bs.frame(blockIdx.z);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const T* F = (const T*)fp.tokens;
    const int D = fp.D, P = fp.P, M = fp.M;
    const int d0 = blockIdx.y * GEMM_MT;
    const unsigned KS = gridDim.x, rank = blockIdx.x;  // the cluster spans the grid's x
    // uniform for the cluster: other dtype or precision, no masks, tile past D
    if (fp.token_bf16 != (sizeof(T) == 2) || fp.precision != PR || M <= 0 || d0 >= D) return;
    // a failed frame: every CTA takes what its cluster's first one read
    if (tid == 0) s_err = *(volatile int32_t*)&sc.ctr->err;
    int frame_err;
    if (KS > 1) {
        cluster_sync();
        frame_err = dsm_ld32(dsm_map(&s_err, 0));
        cluster_sync();  // the first one stays until all have read
    } else {
        __syncthreads();
        frame_err = s_err;
    }
    if (frame_err) return;

    constexpr bool BF = PR == DISC_BF16, F8 = PR == DISC_FP8_E4M3, LO = sizeof(T) == 4;
    constexpr uint32_t EB = F8 ? 1 : (BF ? 2 : 4);  // operand bytes
    constexpr uint32_t A_BYTES = A_TILE_BYTES / 4 * EB;
    const uint32_t B_TILE_BYTES = (uint32_t)NT * GEMM_KC * EB;
    const uint32_t B_LBO = (uint32_t)NT * 16;
    const uint32_t STAGE = gemm_stage_bytes(NT, PR, !LO);
    // the barriers lie past the stages and past the partial sums over them
    const int gp = groups / (int)KS;  // groups of this CTA
    const size_t used = max(2 * (size_t)STAGE, KS > 1 ? (size_t)gp * NT * GEMM_MT * 4 : (size_t)0);
    uint64_t* mbar = (uint64_t*)(smem + used);
    uint32_t* tmem_slot = (uint32_t*)(mbar + 2);
    const bool sums = KS == 1 && gp > 1;
    const uint32_t ncols = columns_of(gemm_columns(NT, (int)KS, groups));

    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)),
                     "r"(ncols)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    if (tid == 0) {
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_u32(&mbar[0])) : "memory");
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_u32(&mbar[1])) : "memory");
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    fence_before();
    __syncthreads();
    fence_after();
    const uint32_t tmem = *tmem_slot;
    const uint32_t idesc = F8 ? idesc_e4m3(GEMM_MT, NT) : (BF ? idesc_bf16(GEMM_MT, NT) : idesc_tf32(GEMM_MT, NT));
    // this CTA's share of the 32-patch chunks
    const int all_chunks = (P + GEMM_KC - 1) / GEMM_KC;
    const int cb = (int)(all_chunks * rank / KS), nchunks = (int)(all_chunks * (rank + 1) / KS) - cb;
    auto group_start = [&](int g) { return all_chunks * ((int)rank * gp + g) / groups - cb; };
    int group = 0, group_at = 0, group_end = group_start(1);  // the group of the current chunk
    bool failed = false;
    int last_commit = -1;  // chunk of the most recent commit (same on all threads)
    const bool stall = g_gemm_stall != 0;  // uniform: read once
    // Thread tid stages half a row of the F^T tile: 16 tokens of row d0 + (tid
    // & 127), and its granules of the weight tile.  Those of the next chunk
    // are loaded into registers while the current chunk is staged and
    // multiplied, so loads stay in flight across the loop.
    constexpr int HALF = GEMM_KC / 2, WPRE = 2;
    const int row = tid & 127, half = tid >> 7;
    using Raw = decltype(ldtok((const T*)nullptr, 0));
    auto load_chunk = [&](int c, Raw (&x)[HALF]) {
        const int d = d0 + row, p0 = (cb + c) * GEMM_KC + half * HALF;
#pragma unroll
        for (int j = 0; j < HALF; j++) {
            const int p = p0 + j;
            x[j] = (d < D && p < P) ? ldtok(F, (size_t)p * D + d) : Raw(0);
        }
    };
    // granule g of the chunk's weight tile: 16 bytes of e4m3, or 16 bytes of
    // fp32 (half a granule of bf16: two per 16 staged bytes)
    constexpr int GPR = F8 ? GEMM_KC / 16 : GEMM_KC / 4;  // granules per weight row
    const int granules = NT * GPR;
    auto load_w = [&](int c, int g) -> float4 {
        const int n = g / GPR, kq = g % GPR, p0 = (cb + c) * GEMM_KC;
        if constexpr (F8) return *(const float4*)(sc.W8 + (size_t)n * fp.Kpad + p0 + 16 * kq);
        else return *(const float4*)(sc.W + (size_t)n * fp.Kpad + p0 + 4 * kq);
    };
    Raw xn[HALF];
    float4 wn[WPRE];
    auto prefetch = [&](int c) {
        load_chunk(c, xn);
#pragma unroll
        for (int i = 0; i < WPRE; i++) {
            const int g = tid + i * GEMM_THREADS;
            wn[i] = g < granules ? load_w(c, g) : make_float4(0.0f, 0.0f, 0.0f, 0.0f);
        }
    };
    if (nchunks > 0) prefetch(0);

    // The accumulators in tensor memory: warp w reads lanes 32 (w & 3) .. + 31
    // (rows of D), columns (masks) in 16s, alternating between the two warps
    // of the same lanes.  add_group: 16 columns of the group's accumulator
    // onto the sum of the groups before.
    const uint32_t tlane = tmem + ((uint32_t)((warp & 3) * 32) << 16);
    const int er = (warp & 3) * 32 + lane;
    float* out = sc.Efast + d0 + er;  // of mask 0
    const bool er_in = d0 + er < D;
    auto add_group = [&](int c0, float (&v)[16]) {
        uint32_t r[16], q[16];
        tmem_ld16(tlane + (uint32_t)c0, r);
        if (group > 0) tmem_ld16(tlane + (uint32_t)(NT + c0), q);
        asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
        tmem_use(r);
        if (group > 0) tmem_use(q);
#pragma unroll
        for (int j = 0; j < 16; j++)
            v[j] = __fadd_rn(group > 0 ? __uint_as_float(q[j]) : 0.0f, __uint_as_float(r[j]));
    };

    for (int c = 0; c < nchunks && !failed; c++) {
        const int s = c & 1;
        uint8_t* st = smem + s * STAGE;
        float x[HALF];
        float4 w[WPRE];
#pragma unroll
        for (int j = 0; j < HALF; j++) x[j] = tok_f32(xn[j]);
#pragma unroll
        for (int i = 0; i < WPRE; i++) w[i] = wn[i];
        if (c + 1 < nchunks) prefetch(c + 1);
        if (c >= 2) {
            // the MMAs of chunk c-2 read this stage: wait for their commit
            bool ok = mbar_wait(smem_u32(&mbar[s]), (uint32_t)(((c >> 1) - 1) & 1));
            if (__syncthreads_or(!ok)) { failed = true; break; }
        }
        if (c == group_end) {
            if (sums) {  // the group is whole once its last chunk's MMAs are done
                const bool ok = mbar_wait(smem_u32(&mbar[s ^ 1]), (uint32_t)(((c - 1) >> 1) & 1));
                if (__syncthreads_or(!ok)) { failed = true; break; }
                fence_after();
                for (int c0 = 16 * (warp >> 2); c0 < NT; c0 += 32) {
                    float v[16];
                    add_group(c0, v);
                    tmem_st16(tlane + (uint32_t)(NT + c0), v);
                }
                asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
                fence_before();  // (the next MMAs overwrite the accumulator after the barrier below)
            }
            group_at = c;
            group++;
            group_end = group_start(group + 1);
        }
        // A: the F^T tile
        if constexpr (F8) {
            // 16 patches of e4m3 in 16 B; one exact multiply by 2^-a_p each
            const float4* qm = (const float4*)(sc.qmul + (cb + c) * GEMM_KC + half * HALF);  // zero past P
#pragma unroll
            for (int q4 = 0; q4 < HALF / 4; q4++) {
                const float4 mu = qm[q4];
                x[4 * q4] = __fmul_rn(x[4 * q4], mu.x);
                x[4 * q4 + 1] = __fmul_rn(x[4 * q4 + 1], mu.y);
                x[4 * q4 + 2] = __fmul_rn(x[4 * q4 + 2], mu.z);
                x[4 * q4 + 3] = __fmul_rn(x[4 * q4 + 3], mu.w);
            }
            const uint4 v = make_uint4(pack_e4m3(x[0], x[1], x[2], x[3]), pack_e4m3(x[4], x[5], x[6], x[7]),
                                       pack_e4m3(x[8], x[9], x[10], x[11]), pack_e4m3(x[12], x[13], x[14], x[15]));
            *(uint4*)(st + half * A_LBO + row * 16) = v;
        } else if constexpr (BF) {
            // 8 patches of bf16 per 16 B
#pragma unroll
            for (int k = 0; k < HALF / 8; k++) {
                const float* y = x + 8 * k;
                const uint4 v = make_uint4(pack_bf16(y[0], y[1]), pack_bf16(y[2], y[3]), pack_bf16(y[4], y[5]),
                                           pack_bf16(y[6], y[7]));
                *(uint4*)(st + (half * (HALF / 8) + k) * A_LBO + row * 16) = v;
            }
        } else {
#pragma unroll
            for (int k = 0; k < HALF / 4; k++) {
                const float* y = x + 4 * k;
                const uint32_t off = (half * (HALF / 4) + k) * A_LBO + row * 16;
                if constexpr (LO) {
                    float4 hi, lo;
                    hi.x = tf32_rna(y[0]); lo.x = tf32_rna(y[0] - hi.x);
                    hi.y = tf32_rna(y[1]); lo.y = tf32_rna(y[1] - hi.y);
                    hi.z = tf32_rna(y[2]); lo.z = tf32_rna(y[2] - hi.z);
                    hi.w = tf32_rna(y[3]); lo.w = tf32_rna(y[3] - hi.w);
                    *(float4*)(st + off) = hi;
                    *(float4*)(st + A_BYTES + off) = lo;
                } else {
                    *(float4*)(st + off) = make_float4(y[0], y[1], y[2], y[3]);  // bf16 values are tf32 values
                }
            }
        }
        // B: the weight rows
        auto stage_w = [&](int g, float4 v) {
            const int n = g / GPR, kq = g % GPR;
            if constexpr (F8) {
                *(float4*)(st + A_BYTES + kq * B_LBO + n * 16) = v;
            } else if constexpr (BF) {
                *(uint2*)(st + A_BYTES + (kq >> 1) * B_LBO + n * 16 + (kq & 1) * 8) =
                    make_uint2(pack_bf16(v.x, v.y), pack_bf16(v.z, v.w));
            } else {
                float4 hi, lo;
                hi.x = tf32_rna(v.x); lo.x = tf32_rna(v.x - hi.x);
                hi.y = tf32_rna(v.y); lo.y = tf32_rna(v.y - hi.y);
                hi.z = tf32_rna(v.z); lo.z = tf32_rna(v.z - hi.z);
                hi.w = tf32_rna(v.w); lo.w = tf32_rna(v.w - hi.w);
                uint8_t* Bhi = st + (LO ? 2 : 1) * A_BYTES;
                const uint32_t off = kq * B_LBO + n * 16;
                *(float4*)(Bhi + off) = hi;
                *(float4*)(Bhi + B_TILE_BYTES + off) = lo;
            }
        };
#pragma unroll
        for (int i = 0; i < WPRE; i++)
            if (tid + i * GEMM_THREADS < granules) stage_w(tid + i * GEMM_THREADS, w[i]);
        for (int g = tid + WPRE * GEMM_THREADS; g < granules; g += GEMM_THREADS) stage_w(g, load_w(c, g));
        // make the generic-proxy stores visible to the tensor core (async proxy)
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        __syncthreads();
        if (tid == 0 && !stall) {
            fence_after();
            const uint32_t acc = tmem + (KS > 1 ? (uint32_t)(group * NT) : 0u);
            if constexpr (F8) {
                // one K step of 32 = two 16-byte core-matrix columns of e4m3
                const uint32_t a0 = smem_u32(st), b0 = a0 + A_BYTES;
                mma_e4m3(acc, smem_desc(a0, A_LBO, 128), smem_desc(b0, B_LBO, 128), idesc, c > group_at ? 1u : 0u);
            } else if constexpr (BF) {
                // K step 16 = two 16-byte core-matrix columns of bf16
                const uint32_t a0 = smem_u32(st), b0 = a0 + A_BYTES;
#pragma unroll
                for (int ks = 0; ks < GEMM_KC / 16; ks++) {
                    const uint32_t ao = ks * 2 * A_LBO, bo = ks * 2 * B_LBO;
                    mma_bf16(acc, smem_desc(a0 + ao, A_LBO, 128), smem_desc(b0 + bo, B_LBO, 128), idesc,
                             (c > group_at || ks > 0) ? 1u : 0u);
                }
            } else {
                const uint32_t a_hi = smem_u32(st), a_lo = a_hi + A_BYTES;
                const uint32_t b_hi = a_hi + (LO ? 2 : 1) * A_BYTES, b_lo = b_hi + B_TILE_BYTES;
#pragma unroll
                for (int ks = 0; ks < GEMM_KC / 8; ks++) {
                    const uint32_t ao = ks * 2 * A_LBO, bo = ks * 2 * B_LBO;
                    const uint64_t dah = smem_desc(a_hi + ao, A_LBO, 128);
                    const uint64_t dbh = smem_desc(b_hi + bo, B_LBO, 128), dbl = smem_desc(b_lo + bo, B_LBO, 128);
                    mma_tf32(acc, dah, dbh, idesc, (c > group_at || ks > 0) ? 1u : 0u);
                    mma_tf32(acc, dah, dbl, idesc, 1u);
                    if constexpr (LO) mma_tf32(acc, smem_desc(a_lo + ao, A_LBO, 128), dbh, idesc, 1u);
                }
            }
            mma_commit(smem_u32(&mbar[s]));
        }
        if (!stall) last_commit = c;
    }
    if (!failed) {
        const int c = nchunks - 1;
        bool ok = mbar_wait(smem_u32(&mbar[c & 1]), (uint32_t)((c >> 1) & 1));
        failed = __syncthreads_or(!ok);
    }
    fence_after();
    // epilogue
    float* part = (float*)smem;  // [gp][NT][128] this CTA's partial sums (KS > 1; every MMA is done)
    if (!failed) {
        for (int c0 = 16 * (warp >> 2); c0 < NT; c0 += 32) {
            if (KS > 1) {
                for (int g = 0; g < gp; g++) {
                    uint32_t r[16];
                    tmem_ld16(tlane + (uint32_t)(g * NT + c0), r);
                    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
                    tmem_use(r);
#pragma unroll
                    for (int j = 0; j < 16; j++) part[(g * NT + c0 + j) * GEMM_MT + er] = __uint_as_float(r[j]);
                }
                continue;
            }
            float v[16];
            add_group(c0, v);
#pragma unroll
            for (int j = 0; j < 16; j++) {
                const int m = c0 + j;
                if (m >= M || !er_in) continue;
                if constexpr (F8) v[j] = scale_pow2(v[j], sc.qexpm[m]);
                out[(size_t)m * D] = v[j];
            }
        }
    } else {
        // give MMAs still in flight one more bounded wait before TMEM is freed
        if (last_commit >= 0 && tid == 0)
            mbar_wait(smem_u32(&mbar[last_commit & 1]), (uint32_t)((last_commit >> 1) & 1));
        if (tid == 0) atomicCAS(&sc.ctr->err, 0, DISC_ERR_TIMEOUT);
    }
    if (KS > 1) {
        // the cluster's partial sums, group after group (a CTA that failed
        // leaves what it had staged: its frame has failed); each CTA takes
        // every KS-th mask
        cluster_sync();
        const int d = d0 + row;
        unsigned at[GEMM_GROUPS];  // the row's partial sums of mask 0 (groups and KS are powers of two)
#pragma unroll
        for (int g = 0; g < GEMM_GROUPS; g++)
            if (g < groups) at[g] = dsm_map(part + (g & (gp - 1)) * NT * GEMM_MT + row, (unsigned)g >> (gp >> 1));
        for (int m = (int)rank + (int)KS * half; m < M; m += 2 * (int)KS) {
            float p[GEMM_GROUPS], v = 0.0f;
#pragma unroll
            for (int g = 0; g < GEMM_GROUPS; g++)  // all on their way before the first is added
                if (g < groups) p[g] = __int_as_float(dsm_ld32(at[g] + (unsigned)(m * GEMM_MT * 4)));
#pragma unroll
            for (int g = 0; g < GEMM_GROUPS; g++)
                if (g < groups) v = __fadd_rn(v, p[g]);
            if constexpr (F8) v = scale_pow2(v, sc.qexpm[m]);
            if (d < D) sc.Efast[(size_t)m * D + d] = v;
        }
        cluster_sync();  // no CTA leaves while another reads its sums
    }
    fence_before();
    __syncthreads();
    if (warp == 0)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(ncols) : "memory");
}

// CTAs per tile. A CTA costs its chunks and as much as four more (set-up, the
// exchange of partial sums, the result), and the CTAs run in waves: one per SM,
// or two where their shared memory lets them, which take 1.4 times as long. That
// orders what was measured, us for 1 | 4 | 8 | 12 | 16 | 32 frames: Room with 8
// CTAs per tile 15.5 | 19.3 | 28.7 | 35.9 | 44.1 | 79, with 4 19.4 | 19.4 | 25.5 |
// 25.5 | 37.8 | 59, with 2 27 | 27 | 27.5 | 29.7 | 37.4 | 54, with one 39 | 39 |
// 40 | 40 | 40 | 54; 200 masks in fp32 (a CTA per SM) with 8 25 | 44 | 79 | 99 |
// 136 | -, with 4 36 | 36 | 64 | 65 | 94 | 159, with one 77 | 77 | 78 | 79 | 79 |
// 158. An SM partition may be too small or too scattered to hold a cluster.
static int gemm_split(int NT, int precision, bool bf16_tokens, int groups, int chunks, int tiles, int B, bool clusters)
{
    int best = 1, least = 0;
    for (int KS = 1; KS <= (clusters ? groups : 1); KS *= 2) {
        const int cols = gemm_columns(NT, KS, groups);
        if (cols > 2 * GEMM_COLS || (KS > 1 && (size_t)(groups / KS) * NT * GEMM_MT * 4 + 128 > GEMM_SMEM)) continue;
        const bool two = 2 * (gemm_smem_bytes(NT, precision, bf16_tokens, KS, groups) + 128 + 1024) <= SMEM_MAX + 1024;
        const int ctas = KS * tiles * B, left = ctas % 304;
        const int waves = two ? ctas / 304 * 7 + (left > 152 ? 7 : left > 0 ? 5 : 0) : (ctas + 151) / 152 * 5;  // in fifths
        const int cost = waves * ((chunks + KS - 1) / KS + 4);
        if (KS == 1 || cost < least) {
            best = KS;
            least = cost;
        }
    }
    return best;
}

template <typename T, int PR>
static void launch_gemm_as(const FrameParams* fps, const BatchScratch& bs, int tiles, int B, int NT, int chunks,
                           bool clusters, cudaStream_t st)
{
    // How the patches are grouped depends on their number alone: two chunks to
    // a group at least, eight groups at most.
    int groups = 1;
    while (groups < GEMM_GROUPS && 4 * groups <= chunks) groups *= 2;
    const int KS = gemm_split(NT, PR, sizeof(T) == 2, groups, chunks, tiles, B, clusters);
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = KS;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    cfg.gridDim = dim3(KS, tiles, B);
    cfg.blockDim = dim3(GEMM_THREADS);
    cfg.dynamicSmemBytes = gemm_smem_bytes(NT, PR, sizeof(T) == 2, KS, groups);
    cfg.stream = st;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    cudaLaunchKernelEx(&cfg, k_pool_gemm<T, PR>, fps, bs, NT, groups);
}

int launch_pool_gemm(const FrameParams* fps, const BatchScratch& bs, int B, int P, int D, int Mmax, const bool any[2][3],
                     bool clusters, cudaStream_t st)
{
    if (Mmax <= 0) return 0;
    const int NT = std::max(16, (Mmax + 15) / 16 * 16);
    const int tiles = (D + GEMM_MT - 1) / GEMM_MT, chunks = (P + GEMM_KC - 1) / GEMM_KC;
    int n = 0;
    if (any[0][0]) { launch_gemm_as<float, DISC_FP32>(fps, bs, tiles, B, NT, chunks, clusters, st); n++; }
    if (any[1][0]) { launch_gemm_as<__nv_bfloat16, DISC_FP32>(fps, bs, tiles, B, NT, chunks, clusters, st); n++; }
    if (any[0][1]) { launch_gemm_as<float, DISC_BF16>(fps, bs, tiles, B, NT, chunks, clusters, st); n++; }
    if (any[1][1]) { launch_gemm_as<__nv_bfloat16, DISC_BF16>(fps, bs, tiles, B, NT, chunks, clusters, st); n++; }
    if (any[0][2]) { launch_gemm_as<float, DISC_FP8_E4M3>(fps, bs, tiles, B, NT, chunks, clusters, st); n++; }
    if (any[1][2]) { launch_gemm_as<__nv_bfloat16, DISC_FP8_E4M3>(fps, bs, tiles, B, NT, chunks, clusters, st); n++; }
    return n;
}

template <typename T, int PR>
static cudaError_t gemm_attr()
{
    cudaFuncAttributes a;
    const cudaError_t e = cudaFuncGetAttributes(&a, k_pool_gemm<T, PR>);
    if (e != cudaSuccess) return e;
    if (3 * GEMM_THREADS * a.numRegs <= 65536) return cudaErrorInvalidConfiguration;  // see GEMM_COLS
    return cudaFuncSetAttribute(k_pool_gemm<T, PR>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                (int)GEMM_SMEM);
}

cudaError_t set_gemm_kernel_attrs()
{
    cudaError_t e = gemm_attr<float, DISC_FP32>();
    if (e == cudaSuccess) e = gemm_attr<__nv_bfloat16, DISC_FP32>();
    if (e == cudaSuccess) e = gemm_attr<float, DISC_BF16>();
    if (e == cudaSuccess) e = gemm_attr<__nv_bfloat16, DISC_BF16>();
    if (e == cudaSuccess) e = gemm_attr<float, DISC_FP8_E4M3>();
    if (e == cudaSuccess) e = gemm_attr<__nv_bfloat16, DISC_FP8_E4M3>();
    return e;
}

}  // namespace disc

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
// A 128-row tile of D belongs to a cluster of KS CTAs, each of which takes a
// KS-th of the patches (K); with KS > 1 the partial sums meet through
// distributed shared memory, added in rank order.  One elected thread issues
// the MMAs; a two-stage shared-memory ring is recycled through mbarriers that
// tcgen05.commit arrives on.  Every wait is bounded by a global-timer limit
// after which the kernel records DISC_ERR_TIMEOUT and returns.
//
// The contraction reads each token once for ~M/2 flop per byte, so it is bound
// by how many token loads are in flight: 256 threads of 16 loads, one chunk
// ahead, two CTAs or more per SM.  With 128 threads, one CTA per SM and one
// CTA per tile whatever the batch, a 32-frame Room batch took 95 us (now 52) and a
// single frame (6 CTAs) 59 us (now 13).
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

__device__ __forceinline__ void fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }

template <typename T>
__device__ __forceinline__ float ldtok(const T* F, size_t i);
template <>
__device__ __forceinline__ float ldtok<float>(const float* F, size_t i) { return __ldg(F + i); }
template <>
__device__ __forceinline__ float ldtok<__nv_bfloat16>(const __nv_bfloat16* F, size_t i) { return __bfloat162float(F[i]); }

}  // namespace

constexpr uint32_t A_TILE_BYTES = GEMM_MT * GEMM_KC * 4;  // 16 KB (tf32); bf16 tiles take half, e4m3 a quarter
constexpr uint32_t A_LBO = (GEMM_MT / 8) * 128;           // 2048: next 16-byte K group (4 tf32 / 8 bf16 / 16 e4m3)

constexpr int GEMM_THREADS = 256;

// The bytes of one CTA: two pipeline stages and the barriers; with a cluster
// also room for the partial sums over the stages; and never less than its
// share of the SM's shared memory by tensor-memory columns (512 columns over
// 227 KB), so that the CTAs that fit an SM also fit its tensor memory and an
// allocation never waits (a cluster's CTA that waited for columns held by
// another cluster could wait for itself).
constexpr size_t SMEM_MAX = 227 * 1024;
__host__ __device__ constexpr uint32_t gemm_columns(int NT) { return NT <= 32 ? 32 : NT <= 64 ? 64 : NT <= 128 ? 128 : 256; }
// operand bytes of one stage: tf32 A hi | A lo (fp32 tokens only: bf16 ones are exact in tf32) | B hi | B lo, or
// bf16 / e4m3 A | B
__host__ __device__ constexpr uint32_t gemm_stage_bytes(int NT, int precision, bool bf16_tokens)
{
    return precision == DISC_FP8_E4M3 ? A_TILE_BYTES / 4 + (uint32_t)NT * GEMM_KC
           : precision == DISC_BF16   ? A_TILE_BYTES / 2 + (uint32_t)NT * GEMM_KC * 2
                                      : A_TILE_BYTES * (bf16_tokens ? 1 : 2) + (uint32_t)NT * GEMM_KC * 8;
}
__host__ size_t gemm_smem_bytes(int NT, int precision, bool bf16_tokens, int KS)
{
    size_t b = 2 * (size_t)gemm_stage_bytes(NT, precision, bf16_tokens);
    if (KS > 1) b = std::max(b, (size_t)NT * GEMM_MT * 4);
    return std::max(b + 128, SMEM_MAX * gemm_columns(NT) / 512);
}
static_assert(2 * gemm_stage_bytes(MAX_MASKS, DISC_FP32, false) + 128 <= SMEM_MAX, "the largest stage pair fits an SM");

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
__global__ void __launch_bounds__(GEMM_THREADS, 2) k_pool_gemm(const FrameParams* fps, BatchScratch bs, int NT)
{
    extern __shared__ __align__(1024) uint8_t smem[];
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
    const size_t used = max(2 * (size_t)STAGE, KS > 1 ? (size_t)NT * GEMM_MT * 4 : (size_t)0);
    uint64_t* mbar = (uint64_t*)(smem + used);
    uint32_t* tmem_slot = (uint32_t*)(mbar + 2);
    const uint32_t ncols = gemm_columns(NT);

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
    bool failed = false;
    int last_commit = -1;  // chunk of the most recent commit (same on all threads)
    const bool stall = g_gemm_stall != 0;  // uniform: read once
    // Thread tid stages half a row of the F^T tile: 16 tokens of row d0 + (tid
    // & 127), and its granules of the weight tile.  Those of the next chunk
    // are loaded into registers while the current chunk is staged and
    // multiplied, so loads stay in flight across the loop.
    constexpr int HALF = GEMM_KC / 2, WPRE = 2;
    const int row = tid & 127, half = tid >> 7;
    auto load_chunk = [&](int c, float (&x)[HALF]) {
        const int d = d0 + row, p0 = (cb + c) * GEMM_KC + half * HALF;
#pragma unroll
        for (int j = 0; j < HALF; j++) {
            const int p = p0 + j;
            x[j] = (d < D && p < P) ? ldtok<T>(F, (size_t)p * D + d) : 0.0f;
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
    float xn[HALF];
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

    for (int c = 0; c < nchunks && !failed; c++) {
        const int s = c & 1;
        uint8_t* st = smem + s * STAGE;
        float x[HALF];
        float4 w[WPRE];
#pragma unroll
        for (int j = 0; j < HALF; j++) x[j] = xn[j];
#pragma unroll
        for (int i = 0; i < WPRE; i++) w[i] = wn[i];
        if (c + 1 < nchunks) prefetch(c + 1);
        if (c >= 2) {
            // the MMAs of chunk c-2 read this stage: wait for their commit
            bool ok = mbar_wait(smem_u32(&mbar[s]), (uint32_t)(((c >> 1) - 1) & 1));
            if (__syncthreads_or(!ok)) { failed = true; break; }
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
            if constexpr (F8) {
                // one K step of 32 = two 16-byte core-matrix columns of e4m3
                const uint32_t a0 = smem_u32(st), b0 = a0 + A_BYTES;
                mma_e4m3(tmem, smem_desc(a0, A_LBO, 128), smem_desc(b0, B_LBO, 128), idesc, c > 0 ? 1u : 0u);
            } else if constexpr (BF) {
                // K step 16 = two 16-byte core-matrix columns of bf16
                const uint32_t a0 = smem_u32(st), b0 = a0 + A_BYTES;
#pragma unroll
                for (int ks = 0; ks < GEMM_KC / 16; ks++) {
                    const uint32_t ao = ks * 2 * A_LBO, bo = ks * 2 * B_LBO;
                    mma_bf16(tmem, smem_desc(a0 + ao, A_LBO, 128), smem_desc(b0 + bo, B_LBO, 128), idesc,
                             (c > 0 || ks > 0) ? 1u : 0u);
                }
            } else {
                const uint32_t a_hi = smem_u32(st), a_lo = a_hi + A_BYTES;
                const uint32_t b_hi = a_hi + (LO ? 2 : 1) * A_BYTES, b_lo = b_hi + B_TILE_BYTES;
#pragma unroll
                for (int ks = 0; ks < GEMM_KC / 8; ks++) {
                    const uint32_t ao = ks * 2 * A_LBO, bo = ks * 2 * B_LBO;
                    const uint64_t dah = smem_desc(a_hi + ao, A_LBO, 128);
                    const uint64_t dbh = smem_desc(b_hi + bo, B_LBO, 128), dbl = smem_desc(b_lo + bo, B_LBO, 128);
                    mma_tf32(tmem, dah, dbh, idesc, (c > 0 || ks > 0) ? 1u : 0u);
                    mma_tf32(tmem, dah, dbl, idesc, 1u);
                    if constexpr (LO) mma_tf32(tmem, smem_desc(a_lo + ao, A_LBO, 128), dbh, idesc, 1u);
                }
            }
            mma_commit(smem_u32(&mbar[s]));
        }
        if (!stall) last_commit = c;
    }
    if (!failed && nchunks > 0) {
        const int c = nchunks - 1;
        bool ok = mbar_wait(smem_u32(&mbar[c & 1]), (uint32_t)((c >> 1) & 1));
        failed = __syncthreads_or(!ok);
    }
    fence_after();
    // epilogue: warp w reads TMEM lanes 32 (w & 3) .. + 31 (rows of D), columns
    // (masks) in 16s, alternating between the two warps of the same lanes
    float* part = (float*)smem;  // [NT][128] this CTA's partial sums (KS > 1; every MMA is done)
    if (!failed) {
        const int er = (warp & 3) * 32 + lane, d = d0 + er;
        for (int c0 = 16 * (warp >> 2); c0 < NT; c0 += 32) {
            uint32_t r[16];
            if (nchunks > 0) {
                const uint32_t taddr = tmem + ((uint32_t)((warp & 3) * 32) << 16) + (uint32_t)c0;
                asm volatile(
                    "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, "
                    "[%16];"
                    : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
                      "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]),
                      "=r"(r[15])
                    : "r"(taddr));
                asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
            } else {
#pragma unroll
                for (int j = 0; j < 16; j++) r[j] = 0u;
            }
#pragma unroll
            for (int j = 0; j < 16; j++) {
                const int m = c0 + j;
                if (KS > 1) {
                    part[m * GEMM_MT + er] = __uint_as_float(r[j]);
                } else if (m < M && d < D) {
                    float v = __uint_as_float(r[j]);
                    if constexpr (F8) v = scale_pow2(v, sc.qexpm[m]);
                    sc.Efast[(size_t)m * D + d] = v;
                }
            }
        }
    } else {
        // give MMAs still in flight one more bounded wait before TMEM is freed
        if (last_commit >= 0 && tid == 0)
            mbar_wait(smem_u32(&mbar[last_commit & 1]), (uint32_t)((last_commit >> 1) & 1));
        if (tid == 0) atomicCAS(&sc.ctr->err, 0, DISC_ERR_TIMEOUT);
    }
    if (KS > 1) {
        // the cluster's partial sums, in rank order (a CTA that failed leaves
        // what it had staged: its frame has failed); each CTA takes every
        // KS-th mask
        cluster_sync();
        const int d = d0 + row;
        for (int m = (int)rank + (int)KS * half; m < M; m += 2 * (int)KS) {
            float v = 0.0f;
            for (unsigned q = 0; q < KS; q++)
                v += __int_as_float(dsm_ld32(dsm_map(part + m * GEMM_MT + row, q)));
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

template <typename T, int PR>
static void launch_gemm_as(const FrameParams* fps, const BatchScratch& bs, int tiles, int B, int NT, int KS,
                           cudaStream_t st)
{
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = KS;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    cfg.gridDim = dim3(KS, tiles, B);
    cfg.blockDim = dim3(GEMM_THREADS);
    cfg.dynamicSmemBytes = gemm_smem_bytes(NT, PR, sizeof(T) == 2, KS);
    cfg.stream = st;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    cudaLaunchKernelEx(&cfg, k_pool_gemm<T, PR>, fps, bs, NT);
}

int launch_pool_gemm(const FrameParams* fps, const BatchScratch& bs, int B, int P, int D, int Mmax, const bool any[2][3],
                     bool clusters, cudaStream_t st)
{
    if (Mmax <= 0) return 0;
    const int NT = std::max(16, (Mmax + 15) / 16 * 16);
    const int tiles = (D + GEMM_MT - 1) / GEMM_MT, chunks = (P + GEMM_KC - 1) / GEMM_KC;
    // As many CTAs per tile as leave every SM one, with two chunks each at
    // least: a single frame's 6 tiles of 18 chunks take 8 CTAs each (one CTA:
    // 59 us, all of it 18 chunks in a row); a batch that fills the SMs by
    // itself takes one, without the exchange of partial sums.  So does an SM
    // partition, which may be too small or too scattered to hold a cluster.
    int KS = 1;
    while (clusters && KS < 8 && 2 * KS * tiles * B <= 152 && 4 * KS <= chunks) KS *= 2;
    int n = 0;
    if (any[0][0]) { launch_gemm_as<float, DISC_FP32>(fps, bs, tiles, B, NT, KS, st); n++; }
    if (any[1][0]) { launch_gemm_as<__nv_bfloat16, DISC_FP32>(fps, bs, tiles, B, NT, KS, st); n++; }
    if (any[0][1]) { launch_gemm_as<float, DISC_BF16>(fps, bs, tiles, B, NT, KS, st); n++; }
    if (any[1][1]) { launch_gemm_as<__nv_bfloat16, DISC_BF16>(fps, bs, tiles, B, NT, KS, st); n++; }
    if (any[0][2]) { launch_gemm_as<float, DISC_FP8_E4M3>(fps, bs, tiles, B, NT, KS, st); n++; }
    if (any[1][2]) { launch_gemm_as<__nv_bfloat16, DISC_FP8_E4M3>(fps, bs, tiles, B, NT, KS, st); n++; }
    return n;
}

template <typename T, int PR>
static cudaError_t gemm_attr()
{
    return cudaFuncSetAttribute(k_pool_gemm<T, PR>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                (int)gemm_smem_bytes(MAX_MASKS, PR, sizeof(T) == 2, 8));
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

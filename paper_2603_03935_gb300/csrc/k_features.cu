// Feature-side kernels of the integration step (Sec. III-C), batched over the
// frames of a batch (blockIdx.z = frame slot):
//   Eq. 1 distinctiveness map, mask->patch coverage, pooling weights with the
//   image-based quality terms (S_size, S_sem, S_dist of Eq. 2), and the exact
//   D-weighted pooled embedding.  None of them touches the map, so all frames
//   of a batch run in one launch.
#include <cuda_bf16.h>

#include <algorithm>

#include "disc_common.cuh"
#include "kernels.h"

namespace disc {

// Four consecutive token values from element i on; the last `n` of a row
// (n < 4 past its end: zeros).  vec: rows and base are aligned to the four.
template <typename T>
__device__ __forceinline__ bool tok_vec(const void* F, int D)
{
    return (D & 3) == 0 && ((size_t)F & (4 * sizeof(T) - 1)) == 0;
}
__device__ __forceinline__ float4 tok4(const float* F, size_t i, int n, bool vec)
{
    if (vec) return __ldg((const float4*)(F + i));
    return make_float4(__ldg(F + i), n > 1 ? __ldg(F + i + 1) : 0.0f, n > 2 ? __ldg(F + i + 2) : 0.0f,
                       n > 3 ? __ldg(F + i + 3) : 0.0f);
}
__device__ __forceinline__ float4 tok4(const __nv_bfloat16* F, size_t i, int n, bool vec)
{
    if (vec) {
        const uint2 v = __ldg((const uint2*)(F + i));
        return make_float4(__uint_as_float(v.x << 16), __uint_as_float(v.x & 0xffff0000u),
                           __uint_as_float(v.y << 16), __uint_as_float(v.y & 0xffff0000u));
    }
    return make_float4(__bfloat162float(F[i]), n > 1 ? __bfloat162float(F[i + 1]) : 0.0f,
                       n > 2 ? __bfloat162float(F[i + 2]) : 0.0f, n > 3 ? __bfloat162float(F[i + 3]) : 0.0f);
}

__device__ __forceinline__ void set_err(FrameCounters* c, int code) { atomicCAS(&c->err, 0, code); }

// ---- Eq. 1, pass 1: column sums of the tokens, range check, mean token -----------
// A block sums TOK_ROWS patches of TOK_COLS columns: 64 threads of four
// columns each side by side, four rows of threads, every load of a thread
// issued before the first sum (16 bytes each where rows are aligned).  The
// last block of a column group to finish then takes the group's mean token,
// global embedding and share of ||g||^2, so no launch of its own waits for
// them (per group, not per frame: its fp64 divisions spread over the SMs).
// (Bound by the latency of one pass of loads.  One column per thread and 64
// patches one after the other took 30 us for a single 576x768 grid.)
constexpr int TOK_ROWS = 32, TOK_PER = TOK_ROWS / 4;

template <typename T>
__global__ void __launch_bounds__(256) k_tok_colsum(const FrameParams* fps, BatchScratch bs)
{
    __shared__ long long part[3][TOK_COLS];
    __shared__ int s_last;
    const FrameParams& fp = fps[blockIdx.z];
    if (fp.token_bf16 != (sizeof(T) == 2)) return;
    const Scratch sc = bs.frame(blockIdx.z);
    const T* F = (const T*)fp.tokens;
    const int D = fp.D, P = fp.P, tid = threadIdx.x;
    const int d0 = blockIdx.x * TOK_COLS, p0 = blockIdx.y * TOK_ROWS;
    if (d0 >= D || p0 >= P) return;  // uniform per block
    const bool vec = tok_vec<T>(F, D);
    const int d = d0 + 4 * (tid & 63), row = tid >> 6, n = D - d;
    long long s[4] = {0, 0, 0, 0};
    bool bad = false;
    if (n > 0) {
        float4 x[TOK_PER];
#pragma unroll
        for (int j = 0; j < TOK_PER; j++) {
            const int p = p0 + row + 4 * j;
            x[j] = p < P ? tok4(F, (size_t)p * D + d, n, vec) : make_float4(0.0f, 0.0f, 0.0f, 0.0f);
        }
#pragma unroll
        for (int j = 0; j < TOK_PER; j++) {
            const float m = fmaxf(fmaxf(fabsf(x[j].x), fabsf(x[j].y)), fmaxf(fabsf(x[j].z), fabsf(x[j].w)));
            // (a comparison with NaN among the four fails; fmaxf drops it)
            bad |= !(m <= TOKEN_LIMIT) || x[j].x != x[j].x || x[j].y != x[j].y || x[j].z != x[j].z || x[j].w != x[j].w;
            s[0] += fix_split<S_TOK>(x[j].x);  // |x| <= 1024 (else the frame fails)
            s[1] += fix_split<S_TOK>(x[j].y);
            s[2] += fix_split<S_TOK>(x[j].z);
            s[3] += fix_split<S_TOK>(x[j].w);
        }
    }
    if (bad) set_err(sc.ctr, DISC_ERR_RANGE);
    const int c = 4 * (tid & 63);
    if (row > 0) {
#pragma unroll
        for (int k = 0; k < 4; k++) part[row - 1][c + k] = s[k];
    }
    __syncthreads();
    if (row == 0) {
#pragma unroll
        for (int k = 0; k < 4; k++)
            if (k < n)
                atomicAdd((unsigned long long*)&sc.sumF[d + k],
                          (unsigned long long)(s[k] + part[0][c + k] + part[1][c + k] + part[2][c + k]));
        __threadfence();
    }
    __syncthreads();
    if (tid == 0) s_last = atomicAdd(&sc.tick[blockIdx.x], 1) == (P + TOK_ROWS - 1) / TOK_ROWS - 1;
    __syncthreads();
    if (!s_last) return;
    __threadfence();
    long long gg = 0;
    const int k = d0 + tid;
    if (k < D) {
        const long long sum = *(volatile long long*)&sc.sumF[k];
        const float fb = __double2float_rn(__ddiv_rn(unfix(sum, S_TOK), (double)P));
        sc.fbar[k] = fb;
        float g = fb;
        if (fp.gembed) {
            g = fp.gembed[k];
            if (!(fabsf(g) <= TOKEN_LIMIT)) set_err(sc.ctr, DISC_ERR_RANGE);
        }
        sc.gvec[k] = g;
        gg = fix32f(__fmul_rn(g, g), S_SQ);
    }
    gg = warp_sum(gg);
    if ((tid & 31) == 0 && gg) atomicAdd((unsigned long long*)sc.gg, (unsigned long long)gg);
}

// ---- Eq. 1, pass 2: residual norms, token . g, ||token||^2 (warp per patch) --
// 32 patches per block: their square roots and cosines (fp64, whose pipe this
// part has little of) are then taken a lane per patch, by two warps side by
// side.  With one lane of every patch's warp taking its own roots and scalar
// loads the kernel took 51 us per 32 Room frames, and 38 so.
constexpr int ROW_PATCHES = 32;

template <typename T>
__global__ void __launch_bounds__(32 * ROW_PATCHES) k_tok_rows(const FrameParams* fps, BatchScratch bs)
{
    __shared__ long long s_ss[ROW_PATCHES], s_dg[ROW_PATCHES], s_ff[ROW_PATCHES];
    __shared__ int s_err;
    const FrameParams& fp = fps[blockIdx.z];
    if (fp.token_bf16 != (sizeof(T) == 2)) return;
    const Scratch sc = bs.frame(blockIdx.z);
    const T* F = (const T*)fp.tokens;
    const int D = fp.D, P = fp.P;
    if ((int)blockIdx.x * ROW_PATCHES >= P) return;  // uniform per block
    if (threadIdx.x == 0) s_err = sc.ctr->err;
    __syncthreads();
    if (s_err) return;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int p = blockIdx.x * ROW_PATCHES + warp;
    if (p < P) {
        const bool vec = tok_vec<T>(F, D);
        const float4* fbar = (const float4*)sc.fbar;  // the slots' rows of [D]: read as four where D allows
        const float4* gvec = (const float4*)sc.gvec;
        const bool vd = (D & 3) == 0;
        long long ss = 0, dg = 0, ff = 0;
        float mx = 0.0f;
        auto add = [&](float f, float b, float g) {
            const float r = __fsub_rn(f, b);
            ss += fix_split<S_SQ>(__fmul_rn(r, r));  // at most 2^22
            dg += fix_split<S_SQ>(__fmul_rn(f, g));
            ff += fix_split<S_SQ>(__fmul_rn(f, f));
            mx = fmaxf(mx, fabsf(f));
        };
        for (int d0 = 4 * lane; d0 < D; d0 += 256) {  // two groups of four in flight
            float4 f[2], b[2], g[2];
#pragma unroll
            for (int j = 0; j < 2; j++) {
                const int d = d0 + 128 * j;
                const int n = D - d;
                f[j] = b[j] = g[j] = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
                if (n <= 0) continue;
                f[j] = tok4(F, (size_t)p * D + d, n, vec);
                b[j] = vd ? fbar[d >> 2] : tok4(sc.fbar, d, n, false);
                g[j] = vd ? gvec[d >> 2] : tok4(sc.gvec, d, n, false);
            }
#pragma unroll
            for (int j = 0; j < 2; j++) {
                add(f[j].x, b[j].x, g[j].x);
                add(f[j].y, b[j].y, g[j].y);
                add(f[j].z, b[j].z, g[j].z);
                add(f[j].w, b[j].w, g[j].w);
            }
        }
        ss = warp_sum(ss);
        dg = warp_sum(dg);
        ff = warp_sum(ff);
        if (lane == 0) {
            s_ss[warp] = ss;
            s_dg[warp] = dg;
            s_ff[warp] = ff;
        }
        if (fp.precision == DISC_FP8_E4M3) {
            // the token's E4M3 operand q_p = rn(f_p / 2^e) and, from its actual
            // residue, bounds of ||2^e q_p - f_p|| and ||q_p||; fp32 sums of at
            // most D/32 + 5 levels stay within (1 + 2^-10) of the exact values
            for (int o = 16; o > 0; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
            // (any e with max |f| <= 448 * 2^e serves; from -127 on, 2^-e is a
            // normal float, so the GEMM scales by one exact multiply)
            const int e = max(e4m3_exp(mx), -127);
            float se = 0.0f, sn = 0.0f;
            auto quant = [&](float f) {
                const float q = from_e4m3(to_e4m3(scale_pow2(f, -e)));
                const float r = __fsub_rn(scale_pow2(q, e), f);
                se = __fadd_rn(se, __fmul_rn(r, r));
                sn = __fadd_rn(sn, __fmul_rn(q, q));
            };
            for (int d = 4 * lane; d < D; d += 128) {
                const float4 f = tok4(F, (size_t)p * D + d, D - d, vec);
                quant(f.x);
                quant(f.y);
                quant(f.z);
                quant(f.w);
            }
            se = warp_sum(se);
            sn = warp_sum(sn);
            if (lane == 0) {
                sc.qexp[p] = e;
                sc.qmul[p] = __int_as_float((127 - e) << 23);
                sc.qerr[p] = __fmul_rn(sqrtf(se), 1.0f + 0x1p-10f);
                sc.qnrm[p] = __fmul_rn(sqrtf(sn), 1.0f + 0x1p-10f);
            }
        }
    }
    __syncthreads();
    const int q = blockIdx.x * ROW_PATCHES + lane;
    if (warp == 0) {  // residual norms
        long long nfix = 0;
        if (q < P) {
            const float n = __double2float_rn(__dsqrt_rn(unfix(s_ss[lane], S_SQ)));
            sc.nrm[q] = n;
            nfix = fix32f(n, S_NRM);
        }
        nfix = warp_sum(nfix);
        if (lane == 0 && nfix) atomicAdd((unsigned long long*)sc.nsum, (unsigned long long)nfix);
    } else if (warp == 1 && q < P) {  // ||f_p|| and cos(f_p, g)
        const long long gg = *sc.gg;
        const double rf = __dsqrt_rn(unfix(s_ff[lane], S_SQ)), rg = __dsqrt_rn(unfix(gg, S_SQ));
        sc.fnorm[q] = __double2float_rn(rf);
        sc.cosg[q] = s_ff[lane] != 0 && gg != 0
                         ? __double2float_rn(__ddiv_rn(unfix(s_dg[lane], S_SQ), __dmul_rn(rf, rg)))
                         : 0.0f;
    }
}

// ---- Eq. 1, pass 3: D_p ----------------------------------------------------------
__global__ void k_tok_finish(const FrameParams* fps, BatchScratch bs)
{
    const FrameParams& fp = fps[blockIdx.z];
    const Scratch sc = bs.frame(blockIdx.z);
    const int p = blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= fp.P || sc.ctr->err) return;
    double nbar = __ddiv_rn(unfix(*sc.nsum, S_NRM), (double)fp.P);
    sc.Dp[p] = __double2float_rn(__ddiv_rn((double)sc.nrm[p], __dadd_rn(nbar, (double)fp.eps)));
}

// ---- mask -> patch coverage: one block per patch row, shared histogram --------
// Rows v with floor(v * Ph / H) == i form the band of patch row i.  A thread
// walks a column of the band top down and adds each run of equal labels at
// once: masks are tall, so a 20-row column is a shared atomic or two, and the
// column's patch is computed once.  (A thread per pixel, with its 64-bit
// modulo and an atomic each, took 36 us for one 640x480 frame.)
__global__ void k_coverage(const FrameParams* fps, BatchScratch bs)
{
    extern __shared__ int32_t hist[];  // [M][Pw]
    const FrameParams& fp = fps[blockIdx.z];
    const Scratch sc = bs.frame(blockIdx.z);
    const int i = blockIdx.x;
    const int M = fp.M, Pw = fp.Pw, W = fp.W;
    if (M <= 0 || i >= fp.Ph) return;
    for (int j = threadIdx.x; j < M * Pw; j += blockDim.x) hist[j] = 0;
    __syncthreads();
    const int v0 = (i * fp.H + fp.Ph - 1) / fp.Ph;
    const int v1 = ((i + 1) * fp.H + fp.Ph - 1) / fp.Ph;
    constexpr int BURST = 8;  // rows loaded before the first is used
    for (int u = threadIdx.x; u < W; u += blockDim.x) {
        int32_t* h = hist + (int)(((long long)u * Pw) / W) - Pw;  // of label 1 at h[Pw]
        const uint16_t* col = fp.labels + u;
        int cur = 0, run = 0;
        for (int v = v0; v < v1; v += BURST) {
            int lab[BURST];
#pragma unroll
            for (int k = 0; k < BURST; k++) lab[k] = v + k < v1 ? (int)col[(size_t)(v + k) * W] : 0;
#pragma unroll
            for (int k = 0; k < BURST; k++) {
                if (lab[k] != cur) {
                    if (run && cur >= 1 && cur <= M) atomicAdd(&h[cur * Pw], run);
                    cur = lab[k];
                    run = 0;
                }
                run++;
            }
        }
        if (cur >= 1 && cur <= M) atomicAdd(&h[cur * Pw], run);
    }
    __syncthreads();
    for (int j = threadIdx.x; j < M * Pw; j += blockDim.x) {
        int m = j / Pw, jj = j % Pw;
        sc.cov[(size_t)m * fp.P + i * Pw + jj] = hist[j];
    }
    for (int m = threadIdx.x; m < M; m += blockDim.x) {
        int s = 0;
        for (int jj = 0; jj < Pw; jj++) s += hist[m * Pw + jj];
        if (s) atomicAdd(&sc.npix[m], s);
    }
}

template <typename T>
__device__ __forceinline__ T block_sum(T v, T* red)
{
    v = warp_sum(v);
    const int w = threadIdx.x >> 5, nw = blockDim.x >> 5;
    if ((threadIdx.x & 31) == 0) red[w] = v;
    __syncthreads();
    T s = 0;
    for (int i = 0; i < nw; i++) s += red[i];
    __syncthreads();
    return s;
}

__device__ __forceinline__ float block_max(float v, float* red)
{
    for (int o = 16; o > 0; o >>= 1) v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, o));
    const int w = threadIdx.x >> 5, nw = blockDim.x >> 5;
    if ((threadIdx.x & 31) == 0) red[w] = v;
    __syncthreads();
    float s = 0.0f;
    for (int i = 0; i < nw; i++) s = fmaxf(s, red[i]);
    __syncthreads();
    return s;
}

// FP8 precision: the weight row of mask m as E4M3 operands and the bound of
// the pooled embedding the tensor cores form from them.  Token p enters the
// GEMM as q_p = rn(f_p / 2^a_p), so its weight is scaled to w'_p = 2^a_p w_p
// (exact) and the row stored as r_p = rn(w'_p / 2^b); the GEMM returns
// 2^b sum_p r_p q_p.  Against e = sum_p w_p f_p its error is at most
//   sum_p |2^b r_p - w'_p| ||q_p||       (weight rounding)
// + sum_p w_p ||2^a_p q_p - f_p||         (token rounding)
// + g 2^b sum_p r_p ||q_p||               (accumulation)
// with g = (Kpad/32 + 2) 2^-12: an allowance of 12 bits per addition of a
// 32-deep MMA step into the accumulator, well below fp32's own rounding.
// The sum is taken in fp32 and widened by (1 + 2^-10).  Returns the bound.
__device__ float fp8_weights(const FrameParams& fp, const Scratch& sc, int m, const float* w, uint8_t* w8,
                             float* red)
{
    float mx = 0.0f;
    for (int p = threadIdx.x; p < fp.P; p += blockDim.x) mx = fmaxf(mx, scale_pow2(w[p], sc.qexp[p]));
    mx = block_max(mx, red);
    const int b = e4m3_exp(mx);
    float g1 = 0.0f, g2 = 0.0f, g3 = 0.0f;
    for (int p = threadIdx.x; p < fp.P; p += blockDim.x) {
        const float ws = scale_pow2(w[p], sc.qexp[p]);
        const uint8_t q = to_e4m3(scale_pow2(ws, -b));
        w8[p] = q;
        const float r = from_e4m3(q);
        g1 = __fadd_rn(g1, __fmul_rn(fabsf(__fsub_rn(scale_pow2(r, b), ws)), sc.qnrm[p]));
        g2 = __fadd_rn(g2, __fmul_rn(w[p], sc.qerr[p]));
        g3 = __fadd_rn(g3, __fmul_rn(r, sc.qnrm[p]));
    }
    g1 = block_sum(g1, red);
    g2 = block_sum(g2, red);
    g3 = block_sum(g3, red);
    if (threadIdx.x == 0) sc.qexpm[m] = b;
    const float gam = ldexpf((float)(fp.Kpad / 32 + 2), -12);
    return __fmul_rn(__fadd_rn(__fadd_rn(g1, g2), __fmul_rn(gam, scale_pow2(g3, b))), 1.0f + 0x1p-10f);
}

// ---- pooling weights and the image-based quality terms (one block per mask) ---
// a_p = c_p * D_p;  w_p = a_p / sum a  (sum a == 0, or the second grid's view:
// w_p = c_p / |M|);
// S_size = min(lambda |M| / (H W), 1);  S_dist = 0.5 + 0.5 * sum a / |M|;
// S_sem = clamp(sum c_p ReLU(cos(f_p, g)) / |M|, 0, 1).
__global__ void k_weights(const FrameParams* fps, BatchScratch bs)
{
    __shared__ long long red_ll[32];
    __shared__ float red_f[32];
    __shared__ int s_err;
    const FrameParams& fp = fps[blockIdx.z];
    const Scratch sc = bs.frame(blockIdx.z);
    const int m = blockIdx.x;
    if (m >= fp.M) return;  // uniform per block
    // read once for the block: the other grid's token kernels, which share the
    // frame's counters, may set it meanwhile
    if (threadIdx.x == 0) s_err = *(volatile int32_t*)&sc.ctr->err;
    __syncthreads();
    if (s_err) return;
    const int npix = sc.npix[m];
    float* w = sc.W + (size_t)m * fp.Kpad;
    float* S = sc.S + 5 * m;
    const int32_t* c = sc.cov + (size_t)m * fp.P;
    const bool fp8 = fp.precision == DISC_FP8_E4M3;
    uint8_t* w8 = sc.W8 + (size_t)m * fp.Kpad;
    if (npix < fp.min_px) {
        for (int p = threadIdx.x; p < fp.P; p += blockDim.x) {
            w[p] = 0.0f;
            if (fp8) w8[p] = 0;
        }
        if (threadIdx.x < 5) S[threadIdx.x] = 0.0f;
        if (threadIdx.x == 0) sc.Bm[m] = 0.0f;
        return;
    }
    long long A = 0, sem = 0;
    for (int p = threadIdx.x; p < fp.P; p += blockDim.x) {
        float cp = (float)c[p];
        A += fix32f(__fmul_rn(cp, sc.Dp[p]), S_A);
        float rc = sc.cosg[p] > 0.0f ? sc.cosg[p] : 0.0f;
        sem += fix32f(__fmul_rn(cp, rc), S_SEM);
    }
    A = block_sum(A, red_ll);
    sem = block_sum(sem, red_ll);
    const float Af = __double2float_rn(unfix(A, S_A));
    float bsum = 0.0f;
    for (int p = threadIdx.x; p < fp.P; p += blockDim.x) {
        float cp = (float)c[p];
        float wp = A > 0 && !fp.uniform_w ? __fdiv_rn(__fmul_rn(cp, sc.Dp[p]), Af) : __fdiv_rn(cp, (float)npix);
        w[p] = wp;
        bsum += wp * sc.fnorm[p];
    }
    bsum = block_sum(bsum, red_f);
    if (fp8) bsum = fp8_weights(fp, sc, m, w, w8, red_f);
    if (threadIdx.x == 0) {
        sc.Bm[m] = bsum;
        S[0] = fminf(__fdiv_rn(__fmul_rn(fp.lambda_size, (float)npix), (float)(fp.H * fp.W)), 1.0f);
        float Dbar = __double2float_rn(__ddiv_rn(unfix(A, S_A), (double)npix));
        S[3] = __fadd_rn(0.5f, __fmul_rn(0.5f, Dbar));
        float sm = __double2float_rn(__ddiv_rn(unfix(sem, S_SEM), (double)npix));
        S[2] = fminf(fmaxf(sm, 0.0f), 1.0f);
        S[1] = 0.0f;
        S[4] = 0.0f;
    }
}

// ---- exact D-weighted pooled embedding: e_m[d] = sum_p w_p f_p[d] -------------
// Each product is rounded to fp32 and added exactly in 2^-40 fixed point, so
// the patches can be visited in any order: the block first gathers the
// patches the mask covers, then walks only those, 64 threads of four columns
// side by side and four rows of threads that share the patches, four loads of
// each in flight (a Room frame alone: 15.6 us with a column per thread and
// one patch after the other; per frame of a 32-frame batch 1.37 -> 1.14 us).
constexpr int POOL_COLS = 256;

template <typename T>
__global__ void __launch_bounds__(256) k_pool_exact(const FrameParams* fps, BatchScratch bs)
{
    extern __shared__ unsigned char pool_smem[];
    __shared__ long long part[3][POOL_COLS];
    __shared__ int nnz, s_skip;
    const FrameParams& fp = fps[blockIdx.z];
    if (fp.token_bf16 != (sizeof(T) == 2)) return;
    const Scratch sc = bs.frame(blockIdx.z);
    int* plist = (int*)pool_smem;                 // [P]
    float* wlist = (float*)(plist + fp.P);        // [P]
    const T* F = (const T*)fp.tokens;
    const int m = blockIdx.x, D = fp.D, tid = threadIdx.x;
    if (m >= fp.M || (int)blockIdx.y * POOL_COLS >= D) return;  // uniform per block
    const bool ok = sc.npix[m] >= fp.min_px;
    if (tid == 0) {
        nnz = 0;
        s_skip = sc.ctr->err;
    }
    __syncthreads();
    if (s_skip) return;
    if (!ok) {  // an ignored mask
        const int d = blockIdx.y * POOL_COLS + tid;
        if (d < D) sc.Ecan[(size_t)m * D + d] = 0.0f;
        return;
    }
    for (int p0 = tid & ~31; p0 < fp.P; p0 += 256) {  // whole warps together: one place claimed per warp
        const int p = p0 + (tid & 31);
        const float wp = p < fp.P ? sc.W[(size_t)m * fp.Kpad + p] : 0.0f;
        const unsigned has = __ballot_sync(0xffffffffu, wp != 0.0f);
        if (!has) continue;
        int at = 0;
        if ((tid & 31) == 0) at = atomicAdd(&nnz, __popc(has));
        at = __shfl_sync(0xffffffffu, at, 0) + __popc(has & ((1u << (tid & 31)) - 1));
        if (wp != 0.0f) {
            plist[at] = p;
            wlist[at] = wp;
        }
    }
    __syncthreads();
    const int c = 4 * (tid & 63), d = blockIdx.y * POOL_COLS + c, row = tid >> 6, n = D - d;
    long long acc[4] = {0, 0, 0, 0};
    if (n > 0) {
        const bool vec = tok_vec<T>(F, D);
        const int cnt = nnz;
        auto add = [&](int k, float x) { acc[k] += fix_split<S_EMB>(x); };  // |x| <= 1024 (weights are at most 1)
        for (int i0 = row; i0 < cnt; i0 += 16) {
            float4 f[4];
            float w[4];
#pragma unroll
            for (int j = 0; j < 4; j++) {
                const int i = i0 + 4 * j;
                w[j] = i < cnt ? wlist[i] : 0.0f;
                f[j] = i < cnt ? tok4(F, (size_t)plist[i] * D + d, n, vec) : make_float4(0.0f, 0.0f, 0.0f, 0.0f);
            }
#pragma unroll
            for (int j = 0; j < 4; j++) {
                add(0, __fmul_rn(w[j], f[j].x));
                add(1, __fmul_rn(w[j], f[j].y));
                add(2, __fmul_rn(w[j], f[j].z));
                add(3, __fmul_rn(w[j], f[j].w));
            }
        }
    }
    if (row > 0) {
#pragma unroll
        for (int k = 0; k < 4; k++) part[row - 1][c + k] = acc[k];
    }
    __syncthreads();
    if (row == 0) {
#pragma unroll
        for (int k = 0; k < 4; k++)
            if (k < n)
                sc.Ecan[(size_t)m * D + d + k] =
                    unfix32f(acc[k] + part[0][c + k] + part[1][c + k] + part[2][c + k], S_EMB);
    }
}

// the sums the second grid's view accumulates per slot: column sums, pixel
// counts, ||g||^2 and the residual-norm sum (its counters are the primary's)
__global__ void k_view_clear(BatchScratch bs, int D, int MM)
{
    const Scratch sc = bs.frame(blockIdx.y);
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < max(max(D, MM), TOK_GROUPS); i += gridDim.x * blockDim.x) {
        if (i < D) sc.sumF[i] = 0;
        if (i < MM) sc.npix[i] = 0;
        if (i == 0) {
            *sc.gg = 0;
            *sc.nsum = 0;
        }
        if (i < TOK_GROUPS) sc.tick[i] = 0;
    }
}

int launch_view_clear(const BatchScratch& bs, int B, int D, int MM, cudaStream_t st)
{
    k_view_clear<<<dim3(4, B), 256, 0, st>>>(bs, D, MM);
    return 1;
}

// ---- host launchers (each returns the number of kernels it enqueued) ----------
// Batched launchers cover B frame slots; P, D, Ph, Pw and Mmax bound the grids.
int launch_token_stats(const FrameParams* fps, const BatchScratch& bs, int B, int P, int D, bool any_bf16,
                       bool any_f32, cudaStream_t st)
{
    int n = 0;
    const dim3 gcol((D + TOK_COLS - 1) / TOK_COLS, (P + TOK_ROWS - 1) / TOK_ROWS, B);
    const dim3 grow((P + ROW_PATCHES - 1) / ROW_PATCHES, 1, B);
    if (any_f32) { k_tok_colsum<float><<<gcol, 256, 0, st>>>(fps, bs); n++; }
    if (any_bf16) { k_tok_colsum<__nv_bfloat16><<<gcol, 256, 0, st>>>(fps, bs); n++; }
    if (any_f32) { k_tok_rows<float><<<grow, 32 * ROW_PATCHES, 0, st>>>(fps, bs); n++; }
    if (any_bf16) { k_tok_rows<__nv_bfloat16><<<grow, 32 * ROW_PATCHES, 0, st>>>(fps, bs); n++; }
    // a warp per block: the fp64 divisions and roots spread over the SMs
    k_tok_finish<<<dim3((P + 31) / 32, 1, B), 32, 0, st>>>(fps, bs);
    return n + 1;
}

int launch_coverage(const FrameParams* fps, const BatchScratch& bs, int B, int Ph, int Pw, int Wmax, int Mmax,
                    cudaStream_t st)
{
    if (Mmax <= 0) return 0;
    const int threads = std::min(1024, std::max(128, (Wmax + 31) / 32 * 32));  // a thread per column
    k_coverage<<<dim3(Ph, 1, B), threads, coverage_smem_bytes(Mmax, Pw), st>>>(fps, bs);
    return 1;
}

int launch_weights(const FrameParams* fps, const BatchScratch& bs, int B, int Mmax, cudaStream_t st)
{
    if (Mmax <= 0) return 0;
    k_weights<<<dim3(Mmax, 1, B), 256, 0, st>>>(fps, bs);
    return 1;
}

int launch_pool_exact(const FrameParams* fps, const BatchScratch& bs, int B, int P, int D, int Mmax, bool any_bf16,
                      bool any_f32, cudaStream_t st)
{
    if (Mmax <= 0) return 0;
    dim3 gp(Mmax, (D + POOL_COLS - 1) / POOL_COLS, B);
    size_t psm = 8 * (size_t)P;
    int n = 0;
    if (any_f32) { k_pool_exact<float><<<gp, 256, psm, st>>>(fps, bs); n++; }
    if (any_bf16) { k_pool_exact<__nv_bfloat16><<<gp, 256, psm, st>>>(fps, bs); n++; }
    return n;
}

// the [M][Pw] coverage histogram of one block
size_t coverage_smem_bytes(int max_masks, int Pw) { return sizeof(int32_t) * (size_t)max_masks * Pw; }

cudaError_t set_feature_kernel_attrs(int max_dyn_smem)
{
    cudaError_t e = cudaFuncSetAttribute(k_coverage, cudaFuncAttributeMaxDynamicSharedMemorySize, max_dyn_smem);
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(k_pool_exact<float>, cudaFuncAttributeMaxDynamicSharedMemorySize, max_dyn_smem);
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(k_pool_exact<__nv_bfloat16>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 max_dyn_smem);
    return e;
}

}  // namespace disc

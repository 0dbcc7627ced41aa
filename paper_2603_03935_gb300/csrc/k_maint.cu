// Map maintenance and query kernels: table growth, checkpoint loading,
// open-vocabulary top-k over the instance embeddings, point -> instance lookup.
#include <climits>

#include "disc_common.cuh"
#include "kernels.h"

namespace disc {

// ---- growth: re-insert every entry of the old table into a larger one ----------
__global__ void k_rehash(VoxelTable from, VoxelTable to, int* err)
{
    const unsigned long long cap = from.mask + 1;
    for (unsigned long long i = (unsigned long long)blockIdx.x * blockDim.x + threadIdx.x; i < cap;
         i += (unsigned long long)gridDim.x * blockDim.x) {
        const unsigned long long key = from.keys[i];
        if (key == EMPTY_KEY) continue;
        unsigned long long h = vt_home(key, to.mask);
        unsigned long long probes = 0;
        while (true) {
            unsigned long long prev = atomicCAS(&to.keys[h], EMPTY_KEY, key);
            if (prev == EMPTY_KEY) { to.labels[h] = from.labels[i]; break; }
            h = vt_next(h, probes + 1, to.mask);
            if (++probes > to.mask) { atomicExch(err, DISC_ERR_TABLE_FULL); return; }
        }
    }
}

// ---- queries -----------------------------------------------------------------------
// cosine of each query against every live instance; scores [nq][nid].  A block
// holds QUERY_TILE queries in shared memory (in chunks of the dimension) and
// each of its warps four instances, whose rows it reads once for all of them;
// the norms are taken beside.  Every sum keeps its order (a lane its dimensions
// in turn, then the lanes by halves), so scores do not depend on the tiling.
// Bound by instruction issue, and by the latency of the rows' loads (24 steps
// of a lane at dimension 768): each row's next two values are on their way
// while one is used, and four queries' values lie side by side for one 16-byte
// read.  4000 instances x 64 queries of 768: 122 us with a warp per (query,
// instance), which read both rows and took both norms each time; 45 us with
// the tile, 33 with the loads ahead (three or four ahead, in more registers,
// 44).
constexpr int QUERY_TILE = 8, QUERY_DIM = 1024, QUERY_INST = 4, QUERY_WARPS = 8, QUERY_AHEAD = 2;
static_assert(QUERY_TILE * QUERY_INST == 32 && QUERY_WARPS == QUERY_TILE, "a lane per product, a warp per query's norm");

__global__ void __launch_bounds__(32 * QUERY_WARPS) k_query_scores(const float* q, int nq, int D, Instances inst,
                                                                   int nid, float* scores)
{
    __shared__ float4 qs[QUERY_TILE / 4][QUERY_DIM];  // four queries side by side
    __shared__ float s_na[QUERY_TILE];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int q0 = blockIdx.y * QUERY_TILE;
    const int i0 = (blockIdx.x * QUERY_WARPS + warp) * QUERY_INST;
    const float* row[QUERY_INST];
    unsigned live = 0;  // (a dropped instance has no observations)
#pragma unroll
    for (int u = 0; u < QUERY_INST; u++) {
        const int i = i0 + u;
        if (i < nid && inst.parent[i] == i && inst.n_obs[i] > 0) live |= 1u << u;
        row[u] = inst.E + (size_t)((live >> u) & 1u ? i : 0) * D;
    }
    float dt[32] = {}, nb[QUERY_INST] = {}, na = 0.0f;  // product (u, t) in dt[u * QUERY_TILE + t]
    for (int c0 = 0; c0 < D; c0 += QUERY_DIM) {
        const int cn = min(QUERY_DIM, D - c0);
        __syncthreads();
        {  // a warp per query: its norm on the way
            const float* src = q + (size_t)min(q0 + warp, nq - 1) * D + c0;
#pragma unroll 8
            for (int d = lane; d < cn; d += 32) {
                const float a = src[d];
                ((float*)&qs[warp / 4][d])[warp % 4] = a;
                na += a * a;
            }
        }
        float ahead[QUERY_INST][QUERY_AHEAD];  // the rows' next values, on their way
#pragma unroll
        for (int k = 0; k < QUERY_AHEAD; k++)
#pragma unroll
            for (int u = 0; u < QUERY_INST; u++)
                ahead[u][k] = lane + 32 * k < cn ? row[u][c0 + lane + 32 * k] : 0.0f;
        __syncthreads();
#pragma unroll QUERY_AHEAD
        for (int d = lane; d < cn; d += 32) {
            float b[QUERY_INST];
#pragma unroll
            for (int u = 0; u < QUERY_INST; u++) {
                b[u] = ahead[u][0];
#pragma unroll
                for (int k = 0; k + 1 < QUERY_AHEAD; k++) ahead[u][k] = ahead[u][k + 1];
                const int dn = d + 32 * QUERY_AHEAD;
                ahead[u][QUERY_AHEAD - 1] = dn < cn ? row[u][c0 + dn] : 0.0f;
            }
#pragma unroll
            for (int u = 0; u < QUERY_INST; u++) nb[u] += b[u] * b[u];
#pragma unroll
            for (int h = 0; h < QUERY_TILE / 4; h++) {
                const float4 a = qs[h][d];
#pragma unroll
                for (int u = 0; u < QUERY_INST; u++) {
                    dt[u * QUERY_TILE + 4 * h] += a.x * b[u];
                    dt[u * QUERY_TILE + 4 * h + 1] += a.y * b[u];
                    dt[u * QUERY_TILE + 4 * h + 2] += a.z * b[u];
                    dt[u * QUERY_TILE + 4 * h + 3] += a.w * b[u];
                }
            }
        }
    }
    na = warp_sum(na);
    if (lane == 0) s_na[warp] = na;
    float nbl = 0.0f;  // of the lane's instance
#pragma unroll
    for (int u = 0; u < QUERY_INST; u++) {
        const float n = warp_sum(nb[u]);
        if (lane / QUERY_TILE == u) nbl = n;
    }
    // the 32 sums, one to a lane: as the lanes halve, so do the sums each holds
    // (the additions of every sum are those of a butterfly of its own)
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        const bool upper = lane & o;
#pragma unroll
        for (int i = 0; i < o; i++) {
            const float keep = upper ? dt[i + o] : dt[i], give = upper ? dt[i] : dt[i + o];
            dt[i] = keep + __shfl_xor_sync(0xffffffffu, give, o);
        }
    }
    __syncthreads();
    const int u = lane / QUERY_TILE, t = lane % QUERY_TILE;
    const float n = s_na[t];
    const float s = (n > 0.0f && nbl > 0.0f) ? dt[0] / (sqrtf(n) * sqrtf(nbl)) : 0.0f;
    if (q0 + t < nq && i0 + u < nid) scores[(size_t)(q0 + t) * nid + i0 + u] = (live >> u) & 1u ? s : -INFINITY;
}

// k best per query (score descending, id ascending).  A thread keeps the best
// of its share of the scores; each round the block takes the best of those,
// and only its owner looks its share over again.  (A pass of the block over
// all scores per round took 22 us for 10 of 4000, 11 us so.)
constexpr int TOPK_THREADS = 512;

__global__ void __launch_bounds__(TOPK_THREADS) k_query_topk(float* scores, int nid, int k, int* ids, float* out)
{
    __shared__ unsigned long long best[TOPK_THREADS / 32];
    const int qi = blockIdx.x, tid = threadIdx.x, lane = tid & 31;
    float* sc = scores + (size_t)qi * nid;
    // score and id as one number (0: no score above -inf, NaN among them):
    // the higher score first (-0 as 0), then the smaller id
    auto mine = [&]() -> unsigned long long {
        unsigned long long m = 0ull;
        for (int i = tid; i < nid; i += TOPK_THREADS) {
            const float s = sc[i];
            if (!(s > -INFINITY)) continue;
            const unsigned b = __float_as_uint(s + 0.0f);
            const unsigned key = (b & 0x80000000u) ? ~b : (b | 0x80000000u);
            m = max(m, ((unsigned long long)key << 32) | (unsigned)~i);
        }
        return m;
    };
    unsigned long long own = mine();
    for (int j = 0; j < k; j++) {
        unsigned long long m = own;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) m = max(m, __shfl_xor_sync(0xffffffffu, m, o));
        if (lane == 0) best[tid >> 5] = m;
        __syncthreads();
        m = best[0];
#pragma unroll
        for (int w = 1; w < TOPK_THREADS / 32; w++) m = max(m, best[w]);
        if (m == 0ull) {  // none left (uniform)
            for (int r = j + tid; r < k; r += TOPK_THREADS) {
                ids[(size_t)qi * k + r] = -1;
                out[(size_t)qi * k + r] = -INFINITY;
            }
            return;
        }
        if (own == m) {
            const int i = (int)~(unsigned)m;
            ids[(size_t)qi * k + j] = i;
            out[(size_t)qi * k + j] = sc[i];
            sc[i] = -INFINITY;
            own = mine();
        }
        __syncthreads();
    }
}

__global__ void k_query_points(const float* xyz, long long n, float voxel, VoxelTable vt, Instances inst, int* ids)
{
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
        unsigned long long key;
        int out = -1;
        if (voxel_key(xyz[3 * i], xyz[3 * i + 1], xyz[3 * i + 2], __fdiv_rn(1.0f, voxel), &key)) {
            unsigned long long h = vt_home(key, vt.mask);
            for (unsigned long long pr = 0; pr <= vt.mask; pr++) {
                unsigned long long kk = vt.keys[h];
                if (kk == key) {
                    const int lab = vt.labels[h];
                    out = lab >= 0 ? inst.parent[lab] : -1;  // -1: the voxel's instance was dropped
                    break;
                }
                if (kk == EMPTY_KEY) break;
                h = vt_next(h, pr + 1, vt.mask);
            }
        }
        ids[i] = out;
    }
}

// insert checkpointed voxels (keys unique, table sized beforehand)
__global__ void k_load_voxels(const unsigned long long* keys, const int* labels, long long n, VoxelTable vt, int* err)
{
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
        const unsigned long long key = keys[i];
        unsigned long long h = vt_home(key, vt.mask);
        unsigned long long probes = 0;
        while (true) {
            unsigned long long prev = atomicCAS(&vt.keys[h], EMPTY_KEY, key);
            if (prev == EMPTY_KEY || prev == key) { vt.labels[h] = labels[i]; break; }
            h = vt_next(h, probes + 1, vt.mask);
            if (++probes > vt.mask) { atomicExch(err, DISC_ERR_TABLE_FULL); return; }
        }
    }
}

// ---- host launchers ------------------------------------------------------------------
void launch_rehash(const VoxelTable& from, const VoxelTable& to, int* err, cudaStream_t st)
{
    k_rehash<<<152 * 8, 256, 0, st>>>(from, to, err);
}

void launch_query_topk(const float* q, int nq, int D, const Instances& inst, int nid, float* scores, int k,
                       int* ids, float* out, cudaStream_t st)
{
    const int per = QUERY_WARPS * QUERY_INST;
    const dim3 g((nid + per - 1) / per, (nq + QUERY_TILE - 1) / QUERY_TILE);
    k_query_scores<<<g, 32 * QUERY_WARPS, 0, st>>>(q, nq, D, inst, nid, scores);
    k_query_topk<<<nq, TOPK_THREADS, 0, st>>>(scores, nid, k, ids, out);
}

void launch_query_points(const float* xyz, long long n, float voxel, const VoxelTable& vt, const Instances& inst,
                         int* ids, cudaStream_t st)
{
    k_query_points<<<152 * 4, 256, 0, st>>>(xyz, n, voxel, vt, inst, ids);
}

void launch_load_voxels(const unsigned long long* keys, const int* labels, long long n, const VoxelTable& vt,
                        int* err, cudaStream_t st)
{
    k_load_voxels<<<152 * 4, 256, 0, st>>>(keys, labels, n, vt, err);
}

}  // namespace disc

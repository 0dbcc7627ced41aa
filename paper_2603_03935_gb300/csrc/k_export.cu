// Export of a map's voxels sorted by key (disc_map_export_voxels).
//
// The keys are distinct points of a 3D grid, and ascending key order is
// ascending (x, y, z).  So no sort is needed: inside the bounding box of the
// occupied voxels every voxel has a dense index in that order, a bitmap over
// the box marks the occupied ones, and a voxel's place in the export is the
// number of set bits before its own.  One pass over the table lists the
// occupied slots and their box; the rest works on the listed voxels and the
// bitmap (a room of 10 x 8 x 3 m at 5 cm: 2 M bits).
//
// Bound by launches and by the copy of the result to the host.  A map of
// 125,000 voxels in 2^18 slots: 0.33 ms for the call, where copying the whole
// table to the host and sorting there took 6.5 ms.
#include <climits>

#include "disc_common.cuh"
#include "kernels.h"

namespace disc {

namespace {

// dense index of a voxel in the box: x major, z minor
__device__ __forceinline__ unsigned long long box_index(const ExportScratch& es, unsigned long long key)
{
    int k[3];
    unpack_key(key, k);
    return ((unsigned long long)(k[0] - es.lo[0]) * es.ny + (unsigned long long)(k[1] - es.lo[1])) * es.nz +
           (unsigned long long)(k[2] - es.lo[2]);
}

}  // namespace

// occupied slots into es.list, their number and box into es.head (n, then
// the least and the largest coordinate per axis)
__global__ void k_export_list(VoxelTable vt, ExportScratch es)
{
    const int lane = threadIdx.x & 31;
    const unsigned long long cap = vt.mask + 1;
    int lo[3] = {INT_MAX, INT_MAX, INT_MAX}, hi[3] = {INT_MIN, INT_MIN, INT_MIN};
    for (unsigned long long i0 = ((unsigned long long)blockIdx.x * blockDim.x + threadIdx.x) & ~31ull; i0 < cap;
         i0 += (unsigned long long)gridDim.x * blockDim.x) {  // whole warps together
        const unsigned long long i = i0 + lane;
        const unsigned long long key = i < cap ? vt.keys[i] : EMPTY_KEY;
        const unsigned has = __ballot_sync(0xffffffffu, key != EMPTY_KEY);
        if (!has) continue;
        int base = 0;
        if (lane == 0) base = atomicAdd(&es.head[0], __popc(has));
        base = __shfl_sync(0xffffffffu, base, 0);
        if (key == EMPTY_KEY) continue;
        const int at = base + __popc(has & ((1u << lane) - 1));
        if (at < es.list_cap) es.list[at] = (unsigned)i;
        int k[3];
        unpack_key(key, k);
#pragma unroll
        for (int a = 0; a < 3; a++) {
            lo[a] = min(lo[a], k[a]);
            hi[a] = max(hi[a], k[a]);
        }
    }
#pragma unroll
    for (int a = 0; a < 3; a++) {
        const int l = __reduce_min_sync(0xffffffffu, lo[a]), h = __reduce_max_sync(0xffffffffu, hi[a]);
        if (lane == 0 && l <= h) {
            atomicMin(&es.head[1 + a], l);
            atomicMax(&es.head[4 + a], h);
        }
    }
}

__global__ void k_export_mark(VoxelTable vt, ExportScratch es)
{
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < es.n; i += gridDim.x * blockDim.x) {
        const unsigned long long x = box_index(es, vt.keys[es.list[i]]);
        atomicOr(&es.bits[x >> 5], 1u << (x & 31));
    }
}

// set bits of every 1024-bit group (a warp each)
__global__ void k_export_count(ExportScratch es)
{
    const int lane = threadIdx.x & 31;
    for (long long b = ((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5; b < es.groups;
         b += ((long long)gridDim.x * blockDim.x) >> 5) {
        const int c = __reduce_add_sync(0xffffffffu, __popc(es.bits[b * 32 + lane]));
        if (lane == 0) es.before[b] = c;
    }
}

// exclusive prefix of n counts, EXPORT_SPAN to a block; the spans' totals into
// totals (a second launch with one block scans those)
__global__ void __launch_bounds__(1024) k_export_scan(int* x, long long n, int* totals)
{
    __shared__ int wsum[32];
    constexpr int PER = EXPORT_SPAN / 1024;
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    const long long at = (long long)blockIdx.x * EXPORT_SPAN + (long long)tid * PER;
    int v[PER], sum = 0;
#pragma unroll
    for (int j = 0; j < PER; j++) {
        v[j] = at + j < n ? x[at + j] : 0;
        sum += v[j];
    }
    int incl = sum;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
        const int y = __shfl_up_sync(0xffffffffu, incl, d);
        if (lane >= d) incl += y;
    }
    if (lane == 31) wsum[wid] = incl;
    __syncthreads();
    int run = incl - sum;
    for (int w = 0; w < wid; w++) run += wsum[w];
#pragma unroll
    for (int j = 0; j < PER; j++) {
        if (at + j < n) x[at + j] = run;
        run += v[j];
    }
    if (totals && tid == 1023) totals[blockIdx.x] = run;
}

__global__ void k_export_place(VoxelTable vt, const int32_t* parent, int nid, ExportScratch es)
{
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < es.n; i += gridDim.x * blockDim.x) {
        const unsigned s = es.list[i];
        const unsigned long long key = vt.keys[s];
        const int lab = vt.labels[s];
        const unsigned long long x = box_index(es, key);
        const long long b = (long long)(x >> 10);
        int at = es.before[b] + es.spans[b / EXPORT_SPAN];
        const unsigned* w = es.bits + b * 32;
        const int word = (int)(x >> 5) & 31;
        for (int k = 0; k < word; k++) at += __popc(w[k]);
        at += __popc(w[word] & ((1u << (x & 31)) - 1));
        es.keys[at] = key;
        es.ids[at] = lab >= 0 && lab < nid ? parent[lab] : -1;
    }
}

// Instance table into pinned host memory, the rows handed out so far (none
// when they are more than fit)
__global__ void k_stage_table(Instances inst, const int* next_id, int D, TableStage ts)
{
    const int n = *next_id;
    const long long at = (long long)blockIdx.x * blockDim.x + threadIdx.x, step = (long long)gridDim.x * blockDim.x;
    if (at == 0) *ts.n = n;
    if (n > ts.rows) return;
    for (long long i = at; i < n; i += step) {
        ts.count[i] = inst.count[i];
        ts.parent[i] = inst.parent[i];
        ts.Q[i] = inst.Q[i];
        ts.n_obs[i] = inst.n_obs[i];
    }
    if (!ts.E) return;
    const long long words = (long long)n * D, quads = words >> 2;
    for (long long i = at; i < quads; i += step) ((float4*)ts.E)[i] = ((const float4*)inst.E)[i];
    for (long long i = 4 * quads + at; i < words; i += step) ts.E[i] = inst.E[i];
}

// ---- host launchers ------------------------------------------------------------------
void launch_export_list(const VoxelTable& vt, const ExportScratch& es, cudaStream_t st)
{
    k_export_list<<<152 * 8, 256, 0, st>>>(vt, es);
}

void launch_stage_table(const Instances& inst, const int* next_id, int D, const TableStage& ts, cudaStream_t st)
{
    const long long quads = (long long)ts.rows * (ts.E ? D / 4 + 1 : 1);
    k_stage_table<<<(int)(quads / 256 + 1 < 152 ? quads / 256 + 1 : 152), 256, 0, st>>>(inst, next_id, D, ts);
}

// es.bits zero; at most EXPORT_SPAN spans
void launch_export_place(const VoxelTable& vt, const int32_t* parent, int nid, const ExportScratch& es,
                         cudaStream_t st)
{
    const int spans = (int)((es.groups + EXPORT_SPAN - 1) / EXPORT_SPAN);
    const int nb = (es.n + 255) / 256 < 152 * 8 ? (es.n + 255) / 256 : 152 * 8;
    k_export_mark<<<nb, 256, 0, st>>>(vt, es);
    k_export_count<<<152 * 8, 256, 0, st>>>(es);
    k_export_scan<<<spans, 1024, 0, st>>>(es.before, es.groups, es.spans);
    k_export_scan<<<1, 1024, 0, st>>>(es.spans, spans, nullptr);
    k_export_place<<<nb, 256, 0, st>>>(vt, parent, nid, es);
}

}  // namespace disc

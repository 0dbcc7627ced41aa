// Geometry kernels of the integration step, batched over the frames of a batch
// (they only read the map):
//   Sec. III-A  masked depth -> world points -> voxel keys and pixel normals;
//               per-segment voxel sets V_m as records by key partition, each
//               partition gathered into distinct entries
//   Eq. 3       per voxel max(0, -r_v . n_v), summed exactly per segment
//   Sec. III-B  label of every voxel in the map as it stood at the start of
//               the batch (voxels absent then are re-probed by the serial
//               overlap kernel, which sees the inserts of earlier frames)
//   Eq. 2       Q = S_size * S_angle * S_sem * S_dist per segment
#include <algorithm>
#include <climits>

#include "disc_common.cuh"
#include "kernels.h"

namespace disc {

// The geometry kernels run beside the token kernels: they neither read nor set
// the frame's err (which those may set meanwhile) but their own geo_err.
__device__ __forceinline__ void set_err(FrameCounters* c, int code) { atomicCAS(&c->geo_err, 0, code); }

// partition of a (mask, voxel) key with hash h (its top bits; the shared
// hash of a partition and its splits take the low ones)
__device__ __forceinline__ int seg_part(unsigned long long h, int parts)
{
    return (int)__umulhi((unsigned)(h >> 32), (unsigned)parts);
}

// one more record of the frame: 256-bit stores and loads move it whole
__device__ __forceinline__ void seg_append(const Scratch& sc, int parts, unsigned long long key, long long n0,
                                           long long n1, long long n2)
{
    const int part = seg_part(mix64(key), parts);
    const int pos = atomicAdd(&sc.scur[(size_t)part * SEG_CUR], 1);
    SegRec* r = pos < SEG_REGION ? sc.srec + (size_t)part * SEG_REGION + pos
                                 : sc.srec + (size_t)sc.sparts * SEG_REGION + atomicAdd(&sc.scur[(size_t)sc.sparts * SEG_CUR], 1);
    asm volatile("st.global.v4.b64 [%0], {%1, %2, %3, %4};" ::"l"(r), "l"(key), "l"(n0), "l"(n1), "l"(n2) : "memory");
}

__device__ __forceinline__ void seg_load(const SegRec* r, unsigned long long* key, long long v[3])
{
    asm volatile("ld.global.v4.b64 {%0, %1, %2, %3}, [%4];" : "=l"(*key), "=l"(v[0]), "=l"(v[1]), "=l"(v[2]) : "l"(r));
}

// ---- slot clearing: the counters and accumulators a frame slot used last time --
__global__ void k_slot_clear(BatchScratch bs, int D, int MM)
{
    const Scratch sc = bs.frame(blockIdx.y);
    const int nc = sc.dkey ? sc.ctr->n_cells : 0;
    const int np = sc.scur ? sc.sparts + 1 : 0;
    const int n = max(max(np, nc), max(D, MM));
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
        if (i < np) sc.scur[(size_t)i * SEG_CUR] = 0;
        if (i < nc) {
            sc.dkey[sc.dlist[i]] = 0ull;
            sc.dcnt[sc.dlist[i]] = 0;
        }
        if (i < D) sc.sumF[i] = 0;
        if (i < MM) {
            sc.npix[i] = 0;
            sc.ang[i] = 0;
            sc.nvox[i] = 0;
            sc.segrep[i] = -1;
            if (sc.newcnt) sc.newcnt[i] = 0;
        }
    }
}

// counters and scalar sums of every slot (after k_slot_clear has read them)
__global__ void k_slot_reset(BatchScratch bs, int B)
{
    const int b = blockIdx.x * blockDim.x + threadIdx.x;
    if (b >= B) return;
    const Scratch sc = bs.frame(b);
    *sc.gg = 0;
    *sc.nsum = 0;
    for (int i = 0; i < TOK_GROUPS; i++) sc.tick[i] = 0;
    FrameCounters z = {};
    *sc.ctr = z;
}

// ---- back-projection (one thread per pixel) --------------------------------------
// A block covers a 32 x 16 pixel tile.  The tile and a one-pixel halo are
// loaded once into shared memory together with each position's world point,
// so neighbours' points (for the pixel normal) are read, not recomputed.
// Each valid pixel becomes a record (its (mask, voxel) key and exact normal)
// of the partition its key hashes to: one counter increment and one 32-byte
// store, no probing and nothing that the frame's next use has to clear.
// Pixels that share a voxel first add up inside a thread and between two
// neighbouring ones. Unless most of what is left is distinct (far surfaces,
// fine voxels), the tile's pixels then meet in a shared hash that sums their
// normals, and only its distinct keys become records: a voxel's records pile
// up in one partition, where k_entries sums them one after the other. The
// line is drawn on the keys themselves, a sample of one per thread counted in
// a bitmap of their hashes, so holes, sparse depth and alternating labels do
// not move it.  (Runs of equal keys along the rows, the line before, are broken
// by a missing column: Room frames with every other column of depth missing
// and 20 cm voxels took 31 us a frame, now 9, with 1 m voxels 201, now 8.)
// Back-projection and entries, us per frame, tiles merged when fewer than 1/4 |
// 1/2 | 5/8 | 3/4 | 7/8 of the sample are distinct: Room 13.3 | 12.6 | 12.7 |
// 12.8 | 13.1 (by runs 12.5); a building of 5 cm voxels 10.7 | 10.1 | 10.0 |
// 10.1 | 10.1 (9.9); Room without the depth noise 11.5 | 11.2 | 11.2 | 11.3 |
// 11.6 (11.5); alternating labels 13.6 | 13.0 | 12.6 | 12.7 | 13.1 (13.7).
// Bound by instruction issue (60 % active) and by the scattered record stores
// and counter increments, one line per lane (L1 70 % busy).  Measured on Room
// frames (640x480, 2.5 cm voxels, 8 frames per launch) in place of one global
// (segment, voxel) hash per frame with 32-byte slots, whose probes and three
// 64-bit atomics per key missed L2: 18.1 -> 7.3 us per frame, and 2.6 -> 0.3 us
// for clearing the slot; with k_entries (4.5 -> 5.3 us, they now also sum the
// pixels) 25.2 -> 12.9 us.  The partition counters lie a cache line apart: side
// by side (8 to a sector) the kernel took 28.8 us.
constexpr int BP_TX = 32, BP_TY = 16, BP_PER = 2;      // tile; pixels per thread (rows 2 ty and 2 ty + 1)
constexpr int BP_ROWS = BP_TY / BP_PER, BP_THREADS = BP_TX * BP_ROWS;
constexpr int BP_HX = BP_TX + 2, BP_HY = BP_TY + 2, BP_HALO = BP_HX * BP_HY;
constexpr int BP_SLOTS = 2 * BP_TX * BP_TY;
constexpr int BP_LOG_BITS = 11, BP_BITS = 1 << BP_LOG_BITS;

struct __align__(16) TilePoint {
    float p[3];
    int lab;   // mask label if the pixel has valid depth (and is inside the image), else 0
};

// Normal of a pixel from its neighbours to the right, left, below and above,
// as three fixed-point components; zero when it has none.
__device__ __forceinline__ void pixel_normal(const float t[3], const TilePoint& me, const TilePoint& right,
                                             const TilePoint& left, const TilePoint& below, const TilePoint& above,
                                             long long nfix[3])
{
    // image-space tangents: forward differences, backward at the mask's
    // edge; a neighbour counts if it has valid depth and the same label
    const bool fa = right.lab == me.lab, fc = below.lab == me.lab;
    if ((!fa && left.lab != me.lab) || (!fc && above.lab != me.lab)) return;
    float e1[3], e2[3], n[3];
#pragma unroll
    for (int r = 0; r < 3; r++) {
        e1[r] = fa ? __fsub_rn(right.p[r], me.p[r]) : __fsub_rn(me.p[r], left.p[r]);
        e2[r] = fc ? __fsub_rn(below.p[r], me.p[r]) : __fsub_rn(me.p[r], above.p[r]);
    }
    n[0] = __fsub_rn(__fmul_rn(e2[1], e1[2]), __fmul_rn(e2[2], e1[1]));
    n[1] = __fsub_rn(__fmul_rn(e2[2], e1[0]), __fmul_rn(e2[0], e1[2]));
    n[2] = __fsub_rn(__fmul_rn(e2[0], e1[1]), __fmul_rn(e2[1], e1[0]));
    const float l2 = __fadd_rn(__fadd_rn(__fmul_rn(n[0], n[0]), __fmul_rn(n[1], n[1])), __fmul_rn(n[2], n[2]));
    if (!(l2 > 0.0f)) return;
    const float il = __frcp_rn(__fsqrt_rn(l2));
#pragma unroll
    for (int r = 0; r < 3; r++) n[r] = __fmul_rn(n[r], il);
    // orient toward the camera
    const float vd = __fadd_rn(__fadd_rn(__fmul_rn(__fsub_rn(me.p[0], t[0]), n[0]),
                                         __fmul_rn(__fsub_rn(me.p[1], t[1]), n[1])),
                               __fmul_rn(__fsub_rn(me.p[2], t[2]), n[2]));
#pragma unroll
    for (int r = 0; r < 3; r++) nfix[r] = fix_split<S_VEC>(vd > 0.0f ? -n[r] : n[r]);
}

__global__ void __launch_bounds__(BP_THREADS) k_backproject(const FrameParams* fps, BatchScratch bs, int f0)
{
    // the tile's points, then (only in tiles that merge pixels) its hash
    constexpr size_t HASH_BYTES = (size_t)BP_SLOTS * (8 + 6 * 4);
    static_assert(sizeof(TilePoint) * BP_HALO <= HASH_BYTES, "the hash lies over the points");
    __shared__ __align__(16) unsigned char smem[HASH_BYTES];
    __shared__ unsigned short tlist[BP_TX * BP_TY];  // claimed tile slots
    __shared__ unsigned s_act[MAX_MASKS / 32];        // masks of at least min_px pixels
    __shared__ uint4 s_bits[BP_BITS / 128];          // a bit per hash value of the tile's keys
    __shared__ int s_valid, s_samples, s_dropped, s_listed, s_err;
    TilePoint* tp = (TilePoint*)smem;
    const FrameParams& fp = fps[f0 + blockIdx.z];
    const Scratch sc = bs.frame(f0 + blockIdx.z);
    const int M = fp.M, W = fp.W, H = fp.H;
    const int u0 = blockIdx.x * BP_TX - 1, v0 = blockIdx.y * BP_TY - 1;  // halo origin
    if (M <= 0 || u0 + 1 >= W || v0 + 1 >= H) return;  // uniform per block
    const int tid = threadIdx.y * BP_TX + threadIdx.x, lane = threadIdx.x;
    if (tid == 0) {
        s_valid = s_samples = s_dropped = s_listed = 0;
        s_err = sc.ctr->geo_err;
    }
    if (tid < BP_BITS / 128) s_bits[tid] = make_uint4(0, 0, 0, 0);
    {
        const unsigned act = __ballot_sync(0xffffffffu, tid < M && sc.npix[tid] >= fp.min_px);
        if (lane == 0) s_act[threadIdx.y] = act;
    }
    // The thread's two pixels and, in the first threads, one of the halo: label
    // (0 unless the depth is valid) and world point, into the tile; all loaded
    // before the first is used.
    static_assert(BP_PER == 2 && BP_HALO - BP_TX * BP_TY <= BP_THREADS, "two pixels and at most one of the halo");
    const Camera cam = fp.cam;
    const int at0 = (2 * threadIdx.y + 1) * BP_HX + threadIdx.x + 1;
    int hx = 0, hy = 0;  // the halo pixel: top and bottom rows, then left and right columns
    const bool halo = tid < BP_HALO - BP_TX * BP_TY;
    if (tid < 2 * BP_HX) {
        hx = tid < BP_HX ? tid : tid - BP_HX;
        hy = tid < BP_HX ? 0 : BP_HY - 1;
    } else {
        const int k = tid - 2 * BP_HX;
        hx = k < BP_TY ? 0 : BP_HX - 1;
        hy = 1 + (k < BP_TY ? k : k - BP_TY);
    }
    int plab[3];
    float pz[3];
#pragma unroll
    for (int j = 0; j < 3; j++) {
        const int u = u0 + (j < 2 ? (int)threadIdx.x + 1 : hx), v = v0 + (j < 2 ? 2 * (int)threadIdx.y + 1 + j : hy);
        plab[j] = 0;
        pz[j] = 0.0f;
        if ((j < 2 || halo) && (unsigned)u < (unsigned)W && (unsigned)v < (unsigned)H) {
            const int idx = v * W + u;
            plab[j] = fp.labels[idx];
            pz[j] = fp.depth[idx];
            // a DBSCAN noise pixel counts as invalid depth
            if (fp.db_min_pts > 0 && (sc.dflag[idx] & 2)) plab[j] = 0;
        }
    }
    const float z_min = fp.z_min, z_max = fp.z_max, inv_voxel = fp.inv_voxel;
    TilePoint me[BP_PER];
#pragma unroll
    for (int j = 0; j < 3; j++) {
        if (j == 2 && !halo) break;
        TilePoint t;
        t.lab = 0;
        t.p[0] = t.p[1] = t.p[2] = 0.0f;
        if (plab[j] >= 1 && plab[j] <= M && pz[j] >= z_min && pz[j] <= z_max) {
            t.lab = plab[j];
            world_point(cam, u0 + (j < 2 ? (int)threadIdx.x + 1 : hx), v0 + (j < 2 ? 2 * (int)threadIdx.y + 1 + j : hy),
                        pz[j], t.p);
        }
        if (j < 2) me[j < 2 ? j : 0] = t;
        tp[j < 2 ? at0 + j * BP_HX : hy * BP_HX + hx] = t;
    }
    __syncthreads();
    if (s_err) return;
    unsigned long long hk[BP_PER];  // 0: no record
    long long nfix[BP_PER][3];
    int nvalid = 0, ndrop = 0;
#pragma unroll
    for (int j = 0; j < BP_PER; j++) {
        const int at = at0 + j * BP_HX;
        hk[j] = 0ull;
        nfix[j][0] = nfix[j][1] = nfix[j][2] = 0;
        const int lab = me[j].lab;
        const bool active = lab > 0 && ((s_act[(lab - 1) >> 5] >> ((lab - 1) & 31)) & 1u);
        unsigned long long key = 0;
        const bool keyed = active && voxel_key(me[j].p[0], me[j].p[1], me[j].p[2], inv_voxel, &key);
        if (keyed) {
            hk[j] = ((unsigned long long)lab << 54) | key;
            pixel_normal(cam.t, me[j], tp[at + 1], tp[at - 1], j == 0 ? me[1] : tp[at + BP_HX],
                         j == 0 ? tp[at - BP_HX] : me[0], nfix[j]);
        }
        nvalid += __popc(__ballot_sync(0xffffffffu, keyed));
        ndrop += __popc(__ballot_sync(0xffffffffu, active && !keyed));
    }
    // the thread's two pixels, then the pixels of two neighbouring threads,
    // add up where they share a voxel
    if (hk[0] == hk[1]) {
        hk[1] = 0ull;
#pragma unroll
        for (int r = 0; r < 3; r++) nfix[0][r] += nfix[1][r];
    }
#pragma unroll
    for (int j = 0; j < BP_PER; j++) {
        const unsigned long long other = __shfl_xor_sync(0xffffffffu, hk[j], 1);
        const bool same = hk[j] == other && other;
        if (!__any_sync(0xffffffffu, same)) continue;
#pragma unroll
        for (int r = 0; r < 3; r++) {
            const long long v = __shfl_xor_sync(0xffffffffu, nfix[j][r], 1);
            if (same) nfix[j][r] += v;
        }
        if (same && (lane & 1)) hk[j] = 0ull;
    }
    // a sum of every thread that has one, and how many distinct keys they have
    // (nearly: a bit may stand for several)
    unsigned* bits = (unsigned*)s_bits;
    const unsigned long long sample = hk[0] ? hk[0] : hk[1];
    const int nsample = __popc(__ballot_sync(0xffffffffu, sample != 0ull));
    if (sample) {
        const unsigned b = ((unsigned)sample * 0x9E3779B1u + (unsigned)(sample >> 32) * 0x85EBCA77u) >> (32 - BP_LOG_BITS);
        atomicOr(&bits[b >> 5], 1u << (b & 31));
    }
    if (lane == 0) {
        if (nvalid) atomicAdd(&s_valid, nvalid);
        if (nsample) atomicAdd(&s_samples, nsample);
        if (ndrop) atomicAdd(&s_dropped, ndrop);
    }
    __syncthreads();
    if (tid == 0) {
        if (s_valid) atomicAdd(&sc.ctr->valid_pixels, s_valid);
        if (s_dropped) atomicAdd(&sc.ctr->dropped_pixels, s_dropped);
    }
    int distinct = 0;
#pragma unroll
    for (int i = 0; i < BP_BITS / 32; i += 32) distinct += __popc(bits[i + lane]);
    distinct = __reduce_add_sync(0xffffffffu, distinct);
    const int parts = seg_parts((long long)W * H);
    if (8 * distinct > 5 * s_samples || s_samples == 0) {  // uniform per block
#pragma unroll
        for (int j = 0; j < BP_PER; j++)
            if (hk[j]) seg_append(sc, parts, hk[j], nfix[j][0], nfix[j][1], nfix[j][2]);
        return;
    }
    // Every sum of up to four pixels adds to its (mask, voxel) slot of the
    // tile's shared hash: each 2^-32 fixed-point component v (|v| <= 2^34)
    // splits exactly into v = (v >> 16) * 2^16 + (v & 0xffff), whose parts
    // add in 32-bit integers for up to a whole tile.  (Summing a warp's equal
    // keys first with a warp match and reductions measured slower: those warp
    // instructions cost more than the shared-memory atomics they save.)  The
    // thread that claims a slot lists it.
    unsigned long long* tkey = (unsigned long long*)smem;
    unsigned* tn = (unsigned*)(tkey + BP_SLOTS);  // [6][BP_SLOTS] per component: sums of (v >> 16) and (v & 0xffff)
    for (int i = tid; i < (int)(HASH_BYTES / 16); i += BP_THREADS) ((uint4*)smem)[i] = make_uint4(0, 0, 0, 0);
    __syncthreads();
#pragma unroll
    for (int j = 0; j < BP_PER; j++) {
        if (!hk[j]) continue;
        // at most BP_TX * BP_TY distinct keys in BP_SLOTS slots
        unsigned t = (unsigned)(mix64(hk[j]) & (BP_SLOTS - 1));
        while (true) {
            const unsigned long long cur = *(volatile unsigned long long*)&tkey[t];
            if (cur == hk[j]) break;
            if (cur == 0ull) {
                const unsigned long long prev = atomicCAS(&tkey[t], 0ull, hk[j]);
                if (prev == 0ull) {
                    tlist[atomicAdd(&s_listed, 1)] = (unsigned short)t;
                    break;
                }
                if (prev == hk[j]) break;
            }
            t = (t + 1) & (BP_SLOTS - 1);
        }
#pragma unroll
        for (int r = 0; r < 3; r++) {
            const unsigned hi = (unsigned)(int)(nfix[j][r] >> 16), lo = (unsigned)(nfix[j][r] & 0xffff);
            if (hi) atomicAdd(&tn[2 * r * BP_SLOTS + t], hi);
            if (lo) atomicAdd(&tn[(2 * r + 1) * BP_SLOTS + t], lo);
        }
    }
    __syncthreads();
    for (int i = tid; i < s_listed; i += BP_THREADS) {
        const int t = tlist[i];
        long long v[3];
#pragma unroll
        for (int r = 0; r < 3; r++)
            v[r] = (long long)(int)tn[2 * r * BP_SLOTS + t] * 65536 + (long long)tn[(2 * r + 1) * BP_SLOTS + t];
        seg_append(sc, parts, tkey[t], v[0], v[1], v[2]);
    }
}

// ---- per unique (segment, voxel): its records gathered, Eq. 3 term, |V_m| ----------
// A block takes one partition of a frame's records.  Their keys meet in a
// shared hash, each slot heading a chain of its records (one shared exchange
// per record; most voxels have one to three).  Each distinct key becomes an
// entry: its thread walks the chain and sums the records' normals in
// registers (integers, so the order does not matter) and takes the S_angle
// term.  Shared-memory sums in the place of the chains (64-bit adds as two
// 32-bit words with the carry) measured 8.3 us per Room frame: 24 KB more
// shared memory per block to clear, and three to six atomics per record.
// The entries are written ordered by mask, so that the lookup's warps see few
// masks.  A partition with more distinct keys than the hash takes (skewed
// frames only) is split by further bits of the keys' hash and walked once
// per part.  Per-segment sums gather in shared memory first (one global
// atomic per block and segment): each term t (0 <= t <= 2^32 in 2^-32 fixed
// point) adds as its two 16-bit halves, whose block sums stay below 2^31.
// Without LOOKUP the labels are left to k_lookup, which runs once the previous
// batch's voxels are in (this kernel then reads no map state).
constexpr int SEG_THREADS = 256;
constexpr int SEG_SLOTS = 1024;
constexpr int SEG_MAX = 760;  // distinct keys per walk; every thread may claim one more slot before it sees the limit
static_assert(SEG_MAX + SEG_THREADS <= SEG_SLOTS - 1, "a probe always finds an empty slot");
static_assert(SEG_THREADS >= MAX_MASKS, "one thread per mask in the prefix sum");

template <bool LOOKUP>
__global__ void __launch_bounds__(SEG_THREADS) k_entries(const FrameParams* fps, BatchScratch bs,
                                                         const MapRefs* refs, int f0)
{
    __shared__ __align__(16) unsigned long long tkey[SEG_SLOTS];
    __shared__ __align__(16) int thead[SEG_SLOTS];         // last record of the slot's chain
    __shared__ int tnext[SEG_REGION];                       // the record before it in its chain
    __shared__ unsigned short tlist[SEG_MAX], trank[SEG_MAX];
    __shared__ unsigned s_hi[MAX_MASKS], s_lo[MAX_MASKS];  // per segment: sums of the terms' halves
    __shared__ int s_nv[MAX_MASKS], s_off[MAX_MASKS];
    __shared__ int s_wsum[SEG_THREADS / 32];
    __shared__ int s_n, s_over, s_base;
    const FrameParams& fp = fps[f0 + blockIdx.y];
    const Scratch sc = bs.frame(f0 + blockIdx.y);
    const int parts = seg_parts((long long)fp.W * fp.H), part = blockIdx.x, M = fp.M;
    if (M <= 0 || part >= parts) return;  // uniform per block
    const int nrec = sc.scur[(size_t)part * SEG_CUR];
    if (nrec == 0) return;
    const SegRec* region = sc.srec + (size_t)part * SEG_REGION;
    const SegRec* overflow = sc.srec + (size_t)sc.sparts * SEG_REGION;
    // past its region, a partition finds its other records in the overflow
    // list; their chain links lie in the absent-entry list, free until the
    // frame chain
    const int nall = nrec <= SEG_REGION ? nrec : SEG_REGION + sc.scur[(size_t)sc.sparts * SEG_CUR];
    int32_t* onext = sc.aent;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    int maxp = 0;
    // the walk (level, q): the keys whose `level` hash bits above the slot's equal q
    int level = 0;
    unsigned q = 0;
    while (true) {
        for (int i = tid; i < SEG_SLOTS / 2; i += SEG_THREADS) ((uint4*)tkey)[i] = make_uint4(0, 0, 0, 0);
        for (int i = tid; i < SEG_SLOTS / 4; i += SEG_THREADS) ((int4*)thead)[i] = make_int4(-1, -1, -1, -1);
        if (tid < M) {
            s_hi[tid] = 0;
            s_lo[tid] = 0;
            s_nv[tid] = 0;
        }
        if (tid == 0) s_n = s_over = 0;
        __syncthreads();
        for (int i = tid; i < nall; i += SEG_THREADS) {
            if (*(volatile int*)&s_over) break;
            const unsigned long long key = i < SEG_REGION ? region[i].key : overflow[i - SEG_REGION].key;
            const unsigned long long h = mix64(key);
            if (i >= SEG_REGION && seg_part(h, parts) != part) continue;
            if (level && (((unsigned)h >> 10) & ((1u << level) - 1)) != q) continue;
            unsigned t = (unsigned)h & (SEG_SLOTS - 1);
            int probes = 0;
            while (true) {
                const unsigned long long prev = atomicCAS(&tkey[t], 0ull, key);
                if (prev == 0ull) {
                    const int at = atomicAdd(&s_n, 1);
                    if (at < SEG_MAX) tlist[at] = (unsigned short)t;
                    else s_over = 1;
                    break;
                }
                if (prev == key) break;
                t = (t + 1) & (SEG_SLOTS - 1);
                probes++;
            }
            maxp = max(maxp, probes);
            const int prev = atomicExch(&thead[t], i);
            if (i < SEG_REGION) tnext[i] = prev;
            else onext[i - SEG_REGION] = prev;
        }
        __syncthreads();
        if (s_over) {  // too many distinct keys: the same walk on half of them
            __syncthreads();
            if (++level > 20) {
                if (tid == 0) set_err(sc.ctr, DISC_ERR_TABLE_FULL);
                return;
            }
            continue;
        }
        const int n = s_n;
        // the entries' base in the frame's list, returned while the terms compute
        int base = 0;
        if (tid == 0 && n) base = atomicAdd(&sc.ctr->n_entries, n);
        for (int i = tid; i < n; i += SEG_THREADS) {
            const int t = tlist[i];
            const unsigned long long hk = tkey[t];
            const int m = (int)(hk >> 54);
            const unsigned long long key = hk & ((1ull << 54) - 1);
            long long sum[3] = {0, 0, 0};
            for (int r = thead[t]; r >= 0;) {
                unsigned long long k_;
                long long v[3];
                seg_load(r < SEG_REGION ? region + r : overflow + (r - SEG_REGION), &k_, v);
                sum[0] += v[0];
                sum[1] += v[1];
                sum[2] += v[2];
                r = r < SEG_REGION ? tnext[r] : onext[r - SEG_REGION];
            }
            float N[3];
#pragma unroll
            for (int r = 0; r < 3; r++) N[r] = unfix32f(sum[r], S_VEC);
            float l2 = __fadd_rn(__fadd_rn(__fmul_rn(N[0], N[0]), __fmul_rn(N[1], N[1])), __fmul_rn(N[2], N[2]));
            float term = 0.0f;
            if (l2 > 0.0f) {
                float l = __fsqrt_rn(l2);
                float nv[3] = {__fdiv_rn(N[0], l), __fdiv_rn(N[1], l), __fdiv_rn(N[2], l)};
                int k[3];
                unpack_key(key, k);
                float r[3];
#pragma unroll
                for (int a = 0; a < 3; a++)
                    r[a] = __fsub_rn(__fmul_rn(__fadd_rn((float)k[a], 0.5f), fp.voxel), fp.cam.t[a]);
                float rl2 = __fadd_rn(__fadd_rn(__fmul_rn(r[0], r[0]), __fmul_rn(r[1], r[1])), __fmul_rn(r[2], r[2]));
                if (rl2 > 0.0f) {
                    float rl = __fsqrt_rn(rl2);
                    float dot = __fadd_rn(__fadd_rn(__fmul_rn(r[0], nv[0]), __fmul_rn(r[1], nv[1])),
                                          __fmul_rn(r[2], nv[2]));
                    term = __fdiv_rn(-dot, rl);
                    if (!(term > 0.0f)) term = 0.0f;
                }
            }
            const long long tf = fix_split<S_VEC>(term);
            const unsigned hi = (unsigned)(tf >> 16), lo = (unsigned)(tf & 0xffff);
            if (hi) atomicAdd(&s_hi[m - 1], hi);
            if (lo) atomicAdd(&s_lo[m - 1], lo);
            trank[i] = (unsigned short)atomicAdd(&s_nv[m - 1], 1);
        }
        if (tid == 0) s_base = base;
        __syncthreads();
        // entry positions: by mask, within a mask in any order
        {
            const int c = tid < M ? s_nv[tid] : 0;
            int incl = c;
#pragma unroll
            for (int d = 1; d < 32; d <<= 1) {
                const int y = __shfl_up_sync(0xffffffffu, incl, d);
                if (lane >= d) incl += y;
            }
            if (lane == 31) s_wsum[warp] = incl;
            __syncthreads();
            int before = s_base;
            for (int w = 0; w < warp; w++) before += s_wsum[w];
            if (tid < M) s_off[tid] = before + incl - c;
        }
        __syncthreads();
        for (int i = tid; i < n; i += SEG_THREADS) {
            const unsigned long long hk = tkey[tlist[i]];
            const int at = s_off[(int)(hk >> 54) - 1] + trank[i];
            sc.sent[at] = hk;
            if constexpr (LOOKUP) {  // label in the map at the start of the batch (-1: absent then)
                const VoxelTable& vt = refs[fp.map].vt;
                const unsigned long long key = hk & ((1ull << 54) - 1);
                unsigned long long h = vt_home(key, vt.mask);
                int lab = -1, probes = 0;
                while (true) {
                    const unsigned long long kk = vt.keys[h];
                    if (kk == key) { lab = vt.labels[h]; break; }
                    if (kk == EMPTY_KEY) break;
                    h = vt_next(h, probes + 1, vt.mask);
                    if (++probes > (int)vt.mask) { set_err(sc.ctr, DISC_ERR_TABLE_FULL); break; }
                }
                maxp = max(maxp, probes);
                sc.elab[at] = lab;
            }
        }
        if (tid < M && s_nv[tid]) {
            const long long sum = (long long)s_hi[tid] * 65536 + (long long)s_lo[tid];
            if (sum) atomicAdd((unsigned long long*)&sc.ang[tid], (unsigned long long)sum);
            atomicAdd(&sc.nvox[tid], s_nv[tid]);
        }
        // the next walk in order: up while this is its level's second half
        while (level > 0 && ((q >> (level - 1)) & 1u)) {
            level--;
            q &= ~(1u << level);
        }
        if (level == 0) break;
        q |= 1u << (level - 1);
        __syncthreads();  // the shared arrays are read above
    }
    const int pm = __reduce_max_sync(0xffffffffu, maxp);
    if (lane == 0 && pm > 0) atomicMax(&sc.ctr->max_probe, pm);
}

// ---- Eq. 2-3: S_angle = mean of the voxel terms; Q per segment -------------------
// Runs after both the token and the geometry kernels: a frame that either
// failed takes its error here, and its geometry counters, voxel counts and
// S_angle read zero.
__global__ void k_quality(const FrameParams* fps, BatchScratch bs)
{
    const FrameParams& fp = fps[blockIdx.x];
    const Scratch sc = bs.frame(blockIdx.x);
    const int err = sc.ctr->err ? sc.ctr->err : sc.ctr->geo_err;
    if (err) {
        __syncthreads();  // every thread has read both
        if (threadIdx.x == 0) {
            FrameCounters* c = sc.ctr;
            c->err = err;
            c->n_entries = c->valid_pixels = c->dropped_pixels = c->max_probe = c->denoised = 0;
        }
        for (int m = threadIdx.x; m < fp.M; m += blockDim.x) {
            sc.nvox[m] = 0;
            sc.S[5 * m + 1] = sc.S[5 * m + 4] = 0.0f;
        }
        return;
    }
    int live = 0;
    for (int m = threadIdx.x; m < fp.M; m += blockDim.x) {
        float* S = sc.S + 5 * m;
        const int nv = sc.nvox[m];
        float sa = 0.0f;
        if (nv > 0) {
            sa = __double2float_rn(__ddiv_rn(unfix(sc.ang[m], S_VEC), (double)nv));
            live++;
        }
        S[1] = sa;
        S[4] = __fmul_rn(__fmul_rn(__fmul_rn(S[0], sa), S[2]), S[3]);
    }
    live = warp_sum(live);
    if ((threadIdx.x & 31) == 0 && live) atomicAdd(&sc.ctr->live_segments, live);
}

// ---- host launchers ------------------------------------------------------------------
int launch_slot_clear(const BatchScratch& bs, int B, int D, int MM, cudaStream_t st)
{
    k_slot_clear<<<dim3(64, B), 256, 0, st>>>(bs, D, MM);
    k_slot_reset<<<(B + 127) / 128, 128, 0, st>>>(bs, B);
    return 2;
}

// launch on frames [f0, f0 + nb) of the batch
int launch_backproject(const FrameParams* fps, const BatchScratch& bs, int f0, int nb, int H, int W, cudaStream_t st)
{
    dim3 b(BP_TX, BP_ROWS), g((W + BP_TX - 1) / BP_TX, (H + BP_TY - 1) / BP_TY, nb);
    k_backproject<<<g, b, 0, st>>>(fps, bs, f0);
    return 1;
}

int launch_entries(const FrameParams* fps, const BatchScratch& bs, const MapRefs* refs, int f0, int nb, bool lookup,
                   cudaStream_t st)
{
    const dim3 g(bs.base.sparts, nb);
    if (lookup) k_entries<true><<<g, SEG_THREADS, 0, st>>>(fps, bs, refs, f0);
    else k_entries<false><<<g, SEG_THREADS, 0, st>>>(fps, bs, refs, f0);
    return 1;
}

int launch_quality(const FrameParams* fps, const BatchScratch& bs, int B, cudaStream_t st)
{
    k_quality<<<B, 256, 0, st>>>(fps, bs);
    return 1;
}

}  // namespace disc

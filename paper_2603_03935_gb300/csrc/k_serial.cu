// The stateful part of the integration step, run frame after frame in order
// (each frame sees the map its predecessors left).  Per frame, four kernels
// (captured with the rest of the batch in one CUDA graph):
//   k_overlap  Sec. III-B  exact overlap histogram ov[m][k] of every segment
//                          with the instances of the map before this frame
//   k_score    Sec. III-B  geometry gate (overlap coefficient) and cosine gate
//                          per (segment, instance) pair; fast tensor-core
//                          score, exact re-score inside its error band
//   k_union    Sec. III-B  union of segments and instances (representative =
//              Sec. III-C  smallest id), new ids, merges, Q-replacement fusion
//                          (one CTA)
//   k_apply    Sec. III-B  embedding copies, insertion of the new voxels,
//                          flattening of the parent table, cleanup
#include <cuda_bf16.h>

#include <algorithm>
#include <climits>

#include "disc_common.cuh"
#include "kernels.h"

namespace disc {

__device__ __forceinline__ void set_err(FrameCounters* c, int code) { atomicCAS(&c->err, 0, code); }

// ---- overlap histogram -----------------------------------------------------------
// Each block takes 1024 entries at a time.  Their (segment, root) pairs are
// counted in a shared-memory hash first; only the block's distinct pairs
// then update the frame's global histogram.  Voxels absent from the map go
// to the new-voxel hash with the lowest segment that contains them.
constexpr int SER_THREADS = 1024;
constexpr int OV_SLOTS = 2 * SER_THREADS;
constexpr int OV_PROBES = 64;  // longest probe of the shared pair hash

// label of a key in the voxel table, -1 if absent, from the n-th place h of
// its probe sequence on
__device__ __noinline__ int far_label(const VoxelTable& vt, unsigned long long key, unsigned long long h,
                                      unsigned long long n)
{
    for (; n <= vt.mask; n++) {
        const unsigned long long kk = vt.keys[h];
        if (kk == key) return vt.labels[h];
        if (kk == EMPTY_KEY) return -1;
        h = vt_next(h, n + 1, vt.mask);
    }
    return -1;
}

// cnt more voxels of segment-instance pair okey in the frame's pair hash
__device__ void add_pair(const Scratch& sc, const SerialScratch& ss, unsigned long long okey, int cnt = 1)
{
    unsigned long long t = mix64(okey) & ss.omask;
    for (unsigned long long pr = 0;; pr++) {
        const unsigned long long cur = ss.okeys[t];
        if (cur == okey) break;
        if (cur == EMPTY_KEY) {
            const unsigned long long prev = atomicCAS(&ss.okeys[t], EMPTY_KEY, okey);
            if (prev == EMPTY_KEY) {
                ss.olist[atomicAdd(&sc.ctr->n_pairs, 1)] = (int)t;
                break;
            }
            if (prev == okey) break;
        }
        t = (t + 1) & ss.omask;
        if (pr > ss.omask) {
            set_err(sc.ctr, DISC_ERR_TABLE_FULL);
            return;
        }
    }
    atomicAdd(&ss.ocnt[t], cnt);
}

// key of a voxel from its biased coordinates
__device__ __forceinline__ unsigned long long key_at(int x, int y, int z)
{
    return ((unsigned long long)(unsigned)x << (2 * KEY_BITS)) | ((unsigned long long)(unsigned)y << KEY_BITS) |
           (unsigned long long)(unsigned)z;
}

// label l's root among the nr distinct roots; returns how many there are now.
// (The rare steps of the neighbourhood are calls: inlined at each place they
// made the loop too long for the instruction cache.)
__device__ __noinline__ int add_root(const int32_t* parent, int l, int roots[27], int nr)
{
    const int root = parent[l];
    for (int t = 0; t < nr; t++)
        if (roots[t] == root) return nr;
    roots[nr] = root;
    return nr + 1;
}

// Neighbourhood overlap (overlap_dilation): segment voxel `key` (label lab,
// -1 if absent) overlaps each distinct instance labelling it or one of its 26
// neighbours, once: their roots into roots[27], returns how many.  The nine
// neighbours of one x offset lie in four blocks of the table, and a block's
// four voxels of one x in four consecutive slots (vt_place: x is the highest
// of the place's three bits, which the block's hash permutes by an exclusive
// or): one 32-byte load of keys and one 16-byte load of labels per block, two
// blocks at a time.  Slots are compared as they lie (the exclusive or goes
// into the expected key), and only a label other than the last three met
// is looked up.  A place that another block's voxel holds is walked past at the
// end, all lanes of a warp together.
// Bound by latency and issue.  Room frames (134,000 segment voxels, the table
// a quarter full): k_overlap 46.5 us per frame with a load of eight bytes, a
// label and a parent per neighbour, 37.6 so (14.4 without the neighbours; 7 of
// the rest for places held by other voxels, 5 for labels looked up).  All four
// blocks' loads at once, with every step inlined, took 78.
__device__ __forceinline__ int dilated_roots(const VoxelTable& vt, const int32_t* parent, unsigned long long key,
                                             int lab, int roots[27])
{
    constexpr int FIELD = (1 << KEY_BITS) - 1;
    int nr = 0, c0 = lab, c1 = lab, c2 = lab;  // labels met last
    if (lab >= 0) roots[nr++] = parent[lab];
    const int xc = (int)(key >> (2 * KEY_BITS)) & FIELD, yc = (int)(key >> KEY_BITS) & FIELD, zc = (int)key & FIELD;
    if (vt.mask < 7) {  // a table of less than a block
#pragma unroll 1
        for (int n = 0; n < 27; n++) {
            const int x = xc + n / 9 - 1, y = yc + n / 3 % 3 - 1, z = zc + n % 3 - 1;
            if (((x | y | z) & ~FIELD) != 0) continue;
            const unsigned long long nk = key_at(x, y, z);
            const int l = far_label(vt, nk, vt_home(nk, vt.mask), 0);
            if (l >= 0) nr = add_root(parent, l, roots, nr);
        }
        return nr;
    }
    // the lower blocks, and which of a block's two y (z) are one of the three:
    // bits for the lower block, then for the upper one
    const int y0 = (yc - 1) >> 1, z0 = (zc - 1) >> 1;
    const unsigned my = (yc == 0 ? 0u : (yc & 1) ? 3u : 2u) | (yc == FIELD ? 0u : (yc & 1) ? 1u : 3u) << 2;
    const unsigned mz = (zc == 0 ? 0u : (zc & 1) ? 3u : 2u) | (zc == FIELD ? 0u : (zc & 1) ? 1u : 3u) << 2;
    unsigned long long walk = 0;  // places held by another voxel: 16 (x offset) + 4 (block) + slot
#pragma unroll 1
    for (int n = 0; n < 6; n++) {
        const int x = xc + (n >> 1) - 1, by = y0 + (n & 1);
        const unsigned ym = my >> 2 * (n & 1);
        if ((x & ~FIELD) != 0 || (ym & 3) == 0) continue;
        unsigned long long kk[2][4], expect[2];
        int4 l4[2];
        unsigned want[2];
#pragma unroll
        for (int q = 0; q < 2; q++) {
            const unsigned long long h = mix64(key_at(x & ~1, 2 * by, 2 * (z0 + q)));
            const unsigned p = (unsigned)(h >> 61);
            const unsigned long long at = ((h << 3) | (((x & 1) << 2) ^ (p & 4))) & vt.mask;
            asm("ld.global.v4.b64 {%0, %1, %2, %3}, [%4];"
                : "=l"(kk[q][0]), "=l"(kk[q][1]), "=l"(kk[q][2]), "=l"(kk[q][3])
                : "l"(vt.keys + at));
            l4[q] = *(const int4*)(vt.labels + at);
            expect[q] = key_at(x, 2 * by, 2 * (z0 + q)) ^ ((unsigned long long)((p >> 1) & 1) << KEY_BITS | (p & 1));
            const unsigned zm = mz >> (2 * q) & 3;
            unsigned w = ((ym & 1) ? zm : 0) | ((ym & 2) ? zm << 2 : 0);
            if (p & 1) w = (w & 5) << 1 | (w >> 1 & 5);
            if (p & 2) w = (w & 3) << 2 | w >> 2;
            want[q] = w;  // bit s: slot s is a neighbour's place
        }
#pragma unroll
        for (int q = 0; q < 2; q++) {
            const int l[4] = {l4[q].x, l4[q].y, l4[q].z, l4[q].w};
            unsigned far = 0;
            unsigned other = 0;
#pragma unroll
            for (int s = 0; s < 4; s++) {
                const int hi = (int)(kk[q][s] >> 32);  // (negative only in an empty slot)
                const bool hit = hi == (int)(expect[q] >> 32) &&
                                 (unsigned)kk[q][s] == ((unsigned)expect[q] ^ ((unsigned)(s >> 1) << KEY_BITS | (s & 1)));
                if (!hit && hi >= 0) far |= 1u << s;
                if (hit && l[s] != c0 && l[s] != c1 && l[s] != c2) other |= 1u << s;
            }
            far &= want[q];
            other &= want[q];
            walk |= (unsigned long long)far << (16 * (n >> 1) + 8 * (n & 1) + 4 * q);
            while (other) {
                const int s = __ffs(other) - 1, x = s < 2 ? (s ? l[1] : l[0]) : s == 2 ? l[2] : l[3];
                other &= other - 1;
                if (x < 0 || x == c0) continue;
                c2 = c1;
                c1 = c0;
                c0 = x;
                nr = add_root(parent, x, roots, nr);
            }
        }
    }
    while (walk) {
        const int n = __ffsll((long long)walk) - 1;
        walk &= walk - 1;
        const int x = xc + (n >> 4) - 1, by = y0 + (n >> 3 & 1), bz = z0 + (n >> 2 & 1);
        const unsigned long long h = mix64(key_at(x & ~1, 2 * by, 2 * bz));
        const unsigned at = (n & 3) ^ ((unsigned)(h >> 61) & 3);
        const unsigned long long nk = key_at(x, 2 * by + (int)(at >> 1), 2 * bz + (int)(at & 1));
        const int l = far_label(vt, nk, vt_next(vt_place(h, nk, vt.mask), 1, vt.mask), 1);
        if (l >= 0) nr = add_root(parent, l, roots, nr);
    }
    return nr;
}

__device__ void phase_overlap(const Scratch& sc, const SerialScratch& ss, const VoxelTable& vt, const Instances& inst,
                              unsigned char* smem, bool dilate)
{
    unsigned long long* pkey = (unsigned long long*)smem;   // [OV_SLOTS]
    int* pcnt = (int*)(pkey + OV_SLOTS);                    // [OV_SLOTS]
    constexpr int OV_THREADS = SER_THREADS;
    const int ne = sc.ctr->n_entries;
    if (blockIdx.x * OV_THREADS >= ne) return;  // no entries for this block (uniform)
    for (int i = threadIdx.x; i < OV_SLOTS; i += OV_THREADS) {
        pkey[i] = EMPTY_KEY;
        pcnt[i] = 0;
    }
    __syncthreads();
    const int lane = threadIdx.x & 31;
    for (int i0 = blockIdx.x * OV_THREADS; i0 < ne; i0 += gridDim.x * OV_THREADS) {
        const int i = i0 + threadIdx.x;
        int new_slot = -1;  // slot of the new-voxel hash this thread claimed
        if (i < ne) {
            const unsigned long long hk = sc.sent[i];
            const int m = (int)(hk >> 54);
            const unsigned long long key = hk & ((1ull << 54) - 1);
            int lab = sc.elab[i];
            if (lab < 0) {
                // absent when the batch started: an earlier frame may have added it
                unsigned long long h = vt_home(key, vt.mask);
                for (int pr = 0;; pr++) {
                    const unsigned long long kk = vt.keys[h];
                    if (kk == key) { lab = vt.labels[h]; break; }
                    if (kk == EMPTY_KEY || pr > (int)vt.mask) break;
                    h = vt_next(h, pr + 1, vt.mask);
                }
            }
            // an entry adds one pair, or up to 27 (then a pair that finds no
            // place in the shared hash goes straight to the frame's)
            int roots[27];
            const int nr = dilate ? dilated_roots(vt, inst.parent, key, lab, roots)
                                  : lab >= 0 ? (roots[0] = inst.parent[lab], 1) : 0;
            for (int r = 0; r < nr; r++) {
                const unsigned long long okey = ((unsigned long long)m << 32) | (unsigned)roots[r];
                unsigned t = ((unsigned)roots[r] * 0x9E3779B1u + (unsigned)m * 0x85EBCA77u) / (unsigned)(0x100000000ull / OV_SLOTS);
                int pr = 0;
                for (; pr < OV_PROBES; pr++) {
                    const unsigned long long prev = atomicCAS(&pkey[t], EMPTY_KEY, okey);
                    if (prev == EMPTY_KEY || prev == okey) break;
                    t = (t + 1) & (OV_SLOTS - 1);
                }
                if (pr < OV_PROBES) atomicAdd(&pcnt[t], 1);
                else add_pair(sc, ss, okey);
            }
            if (lab < 0) {
                unsigned long long t = mix64(key) & ss.nmask;
                for (int pr = 0;; pr++) {
                    const unsigned long long cur = ss.nkeys[t];
                    if (cur == key) break;
                    if (cur == EMPTY_KEY) {
                        const unsigned long long prev = atomicCAS(&ss.nkeys[t], EMPTY_KEY, key);
                        if (prev == EMPTY_KEY) { new_slot = (int)t; break; }
                        if (prev == key) break;
                    }
                    t = (t + 1) & ss.nmask;
                    if (pr > (int)ss.nmask) { set_err(sc.ctr, DISC_ERR_TABLE_FULL); break; }
                }
                atomicMin(&ss.nown[t], m);
            }
        }
        // warp-aggregated append of the claimed new-voxel slots
        {
            const unsigned want = __ballot_sync(0xffffffffu, new_slot >= 0);
            int base = 0;
            if (lane == 0 && want) base = atomicAdd(&sc.ctr->n_new, __popc(want));
            base = __shfl_sync(0xffffffffu, base, 0);
            if (new_slot >= 0) ss.nlist[base + __popc(want & ((1u << lane) - 1))] = new_slot;
        }
        __syncthreads();
        // flush the block's distinct pairs, then clear them for the next pass
        for (int j0 = 0; j0 < OV_SLOTS; j0 += OV_THREADS) {
            const int j = j0 + threadIdx.x;
            const unsigned long long okey = pkey[j];
            int pair_slot = -1;
            if (okey != EMPTY_KEY) {
                unsigned long long t = mix64(okey) & ss.omask;
                for (int pr = 0;; pr++) {
                    const unsigned long long cur = ss.okeys[t];
                    if (cur == okey) break;
                    if (cur == EMPTY_KEY) {
                        const unsigned long long prev = atomicCAS(&ss.okeys[t], EMPTY_KEY, okey);
                        if (prev == EMPTY_KEY) { pair_slot = (int)t; break; }
                        if (prev == okey) break;
                    }
                    t = (t + 1) & ss.omask;
                    if (pr > (int)ss.omask) { set_err(sc.ctr, DISC_ERR_TABLE_FULL); break; }
                }
                atomicAdd(&ss.ocnt[t], pcnt[j]);
                pkey[j] = EMPTY_KEY;
                pcnt[j] = 0;
            }
            const unsigned want = __ballot_sync(0xffffffffu, pair_slot >= 0);
            int base = 0;
            if (lane == 0 && want) base = atomicAdd(&sc.ctr->n_pairs, __popc(want));
            base = __shfl_sync(0xffffffffu, base, 0);
            if (pair_slot >= 0) ss.olist[base + __popc(want & ((1u << lane) - 1))] = pair_slot;
        }
        __syncthreads();
    }
}

// ---- gates per (segment, instance) pair: one warp per pair -----------------------
// The fast cosine takes the tensor-core pooled embedding and the instance's
// scoring copy (fp32, bf16 at BF16 precision, E4M3 at FP8 precision: the
// copy's power-of-two scale cancels in the cosine); inside its error band the
// pair is re-scored exactly.
__device__ __forceinline__ unsigned bf16_pair(float lo, float hi)
{
    return (unsigned)__bfloat16_as_ushort(__float2bfloat16_rn(lo)) |
           ((unsigned)__bfloat16_as_ushort(__float2bfloat16_rn(hi)) << 16);
}

__device__ __forceinline__ float4 bf16x4_to_f32(uint2 v)
{
    return make_float4(__uint_as_float(v.x << 16), __uint_as_float(v.x & 0xffff0000u), __uint_as_float(v.y << 16),
                       __uint_as_float(v.y & 0xffff0000u));
}

// With a second grid (inst.A), the fast and exact features, their bounds and
// the instance side all come from the association features (view scratch va).
struct GateFeatures {
    const float* fast;    // [M][D] tensor-core pooled features
    const float* exact;   // [M][D] exact pooled features
    const float* bm;      // [M] sum_p w ||f_p|| (error-bound scale)
    const float* Sm;      // [cap][D] instances' scoring master
    int D;
};

__device__ __forceinline__ GateFeatures gate_features(const FrameParams& fp, const Scratch& sc, const Scratch& va,
                                                      const Instances& inst)
{
    GateFeatures g;
    g.D = scoring_dim(inst, fp.D);
    g.Sm = scoring_master(inst);
    g.fast = inst.A ? va.Efast : sc.Efast;
    g.exact = inst.A ? va.Ecan : sc.Ecan;
    g.bm = inst.A ? va.Bm : sc.Bm;
    return g;
}

// The cosine gate of segment m against instance k, by one warp (all 32 lanes
// call; every lane returns the decision).  The fast cosine takes the
// tensor-core pooled feature and the instance's scoring copy; inside its
// error band the pair is re-scored exactly (*border counts those).
__device__ bool warp_cosine_gate(const FrameParams& fp, const GateFeatures& gf, const Instances& inst, int m, int k,
                                 int* border)
{
    const int lane = threadIdx.x & 31;
    const int D = gf.D;
    const float* fast = gf.fast;
    const float* exact = gf.exact;
    const float* bm = gf.bm;
    const float* Sm = gf.Sm;
    const float* a = fast + (size_t)m * D;
    const float* b = Sm + (size_t)k * D;
    const float bmm = bm[m], erk = inst.Er ? inst.Er[k] : 0.0f;  // loaded beside the rows
    float dt = 0.0f, na = 0.0f, nb = 0.0f;
    if (inst.Eb && (D & 3) == 0) {  // bf16 scoring copy: 8-byte rows of 4
        const float4* a4 = (const float4*)a;
        const uint2* b4 = (const uint2*)(inst.Eb + (size_t)k * D);
        const int n4 = D >> 2;
        for (int d0 = 0; d0 < n4; d0 += 32 * 4) {
            float4 xs[4];
            uint2 ys[4];
#pragma unroll
            for (int j = 0; j < 4; j++) {
                const int d = d0 + j * 32 + lane;
                xs[j] = d < n4 ? a4[d] : make_float4(0.f, 0.f, 0.f, 0.f);
                ys[j] = d < n4 ? b4[d] : make_uint2(0u, 0u);
            }
#pragma unroll
            for (int j = 0; j < 4; j++) {
                const float4 x = xs[j], y = bf16x4_to_f32(ys[j]);
                dt += x.x * y.x + x.y * y.y + x.z * y.z + x.w * y.w;
                na += x.x * x.x + x.y * x.y + x.z * x.z + x.w * x.w;
                nb += y.x * y.x + y.y * y.y + y.z * y.z + y.w * y.w;
            }
        }
    } else if (inst.E8 && (D & 3) == 0) {  // E4M3 scoring copy: 4-byte words of 4
        const float4* a4 = (const float4*)a;
        const uint32_t* b4 = (const uint32_t*)(inst.E8 + (size_t)k * D);
        const int n4 = D >> 2;
        for (int d0 = 0; d0 < n4; d0 += 32 * 4) {
            float4 xs[4];
            uint32_t ys[4];
#pragma unroll
            for (int j = 0; j < 4; j++) {
                const int d = d0 + j * 32 + lane;
                xs[j] = d < n4 ? a4[d] : make_float4(0.f, 0.f, 0.f, 0.f);
                ys[j] = d < n4 ? b4[d] : 0u;
            }
#pragma unroll
            for (int j = 0; j < 4; j++) {
                const float4 x = xs[j];
                const float y0 = from_e4m3(ys[j] & 0xffu), y1 = from_e4m3((ys[j] >> 8) & 0xffu);
                const float y2 = from_e4m3((ys[j] >> 16) & 0xffu), y3 = from_e4m3(ys[j] >> 24);
                dt += x.x * y0 + x.y * y1 + x.z * y2 + x.w * y3;
                na += x.x * x.x + x.y * x.y + x.z * x.z + x.w * x.w;
                nb += y0 * y0 + y1 * y1 + y2 * y2 + y3 * y3;
            }
        }
    } else if (inst.E8) {
        const uint8_t* b8 = inst.E8 + (size_t)k * D;
        for (int d = lane; d < D; d += 32) {
            const float x = a[d], y = from_e4m3(b8[d]);
            dt += x * y;
            na += x * x;
            nb += y * y;
        }
    } else if (inst.Eb) {
        const uint16_t* bb = inst.Eb + (size_t)k * D;
        for (int d = lane; d < D; d += 32) {
            const float x = a[d], y = __uint_as_float((unsigned)bb[d] << 16);
            dt += x * y;
            na += x * x;
            nb += y * y;
        }
    } else if ((D & 3) == 0 && D <= 1024) {  // 16-byte rows of up to 1024: every load in flight at once
        const float4* a4 = (const float4*)a;
        const float4* b4 = (const float4*)b;
        const int n4 = D >> 2;
        float4 xs[8], ys[8];
#pragma unroll
        for (int j = 0; j < 8; j++) {
            const int d = j * 32 + lane;
            xs[j] = d < n4 ? a4[d] : make_float4(0.f, 0.f, 0.f, 0.f);
            ys[j] = d < n4 ? b4[d] : make_float4(0.f, 0.f, 0.f, 0.f);
        }
#pragma unroll
        for (int j = 0; j < 8; j++) {
            const float4 x = xs[j], y = ys[j];
            dt += x.x * y.x + x.y * y.y + x.z * y.z + x.w * y.w;
            na += x.x * x.x + x.y * x.y + x.z * x.z + x.w * x.w;
            nb += y.x * y.x + y.y * y.y + y.z * y.z + y.w * y.w;
        }
    } else if ((D & 3) == 0) {  // rows are 16-byte aligned: vector loads, 8 in flight per lane
        const float4* a4 = (const float4*)a;
        const float4* b4 = (const float4*)b;
        const int n4 = D >> 2;
        for (int d0 = 0; d0 < n4; d0 += 32 * 4) {
            float4 xs[4], ys[4];
#pragma unroll
            for (int j = 0; j < 4; j++) {
                const int d = d0 + j * 32 + lane;
                xs[j] = d < n4 ? a4[d] : make_float4(0.f, 0.f, 0.f, 0.f);
                ys[j] = d < n4 ? b4[d] : make_float4(0.f, 0.f, 0.f, 0.f);
            }
#pragma unroll
            for (int j = 0; j < 4; j++) {
                const float4 x = xs[j], y = ys[j];
                dt += x.x * y.x + x.y * y.y + x.z * y.z + x.w * y.w;
                na += x.x * x.x + x.y * x.y + x.z * x.z + x.w * x.w;
                nb += y.x * y.x + y.y * y.y + y.z * y.z + y.w * y.w;
            }
        }
    } else {
        for (int d = lane; d < D; d += 32) {
            const float x = a[d], y = b[d];
            dt += x * y;
            na += x * x;
            nb += y * y;
        }
    }
    dt = warp_sum(dt);
    na = warp_sum(na);
    nb = warp_sum(nb);
    bool edge;
    const float cf = (na > 0.0f && nb > 0.0f) ? dt / (sqrtf(na) * sqrtf(nb)) : 0.0f;
    // |cos(a, b') - cos(e, b)| <= 2 |a - e| / |a| + 2 |b' - b| / |b|, plus
    // the fp32 arithmetic of cf; 10 % slack on the bounds
    float band = (na > 0.0f) ? 2.2f * fp.eta * bmm / sqrtf(na) + fp.dot_err + 1e-6f : 2.0f;
    if (inst.Er) band += 2.2f * erk;
    if (fabsf(cf - fp.tau) > band) {
        edge = cf >= fp.tau;
    } else {
        // exact re-score with the exact pooled embedding
        const float* ae = exact + (size_t)m * D;
        long long xd = 0, xa = 0, xb = 0;
        if ((D & 3) == 0) {  // all of a lane's loads in flight before the exact sums
            const float4* a4 = (const float4*)ae;
            const float4* b4 = (const float4*)b;
            const int n4 = D >> 2;
            for (int d0 = 0; d0 < n4; d0 += 32 * 4) {
                float4 xs[4], ys[4];
#pragma unroll
                for (int j = 0; j < 4; j++) {
                    const int d = d0 + j * 32 + lane;
                    xs[j] = d < n4 ? a4[d] : make_float4(0.f, 0.f, 0.f, 0.f);
                    ys[j] = d < n4 ? b4[d] : make_float4(0.f, 0.f, 0.f, 0.f);
                }
#pragma unroll
                for (int j = 0; j < 4; j++) {
                    const float xv[4] = {xs[j].x, xs[j].y, xs[j].z, xs[j].w};
                    const float yv[4] = {ys[j].x, ys[j].y, ys[j].z, ys[j].w};
#pragma unroll
                    for (int c = 0; c < 4; c++) {
                        xd += fix32f(__fmul_rn(xv[c], yv[c]), S_SQ);
                        xa += fix32f(__fmul_rn(xv[c], xv[c]), S_SQ);
                        xb += fix32f(__fmul_rn(yv[c], yv[c]), S_SQ);
                    }
                }
            }
        } else {
            for (int d = lane; d < D; d += 32) {
                const float x = ae[d], y = b[d];
                xd += fix32f(__fmul_rn(x, y), S_SQ);
                xa += fix32f(__fmul_rn(x, x), S_SQ);
                xb += fix32f(__fmul_rn(y, y), S_SQ);
            }
        }
        xd = warp_sum(xd);
        xa = warp_sum(xa);
        xb = warp_sum(xb);
        float ce = 0.0f;
        if (xa != 0 && xb != 0)
            ce = __double2float_rn(__ddiv_rn(unfix(xd, S_SQ),
                                             __dmul_rn(__dsqrt_rn(unfix(xa, S_SQ)), __dsqrt_rn(unfix(xb, S_SQ)))));
        edge = ce >= fp.tau;
        (*border)++;
    }
    return edge;
}

// Warps w0, w0 + nw, ... of the launch take the pairs in turn.
__device__ void phase_score(const FrameParams& fp, const Scratch& sc, const Scratch& va, const SerialScratch& ss,
                            const Instances& inst, int w0, int nw)
{
    const int lane = threadIdx.x & 31;
    const int npairs = sc.ctr->n_pairs;
    const GateFeatures gf = gate_features(fp, sc, va, inst);
    int border = 0, scored = 0;
    for (int i = w0; i < npairs; i += nw) {
        const int slot = ss.olist[i];
        const unsigned long long okey = ss.okeys[slot];
        const int m = (int)(okey >> 32) - 1;
        const int k = (int)(okey & 0xffffffffu);
        const long long ov = ss.ocnt[slot];
        // overlap coefficient |V_m & V_k| / min(|V_m|, |V_k|) >= ov_num / ov_den
        const long long denom = min((long long)sc.nvox[m], inst.count[k]);
        if (ov * (long long)fp.ov_den < (long long)fp.ov_num * denom) continue;
        scored++;
        const bool edge = warp_cosine_gate(fp, gf, inst, m, k, &border);
        if (edge && lane == 0) {
            const int e = atomicAdd(ss.edge_n, 1);
            if (e < ss.edge_cap) {
                ss.edge_m[e] = m;
                ss.edge_k[e] = k;
            } else {
                set_err(sc.ctr, DISC_ERR_CAPACITY);
            }
        }
    }
    if (lane == 0 && border) atomicAdd(&sc.ctr->borderline, border);
    if (lane == 0 && scored) atomicAdd(&sc.ctr->n_scored, scored);
}

// ---- union, new ids, merges, fusion (one block) ------------------------------------
// Shared memory: a hash set of the frame's active roots (all overlap pairs)
// that also hands out local indices to the roots that carry an edge, and
// per-local-root arrays for the union-find and the fusion.  Every step runs
// in parallel on shared memory.  Any block of a multiple of 32 threads, at
// least MAX_MASKS, runs it.
constexpr int UNION_THREADS = 256;
constexpr int PAIR_CAP = 8192;             // distinct (segment, instance) overlaps per frame
constexpr int EDGE_ROOT_CAP = 2048;        // distinct instances with an accepted edge per frame
constexpr int EDGE_CAP = 4096;             // accepted (segment, instance) edges per frame
constexpr int UHASH = 2 * PAIR_CAP;        // hash slots at most (load <= 1/2); a frame uses
                                           // the next power of two >= 2 * its pairs
constexpr unsigned UH_EMPTY = 0xffffffffu;
constexpr unsigned UH_UNUSED = 0xffffffffu;
constexpr unsigned UH_LOCAL = 0x80000000u;
constexpr size_t UNION_SMEM = (size_t)UHASH * 8 + (size_t)EDGE_ROOT_CAP * 24 + (size_t)EDGE_CAP * 8;

// slot of root id k in the union's root hash (32-bit multiplicative mix)
__device__ __forceinline__ unsigned uhash(unsigned k, unsigned mask)
{
    unsigned h = k * 0x9E3779B1u;
    h ^= h >> 15;
    return h & mask;
}

// float <-> unsigned key with the same order (for atomicMax over floats)
__device__ __forceinline__ unsigned f2key(float x)
{
    const unsigned b = __float_as_uint(x);
    return (b & 0x80000000u) ? ~b : (b | 0x80000000u);
}
__device__ __forceinline__ float key2f(unsigned k)
{
    return __uint_as_float((k & 0x80000000u) ? (k & 0x7fffffffu) : ~k);
}

__device__ __forceinline__ int uf_find(const int* uf, int x)
{
    while (true) {
        const int p = ((volatile const int*)uf)[x];
        if (p == x) return x;
        x = p;
    }
}

__device__ __forceinline__ int local_of(const unsigned* hkey, const unsigned* hval, unsigned mask, unsigned k)
{
    unsigned h = uhash(k, mask);
    while (hkey[h] != k) h = (h + 1) & mask;
    return (int)(hval[h] & ~UH_LOCAL);
}

// The arrays of a union region (UNION_SMEM bytes): the root hash, the
// per-local-root arrays and the edge arrays.
struct UnionRegion {
    unsigned* hkey;      // [UHASH] root id
    unsigned* hval;      // [UHASH] claimant edge, then UH_LOCAL | local index
    int* gid;            // [EDGE_ROOT_CAP] local -> instance id
    int* uf;             // union-find over local indices
    int* best_src;       // fusion winner per component
    float* best_q;
    float* qloc;         // Q of the local roots
    int* oloc;           // observations of the local roots
    int* em;             // [EDGE_CAP] edge segment
    int* ek;             // [EDGE_CAP] edge instance id
    __device__ __forceinline__ explicit UnionRegion(unsigned char* base)
    {
        hkey = (unsigned*)base;
        hval = hkey + UHASH;
        gid = (int*)(hval + UHASH);
        uf = gid + EDGE_ROOT_CAP;
        best_src = uf + EDGE_ROOT_CAP;
        best_q = (float*)(best_src + EDGE_ROOT_CAP);
        qloc = best_q + EDGE_ROOT_CAP;
        oloc = (int*)(qloc + EDGE_ROOT_CAP);
        em = oloc + EDGE_ROOT_CAP;
        ek = em + EDGE_CAP;
    }
};

// The frame's npairs overlap pairs give their roots through pair_root(i);
// its nedge accepted edges are in ss.edge_m/k.  union_smem: a union region in
// shared or global memory (the fusion step lays EDGE_ROOT_CAP 64-bit words
// over em).  Past a capacity the frame fails with DISC_ERR_CAPACITY.
template <class PairRoot>
__device__ void union_frame(const FrameParams& fp, const Scratch& sc, const SerialScratch& ss, const Instances& inst,
                            int* next_id, unsigned char* union_smem, int npairs, int nedge, PairRoot pair_root)
{
    const UnionRegion U(union_smem);
    unsigned* hkey = U.hkey;
    unsigned* hval = U.hval;
    int* gid = U.gid;
    int* uf = U.uf;
    int* best_src = U.best_src;
    float* best_q = U.best_q;
    float* qloc = U.qloc;
    int* oloc = U.oloc;
    int* em = U.em;
    int* ek = U.ek;
    __shared__ int anchor[MAX_MASKS];                 // smallest local root of a segment's edges
    __shared__ int srep[MAX_MASKS];
    __shared__ int snv[MAX_MASKS];
    __shared__ float sq[MAX_MASKS];
    __shared__ int s_nroots, s_nloc, s_merges, s_new, s_ncopy, s_next;
    const int tid = threadIdx.x, NT = blockDim.x;
    FrameCounters* ctr = sc.ctr;
    const int M = fp.M;
    if (2u * (unsigned)npairs > (unsigned)UHASH || nedge > EDGE_CAP) {
        if (tid == 0) set_err(ctr, DISC_ERR_CAPACITY);
        return;
    }
    unsigned hsize = 64;
    while (hsize < 2u * (unsigned)npairs) hsize <<= 1;
    const unsigned hm = hsize - 1;
    // the edges, once, into shared memory (segment, root)
    for (int e = tid; e < nedge; e += NT) {
        em[e] = ss.edge_m[e];
        ek[e] = ss.edge_k[e];
    }
    for (int i = tid; i < (int)hsize; i += NT) {
        hkey[i] = UH_EMPTY;
        hval[i] = UH_UNUSED;
    }
    for (int m = tid; m < M; m += NT) {
        anchor[m] = INT_MAX;
        snv[m] = sc.nvox[m];
        sq[m] = sc.S[5 * m + 4];
    }
    if (tid == 0) {
        s_nroots = 0;
        s_nloc = 0;
        s_merges = 0;
        s_new = 0;
        s_ncopy = 0;
        s_next = *next_id;
    }
    __syncthreads();
    // (1) active set: distinct roots of all overlap pairs (counted per warp)
    {
        int mine = 0;
        for (int i = tid; i < npairs; i += NT) {
            const unsigned k = pair_root(i);
            unsigned h = uhash(k, hm);
            while (true) {
                const unsigned cur = hkey[h];
                if (cur == k) break;
                if (cur == UH_EMPTY) {
                    const unsigned prev = atomicCAS(&hkey[h], UH_EMPTY, k);
                    if (prev == UH_EMPTY) { mine++; break; }
                    if (prev == k) break;
                }
                h = (h + 1) & hm;
            }
        }
        mine = warp_sum(mine);
        if ((tid & 31) == 0 && mine) atomicAdd(&s_nroots, mine);
    }
    __syncthreads();
    // (2) local indices for the roots that carry an edge: the first edge to
    //     claim a root's slot assigns the index
    for (int e = tid; e < nedge; e += NT) {
        const unsigned k = (unsigned)ek[e];
        unsigned h = uhash(k, hm);
        while (hkey[h] != k) h = (h + 1) & hm;
        atomicCAS(&hval[h], UH_UNUSED, (unsigned)e);
    }
    __syncthreads();
    for (int e = tid; e < nedge; e += NT) {
        const unsigned k = (unsigned)ek[e];
        unsigned h = uhash(k, hm);
        while (hkey[h] != k) h = (h + 1) & hm;
        if (hval[h] == (unsigned)e) {
            const int x = atomicAdd(&s_nloc, 1);
            if (x < EDGE_ROOT_CAP) {
                gid[x] = (int)k;
                uf[x] = x;
                qloc[x] = inst.Q[k];
                oloc[x] = inst.n_obs[k];
            }
            hval[h] = UH_LOCAL | (unsigned)x;
        }
    }
    __syncthreads();
    const int nloc = s_nloc;
    if (nloc > EDGE_ROOT_CAP) {
        if (tid == 0) set_err(ctr, DISC_ERR_CAPACITY);
        return;
    }
    // (3) union of the instances one segment joins: every edge hooks its
    //     root onto the segment's anchor; a hook always links the root with
    //     the larger instance id under the smaller one, so each set's root is
    //     its smallest instance id
    for (int e = tid; e < nedge; e += NT) atomicMin(&anchor[em[e]], local_of(hkey, hval, hm, (unsigned)ek[e]));
    __syncthreads();
    for (int e = tid; e < nedge; e += NT) {
        int x = local_of(hkey, hval, hm, (unsigned)ek[e]);
        int y = anchor[em[e]];
        while (true) {
            x = uf_find(uf, x);
            y = uf_find(uf, y);
            if (x == y) break;
            const int lo = gid[x] < gid[y] ? x : y, hi = lo == x ? y : x;
            if (atomicCAS(&uf[hi], hi, lo) == hi) break;
        }
    }
    __syncthreads();
    for (int x = tid; x < nloc; x += NT) uf[x] = uf_find(uf, x);  // stores only roots
    __syncthreads();
    for (int m = tid; m < M; m += NT) srep[m] = anchor[m] != INT_MAX ? gid[uf[anchor[m]]] : -1;
    __syncthreads();
    // (4) new instances for live segments without an edge, in mask order:
    //     the id of mask m is next_id plus the number of such masks before it
    //     (a block-wide exclusive scan; M <= MAX_MASKS <= NT)
    {
        __shared__ int wtot[32];
        const int lane = tid & 31, wid = tid >> 5;
        const bool want = tid < M && snv[tid] > 0 && srep[tid] < 0;
        const unsigned bal = __ballot_sync(0xffffffffu, want);
        if (lane == 0) wtot[wid] = __popc(bal);
        __syncthreads();
        int before = __popc(bal & ((1u << lane) - 1)), total = 0;
        for (int w = 0; w < (NT >> 5); w++) {
            before += w < wid ? wtot[w] : 0;
            total += wtot[w];
        }
        const int base = s_next;
        if (base + total > inst.cap) {  // uniform: every thread summed the same counts
            if (tid == 0) set_err(ctr, DISC_ERR_CAPACITY);
            return;
        }
        if (want) {
            const int id = base + before, m = tid;
            srep[m] = id;
            inst.parent[id] = id;
            inst.count[id] = 0;
            inst.Q[id] = sq[m];
            inst.n_obs[id] = 1;
            ss.copy_dst[before] = id;
            ss.copy_src[before] = -(m + 1);
        }
        __syncthreads();  // every thread has read s_next
        if (tid == 0) {
            *next_id = base + total;
            s_next = base + total;
            s_new = total;
            s_ncopy = total;
        }
    }
    __syncthreads();
    for (int m = tid; m < M; m += NT) sc.segrep[m] = srep[m];
    // (5) fusion per component: the candidates in the order (members by
    //     ascending id, then segments by ascending mask) keep the first one
    //     whose Q is the component's maximum (strict '>' while scanning):
    //     the component's maximum (an atomic max on order-preserving keys),
    //     then the smallest member id with that Q, else the smallest mask;
    //     the stored Q is the winner's own value.  The edge arrays are no
    //     longer needed and hold part of the per-root scratch.
    unsigned* qmax = (unsigned*)best_q;                              // [nloc] key of the max Q
    int* obs = best_src;                                             // [nloc] observations
    unsigned long long* src_inst = (unsigned long long*)em;          // [nloc] (id << 32 | local) at the max
    int* src_seg = ek;                                               // [nloc] smallest mask at the max
    for (int r = tid; r < nloc; r += NT) {
        qmax[r] = 0u;
        obs[r] = 0;
        src_inst[r] = ~0ull;
        src_seg[r] = INT_MAX;
    }
    // the local root of each segment that joined a component
    for (int m = tid; m < M; m += NT) snv[m] = anchor[m] != INT_MAX ? uf[anchor[m]] : -1;
    __syncthreads();
    for (int x = tid; x < nloc; x += NT) {
        atomicMax(&qmax[uf[x]], f2key(qloc[x]));
        atomicAdd(&obs[uf[x]], oloc[x]);
    }
    for (int m = tid; m < M; m += NT)
        if (snv[m] >= 0) {
            atomicMax(&qmax[snv[m]], f2key(sq[m]));
            atomicAdd(&obs[snv[m]], 1);
        }
    __syncthreads();
    for (int x = tid; x < nloc; x += NT)
        if (qloc[x] == key2f(qmax[uf[x]]))
            atomicMin(&src_inst[uf[x]], ((unsigned long long)(unsigned)gid[x] << 32) | (unsigned)x);
    for (int m = tid; m < M; m += NT)
        if (snv[m] >= 0 && sq[m] == key2f(qmax[snv[m]])) atomicMin(&src_seg[snv[m]], m);
    __syncthreads();
    for (int r = tid; r < nloc; r += NT) {
        if (uf[r] != r) continue;
        const int rep = gid[r];
        inst.n_obs[rep] = obs[r];
        int src;
        float q;
        if (src_inst[r] != ~0ull) {
            const int x = (int)(src_inst[r] & 0xffffffffu);
            src = gid[x];
            q = qloc[x];
        } else {
            src = -(src_seg[r] + 1);
            q = sq[src_seg[r]];
        }
        if (src == rep) continue;
        const int c = atomicAdd(&s_ncopy, 1);
        ss.copy_dst[c] = rep;
        ss.copy_src[c] = src;
        inst.Q[rep] = q;
    }
    // (6) merge members into their representative
    for (int x = tid; x < nloc; x += NT) {
        const int r = uf[x];
        if (r == x) continue;
        const int k = gid[x], rep = gid[r];
        inst.parent[k] = rep;
        atomicAdd((unsigned long long*)&inst.count[rep], (unsigned long long)inst.count[k]);
        inst.count[k] = 0;
        atomicAdd(&s_merges, 1);
    }
    __syncthreads();
    if (tid == 0) {
        *ss.copy_n = s_ncopy;
        *ss.edge_n = 0;  // the next frame's gates start a new edge list
        ctr->active_instances = s_nroots;
        ctr->new_instances = s_new;
        ctr->merges = s_merges;
        ctr->next_id = s_next;
        ctr->n_copies = s_ncopy;
    }
}

// The frame's pairs in the map's global pair hash, its edges in ss.edge_m/k;
// union_smem: a region of UNION_SMEM bytes (shared or global memory).
__device__ void phase_union(const FrameParams& fp, const Scratch& sc, const SerialScratch& ss, const Instances& inst,
                            int* next_id, unsigned char* union_smem)
{
    const int npairs = sc.ctr->n_pairs;
    const int nedge = min(*ss.edge_n, ss.edge_cap);
    union_frame(fp, sc, ss, inst, next_id, union_smem, npairs, nedge,
                [&](int i) { return (unsigned)(ss.okeys[ss.olist[i]] & 0xffffffffu); });
}

// One warp copies an embedding row (and writes its bf16 copy when tb is set).
__device__ __forceinline__ void copy_row(const float* from, float* to, uint16_t* tb, int D, int lane)
{
    if ((D & 3) == 0) {
        const float4* f4 = (const float4*)from;
        float4* t4 = (float4*)to;
        const int n4 = D >> 2;
        for (int d0 = 0; d0 < n4; d0 += 32 * 8) {
            float4 r[8];
#pragma unroll
            for (int j = 0; j < 8; j++) {
                const int d = d0 + j * 32 + lane;
                if (d < n4) r[j] = f4[d];
            }
#pragma unroll
            for (int j = 0; j < 8; j++) {
                const int d = d0 + j * 32 + lane;
                if (d < n4) {
                    t4[d] = r[j];
                    if (tb) ((uint2*)tb)[d] = make_uint2(bf16_pair(r[j].x, r[j].y), bf16_pair(r[j].z, r[j].w));
                }
            }
        }
    } else {
        for (int d = lane; d < D; d += 32) {
            to[d] = from[d];
            if (tb) tb[d] = __bfloat16_as_ushort(__float2bfloat16_rn(from[d]));
        }
    }
}

// ---- embeddings, new voxels, parent flattening, cleanup ---------------------------
__device__ void phase_apply(const FrameParams& fp, const Scratch& sc, const Scratch& va, const SerialScratch& ss,
                            const VoxelTable& vt,
                            const Instances& inst, const int* next_id, bool ok)
{
    const int gtid = blockIdx.x * blockDim.x + threadIdx.x;
    const int gsz = gridDim.x * blockDim.x;
    const int lane = threadIdx.x & 31;
    const int D = fp.D;
    if (ok) {
        // winning embeddings (the sources are never written in this frame):
        // one warp per vector, all loads in flight before the stores; the
        // scoring copies follow the scoring master (the association feature
        // with a second grid)
        const int nc = *ss.copy_n;
        for (int c = gtid >> 5; c < nc; c += gsz >> 5) {
            const int src = ss.copy_src[c], dst = ss.copy_dst[c];
            const float* from = src >= 0 ? inst.E + (size_t)src * D : sc.Ecan + (size_t)(-src - 1) * D;
            if (inst.A) {
                const int Da = inst.Da;
                const float* fa = src >= 0 ? inst.A + (size_t)src * Da : va.Ecan + (size_t)(-src - 1) * Da;
                copy_row(from, inst.E + (size_t)dst * D, nullptr, D, lane);
                copy_row(fa, inst.A + (size_t)dst * Da, inst.Eb ? inst.Eb + (size_t)dst * Da : nullptr, Da, lane);
                if (inst.E8) e4m3_copy_row(fa, Da, inst.E8 + (size_t)dst * Da, inst.Er + dst);
            } else {
                copy_row(from, inst.E + (size_t)dst * D, inst.Eb ? inst.Eb + (size_t)dst * D : nullptr, D, lane);
                if (inst.E8) e4m3_copy_row(from, D, inst.E8 + (size_t)dst * D, inst.Er + dst);
            }
        }
        // new voxels: the lowest segment index owns a voxel
        const int nn = sc.ctr->n_new;
        for (int i = gtid; i < nn; i += gsz) {
            const int t = ss.nlist[i];
            const unsigned long long key = ss.nkeys[t];
            const int lab = sc.segrep[ss.nown[t] - 1];
            unsigned long long h = vt_home(key, vt.mask);
            for (int pr = 0;; pr++) {
                const unsigned long long prev = atomicCAS(&vt.keys[h], EMPTY_KEY, key);
                if (prev == EMPTY_KEY) { vt.labels[h] = lab; break; }
                h = vt_next(h, pr + 1, vt.mask);
                if (pr > (int)vt.mask) { set_err(sc.ctr, DISC_ERR_TABLE_FULL); break; }
            }
            // one count update per distinct instance of the warp
            const unsigned grp = __match_any_sync(__activemask(), lab);
            if (lane == __ffs(grp) - 1) atomicAdd((unsigned long long*)&inst.count[lab], (unsigned long long)__popc(grp));
        }
        if (gtid == 0) atomicAdd(vt.used, (unsigned long long)nn);
        // keep the parent table flat (two levels at most after this frame)
        if (sc.ctr->merges > 0) {
            const int nid = *next_id;
            for (int i = gtid; i < nid; i += gsz) inst.parent[i] = inst.parent[inst.parent[i]];
        }
    }
    // cleanup of the serial hashes, whatever happened above
    const int np = sc.ctr->n_pairs, nn = sc.ctr->n_new;
    for (int i = gtid; i < np; i += gsz) {
        const int s = ss.olist[i];
        ss.okeys[s] = EMPTY_KEY;
        ss.ocnt[s] = 0;
    }
    for (int i = gtid; i < nn; i += gsz) {
        const int s = ss.nlist[i];
        // inserted above before this thread reset it: same thread, same i
        ss.nkeys[s] = EMPTY_KEY;
        ss.nown[s] = INT_MAX;
    }
}

// ---- kernels ------------------------------------------------------------------------
// Block row g runs frame j of map g.  Whether the frame is blocked is decided
// once per block (another block may raise an error while this one reads), so
// every thread of the block takes the same path.  Returns the frame slot, or
// -1 when map g has no frame j or the frame is blocked.
// The frame slot of this block's map (block row g) and whether the frame is
// blocked: by its own error, or (full check, the frame's first serial kernel)
// by an error of the map's previous frame, which is then copied into this
// frame's counters so that its later kernels need only their own.  Warp 0
// loads the slot indices side by side, then both status words: two round
// trips before the block's barrier.
__device__ int block_slot(const BatchScratch& bs, const SerialStep& st, bool* blocked, bool full)
{
    __shared__ int s_slot, s_blocked;
    const int g = blockIdx.y;
    if (threadIdx.x < 32) {
        const int lane = threadIdx.x;
        const bool prev_in_batch = st.j > 0;
        int v = -1;
        if (lane == 0)
            v = st.slot_of[g * st.J + st.j];
        else if (lane == 1 && full)
            v = prev_in_batch ? st.slot_of[g * st.J + st.j - 1] : st.prev_hist[g];
        const int slot = __shfl_sync(0xffffffffu, v, 0);
        const int pidx = __shfl_sync(0xffffffffu, v, 1);
        int e = 0;
        if (lane == 0 && slot >= 0)
            e = bs.frame(slot).ctr->err;
        else if (lane == 1 && full && pidx >= 0)
            e = prev_in_batch ? bs.frame(pidx).ctr->err : st.hist[pidx].err;
        const int own = __shfl_sync(0xffffffffu, e, 0);
        const int prev = __shfl_sync(0xffffffffu, e, 1);
        if (lane == 0) {
            bool b = slot >= 0 && own != 0;
            if (slot >= 0 && !b && full && prev) {
                set_err(bs.frame(slot).ctr, prev);
                b = true;
            }
            s_slot = slot;
            s_blocked = b ? 1 : 0;
        }
    }
    __syncthreads();
    const int slot = s_slot;
    *blocked = s_blocked != 0;
    __syncthreads();
    return slot;
}

constexpr size_t OV_SMEM = (size_t)OV_SLOTS * 12;

__global__ void __launch_bounds__(SER_THREADS) k_overlap(const FrameParams* fps, BatchScratch bs, SerialStep st)
{
    extern __shared__ __align__(16) unsigned char ov_smem[];
    bool blocked;
    const int slot = block_slot(bs, st, &blocked, true);
    if (slot < 0 || blocked) return;
    const MapRefs& R = st.refs[blockIdx.y];
    const SerialScratch ss = R.ss;
    const VoxelTable vt = R.vt;
    const Instances inst = R.inst;
    phase_overlap(bs.frame(slot), ss, vt, inst, ov_smem, fps[slot].dilate != 0);
}

__global__ void k_score(const FrameParams* fps, BatchScratch bs, SerialStep st)
{
    bool blocked;
    const int slot = block_slot(bs, st, &blocked, false);
    if (slot < 0 || blocked) return;
    const MapRefs& R = st.refs[blockIdx.y];
    const SerialScratch ss = R.ss;
    const Instances inst = R.inst;
    phase_score(fps[slot], bs.frame(slot), st.view.frame(slot), ss, inst, (blockIdx.x * blockDim.x + threadIdx.x) >> 5,
                (gridDim.x * blockDim.x) >> 5);
}

__global__ void __launch_bounds__(UNION_THREADS, 1) k_union(const FrameParams* fps, BatchScratch bs, SerialStep st)
{
    extern __shared__ __align__(16) unsigned char union_smem[];
    bool blocked;
    const int slot = block_slot(bs, st, &blocked, false);
    if (slot < 0 || blocked) return;
    const MapRefs& R = st.refs[blockIdx.y];
    const SerialScratch ss = R.ss;
    const Instances inst = R.inst;
    phase_union(fps[slot], bs.frame(slot), ss, inst, R.next_id, union_smem);
}

__global__ void k_apply(const FrameParams* fps, BatchScratch bs, SerialStep st)
{
    bool blocked;
    const int slot = block_slot(bs, st, &blocked, false);
    if (slot < 0) return;
    const MapRefs& R = st.refs[blockIdx.y];
    const SerialScratch ss = R.ss;
    const VoxelTable vt = R.vt;
    const Instances inst = R.inst;
    phase_apply(fps[slot], bs.frame(slot), st.view.frame(slot), ss, vt, inst, R.next_id, !blocked);
}

__global__ void k_serial_begin(const MapRefs* refs, int G)
{
    const int g = blockIdx.x * blockDim.x + threadIdx.x;
    if (g < G) {
        *refs[g].ss.edge_n = 0;
        *refs[g].ss.copy_n = 0;
    }
}

// ==== The frame chain as one pass per batch ==========================================
// The overlap histogram of frame j (Sec. III-B) counts, per segment m and
// instance root k, the segment's voxels whose label resolves to k in the map
// as frame j finds it.  A voxel of frame j is either
//   (a) in the map when the batch starts: its label is known before any frame
//       of the batch runs, only its root may change as earlier frames merge;
//   (b) absent then, and first seen in this batch by an earlier frame j0 of
//       the same map: that frame inserts it with the instance its lowest
//       segment m0 joins (Sec. III-B, reading O11), known once frame j0 is
//       associated;
//   (c) absent until frame j itself: a new voxel of frame j (no overlap),
//       owned by its lowest segment.
// So the per-voxel work of the whole batch runs before the frames run in
// order: k_lookup probes every (segment, voxel) entry of every frame in the
// map as it stands at the batch start and gathers each absent voxel's first
// (frame, segment) of the batch in one batch-wide hash; k_absent sorts the
// absent entries into (b) and (c).  Each frame is left with a few hundred
// to a few thousand items, (m, label) and (m, j0, m0), with voxel counts.
// k_associate then runs each map's frames in order in one CTA (overlap pairs
// from the items, the gates, the union, fusion and the voxel counts; a
// cluster's other CTAs take crowded frames' pairs and copies), and
// k_commit inserts the batch's new voxels with their first frame's labels and
// flattens the parent tables.  A frame that fails inserts nothing, and the
// frames after it in its map are blocked.

constexpr unsigned long long KEY54 = (1ull << 54) - 1;

// `cnt` more voxels of overlap item `key` of the frame
__device__ __forceinline__ void add_item(const Scratch& sc, unsigned long long key, int cnt)
{
    unsigned long long t = mix64(key) & sc.smask;
    for (unsigned long long pr = 0;; pr++) {
        const unsigned long long cur = sc.pkey[t];
        if (cur == key) break;
        if (cur == EMPTY_KEY) {
            const unsigned long long prev = atomicCAS(&sc.pkey[t], EMPTY_KEY, key);
            if (prev == EMPTY_KEY) {
                sc.plist[atomicAdd(&sc.ctr->n_pre, 1)] = (int)t;
                break;
            }
            if (prev == key) break;
        }
        t = (t + 1) & sc.smask;
        if (pr > sc.smask) {
            set_err(sc.ctr, DISC_ERR_TABLE_FULL);
            return;
        }
    }
    atomicAdd(&sc.pcnt[t], cnt);
}

// The warp's lanes with `want` set add one voxel each to overlap item `key`
// of the frame: lanes with the same key add together (one atomic per
// distinct key of the warp).  All 32 lanes call.
__device__ __forceinline__ void add_item_warp(const Scratch& sc, unsigned long long key, bool want)
{
    const unsigned act = __ballot_sync(0xffffffffu, want);
    if (!want) return;
    const unsigned grp = __match_any_sync(act, key);
    if ((int)(threadIdx.x & 31) != __ffs(grp) - 1) return;
    add_item(sc, key, __popc(grp));
}

// Warp-aggregated append: each lane with `want` gets a distinct index from
// the counter; all 32 lanes call.
__device__ __forceinline__ int warp_append(int* counter, bool want)
{
    const unsigned b = __ballot_sync(0xffffffffu, want);
    const int lane = threadIdx.x & 31;
    int base = 0;
    if (lane == 0 && b) base = atomicAdd(counter, __popc(b));
    base = __shfl_sync(0xffffffffu, base, 0);
    return base + __popc(b & ((1u << lane) - 1));
}

// Label of `key` in the voxel table (-1: absent), probed by the PW lanes of
// an aligned lane group together (warp-cooperative probing): each round the
// group loads PW consecutive slots of the probe sequence, and the first slot
// in probe order that holds the key or is empty decides.  All lanes of a
// group pass the same key and `active`; inactive groups return -1 at once.
// *probes: slots passed before the deciding one; *full: no empty slot found.
template <int PW>
__device__ __forceinline__ int probe_label(const VoxelTable& vt, unsigned long long key, bool active, int* probes,
                                           bool* full)
{
    *probes = 0;
    *full = false;
    if (!active) return -1;
    const int lane = threadIdx.x & 31, base = lane & ~(PW - 1), sub = lane - base;
    const unsigned gmask = (PW == 32 ? 0xffffffffu : ((1u << PW) - 1u)) << base;
    const unsigned long long h = vt_home(key, vt.mask);
    for (unsigned long long pr = 0; pr <= vt.mask; pr += PW) {
        const unsigned long long slot = vt_slot(h, pr + sub, vt.mask);
        const unsigned long long kk = vt.keys[slot];
        const unsigned hit = (__ballot_sync(gmask, kk == key || kk == EMPTY_KEY) & gmask) >> base;
        if (hit) {
            const int first = __ffs(hit) - 1;
            const bool found = __shfl_sync(gmask, kk == key, base + first);
            int lab = -1;
            if (found && sub == first) lab = vt.labels[slot];
            *probes = (int)pr + first;
            return found ? __shfl_sync(gmask, lab, base + first) : -1;
        }
    }
    *full = true;
    return -1;
}

// Absent voxel `key` of segment m of frame fp, into the batch's absent-voxel
// hash: its slot (-1 on failure); *claimed: the first to name the voxel.
__device__ __forceinline__ int add_absent(const FrameParams& fp, const Scratch& sc, const AbsentHash& ah, int m,
                                          unsigned long long key, bool* claimed)
{
    const unsigned long long ak = ((unsigned long long)(fp.map + 1) << 54) | key;
    unsigned long long t = mix64(ak) & ah.mask;
    for (unsigned long long pr = 0;; pr++) {
        const unsigned long long cur = ah.key[t];
        if (cur == ak) break;
        if (cur == 0ull) {
            const unsigned long long prev = atomicCAS(&ah.key[t], 0ull, ak);
            if (prev == 0ull) { *claimed = true; break; }
            if (prev == ak) break;
        }
        t = (t + 1) & ah.mask;
        if (pr > ah.mask) { set_err(sc.ctr, DISC_ERR_TABLE_FULL); return -1; }
    }
    atomicMin(&ah.val[t], (fp.jpos << 9) | m);
    return (int)t;
}

// Every entry of every frame slot of the batch (block row = slot), one lane
// per entry: as k_lookup below.  A thread takes four entries, whose keys,
// table slots and labels are each loaded together: the kernel waits for
// random table sectors, and one entry per thread kept too few of them in
// flight.  A block's 1024 entries (sorted by mask within their partitions)
// meet in a shared hash of items, so that only its distinct ones reach the
// frame's.
// Bound by the latency of random table sectors.  Room frames, 32 per launch,
// with k_absent and k_items: 4.8 us per frame with one entry per thread and a
// warp match, 4.0 so, 3.2 with a block's voxels in one place of the table
// (vt_home).
constexpr int LK_PER = 4, LK_THREADS = 256, LK_TILE = LK_PER * LK_THREADS, LK_SLOTS = 2 * LK_TILE;

__global__ void __launch_bounds__(LK_THREADS) k_lookup1(const FrameParams* fps, BatchScratch bs, const MapRefs* refs,
                                                        AbsentHash ah)
{
    __shared__ __align__(16) unsigned long long tkey[LK_SLOTS];
    __shared__ __align__(16) int tcnt[LK_SLOTS];
    __shared__ unsigned short tlist[LK_TILE];
    __shared__ int s_n, s_err;
    const int f = blockIdx.y;
    const FrameParams& fp = fps[f];
    const Scratch sc = bs.frame(f);
    const int ne = sc.ctr->n_entries, tid = threadIdx.x;
    if (tid == 0) s_err = *(volatile int32_t*)&sc.ctr->err;  // blocks of this launch may set it
    __syncthreads();
    if (fp.M <= 0 || s_err) return;  // a failed frame's items are never read
    const VoxelTable vt = refs[fp.map].vt;
    int maxp = 0;
    for (int i0 = blockIdx.x * LK_TILE; i0 < ne; i0 += gridDim.x * LK_TILE) {  // uniform per block
        unsigned long long hk[LK_PER], h[LK_PER], cur[LK_PER];
        int lab[LK_PER];
#pragma unroll
        for (int j = 0; j < LK_PER; j++) {
            const int i = i0 + j * LK_THREADS + tid;
            hk[j] = i < ne ? sc.sent[i] : 0ull;
        }
        for (int i = tid; i < LK_SLOTS / 2; i += LK_THREADS) ((uint4*)tkey)[i] = make_uint4(~0u, ~0u, ~0u, ~0u);
        for (int i = tid; i < LK_SLOTS / 4; i += LK_THREADS) ((int4*)tcnt)[i] = make_int4(0, 0, 0, 0);
        if (tid == 0) s_n = 0;
#pragma unroll
        for (int j = 0; j < LK_PER; j++) {
            h[j] = vt_home(hk[j] & KEY54, vt.mask);
            cur[j] = hk[j] ? vt.keys[h[j]] : EMPTY_KEY;
        }
        // the first slot decides most entries; the others walk on
#pragma unroll
        for (int j = 0; j < LK_PER; j++) {
            int pr = 0;
            while (cur[j] != EMPTY_KEY && cur[j] != (hk[j] & KEY54)) {
                if ((unsigned long long)++pr > vt.mask) {
                    set_err(sc.ctr, DISC_ERR_TABLE_FULL);
                    hk[j] = 0ull;
                    break;
                }
                h[j] = vt_next(h[j], pr, vt.mask);
                cur[j] = vt.keys[h[j]];
            }
            maxp = max(maxp, pr);
        }
#pragma unroll
        for (int j = 0; j < LK_PER; j++) lab[j] = hk[j] && cur[j] != EMPTY_KEY ? vt.labels[h[j]] : -1;
        __syncthreads();
#pragma unroll
        for (int j = 0; j < LK_PER; j++) {
            if (lab[j] >= 0) {
                const unsigned long long key = ((hk[j] >> 54) << 33) | (unsigned)lab[j];
                unsigned t = (unsigned)mix64(key) & (LK_SLOTS - 1);
                while (true) {  // at most LK_TILE distinct keys in LK_SLOTS slots
                    const unsigned long long prev = atomicCAS(&tkey[t], EMPTY_KEY, key);
                    if (prev == EMPTY_KEY) {
                        tlist[atomicAdd(&s_n, 1)] = (unsigned short)t;
                        break;
                    }
                    if (prev == key) break;
                    t = (t + 1) & (LK_SLOTS - 1);
                }
                atomicAdd(&tcnt[t], 1);
            }
            const bool absent = hk[j] && lab[j] < 0;
            if (!__any_sync(0xffffffffu, absent)) continue;
            bool claimed = false;
            int at = -1;
            if (absent) at = add_absent(fp, sc, ah, (int)(hk[j] >> 54), hk[j] & KEY54, &claimed);
            const int li = warp_append(ah.n, claimed);
            if (claimed) ah.list[li] = at;
            const int ai = warp_append(&sc.ctr->n_absent, at >= 0);
            if (at >= 0) {
                sc.aent[ai] = i0 + j * LK_THREADS + tid;
                sc.aslot[ai] = at;
            }
        }
        __syncthreads();
        for (int i = tid; i < s_n; i += LK_THREADS) add_item(sc, tkey[tlist[i]], tcnt[tlist[i]]);
        __syncthreads();
    }
    const int pm = __reduce_max_sync(0xffffffffu, maxp);
    if ((tid & 31) == 0 && pm > 0) atomicMax(&sc.ctr->max_probe, pm);
}

// Every entry of every frame slot of the batch (block row = slot): its label
// in the map at the batch start (tag-0 item), or, when absent, its slot in
// the batch's absent-voxel hash, where the least (frame position, segment)
// containing it is kept.  PW lanes (2, 4 or 8) look each entry up together;
// the group's first lane carries the entry afterwards.
template <int PW>
__global__ void __launch_bounds__(256) k_lookup(const FrameParams* fps, BatchScratch bs, const MapRefs* refs,
                                               AbsentHash ah)
{
    const int f = blockIdx.y;
    const FrameParams& fp = fps[f];
    const Scratch sc = bs.frame(f);
    const int ne = sc.ctr->n_entries;
    if (fp.M <= 0 || sc.ctr->err) return;  // a failed frame's items are never read
    const VoxelTable vt = refs[fp.map].vt;
    const int lane = threadIdx.x & 31;
    constexpr int PER = 32 / PW;  // entries of a warp per round
    const int warp = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, nwarps = (gridDim.x * blockDim.x) >> 5;
    int maxp = 0;
    for (int i0 = warp * PER; i0 < ne; i0 += nwarps * PER) {  // whole warps iterate together
        const int i = i0 + lane / PW;
        const bool valid = i < ne;
        const bool lead = valid && (lane & (PW - 1)) == 0;
        const unsigned long long hk = valid ? sc.sent[i] : 0ull;
        const int m = (int)(hk >> 54);
        const unsigned long long key = hk & KEY54;
        int probes;
        bool full;
        const int lab = probe_label<PW>(vt, key, valid, &probes, &full);
        if (lead && full) set_err(sc.ctr, DISC_ERR_TABLE_FULL);
        maxp = max(maxp, probes);
        int at = -1;
        bool claimed = false;
        if (lead && !full && lab < 0) {
            at = add_absent(fp, sc, ah, m, key, &claimed);
        }
        add_item_warp(sc, ((unsigned long long)m << 33) | (unsigned)lab, lead && lab >= 0);
        const int li = warp_append(ah.n, claimed);
        if (claimed) ah.list[li] = at;
        const int ai = warp_append(&sc.ctr->n_absent, at >= 0);
        if (at >= 0) {
            sc.aent[ai] = i;
            sc.aslot[ai] = at;
        }
    }
    const int pm = __reduce_max_sync(0xffffffffu, maxp);
    if (lane == 0 && pm > 0) atomicMax(&sc.ctr->max_probe, pm);
}

// Every entry absent at the batch start, once the batch-wide hash holds each
// voxel's first (frame position j0, segment m0): j0 before this frame makes a
// tag-1 item (m, j0 << 9 | m0); j0 this frame makes a new voxel, counted for
// its owner m0 once (by the entry of m0 itself).
__global__ void __launch_bounds__(256) k_absent(const FrameParams* fps, BatchScratch bs, AbsentHash ah)
{
    __shared__ int s_new[MAX_MASKS];
    const int f = blockIdx.y;
    const FrameParams& fp = fps[f];
    const Scratch sc = bs.frame(f);
    const int na = sc.ctr->n_absent;
    if (fp.M <= 0 || sc.ctr->err || (int)(blockIdx.x * blockDim.x) >= na) return;  // uniform per block
    for (int m = threadIdx.x; m < fp.M; m += blockDim.x) s_new[m] = 0;
    __syncthreads();
    const int lane = threadIdx.x & 31;
    for (int a0 = blockIdx.x * blockDim.x + (threadIdx.x & ~31); a0 < na; a0 += gridDim.x * blockDim.x) {
        const int a = a0 + lane;
        const bool valid = a < na;
        int m = 0, pv = 0;
        if (valid) {
            m = (int)(sc.sent[sc.aent[a]] >> 54);
            pv = ah.val[sc.aslot[a]];
        }
        const int j0 = pv >> 9, m0 = pv & 511;
        add_item_warp(sc, ((unsigned long long)m << 33) | (1ull << 32) | (unsigned)pv, valid && j0 < fp.jpos);
        if (valid && j0 == fp.jpos && m0 == m) atomicAdd(&s_new[m - 1], 1);
    }
    __syncthreads();
    int tot = 0;
    for (int m = threadIdx.x; m < fp.M; m += blockDim.x)
        if (s_new[m]) {
            atomicAdd(&sc.newcnt[m], s_new[m]);
            tot += s_new[m];
        }
    tot = warp_sum(tot);
    if (lane == 0 && tot) atomicAdd(&sc.ctr->n_new, tot);
}

// Every slot's overlap items, once k_absent is done: the hash slots listed
// in plist become dense (key, count) arrays in claim order (ikey over the
// free aent | aslot, icnt over plist itself: each thread reads plist[i]
// before it writes icnt[i]), tag-0 items under their label's root as the
// batch starts, and the hash is emptied for the slot's next batch.  Items of
// a failed frame are emptied as well.
__global__ void __launch_bounds__(256) k_items(const FrameParams* fps, BatchScratch bs, const MapRefs* refs)
{
    const Scratch sc = bs.frame(blockIdx.y);
    const int n = sc.ctr->n_pre;
    const int32_t* parent = refs[fps[blockIdx.y].map].inst.parent;  // flat between batches
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
        const int t = sc.plist[i];
        unsigned long long key = sc.pkey[t];
        const int cnt = sc.pcnt[t];
        sc.pkey[t] = EMPTY_KEY;
        sc.pcnt[t] = 0;
        if (!((key >> 32) & 1ull)) key = (key & ~0xffffffffull) | (unsigned)parent[(unsigned)key];
        sc.ikey[i] = key;
        sc.icnt[i] = cnt;
    }
}

// root of instance id x (parent chains may be longer than one step between
// the merges of a batch and its k_commit).  A parent is never above its
// child (a merge hooks an instance under the component's smallest id), so a
// chain ends within one step per merging frame of the batch; the step limit
// only keeps a damaged table from looping.
__device__ __forceinline__ int find_root(const int32_t* parent, int x)
{
    for (int it = 0; it < (1 << 16); it++) {
        const int p = parent[x];
        if (p == x) break;
        x = p;
    }
    return x;
}

// one thread reads a counter word another thread of the launch may have
// written by an atomic; every thread then takes the same branch
__device__ __forceinline__ int block_read(const int32_t* w)
{
    __shared__ int s_v;
    __syncthreads();
    if (threadIdx.x == 0) s_v = *(volatile const int32_t*)w;
    __syncthreads();
    const int v = s_v;
    __syncthreads();
    return v;
}

constexpr int ASSOC_THREADS = 512;
constexpr int APH = 2048;         // slots of the pair hash (shared memory)
constexpr int APH_MAX = 1536;     // pairs it takes (load <= 3/4)
constexpr int APH_PROBES = 64;    // longest probe of the pair hash
constexpr int ARH = 2048;         // slots of the hash of active roots
constexpr int ASSOC_ROOTS = 256;  // instances with an accepted edge, in shared memory
constexpr int ASSOC_EDGES = 512;  // accepted edges, in shared memory
constexpr int ASSOC_CHG = 512;    // words of the bitmap of instances whose embedding changed in the batch
// A frame past one of these shared capacities runs steps (1)-(3) with the
// map's global pair hash and union region.
constexpr int ASSOC_FRAMES = 64;  // frames whose slot, items and masks are read once, at the start

// an overlap item's icnt word: its voxels, and what k_gates found of its
// segment against its instance as the batch starts
constexpr int ITEM_COUNT = (1 << 26) - 1;
constexpr int ITEM_KNOWN = 1 << 28, ITEM_EDGE = 1 << 29, ITEM_BORDER = 1 << 30;

// The state of the frame a CTA works on.
struct __align__(16) AssocShared {
    unsigned long long pk[APH];             // (segment + 1) << 32 | root
    unsigned long long best[ASSOC_ROOTS];   // per local root: best candidate of its component (cand_key)
    long long cloc[ASSOC_ROOTS];            // voxel count
    int pc[APH];                            // voxels of the pair
    int pd[APH];                            // its ITEM_* flags
    unsigned short pl[APH_MAX];             // used slots
    unsigned rkey[ARH];                     // active roots
    int rval[ARH];                          // local index of a root with an edge
    int2 live[APH_MAX];                     // pairs to score now: (segment | root slot << 9, instance)
    int gid[ASSOC_ROOTS];                   // local root -> instance id
    int uf[ASSOC_ROOTS];                    // union-find over local roots
    int obs[ASSOC_ROOTS];                   // observations of its component
    int oloc[ASSOC_ROOTS];                  // observations
    int em[ASSOC_EDGES];                    // accepted edges: segment and root slot
    int eh[ASSOC_EDGES];
    int anchor[MAX_MASKS];                  // smallest local root of a segment's edges
    unsigned chg[ASSOC_CHG];                // bit hash(id): id's embedding changed in this batch
    unsigned want[MAX_MASKS / 32];          // segments that open an instance
    int err, ncopies;                       // the frame's status and embedding copies
    int4 meta[ASSOC_FRAMES];                // the first frames' slot, n_pre, own error and masks
    int4 job;                               // for the cluster's other CTAs: kind, items, frame slot
    int ne, nlive, nloc, nroots, np, nsc, border, ovf, multi, ncopy, merges, next, merged_any, all_changed;
};
constexpr size_t ASSOC_SMEM = sizeof(AssocShared);
constexpr size_t ASSOC_SMEM_ALONE = 216 * 1024;
constexpr int RV_FREE = -1, RV_TAKEN = -2;

// A fusion candidate as a number: the higher Q first, then the smaller order
// (an instance id, or 2^31 + mask: members by id, then segments by mask).
__device__ __forceinline__ unsigned long long cand_key(float q, unsigned order)
{
    return ((unsigned long long)f2key(q) << 32) | (unsigned)~order;
}

__device__ __forceinline__ unsigned chg_bit(int id) { return ((unsigned)id * 0x9E3779B1u) >> 18; }  // 14 bits
static_assert(ASSOC_CHG * 32 == 1 << 14, "one bit per hash value");

// Accepted edge (segment m, root slot h) number e: the first edge of a root
// opens its local index with the instance's values.
__device__ __forceinline__ void claim_root(AssocShared& A, int h, int k, long long cnt, float q, int obs)
{
    if (atomicCAS(&A.rval[h], RV_FREE, RV_TAKEN) != RV_FREE) return;
    const int x = atomicAdd(&A.nloc, 1);
    if (x < ASSOC_ROOTS) {
        A.gid[x] = k;
        A.uf[x] = x;
        A.cloc[x] = cnt;
        A.oloc[x] = A.obs[x] = obs;
        A.best[x] = cand_key(q, (unsigned)k);
    }
    A.rval[h] = x;
}

// The cosine gate of every tag-0 item's segment against its instance as the
// batch starts, one warp per item, all frames of the batch at once: most
// instances keep their embedding through a batch, and k_associate then finds
// the decision beside the item.  (Also for one frame per map: a Room frame's
// 43 passing pairs, three rounds of k_associate's warps, cost it 8 us and the
// launch 5.)
__global__ void __launch_bounds__(256) k_gates(const FrameParams* fps, BatchScratch bs, BatchScratch view,
                                               const MapRefs* refs)
{
    const int f = blockIdx.y;
    const FrameParams& fp = fps[f];
    const Scratch sc = bs.frame(f);
    if (fp.M <= 0 || sc.ctr->err) return;  // a failed frame's items are never read
    const int n = sc.ctr->n_pre, nw = (gridDim.x * blockDim.x) >> 5;
    const Instances inst = refs[fp.map].inst;
    const GateFeatures gf = gate_features(fp, sc, view.frame(f), inst);
    for (int i = (blockIdx.x * blockDim.x + threadIdx.x) >> 5; i < n; i += nw) {
        const unsigned long long key = sc.ikey[i];
        if ((key >> 32) & 1ull) continue;
        int border = 0;
        const bool edge = warp_cosine_gate(fp, gf, inst, (int)(key >> 33) - 1, (int)(unsigned)key, &border);
        if ((threadIdx.x & 31) == 0)
            sc.icnt[i] |= ITEM_KNOWN | (edge ? ITEM_EDGE : 0) | (border ? ITEM_BORDER : 0);
    }
}

// ---- what the other CTAs of a map's cluster do for its leader ---------------------
// They wait at the cluster's barrier for a job, read it and its items from the
// leader's shared memory, and meet the leader at the barrier again when it is
// done.
constexpr int JOB_END = 0, JOB_SCORE = 1, JOB_COPY = 2, JOB_PAIRS = 3;
constexpr int JOB_MIN = 48;  // items that are worth one: three rounds of the leader's warps
constexpr int LIVE_EDGE = 1 << 30, LIVE_BORDER = 1 << 29;  // what became of a pair, in its live word

// Pairs w, w + nw, ... of the leader's n live pairs through the cosine gate.
__device__ __noinline__ void job_score(const AssocShared& A, const FrameParams& fp, const GateFeatures& gf,
                                       const Instances& inst, int n, int w, int nw)
{
    const unsigned live = dsm_map(A.live, 0);
    for (int q = w; q < n; q += nw) {
        const int x = dsm_ld32(live + 8u * q), k = dsm_ld32(live + 8u * q + 4u);
        int border = 0;
        const bool edge = warp_cosine_gate(fp, gf, inst, x & 511, k, &border);
        if ((threadIdx.x & 31) == 0)
            dsm_st32(live + 8u * q, x | (edge ? LIVE_EDGE : 0) | (border ? LIVE_BORDER : 0));
    }
}

// One warp writes the embedding (and, with a second grid, the association
// feature) that copy c of the frame names, and its scoring copy.
__device__ __forceinline__ void copy_embedding(const MapRefs& R, const Scratch& sc, const Scratch& va, int D, int c)
{
    const Instances& inst = R.inst;
    const int lane = threadIdx.x & 31;
    const int src = R.ss.copy_src[c], dst = R.ss.copy_dst[c];
    const float* from = src >= 0 ? inst.E + (size_t)src * D : sc.Ecan + (size_t)(-src - 1) * D;
    if (inst.A) {
        const int Da = inst.Da;
        const float* fa = src >= 0 ? inst.A + (size_t)src * Da : va.Ecan + (size_t)(-src - 1) * Da;
        copy_row(from, inst.E + (size_t)dst * D, nullptr, D, lane);
        copy_row(fa, inst.A + (size_t)dst * Da, inst.Eb ? inst.Eb + (size_t)dst * Da : nullptr, Da, lane);
        if (inst.E8) e4m3_copy_row(fa, Da, inst.E8 + (size_t)dst * Da, inst.Er + dst);
    } else {
        copy_row(from, inst.E + (size_t)dst * D, inst.Eb ? inst.Eb + (size_t)dst * D : nullptr, D, lane);
        if (inst.E8) e4m3_copy_row(from, D, inst.E8 + (size_t)dst * D, inst.Er + dst);
    }
}

__device__ __noinline__ void assoc_help(const AssocShared& A, const MapRefs& R, const FrameParams* fps,
                                        const BatchScratch& bs, const BatchScratch& view, int rank, int nranks)
{
    const int wid = threadIdx.x >> 5, nw = ASSOC_THREADS >> 5;
    const unsigned job = dsm_map(&A.job, 0);
    while (true) {
        cluster_sync();  // the leader has a job
        const int kind = dsm_ld32(job), n = dsm_ld32(job + 4), slot = dsm_ld32(job + 8);
        if (kind != JOB_END) {
            const FrameParams& fp = fps[slot];
            const Scratch sc = bs.frame(slot), va = view.frame(slot);
            if (kind == JOB_PAIRS) {  // (past the shared capacities: the pairs of the map's global hash)
                phase_score(fp, sc, va, R.ss, R.inst, rank * nw + wid, nranks * nw);
            } else if (kind == JOB_SCORE) {
                job_score(A, fp, gate_features(fp, sc, va, R.inst), R.inst, n, rank * nw + wid, nranks * nw);
            } else {  // (the leader goes on to the next frame meanwhile)
                for (int c = (rank - 1) * nw + wid; c < n; c += (nranks - 1) * nw) copy_embedding(R, sc, va, fp.D, c);
            }
        }
        cluster_sync();  // it is done, and the leader's shared memory read
        if (kind == JOB_END) return;
    }
}

// One CTA per map of the batch walks the map's frames in order.  Per frame:
//   (1) every item (its label resolved to the root as of now) adds to its
//       (segment, root) pair in the shared pair hash;
//   (2) a thread per pair: the overlap gate, the active roots, and the cosine
//       gate where k_gates took it for the instance's embedding at the batch
//       start and no frame has changed that since; the pairs left are scored
//       now, a warp each;
//   (3) components, new ids, merges and fusion winners, and the frame's new
//       voxels into the counts;
//   (4) a warp per embedding copy.
// with a block barrier after each; step (4) runs beside the next frame's
// step (1), which reads no embedding.  The next frame's items and segment
// values are loaded while this one is united.  A frame past the shared
// capacities runs steps (1)-(3) with the map's global pair hash and union
// region.
//
// Bound by latency: a row of dependent steps per frame.  Room frames, 32 per
// launch: 9.5 us per frame.  A cluster of 8 CTAs per map, whose leader's state
// the others reached through distributed shared memory, took 15.2 us (every
// passing pair scored between two cluster barriers, the union in fourteen
// block barriers) and 11.8 with k_gates and this union: a cluster barrier that
// orders global memory costs 1.2 us and empties the L1, a block barrier 0.03
// us.  So one CTA, the leader, walks the frames, and the others of a cluster
// only wait for jobs: the pairs left to score and the embeddings to copy where
// a frame has more than JOB_MIN of them (the copies while the leader goes on to
// the next frame's steps (1) and (2)).  Frames of 240 masks, us per frame, one
// CTA | 8 with jobs: views that stay alike 42 | 18, views that improve 72 | 25,
// masks that drift over the instances 88 | 26; 100 masks 23 | 14, 32 | 19,
// 41 | 18; 40 masks 14.8 | 14.6, 17.2 | 17.1, 19.5 | 14.6.  Spills about 500
// bytes a thread at 128 registers, the most that 512 threads can have.
__global__ void __launch_bounds__(ASSOC_THREADS, 1) k_associate(const FrameParams* fps, BatchScratch bs,
                                                                SerialStep st)
{
    extern __shared__ __align__(16) unsigned char assoc_smem[];
    AssocShared& A = *(AssocShared*)assoc_smem;
    const int g = blockIdx.y, rank = blockIdx.x, nranks = gridDim.x;  // a cluster spans the grid's x
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    constexpr int NT = ASSOC_THREADS;
    // the map's table pointers, in shared memory: read there, they are never
    // reloaded from global memory after the kernel's own global stores
    __shared__ MapRefs s_refs;
    static_assert(sizeof(MapRefs) % 8 == 0, "copied in 8-byte words");
    for (int i = tid; i < (int)(sizeof(MapRefs) / 8); i += NT)
        ((unsigned long long*)&s_refs)[i] = ((const unsigned long long*)&st.refs[g])[i];
    if (rank > 0) {  // uniform per block
        __syncthreads();
        assoc_help(A, s_refs, fps, bs, st.view, rank, nranks);
        return;
    }
    // a job for the cluster's other CTAs, and the wait until the last one is done
    bool helping = false;
    auto finish = [&] {
        if (helping) cluster_sync();
        helping = false;
    };
    auto give = [&](int kind, int n, int slot) {
        finish();
        if (tid == 0) A.job = make_int4(kind, n, slot, 0);
        cluster_sync();
        helping = true;
    };
    for (int j = tid; j < min(st.J, ASSOC_FRAMES); j += NT) {
        const int slot = st.slot_of[g * st.J + j];
        A.meta[j] = slot < 0 ? make_int4(-1, 0, 0, 0)
                             : make_int4(slot, bs.frame(slot).ctr->n_pre,
                                         *(volatile const int32_t*)&bs.frame(slot).ctr->err, fps[slot].M);
    }
    __syncthreads();
    auto meta = [&](int j) -> int4 {
        if (j < ASSOC_FRAMES) return A.meta[j];
        const int slot = st.slot_of[g * st.J + j];
        return slot < 0 ? make_int4(-1, 0, 0, 0)
                        : make_int4(slot, bs.frame(slot).ctr->n_pre,
                                    *(volatile const int32_t*)&bs.frame(slot).ctr->err, fps[slot].M);
    };
    const MapRefs& R = s_refs;
    const Instances& inst = R.inst;
    for (int i = tid; i < APH; i += NT) {
        A.pk[i] = EMPTY_KEY;
        A.pc[i] = A.pd[i] = 0;
    }
    for (int i = tid; i < ARH; i += NT) {
        A.rkey[i] = UH_EMPTY;
        A.rval[i] = RV_FREE;
    }
    for (int i = tid; i < MAX_MASKS; i += NT) A.anchor[i] = INT_MAX;
    for (int i = tid; i < ASSOC_CHG; i += NT) A.chg[i] = 0u;
    if (tid == 0) {
        *R.ss.edge_n = 0;
        *R.ss.copy_n = 0;
        A.ne = A.nlive = A.nloc = A.nroots = A.np = A.nsc = A.border = A.ovf = A.multi = A.ncopy = A.merges = 0;
        A.merged_any = A.all_changed = A.err = A.ncopies = 0;
        A.next = *(volatile const int*)R.next_id;
    }
    // an item's (segment, root) pair: tag-1 items through the segment their
    // voxel's first frame gave it to; known: the root is the one k_gates took
    auto label_of = [&](unsigned long long key) -> int {
        const unsigned x = (unsigned)key;
        return ((key >> 32) & 1ull) ? bs.frame(st.slot_of[g * st.J + (int)(x >> 9)]).segrep[(x & 511u) - 1] : (int)x;
    };
    // the thread's first item of a frame and its segment's values, loaded ahead
    unsigned long long pre_key = EMPTY_KEY;
    int pre_cnt = 0, pre_nv = 0, pre_new = 0;
    float pre_q = 0.0f;
    auto prefetch = [&](int j) {
        if (j >= st.J) return;
        const int4 mt = meta(j);
        if (mt.x < 0) return;
        const Scratch sc = bs.frame(mt.x);
        if (tid < mt.w) {
            pre_nv = sc.nvox[tid];
            pre_q = sc.S[5 * tid + 4];
            pre_new = sc.newcnt[tid];
        }
        if (tid < mt.y) {
            pre_key = sc.ikey[tid];
            pre_cnt = sc.icnt[tid];
        }
    };
    prefetch(0);
    const int4 meta0 = meta(0);
    const int ov_num = meta0.x < 0 ? 0 : fps[meta0.x].ov_num, ov_den = meta0.x < 0 ? 1 : fps[meta0.x].ov_den;
    __syncthreads();
    for (int j = 0; j < st.J; j++) {
        const int4 mt = meta(j);
        const int slot = mt.x;
        if (slot < 0) break;
        const FrameParams& fp = fps[slot];
        const Scratch sc = bs.frame(slot);
        const int M = mt.w;
        // blocked: the frame's own error (set before the launch), or its
        // predecessor's status (staged before the last barrier)
        const int prev = j > 0 ? A.err : (st.prev_hist[g] >= 0 ? st.hist[st.prev_hist[g]].err : 0);
        const int own = mt.z;
        const bool blocked = own || prev;
        if (tid == 0 && !own && prev) set_err(sc.ctr, prev);
        bool global_pairs = false, united = false;
        if (!blocked) {
            const int nv = pre_nv, nnew = pre_new;
            const float sq = pre_q;
            // (1) overlap pairs
            for (int i = tid; i < mt.y; i += NT) {
                const unsigned long long key = i == tid ? pre_key : sc.ikey[i];
                const int cnt = i == tid ? pre_cnt : sc.icnt[i];
                const int lab = label_of(key);
                if (lab < 0) continue;
                const int root = find_root(inst.parent, lab);
                const unsigned long long okey = ((key >> 33) << 32) | (unsigned)root;
                unsigned h = (unsigned)(mix64(okey) & (APH - 1));
                int pr = 0;
                for (; pr < APH_PROBES; pr++) {
                    const unsigned long long prv = atomicCAS(&A.pk[h], EMPTY_KEY, okey);
                    if (prv == EMPTY_KEY) {
                        const int at = atomicAdd(&A.np, 1);
                        if (at < APH_MAX) A.pl[at] = (unsigned short)h;
                    }
                    if (prv == EMPTY_KEY || prv == okey) break;
                    h = (h + 1) & (APH - 1);
                }
                if (pr == APH_PROBES) {
                    A.ovf = 1;
                    continue;
                }
                atomicAdd(&A.pc[h], cnt & ITEM_COUNT);
                // k_gates' decision holds for the root it saw
                if ((cnt & ITEM_KNOWN) && root == lab) atomicOr(&A.pd[h], cnt & ~ITEM_COUNT);
            }
            __syncthreads();
            const int np = A.np;
            global_pairs = A.ovf || np > APH_MAX;  // uniform
            if (!global_pairs) {
                // (2) |V_m & V_k| / min(|V_m|, |V_k|) >= ov_num / ov_den; the
                //     hash is emptied on the way
                int nsc = 0, nroot = 0, border = 0;
                for (int i = tid; i < np; i += NT) {
                    const int t = A.pl[i];
                    const unsigned long long okey = A.pk[t];
                    const int ov = A.pc[t], fl = A.pd[t];
                    const int m = (int)(okey >> 32) - 1, k = (int)(okey & 0xffffffffu);
                    const int nvm = sc.nvox[m], obs = inst.n_obs[k];
                    const long long count = inst.count[k];
                    const float q = inst.Q[k];
                    A.pk[t] = EMPTY_KEY;
                    A.pc[t] = A.pd[t] = 0;
                    // active set: the distinct roots of all overlap pairs
                    unsigned h = uhash((unsigned)k, ARH - 1);
                    while (true) {  // at most APH_MAX roots in ARH slots
                        const unsigned prv = atomicCAS(&A.rkey[h], UH_EMPTY, (unsigned)k);
                        if (prv == UH_EMPTY) nroot++;
                        if (prv == UH_EMPTY || prv == (unsigned)k) break;
                        h = (h + 1) & (ARH - 1);
                    }
                    if ((long long)ov * ov_den < (long long)ov_num * min((long long)nvm, count)) continue;
                    nsc++;
                    const unsigned bit = chg_bit(k);
                    if (!(fl & ITEM_KNOWN) || A.all_changed || ((A.chg[bit >> 5] >> (bit & 31)) & 1u)) {
                        A.live[atomicAdd(&A.nlive, 1)] = make_int2(m | ((int)h << 9), k);
                        continue;
                    }
                    if (fl & ITEM_BORDER) border++;
                    if (!(fl & ITEM_EDGE)) continue;
                    const int e = atomicAdd(&A.ne, 1);
                    if (e < ASSOC_EDGES) {
                        A.em[e] = m;
                        A.eh[e] = (int)h;
                    }
                    claim_root(A, (int)h, k, count, q, obs);
                }
                const int sums = warp_sum(nroot | (nsc << 16));  // each at most APH_MAX / 16
                border = warp_sum(border);
                if (lane == 0 && sums) {
                    atomicAdd(&A.nroots, sums & 0xffff);
                    atomicAdd(&A.nsc, sums >> 16);
                    if (border) atomicAdd(&A.border, border);
                }
                __syncthreads();
            }
            // the copies of the frame before, where the other CTAs make them:
            // the gates read embeddings, step (3) writes the copy lists
            finish();
            if (!global_pairs) {
                const int nlive = A.nlive;
                if (nranks > 1 && nlive > JOB_MIN) {
                    give(JOB_SCORE, nlive, slot);
                    job_score(A, fp, gate_features(fp, sc, st.view.frame(slot), inst), inst, nlive, wid,
                              nranks * (NT >> 5));
                    finish();
                    int border = 0;
                    for (int q = tid; q < nlive; q += NT) {
                        const int x = A.live[q].x, k = A.live[q].y, h = (x >> 9) & (ARH - 1);
                        if (x & LIVE_BORDER) border++;
                        if (!(x & LIVE_EDGE)) continue;
                        const int e = atomicAdd(&A.ne, 1);
                        if (e < ASSOC_EDGES) {
                            A.em[e] = x & 511;
                            A.eh[e] = h;
                        }
                        claim_root(A, h, k, inst.count[k], inst.Q[k], inst.n_obs[k]);
                    }
                    border = warp_sum(border);
                    if (lane == 0 && border) atomicAdd(&A.border, border);
                    __syncthreads();
                } else if (nlive > 0) {
                    const GateFeatures gf = gate_features(fp, sc, st.view.frame(slot), inst);
                    int rescored = 0;
                    for (int q = wid; q < nlive; q += NT >> 5) {
                        const int m = A.live[q].x & 511, h = A.live[q].x >> 9, k = A.live[q].y;
                        // the instance's values the union needs, read beside the gate
                        const long long ck = lane == 0 ? inst.count[k] : 0;
                        const float qk = lane == 0 ? inst.Q[k] : 0.0f;
                        const int ok = lane == 0 ? inst.n_obs[k] : 0;
                        if (!warp_cosine_gate(fp, gf, inst, m, k, &rescored) || lane != 0) continue;
                        const int e = atomicAdd(&A.ne, 1);
                        if (e < ASSOC_EDGES) {
                            A.em[e] = m;
                            A.eh[e] = h;
                        }
                        claim_root(A, h, k, ck, qk, ok);
                    }
                    if (lane == 0 && rescored) atomicAdd(&A.border, rescored);
                    __syncthreads();
                }
                global_pairs = A.ne > ASSOC_EDGES || A.nloc > ASSOC_ROOTS;  // uniform
            }
            // the next frame's items and segment values, on their way while
            // this one is united
            prefetch(j + 1);
            if (!global_pairs) {
                // (3) components: a segment joins every root it has an edge
                //     with; a set's root is its smallest instance id
                const int ne = A.ne, nloc = A.nloc;
                for (int e = tid; e < ne; e += NT)
                    if (atomicMin(&A.anchor[A.em[e]], A.rval[A.eh[e]]) != INT_MAX) A.multi = 1;
                __syncthreads();
                if (A.multi) {  // some segment has several edges: every edge hooks its root onto the segment's anchor
                    for (int e = tid; e < ne; e += NT) {
                        int x = A.rval[A.eh[e]], y = A.anchor[A.em[e]];
                        while (true) {
                            x = uf_find(A.uf, x);
                            y = uf_find(A.uf, y);
                            if (x == y) break;
                            const int lo = A.gid[x] < A.gid[y] ? x : y, hi = lo == x ? y : x;
                            if (atomicCAS(&A.uf[hi], hi, lo) == hi) break;
                        }
                    }
                    __syncthreads();
                    int root = -1;
                    if (tid < nloc) root = uf_find(A.uf, tid);
                    __syncthreads();
                    if (tid < nloc) A.uf[tid] = root;
                    __syncthreads();
                }
                // fusion candidates: the members of a component by id, then its
                // segments by mask; the first with the highest Q wins.  New
                // instances: live segments without an edge, in mask order.
                int comp = -1;  // the segment's component
                if (tid < MAX_MASKS) {
                    if (tid < M && A.anchor[tid] != INT_MAX) comp = A.uf[A.anchor[tid]];
                    const unsigned w = __ballot_sync(0xffffffffu, tid < M && nv > 0 && comp < 0);
                    if (lane == 0) A.want[wid] = w;
                    if (comp >= 0) {
                        atomicMax(&A.best[comp], cand_key(sq, 0x80000000u | (unsigned)tid));
                        atomicAdd(&A.obs[comp], 1);
                    }
                } else {
                    const int x = tid - MAX_MASKS;
                    if (x < nloc && A.uf[x] != x) {
                        atomicMax(&A.best[A.uf[x]], A.best[x]);  // (only roots' entries change)
                        atomicAdd(&A.obs[A.uf[x]], A.oloc[x]);
                    }
                }
                __syncthreads();
                int first = 0, total = 0;
#pragma unroll
                for (int w = 0; w < MAX_MASKS / 32; w++) {
                    const int c = __popc(A.want[w]);
                    if (w < wid) first += c;
                    total += c;
                }
                const int base = A.next;
                if (base + total > inst.cap) {  // uniform
                    if (tid == 0) set_err(sc.ctr, DISC_ERR_CAPACITY);
                    __syncthreads();
                } else {
                    united = true;
                    if (tid < MAX_MASKS) {
                        if (tid < M) {
                            int rep = comp >= 0 ? A.gid[comp] : -1;
                            if ((A.want[wid] >> lane) & 1u) {
                                first += __popc(A.want[wid] & ((1u << lane) - 1));
                                rep = base + first;
                                inst.parent[rep] = rep;
                                inst.count[rep] = nnew;
                                inst.Q[rep] = sq;
                                inst.n_obs[rep] = 1;
                                R.ss.copy_dst[first] = rep;
                                R.ss.copy_src[first] = -(tid + 1);
                            } else if (rep >= 0 && nnew) {
                                atomicAdd((unsigned long long*)&inst.count[rep], (unsigned long long)nnew);
                            }
                            sc.segrep[tid] = rep;
                        }
                    } else if (tid - MAX_MASKS < nloc) {
                        const int x = tid - MAX_MASKS, r = A.uf[x], k = A.gid[x];
                        if (r != x) {  // merged into its representative
                            inst.parent[k] = A.gid[r];
                            atomicAdd((unsigned long long*)&inst.count[A.gid[r]], (unsigned long long)A.cloc[x]);
                            inst.count[k] = 0;
                            atomicAdd(&A.merges, 1);
                        } else {
                            const unsigned order = ~(unsigned)A.best[x];
                            inst.n_obs[k] = A.obs[x];
                            if (order != (unsigned)k) {  // another member's or a segment's embedding
                                const int c = total + atomicAdd(&A.ncopy, 1);
                                R.ss.copy_dst[c] = k;
                                R.ss.copy_src[c] = (order & 0x80000000u) ? -(int)(order & 0x7fffffffu) - 1 : (int)order;
                                inst.Q[k] = key2f((unsigned)(A.best[x] >> 32));
                                const unsigned bit = chg_bit(k);
                                atomicOr(&A.chg[bit >> 5], 1u << (bit & 31));
                            }
                        }
                    }
                    __syncthreads();
                    if (tid == 0) {
                        FrameCounters* ctr = sc.ctr;
                        ctr->n_pairs = np;
                        ctr->n_scored = A.nsc;
                        if (A.border) atomicAdd(&ctr->borderline, A.border);
                        ctr->active_instances = A.nroots;
                        ctr->new_instances = total;
                        ctr->merges = A.merges;
                        ctr->next_id = base + total;
                        ctr->n_copies = total + A.ncopy;
                        *R.next_id = base + total;
                        A.next = base + total;
                        if (A.merges) A.merged_any = 1;
                        A.err = 0;
                        A.ncopies = total + A.ncopy;
                    }
                }
            }
            if (global_pairs) {
                // more pairs, edges or edge roots than the shared memory holds:
                // with the map's global pair hash and union region
                __syncthreads();
                for (int i = tid; i < mt.y; i += NT) {
                    const unsigned long long key = sc.ikey[i];
                    const int lab = label_of(key);
                    if (lab >= 0)
                        add_pair(sc, R.ss, ((key >> 33) << 32) | (unsigned)find_root(inst.parent, lab),
                                 sc.icnt[i] & ITEM_COUNT);
                }
                if (!block_read(&sc.ctr->err)) {
                    if (nranks > 1) give(JOB_PAIRS, 0, slot);
                    phase_score(fp, sc, st.view.frame(slot), R.ss, inst, wid, nranks * (NT >> 5));
                    finish();
                }
                if (!block_read(&sc.ctr->err)) phase_union(fp, sc, R.ss, inst, R.next_id, R.ss.ureg);
                // empty the global pair hash
                __syncthreads();
                const int ng = *(volatile int32_t*)&sc.ctr->n_pairs;
                for (int i = tid; i < ng; i += NT) {
                    const int t = R.ss.olist[i];
                    R.ss.okeys[t] = EMPTY_KEY;
                    R.ss.ocnt[t] = 0;
                }
            }
        }
        // the frame closes: its status and copy count for step (4) and the next
        // frame, the shared state emptied
        __syncthreads();
        if (!united && tid == 0) {
            const int err = *(volatile int32_t*)&sc.ctr->err;
            A.err = err;
            A.ncopies = err ? 0 : *(volatile int32_t*)R.ss.copy_n;
            A.next = *(volatile const int*)R.next_id;
            if (!err && *(volatile int32_t*)&sc.ctr->merges > 0) A.merged_any = 1;
            if (!blocked) A.all_changed = 1;  // the global path keeps no record of changed embeddings
        }
        for (int i = tid; i < ARH / 4; i += NT) {
            ((uint4*)A.rkey)[i] = make_uint4(UH_EMPTY, UH_EMPTY, UH_EMPTY, UH_EMPTY);
            ((int4*)A.rval)[i] = make_int4(RV_FREE, RV_FREE, RV_FREE, RV_FREE);
        }
        if (tid < MAX_MASKS) A.anchor[tid] = INT_MAX;
        if (tid == 0)
            A.ne = A.nlive = A.nloc = A.nroots = A.np = A.nsc = A.border = A.ovf = A.multi = A.ncopy = A.merges = 0;
        if (global_pairs)  // pairs may be left where the walk never came
            for (int i = tid; i < APH; i += NT) {
                A.pk[i] = EMPTY_KEY;
                A.pc[i] = A.pd[i] = 0;
            }
        if (blocked) prefetch(j + 1);
        __syncthreads();
        // (4) the winners' embeddings; on the global path also the new voxels
        //     into the counts
        if (!A.err) {
            const int nc = A.ncopies;
            if (nranks > 1 && nc > JOB_MIN) {
                give(JOB_COPY, nc, slot);
            } else {
                // from the last warp down: the first warps take the next
                // frame's items, so the two run side by side
                const Scratch va = st.view.frame(slot);
                for (int c = (NT >> 5) - 1 - wid; c < nc; c += NT >> 5) copy_embedding(R, sc, va, fp.D, c);
            }
            if (!united && !blocked)
                for (int m = tid; m < M; m += NT) {
                    const int n = sc.newcnt[m], rep = sc.segrep[m];
                    if (n && rep >= 0) atomicAdd((unsigned long long*)&inst.count[rep], (unsigned long long)n);
                }
        }
        if (tid == 0 && !united) {
            *R.ss.edge_n = 0;
            *R.ss.copy_n = 0;
        }
    }
    if (tid == 0) st.merged[g] = A.merged_any;
    if (nranks > 1) {
        give(JOB_END, 0, 0);
        finish();
    }
}

// After the batch's frames: every voxel of the absent-voxel hash whose first
// frame succeeded goes into its map with the instance that frame's lowest
// segment joined; the hash is emptied on the way.  Then the parent table of
// every map whose frames merged is flattened (each id to its root).
__global__ void k_commit(BatchScratch bs, SerialStep st, AbsentHash ah, int G)
{
    const int gtid = blockIdx.x * blockDim.x + threadIdx.x, gsz = gridDim.x * blockDim.x;
    const int lane = threadIdx.x & 31;
    const int n = *ah.n;
    for (int i0 = gtid & ~31; i0 < n; i0 += gsz) {
        const int i = i0 + lane;
        int g = -1, lab = -1;
        unsigned long long key = 0;
        if (i < n) {
            const int t = ah.list[i];
            const unsigned long long ak = ah.key[t];
            const int pv = ah.val[t];
            ah.key[t] = 0ull;
            ah.val[t] = INT_MAX;
            g = (int)(ak >> 54) - 1;
            key = ak & KEY54;
            const int slot = st.slot_of[g * st.J + (pv >> 9)];
            const Scratch sc = bs.frame(slot);
            if (sc.ctr->err == 0) lab = sc.segrep[(pv & 511) - 1];
        }
        const bool ins = lab >= 0;
        if (ins) {
            const VoxelTable vt = st.refs[g].vt;
            unsigned long long h = vt_home(key, vt.mask);
            for (unsigned long long pr = 0;; pr++) {
                const unsigned long long prev = atomicCAS(&vt.keys[h], EMPTY_KEY, key);
                if (prev == EMPTY_KEY) {
                    vt.labels[h] = lab;
                    break;
                }
                h = vt_next(h, pr + 1, vt.mask);
                if (pr > vt.mask) break;  // not reached: the batch's room was checked before it ran
            }
        }
        // one count update per map of the warp
        const unsigned act = __ballot_sync(0xffffffffu, ins);
        if (ins) {
            const unsigned grp = __match_any_sync(act, g);
            if (lane == __ffs(grp) - 1) atomicAdd(st.refs[g].vt.used, (unsigned long long)__popc(grp));
        }
    }
    for (int g = 0; g < G; g++) {
        if (!st.merged[g]) continue;
        const Instances inst = st.refs[g].inst;
        const int nid = *st.refs[g].next_id;
        for (int i = gtid; i < nid; i += gsz) inst.parent[i] = find_root(inst.parent, i);
    }
}

// ---- host launcher ----------------------------------------------------------------
// E4M3 scoring copies of instances [0, n) from their scoring master (one
// warp per instance), as the apply phase writes them
__global__ void k_e4m3_copies(Instances inst, int n, int D)
{
    const float* Sm = scoring_master(inst);
    const int Ds = scoring_dim(inst, D);
    for (int k = (blockIdx.x * blockDim.x + threadIdx.x) >> 5; k < n; k += (gridDim.x * blockDim.x) >> 5)
        e4m3_copy_row(Sm + (size_t)k * Ds, Ds, inst.E8 + (size_t)k * Ds, inst.Er + k);
}

int launch_e4m3_copies(const Instances& inst, int n, int D, cudaStream_t st)
{
    if (n <= 0 || !inst.E8) return 0;
    k_e4m3_copies<<<std::min((n + 7) / 8, 1216), 256, 0, st>>>(inst, n, D);
    return 1;
}

// Room check between a batch's two parts: per map of the batch, its voxel
// count (after every earlier batch) and the unique (segment, voxel) pairs of
// its frames in this batch, an upper bound of the voxels the batch inserts.
__global__ void k_room(const MapRefs* refs, int G, const int* slot_of, int J, BatchScratch bs,
                       unsigned long long* out)
{
    for (int g = blockIdx.x * blockDim.x + threadIdx.x; g < G; g += gridDim.x * blockDim.x) {
        unsigned long long inc = 0;
        for (int j = 0; j < J; j++) {
            const int slot = slot_of[g * J + j];
            if (slot >= 0) inc += (unsigned long long)max(bs.frame(slot).ctr->n_entries, 0);
        }
        out[2 * g] = *refs[g].vt.used;
        out[2 * g + 1] = inc;
    }
}

int launch_room(const MapRefs* refs, int G, const int* slot_of, int J, const BatchScratch& bs, unsigned long long* out,
                cudaStream_t st)
{
    k_room<<<(G + 127) / 128, 128, 0, st>>>(refs, G, slot_of, J, bs, out);
    return 1;
}

int launch_serial_begin(const MapRefs* refs, int G, cudaStream_t st)
{
    k_serial_begin<<<(G + 127) / 128, 128, 0, st>>>(refs, G);
    return 1;
}

// Blocks per map: the whole GPU for a single map, fewer per map as the maps
// of a batch multiply (they run side by side).
static int per_map(int full, int G, int least)
{
    return std::max(least, (full + G - 1) / G);
}

int launch_serial_step(const FrameParams* fps, const BatchScratch& bs, const SerialStep& st, int G, int phase,
                       cudaStream_t st_)
{
    const int q = st.cta_scale > 0 ? st.cta_scale : 4;  // quarters of the default CTA counts
    switch (phase) {
        case 0:
            k_overlap<<<dim3(per_map(76 * 2 * q / 2, G, 8), G), SER_THREADS, OV_SMEM, st_>>>(fps, bs, st);
            return 1;
        case 1:
            k_score<<<dim3(per_map(38 * q, G, 4), G), 256, 0, st_>>>(fps, bs, st);
            return 1;
        case 2:
            k_union<<<dim3(1, G), UNION_THREADS, UNION_SMEM, st_>>>(fps, bs, st);
            return 1;
        default:
            k_apply<<<dim3(per_map(76 * q, G, 8), G), 256, 0, st_>>>(fps, bs, st);
            return 1;
    }
}

int launch_lookup(const FrameParams* fps, const BatchScratch& bs, const BatchScratch& view, const MapRefs* refs,
                  const AbsentHash& ah, int S, int probe_width, cudaStream_t st)
{
    const dim3 grid(152, S);
    switch (probe_width) {
        case 2: k_lookup<2><<<grid, 256, 0, st>>>(fps, bs, refs, ah); break;
        case 4: k_lookup<4><<<grid, 256, 0, st>>>(fps, bs, refs, ah); break;
        case 8: k_lookup<8><<<grid, 256, 0, st>>>(fps, bs, refs, ah); break;
        default: k_lookup1<<<grid, LK_THREADS, 0, st>>>(fps, bs, refs, ah); break;
    }
    k_absent<<<dim3(38, S), 256, 0, st>>>(fps, bs, ah);
    k_items<<<dim3(16, S), 256, 0, st>>>(fps, bs, refs);
    k_gates<<<dim3(32, S), 256, 0, st>>>(fps, bs, view, refs);
    return 4;
}

size_t union_region_bytes_full() { return UNION_SMEM; }

// A CTA of this kernel fills an SM's registers, so the clusters of a batch's
// maps together leave most SMs to the kernels beside them. 16 maps of 240
// masks, us per frame of the call (association alone): one CTA per map 25.1
// (2.8), clusters of 8, 128 CTAs, 25.3 (2.2), of 4 24.5 (1.5), of 2 24.9 (2.1).
constexpr int ASSOC_CTAS = 64;
// CTAs per map of the association kernel that the device can place together
static int g_assoc_max_cluster = 1;  // set once by set_serial_kernel_attrs

static cudaLaunchConfig_t assoc_config(int G, int cluster, size_t smem, cudaLaunchAttribute* at, cudaStream_t s)
{
    cudaLaunchConfig_t cfg = {};
    at->id = cudaLaunchAttributeClusterDimension;
    at->val.clusterDim.x = cluster;
    at->val.clusterDim.y = 1;
    at->val.clusterDim.z = 1;
    cfg.gridDim = dim3(cluster, G);
    cfg.blockDim = dim3(ASSOC_THREADS);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    return cfg;
}

int launch_associate(const FrameParams* fps, const BatchScratch& bs, const SerialStep& st, int G, int cluster,
                     cudaStream_t s)
{
    int c = 1;
    while (2 * c <= std::min(cluster, g_assoc_max_cluster) && 2 * c * G <= ASSOC_CTAS) c *= 2;
    // A CTA of few maps keeps its SM to itself (a row of dependent steps that
    // shares its issue slots with stateless blocks runs 1.4 times as long):
    // it asks for all of the SM's shared memory.
    cudaLaunchAttribute at;
    const cudaLaunchConfig_t cfg = assoc_config(G, c, G <= 4 ? ASSOC_SMEM_ALONE : ASSOC_SMEM, &at, s);
    cudaLaunchKernelEx(&cfg, k_associate, fps, bs, st);
    return 1;
}

int launch_commit(const BatchScratch& bs, const SerialStep& st, const AbsentHash& ah, int G, cudaStream_t s)
{
    k_commit<<<152 * 2, 512, 0, s>>>(bs, st, ah, G);
    return 1;
}

cudaError_t set_serial_kernel_attrs()
{
    cudaError_t e = cudaFuncSetAttribute(k_union, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)UNION_SMEM);
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(k_associate, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)ASSOC_SMEM_ALONE);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(k_overlap, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)OV_SMEM);
    for (int c = 8; e == cudaSuccess && c > 1; c /= 2) {
        cudaLaunchAttribute at;
        const cudaLaunchConfig_t cfg = assoc_config(1, c, ASSOC_SMEM_ALONE, &at, nullptr);
        int n = 0;
        if (cudaOccupancyMaxActiveClusters(&n, k_associate, &cfg) == cudaSuccess && n > 0) {
            g_assoc_max_cluster = c;
            break;
        }
        cudaGetLastError();
    }
    return e;
}

}  // namespace disc

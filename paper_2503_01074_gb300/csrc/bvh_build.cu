// LBVH construction for the sonar geometry query (OceanSim Sec. III-A-2:
// the scene is queried by ray casting; this builds the acceleration structure).
//
//   1. validate + bounds              of box centres and of vertices; grid-stride, one set
//                                     of atomics per block
//   2. Morton codes                   63-bit keys (21 bits per axis) of triangles' box centres
//   3. radix sort                     stable LSD, 8-bit digits, three launches a digit
//   4. Karras hierarchy               one thread per internal node (Karras, HPG 2012)
//   5. climb                          leaf to root, the second visitor of a node goes on:
//                                     packed triangles, boxes (runs of <= kLeafMax
//                                     triangles become leaves), and the SAH programme
//                                     of both wide trees
//   6. wide collapse                  top-down, one launch a level for the 4-wide and
//                                     the 8-wide tree together; then the nodes
//                                     (128 or 256 bytes) in breadth-first order
//
// Every step reads the state that the one before left on the device, so the host
// waits twice: for the counts that size the nodes, and for the end.  Kernels after
// the validation return at once if it found a fault.  Measured, one upload: 2.1
// million triangles 4.1 ms with five launches a digit, three separate climbs, a
// host round trip per level and tree and a fresh mapping of the memory per build,
// now 1.03 ms; 183,360 triangles 2.2 -> 0.42 ms; 1,282 triangles 1.28 -> 0.32 ms;
// 33.6 million 33.7 -> 26.8 ms (there the scratch, 6 GB, is mapped anew each time).
#include <cuda_runtime.h>
#include <stdint.h>

#include <algorithm>
#include <string>

#include "sonar_internal.cuh"
#include "sonar_host.h"

namespace sonar {
namespace {

constexpr int kThreads = 256;
constexpr int kRsItems = 12;
constexpr int kRsTile = kThreads * kRsItems;   // keys per sort block (36 KB staged in shared memory)
constexpr int kLevels = 32;   // (3 kLevels + 1 > kStackMax): a deeper 4-wide tree is refused

// What the steps of a build pass on, in device memory.
struct BuildState {
    uint32_t flags;        // 1: index out of range, 2: negative material, 4: non-finite vertex
    int32_t max_mat;
    // ordered-encoded bounds: of the box centres (the Morton grid), of the triangles'
    // vertices (the padding)
    uint32_t lo[3], hi[3], vlo[3], vhi[3];
    int32_t height;        // of the binary hierarchy
    int32_t level[2][kLevels + 1];   // wide nodes per level of the 4-wide and 8-wide tree
};

__global__ void k_build_init(BuildState* st, int32_t* list4, int32_t* list8) {
    const int t = threadIdx.x;
    if (t < kLevels + 1) st->level[0][t] = st->level[1][t] = t == 0 ? 1 : 0;
    if (t < 3) { st->lo[t] = st->vlo[t] = 0xFFFFFFFFu; st->hi[t] = st->vhi[t] = 0u; }
    if (t == 0) {
        st->flags = 0u;
        st->max_mat = -1;
        st->height = 0;
        list4[0] = list8[0] = 0;   // both trees start at the binary root
    }
}

// ---------------------------------------------------------------------------
// 1. validation and bounds of the box centres and vertices
// ---------------------------------------------------------------------------

__device__ __forceinline__ float3 load_v(const float* v, int32_t i) {
    return make_float3(v[3 * (int64_t)i], v[3 * (int64_t)i + 1], v[3 * (int64_t)i + 2]);
}

// The centre of a triangle's box stands for it in the Morton order.  The two
// triangles of a heightfield cell have the same box seen from above, so they get
// neighbouring keys and become one leaf, and a grid of 2^k cells falls into a
// quadtree of its cells (the bounds are those of the centres too); their centroids
// lie a third of a cell apart, which paired triangles of different cells.  Ray cast
// of 64 frames of 32,768 rays by centroids -> by box centres 383 -> 360 us, of 32
// frames of 8,192 rays 79 -> 66, of 7.3 million rays of three sensor types 1132 ->
// 998, of 32 frames of 262,144 rays over 33.6 million triangles 1791 -> 1686.
__device__ __forceinline__ float3 box_centre(float3 p, float3 q, float3 r) {
    return make_float3(0.5f * fminf(p.x, fminf(q.x, r.x)) + 0.5f * fmaxf(p.x, fmaxf(q.x, r.x)),
                       0.5f * fminf(p.y, fminf(q.y, r.y)) + 0.5f * fmaxf(p.y, fmaxf(q.y, r.y)),
                       0.5f * fminf(p.z, fminf(q.z, r.z)) + 0.5f * fmaxf(p.z, fmaxf(q.z, r.z)));
}

__global__ void __launch_bounds__(kThreads) k_validate(const float* verts, int64_t nv, const int32_t* tris,
                                                       const int32_t* mat, int64_t nt, BuildState* st) {
    // bounds 0-2 of the box centres, 3-5 of the vertices
    __shared__ uint32_t s_lo[6], s_hi[6], s_flags;
    __shared__ int32_t s_mat;
    if (threadIdx.x < 6) { s_lo[threadIdx.x] = 0xFFFFFFFFu; s_hi[threadIdx.x] = 0u; }
    if (threadIdx.x == 0) { s_flags = 0; s_mat = -1; }
    __syncthreads();
    uint32_t lo[6], hi[6], flags = 0u;
#pragma unroll
    for (int k = 0; k < 6; ++k) { lo[k] = 0xFFFFFFFFu; hi[k] = 0u; }
    int32_t most_mat = -1;
    for (int64_t t = (int64_t)blockIdx.x * kThreads + threadIdx.x; t < nt; t += (int64_t)gridDim.x * kThreads) {
        const int32_t a = tris[3 * t], b = tris[3 * t + 1], c = tris[3 * t + 2];
        uint32_t f = 0;
        if (a < 0 || b < 0 || c < 0 || a >= nv || b >= nv || c >= nv) f |= 1u;
        const int32_t m = mat[t];
        if (m < 0) f |= 2u;
        most_mat = max(most_mat, m);
        if (!f) {
            const float3 p = load_v(verts, a), q = load_v(verts, b), r = load_v(verts, c);
            const bool fin = isfinite(p.x) && isfinite(p.y) && isfinite(p.z) && isfinite(q.x) &&
                             isfinite(q.y) && isfinite(q.z) && isfinite(r.x) && isfinite(r.y) &&
                             isfinite(r.z);
            if (!fin) {
                f |= 4u;
            } else {
                const float3 g = box_centre(p, q, r);
                const float most[6] = {g.x, g.y, g.z, fmaxf(p.x, fmaxf(q.x, r.x)), fmaxf(p.y, fmaxf(q.y, r.y)),
                                       fmaxf(p.z, fmaxf(q.z, r.z))};
                const float least[6] = {g.x, g.y, g.z, fminf(p.x, fminf(q.x, r.x)), fminf(p.y, fminf(q.y, r.y)),
                                        fminf(p.z, fminf(q.z, r.z))};
#pragma unroll
                for (int k = 0; k < 6; ++k) {
                    lo[k] = min(lo[k], ord_enc(least[k]));
                    hi[k] = max(hi[k], ord_enc(most[k]));
                }
            }
        }
        flags |= f;
    }
    for (int k = 0; k < 6; ++k) {
        lo[k] = __reduce_min_sync(0xFFFFFFFFu, lo[k]);
        hi[k] = __reduce_max_sync(0xFFFFFFFFu, hi[k]);
    }
    flags = __reduce_or_sync(0xFFFFFFFFu, flags);
    most_mat = __reduce_max_sync(0xFFFFFFFFu, most_mat);
    if ((threadIdx.x & 31) == 0) {
        for (int k = 0; k < 6; ++k) { atomicMin(&s_lo[k], lo[k]); atomicMax(&s_hi[k], hi[k]); }
        if (flags) atomicOr(&s_flags, flags);
        atomicMax(&s_mat, most_mat);
    }
    __syncthreads();
    if (threadIdx.x < 6) {
        const int k = threadIdx.x;
        atomicMin(k < 3 ? &st->lo[k] : &st->vlo[k - 3], s_lo[k]);
        atomicMax(k < 3 ? &st->hi[k] : &st->vhi[k - 3], s_hi[k]);
    }
    if (threadIdx.x == 0) {
        if (s_flags) atomicOr(&st->flags, s_flags);
        atomicMax(&st->max_mat, s_mat);
    }
}

// Box padding: covers the difference between the FP32 traversal ray and the
// exact ray, so that the FP32 box test never culls an exact hit.  That difference
// grows with the coordinates and the ranges in the scene, so the padding follows the
// vertices: a few coarse triangles about one middle (a seabed quad) would leave the
// bounds of their centres as small as the object between them.
__device__ __forceinline__ float box_pad(const BuildState* st) {
    float ext = 0.0f, mag = 0.0f;
    for (int a = 0; a < 3; ++a) {
        const float l = ord_dec(st->vlo[a]), h = ord_dec(st->vhi[a]);
        ext = fmaxf(ext, __fsub_rn(h, l));
        mag = fmaxf(mag, fmaxf(fabsf(l), fabsf(h)));
    }
    return fmaxf(__fmul_rn(1e-5f, fminf(__fadd_rn(ext, mag), 3.0e38f)), 1e-6f);   // finite at any extent
}

// ---------------------------------------------------------------------------
// 2. Morton codes
// ---------------------------------------------------------------------------

// The low 21 bits of v with two zero bits between neighbours.
__device__ __forceinline__ uint64_t spread3(uint32_t v) {
    uint64_t x = v & 0x1FFFFFu;
    x = (x | x << 32) & 0x001F00000000FFFFull;
    x = (x | x << 16) & 0x001F0000FF0000FFull;
    x = (x | x << 8) & 0x100F00F00F00F00Full;
    x = (x | x << 4) & 0x10C30C30C30C30C3ull;
    x = (x | x << 2) & 0x1249249249249249ull;
    return x;
}

__global__ void k_morton(const float* verts, const int32_t* tris, int64_t nt, const BuildState* st,
                         uint64_t* keys, uint32_t* vals) {
    const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= nt || st->flags) return;
    const float3 m = box_centre(load_v(verts, tris[3 * t]), load_v(verts, tris[3 * t + 1]), load_v(verts, tris[3 * t + 2]));
    const float c[3] = {m.x, m.y, m.z};
    // one scale for all axes (the largest extent): a flat scene (a seabed is
    // ~100 m wide and a few m high) then splits across its width first and in
    // height only at fine levels; per-axis scaling split it in height as early
    // as in x and y, into wide overlapping boxes (+30 % node visits per ray)
    uint32_t g[3];
    float ext = 0.0f;
    for (int a = 0; a < 3; ++a) ext = fmaxf(ext, ord_dec(st->hi[a]) - ord_dec(st->lo[a]));
    for (int a = 0; a < 3; ++a) {
        const float lo = ord_dec(st->lo[a]);
        float u = ext > 0.0f ? (c[a] - lo) / ext : 0.0f;
        u = fminf(fmaxf(u, 0.0f), 1.0f);
        g[a] = (uint32_t)fminf(u * 2097152.0f, 2097151.0f);    // 21 bits
    }
    keys[t] = spread3(g[0]) << 2 | spread3(g[1]) << 1 | spread3(g[2]);
    vals[t] = (uint32_t)t;
}

// ---------------------------------------------------------------------------
// 3. stable LSD radix sort (8-bit digits)
// ---------------------------------------------------------------------------

// Digit counts of every tile, hist[digit][tile].
__global__ void __launch_bounds__(kThreads) k_rs_hist(const uint64_t* keys, int64_t n, int shift,
                                                      const BuildState* st, uint32_t* hist, int tiles) {
    __shared__ uint32_t h[256];
    if (st->flags) return;
    h[threadIdx.x] = 0;
    __syncthreads();
    const int64_t base = (int64_t)blockIdx.x * kRsTile;
#pragma unroll
    for (int k = 0; k < kRsItems; ++k) {
        const int64_t i = base + k * kThreads + threadIdx.x;
        if (i < n) atomicAdd(&h[(keys[i] >> shift) & 255u], 1u);
    }
    __syncthreads();
    hist[(int64_t)threadIdx.x * tiles + blockIdx.x] = h[threadIdx.x];
}

// Exclusive scan of one value per thread of a block (s_warp: 32 words).
__device__ __forceinline__ uint32_t block_exclusive_scan(uint32_t v, uint32_t* s_warp, uint32_t& total) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    uint32_t x = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_up_sync(0xFFFFFFFFu, x, o);
        if (lane >= o) x += y;
    }
    if (lane == 31) s_warp[warp] = x;
    __syncthreads();
    uint32_t before = 0u;
    total = 0u;
    for (int w = 0; w < (int)(blockDim.x >> 5); ++w) {
        const uint32_t s = s_warp[w];
        if (w < warp) before += s;
        total += s;
    }
    __syncthreads();
    return before + x - v;
}

// One block per digit: its tiles' counts become their exclusive prefix, and
// total[digit] their sum.
__global__ void __launch_bounds__(kThreads) k_rs_rows(const BuildState* st, uint32_t* hist, int tiles, uint32_t* total) {
    __shared__ uint32_t s_warp[32];
    if (st->flags) return;
    uint32_t* row = hist + (int64_t)blockIdx.x * tiles;
    uint32_t carry = 0u;
    for (int base = 0; base < tiles; base += kThreads * 4) {
        uint32_t v[4], sum = 0u;
        const int i = base + 4 * threadIdx.x;
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            v[k] = i + k < tiles ? row[i + k] : 0u;
            sum += v[k];
        }
        uint32_t all;
        uint32_t run = carry + block_exclusive_scan(sum, s_warp, all);
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            if (i + k < tiles) row[i + k] = run;
            run += v[k];
        }
        carry += all;
    }
    if (threadIdx.x == 0) total[blockIdx.x] = carry;
}

// Stable scatter of a tile.  Each warp takes a run of consecutive keys, 32 at a
// time, and ranks them by digit against its own counters (lanes of equal digit
// in lane order); one pass over the counters turns them into places within the
// tile; the tile is then ordered in shared memory and written out as runs of
// consecutive places.  2.1 million keys: 23 us a digit, 34 us with a block-wide
// round (four barriers) per 256 keys and unordered stores.
__global__ void __launch_bounds__(kThreads) k_rs_scatter(const uint64_t* kin, const uint32_t* vin, uint64_t* kout,
                                                         uint32_t* vout, int64_t n, int shift, const BuildState* st,
                                                         const uint32_t* hist, const uint32_t* total, int tiles) {
    constexpr int kWarps = kThreads / 32;
    __shared__ uint64_t s_key[kRsTile];
    __shared__ uint32_t s_val[kRsTile];
    __shared__ uint32_t s_count[kWarps][256];   // per warp and digit: count, then first place in the tile
    __shared__ uint32_t s_to[256];              // per digit: output place of the tile's place 0
    __shared__ uint32_t s_warp[32];
    if (st->flags) return;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    for (int w = 0; w < kWarps; ++w) s_count[w][tid] = 0u;
    __syncthreads();
    const int64_t base = (int64_t)blockIdx.x * kRsTile;
    const int count = (int)min((int64_t)kRsTile, n - base);
    const int first = warp * (32 * kRsItems);
    const uint32_t lt = (1u << lane) - 1u;
    uint64_t key[kRsItems];
    uint32_t val[kRsItems], rank[kRsItems];
#pragma unroll
    for (int k = 0; k < kRsItems; ++k) {
        const int i = first + 32 * k + lane;
        key[k] = i < count ? kin[base + i] : 0ull;
        val[k] = i < count ? vin[base + i] : 0u;
    }
#pragma unroll
    for (int k = 0; k < kRsItems; ++k) {
        // lanes of equal digit by eight votes (a match instruction costs several
        // times as much: its unit serves one warp at a time)
        const bool ok = first + 32 * k + lane < count;
        const uint32_t digit = (uint32_t)((key[k] >> shift) & 255u);
        uint32_t peers = __ballot_sync(0xFFFFFFFFu, ok);
#pragma unroll
        for (int b = 0; b < 8; ++b) {
            const bool one = (digit >> b) & 1u;
            const uint32_t votes = __ballot_sync(0xFFFFFFFFu, one);
            peers &= one ? votes : ~votes;
        }
        const uint32_t before = __popc(peers & lt);
        const uint32_t have = ok ? s_count[warp][digit] : 0u;
        rank[k] = have + before;
        __syncwarp();
        if (ok && before == 0u) s_count[warp][digit] = have + __popc(peers);
        __syncwarp();
    }
    __syncthreads();
    {
        // thread = digit: places of the digit's first key of each warp within the tile
        uint32_t sum = 0u;
        for (int w = 0; w < kWarps; ++w) sum += s_count[w][tid];
        uint32_t all;
        uint32_t place = block_exclusive_scan(sum, s_warp, all);
        const uint32_t start = place;
        for (int w = 0; w < kWarps; ++w) {
            const uint32_t c = s_count[w][tid];
            s_count[w][tid] = place;
            place += c;
        }
        const uint32_t digit_base = block_exclusive_scan(total[tid], s_warp, all);
        s_to[tid] = digit_base + hist[(int64_t)tid * tiles + blockIdx.x] - start;
    }
    __syncthreads();
#pragma unroll
    for (int k = 0; k < kRsItems; ++k) {
        if (first + 32 * k + lane < count) {
            const uint32_t at = s_count[warp][(key[k] >> shift) & 255u] + rank[k];
            s_key[at] = key[k];
            s_val[at] = val[k];
        }
    }
    __syncthreads();
    for (int i = tid; i < count; i += kThreads) {
        const uint64_t x = s_key[i];
        const uint32_t to = s_to[(x >> shift) & 255u] + (uint32_t)i;
        kout[to] = x;
        vout[to] = s_val[i];
    }
}

// ---------------------------------------------------------------------------
// 4. Karras hierarchy
// ---------------------------------------------------------------------------

// Length of the common prefix of keys i and j; equal keys are told apart by
// their indices (64 + common prefix of i and j); -1 outside [0, n).
__device__ __forceinline__ int delta(const uint64_t* k, int64_t n, int64_t i, int64_t j) {
    if (j < 0 || j >= n) return -1;
    const uint64_t a = k[i], b = k[j];
    if (a != b) return __clzll((long long)(a ^ b));
    return 64 + __clz((int)((uint32_t)i ^ (uint32_t)j));
}

// up[c] of internal node c, up[n - 1 + i] of leaf i: 2 * parent + side (-1: the
// root); range[p] = covered leaves [lo, hi].
__global__ void k_karras(const uint64_t* keys, int64_t n, const BuildState* st, int32_t* up, int2* range) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n - 1 || st->flags) return;
    const int d = delta(keys, n, i, i + 1) > delta(keys, n, i, i - 1) ? 1 : -1;
    const int dmin = delta(keys, n, i, i - d);
    int64_t lmax = 2;
    while (delta(keys, n, i, i + lmax * d) > dmin) lmax <<= 1;
    int64_t l = 0;
    for (int64_t t = lmax >> 1; t >= 1; t >>= 1)
        if (delta(keys, n, i, i + (l + t) * d) > dmin) l += t;
    const int64_t j = i + l * d;
    const int dnode = delta(keys, n, i, j);
    int64_t s = 0, t = l;
    do {
        t = (t + 1) >> 1;
        if (delta(keys, n, i, i + (s + t) * d) > dnode) s += t;
    } while (t > 1);
    const int64_t gamma = i + s * d + (d < 0 ? -1 : 0);
    const int64_t lo = i < j ? i : j, hi = i < j ? j : i;
    up[lo == gamma ? (n - 1) + gamma : gamma] = (int32_t)(2 * i);
    up[hi == gamma + 1 ? (n - 1) + gamma + 1 : gamma + 1] = (int32_t)(2 * i + 1);
    range[i] = make_int2((int)lo, (int)hi);
    if (i == 0) up[0] = -1;
}

// ---------------------------------------------------------------------------
// 5. climb: boxes and the SAH programme of both wide trees
// ---------------------------------------------------------------------------

__device__ __forceinline__ float half_area(float4 lo, float4 hi) {
    const float dx = hi.x - lo.x, dy = hi.y - lo.y, dz = hi.z - lo.z;
    return dx * dy + dy * dz + dz * dx;
}

static_assert(kLeafMax == 2, "k_climb starts at single triangles and at pairs");
constexpr float kSahTri = 0.7f;   // SAH cost of a triangle test relative to a wide-node visit
// The programme, bottom-up over the binary tree: cost(x, k) is the least SAH cost
// of the subtree at side x (a leaf run or a binary node) when it may take up to k
// (1..W) child slots of the W-wide node above it.  One slot: the side itself, a
// leaf (area x triangles x kSahTri) or a W-wide node (area + the cost of its
// subtree spread over W slots); k slots: the better of that and opening the node,
// its two sides sharing the k slots.  dec[p] keeps, for k = 2..W, the split of
// p's slots between its sides (kSplitBits each, from bit 0) and whether p is
// better opened (one bit each above the splits).  cost holds W floats per binary
// node.
template <int W>
struct Wide {
    static constexpr int kSplitBits = W == 8 ? 3 : 2;
    static constexpr int kOpenBit = kSplitBits * (W - 1);
    __host__ __device__ static constexpr int split(int32_t d, int k) {
        return (d >> (kSplitBits * (k - 2))) & ((1 << kSplitBits) - 1);
    }
    __host__ __device__ static constexpr bool opened(int32_t d, int k) { return (d >> (kOpenBit + k - 2)) & 1; }
};

// A node's cost per slot count from its sides' (a0, a1 [W]) and its own area;
// returns the decisions.
template <int W>
__device__ __forceinline__ int32_t programme(const float (&a0)[W], const float (&a1)[W], float area, float (&out)[W]) {
    float open[W + 1];
    int split[W + 1];
#pragma unroll
    for (int m = 2; m <= W; ++m) {
        open[m] = 3.0e38f;
        split[m] = 1;
#pragma unroll
        for (int j = 1; j < m; ++j) {
            const float v = a0[j - 1] + a1[m - j - 1];
            if (v < open[m]) { open[m] = v; split[m] = j; }
        }
    }
    const float wide = area + open[W];   // one slot: a W-wide node, its two sides sharing the W slots
    out[0] = wide;
    int32_t d = 0;
#pragma unroll
    for (int k = 2; k <= W; ++k) {
        const bool opened = open[k] < wide;
        out[k - 1] = opened ? open[k] : wide;
        d |= (split[k] << (Wide<W>::kSplitBits * (k - 2))) | (opened ? (1 << (Wide<W>::kOpenBit + k - 2)) : 0);
    }
    return d;
}

// The costs of one side: a leaf run's for every slot count, or a node's stored ones.
template <int W>
__device__ __forceinline__ void side_costs(float4 lo, float4 hi, const float* cost, float (&a)[W]) {
    const int32_t h = __float_as_int(lo.w);
    if (h < 0) {
        const float v = half_area(lo, hi) * kSahTri * (float)(((~h) & 7) + 1);
#pragma unroll
        for (int k = 0; k < W; ++k) a[k] = v;
        return;
    }
#pragma unroll
    for (int k = 0; k < W; k += 4) {
        const float4 v = __ldcg(reinterpret_cast<const float4*>(cost + (int64_t)W * h + k));
        a[k] = v.x; a[k + 1] = v.y; a[k + 2] = v.z; a[k + 3] = v.w;
    }
}

// One thread per leaf i: writes its packed triangle and hands its padded box to
// its parent's slot of `pairs` (pairs[2 x] = (lo, handle), pairs[2 x + 1] = (hi,
// height) of side x = 2 * parent + side); the second of a node's two visitors
// unites the boxes, runs the programme and climbs on with the node's own box.
// Padded boxes unite to the padded union (rounding is monotone).
// Bound by the latency of a level (an atomic, a fence and the sides' loads), some
// 20 levels of it: one climb (343 us for 2.1 million triangles) does what refit,
// packing and the programmes of the two trees took four passes for (750 us).
__global__ void __launch_bounds__(kThreads) k_climb(const float* verts, const int32_t* tris, const int32_t* mat,
                                                    const uint32_t* vals, int64_t n, BuildState* st,
                                                    const int32_t* up, const int2* range, int32_t* visits,
                                                    float4* out, int32_t* mat_orig, float4* pairs, float* cost4,
                                                    float* cost8, int4* info) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n || st->flags) return;
    const uint32_t o = vals[i];
    const float3 p = load_v(verts, tris[3 * (int64_t)o]), q = load_v(verts, tris[3 * (int64_t)o + 1]),
                 r = load_v(verts, tris[3 * (int64_t)o + 2]);
    const int32_t m = mat[o];
    out[3 * i] = make_float4(p.x, p.y, p.z, __int_as_float(m));
    out[3 * i + 1] = make_float4(q.x, q.y, q.z, __uint_as_float(o));
    out[3 * i + 2] = make_float4(r.x, r.y, r.z, 0.0f);
    mat_orig[o] = m;
    if (n <= kLeafMax) return;   // the scene is one leaf
    const float pad = box_pad(st);
    float4 lo = make_float4(fminf(p.x, fminf(q.x, r.x)) - pad, fminf(p.y, fminf(q.y, r.y)) - pad,
                            fminf(p.z, fminf(q.z, r.z)) - pad, __int_as_float(leaf_handle((int32_t)i, 1)));
    float4 hi = make_float4(fmaxf(p.x, fmaxf(q.x, r.x)) + pad, fmaxf(p.y, fmaxf(q.y, r.y)) + pad,
                            fmaxf(p.z, fmaxf(q.z, r.z)) + pad, __int_as_float(0));
    int32_t x = up[(n - 1) + i];
    // a run of two triangles (one leaf of the wide trees): the left one's thread
    // takes both and starts above their node, whose sides nothing reads
    const int2 around = range[x >> 1];
    if (around.y - around.x + 1 == kLeafMax) {
        if (x & 1) return;
        const uint32_t o2 = vals[i + 1];
        const float3 p2 = load_v(verts, tris[3 * (int64_t)o2]), q2 = load_v(verts, tris[3 * (int64_t)o2 + 1]),
                     r2 = load_v(verts, tris[3 * (int64_t)o2 + 2]);
        lo = make_float4(fminf(lo.x, fminf(p2.x, fminf(q2.x, r2.x)) - pad), fminf(lo.y, fminf(p2.y, fminf(q2.y, r2.y)) - pad),
                         fminf(lo.z, fminf(p2.z, fminf(q2.z, r2.z)) - pad), __int_as_float(leaf_handle(around.x, kLeafMax)));
        hi = make_float4(fmaxf(hi.x, fmaxf(p2.x, fmaxf(q2.x, r2.x)) + pad), fmaxf(hi.y, fmaxf(p2.y, fmaxf(q2.y, r2.y)) + pad),
                         fmaxf(hi.z, fmaxf(p2.z, fmaxf(q2.z, r2.z)) + pad), __int_as_float(1));
        x = up[x >> 1];
    }
    while (x >= 0) {
        __stcg(pairs + 2 * (int64_t)x, lo);
        __stcg(pairs + 2 * (int64_t)x + 1, hi);
        __threadfence();
        const int32_t node = x >> 1;
        if (atomicAdd(&visits[node], 1) == 0) return;   // the other child is still on its way
        __threadfence();
        const float4 l2 = __ldcg(pairs + 2 * (int64_t)(x ^ 1)), h2 = __ldcg(pairs + 2 * (int64_t)(x ^ 1) + 1);
        const bool left = (x & 1) == 0;
        const float4 l0 = left ? lo : l2, h0 = left ? hi : h2, l1 = left ? l2 : lo, h1 = left ? h2 : hi;
        const int height = 1 + max(__float_as_int(h0.w), __float_as_int(h1.w));
        lo = make_float4(fminf(l0.x, l1.x), fminf(l0.y, l1.y), fminf(l0.z, l1.z), 0.0f);
        hi = make_float4(fmaxf(h0.x, h1.x), fmaxf(h0.y, h1.y), fmaxf(h0.z, h1.z), __int_as_float(height));
        const float area = half_area(lo, hi);
        int32_t d4;
        {
            float a0[4], a1[4], c[4];
            side_costs<4>(l0, h0, cost4, a0);
            side_costs<4>(l1, h1, cost4, a1);
            d4 = programme<4>(a0, a1, area, c);
            __stcg(reinterpret_cast<float4*>(cost4 + 4 * (int64_t)node), make_float4(c[0], c[1], c[2], c[3]));
        }
        float a0[8], a1[8], c[8];
        side_costs<8>(l0, h0, cost8, a0);
        side_costs<8>(l1, h1, cost8, a1);
        const int32_t d8 = programme<8>(a0, a1, area, c);
        info[node] = make_int4(__float_as_int(l0.w), __float_as_int(l1.w), d4, d8);
        __stcg(reinterpret_cast<float4*>(cost8 + 8 * (int64_t)node), make_float4(c[0], c[1], c[2], c[3]));
        __stcg(reinterpret_cast<float4*>(cost8 + 8 * (int64_t)node + 4), make_float4(c[4], c[5], c[6], c[7]));
        lo.w = __int_as_float(node);
        x = up[node];
        if (x < 0) st->height = height;
    }
}

// ---------------------------------------------------------------------------
// 6. wide collapse
// ---------------------------------------------------------------------------

// The children of the wide node rooted at binary node p from the programme: p's
// W slots split between its sides, each side taking its slots as a leaf, a
// W-wide node (one slot) or opened further.  Every side keeps at least one slot,
// so at most W sides are pending at once.  side[0..W): sides in slot order, -1
// empty; handle: the handles of those sides.  info[p] = (handles of p's sides,
// decisions of the 4-wide and of the 8-wide programme): one load per opened node.
template <int W>
__device__ __forceinline__ int pick_children(int32_t p, const int4* info, int32_t (&side)[W], int32_t (&handle)[W]) {
    int cnt = 0, nw = 0;
    int32_t ws[W + 1], wh[W + 1];   // work list of (side, handle, slots)
    int wk[W + 1];
    auto open = [&](int32_t q, int k) {
        const int4 v = __ldg(info + q);
        const int j = Wide<W>::split(W == 4 ? v.z : v.w, k);
        ws[nw] = 2 * q + 1; wh[nw] = v.y; wk[nw++] = k - j;
        ws[nw] = 2 * q;     wh[nw] = v.x; wk[nw++] = j;
    };
    open(p, W);
    while (nw > 0) {
        --nw;
        const int32_t x = ws[nw], h = wh[nw];
        const int k = wk[nw];
        if (h >= 0 && k >= 2) {
            const int4 v = __ldg(info + h);
            if (Wide<W>::opened(W == 4 ? v.z : v.w, k)) {
                open(h, k);
                continue;
            }
        }
        side[cnt] = x;
        handle[cnt++] = h;
    }
    return cnt;
}

// Entries of the level lists before level `upto` of tree t.
__device__ __forceinline__ int level_base(const BuildState* st, int t, int upto) {
    int b = 0;
    for (int k = 0; k < upto; ++k) b += st->level[t][k];
    return b;
}

// One level: the wide nodes list[base .. base + level[l]) (entry = the node's
// index, value = the binary node it is rooted at) append their internal children
// to the next level, each node's side by side, and keep the first one's index.
// Places come from one atomic per warp: the order of a level's nodes may differ
// from build to build, which no result depends on.
template <int W>
__device__ void mark_level(int t, int l, BuildState* st, const int4* info, int32_t* list, int32_t* first_child) {
    const int lane = threadIdx.x & 31;
    const int count = st->level[t][l], base = level_base(st, t, l), next = base + count;
    const int stride = gridDim.x * blockDim.x;
    for (int e0 = blockIdx.x * blockDim.x + (threadIdx.x & ~31); e0 < count; e0 += stride) {
        const int e = e0 + lane;
        int32_t side[W], h[W];
        int n = 0, ni = 0;
        if (e < count) {
            n = pick_children<W>(list[base + e], info, side, h);
            for (int k = 0; k < n; ++k) ni += h[k] >= 0;
        }
        int x = ni;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int y = __shfl_up_sync(0xFFFFFFFFu, x, o);
            if (lane >= o) x += y;
        }
        int at = 0;
        if (lane == 31) at = x > 0 ? atomicAdd(&st->level[t][l + 1], x) : 0;
        at = next + __shfl_sync(0xFFFFFFFFu, at, 31) + x - ni;
        if (e < count) {
            first_child[base + e] = at;
            for (int k = 0; k < n; ++k)
                if (h[k] >= 0) list[at++] = h[k];
        }
    }
}

__global__ void __launch_bounds__(kThreads) k_mark(int l, BuildState* st, const int4* info, int32_t* list4,
                                                   int32_t* list8, int32_t* first4, int32_t* first8) {
    if (st->flags) return;
    if (blockIdx.y == 0) mark_level<4>(0, l, st, info, list4, first4);
    else mark_level<8>(1, l, st, info, list8, first8);
}

// Writes wide node e.  Empty slots hold a point at +inf that no ray enters and the
// empty handle.  The 4-wide layout keeps the planes axis by axis, the 8-wide one
// child by child (sonar_internal.cuh).
template <int W>
__device__ void write_node(int64_t e, const int32_t* list, const int32_t* first_child, const float4* pairs,
                           const int4* info, float4* nodes) {
    int32_t side[W], handle[W];
    const int n = pick_children<W>(list[e], info, side, handle);
    int32_t r = first_child[e];
    const float inf = __int_as_float(0x7F800000);
    // centre and half-width: the half-width rounded up, so that the box only grows
    float c[3][W], h[3][W];
    int32_t hs[W];
#pragma unroll
    for (int k = 0; k < W; ++k) {
        c[0][k] = c[1][k] = c[2][k] = inf;
        h[0][k] = h[1][k] = h[2][k] = 0.0f;
        hs[k] = kEmpty;
        if (k >= n) continue;
        const float4 l4 = pairs[2 * (int64_t)side[k]], h4 = pairs[2 * (int64_t)side[k] + 1];
        const float lo[3] = {l4.x, l4.y, l4.z}, hi[3] = {h4.x, h4.y, h4.z};
        for (int a = 0; a < 3; ++a) {
            c[a][k] = 0.5f * lo[a] + 0.5f * hi[a];
            h[a][k] = fmaxf(__fsub_ru(hi[a], c[a][k]), __fsub_ru(c[a][k], lo[a]));
        }
        hs[k] = handle[k] >= 0 ? r++ : handle[k];
    }
    float4* o = nodes + 2 * W * e;
    if constexpr (W == 4) {
        for (int a = 0; a < 3; ++a) {
            o[2 * a] = make_float4(c[a][0], c[a][1], c[a][2], c[a][3]);
            o[2 * a + 1] = make_float4(h[a][0], h[a][1], h[a][2], h[a][3]);
        }
        o[6] = make_float4(__int_as_float(hs[0]), __int_as_float(hs[1]), __int_as_float(hs[2]), __int_as_float(hs[3]));
        o[7] = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
    } else {
#pragma unroll
        for (int k = 0; k < W; ++k) {
            o[2 * k] = make_float4(c[0][k], h[0][k], c[1][k], h[1][k]);
            o[2 * k + 1] = make_float4(c[2][k], h[2][k], __int_as_float(hs[k]), 0.0f);
        }
    }
}

__global__ void __launch_bounds__(kThreads) k_write_nodes(int64_t n4, int64_t n8, const float4* pairs,
                                                          const int4* info, const int32_t* list4,
                                                          const int32_t* list8, const int32_t* first4,
                                                          const int32_t* first8, float4* nodes, float4* nodes8) {
    const int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (blockIdx.y == 0) {
        if (e < n4) write_node<4>(e, list4, first4, pairs, info, nodes);
    } else if (e < n8) {
        write_node<8>(e, list8, first8, pairs, info, nodes8);
    }
}

inline unsigned blocks_for(int64_t n, int t) { return (unsigned)((n + t - 1) / t); }

}  // namespace

// Temporary device buffers of one build: parts of one allocation from the
// context's pool, returned to it in stream order on exit.
struct BuildScratch {
    cudaStream_t st;
    char* base = nullptr;
    size_t used = 0;
    template <class T>
    size_t reserve(size_t count) {   // offset of a part (256-byte aligned)
        const size_t at = used;
        used += (count * sizeof(T) + 255) / 256 * 256;
        return at;
    }
    template <class T>
    T* at(size_t offset) const { return reinterpret_cast<T*>(base + offset); }
    ~BuildScratch() {
        if (base) cudaFreeAsync(base, st);
    }
};

sonar_status build_scene(const float* verts, int64_t nv, const int32_t* tris, const int32_t* mat,
                         int64_t nt, int sm_count, cudaMemPool_t pool, cudaStream_t st, SceneStore* out,
                         std::string* msg) {
    *out = SceneStore{};
    out->n_tris = nt;
    out->max_mat = -1;
    if (nt == 0) {
        out->root = kEmpty;
        return SONAR_OK;
    }
    const int64_t n = nt;
    const bool tree = n > kLeafMax;
    const int tiles = (int)blocks_for(n, kRsTile);
    BuildScratch S{st};
    const size_t o_state = S.reserve<BuildState>(1);
    const size_t o_k0 = S.reserve<uint64_t>(n), o_k1 = S.reserve<uint64_t>(n);
    const size_t o_v0 = S.reserve<uint32_t>(n), o_v1 = S.reserve<uint32_t>(n);
    const size_t o_hist = S.reserve<uint32_t>(256ll * tiles), o_total = S.reserve<uint32_t>(256);
    const size_t o_up = S.reserve<int32_t>(2 * n), o_range = S.reserve<int2>(n), o_visits = S.reserve<int32_t>(n);
    const size_t o_pairs = S.reserve<float4>(4 * n);
    const size_t o_cost4 = S.reserve<float>(4 * n), o_cost8 = S.reserve<float>(8 * n);
    const size_t o_info = S.reserve<int4>(n);
    const size_t o_list4 = S.reserve<int32_t>(n), o_list8 = S.reserve<int32_t>(n);
    const size_t o_first4 = S.reserve<int32_t>(n), o_first8 = S.reserve<int32_t>(n);
    cudaError_t e = cudaMallocFromPoolAsync((void**)&S.base, S.used, pool, st);
    if (e != cudaSuccess) {
        S.base = nullptr;
        cudaGetLastError();
        *msg = "out of device memory (build scratch)";
        return SONAR_ERR_OOM;
    }
    // persistent buffers: triangles now, nodes once their count is known
    e = cudaMallocFromPoolAsync((void**)&out->tris, sizeof(float4) * 3 * n, pool, st);
    if (e == cudaSuccess) e = cudaMallocFromPoolAsync((void**)&out->mat_orig, sizeof(int32_t) * n, pool, st);
    if (e != cudaSuccess) {
        cudaGetLastError();
        *msg = "out of device memory (scene)";
        return SONAR_ERR_OOM;
    }
    out->bytes = sizeof(float4) * 3 * n + sizeof(int32_t) * n;
    BuildState* state = S.at<BuildState>(o_state);
    uint64_t *k0 = S.at<uint64_t>(o_k0), *k1 = S.at<uint64_t>(o_k1);
    uint32_t *v0 = S.at<uint32_t>(o_v0), *v1 = S.at<uint32_t>(o_v1);
    uint32_t *hist = S.at<uint32_t>(o_hist), *total = S.at<uint32_t>(o_total);
    int32_t* up = S.at<int32_t>(o_up);
    int2* range = S.at<int2>(o_range);
    float4* pairs = S.at<float4>(o_pairs);
    int4* info = S.at<int4>(o_info);
    int32_t *list4 = S.at<int32_t>(o_list4), *list8 = S.at<int32_t>(o_list8);
    int32_t *first4 = S.at<int32_t>(o_first4), *first8 = S.at<int32_t>(o_first8);

    k_build_init<<<1, 64, 0, st>>>(state, list4, list8);
    k_validate<<<(unsigned)std::min<int64_t>(blocks_for(n, kThreads), 4ll * sm_count), kThreads, 0, st>>>(
        verts, nv, tris, mat, n, state);
    k_morton<<<blocks_for(n, kThreads), kThreads, 0, st>>>(verts, tris, n, state, k0, v0);
    for (int shift = 0; shift < 63; shift += 8) {
        k_rs_hist<<<tiles, kThreads, 0, st>>>(k0, n, shift, state, hist, tiles);
        k_rs_rows<<<256, kThreads, 0, st>>>(state, hist, tiles, total);
        k_rs_scatter<<<tiles, kThreads, 0, st>>>(k0, v0, k1, v1, n, shift, state, hist, total, tiles);
        std::swap(k0, k1);
        std::swap(v0, v1);
    }
    if (tree) {
        k_karras<<<blocks_for(n - 1, kThreads), kThreads, 0, st>>>(k0, n, state, up, range);
        e = cudaMemsetAsync(S.at<int32_t>(o_visits), 0, sizeof(int32_t) * (n - 1), st);
    }
    k_climb<<<blocks_for(n, kThreads), kThreads, 0, st>>>(verts, tris, mat, v0, n, state, up, range,
                                                          S.at<int32_t>(o_visits), out->tris, out->mat_orig, pairs,
                                                          S.at<float>(o_cost4), S.at<float>(o_cost8), info);
    // levels: a 4-wide tree over a surface has about 0.65 log2(n) of them; a few
    // more at a time for a tree that is deeper
    int guess = 2;
    for (int64_t m = n; m > 1; m >>= 1) ++guess;
    guess = guess * 2 / 3;
    BuildState hs{};
    int64_t count[2] = {0, 0};
    int depth[2] = {0, 0};
    const unsigned mark_blocks = (unsigned)std::min<int64_t>(blocks_for(n, 4 * kThreads), 4ll * sm_count);
    for (int l = 0; e == cudaSuccess;) {
        const int stop = tree ? std::min(kLevels, l == 0 ? guess : l + 4) : 0;
        for (; l < stop; ++l)
            k_mark<<<dim3(mark_blocks, 2), kThreads, 0, st>>>(l, state, info, list4, list8, first4, first8);
        e = cudaMemcpyAsync(&hs, state, sizeof hs, cudaMemcpyDeviceToHost, st);
        if (e == cudaSuccess) e = cudaStreamSynchronize(st);
        if (!tree || hs.flags || l >= kLevels || hs.level[0][l] + hs.level[1][l] == 0) break;
    }
    if (e == cudaSuccess) e = cudaGetLastError();
    if (e != cudaSuccess) { *msg = std::string("build failed: ") + cudaGetErrorString(e); return SONAR_ERR_CUDA; }
    if (hs.flags & 1u) { *msg = "triangle vertex index out of range"; return SONAR_ERR_ARG; }
    if (hs.flags & 2u) { *msg = "negative material id"; return SONAR_ERR_ARG; }
    if (hs.flags & 4u) { *msg = "non-finite vertex coordinate"; return SONAR_ERR_ARG; }
    out->max_mat = hs.max_mat;
    if (!tree) {
        out->root = leaf_handle(0, (int32_t)n);
        return SONAR_OK;
    }
    out->height = hs.height;
    for (int t = 0; t < 2; ++t)
        for (int l = 0; l <= kLevels; ++l) {
            count[t] += hs.level[t][l];
            if (hs.level[t][l] > 0) depth[t] = l + 1;
        }
    // a visit pushes at most W - 1 children, one visit per level of the W-wide
    // tree on any path: the walk never needs more than (W - 1) depth + 1
    // entries.  An 8-wide tree too deep for the stack is not kept (rays then
    // walk the 4-wide one).
    if (3 * depth[0] + 1 > kStackMax) {
        *msg = "hierarchy too deep for the traversal stack (4-wide depth " + std::to_string(depth[0]) + ")";
        return SONAR_ERR_ARG;
    }
    const bool wide = 7 * depth[1] + 1 <= kStackMax;
    e = cudaMallocFromPoolAsync((void**)&out->nodes, sizeof(float4) * 8 * count[0], pool, st);
    if (e == cudaSuccess && wide) e = cudaMallocFromPoolAsync((void**)&out->nodes8, sizeof(float4) * 16 * count[1], pool, st);
    if (e != cudaSuccess) {
        cudaGetLastError();
        *msg = "out of device memory (scene)";
        return SONAR_ERR_OOM;
    }
    out->n_pairs = count[0];
    out->n_nodes8 = wide ? count[1] : 0;
    out->bytes += sizeof(float4) * (8 * out->n_pairs + 16 * out->n_nodes8);
    out->root = 0;
    k_write_nodes<<<dim3(blocks_for(count[0], kThreads), wide ? 2 : 1), kThreads, 0, st>>>(
        count[0], out->n_nodes8, pairs, info, list4, list8, first4, first8, out->nodes, out->nodes8);
    e = cudaGetLastError();
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    if (e != cudaSuccess) { *msg = std::string("build failed: ") + cudaGetErrorString(e); return SONAR_ERR_CUDA; }
    return SONAR_OK;
}

// The caller has synchronised the device: nothing reads the scene any more.
void free_scene(SceneStore* s) {
    for (void* p : {(void*)s->nodes, (void*)s->nodes8, (void*)s->tris, (void*)s->mat_orig})
        if (p) cudaFreeAsync(p, 0);
    *s = SceneStore{};
}

}  // namespace sonar

// Sonar ray casting (OceanSim, arXiv 2503.01074, Sec. III-A-2).
//
// k_trig              float-float sin/cos tables of each sensor's beam azimuths
//                     and elevations (FP64 once per sensor).
// k_trace             one ray per lane, warps on compact beam x elevation
//                     patches: ray generation -> closest hit (LBVH walk,
//                     Moller-Trumbore) -> range/azimuth bin -> 16-byte hit record.
//                     The STATS variant counts node visits and triangle tests and
//                     marks the nodes and triangles it touches.
// k_trace_group       the same with eight or four lanes per ray, for small launches.
// k_popcount          counts the marked nodes and triangles.
//
// Ray casting precision: the walk and the triangle tests run in FP32.  A test
// whose barycentric or distance outcome lies inside a certified FP32 error
// bound, and any two candidates within 2e-5 t of each other, are re-decided
// exactly in float-float arithmetic (about 48 significant bits, on the FP32
// pipes) against the exact ray, whose direction comes from per-sensor sin/cos
// tables computed in FP64 once; hit decisions therefore agree with an FP64
// reference except for genuinely ambiguous rays.
#include <cuda_runtime.h>
#include <math_constants.h>
#include <stdint.h>

#include "sonar_host.h"
#include "sonar_internal.cuh"
#include "devmath.cuh"

namespace sonar {
namespace {

// ---------------------------------------------------------------------------
// rays
// ---------------------------------------------------------------------------

__device__ __forceinline__ float3 ray_dir32(const SensorDev& s, int i, int j) {
    const float phi = fmaf((float)i + 0.5f, s.hfov / (float)s.nb, -0.5f * s.hfov);
    const float th = fmaf((float)j + 0.5f, s.vfov / (float)s.ne, -0.5f * s.vfov);
    float sp, cp, st, ct;
    sincosf(phi, &sp, &cp);
    sincosf(th, &st, &ct);
    const float dx = sp * ct, dy = cp * ct, dz = st;
    const float3 w = f3(fmaf(s.rot[0], dx, fmaf(s.rot[1], dy, s.rot[2] * dz)),
                        fmaf(s.rot[3], dx, fmaf(s.rot[4], dy, s.rot[5] * dz)),
                        fmaf(s.rot[6], dx, fmaf(s.rot[7], dy, s.rot[8] * dz)));
    const float inv = 1.0f / sqrtf(dot3(w, w));
    return f3(w.x * inv, w.y * inv, w.z * inv);
}

// The exact ray of (i, j) in float-float, unnormalised: w = R ds with ds from
// the sensor's float-float sine/cosine tables (beam i, elevation j).  The hit
// decisions below only use signs and ratios, which a positive scale leaves
// unchanged.
__device__ __forceinline__ void ray_dir_ff(const SensorDev& s, int i, int j, ff w[3]) {
    const float4 bp = s.trig[i], el = s.trig[s.nb + j];
    const ff sp{bp.x, bp.y}, cp{bp.z, bp.w}, st{el.x, el.y}, ct{el.z, el.w};
    const ff ds[3] = {ff_mul(sp, ct), ff_mul(cp, ct), st};
    for (int a = 0; a < 3; ++a)
        w[a] = ff_add(ff_add(ff_mulf(ds[0], s.rot[3 * a]), ff_mulf(ds[1], s.rot[3 * a + 1])),
                      ff_mulf(ds[2], s.rot[3 * a + 2]));
}


// ---------------------------------------------------------------------------
// closest hit: LBVH walk with a short stack
// ---------------------------------------------------------------------------

// The exact decisions, out of line (rarely needed; they would otherwise add
// registers to the FP32 walk) and in float-float on the FP32 pipes.
//
// exact_hit: does the exact ray of (i, j) hit the triangle?  *t = the hit
// distance in FP32.
__device__ __noinline__ bool exact_hit(const SensorDev& s, int i, int j, float4 a, float4 b, float4 c, float* t) {
    ff w[3];
    ray_dir_ff(s, i, j, w);
    const float o[3] = {s.pos[0], s.pos[1], s.pos[2]};
    ff D, T;
    if (!mt_ff(o, w, a, b, c, D, T)) return false;
    const float len = sqrtf(w[0].hi * w[0].hi + w[1].hi * w[1].hi + w[2].hi * w[2].hi);
    *t = (T.hi / D.hi) * len;
    return true;
}

// exact_closer: along the exact ray of (i, j), is triangle `p` (index id_p) the
// closest-hit choice over triangle `q` (index id_q)?  Nearer exact distance
// first (T_p / D_p < T_q / D_q, compared as T_p D_q < T_q D_p), then the lower
// index; a triangle the exact ray misses never wins.
__device__ __noinline__ bool exact_closer(const SensorDev& s, int i, int j, const float4* p, uint32_t id_p,
                                          const float4* q, uint32_t id_q) {
    ff w[3];
    ray_dir_ff(s, i, j, w);
    const float o[3] = {s.pos[0], s.pos[1], s.pos[2]};
    ff Dp, Tp, Dq, Tq;
    if (!mt_ff(o, w, __ldg(p), __ldg(p + 1), __ldg(p + 2), Dp, Tp)) return false;
    if (!mt_ff(o, w, __ldg(q), __ldg(q + 1), __ldg(q + 2), Dq, Tq)) return true;
    const int c = ff_sign(ff_sub(ff_mul(Tp, Dq), ff_mul(Tq, Dp)));
    return c < 0 || (c == 0 && id_p < id_q);
}

// The exact test of two triangles along the exact ray of (i, j), by a whole warp:
// each half takes one (triangles f0 and f1 in leaf order), a lane per component of
// a vector or per product, the same operations in the same order as mt_ff, so the
// same bits.  Returns in every lane whether each is hit and its D and T, and the
// length of the unnormalised direction.  An undecided test falls to about one ray
// of a 32-ray tile; by its lane alone it took ~750 instructions in a row.
struct ExactPair {
    bool hit0, hit1;
    ff D0, T0, D1, T1;
    float len;
};
__device__ __forceinline__ ff shfl16(ff v, int src) {
    return ff{__shfl_sync(0xFFFFFFFFu, v.hi, src, 16), __shfl_sync(0xFFFFFFFFu, v.lo, src, 16)};
}
__device__ __forceinline__ float axis_of(float4 v, int a) { return a == 0 ? v.x : a == 1 ? v.y : v.z; }

__device__ __noinline__ ExactPair exact_pair(const SensorDev& s, const float4* tris, int i, int j, int f0, int f1) {
    const int lane = threadIdx.x & 31, l = min(lane & 15, 11), kind = l / 3, ax = l - 3 * kind;
    const float4* tp = tris + 3 * (int64_t)(lane < 16 ? f0 : f1);
    const float4 a = __ldg(tp), b = __ldg(tp + 1), c = __ldg(tp + 2);
    // components: lanes 0-2 e1, 3-5 e2, 6-8 s = o - v0, 9-11 the direction w
    const ff e = ff_two_sum(kind == 0 ? axis_of(b, ax) : kind == 1 ? axis_of(c, ax) : s.pos[ax], -axis_of(a, ax));
    const float4 bp = s.trig[i], el = s.trig[s.nb + j];
    const ff sp{bp.x, bp.y}, cp{bp.z, bp.w}, st{el.x, el.y}, ct{el.z, el.w};
    const ff w = ff_add(ff_add(ff_mulf(ff_mul(sp, ct), s.rot[3 * ax]), ff_mulf(ff_mul(cp, ct), s.rot[3 * ax + 1])),
                        ff_mulf(st, s.rot[3 * ax + 2]));
    const ff v{kind == 3 ? w.hi : e.hi, kind == 3 ? w.lo : e.lo};
    // cross products: lanes 0-2 p = w x e2, 3-5 q = s x e1
    const int y = ax == 2 ? 0 : ax + 1, z = ax == 0 ? 2 : ax - 1;
    const int ka = kind == 0 ? 9 : 6, kb = kind == 0 ? 3 : 0;
    const ff ay = shfl16(v, ka + y), bz = shfl16(v, kb + z), az = shfl16(v, ka + z), by = shfl16(v, kb + y);
    const ff cr = ff_sub(ff_mul(ay, bz), ff_mul(az, by));
    // dot products, three lanes each: det = e1 p, u = s p, v = w q, t = e2 q
    const ff x0 = shfl16(v, (kind == 0 ? 0 : kind == 1 ? 6 : kind == 2 ? 9 : 3) + ax);
    const ff x1 = shfl16(cr, (kind < 2 ? 0 : 3) + ax);
    const ff m = ff_mul(x0, x1);
    const ff dot = ff_add(ff_add(shfl16(m, 3 * kind), shfl16(m, 3 * kind + 1)), shfl16(m, 3 * kind + 2));
    const ff det = shfl16(dot, 0);
    ff un = shfl16(dot, 3), vn = shfl16(dot, 6), tn = shfl16(dot, 9);
    const int sg = ff_sign(det);
    ff D = det;
    if (sg < 0) { D = ff_neg(det); un = ff_neg(un); vn = ff_neg(vn); tn = ff_neg(tn); }
    const bool hit = sg != 0 && !(ff_sign(un) < 0 || ff_sign(vn) < 0 || ff_sign(ff_sub(ff_sub(D, un), vn)) < 0 ||
                                  ff_sign(tn) <= 0);
    const uint32_t hits = __ballot_sync(0xFFFFFFFFu, hit);
    auto of = [&](float x, int half) { return __shfl_sync(0xFFFFFFFFu, x, 16 * half); };
    ExactPair r;
    r.hit0 = hits & 1u;
    r.hit1 = (hits >> 16) & 1u;
    r.D0 = ff{of(D.hi, 0), of(D.lo, 0)};
    r.T0 = ff{of(tn.hi, 0), of(tn.lo, 0)};
    r.D1 = ff{of(D.hi, 1), of(D.lo, 1)};
    r.T1 = ff{of(tn.hi, 1), of(tn.lo, 1)};
    const float w0 = __shfl_sync(0xFFFFFFFFu, w.hi, 0), w1 = __shfl_sync(0xFFFFFFFFu, w.hi, 1),
                w2 = __shfl_sync(0xFFFFFFFFu, w.hi, 2);
    r.len = sqrtf(w0 * w0 + w1 * w1 + w2 * w2);
    return r;
}

// Float-float sine and cosine tables of the sensor's beam azimuths
// phi_i = -H/2 + (i + 1/2) H / N_b and elevations theta_j = -V/2 + (j + 1/2) V / N_e
// (computed in FP64 once per sensor, split into hi + lo floats): trig[i] for
// beams, trig[N_b + j] for elevations, each (sin hi, sin lo, cos hi, cos lo).
__global__ void k_trig(const SensorDev* sensors, SensorDev one) {
    __shared__ bool s_current;
    let_next_start();
    const SensorDev& s = sensors ? sensors[blockIdx.y] : one;
    // a batch block whose entries were built for the sensor's current fields of
    // view has nothing to do (only later launches read the table).  One thread reads
    // the stamp for all: a warp that read it after it was written would skip its entries
    if (threadIdx.x == 0) s_current = s.trig_stamp && s.trig_stamp[blockIdx.x] == s.trig_version;
    __syncthreads();
    if (s_current) return;
    if (s.trig_stamp && threadIdx.x == 0) s.trig_stamp[blockIdx.x] = s.trig_version;
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= s.nb + s.ne) return;
    double a;
    if (k < s.nb) {
        const double H = s.hfov;
        a = -H / 2.0 + (k + 0.5) * H / s.nb;
    } else {
        const double V = s.vfov;
        a = -V / 2.0 + (k - s.nb + 0.5) * V / s.ne;
    }
    double sn, cs;
    sincos(a, &sn, &cs);
    const float sh = (float)sn, ch = (float)cs;
    s.trig[k] = make_float4(sh, (float)(sn - (double)sh), ch, (float)(cs - (double)ch));
}

// Range bin of a hit, or -1 when r is outside [r_min, r_max).
__device__ __forceinline__ int range_bin(const SensorDev& s, float r) {
    if (!(r >= s.rmin && r < s.rmax)) return -1;
    const int br = (int)floorf((r - s.rmin) * s.inv_dr);
    return br < s.nr - 1 ? br : s.nr - 1;
}

// Azimuth bin of beam i: floor((2i + 1) naz / (2 nb)), in 32-bit integers when
// the product fits (it does whenever nb * naz < 2^30).
__device__ __forceinline__ int az_bin(const SensorDev& s, int i) {
    if ((int64_t)s.nb * s.naz < (1ll << 30)) return (int)(((2u * i + 1u) * (uint32_t)s.naz) / (2u * (uint32_t)s.nb));
    return (int)(((2ll * i + 1) * s.naz) / (2ll * s.nb));
}


// ---------------------------------------------------------------------------
// trace: one ray per thread, hit record out
// ---------------------------------------------------------------------------

// The hit record of ray (ri, rj) of direction d: `best` the triangle hit (leaf
// order, -1: none) at distance best_t.
__device__ __forceinline__ uint4 record_of(const SensorDev& S, const SceneDev& sc, const sonar_params& p, float3 d,
                                           int ri, int best, float best_t) {
    uint32_t key = kNoKey, orig = 0xFFFFFFFFu, cosb = 0u;
    float tr = CUDART_INF_F;
    if (best >= 0) {
        const float4* tp = sc.tris + 3 * (int64_t)best;
        const float4 va = __ldg(tp), vb = __ldg(tp + 1), vc = __ldg(tp + 2);
        const float3 v0 = f3(va.x, va.y, va.z);
        const float3 n = cross3(sub(f3(vb.x, vb.y, vb.z), v0), sub(f3(vc.x, vc.y, vc.z), v0));
        const float dn = dot3(d, n) / sqrtf(dot3(n, n));
        orig = __float_as_uint(vb.w);
        tr = best_t;
        cosb = __float_as_uint(p.two_sided ? fabsf(dn) : fmaxf(-dn, 0.0f));
        const int br = range_bin(S, best_t);
        if (br >= 0) key = (uint32_t)(br * S.naz + az_bin(S, ri));
    }
    return make_uint4(key, orig, __float_as_uint(tr), cosb);
}

// Each warp takes a tile of tb beams x (32 / tb) elevations of one sensor: lane l
// traces beam i0 + l % tb, elevation j0 + l / tb, so that the warp's rays sample
// a compact patch of the field of view.  Records go to their canonical index
// i * n_elev + j.
//
// The walk over the W-wide hierarchy (W = 4, or 8 for launches too small to
// fill the GPU, where fewer dependent node loads per ray matter more than the
// extra box tests per visit) is a while-while loop in step: lanes descend nearest
// child first, pushing the other entered children; a lane that reaches a leaf
// parks it and keeps descending until no lane is without one, so that the
// triangle tests run together, and the whole warp settles the undecided ones
// (exact_pair).  A lane whose ray is finished writes its record at once and
// idles until the warp is done.
//
// Bound by issue, the pipe of comparisons, minima and selections first, with the
// latency of node loads next (about 62 % of the issue slots, 25 of 32 warps).
// What that came to, ray cast of 64 frames of 512 x 64 rays / 128 mixed sensors /
// 32 frames of 1024 x 256 rays over 33.6 million triangles, hit records the same:
// 432 / 1277 / 1994 us, undecided tests by their lane alone; 426 / 1261 / 1979 by
// the warp, which also takes the walk from 95 registers to 69; 405 / 1200 / 1882
// with handles selected by the bits of their slot and no count of entered
// children; 393 / 1163 / 1838 with a bottom stack entry instead of an empty test
// and two tiles a block (the block limit is 32 per SM, and two warps share the
// slot of one); 383 / 1132 / 1791 with boxes as centre and half-width; 360 / 998 /
// 1686 on a hierarchy over the triangles' box centres.
// With STATS the kernel also counts node visits and triangle tests and marks
// the nodes and triangles it touches (records are then not written).
constexpr int kTraceWarps = 2;   // tiles per block, each a warp's own
template <int MINB, bool STATS, int W>
__global__ void __launch_bounds__(32 * kTraceWarps, MINB) k_trace(const __grid_constant__ TraceArgs a) {
    __shared__ SensorDev s_S[kTraceWarps];
    __shared__ SceneDev s_SC[kTraceWarps];
    let_next_start();
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    int tile = blockIdx.x * kTraceWarps + wid;
    if (tile >= a.n_tiles) return;
    SensorDev& S = s_S[wid];
    SceneDev& SC = s_SC[wid];
    if (a.sensors) {
        // the warp copies the sensor and scene descriptors word by word, both at
        // once (the map carries the scene index): one round trip after the map
        const int4 m = a.block_map[tile];
        copy_words(&S, a.sensors + m.x, lane);
        copy_words(&SC, a.scenes + m.z, lane);
        tile = m.y;
    } else {
        copy_param(&S, &a.one, lane);
        copy_param(&SC, &a.one_scene, lane);
        if (a.from_last) tile = a.n_tiles - 1 - tile;
    }
    __syncwarp();
    wait_for_previous();   // the exact-ray tables
    if (a.zero_word && blockIdx.x == 0 && threadIdx.x == 0) *a.zero_word = 0;   // read by a later launch only
    const int tb = S.tb, te = 32 / S.tb;
    const int tiles_b = (S.nb + tb - 1) / tb;
    const int ty = tile / tiles_b, tx = tile - ty * tiles_b;
    const int ri = tx * tb + (lane % tb);
    const int rj = ty * te + lane / tb;
    const SceneDev& sc = SC;
    const sonar_params& p = a.params;
    // without clipping any finite distance counts: 3e38 stands for infinity so
    // that the box cut below (1.00002 times the best distance) stays finite
    const float tlimit = p.clip_tmax ? S.rmax : 3.0e38f;
    const float3 o = f3(S.pos[0], S.pos[1], S.pos[2]);
    const bool inside = ri < S.nb && rj < S.ne;
    const float3 d = inside ? ray_dir32(S, ri, rj) : f3(0.0f, 0.0f, 1.0f);
    const float tiny = 1e-20f;
    const float3 inv = f3(1.0f / (fabsf(d.x) > tiny ? d.x : copysignf(tiny, d.x)),
                          1.0f / (fabsf(d.y) > tiny ? d.y : copysignf(tiny, d.y)),
                          1.0f / (fabsf(d.z) > tiny ? d.z : copysignf(tiny, d.z)));
    const float3 oinv = f3(o.x * inv.x, o.y * inv.y, o.z * inv.z);
    // (inv, inv) and (-o inv, -o inv) per axis as packed pairs for the box tests
    const unsigned long long ivx = pk2(inv.x), ivy = pk2(inv.y), ivz = pk2(inv.z);
    const unsigned long long novx = pk2(-oinv.x), novy = pk2(-oinv.y), novz = pk2(-oinv.z);
    const float3 ainv = f3(fabsf(inv.x), fabsf(inv.y), fabsf(inv.z));
    int32_t stack[kStackMax + 1];   // above a bottom entry that ends the walk
    stack[0] = kEmpty;
    int sp = 1, best = -1;
    uint32_t best_id = 0xFFFFFFFFu;
    float best_t = tlimit;
    uint64_t visits = 0, tests = 0, exact_n = 0;
    // `node`: the internal node to visit next (or kEmpty); `leaf`: a parked
    // leaf whose triangles wait to be tested (0 = none; leaf handles are negative)
    int32_t node = inside ? sc.root : kEmpty, leaf = 0;
    if (node < 0 && node != kEmpty) { leaf = node; node = kEmpty; }
    bool live = inside;
    for (;;) {
        // descend while some lane has a node to visit and no leaf yet
        while (__any_sync(0xFFFFFFFFu, node >= 0 && leaf == 0)) {
            if (node >= 0) {
                const float4* pn = W == 4 ? sc.nodes + 8 * (int64_t)node : sc.nodes8 + 16 * (int64_t)node;
                if (STATS) {
                    ++visits;
                    atomicOr(a.tc.node_bits + (node >> 5), 1u << (node & 31));
                }
                const float tcut = best_t * 1.00002f;
                // sort key per child: entry distance bits (>= 0, so integer order
                // is distance order) with the child slot in the low bits; a
                // missed child sorts last as 0xFFFFFFFF
                uint32_t key[W];
                int32_t hs[W];
                // per axis, the centre and half-width of every child's box
                float cx[W], hx[W], cy[W], hy[W], cz[W], hz[W];
                if constexpr (W == 4) {
                    ld_node_pair(pn, cx, hx);
                    ld_node_pair(pn + 2, cy, hy);
                    ld_node_pair(pn + 4, cz, hz);
                    float h[4], none[4];
                    ld_node_pair(pn + 6, h, none);
#pragma unroll
                    for (int c = 0; c < 4; ++c) hs[c] = __float_as_int(h[c]);
                } else {
#pragma unroll
                    for (int c = 0; c < W; ++c) {
                        const Child ch = ld_child(pn + 2 * c);
                        cx[c] = ch.cx; hx[c] = ch.hx;
                        cy[c] = ch.cy; hy[c] = ch.hy;
                        cz[c] = ch.cz; hz[c] = ch.hz;
                        hs[c] = ch.handle;
                    }
                }
                // the ray's distance to a box's centre plane, two children at a time
                float tx[W], ty[W], tz[W];
#pragma unroll
                for (int c = 0; c < W; c += 2) {
                    fma2(cx[c], cx[c + 1], ivx, novx, tx[c], tx[c + 1]);
                    fma2(cy[c], cy[c + 1], ivy, novy, ty[c], ty[c + 1]);
                    fma2(cz[c], cz[c + 1], ivz, novz, tz[c], tz[c + 1]);
                }
#pragma unroll
                for (int c = 0; c < W; ++c) {
                    const float lo = fmaxf(fmaxf(fmaf(-hx[c], ainv.x, tx[c]), fmaf(-hy[c], ainv.y, ty[c])),
                                           fmaxf(fmaf(-hz[c], ainv.z, tz[c]), 0.0f));
                    const float hi = fminf(fminf(fmaf(hx[c], ainv.x, tx[c]), fmaf(hy[c], ainv.y, ty[c])),
                                           fminf(fmaf(hz[c], ainv.z, tz[c]), tcut));
                    // an empty slot's box is a point at +inf on every axis: along an axis
                    // the ray travels in the + direction its entry distance is +inf,
                    // and if it travels in the - direction along all three its exit
                    // distance is -inf; the exit is also at most tcut, which is
                    // finite, so an empty slot never passes and needs no handle check
                    const bool hit = lo <= hi * 1.0000005f;
                    key[c] = hit ? ((__float_as_uint(lo) & ~(uint32_t)(W - 1)) | (uint32_t)c) : 0xFFFFFFFFu;
                }
                sort_keys<W>(key);
                if (sp + W - 1 > kStackMax) {   // cannot happen for a checked height: give up the ray
                    atomicOr(a.err, SONAR_DEVERR_STACK);
                    node = kEmpty;
                    leaf = 0;
                    sp = 1;
                    best = -1;
                } else {
#pragma unroll
                    for (int c = W - 1; c >= 1; --c) {
                        if (key[c] != 0xFFFFFFFFu) stack[sp++] = child_at<W>(hs, key[c] & (uint32_t)(W - 1));
                    }
                    if (key[0] != 0xFFFFFFFFu) node = child_at<W>(hs, key[0] & (uint32_t)(W - 1));
                    else node = stack[--sp];
                }
                if (node < 0 && node != kEmpty && leaf == 0) {   // park the leaf, keep descending
                    leaf = node;
                    node = stack[--sp];
                }
            }
            __syncwarp();
        }
        // the triangles of the parked leaves, a triangle of every lane's at a time;
        // undecided tests and near ties are settled by the whole warp, one after another
        while (__any_sync(0xFFFFFFFFu, leaf != 0)) {
            const int32_t x = ~leaf;
            const int32_t first = x >> 3, count = leaf != 0 ? (x & 7) + 1 : 0;
            for (int k = 0; __any_sync(0xFFFFFFFFu, k < count); ++k) {
                const int32_t f = first + k;
                int r = 0;
                float t = 0.0f;
                uint32_t id = 0u;
                if (k < count) {
                    if (f >= sc.n_tris) {
                        atomicOr(a.err, SONAR_DEVERR_INDEX);
                    } else {
                        const float4* tp = sc.tris + 3 * (int64_t)f;
                        const float4 va = __ldg(tp), vb = __ldg(tp + 1), vc = __ldg(tp + 2);
                        if (STATS) {
                            ++tests;
                            atomicOr(a.tc.tri_bits + (f >> 5), 1u << (f & 31));
                        }
                        r = mt32(o, d, va, vb, vc, t);
                        id = __float_as_uint(vb.w);
                    }
                }
                for (uint32_t m = __ballot_sync(0xFFFFFFFFu, r == 2); m; m &= m - 1) {
                    const int src = __ffs(m) - 1;
                    const int fs = __shfl_sync(0xFFFFFFFFu, f, src);
                    const ExactPair e = exact_pair(S, sc.tris, __shfl_sync(0xFFFFFFFFu, ri, src),
                                                   __shfl_sync(0xFFFFFFFFu, rj, src), fs, fs);
                    if (lane == src) {
                        if (STATS) ++exact_n;
                        r = e.hit0;
                        t = (e.T0.hi / e.D0.hi) * e.len;
                    }
                }
                const bool cand = r != 0 && t < tlimit;
                bool take = cand && (best < 0 || t < best_t);
                // near tie: decide on the exact distances, then on the caller's index
                const bool tie = cand && best >= 0 && fabsf(t - best_t) <= 2e-5f * fmaxf(t, best_t);
                for (uint32_t m = __ballot_sync(0xFFFFFFFFu, tie); m; m &= m - 1) {
                    const int src = __ffs(m) - 1;
                    const ExactPair e = exact_pair(S, sc.tris, __shfl_sync(0xFFFFFFFFu, ri, src),
                                                   __shfl_sync(0xFFFFFFFFu, rj, src), __shfl_sync(0xFFFFFFFFu, f, src),
                                                   __shfl_sync(0xFFFFFFFFu, best, src));
                    if (lane == src) {
                        if (STATS) ++exact_n;
                        const int c = ff_sign(ff_sub(ff_mul(e.T0, e.D1), ff_mul(e.T1, e.D0)));
                        take = e.hit0 && (!e.hit1 || c < 0 || (c == 0 && id < best_id));
                    }
                }
                if (take) {
                    best = f;
                    best_id = id;
                    best_t = t;
                }
            }
            leaf = 0;
            if (node < 0 && node != kEmpty) {   // the next stacked entry is a leaf too
                leaf = node;
                node = stack[--sp];
            }
        }
        if (live && node == kEmpty) {
            // the ray is finished: its hit record (bin key, triangle, range, incidence)
            live = false;
            if (!STATS) {
                *reinterpret_cast<uint4*>(a.hits + S.hits_off + (int64_t)ri * S.ne + rj) =
                    record_of(S, sc, p, d, ri, best, best_t);
            }
        }
        if (__ballot_sync(0xFFFFFFFFu, live) == 0u) break;
    }
    if (STATS) {
        atomicAdd(a.tc.visits, (unsigned long long)visits);
        atomicAdd(a.tc.tests, (unsigned long long)tests);
        atomicAdd(a.tc.exact, (unsigned long long)exact_n);
    }
}
// Several lanes (G = 8 or 4) per ray, for launches that cannot fill the GPU.
// Such a launch lasts as long as its longest chain of dependent node visits (a
// frame of 32,768 rays is a fifth of a wave of k_trace's warps), and there a
// visit costs its ~300 instructions in a row and waits for the slowest of 32
// rays.  Here a lane loads and tests 8 / G children of an 8-wide node; the
// nearest entered child is next (a minimum over the ray's lanes), the others
// go to the ray's stack in shared memory with their entry distances, and an
// entry beyond the ray's cut is dropped when it comes up.  Entered leaves are
// parked by their lanes until every ray of the warp holds one or has nothing
// left to visit; then the triangles are spread over the ray's lanes, two lanes
// a leaf.  Every lane keeps the closest of the triangles it tested itself; the
// ray's cut is the least of them, and the candidates are compared at the end
// by the same rule as in k_trace (distance, exact decision for near ties), so
// the records are the same.
// Bound by the longest rays' chains of visits up to about 20,000 rays, above that
// by issue (four lanes a ray: 15 us per 32,768 rays, against 24 us by eight and
// 6.5 us by one lane in a launch that fills the GPU).  Ray cast of one frame, one
// lane a ray -> four -> eight lanes: 1,024 rays over a plane and a sphere 29.6 ->
// 17.9 -> 17.1 us; 8,192 rays over a seabed 40.4 -> 22.2 -> 21.0; 16,403 rays to
// 27 m 140 -> 55 -> 42; 32,768 rays 42.7 -> 29.1 -> 34.5; 65,536 rays (two frames)
// 57.2 -> 41.6 -> 53.2; 131,072 rays 61.2 -> 71.1 -> 96.5 (all on a hierarchy over
// centroids; over box centres the first three are 15.0, 18.8 and 37.0 as launched).
constexpr int kGroupThreads = 64;       // threads per block

template <int G>
__global__ void __launch_bounds__(kGroupThreads, 12) k_trace_group(const __grid_constant__ TraceArgs a) {
    constexpr int kRays = kGroupThreads / G;            // rays per block
    constexpr int kParts = 32 / kRays;                  // blocks per 32-ray tile
    constexpr int J = 8 / G;                            // children per lane: c, c + G, ...
    constexpr uint32_t kLanes = (1u << G) - 1u;
    __shared__ SensorDev S;
    __shared__ SceneDev SC;
    __shared__ int s_tile;
    __shared__ float2 s_stack[kRays][kStackMax];        // (handle bits, entry distance)
    let_next_start();
    if (threadIdx.x < 32) {
        const int tile = blockIdx.x / kParts;
        if (a.sensors) {
            const int4 m = __ldg(a.block_map + tile);
            copy_words(&S, a.sensors + m.x, threadIdx.x);
            copy_words(&SC, a.scenes + m.z, threadIdx.x);
            if (threadIdx.x == 0) s_tile = m.y;
        } else {
            copy_param(&S, &a.one, threadIdx.x);
            copy_param(&SC, &a.one_scene, threadIdx.x);
            if (threadIdx.x == 0) s_tile = a.from_last ? a.one.trace_blocks - 1 - tile : tile;
        }
    }
    wait_for_previous();   // the exact-ray tables
    if (a.zero_word && blockIdx.x == 0 && threadIdx.x == 0) *a.zero_word = 0;   // read by a later launch only
    __syncthreads();
    const int tb = S.tb, te = 32 / tb, tiles_b = (S.nb + tb - 1) / tb;
    const int ty = s_tile / tiles_b, tx = s_tile - ty * tiles_b;
    const int group = threadIdx.x / G, c = threadIdx.x & (G - 1);
    const int l = (blockIdx.x % kParts) * kRays + group;   // the ray within its tile
    const int ri = tx * tb + l % tb, rj = ty * te + l / tb;
    const SceneDev& sc = SC;
    const float tlimit = a.params.clip_tmax ? S.rmax : 3.0e38f;
    const float3 o = f3(S.pos[0], S.pos[1], S.pos[2]);
    const bool inside = ri < S.nb && rj < S.ne;
    const float3 d = inside ? ray_dir32(S, ri, rj) : f3(0.0f, 0.0f, 1.0f);
    const float tiny = 1e-20f;
    const float3 inv = f3(1.0f / (fabsf(d.x) > tiny ? d.x : copysignf(tiny, d.x)),
                          1.0f / (fabsf(d.y) > tiny ? d.y : copysignf(tiny, d.y)),
                          1.0f / (fabsf(d.z) > tiny ? d.z : copysignf(tiny, d.z)));
    const float3 oinv = f3(o.x * inv.x, o.y * inv.y, o.z * inv.z);
    const float3 ainv = f3(fabsf(inv.x), fabsf(inv.y), fabsf(inv.z));
    const int lane = threadIdx.x & 31, shift = lane & ~(G - 1);
    const uint32_t mine = kLanes << shift;
    float2* stack = s_stack[group];
    int sp = 0, best = -1;
    uint32_t best_id = 0xFFFFFFFFu;
    float best_t = tlimit, cut = tlimit;   // this lane's closest; the ray's
    float node_t = 0.0f;                   // entry distance of `node`
    int32_t leaf[J], late[J];              // leaves parked by this lane (0: none); `late` came while it held one
#pragma unroll
    for (int j = 0; j < J; ++j) leaf[j] = late[j] = 0;
    int32_t node = inside ? sc.root : kEmpty;
    if (node < 0 && node != kEmpty) {      // a scene of one leaf
        if (c == 0) leaf[0] = node;
        node = kEmpty;
    }
    // the ray's 8-bit mask of the children (slot c + G j) whose lanes say yes
    auto slots = [&](const bool (&yes)[J]) {
        uint32_t m = 0u;
#pragma unroll
        for (int j = 0; j < J; ++j) m |= ((__ballot_sync(0xFFFFFFFFu, yes[j]) >> shift) & kLanes) << (G * j);
        return m;
    };
    for (;;) {
        int32_t h[J];
        float lo[J];
        bool inner[J];
        uint32_t kmin = 0xFFFFFFFFu;
#pragma unroll
        for (int j = 0; j < J; ++j) {
            h[j] = kEmpty;
            lo[j] = 0.0f;
            inner[j] = false;
        }
        if (node >= 0) {
            Child ch[J];
#pragma unroll
            for (int j = 0; j < J; ++j) ch[j] = ld_child(sc.nodes8 + 16 * (int64_t)node + 2 * (c + G * j));
            const float tcut = cut * 1.00002f;
#pragma unroll
            for (int j = 0; j < J; ++j) {
                const float tx = fmaf(ch[j].cx, inv.x, -oinv.x), ty = fmaf(ch[j].cy, inv.y, -oinv.y),
                            tz = fmaf(ch[j].cz, inv.z, -oinv.z);
                h[j] = ch[j].handle;
                lo[j] = fmaxf(fmaxf(fmaf(-ch[j].hx, ainv.x, tx), fmaf(-ch[j].hy, ainv.y, ty)),
                              fmaxf(fmaf(-ch[j].hz, ainv.z, tz), 0.0f));
                const float hi = fminf(fminf(fmaf(ch[j].hx, ainv.x, tx), fmaf(ch[j].hy, ainv.y, ty)),
                                       fminf(fmaf(ch[j].hz, ainv.z, tz), tcut));
                const bool enter = lo[j] <= hi * 1.0000005f;   // never an empty slot (see k_trace)
                inner[j] = enter && h[j] >= 0;
                if (enter && h[j] < 0) {
                    if (leaf[j] == 0) leaf[j] = h[j];
                    else late[j] = h[j];
                }
                if (inner[j]) kmin = min(kmin, (__float_as_uint(lo[j]) & ~7u) | (uint32_t)(c + G * j));
            }
        }
#pragma unroll
        for (int k = 1; k < G; k <<= 1) kmin = min(kmin, __shfl_xor_sync(0xFFFFFFFFu, kmin, k));
        const uint32_t near = kmin & 7u;   // the slot of the nearest
        int32_t next = h[0];
        float next_t = lo[0];
        if constexpr (J == 2) {
            if (near >= G) { next = h[1]; next_t = lo[1]; }
        }
        next = __shfl_sync(0xFFFFFFFFu, next, shift + (near & (G - 1)));
        next_t = __shfl_sync(0xFFFFFFFFu, next_t, shift + (near & (G - 1)));
        const uint32_t entered = slots(inner);
        if (entered) {
            const uint32_t others = entered & ~(1u << near);
            const int n = __popc(others);
            if (sp + n > kStackMax) {   // cannot happen for a checked height: give up the ray
                atomicOr(a.err, SONAR_DEVERR_STACK);
                node = kEmpty;
                sp = 0;
#pragma unroll
                for (int j = 0; j < J; ++j) leaf[j] = late[j] = 0;
                best = -1;
                best_t = cut = tlimit;
            } else {
#pragma unroll
                for (int j = 0; j < J; ++j) {
                    const uint32_t slot = (uint32_t)(c + G * j);
                    if ((others >> slot) & 1u)
                        stack[sp + __popc(others & ((1u << slot) - 1u))] = make_float2(__int_as_float(h[j]), lo[j]);
                }
                sp += n;
                node = next;
                node_t = next_t;
            }
            __syncwarp(mine);
        } else {
            node = kEmpty;
        }
        bool has_leaf[J], has_late = false;
#pragma unroll
        for (int j = 0; j < J; ++j) {
            has_leaf[j] = leaf[j] != 0;
            has_late = has_late || late[j] != 0;
        }
        uint32_t parked = slots(has_leaf);
        const bool waits = (node == kEmpty && sp == 0) || parked != 0u;
        const bool all_wait = __all_sync(0xFFFFFFFFu, waits), any_late = __any_sync(0xFFFFFFFFu, has_late);
        if ((all_wait || any_late) && __any_sync(0xFFFFFFFFu, parked != 0u)) {
            do {
                uint32_t m = parked;   // this lane's leaf: set bit number c / 2
                if ((c >> 1) > 0) m &= m - 1;
                if (G > 4 && (c >> 1) > 1) m &= m - 1;
                if (G > 4 && (c >> 1) > 2) m &= m - 1;
                const int slot = (__ffs(m) - 1) & 7;
                int32_t x = __shfl_sync(0xFFFFFFFFu, leaf[0], shift + (slot & (G - 1)));
                if constexpr (J == 2) {
                    const int32_t x1 = __shfl_sync(0xFFFFFFFFu, leaf[1], shift + (slot & (G - 1)));
                    if (slot >= G) x = x1;
                }
                x = ~x;
                const int32_t first = x >> 3, count = m ? (x & 7) + 1 : 0;
                for (int k = c & 1; k < count; k += 2) {
                    const int32_t f = first + k;
                    if (f >= sc.n_tris) {
                        atomicOr(a.err, SONAR_DEVERR_INDEX);
                        break;
                    }
                    const float4* tp = sc.tris + 3 * (int64_t)f;
                    const float4 va = __ldg(tp), vb = __ldg(tp + 1), vc = __ldg(tp + 2);
                    float t;
                    const int r = mt32(o, d, va, vb, vc, t);
                    if (r == 0 || (r == 2 && !exact_hit(S, ri, rj, va, vb, vc, &t)) || !(t < tlimit)) continue;
                    const uint32_t id = __float_as_uint(vb.w);
                    bool take;
                    if (best < 0) take = true;
                    else if (fabsf(t - best_t) <= 2e-5f * fmaxf(t, best_t))
                        take = exact_closer(S, ri, rj, tp, id, sc.tris + 3 * (int64_t)best, best_id);
                    else take = t < best_t;
                    if (take) {
                        best = f;
                        best_id = id;
                        best_t = t;
                    }
                }
                __syncwarp();
#pragma unroll
                for (int k = 0; k < G / 2; ++k) parked &= parked - 1;
            } while (__any_sync(0xFFFFFFFFu, parked != 0u));
#pragma unroll
            for (int j = 0; j < J; ++j) {
                leaf[j] = late[j];
                late[j] = 0;
            }
            cut = best_t;
#pragma unroll
            for (int k = 1; k < G; k <<= 1) cut = fminf(cut, __shfl_xor_sync(0xFFFFFFFFu, cut, k));
        }
        if (node != kEmpty && !(node_t <= cut * 1.00002f)) node = kEmpty;
        while (node == kEmpty && sp > 0) {   // an entry beyond the cut would fail its box test now
            const float2 e = stack[--sp];
            if (e.y <= cut * 1.00002f) {
                node = __float_as_int(e.x);
                node_t = e.y;
            }
        }
        bool more = node != kEmpty;
#pragma unroll
        for (int j = 0; j < J; ++j) more = more || leaf[j] != 0;
        if (!__any_sync(0xFFFFFFFFu, more)) break;
    }
    // the ray's closest of its lanes' candidates
#pragma unroll
    for (int k = 1; k < G; k <<= 1) {
        const float t2 = __shfl_xor_sync(0xFFFFFFFFu, best_t, k);
        const int b2 = __shfl_xor_sync(0xFFFFFFFFu, best, k);
        const uint32_t id2 = __shfl_xor_sync(0xFFFFFFFFu, best_id, k);
        if (b2 < 0) continue;
        bool take;
        if (best < 0) take = true;
        else if (b2 == best) take = false;
        else if (fabsf(t2 - best_t) <= 2e-5f * fmaxf(t2, best_t))
            take = exact_closer(S, ri, rj, sc.tris + 3 * (int64_t)b2, id2, sc.tris + 3 * (int64_t)best, best_id);
        else take = t2 < best_t;
        if (take) {
            best = b2;
            best_id = id2;
            best_t = t2;
        }
    }
    if (inside && c == 0)
        *reinterpret_cast<uint4*>(a.hits + S.hits_off + (int64_t)ri * S.ne + rj) =
            record_of(S, sc, a.params, d, ri, best, best_t);
}

// ---------------------------------------------------------------------------
// counters
// ---------------------------------------------------------------------------

__global__ void k_popcount(const uint32_t* bits, int64_t words, unsigned long long* out) {
    unsigned long long c = 0;
    for (int64_t w = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; w < words; w += (int64_t)gridDim.x * blockDim.x)
        c += __popc(bits[w]);
    for (int o = 16; o; o >>= 1) c += __shfl_down_sync(0xFFFFFFFFu, c, o);
    if ((threadIdx.x & 31) == 0) atomicAdd(out, c);
}

}  // namespace

// ---------------------------------------------------------------------------
// launchers
// ---------------------------------------------------------------------------

cudaError_t launch_trig(const SensorDev* sensors, const SensorDev& one, int n_sensors, int max_angles,
                        cudaStream_t st) {
    const dim3 grid((unsigned)((max_angles + 127) / 128), (unsigned)n_sensors);
    k_trig<<<grid, 128, 0, st>>>(sensors, one);
    return cudaGetLastError();
}

cudaError_t launch_trace(const TraceArgs& a, int blocks, int occupancy, cudaStream_t st, bool early) {
    if (blocks <= 0) return cudaSuccess;
    const bool cap = occupancy & kTraceCap;
    // one sensor's launch on a scene without an 8-wide tree walks the 4-wide
    // one (a batch's variant is checked against all its scenes on the host)
    const bool wide = (occupancy & kTraceWide) && (a.sensors || a.one_scene.nodes8);
    if (wide && (occupancy & kTraceGroup8))
        return launch_kernel(k_trace_group<8>, (unsigned)blocks * (32 * 8 / kGroupThreads), kGroupThreads, 0, st, early, a);
    if (wide && (occupancy & kTraceGroup4))
        return launch_kernel(k_trace_group<4>, (unsigned)blocks * (32 * 4 / kGroupThreads), kGroupThreads, 0, st, early, a);
    TraceArgs b = a;
    b.n_tiles = blocks;
    return launch_kernel(wide ? (cap ? k_trace<16, false, 8> : k_trace<4, false, 8>)
                              : (cap ? k_trace<16, false, 4> : k_trace<4, false, 4>),
                         (unsigned)((blocks + kTraceWarps - 1) / kTraceWarps), 32 * kTraceWarps, 0, st, early, b);
}

cudaError_t launch_stats(const SensorDev& s, const SceneDev& sc, const sonar_params& p,
                         const TraceCounters& tc, uint32_t* err, cudaStream_t st) {
    TraceArgs a{};
    a.one = s;
    a.one_scene = sc;
    a.n_sensors = 1;
    a.params = p;
    a.err = err;
    a.tc = tc;
    if (s.trace_blocks > 0) {
        a.n_tiles = s.trace_blocks;
        const unsigned grid = (unsigned)((s.trace_blocks + kTraceWarps - 1) / kTraceWarps);
        if ((s.occ & kTraceWide) && sc.nodes8) k_trace<4, true, 8><<<grid, 32 * kTraceWarps, 0, st>>>(a);
        else k_trace<4, true, 4><<<grid, 32 * kTraceWarps, 0, st>>>(a);
    }
    return cudaGetLastError();
}

cudaError_t launch_popcount(const uint32_t* bits, int64_t words, unsigned long long* out, cudaStream_t st) {
    k_popcount<<<1024, 256, 0, st>>>(bits, words, out);
    return cudaGetLastError();
}

}  // namespace sonar

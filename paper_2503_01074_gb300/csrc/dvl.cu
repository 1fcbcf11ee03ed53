// DVL kernels (OceanSim, arXiv 2503.01074, Sec. III-A-3): four-beam Janus ranges by
// a per-thread walk of the 4-wide hierarchy, least-squares velocity, range-
// dependent ping period and dropout, and the per-vehicle emission schedule.
#include <cuda_runtime.h>
#include <math_constants.h>
#include <stdint.h>

#include "sonar_host.h"
#include "sonar_internal.cuh"
#include "devmath.cuh"

namespace sonar {
namespace {

// ---------------------------------------------------------------------------
// DVL (Sec. III-A-3): four-beam Janus ranges, least-squares velocity, rate
// ---------------------------------------------------------------------------

// The exact decision of an uncertain FP32 test, on the FP32 direction (out of
// line: rarely needed).
__device__ __noinline__ bool exact_distance(float3 o, float3 d, float4 a, float4 b, float4 c, float* t) {
    const float of[3] = {o.x, o.y, o.z};
    const ff df[3] = {ff{d.x, 0.0f}, ff{d.y, 0.0f}, ff{d.z, 0.0f}};
    ff D, T;
    if (!mt_ff(of, df, a, b, c, D, T)) return false;
    *t = T.hi / D.hi;
    return true;
}

// Closest hit along one ray (any origin and direction) by a walk of the 4-wide
// hierarchy, a lane per ray: certified FP32 Moller-Trumbore, undecided tests
// decided exactly in float-float on the FP32 direction; ties go to the lower
// caller index.  Lanes park a leaf and descend on until every active lane of the
// warp holds one, as in the sonar's ray cast.  Returns the distance (+inf for a
// miss, and for a lane without a ray).
__device__ __forceinline__ float closest_distance(const SceneDev& sc, bool live, float3 o, float3 d, uint32_t* err) {
    const float tiny = 1e-20f;
    const float3 inv = f3(1.0f / (fabsf(d.x) > tiny ? d.x : copysignf(tiny, d.x)),
                          1.0f / (fabsf(d.y) > tiny ? d.y : copysignf(tiny, d.y)),
                          1.0f / (fabsf(d.z) > tiny ? d.z : copysignf(tiny, d.z)));
    const unsigned long long ivx = pk2(inv.x), ivy = pk2(inv.y), ivz = pk2(inv.z);
    const unsigned long long novx = pk2(-(o.x * inv.x)), novy = pk2(-(o.y * inv.y)), novz = pk2(-(o.z * inv.z));
    const float3 ainv = f3(fabsf(inv.x), fabsf(inv.y), fabsf(inv.z));
    int32_t stack[kStackMax + 1];   // above a bottom entry that ends the walk
    stack[0] = kEmpty;
    int sp = 1;
    float best_t = 3.0e38f;   // a finite cut keeps empty slots (boxes at +inf) out, see k_trace
    uint32_t best_id = 0xFFFFFFFFu;
    int32_t node = live ? sc.root : kEmpty, leaf = 0;
    if (node < 0 && node != kEmpty) { leaf = node; node = kEmpty; }
    while (__any_sync(0xFFFFFFFFu, node != kEmpty || leaf != 0)) {
        // descend while some lane has a node to visit and no leaf yet
        while (__any_sync(0xFFFFFFFFu, node >= 0 && leaf == 0)) {
            if (node >= 0) {
                const float4* pn = sc.nodes + 8 * (int64_t)node;
                const float tcut = best_t * 1.00002f;
                // centres and half-widths of the children's boxes, handles (see k_trace)
                float cx[4], hx[4], cy[4], hy[4], cz[4], hz[4], ch[4], none[4];
                ld_node_pair(pn, cx, hx);
                ld_node_pair(pn + 2, cy, hy);
                ld_node_pair(pn + 4, cz, hz);
                ld_node_pair(pn + 6, ch, none);
                int32_t hs[4];
                uint32_t key[4];
                float tx[4], ty[4], tz[4];
#pragma unroll
                for (int c = 0; c < 4; c += 2) {
                    fma2(cx[c], cx[c + 1], ivx, novx, tx[c], tx[c + 1]);
                    fma2(cy[c], cy[c + 1], ivy, novy, ty[c], ty[c + 1]);
                    fma2(cz[c], cz[c + 1], ivz, novz, tz[c], tz[c + 1]);
                }
#pragma unroll
                for (int c = 0; c < 4; ++c) {
                    hs[c] = __float_as_int(ch[c]);
                    const float lo = fmaxf(fmaxf(fmaf(-hx[c], ainv.x, tx[c]), fmaf(-hy[c], ainv.y, ty[c])),
                                           fmaxf(fmaf(-hz[c], ainv.z, tz[c]), 0.0f));
                    const float hi = fminf(fminf(fmaf(hx[c], ainv.x, tx[c]), fmaf(hy[c], ainv.y, ty[c])),
                                           fminf(fmaf(hz[c], ainv.z, tz[c]), tcut));
                    const bool hit = lo <= hi * 1.0000005f;
                    key[c] = hit ? ((__float_as_uint(lo) & ~3u) | (uint32_t)c) : 0xFFFFFFFFu;
                }
                sort_keys<4>(key);
                if (sp + 3 > kStackMax) {   // cannot happen for a checked depth: give up the ray
                    atomicOr(err, SONAR_DEVERR_STACK);
                    node = kEmpty;
                    leaf = 0;
                    sp = 1;
                    best_id = 0xFFFFFFFFu;
                    best_t = 0.0f;
                } else {
#pragma unroll
                    for (int c = 3; c >= 1; --c)
                        if (key[c] != 0xFFFFFFFFu) stack[sp++] = child_at<4>(hs, key[c] & 3u);
                    if (key[0] != 0xFFFFFFFFu) node = child_at<4>(hs, key[0] & 3u);
                    else node = stack[--sp];
                }
                if (node < 0 && node != kEmpty && leaf == 0) {   // park the leaf, keep descending
                    leaf = node;
                    node = stack[--sp];
                }
            }
            __syncwarp();
        }
        while (leaf != 0) {
            const int32_t x = ~leaf;
            const int32_t first = x >> 3, count = (x & 7) + 1;
            for (int k = 0; k < count; ++k) {
                const int32_t f = first + k;
                if (f >= sc.n_tris) {
                    atomicOr(err, SONAR_DEVERR_INDEX);
                    break;
                }
                const float4* tp = sc.tris + 3 * (int64_t)f;
                const float4 va = __ldg(tp), vb = __ldg(tp + 1), vc = __ldg(tp + 2);
                float t;
                const int r = mt32(o, d, va, vb, vc, t);
                if (r == 0 || (r == 2 && !exact_distance(o, d, va, vb, vc, &t))) continue;
                const uint32_t id = __float_as_uint(vb.w);
                if (t < best_t || (t == best_t && id < best_id)) {
                    best_t = t;
                    best_id = id;
                }
            }
            leaf = 0;
            if (node < 0 && node != kEmpty) {   // the next stacked entry is a leaf too
                leaf = node;
                node = stack[--sp];
            }
        }
    }
    return best_id == 0xFFFFFFFFu ? CUDART_INF_F : best_t;
}

// A standard normal from two Philox words: the cosine branch of Box-Muller.
__device__ __forceinline__ float normal_of(uint32_t a, uint32_t b) {
    const float u2 = fmaf((float)b, 0x1p-32f, 0x1p-32f);
    return sqrt_nonneg(neg2log_u(a)) * cospif(2.0f * u2);
}

// 32 poses per block, warp k casting beam k of them; then a thread per pose fits
// the velocity by least squares over the valid beams (Cramer's rule on the 3 x 3
// normal equations) and writes the pose's outputs.  Consecutive poses are mostly
// steps of one track, so the rays of a warp are nearly parallel and close, and
// visit much the same nodes.
// Bound by issue like the sonar's ray cast.  1M poses (4M beams) over 524,288
// triangles: 707 us with the four beams of a pose side by side in a warp, scalar
// plane distances and seven loads a node; 624 us by beams; 444 us with the
// boxes and the descent in step of k_trace.
constexpr int kDvlPoses = 32;
__global__ void __launch_bounds__(4 * kDvlPoses) k_dvl(const __grid_constant__ DvlArgs a) {
    __shared__ float s_range[4][kDvlPoses], s_u[4][kDvlPoses];
    const int k = threadIdx.x / kDvlPoses, q = threadIdx.x & (kDvlPoses - 1);
    const int64_t p = (int64_t)blockIdx.x * kDvlPoses + q;
    const bool live = p < a.n;
    float3 o = f3(0.0f, 0.0f, 0.0f), d = f3(0.0f, 0.0f, 1.0f);
    float u = 0.0f;
    if (live) {
        const float* pose = a.pose + 12 * p;
        o = f3(pose[0], pose[1], pose[2]);
        const float* R = pose + 3;
        const float bx = a.beam[k][0], by = a.beam[k][1], bz = a.beam[k][2];
        d = f3(fmaf(R[0], bx, fmaf(R[1], by, R[2] * bz)), fmaf(R[3], bx, fmaf(R[4], by, R[5] * bz)),
               fmaf(R[6], bx, fmaf(R[7], by, R[8] * bz)));
        // sensor-frame velocity R^T v and this beam's radial velocity with noise
        const float* vw = a.vel_world + 3 * p;
        const float vs0 = fmaf(R[0], vw[0], fmaf(R[3], vw[1], R[6] * vw[2]));
        const float vs1 = fmaf(R[1], vw[0], fmaf(R[4], vw[1], R[7] * vw[2]));
        const float vs2 = fmaf(R[2], vw[0], fmaf(R[5], vw[1], R[8] * vw[2]));
        const U4 x = philox10(U4{(uint32_t)p, (uint32_t)((uint64_t)p >> 32), 2u, (uint32_t)(k >> 1)},
                              a.seed_lo, a.seed_hi);
        const float w = (k & 1) ? normal_of(x.z, x.w) : normal_of(x.x, x.y);
        u = fmaf(bx, vs0, fmaf(by, vs1, bz * vs2)) + a.sigma_b * w;
    }
    s_range[k][q] = closest_distance(a.scene, live, o, d, a.err);
    s_u[k][q] = u;
    __syncthreads();
    if (!live || k != 0) return;
    float rr[4], uu[4];
    unsigned bits = 0u;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        rr[j] = s_range[j][q];
        uu[j] = s_u[j][q];
        if (rr[j] >= a.r_min && rr[j] <= a.r_max) bits |= 1u << j;
    }
    if ((reinterpret_cast<uintptr_t>(a.ranges) & 15u) == 0) {
        reinterpret_cast<float4*>(a.ranges)[p] = make_float4(rr[0], rr[1], rr[2], rr[3]);
    } else {
#pragma unroll
        for (int j = 0; j < 4; ++j) a.ranges[4 * p + j] = rr[j];
    }
    const int nvalid = __popc(bits);
    float A[3][3] = {{0.f, 0.f, 0.f}, {0.f, 0.f, 0.f}, {0.f, 0.f, 0.f}}, y[3] = {0.f, 0.f, 0.f};
    float far = 0.0f;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        if (!((bits >> j) & 1u)) continue;
        far = fmaxf(far, rr[j]);
#pragma unroll
        for (int r = 0; r < 3; ++r) {
            y[r] = fmaf(a.beam[j][r], uu[j], y[r]);
#pragma unroll
            for (int c = 0; c < 3; ++c) A[r][c] = fmaf(a.beam[j][r], a.beam[j][c], A[r][c]);
        }
    }
    int32_t flags = (int32_t)bits;
    float v0 = 0.0f, v1 = 0.0f, v2 = 0.0f;
    const float det = A[0][0] * (A[1][1] * A[2][2] - A[1][2] * A[2][1]) -
                      A[0][1] * (A[1][0] * A[2][2] - A[1][2] * A[2][0]) +
                      A[0][2] * (A[1][0] * A[2][1] - A[1][1] * A[2][0]);
    if (nvalid >= a.min_beams && det != 0.0f) {
        const float id = 1.0f / det;
        v0 = (y[0] * (A[1][1] * A[2][2] - A[1][2] * A[2][1]) - A[0][1] * (y[1] * A[2][2] - A[1][2] * y[2]) +
              A[0][2] * (y[1] * A[2][1] - A[1][1] * y[2])) * id;
        v1 = (A[0][0] * (y[1] * A[2][2] - A[1][2] * y[2]) - y[0] * (A[1][0] * A[2][2] - A[1][2] * A[2][0]) +
              A[0][2] * (A[1][0] * y[2] - y[1] * A[2][0])) * id;
        v2 = (A[0][0] * (A[1][1] * y[2] - y[1] * A[2][1]) - A[0][1] * (A[1][0] * y[2] - y[1] * A[2][0]) +
              y[0] * (A[1][0] * A[2][1] - A[1][1] * A[2][0])) * id;
        flags |= 16;
    }
    a.vel[3 * p] = v0;
    a.vel[3 * p + 1] = v1;
    a.vel[3 * p + 2] = v2;
    a.flags[p] = flags;
    a.period[p] = (flags & 16) ? fmaf(a.t1, far, a.t0) : a.t_lost;
}

// Emission schedule: one warp per vehicle walks its steps (a measurement at step
// 0, then max(1, ceil(period / dt)) steps after each measurement), a chunk of
// steps at a time: the lanes turn the chunk's periods into step counts in shared
// memory, lane 0 walks those, and the chunk is written as whole rows.
// 4096 vehicles x 256 steps: 17 us, against 78 us with a thread per vehicle (below).
constexpr int kSchedWarps = 4, kSchedChunk = 256;
__global__ void __launch_bounds__(32 * kSchedWarps) k_dvl_schedule(const float* period, int64_t n_veh, int64_t n_steps,
                                                                   float dt, int32_t* emit) {
    __shared__ int32_t s_next[kSchedWarps][kSchedChunk];
    __shared__ uint32_t s_bits[kSchedWarps][kSchedChunk / 32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int64_t v = (int64_t)blockIdx.x * kSchedWarps + warp;
    if (v >= n_veh) return;
    const float* P = period + v * n_steps;
    int32_t* E = emit + v * n_steps;
    int64_t at = 0;   // the next measurement (the same in every lane)
    for (int64_t s0 = 0; s0 < n_steps; s0 += kSchedChunk) {
        const int count = (int)min((int64_t)kSchedChunk, n_steps - s0);
        if (lane < kSchedChunk / 32) s_bits[warp][lane] = 0u;
        if (at < s0 + count) {
            for (int i = lane; i < count; i += 32) {
                const float q = ceilf(P[s0 + i] / dt);
                s_next[warp][i] = q >= 1073741824.0f ? 0 : q >= 1.0f ? (int32_t)q : 1;   // 0: beyond 32 bits
            }
            __syncwarp();
            if (lane == 0) {
                while (at < s0 + count) {
                    const int i = (int)(at - s0);
                    s_bits[warp][i >> 5] |= 1u << (i & 31);
                    const int32_t step = s_next[warp][i];
                    at += step > 0 ? step : (int64_t)fminf(ceilf(P[at] / dt), 4.0e18f);
                }
            }
            at = __shfl_sync(0xFFFFFFFFu, at, 0);
        }
        __syncwarp();
        for (int i = lane; i < count; i += 32) E[s0 + i] = (int32_t)((s_bits[warp][i >> 5] >> (i & 31)) & 1u);
        __syncwarp();
    }
}

// The same, a thread per vehicle that clears, walks and marks its row alone: short
// schedules of many vehicles, where a warp per vehicle leaves most of its lanes idle.
// Bound by the chain of a row's loads, then by its scattered stores.
__global__ void __launch_bounds__(128) k_dvl_schedule_short(const float* period, int64_t n_veh, int64_t n_steps,
                                                            float dt, int32_t* emit) {
    const int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (v >= n_veh) return;
    const float* P = period + v * n_steps;
    int32_t* E = emit + v * n_steps;
    for (int64_t s = 0; s < n_steps; ++s) E[s] = 0;
    for (int64_t s = 0; s < n_steps;) {
        E[s] = 1;
        const float q = ceilf(P[s] / dt);
        s += q >= 1.0f ? (int64_t)fminf(q, 4.0e18f) : 1;
    }
}

// Which of the two: measured by warps -> by threads, periods of 1, 4 and 20 steps:
// 1,048,576 vehicles x 1 step 150 -> 12, 151 -> 12, 151 -> 11 us; x 16 413 -> 140, 205 ->
// 92, 156 -> 80; x 48 1017 -> 577, 396 -> 358, 250 -> 323; x 64 1280 -> 844, 458 -> 445, 269 ->
// 389; 100,000 x 32 70 -> 50, 29 -> 28, 19 -> 23; 32,768 x 48 37 -> 25, 16 -> 15, 10 -> 14;
// 4,096 x 32 by warps 7, by threads 14 with every step a measurement (one
// row's chain of loads).
constexpr int64_t kShortSteps = 48, kShortVehicles = 32768;

}  // namespace

// ---------------------------------------------------------------------------
// launchers
// ---------------------------------------------------------------------------

cudaError_t launch_dvl(const DvlArgs& a, cudaStream_t st) {
    if (a.n > 0) k_dvl<<<(unsigned)((a.n + kDvlPoses - 1) / kDvlPoses), 4 * kDvlPoses, 0, st>>>(a);
    return cudaGetLastError();
}

cudaError_t launch_dvl_schedule(const float* period, int64_t n_veh, int64_t n_steps, float dt, int32_t* emit,
                                cudaStream_t st) {
    if (n_veh >= kShortVehicles && n_steps <= kShortSteps && n_steps > 0)
        k_dvl_schedule_short<<<(unsigned)((n_veh + 127) / 128), 128, 0, st>>>(period, n_veh, n_steps, dt, emit);
    else if (n_veh > 0 && n_steps > 0)
        k_dvl_schedule<<<(unsigned)((n_veh + kSchedWarps - 1) / kSchedWarps), 32 * kSchedWarps, 0, st>>>(
            period, n_veh, n_steps, dt, emit);
    return cudaGetLastError();
}

}  // namespace sonar

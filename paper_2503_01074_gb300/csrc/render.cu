// Sonar post-processing kernels (OceanSim, arXiv 2503.01074, Sec. III-A-2).
//
// k_fold              one warp (or block) = one azimuth column of one sensor: the
//                     column's hit records -> intensity (Eq. 2, two-way) -> the sums
//                     of its bins with returns, compactly (a bitmap, ranks, values):
//                     no global atomics, no memset and no dense image of P.
// k_rows              one warp = one range row: Eq. 3-6 noise of every bin, the row
//                     maximum and N = I~ / max; writes I~ and N, reads neither.
// k_norm_rows         whole-image normalisation only: N = I~ / max.
// k_fan_*             fan resample of the normalised image: per-pixel polar
//                     coordinate tables, then bilinear gathers for two frames
//                     per table read.
// adjoint             per-group (row) Jacobian terms, then a per-ray gather of
//                     dL/dP into (dalpha, dgain, dmu) over ray chunks, and a
//                     fixed-order final reduction (deterministic).
#include <cuda_runtime.h>
#include <math_constants.h>
#include <stdint.h>

#include "sonar_host.h"
#include "sonar_internal.cuh"
#include "devmath.cuh"

namespace sonar {
namespace {

// ---------------------------------------------------------------------------
// fold: the rays of every azimuth column -> the column's bins with returns
// ---------------------------------------------------------------------------

// The score of a hit record of material m: s = mu[m] cos exp(-2 alpha r) gain (Eq. 2).
__device__ __forceinline__ float score_of(const FoldArgs& a, int m, float r, float cosine, float alpha, float gain) {
    m = m < a.n_mat ? m : a.n_mat - 1;
    return __ldg(a.theta + 2 + m) * cosine * expf(-2.0f * alpha * r) * gain;
}

// Division by naz of multiples of it: a shift by its trailing zeros and a
// multiplication by the inverse of its odd part modulo 2^32 (Newton's iteration
// doubles the correct low bits, from 5).
struct ExactDiv {
    uint32_t naz, inv;
    int shift;
};
__device__ __forceinline__ ExactDiv exact_div(uint32_t naz) {
    const int shift = __ffs((int)naz) - 1;
    const uint32_t odd = naz >> shift;
    uint32_t x = (odd * 3u) ^ 2u;
#pragma unroll
    for (int k = 0; k < 3; ++k) x *= 2u - odd * x;
    return ExactDiv{naz, x, shift};
}

// Range row of a record of azimuth column `col`, or -1: no return, or a
// corrupt record (reported in the error word).
__device__ __forceinline__ int row_of(const FoldArgs& a, const ExactDiv& div, uint32_t nr, uint32_t n_tris,
                                      uint32_t key, uint32_t tri, uint32_t col) {
    if (key == kNoKey) return -1;
    const uint32_t row = ((key - col) >> div.shift) * div.inv;
    if (row >= nr || row * div.naz + col != key || tri >= n_tris) {
        atomicOr(a.err, SONAR_DEVERR_INDEX);
        return -1;
    }
    return (int)row;
}

// Exclusive prefix of the set bits of bits[0..nwords) into pre (one warp); returns their number.
__device__ __forceinline__ int bit_prefix(const uint32_t* bits, uint32_t* pre, int nwords, int lane) {
    int total = 0;
    for (int w0 = 0; w0 < nwords; w0 += 32) {
        const int w = w0 + lane;
        const int n = w < nwords ? __popc(bits[w]) : 0;
        int x = n;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int y = __shfl_up_sync(0xFFFFFFFFu, x, o);
            if (lane >= o) x += y;
        }
        if (w < nwords) pre[w] = (uint32_t)(total + x - n);
        total += __shfl_sync(0xFFFFFFFFu, x, 31);
    }
    return total;
}

__device__ __forceinline__ int bit_rank(const uint32_t* bits, const uint32_t* pre, int row) {
    return (int)pre[row >> 5] + __popc(bits[row >> 5] & ((1u << (row & 31)) - 1u));
}

// Adds each lane's score to acc[idx] (idx < 0: none), equal bins in lane
// order onto the bin's running sum: with the rays taken 32 at a time in
// canonical order, every bin is the sequential sum of its returns.  The lowest
// lane of a bin reads its peers' scores from shared memory (32 words of the
// warp's own): shuffles among the peers would run the bins one after another
// (64 frames: 63 us with them).
__device__ __forceinline__ void fold_step(float* acc, float* scores, int idx, float score, int lane) {
    scores[lane] = score;
    const uint32_t peers = __match_any_sync(0xFFFFFFFFu, idx);
    __syncwarp();
    if (idx >= 0 && lane == __ffs(peers) - 1) {
        float v = acc[idx] + score;
        for (uint32_t m = peers & (peers - 1); m; m &= m - 1) v += scores[__ffs(m) - 1];
        acc[idx] = v;
    }
    __syncwarp();
}

// A finished bin (rank k of its column): P and the speckle factor 0.5 + w_sm
// of Eq. 3, compactly; or P into the image itself where no scratch holds them.
__device__ __forceinline__ void put_bin(const FoldArgs& a, const SensorDev& S, int64_t first, int k, int row, int col,
                                        float P) {
    const uint32_t b = (uint32_t)row * (uint32_t)S.naz + (uint32_t)col;
    if (a.dense) {
        a.dense[S.polar_off + b] = P;
    } else {
        a.vals[S.val_off + first + k] = make_float2(P, 0.5f + gauss_of(philox10(U4{b, S.frame_lo, 0u, S.frame_hi}, S.seed_lo, S.seed_hi), a.sigma_sm));
    }
}

constexpr int kFoldAhead = 2;   // chunks of 32 rays whose loads are issued together

// Marks the rows of rays first, first + step, ... (step a multiple of 32) of a
// column's n records.
__device__ __forceinline__ void mark_rows(const FoldArgs& a, const ExactDiv& div, const SensorDev& S,
                                          const SceneDev& sc, const sonar_hit* H, uint32_t n, uint32_t first, uint32_t step,
                                          int col, uint32_t* bits) {
    for (uint32_t j = first; j < n; j += kFoldAhead * step) {
        uint2 h[kFoldAhead];   // key, triangle
#pragma unroll
        for (int u = 0; u < kFoldAhead; ++u)
            h[u] = j + u * step < n ? *reinterpret_cast<const uint2*>(H + j + u * step) : make_uint2(kNoKey, 0u);
#pragma unroll
        for (int u = 0; u < kFoldAhead; ++u) {
            const int row = row_of(a, div, S.nr, sc.n_tris, h[u].x, h[u].y, col);
            if (row >= 0) atomicOr(bits + (row >> 5), 1u << (row & 31));
        }
    }
}

// Sums the scores of n consecutive records, in order, at the ranks of their rows
// (one warp): the records of several chunks, then their materials, are loaded
// together, so that a chunk does not wait for both in turn.
__device__ __forceinline__ void sum_rows(const FoldArgs& a, const ExactDiv& div, const SensorDev& S,
                                         const SceneDev& sc, const sonar_hit* H, uint32_t n, int col,
                                         const uint32_t* bits, const uint32_t* pre, int* rows, float* acc,
                                         float* scores, float alpha, float gain, int lane) {
    for (uint32_t jb = 0; jb < n; jb += 32 * kFoldAhead) {
        uint4 h[kFoldAhead];
#pragma unroll
        for (int u = 0; u < kFoldAhead; ++u)
            h[u] = jb + 32 * u + lane < n ? *reinterpret_cast<const uint4*>(H + jb + 32 * u + lane)
                                          : make_uint4(kNoKey, 0u, 0u, 0u);
        int row[kFoldAhead], mat[kFoldAhead];
#pragma unroll
        for (int u = 0; u < kFoldAhead; ++u) {
            row[u] = row_of(a, div, S.nr, sc.n_tris, h[u].x, h[u].y, col);
            mat[u] = row[u] >= 0 ? __ldg(sc.mat_orig + h[u].y) : 0;
        }
#pragma unroll
        for (int u = 0; u < kFoldAhead; ++u) {
            if (jb + 32 * u >= n) break;
            int idx = -1;
            float score = 0.0f;
            if (row[u] >= 0) {
                idx = bit_rank(bits, pre, row[u]);
                rows[idx] = row[u];   // every writer of a rank writes the same row
                score = score_of(a, mat[u], __uint_as_float(h[u].z), __uint_as_float(h[u].w), alpha, gain);
            }
            fold_step(acc, scores, idx, score, lane);
        }
    }
}

// One warp per azimuth column (sensors with at most one beam per column, and
// those whose per-beam rows do not fit in shared memory), or one block per
// column (S.fold_block): its warps on the column's beams (S.fold_beams), or, where few
// columns hold many rays, all of them in pass 1 and one in pass 2.
//
// Only the bins that a ray lands in (about 6 % of them) are stored: pass 1 marks
// the column's rows with returns in a bitmap, a prefix over its words ranks
// them, pass 2 sums the scores at the ranks, and the bitmap with its ranks is
// what the row kernel looks bins up in (a bit per bin plus 8 bytes per ray,
// against the 8 bytes per bin of a dense image written and read back).  A
// column's working set is so a few hundred words rather than a row of floats
// per range bin, and no pass over all bins is left here.
//
// Bound by the latency of its dependent steps (record, material, rank, sum),
// which the resident columns hide (40 registers: 48 warps an SM), and by issue where
// columns hold many rays.  Measured, this kernel and k_rows against the binning
// kernel over dense column blocks and the normalisation pass that they replace:
// 64 frames of 512 x 64 rays into 1000 x 512 bins 39 + 90 us against 231 + 43 us
// (132 + 43 us with hand-picked units); 32 frames of 1024 x 256 rays into 4000 x
// 1024 bins 474 us together against 1122 + 153; one frame of 3000 x 460 rays into
// 350 x 220 bins 39 + 6 us against 462 + 5.  Rows by exact division instead of a
// general one, fewer registers and two chunks of loads at a time were 17 % of it.
__global__ void __launch_bounds__(512, 3) k_fold(const __grid_constant__ FoldArgs a) {
    extern __shared__ __align__(16) uint32_t fold_smem[];
    __shared__ SensorDev S;
    __shared__ SceneDev SC;
    __shared__ int s_col, s_n;
    __shared__ float s_scores[16][32];
    let_next_start();
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nw = blockDim.x >> 5;
    if (warp == 0) {
        if (a.sensors) {
            const int4 m = __ldg(a.block_map + blockIdx.x);
            copy_words(&S, a.sensors + m.x, lane);
            copy_words(&SC, a.scenes + m.z, lane);
            if (lane == 0) s_col = m.y;
        } else {
            copy_param(&S, &a.one, lane);
            copy_param(&SC, &a.one_scene, lane);
            if (lane == 0) s_col = blockIdx.x * (a.one.fold_block ? 1 : nw);
        }
    }
    __syncthreads();
    const float alpha = __ldg(a.theta), gain = __ldg(a.theta + 1);
    const ExactDiv div = exact_div((uint32_t)S.naz);
    const int ne = S.ne, nwords = (S.nr + 31) >> 5;
    const int col = s_col + (S.fold_block ? 0 : warp);
    if (col >= S.naz) return;   // whole warps only (the last block of a sensor)
    const int i0 = first_beam_of_col(col, S.nb, S.naz), i1 = first_beam_of_col(col + 1, S.nb, S.naz);
    const int64_t first = (int64_t)i0 * ne;          // the column's first ray, and its first value slot
    const int n = (i1 - i0) * ne;                    // a sensor's rays fit 31 bits
    const sonar_hit* H = a.hits + S.hits_off + first;
    const int most = min(S.nr, n);                   // bins with returns, at most
    wait_for_previous();   // the hit records
    if (!S.fold_block) {
        uint32_t* bits = fold_smem + (int64_t)warp * a.words_per_warp;
        uint32_t* pre = bits + nwords;
        float* acc = reinterpret_cast<float*>(pre + nwords);
        int* rows = reinterpret_cast<int*>(acc + most);
        for (int w = lane; w < nwords; w += 32) bits[w] = 0u;
        __syncwarp();
        mark_rows(a, div, S, SC, H, n, lane, 32, col, bits);
        __syncwarp();
        const int nd = bit_prefix(bits, pre, nwords, lane);
        for (int k = lane; k < nd; k += 32) acc[k] = 0.0f;
        __syncwarp();
        sum_rows(a, div, S, SC, H, n, col, bits, pre, rows, acc, s_scores[warp], alpha, gain, lane);
        for (int k = lane; k < nd; k += 32) put_bin(a, S, first, k, rows[k], col, acc[k]);
        if (a.bands)
            for (int w = lane; w < nwords; w += 32)
                a.bands[S.band_off + (int64_t)w * S.naz + col] = make_uint2(bits[w], (uint32_t)first + pre[w]);
        return;
    }
    // block form: each part (a beam, in elevation order; or the whole column) sums its own
    // rows, a bin then adds its column's parts in order
    const int parts = S.fold_beams ? i1 - i0 : 1, len = S.fold_beams ? ne : n, nt = blockDim.x;
    uint32_t* bits = fold_smem;
    uint32_t* pre = bits + nwords;
    int* rows = reinterpret_cast<int*>(pre + nwords);
    float* acc = reinterpret_cast<float*>(rows + most);   // [parts][nd]
    for (int w = tid; w < nwords; w += nt) bits[w] = 0u;
    __syncthreads();
    mark_rows(a, div, S, SC, H, n, tid, nt, col, bits);
    __syncthreads();
    if (warp == 0) {
        const int total = bit_prefix(bits, pre, nwords, lane);
        if (lane == 0) s_n = total;
    }
    __syncthreads();
    const int nd = s_n;
    for (int k = tid; k < parts * nd; k += nt) acc[k] = 0.0f;
    __syncthreads();
    for (int p = warp; p < parts; p += nw)
        sum_rows(a, div, S, SC, H + (int64_t)p * len, len, col, bits, pre, rows, acc + p * nd, s_scores[warp], alpha, gain,
                 lane);
    __syncthreads();
    for (int k = tid; k < nd; k += nt) {
        float P = 0.0f;
        for (int p = 0; p < parts; ++p) P += acc[p * nd + k];
        put_bin(a, S, first, k, rows[k], col, P);
    }
    if (a.bands)
        for (int w = tid; w < nwords; w += nt)
            a.bands[S.band_off + (int64_t)w * S.naz + col] = make_uint2(bits[w], (uint32_t)first + pre[w]);
}

// ---------------------------------------------------------------------------
// rows: noise (Eq. 3-6) and range-wise normalisation, one warp per range row
// ---------------------------------------------------------------------------

// The additive term of Eq. 3 for a range row (`rc` its centre, squared over
// r_max^2) and a column whose beam-pattern factor 0.5 exp(-phi_c^2 / sigma_phi)
// is `pat`, from the bin's uniform word of the additive stream:
// (r_c^2 / r_max^2)(1 + pat w_sa), w_sa ~ Rayleigh(sigma_sa) (Eq. 4).
__device__ __forceinline__ float additive_term(float rc, float inv_rmax2, float pat, uint32_t word, float sig_sa) {
    const float w_sa = rayleigh_of(word, sig_sa);
    return rc * rc * inv_rmax2 * (1.0f + pat * w_sa);
}

__device__ __forceinline__ float pattern_of(const SensorDev& S, int col, float da, float inv_sphi) {
    const float pc = fmaf(small_u2f((uint32_t)col) + 0.5f, da, -0.5f * S.hfov);
    return 0.5f * expf(-pc * pc * inv_sphi);
}

// A bin of a row or image of maximum m (which is not divided where it is not positive).
__device__ __forceinline__ float norm_value(float In, float m, int mode) {
    return (mode != 0 && m > 0.0f) ? In / m : In;
}

// v / m correctly rounded, given y = 1 / m correctly rounded, for 2^-60 <= v <= m
// <= 2^60 (the quotient is at least 2^-120, a residual's last bit at least 2^-106:
// nothing under- or overflows): v y is within two ulp,
// one residual step brings it within one, and a second one rounds correctly
// (P. Markstein, IBM J. Res. Dev. 34(1), 1990).  Five FMA-pipe operations,
// against nine and two on the quarter-rate unit for the general division.
__device__ __forceinline__ float div_by(float v, float m, float y) {
    float q = v * y;
    q = fmaf(fmaf(-m, q, v), y, q);
    return fmaf(fmaf(-m, q, v), y, q);
}

// Four neighbouring bins of one row share a Philox block (their index over
// four), so a lane takes quads: q-th quad of the row, its columns
// 4 q - sh + (0..3), sh = row * naz mod 4 (nonzero only where naz is not a
// multiple of 4; the row's first and last quads then reach over its ends).
//
// A block takes a.rows_per_block rows of one band of 32, so the bitmap words of
// its columns (and the columns' beam pattern) are read once into shared memory
// and serve all its rows.  A bin with a return fetches P and the speckle factor
// from its column's compact list; every other bin is the additive term alone.
// REG > 0: a row of up to 128 REG bins stays in registers between its maximum
// and the division, so I~ and N are written and nothing is read back; REG = 0
// (wider rows, and the dense form of the fold's result): I~ is written, then read
// back by the same lanes and divided.  Where such rows are few, a block's warps share
// one (rows_per_block 1): a warp alone takes some 10 ns a bin, 95 us for 8192.
//
// Bound by instruction issue (about 75 per bin, most of them the logarithm and a
// quarter of a Philox block): 64 frames of 1000 x 512 bins in 92 us, 2.8 TB/s of
// stores (the 262 MB that it writes would take 39 us); 125 us with an IEEE division,
// two integer conversions and general square roots and divisions per bin.  32 rows
// a block: 16 take 4 to 8 % longer, 8 up to 25 % (the column tables are read again).
template <int REG, bool VEC>
__global__ void __launch_bounds__(256, REG == 4 ? 3 : 2) k_rows(const __grid_constant__ RowsArgs a) {
    extern __shared__ __align__(16) uint32_t rows_smem[];
    __shared__ SensorDev S;
    __shared__ int s_row0;
    __shared__ float s_top[8];
    let_next_start();
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const bool shared_row = REG == 0 && a.rows_per_block == 1;   // by all warps of the block
    const int q0 = shared_row ? warp : 0, dq = shared_row ? 8 : 1;   // a lane's quads: q0, q0 + dq, ...
    if (warp == 0) {
        // the rows run from the last sensor back to the first, so that the first
        // sensors' N is the last written and the fan finds it in L2
        const int blk = gridDim.x - 1 - blockIdx.x;
        if (a.sensors) {
            const int2 m = __ldg(a.block_map + blk);
            copy_words(&S, a.sensors + m.x, lane);
            if (lane == 0) s_row0 = m.y;
        } else {
            copy_param(&S, &a.one, lane);
            if (lane == 0) s_row0 = blk * a.rows_per_block;
        }
    }
    __syncthreads();
    const int naz = S.naz, nr = S.nr, row0 = s_row0;
    const float dr = (S.rmax - S.rmin) / (float)nr, da = S.hfov / (float)naz;
    const float inv_rmax2 = 1.0f / (S.rmax * S.rmax), inv_sphi = 1.0f / a.params.sigma_phi;
    const float sig_sa = a.params.sigma_sa;
    const int mode = a.params.normalise;
    const bool dense = REG == 0 && a.dense;
    const uint2* bands = a.bands + S.band_off + (int64_t)(row0 >> 5) * naz;
    const bool staged = REG > 0 || naz <= kRowsStaged;   // the launch has room for every such sensor
    float* pat = reinterpret_cast<float*>(rows_smem);
    uint2* mask = reinterpret_cast<uint2*>(rows_smem + ((naz + 3) & ~3));
    if (staged) {
        for (int c = tid; c < naz; c += blockDim.x) pat[c] = pattern_of(S, c, da, inv_sphi);
    }
    wait_for_previous();   // the fold's bitmaps and values
    if (staged) {
        if (!dense)
            for (int c = tid; c < naz; c += blockDim.x) mask[c] = bands[c];
        __syncthreads();
    }
    const PhiloxKey K = philox_key(S.seed_lo, S.seed_hi);
    const uint32_t flo = S.frame_lo, fhi = S.frame_hi;
    const float2* vals = a.vals + S.val_off;
    float image_max = -CUDART_INF_F;
    for (int r = shared_row ? 0 : warp; r < a.rows_per_block; r += 8) {
        const int row = row0 + r;
        if (row >= nr) break;
        const uint32_t b0 = (uint32_t)row * (uint32_t)naz;
        const int sh = VEC ? 0 : (int)(b0 & 3u), nq = (sh + naz + 3) >> 2;
        const int64_t off = S.polar_off + (int64_t)b0 - sh + 4 * lane;   // of the lane's first quad's first bin
        const float rc = fmaf(small_u2f((uint32_t)row) + 0.5f, dr, S.rmin);
        const uint32_t bit = 1u << (row & 31), below = bit - 1u;
        // The four bins of the lane's k-th quad (quad q = lane + 32 k of the row, at
        // 128 k elements from the first): I~ in v, P in p.
        auto quad = [&](int k, float (&v)[4], float (&p)[4]) {
            const int q = lane + 32 * k;
            float2 ret[4];
            float pt[4];
            uint2 w[4];
            if (VEC && staged) {   // 16-byte shared-memory reads
                const float4 p4 = reinterpret_cast<const float4*>(pat)[q];
                pt[0] = p4.x; pt[1] = p4.y; pt[2] = p4.z; pt[3] = p4.w;
                const uint4 w0 = reinterpret_cast<const uint4*>(mask)[2 * q];
                const uint4 w1 = reinterpret_cast<const uint4*>(mask)[2 * q + 1];
                w[0] = make_uint2(w0.x, w0.y); w[1] = make_uint2(w0.z, w0.w);
                w[2] = make_uint2(w1.x, w1.y); w[3] = make_uint2(w1.z, w1.w);
            }
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const int c = 4 * q - sh + j;
                ret[j] = make_float2(0.0f, 0.0f);
                if (VEC || (c >= 0 && c < naz)) {
                    if (!(VEC && staged)) pt[j] = staged ? pat[c] : pattern_of(S, c, da, inv_sphi);
                    if (dense) {
                        ret[j].x = a.dense[off + 128 * k + j];
                        w[j].x = 0u;
                    } else if (!(VEC && staged)) {
                        w[j] = staged ? mask[c] : bands[c];
                    }
                } else {
                    w[j].x = 0u;
                }
            }
            if ((w[0].x | w[1].x | w[2].x | w[3].x) & bit) {
#pragma unroll
                for (int j = 0; j < 4; ++j)
                    if (w[j].x & bit) ret[j] = vals[w[j].y + __popc(w[j].x & below)];
            }
            const U4 x = additive_words((b0 >> 2) + (uint32_t)q, flo, fhi, K);
            const uint32_t xw[4] = {x.x, x.y, x.z, x.w};
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const int c = 4 * q - sh + j;
                v[j] = -CUDART_INF_F;
                p[j] = ret[j].x;
                if (VEC || (c >= 0 && c < naz)) {
                    const float add = additive_term(rc, inv_rmax2, pt[j], xw[j], sig_sa);
                    if (dense) {
                        v[j] = add;
                        if (ret[j].x != 0.0f)
                            v[j] = fmaf(ret[j].x, 0.5f + gauss_of(bin_draws(b0 + (uint32_t)c, S, K), a.params.sigma_sm), add);
                    } else {
                        v[j] = fmaf(ret[j].x, ret[j].y, add);
                    }
                }
            }
            if (!VEC) {   // bins over the row's ends (by column: a bin may be -inf): no part in its maximum
                const float most = fmaxf(fmaxf(v[0], v[1]), fmaxf(v[2], v[3]));   // (nor in the least value)
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    const int c = 4 * q - sh + j;
                    if (c < 0 || c >= naz) v[j] = most;
                }
            }
        };
        auto store = [&](float* to, int k, const float (&v)[4]) {   // `to`: the image at `off`
            if (VEC) {
                reinterpret_cast<float4*>(to)[32 * k] = make_float4(v[0], v[1], v[2], v[3]);
            } else {
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    const int c = 4 * (lane + 32 * k) - sh + j;
                    if (c >= 0 && c < naz) to[128 * k + j] = v[j];
                }
            }
        };
        float* const noised = a.noised + off;
        float* const polar = a.polar + off;
        const int nk = (nq - lane + 31) >> 5;   // the lane's quads
        float m = -CUDART_INF_F;
        if constexpr (REG > 0) {
            float v[REG][4];
            float least = CUDART_INF_F;
#pragma unroll
            for (int k = 0; k < REG; ++k) {
                if (k < nk) {
                    float p[4];
                    quad(k, v[k], p);
                    if (a.binned) store(a.binned + off, k, p);
                    store(noised, k, v[k]);
                    m = fmaxf(m, fmaxf(fmaxf(v[k][0], v[k][1]), fmaxf(v[k][2], v[k][3])));
                    least = fminf(least, fminf(fminf(v[k][0], v[k][1]), fminf(v[k][2], v[k][3])));
                }
            }
            for (int o = 16; o; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xFFFFFFFFu, m, o));
            // the row's values are the additive term (positive) and more unless a
            // reflectivity is negative: the general division is the exception
            if (__all_sync(0xFFFFFFFFu, least >= 0x1p-60f && m <= 0x1p60f) && mode == 1) {
                const float y = 1.0f / m;
#pragma unroll
                for (int k = 0; k < REG; ++k) {
                    if (k < nk) {
#pragma unroll
                        for (int j = 0; j < 4; ++j) v[k][j] = div_by(v[k][j], m, y);
                        store(polar, k, v[k]);
                    }
                }
            } else if (mode != 2) {
#pragma unroll
                for (int k = 0; k < REG; ++k) {
                    if (k < nk) {
#pragma unroll
                        for (int j = 0; j < 4; ++j) v[k][j] = norm_value(v[k][j], m, mode);
                        store(polar, k, v[k]);
                    }
                }
            }
        } else {
            for (int k = q0; k < nk; k += dq) {
                float v[4], p[4];
                quad(k, v, p);
                if (a.binned) store(a.binned + off, k, p);
                store(noised, k, v);
                m = fmaxf(m, fmaxf(fmaxf(v[0], v[1]), fmaxf(v[2], v[3])));
            }
            for (int o = 16; o; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xFFFFFFFFu, m, o));
            if (shared_row) {
                if (lane == 0) s_top[warp] = m;
                __syncthreads();   // the block has one row, and all its warps are here
#pragma unroll
                for (int w = 0; w < 8; ++w) m = fmaxf(m, s_top[w]);
            }
            if (mode != 2) {
                for (int k = q0; k < nk; k += dq) {
                    float v[4];
#pragma unroll
                    for (int j = 0; j < 4; ++j) {
                        const int c = 4 * (lane + 32 * k) - sh + j;
                        v[j] = VEC || (c >= 0 && c < naz) ? norm_value(noised[128 * k + j], m, mode) : 0.0f;
                    }
                    store(polar, k, v);
                }
            }
        }
        image_max = fmaxf(image_max, m);
    }
    // whole-image normalisation: the maximum of the image, divided by in a launch of its own
    if (mode == 2 && lane == 0) atomicMax(a.gmax + S.rowmax_off, ord_enc(image_max));
}

// The noise stream itself: Philox4x32-10 of n counters under one key, the
// same round function the fold, row, adjoint and DVL kernels draw from.
__global__ void __launch_bounds__(256) k_philox_words(const uint4* ctr, int64_t n, uint32_t k0, uint32_t k1,
                                                      uint4* out) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const uint4 c = ctr[i];
    const U4 x = philox10(U4{c.x, c.y, c.z, c.w}, philox_key(k0, k1));
    out[i] = make_uint4(x.x, x.y, x.z, x.w);
}

// ---------------------------------------------------------------------------
// phase 2a: whole-image normalisation
// ---------------------------------------------------------------------------

// N = I~ / max of the image, rows of up to 1024 16-byte-aligned bins: one warp per pair
// of adjacent rows, the pairs from the last to the first (the row kernel went the same
// way, so the first rows, written last, are in L2, and so is N for the fan).  Rows of up
// to 512 bins are loaded both before either is stored (4 KB in flight per warp), wider
// ones go one after the other.
__global__ void __launch_bounds__(256, 4) k_norm_rows(const __grid_constant__ NormArgs a) {
    let_next_start();
    wait_for_previous();   // I~ and its maximum
    const int64_t t = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int lane = threadIdx.x & 31;
    const int64_t pairs = (a.total_rows + 1) >> 1;
    if (t >= pairs) return;
    const int64_t g0 = 2 * (pairs - 1 - t);
    const int rows = (int)min((int64_t)2, a.total_rows - g0);
    float4 v[8];
    const float4* in[2];
    float4* out[2];
    int n4[2] = {0, 0};
    float m[2];
#pragma unroll
    for (int r = 0; r < 2; ++r) {
        if (r >= rows) continue;
        const SensorDev& s = a.sensors ? a.sensors[a.row_map[g0 + r]] : a.one;
        const int64_t off = s.polar_off + (g0 + r - s.rowmax_off) * s.naz;
        in[r] = reinterpret_cast<const float4*>(a.noised + off);
        out[r] = reinterpret_cast<float4*>(a.polar + off);
        n4[r] = s.naz >> 2;
        m[r] = ord_dec(a.gmax[s.rowmax_off]);
    }
    auto divided = [](float4 x, float top) {
        return make_float4(norm_value(x.x, top, 2), norm_value(x.y, top, 2), norm_value(x.z, top, 2), norm_value(x.w, top, 2));
    };
    if (max(n4[0], n4[1]) <= 128) {
#pragma unroll
        for (int k = 0; k < 8; ++k) {
            const int r = k >> 2, q = lane + 32 * (k & 3);
            if (q < n4[r]) v[k] = in[r][q];
        }
#pragma unroll
        for (int k = 0; k < 8; ++k) {
            const int r = k >> 2, q = lane + 32 * (k & 3);
            if (q < n4[r]) out[r][q] = divided(v[k], m[r]);
        }
        return;
    }
#pragma unroll
    for (int r = 0; r < 2; ++r) {
#pragma unroll
        for (int k = 0; k < 8; ++k)
            if (lane + 32 * k < n4[r]) v[k] = in[r][lane + 32 * k];
#pragma unroll
        for (int k = 0; k < 8; ++k)
            if (lane + 32 * k < n4[r]) out[r][lane + 32 * k] = divided(v[k], m[r]);
    }
}

// The same for rows of any width and alignment: one warp per run of 512 bins of a row
// (every a.runs-th run of it).  A frame of 50 x 20000 bins 523 us with a warp per pair
// of rows, 46 with this; 64 frames of 1000 x 511 333 -> 242; 64 frames of 1000 x 512, which
// the kernel above takes, 171 there and 184 here.
__global__ void __launch_bounds__(256) k_norm_runs(const __grid_constant__ NormArgs a) {
    let_next_start();
    wait_for_previous();   // I~ and its maximum
    const int64_t t = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int lane = threadIdx.x & 31;
    if (t >= a.total_rows * a.runs) return;
    const int64_t g = a.total_rows - 1 - t / a.runs;
    const SensorDev& s = a.sensors ? a.sensors[a.row_map[g]] : a.one;
    const int naz = s.naz;
    const int64_t off = s.polar_off + (g - s.rowmax_off) * naz;
    const float* In = a.noised + off;
    float* out = a.polar + off;
    const float m = ord_dec(a.gmax[s.rowmax_off]);
#pragma unroll 1
    for (int64_t j = 512 * (t % a.runs) + lane; j < naz; j += 512ll * a.runs) {
        float v[16];
#pragma unroll
        for (int k = 0; k < 16; ++k)
            if (j + 32 * k < naz) v[k] = In[j + 32 * k];
#pragma unroll
        for (int k = 0; k < 16; ++k)
            if (j + 32 * k < naz) out[j + 32 * k] = norm_value(v[k], m, 2);
    }
}

// ---------------------------------------------------------------------------
// phase 2b: fan resample of the normalised image
// ---------------------------------------------------------------------------

// What the pixels of one fan have in common.
struct FanGeo {
    float inv_scale, mid, top, rmin, rmax, inv_dr, half, az_scale;
    int nr, naz;
};
__device__ __forceinline__ FanGeo fan_geo(const SensorDev& s) {
    return FanGeo{1.0f / s.fan_scale, 0.5f * (float)s.fan_w, (float)s.fan_h, s.rmin, s.rmax, s.inv_dr, 0.5f * s.hfov,
                  (float)s.naz / s.hfov, s.nr, s.naz};
}

// Pixel (u, v) in metres: x to the right of the sensor, y ahead of it.
__device__ __forceinline__ float fan_x(const FanGeo& g, int u) { return ((float)u + 0.5f - g.mid) * g.inv_scale; }
__device__ __forceinline__ float fan_y(const FanGeo& g, int v) { return (g.top - (float)v - 0.5f) * g.inv_scale; }
__device__ __forceinline__ float fan_range(float x, float y) {
    return sqrtf(__fadd_rn(__fmul_rn(x, x), __fmul_rn(y, y)));
}

// A sample between two neighbouring bins of one axis, clamped to the edge bins:
// the lower bin, whether the upper one is another, and the weight towards it.
struct FanSpan {
    int at, more;
    float w;
};
__device__ __forceinline__ FanSpan fan_span(float f, int n) {
    const float f0 = floorf(f);
    const int i = (int)f0;
    const int lo = min(max(i, 0), n - 1), hi = min(max(i + 1, 0), n - 1);
    return FanSpan{lo, hi != lo ? 1 : 0, f - f0};
}
__device__ __forceinline__ FanSpan fan_row(const FanGeo& g, float r) {
    return fan_span(__fsub_rn(__fmul_rn(r - g.rmin, g.inv_dr), 0.5f), g.nr);
}
__device__ __forceinline__ FanSpan fan_col(const FanGeo& g, float phi) {
    return fan_span(__fsub_rn(__fmul_rn(phi + g.half, g.az_scale), 0.5f), g.naz);
}

// Where fan pixel `pix` samples the polar image: x = index of bin (ia, ja),
// y = (ib != ia ? naz : 0) << 1 | (jb != ja), z, w = the bilinear weights wr,
// wa (bit patterns); x = 0xFFFFFFFF outside the fan.  Bilinear over bin
// centres, clamped to the edge bins.
__device__ __forceinline__ uint4 fan_coord(const SensorDev& s, int64_t pix) {
    int v, u;
    if ((int64_t)s.fan_w * s.fan_h < (1ll << 31)) {
        v = (int)((uint32_t)pix / (uint32_t)s.fan_w);
        u = (int)pix - v * s.fan_w;
    } else {
        v = (int)(pix / s.fan_w);
        u = (int)(pix - (int64_t)v * s.fan_w);
    }
    const FanGeo g = fan_geo(s);
    const float x = fan_x(g, u), y = fan_y(g, v), r = fan_range(x, y), phi = atan2f(x, y);
    if (r < g.rmin || r > g.rmax || fabsf(phi) > g.half) return make_uint4(0xFFFFFFFFu, 0u, 0u, 0u);
    const FanSpan row = fan_row(g, r), col = fan_col(g, phi);
    return make_uint4((uint32_t)(row.at * g.naz + col.at),
                      ((row.more ? (uint32_t)g.naz : 0u) << 1) | (col.more ? 1u : 0u), __float_as_uint(row.w),
                      __float_as_uint(col.w));
}

// The same out of line, for kernels that read a table and need it rarely.
__device__ __noinline__ uint4 fan_coord_apart(const SensorDev& s, int64_t pix) { return fan_coord(s, pix); }

// The bilinear value at q = bin (ia, ja), dn and dj bins to the next row and
// column (explicit roundings: the table and the direct path give the same bits).
__device__ __forceinline__ float fan_bilinear(const float* q, uint32_t dn, uint32_t dj, float wr, float wa) {
    const float ua = 1.0f - wa, ur = 1.0f - wr;
    const float top = __fadd_rn(__fmul_rn(ua, q[0]), __fmul_rn(wa, q[dj]));
    const float bot = __fadd_rn(__fmul_rn(ua, q[dn]), __fmul_rn(wa, q[dn + dj]));
    return __fadd_rn(__fmul_rn(ur, top), __fmul_rn(wr, bot));
}

// The fan value at coordinates c over polar image P.
__device__ __forceinline__ float fan_blend(uint4 c, const float* P) {
    if (c.x == 0xFFFFFFFFu) return 0.0f;
    return fan_bilinear(P + c.x, c.y >> 1, c.y & 1u, __uint_as_float(c.z), __uint_as_float(c.w));
}

// The fan of sensors that share no coordinate table.  The fan is symmetric about
// its middle column: pixels u and fan_w - 1 - u have x and -x exactly, so the
// same range and opposite bearings, and one square root and arctangent serve
// both.  One block = kTileCols columns of the left half and their mirror
// columns, by kTileRows rows of one sensor (compact patches of the polar image,
// so the gathers stay in cache); a lane takes a column, a warp every eighth row.
// A pixel out of range needs no bearing.
// Bound by issue: 128 fans of unlike geometry (132 million pixels) 790 -> 428 us
// against a pixel per coordinate computation (and two integer divisions more),
// 397 with all 64 warps of an SM (32 registers instead of 40; both rows' gathers
// before the first store, which takes more of them: 407); one 1024 x 576 fan 9.1 ->
// 6.7 us.
__global__ void __launch_bounds__(256, 8) k_fan_tiles(const __grid_constant__ FanArgs a) {
    __shared__ SensorDev S;
    __shared__ int s_sq;
    let_next_start();
    if (threadIdx.x < 32) {
        if (a.block_map) {
            const int2 m = __ldg(a.block_map + blockIdx.x);
            copy_words(&S, a.sensors + m.x, threadIdx.x);
            if (threadIdx.x == 0) s_sq = m.y;
        } else {
            copy_param(&S, &a.one, threadIdx.x);
            if (threadIdx.x == 0) s_sq = blockIdx.x;
        }
    }
    __syncthreads();
    const int w = S.fan_w, half = (w + 1) / 2;
    const int sx = (half + kTileCols - 1) / kTileCols;
    const int u = (s_sq % sx) * kTileCols + (threadIdx.x & (kTileCols - 1));
    const int v0 = (s_sq / sx) * kTileRows + threadIdx.x / kTileCols;
    if (u >= half) return;
    const FanGeo g = fan_geo(S);
    const float* P = a.polar + S.polar_off;
    float* F = a.fan + S.fan_off;
    const int um = w - 1 - u;   // the mirror pixel (u itself in the middle of an odd width)
    const float x = fan_x(g, um);
    wait_for_previous();   // the normalised image
#pragma unroll
    for (int k = 0; k < kTileRows; k += 256 / kTileCols) {
        const int v = v0 + k;
        if (v >= S.fan_h) break;
        const float y = fan_y(g, v), r = fan_range(x, y);
        float left = 0.0f, right = 0.0f;
        if (!(r < g.rmin || r > g.rmax)) {
            const float phi = atan2f(x, y);
            if (!(fabsf(phi) > g.half)) {
                const FanSpan row = fan_row(g, r), cr = fan_col(g, phi), cl = fan_col(g, -phi);
                const float* q = P + (int64_t)row.at * g.naz;
                const uint32_t dn = row.more ? (uint32_t)g.naz : 0u;
                right = fan_bilinear(q + cr.at, dn, (uint32_t)cr.more, row.w, cr.w);
                left = fan_bilinear(q + cl.at, dn, (uint32_t)cl.more, row.w, cl.w);
            }
        }
        const int64_t at = (int64_t)v * w;   // never re-read here: stream past L2
        __stcs(F + at + um, right);
        if (um != u) __stcs(F + at + u, left);
    }
}

// The fan of the frames that share one coordinate table, in the same squares:
// one thread reads a pixel's table entry once and resamples that pixel for up
// to kFanGroup frames (a frame whose geometry no longer matches the table
// computes its own coordinates).  Bound by the latency of the table (16 bytes a
// pixel, read once from HBM) and of the frames' rows behind it: a thread takes two
// rows of two frames at a time, sixteen gathers in flight, and has asked for its next
// two table entries before.  That takes 64 registers, four blocks an SM, and is
// faster than more blocks with fewer gathers each (one pixel of one frame at a time,
// eight blocks -> this): 64 frames of 1024 x 576 131 -> 110 us (151 MB written, 131 MB
// read), 32 frames of 512 x 288 24 -> 14.  Four rows, four frames or squares of 32
// are slower by 5 to 30 %.
__global__ void __launch_bounds__(256, 4) k_fan_group(const __grid_constant__ FanGroupArgs a) {
    __shared__ SensorDev M[kFanGroup];
    __shared__ int4 s_m;
    __shared__ int s_w, s_h;
    __shared__ const uint4* s_lut;
    let_next_start();
    if (threadIdx.x == 0) {
        s_m = a.block_map[blockIdx.x];
        const SensorDev& o = a.sensors[s_m.x];
        s_w = o.fan_w;
        s_h = o.fan_h;
        s_lut = o.fan_lut;
    }
    __syncthreads();
    const int nm = s_m.w - s_m.z;
    constexpr int kWords = (int)(sizeof(SensorDev) / 4);
    for (int i = threadIdx.x; i < nm * kWords; i += blockDim.x) {
        const int q = i / kWords;
        reinterpret_cast<uint32_t*>(M)[i] =
            reinterpret_cast<const uint32_t*>(a.sensors + a.members[s_m.z + q])[i - q * kWords];
    }
    wait_for_previous();   // the normalised images and the table
    __syncthreads();
    const int w = s_w, h = s_h;
    const int sx = (w + kFanSide - 1) / kFanSide;
    const int u = (s_m.y % sx) * kFanSide + (threadIdx.x & (kFanSide - 1));
    const int v0 = (s_m.y / sx) * kFanSide + (threadIdx.x / kFanSide);
    if (u >= w) return;
    const uint4* lut = s_lut;
    constexpr int kStep = 256 / kFanSide, kRows = 2;
    bool shared = lut != nullptr;   // every frame here goes by the table
    const float* P[kFanGroup];
    float* F[kFanGroup];
#pragma unroll
    for (int q = 0; q < kFanGroup; ++q) {
        const SensorDev& m = M[q < nm ? q : 0];
        shared = shared && m.fan_lut != nullptr;
        P[q] = a.polar + m.polar_off;
        F[q] = a.fan + m.fan_off;
    }
    // the fan is never re-read by the step: streaming stores leave L2 to the polar
    // images and the coordinate table
    if (!shared) {
#pragma unroll 1
        for (int v = v0; v < min(v0 + kFanSide, h); v += kStep) {
            const int64_t pix = (int64_t)v * w + u;
            for (int q = 0; q < nm; ++q) {
                const uint4 c = lut && M[q].fan_lut ? lut[pix] : fan_coord_apart(M[q], pix);
                __stcs(a.fan + M[q].fan_off + pix, fan_blend(c, a.polar + M[q].polar_off));
            }
        }
        return;
    }
    const uint4 outside = make_uint4(0xFFFFFFFFu, 0u, 0u, 0u);
    uint4 ahead[kRows];   // the table's entries of the next rows, on their way during these
#pragma unroll
    for (int r = 0; r < kRows; ++r)
        ahead[r] = v0 + r * kStep < h ? lut[(int64_t)(v0 + r * kStep) * w + u] : outside;
#pragma unroll 1
    for (int k = 0; k < kFanSide; k += kRows * kStep) {
        const int v = v0 + k;
        if (v >= h) break;
        const int64_t pix = (int64_t)v * w + u, step = (int64_t)kStep * w;
        uint4 c[kRows];
#pragma unroll
        for (int r = 0; r < kRows; ++r) {
            c[r] = ahead[r];
            ahead[r] = v + (r + kRows) * kStep < h ? lut[pix + (r + kRows) * step] : outside;
        }
        // every gather before the first store: the compiler must not move a load
        // above a store that might alias it
        float value[kRows][kFanGroup];
#pragma unroll
        for (int r = 0; r < kRows; ++r) {
            const bool in = c[r].x != 0xFFFFFFFFu;   // else the image's first bin is read and dropped
            const uint32_t at = in ? c[r].x : 0u, dn = c[r].y >> 1, dj = c[r].y & 1u;
#pragma unroll
            for (int q = 0; q < kFanGroup; ++q) {
                const float x = fan_bilinear(P[q] + at, dn, dj, __uint_as_float(c[r].z), __uint_as_float(c[r].w));
                value[r][q] = in ? x : 0.0f;
            }
        }
#pragma unroll
        for (int r = 0; r < kRows; ++r)
            if (v + r * kStep < h) {
#pragma unroll
                for (int q = 0; q < kFanGroup; ++q)
                    if (q < nm) __stcs(F[q] + pix + r * step, value[r][q]);
            }
    }
}

// Fills the coordinate table of each owner sensor (one block = kFanTile
// pixels).  A block whose stamp already holds the owner's fan_version has
// nothing to do: the table depends on the fan geometry only, and the host bumps
// the version whenever an update changes it.
// The tables depend on nothing that the kernels before it in a forward write, so it
// works first and waits last (the kernel after it waits for this one alone).
__global__ void __launch_bounds__(256) k_fan_lut(const __grid_constant__ FanLutArgs a) {
    let_next_start();
    __shared__ SensorDev S;
    __shared__ int s_blk;
    __shared__ bool s_current;
    __shared__ uint4* s_lut;
    if (threadIdx.x == 0) {
        const int2 m = a.block_map[blockIdx.x];
        S = a.sensors[m.x];
        s_blk = m.y;
        s_lut = a.luts[m.x];
        s_current = S.fan_stamp && S.fan_stamp[m.y] == S.fan_version;   // read once for all (see k_trig)
    }
    __syncthreads();
    if (s_current) {
        wait_for_previous();
        return;
    }
    const int64_t base = (int64_t)s_blk * kFanTile;
    const int64_t n = (int64_t)S.fan_w * S.fan_h;
#pragma unroll 1
    for (int k = 0; k < kFanTile / 256; ++k) {
        const int64_t pix = base + k * 256 + threadIdx.x;
        if (pix < n) s_lut[pix] = fan_coord(S, pix);
    }
    // the entries are read by later launches only, which see both them and the stamp
    if (threadIdx.x == 0 && S.fan_stamp) S.fan_stamp[s_blk] = S.fan_version;
    wait_for_previous();
}

// ---------------------------------------------------------------------------
// adjoint
// ---------------------------------------------------------------------------

// Group terms of the normalisation Jacobian: m, argmax (lowest index on
// ties) and c = sum G I~ / m^2, one warp per range row, or per `per_warp` of them
// one after another.
// Bound by HBM, and by what a warp waits for between rows: the place of its row (two
// dependent loads), its bins, the reduction.  So every load of up to 512 bins is
// issued before the first compare, and what follows (the row's next 512 bins, the
// next row) is asked for before the reduction.  128,000 rows of 1024 bins 192 -> 157
// us (6.7 TB/s), 64,000 rows of 512 bins 55 -> 53 (57 with a row per warp); more
// warps of fewer registers spill.
__global__ void __launch_bounds__(256, 4) k_adj_rows(const SensorDev* sensors, const int32_t* row_map, SensorDev one,
                                                  int64_t total, int per_warp, int aligned, const float* noised,
                                                  const float* grad, RowInfo* info, int32_t* zero_word) {
    let_next_start();
    wait_for_previous();
    const int lane = threadIdx.x & 31;
    if (zero_word && blockIdx.x == 0 && threadIdx.x == 0) *zero_word = 0;   // the gather's work counter
    const int64_t g0 = (((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5) * per_warp;
    float4 xs[4], ys[4];   // 512 bins of I~ and G, each lane's vectors
    int naz = 0, row = 0;
    int64_t off = 0;
    bool vec = false;
    auto place = [&](int64_t g) {
        const SensorDev& s = sensors ? sensors[__ldg(row_map + g)] : one;
        naz = s.naz;
        row = (int)(g - s.rowmax_off);
        off = s.polar_off + (int64_t)row * naz;
        vec = aligned && ((s.polar_off | naz) & 3) == 0;
    };
    auto ask = [&](int j0) {   // bins j0 .. j0 + 511 of the row
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const int j = j0 + 4 * (lane + 32 * k);
            if (j < naz) {   // I~ is not read again by the adjoint: evict first, keep G in L2
                xs[k] = __ldcs(reinterpret_cast<const float4*>(noised + off + j));
                ys[k] = __ldg(reinterpret_cast<const float4*>(grad + off + j));
            }
        }
    };
    if (g0 < total) {
        place(g0);
        if (vec) ask(0);
    }
    for (int64_t g = g0; g < g0 + per_warp && g < total; ++g) {
        const bool more = g + 1 < g0 + per_warp && g + 1 < total;
        const int base = row * naz;
        float m = -CUDART_INF_F;
        int am = 0x7FFFFFFF;
        float dl = 0.0f;                      // per-lane partial of sum G I~ (few terms)
        if (vec) {
            // what follows is asked for as soon as these bins are taken: the row's
            // next 512, or the next row, on its way during the reduction
#pragma unroll 1
            for (int j0 = 0, n = naz; j0 < n; j0 += 512) {
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    const int j = j0 + 4 * (lane + 32 * k);
                    if (j >= n) continue;
                    const float4 x = xs[k], y = ys[k];   // four consecutive bins, in index order
                    if (x.x > m) { m = x.x; am = j; }
                    if (x.y > m) { m = x.y; am = j + 1; }
                    if (x.z > m) { m = x.z; am = j + 2; }
                    if (x.w > m) { m = x.w; am = j + 3; }
                    dl = fmaf(y.x, x.x, dl);
                    dl = fmaf(y.y, x.y, dl);
                    dl = fmaf(y.z, x.z, dl);
                    dl = fmaf(y.w, x.w, dl);
                }
                if (j0 + 512 < n) {
                    ask(j0 + 512);
                } else if (more) {
                    place(g + 1);
                    if (vec) ask(0);
                }
            }
        } else {
            for (int j = lane; j < naz; j += 32) {
                const float x = noised[off + j];
                if (x > m) { m = x; am = j; }
                dl = fmaf(grad[off + j], x, dl);
            }
            if (more) {
                place(g + 1);
                if (vec) ask(0);
            }
        }
        // lane partials added across the warp in float-float (error-free
        // two-sums on the FP32 pipes: FP64 would cost more than the row's loads)
        ff dot{dl, 0.0f};
        for (int o = 16; o; o >>= 1) {
            const float m2 = __shfl_xor_sync(0xFFFFFFFFu, m, o);
            const int a2 = __shfl_xor_sync(0xFFFFFFFFu, am, o);
            if (m2 > m || (m2 == m && a2 < am)) { m = m2; am = a2; }
            const ff d2{__shfl_xor_sync(0xFFFFFFFFu, dot.hi, o), __shfl_xor_sync(0xFFFFFFFFu, dot.lo, o)};
            dot = ff_add(dot, d2);
        }
        if (lane == 0) {
            RowInfo r;
            r.m = m;
            r.valid = m > 0.0f;
            r.c = r.valid ? (__fadd_rn(dot.hi, dot.lo) / m) / m : 0.0f;
            r.arg = base + am;
            info[g] = r;
        }
    }
}

// The same for whole images: one block per image.
__global__ void __launch_bounds__(1024) k_adj_images(const SensorDev* sensors, SensorDev one, int64_t total,
                                                     const float* noised, const float* grad, RowInfo* info,
                                                     int32_t* zero_word) {
    let_next_start();
    wait_for_previous();
    const int lane = threadIdx.x & 31;
    if (zero_word && blockIdx.x == 0 && threadIdx.x == 0) *zero_word = 0;   // the gather's work counter
    __shared__ float s_m[32];
    __shared__ int s_a[32];
    __shared__ ff s_d[32];
    const int si = blockIdx.x;
    if (si >= total) return;
    const SensorDev& s = sensors ? sensors[si] : one;
    const int64_t n = (int64_t)s.nr * s.naz;
    const float* In = noised + s.polar_off;
    const float* G = grad + s.polar_off;
    float m = -CUDART_INF_F;
    int am = 0x7FFFFFFF;
    ff dot{0.0f, 0.0f};   // float-float: products exact (FMA), sums error-free
    for (int64_t j = threadIdx.x; j < n; j += blockDim.x) {
        const float x = In[j], y = G[j];
        if (x > m) { m = x; am = (int)j; }
        const float p = __fmul_rn(y, x);
        dot = ff_add(dot, ff{p, fmaf(y, x, -p)});
    }
    for (int o = 16; o; o >>= 1) {
        const float m2 = __shfl_xor_sync(0xFFFFFFFFu, m, o);
        const int a2 = __shfl_xor_sync(0xFFFFFFFFu, am, o);
        if (m2 > m || (m2 == m && a2 < am)) { m = m2; am = a2; }
        const ff d2{__shfl_xor_sync(0xFFFFFFFFu, dot.hi, o), __shfl_xor_sync(0xFFFFFFFFu, dot.lo, o)};
        dot = ff_add(dot, d2);
    }
    const int w = threadIdx.x >> 5;
    if (lane == 0) { s_m[w] = m; s_a[w] = am; s_d[w] = dot; }
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int k = 1; k < (int)(blockDim.x >> 5); ++k) {
            if (s_m[k] > m || (s_m[k] == m && s_a[k] < am)) { m = s_m[k]; am = s_a[k]; }
            dot = ff_add(dot, s_d[k]);
        }
        RowInfo r;
        r.m = m;
        r.valid = m > 0.0f;
        r.c = r.valid ? (__fadd_rn(dot.hi, dot.lo) / m) / m : 0.0f;
        r.arg = am;
        info[s.rowmax_off] = r;
    }
}

// Per-ray gather of dL/dP and accumulation of dtheta over a unit of rays,
// reading the hit records (stored by the forward, or recomputed by the ray-cast
// kernel just before: bitwise the same records).
// Deterministic: each unit's sums go to its own row of `partials` (material
// sums per warp in lane order, warp slabs added in warp order, alpha/gain per
// thread then in a fixed tree); k_adj_final adds the rows in a fixed order.
// A unit holds a few hundred rays: its sums are FP32 (float-float across
// lanes), its row of partials FP64.
__global__ void __launch_bounds__(512) k_adjoint(const __grid_constant__ AdjArgs a) {
    extern __shared__ double slab_d[];   // [n_warps][n_mat] (FP32 sums; sized in doubles by the host)
    float* slab = reinterpret_cast<float*>(slab_d);
    __shared__ SensorDev S;
    __shared__ SceneDev SC;
    __shared__ AdjUnit U;
    __shared__ int s_unit;
    __shared__ ff s_ag[2][32];
    let_next_start();
    const int tid = threadIdx.x, nt = blockDim.x;
    const int lane = tid & 31, warp = tid >> 5, nw = nt >> 5;
    const int nm = a.n_mat, nq = nm + 2;
    const float alpha = __ldg(a.theta), gain = __ldg(a.theta + 1);
    const int mode = a.params.normalise;
    int next_u = 0;   // thread 0: the unit taken ahead
    wait_for_previous();   // the row terms, the work counter
    for (int iter = 0;; ++iter) {
        int u;
        if (a.work_counter) {
            if (tid == 0) s_unit = iter == 0 ? atomicAdd(a.work_counter, 1) : next_u;
            __syncthreads();
            u = s_unit;
            if (tid == 0 && u < a.n_units) next_u = atomicAdd(a.work_counter, 1);
        } else {
            if (iter > 0) break;
            u = blockIdx.x;
        }
        if (u >= a.n_units) break;
        if (a.units && warp == 0) {   // warp 0 fetches the unit, then its sensor and scene descriptors at once
            const AdjUnit un = a.units[u];
            copy_words(&S, a.sensors + un.sensor, lane);
            copy_words(&SC, a.scenes + un.scene, lane);
            if (lane == 0) U = un;
        }
        if (!a.units && warp == 0) {
            copy_param(&S, &a.one, lane);
            copy_param(&SC, &a.one_scene, lane);
        }
        if (!a.units && tid == 0) {
            U.sensor = 0;
            U.r0 = u * a.chunk;
            U.r1 = min(U.r0 + a.chunk, a.one.nb * a.one.ne);
        }
        for (int k = tid; k < nw * nm; k += nt) slab[k] = 0.0f;
        __syncthreads();
        const PhiloxKey K = philox_key(S.seed_lo, S.seed_hi);
        float acc_a = 0.0f, acc_g = 0.0f;
        for (int base = U.r0; base < U.r1; base += nt) {
            const int r = base + tid;
            bool valid = false;
            int mat = 0;
            float v_mu = 0.0f;
            if (r < U.r1) {
                const uint4 h = *reinterpret_cast<const uint4*>(a.hits + S.hits_off + r);
                const uint32_t key = h.x, orig = h.y;
                const float rr = __uint_as_float(h.z), cf = __uint_as_float(h.w);
                if (key != kNoKey) {
                    if (key >= (uint32_t)(S.nr * S.naz) || orig >= (uint32_t)SC.n_tris) {
                        atomicOr(a.err, SONAR_DEVERR_INDEX);
                    } else {
                        const float G = a.grad[S.polar_off + key];
                        float gI = G;
                        if (mode != 0) {
                            const RowInfo ri = a.rowinfo[S.rowmax_off + (mode == 1 ? (int)(key / S.naz) : 0)];
                            if (ri.valid) gI = G / ri.m - ((int)key == ri.arg ? ri.c : 0.0f);
                        }
                        const float gP = gI * (0.5f + w_sm_of(key, S, a.params.sigma_sm, K));
                        mat = SC.mat_orig[orig];
                        mat = mat < nm ? mat : nm - 1;
                        const float mu = __ldg(a.theta + 2 + mat);
                        const float ca = gP * cf * expf(-2.0f * alpha * rr);
                        v_mu = ca * gain;
                        acc_a = fmaf(ca * gain * mu, -2.0f * rr, acc_a);
                        acc_g = fmaf(ca, mu, acc_g);
                        valid = true;
                    }
                }
            }
            // material sums of this warp: one butterfly reduction (a fixed order,
            // so deterministic) per distinct material among the valid lanes,
            // added to the slab by the material's lowest lane
            uint32_t todo = __ballot_sync(0xFFFFFFFFu, valid);
            while (todo) {
                const int leader = __ffs(todo) - 1;
                const int m = __shfl_sync(0xFFFFFFFFu, mat, leader);
                const bool mine = valid && mat == m;
                float x = mine ? v_mu : 0.0f;
                for (int o = 16; o; o >>= 1) x += __shfl_xor_sync(0xFFFFFFFFu, x, o);
                if (lane == leader) slab[warp * nm + m] += x;
                todo &= ~__ballot_sync(0xFFFFFFFFu, mine);
            }
        }
        ff da{acc_a, 0.0f}, dg{acc_g, 0.0f};
        for (int o = 16; o; o >>= 1) {
            da = ff_add(da, ff{__shfl_down_sync(0xFFFFFFFFu, da.hi, o), __shfl_down_sync(0xFFFFFFFFu, da.lo, o)});
            dg = ff_add(dg, ff{__shfl_down_sync(0xFFFFFFFFu, dg.hi, o), __shfl_down_sync(0xFFFFFFFFu, dg.lo, o)});
        }
        if (lane == 0) { s_ag[0][warp] = da; s_ag[1][warp] = dg; }
        __syncthreads();
        double* out = a.partials + (int64_t)u * nq;
        for (int m = tid; m < nm; m += nt) {
            ff v{0.0f, 0.0f};
            for (int w = 0; w < nw; ++w) v = ff_add(v, ff{slab[w * nm + m], 0.0f});
            out[2 + m] = (double)v.hi + (double)v.lo;
        }
        if (tid == 0) {
            ff va{0.0f, 0.0f}, vg{0.0f, 0.0f};
            for (int w = 0; w < nw; ++w) { va = ff_add(va, s_ag[0][w]); vg = ff_add(vg, s_ag[1][w]); }
            out[0] = (double)va.hi + (double)va.lo;
            out[1] = (double)vg.hi + (double)vg.lo;
        }
        __syncthreads();
    }
}

// dtheta[q] = sum over units of partials[u][q]: a fixed strided split over the
// threads, then a fixed tree.
__global__ void __launch_bounds__(256) k_adj_final(const double* partials, int n_units, int nq, float* dtheta) {
    __shared__ double red[256];
    const int q = blockIdx.x;
    wait_for_previous();   // the partial sums
    double v = 0.0;
    for (int u = threadIdx.x; u < n_units; u += 256) v += partials[(int64_t)u * nq + q];
    red[threadIdx.x] = v;
    __syncthreads();
    for (int w = 128; w > 0; w >>= 1) {
        if (threadIdx.x < w) red[threadIdx.x] += red[threadIdx.x + w];
        __syncthreads();
    }
    if (threadIdx.x == 0) dtheta[q] = (float)red[0];
}
}  // namespace

// ---------------------------------------------------------------------------
// launchers
// ---------------------------------------------------------------------------

void set_kernel_attributes() {
    cudaFuncSetAttribute(k_fold, cudaFuncAttributeMaxDynamicSharedMemorySize, kMaxDynSmem);
    cudaFuncSetAttribute(k_rows<0, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, kMaxDynSmem);
    cudaFuncSetAttribute(k_rows<0, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, kMaxDynSmem);
    cudaFuncSetAttribute(k_adjoint, cudaFuncAttributeMaxDynamicSharedMemorySize, kMaxDynSmem);
}

cudaError_t launch_fold(const FoldArgs& a, int grid, int block, size_t smem, cudaStream_t st, bool early) {
    return grid > 0 ? launch_kernel(k_fold, grid, block, smem, st, early, a) : cudaSuccess;
}

// The row kernel for rows of up to `naz` bins: in registers up to 512 and up to
// 1024 bins, else written and read back.  `staged`: the widest of the launch's
// sensors whose column tables are staged (no wider than kRowsStaged; 0: none), which
// may be a narrower one than the widest.  `vec`: 16-byte stores (every row of
// every sensor starts on a 16-byte boundary of each image).
cudaError_t launch_rows(const RowsArgs& a, int grid, int naz, int staged, bool vec, cudaStream_t st, bool early) {
    if (grid <= 0) return cudaSuccess;
    // a row whose first bin is not a multiple of 4 may need one quad more
    const int reach = vec ? naz : naz + 3;
    const size_t smem = ((size_t)((staged + 3) & ~3) + 2 * (size_t)staged) * sizeof(uint32_t);
    if (reach <= 512 && !a.dense)
        return launch_kernel(vec ? k_rows<4, true> : k_rows<4, false>, grid, 256, smem, st, early, a);
    if (reach <= 1024 && !a.dense)
        return launch_kernel(vec ? k_rows<8, true> : k_rows<8, false>, grid, 256, smem, st, early, a);
    return launch_kernel(vec ? k_rows<0, true> : k_rows<0, false>, grid, 256, smem, st, early, a);
}

cudaError_t launch_philox(const void* ctr, int64_t n, uint32_t k0, uint32_t k1, void* out, cudaStream_t st) {
    if (n > 0)
        k_philox_words<<<(unsigned)((n + 255) / 256), 256, 0, st>>>(static_cast<const uint4*>(ctr), n, k0, k1,
                                                                      static_cast<uint4*>(out));
    return cudaGetLastError();
}

cudaError_t launch_norm(const NormArgs& a, cudaStream_t st, bool early) {
    const int64_t warps = a.runs ? a.total_rows * a.runs : (a.total_rows + 1) / 2;
    return launch_kernel(a.runs ? k_norm_runs : k_norm_rows, (unsigned)((warps + 7) / 8), 256, 0, st, early, a);
}

cudaError_t launch_fan_tiles(const FanArgs& a, int blocks, cudaStream_t st, bool early) {
    return blocks > 0 ? launch_kernel(k_fan_tiles, blocks, 256, 0, st, early, a) : cudaSuccess;
}

cudaError_t launch_fan_group(const FanGroupArgs& a, int blocks, cudaStream_t st, bool early) {
    return blocks > 0 ? launch_kernel(k_fan_group, blocks, 256, 0, st, early, a) : cudaSuccess;
}

cudaError_t launch_fan_lut(const FanLutArgs& a, int blocks, cudaStream_t st, bool early) {
    return blocks > 0 ? launch_kernel(k_fan_lut, blocks, 256, 0, st, early, a) : cudaSuccess;
}

cudaError_t launch_adj_rows(const SensorDev* sensors, const int32_t* row_map, const SensorDev& one,
                            int64_t total_groups, int normalise, bool aligned, const float* noised,
                            const float* grad, RowInfo* info, int32_t* zero_word, cudaStream_t st, bool early) {
    if (normalise == 0) return cudaSuccess;
    if (normalise != 1)
        return launch_kernel(k_adj_images, (unsigned)total_groups, 1024, 0, st, early, sensors, one, total_groups, noised,
                             grad, info, zero_word);
    // two rows a warp once the launch is four waves or so (32 warps on each of 152 SMs);
    // four are no faster
    const int per_warp = total_groups >= 20000 ? 2 : 1;
    const int64_t warps = (total_groups + per_warp - 1) / per_warp;
    return launch_kernel(k_adj_rows, (unsigned)((warps + 7) / 8), 256, 0, st, early, sensors, row_map, one, total_groups,
                         per_warp, (int)aligned, noised, grad, info, zero_word);
}

cudaError_t launch_adjoint(const AdjArgs& a, int grid, int block, size_t smem, float* dtheta, cudaStream_t st,
                           bool early, bool early_final) {
    const cudaError_t e = launch_kernel(k_adjoint, grid, block, smem, st, early, a);
    if (e != cudaSuccess) return e;
    return launch_kernel(k_adj_final, a.n_mat + 2, 256, 0, st, early_final, (const double*)a.partials, (int)a.n_units,
                         (int)(a.n_mat + 2), dtheta);
}

int adjoint_blocks_per_sm(int block, size_t smem) {
    int n = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, (const void*)k_adjoint, block, smem) != cudaSuccess) return 1;
    return n > 0 ? n : 1;
}

}  // namespace sonar

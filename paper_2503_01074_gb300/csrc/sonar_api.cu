// C ABI of libsonar: contexts, scenes, single-frame and batched rendering,
// the adjoint, the autotuner and the counter mode.  Host code only; kernels
// live in bvh_build.cu, trace.cu, render.cu, image.cu and dvl.cu.
#include <cuda_runtime.h>
#include <stdint.h>

#include <algorithm>
#include <array>
#include <cmath>
#include <cstring>
#include <map>
#include <mutex>
#include <string>
#include <vector>

#include "sonar_host.h"
#include "sonar_internal.cuh"

using namespace sonar;

namespace {

struct Tune {
    int cols = 1;     // kept for saved rows: the fold takes one azimuth column per warp
    int tb = 0;       // tracing: beams per warp tile, elevations = 32 / tb (0: derive)
    int block = 128;  // adjoint: threads per block (which also sets its ray chunks)
    int occ = 0;      // tracing variant: kTraceCap caps registers at 64 (32 warps per SM),
                      // kTraceWide walks the 8-wide tree
};

using ShapeKey = std::array<int, 4>;   // n_beams, n_elev, n_range_bins, n_az_bins

// A device buffer that grows on demand (stream-ordered allocation).
struct Scratch {
    void* p = nullptr;
    size_t bytes = 0;
};

}  // namespace

struct sonar_ctx {
    int device = 0;
    int sm_count = 1;
    std::vector<SceneStore> scenes;
    std::vector<bool> alive;
    std::string last_error;
    uint32_t* d_err = nullptr;
    cudaMemPool_t pool = nullptr;   // scenes and the scratch of their builds
    Scratch rowmax, noised, rowinfo, partials, counters, hits, trig, vals, bands;
    // the exact-ray tables last built by a single-sensor call: their buffer and
    // the angular geometry they hold (beams, elevations, fields of view)
    const float4* trig_at = nullptr;
    int trig_nb = 0, trig_ne = 0;
    float trig_hfov = 0.0f, trig_vfov = 0.0f;
    std::map<ShapeKey, Tune> tune;
};

struct sonar_batch;

namespace {

sonar_status fail(sonar_ctx* ctx, sonar_status st, const std::string& msg) {
    if (ctx) ctx->last_error = msg;
    return st;
}

// The runtime keeps a failed call's error until it is read, and the next launch that
// looks (cudaGetLastError) would report it again: taken here, where it is reported.
sonar_status cuda_fail(sonar_ctx* ctx, cudaError_t e, const char* what) {
    cudaGetLastError();
    return fail(ctx, e == cudaErrorMemoryAllocation ? SONAR_ERR_OOM : SONAR_ERR_CUDA,
                std::string(what) + ": " + cudaGetErrorString(e));
}

#define CU(call, what)                                   \
    do {                                                 \
        cudaError_t e_ = (call);                         \
        if (e_ != cudaSuccess) return cuda_fail(ctx, e_, what); \
    } while (0)

cudaError_t grow(Scratch& s, size_t bytes, cudaStream_t st) {
    if (s.bytes >= bytes && s.p) return cudaSuccess;
    if (s.p) cudaFreeAsync(s.p, st);
    s.p = nullptr;
    s.bytes = 0;
    size_t want = std::max(bytes, (size_t)256);
    cudaError_t e = cudaMallocAsync(&s.p, want, st);
    if (e == cudaSuccess) s.bytes = want;
    return e;
}

bool finite_f(float x) { return std::isfinite(x); }

sonar_status check_sensor(sonar_ctx* ctx, const sonar_sensor* s) {
    if (!s) return fail(ctx, SONAR_ERR_ARG, "sensor is NULL");
    if (s->n_beams < 1 || s->n_elev < 1 || s->n_range_bins < 1 || s->n_az_bins < 1)
        return fail(ctx, SONAR_ERR_ARG, "sensor counts must be >= 1");
    if ((int64_t)s->n_beams * s->n_elev > 0x7FFFFFFFll)
        return fail(ctx, SONAR_ERR_ARG, "n_beams * n_elev exceeds 2^31 - 1");
    if ((int64_t)s->n_range_bins * s->n_az_bins > 0x7FFFFFFEll)
        return fail(ctx, SONAR_ERR_ARG, "n_range_bins * n_az_bins exceeds 2^31 - 2");
    for (int k = 0; k < 3; ++k)
        if (!finite_f(s->pos[k])) return fail(ctx, SONAR_ERR_ARG, "sensor position not finite");
    for (int k = 0; k < 9; ++k)
        if (!finite_f(s->rot[k])) return fail(ctx, SONAR_ERR_ARG, "sensor rotation not finite");
    const float pi = 3.14159265358979f;
    if (!(s->hfov > 0.0f && s->hfov <= pi)) return fail(ctx, SONAR_ERR_ARG, "hfov must be in (0, pi]");
    if (!(s->vfov > 0.0f && s->vfov <= pi)) return fail(ctx, SONAR_ERR_ARG, "vfov must be in (0, pi]");
    if (!(s->r_min >= 0.0f && s->r_max > s->r_min && finite_f(s->r_max)))
        return fail(ctx, SONAR_ERR_ARG, "need 0 <= r_min < r_max < inf");
    return SONAR_OK;
}

sonar_status check_params(sonar_ctx* ctx, const sonar_params* p) {
    if (!p) return fail(ctx, SONAR_ERR_ARG, "params is NULL");
    if (!(p->sigma_sa >= 0.0f && finite_f(p->sigma_sa))) return fail(ctx, SONAR_ERR_ARG, "sigma_sa must be >= 0");
    if (!(p->sigma_sm >= 0.0f && finite_f(p->sigma_sm))) return fail(ctx, SONAR_ERR_ARG, "sigma_sm must be >= 0");
    if (!(p->sigma_phi > 0.0f && finite_f(p->sigma_phi))) return fail(ctx, SONAR_ERR_ARG, "sigma_phi must be > 0");
    if (p->normalise < 0 || p->normalise > 2) return fail(ctx, SONAR_ERR_ARG, "normalise must be 0, 1 or 2");
    if (p->two_sided < 0 || p->two_sided > 1) return fail(ctx, SONAR_ERR_ARG, "two_sided must be 0 or 1");
    if (p->clip_tmax < 0 || p->clip_tmax > 1) return fail(ctx, SONAR_ERR_ARG, "clip_tmax must be 0 or 1");
    if (p->accumulate < 0 || p->accumulate > 1) return fail(ctx, SONAR_ERR_ARG, "accumulate must be 0 or 1");
    return SONAR_OK;
}

sonar_status check_scene(sonar_ctx* ctx, int32_t id) {
    if (id < 0 || id >= (int32_t)ctx->scenes.size() || !ctx->alive[id])
        return fail(ctx, SONAR_ERR_ARG, "unknown scene id " + std::to_string(id));
    return SONAR_OK;
}

sonar_status check_nmat(sonar_ctx* ctx, int32_t scene, int32_t n_mat) {
    if (n_mat < 1 || n_mat > kMaxMat) return fail(ctx, SONAR_ERR_ARG, "n_mat must be in [1, 1024]");
    if (ctx->scenes[scene].max_mat >= n_mat)
        return fail(ctx, SONAR_ERR_ARG, "scene uses material id " + std::to_string(ctx->scenes[scene].max_mat) +
                                             " >= n_mat " + std::to_string(n_mat));
    return SONAR_OK;
}

bool aligned16(const void* p) { return ((uintptr_t)p & 15u) == 0; }

// Launch shapes for a sensor: the tuning cache entry, else the defaults.
Tune tune_for(const sonar_ctx* ctx, const sonar_sensor& s) {
    Tune t;
    auto it = ctx->tune.find(ShapeKey{s.n_beams, s.n_elev, s.n_range_bins, s.n_az_bins});
    if (it != ctx->tune.end()) t = it->second;
    if (t.block < 32 || t.block > 512 || (t.block & 31)) t.block = 128;
    if (t.tb <= 0) t.tb = 8;
    if (t.tb > 32 || (t.tb & (t.tb - 1))) t.tb = 8;
    return t;
}

// Several lanes per ray (0: one) for a launch of `tiles` 32-ray tiles, while it is a
// small part of a wave: the crossings, measured with k_trace_group, lie near 20,000
// rays (eight lanes against four) and 105,000 rays (four against one).
int group_lanes(const sonar_ctx* ctx, int64_t tiles) {
    if (tiles <= 4ll * ctx->sm_count) return kTraceGroup8;
    return tiles <= 22ll * ctx->sm_count ? kTraceGroup4 : 0;
}

// The variant of a launch of `tiles` 32-ray tiles that no tuning row names: several
// lanes per ray on the 8-wide tree for small launches, else a lane per ray on the
// 4-wide one, capped at 64 registers (32 resident warps per SM instead of 28)
// once the launch is at least two waves.  Uncapped / capped / on the 8-wide tree:
// 4,096 tiles 56.1 / 56.4 / 59.8 us, 8,192 tiles of shorter rays 63.8 / 66.1 / 80.4
// us, 65,536 tiles 372 / 362 / 573 us, 227,072 tiles of three sensor types 1027 /
// 999 / 1625 us.
int default_variant(const sonar_ctx* ctx, int64_t tiles) {
    if (const int lanes = group_lanes(ctx, tiles)) return kTraceWide | lanes;
    return tiles >= 64ll * ctx->sm_count ? kTraceCap : 0;
}

// The ray-cast variant of one sensor's own launch (tile tb, variant `occ` of its
// tuning row, if it has one): a launch of at most one wave takes the default of
// its size (tuning rows are made by batches), a larger one the 4-wide tree with
// its row's cap.
int single_variant(const sonar_ctx* ctx, const sonar_sensor& s, int tb, int occ) {
    const int64_t be = 32 / tb;
    const int64_t tiles = ((s.n_beams + tb - 1) / tb) * ((s.n_elev + be - 1) / be);
    const bool tuned = ctx->tune.count(ShapeKey{s.n_beams, s.n_elev, s.n_range_bins, s.n_az_bins}) != 0;
    if (!tuned || tiles <= 32ll * ctx->sm_count) return default_variant(ctx, tiles);
    return occ & ~kTraceWide;
}

// A single frame alone on the GPU: the tuned shapes, and the ray-cast variant
// chosen by the frame's own launch size.
Tune single_tune(const sonar_ctx* ctx, const sonar_sensor& s) {
    Tune t = tune_for(ctx, s);
    t.occ = single_variant(ctx, s, t.tb, t.occ);
    return t;
}

// Most beams of an azimuth column (n_beams spread over n_az_bins columns).
int64_t col_beams_max(const SensorDev& s) { return (s.nb + (int64_t)s.naz - 1) / s.naz; }

int64_t band_count(const SensorDev& s) { return ((int64_t)s.nr + 31) / 32; }

// Shared-memory words of a column in the fold: the rows' bitmap and its ranks,
// then the rows and sums of the bins with returns (no more than rays, nor than
// rows), the sums per beam in the per-beam form.
int64_t fold_words(const SensorDev& s) {
    const int64_t most = std::min<int64_t>(s.nr, col_beams_max(s) * s.ne);
    return 2 * band_count(s) + most * (1 + (s.fold_beams ? col_beams_max(s) : 1));
}

// Whether a sensor's columns take a block each in a launch of `columns` columns, also
// without per-beam rows (the sums are the same either way): few columns of many rays,
// whose rows the block's warps then mark together.  Frames, a warp a column -> a block:
// 256 columns of 1024 rays into 100 range bins 165 -> 91 us; 64 of 4096 310 -> 167; 4 of 1024 into
// 8000 57 -> 45, of 16,384 468 -> 366; fewer rays a column gain nothing, and 512 columns of
// 4096 in a batch take 456 instead of 418.
bool fold_by_block(const SensorDev& s, int64_t columns) {
    return s.fold_beams || (columns <= 256 && col_beams_max(s) * s.ne >= 1024);
}

// Warps of a fold block: four columns; or the beams of one column, up to 16; or 16 to mark
// the rows of one column.
int fold_warps(const SensorDev& s) {
    if (!s.fold_block) return 4;
    return s.fold_beams ? (int)std::max<int64_t>(4, std::min<int64_t>(16, col_beams_max(s))) : 16;
}

// Rows per block of the row kernel: a whole band of 32, which reads the band's
// column tables once, while that leaves at least eight blocks an SM; else 16 or 8.  A
// launch of few rows, some of them wider than a warp's registers hold, takes a block
// a row: a frame of 1 x 8192 bins 94 -> 35 us, 9 x 9000 some 95 -> 35, 500 x 1100 30 -> 29, 500 x
// 20000 231 -> 82; 1000 x 1100 would take 35 instead of 31.
int rows_per_block(int64_t total_rows, int max_naz, int sm_count) {
    if (max_naz > 1024 && total_rows < 4ll * sm_count) return 1;
    for (int r : {32, 16})
        if (total_rows / r >= 8ll * sm_count) return r;
    return 8;
}

// Azimuth bins of a sensor whose column tables the row kernel keeps in shared memory, or 0.
int staged_naz(const SensorDev& s) { return s.naz <= kRowsStaged ? s.naz : 0; }

// Warps per row of the whole-image normalisation: none (a warp per pair of rows) where
// every row is up to 1024 bins on 16-byte boundaries, else one for every 512 bins of the
// widest row, as far as a launch of 2^24 warps goes.
int norm_runs(int max_naz, int64_t total_rows, bool vec) {
    if (vec && max_naz <= 1024) return 0;
    const int64_t runs = ((int64_t)max_naz + 511) / 512;
    return (int)std::max<int64_t>(1, std::min<int64_t>(runs, (1ll << 24) / total_rows));
}

SensorDev make_sensor(const sonar_sensor& s, uint64_t seed, uint64_t frame, const Tune& t, int fan_w,
                      int fan_h) {
    SensorDev d{};
    memcpy(d.pos, s.pos, sizeof d.pos);
    memcpy(d.rot, s.rot, sizeof d.rot);
    d.nb = s.n_beams;
    d.ne = s.n_elev;
    d.nr = s.n_range_bins;
    d.naz = s.n_az_bins;
    d.hfov = s.hfov;
    d.vfov = s.vfov;
    d.rmin = s.r_min;
    d.rmax = s.r_max;
    d.inv_dr = (float)((double)s.n_range_bins / ((double)s.r_max - (double)s.r_min));
    d.fan_w = fan_w;
    d.fan_h = fan_h;
    if (fan_w > 0 && fan_h > 0) {
        const double sx = fan_w / (2.0 * (double)s.r_max * std::sin((double)s.hfov / 2.0));
        const double sy = fan_h / (double)s.r_max;
        d.fan_scale = (float)std::min(sx, sy);
    }
    d.seed_lo = (uint32_t)seed;
    d.seed_hi = (uint32_t)(seed >> 32);
    d.frame_lo = (uint32_t)frame;
    d.frame_hi = (uint32_t)(frame >> 32);
    const int tb = (t.tb >= 1 && t.tb <= 32 && (t.tb & (t.tb - 1)) == 0) ? t.tb : 8;   // beams per warp tile
    d.tb = tb;
    d.occ = t.occ;
    const int64_t be = 32 / tb;   // ray-cast blocks: one warp on tb beams x be elevations
    d.trace_blocks = (int32_t)(((s.n_beams + tb - 1) / tb) * ((s.n_elev + be - 1) / be));
    // The per-beam fold when columns hold several beams (n_beams > n_az_bins)
    // and a column's dense rows, one per beam, would fit 200 KB of shared memory.
    // The choice depends on the sensor shape alone, so a bin's order of summation
    // never depends on how the frame is launched.
    const int64_t beams = col_beams_max(d), dense = (int64_t)d.nr * (1 + beams) + (d.nr + 31) / 32 +
                                                    std::min<int64_t>(beams * d.ne, d.nr);
    d.fold_beams = (s.n_beams > s.n_az_bins && dense * (int64_t)sizeof(float) <= 200 * 1024) ? 1 : 0;
    d.fold_block = d.fold_beams;
    return d;
}

}  // namespace

// ===========================================================================
// context
// ===========================================================================

extern "C" const char* sonar_version(void) {
    return "libsonar 1.0 (sm_103a; 4-wide LBVH + certified FP32 Moller-Trumbore with float-float exact decisions; Philox4x32-10)";
}

extern "C" sonar_status sonar_create(int32_t device, sonar_ctx_t* out) {
    if (!out) return SONAR_ERR_ARG;
    *out = nullptr;
    int n = 0;
    if (cudaGetDeviceCount(&n) != cudaSuccess || device < 0 || device >= n) return SONAR_ERR_ARG;
    if (cudaSetDevice(device) != cudaSuccess) return SONAR_ERR_CUDA;
    sonar_ctx* ctx = new sonar_ctx();
    ctx->device = device;
    cudaDeviceGetAttribute(&ctx->sm_count, cudaDevAttrMultiProcessorCount, device);
    if (cudaMalloc(&ctx->d_err, sizeof(uint32_t)) != cudaSuccess ||
        cudaMemset(ctx->d_err, 0, sizeof(uint32_t)) != cudaSuccess) {
        delete ctx;
        return SONAR_ERR_OOM;
    }
    // scenes come from a pool of the context's own, which keeps up to 1 GiB of
    // freed memory mapped (the scratch of a two-million-triangle build and its
    // scene) for the next build, and gives the rest back at the next
    // synchronisation and everything when the context goes
    cudaMemPoolProps props{};
    props.allocType = cudaMemAllocationTypePinned;
    props.handleTypes = cudaMemHandleTypeNone;
    props.location.type = cudaMemLocationTypeDevice;
    props.location.id = device;
    uint64_t keep = 1ull << 30;
    if (cudaMemPoolCreate(&ctx->pool, &props) != cudaSuccess ||
        cudaMemPoolSetAttribute(ctx->pool, cudaMemPoolAttrReleaseThreshold, &keep) != cudaSuccess) {
        cudaGetLastError();
        if (ctx->pool) cudaMemPoolDestroy(ctx->pool);
        cudaFree(ctx->d_err);
        delete ctx;
        return SONAR_ERR_CUDA;
    }
    set_kernel_attributes();
    cudaGetLastError();
    *out = ctx;
    return SONAR_OK;
}

extern "C" sonar_status sonar_destroy(sonar_ctx_t ctx) {
    if (!ctx) return SONAR_OK;
    cudaSetDevice(ctx->device);
    cudaDeviceSynchronize();
    for (auto& s : ctx->scenes) free_scene(&s);
    for (Scratch* s : {&ctx->rowmax, &ctx->noised, &ctx->rowinfo, &ctx->partials, &ctx->counters, &ctx->hits,
                       &ctx->trig, &ctx->vals, &ctx->bands})
        if (s->p) cudaFreeAsync(s->p, 0);
    cudaDeviceSynchronize();
    cudaMemPoolDestroy(ctx->pool);
    cudaFree(ctx->d_err);
    delete ctx;
    return SONAR_OK;
}

extern "C" const char* sonar_last_error(sonar_ctx_t ctx) {
    return ctx ? ctx->last_error.c_str() : "";
}

extern "C" sonar_status sonar_check(sonar_ctx_t ctx, uint32_t* bits) {
    if (!ctx) return SONAR_ERR_ARG;
    CU(cudaSetDevice(ctx->device), "cudaSetDevice");
    CU(cudaDeviceSynchronize(), "device synchronisation");
    uint32_t w = 0;
    CU(cudaMemcpy(&w, ctx->d_err, sizeof w, cudaMemcpyDeviceToHost), "reading the error word");
    if (bits) *bits = w;
    if (w) {
        CU(cudaMemset(ctx->d_err, 0, sizeof(uint32_t)), "clearing the error word");
        return fail(ctx, SONAR_ERR_DEVICE, "device error word 0x" + std::to_string(w));
    }
    return SONAR_OK;
}

// ===========================================================================
// scenes
// ===========================================================================

extern "C" sonar_status sonar_scene_upload(sonar_ctx_t ctx, const float* d_verts, int64_t n_verts,
                                           const int32_t* d_tris, const int32_t* d_mat, int64_t n_tris,
                                           void* stream, int32_t* scene_id) {
    if (!ctx || !scene_id) return fail(ctx, SONAR_ERR_ARG, "NULL context or scene_id");
    if (n_tris < 0 || n_verts < 0) return fail(ctx, SONAR_ERR_ARG, "negative counts");
    if (n_tris >= (1ll << 28) - 2) return fail(ctx, SONAR_ERR_ARG, "n_tris must be < 2^28 - 2");
    if (n_verts >= (1ll << 31)) return fail(ctx, SONAR_ERR_ARG, "n_verts must be < 2^31");
    if (n_tris > 0 && (!d_verts || !d_tris || !d_mat || n_verts == 0))
        return fail(ctx, SONAR_ERR_ARG, "NULL scene arrays");
    CU(cudaSetDevice(ctx->device), "cudaSetDevice");
    SceneStore s;
    std::string msg;
    const sonar_status st = build_scene(d_verts, n_verts, d_tris, d_mat, n_tris, ctx->sm_count, ctx->pool,
                                        (cudaStream_t)stream, &s, &msg);
    if (st != SONAR_OK) {
        cudaStreamSynchronize((cudaStream_t)stream);   // what was allocated on it is freed on another
        free_scene(&s);
        return fail(ctx, st, msg);
    }
    ctx->scenes.push_back(s);
    ctx->alive.push_back(true);
    *scene_id = (int32_t)ctx->scenes.size() - 1;
    return SONAR_OK;
}

extern "C" sonar_status sonar_scene_release(sonar_ctx_t ctx, int32_t id) {
    if (!ctx) return SONAR_ERR_ARG;
    sonar_status st = check_scene(ctx, id);
    if (st) return st;
    CU(cudaSetDevice(ctx->device), "cudaSetDevice");
    CU(cudaDeviceSynchronize(), "device synchronisation");
    free_scene(&ctx->scenes[id]);
    ctx->alive[id] = false;
    return SONAR_OK;
}

extern "C" sonar_status sonar_scene_info(sonar_ctx_t ctx, int32_t id, int64_t out[5]) {
    if (!ctx || !out) return fail(ctx, SONAR_ERR_ARG, "NULL argument");
    sonar_status st = check_scene(ctx, id);
    if (st) return st;
    const SceneStore& s = ctx->scenes[id];
    out[0] = s.n_tris;
    out[1] = s.n_pairs;
    out[2] = s.height;
    out[3] = s.max_mat;
    out[4] = (int64_t)s.bytes;
    return SONAR_OK;
}

// ===========================================================================
// single-frame rendering
// ===========================================================================

namespace {


// The context's exact-ray table buffer, grown to `entries`; a new buffer holds
// no tables yet.
cudaError_t grow_trig(sonar_ctx* ctx, size_t entries, cudaStream_t s) {
    const void* before = ctx->trig.p;
    const cudaError_t e = grow(ctx->trig, sizeof(float4) * entries, s);
    if (e != cudaSuccess || ctx->trig.p != before || ctx->trig.bytes < sizeof(float4) * entries) ctx->trig_at = nullptr;
    return e;
}

// The exact-ray tables of one sensor's call.  They depend on the angular
// geometry only, so a call with the same geometry and table buffer as the last
// build skips the launch (calls on a context are stream-ordered); while the
// stream is being captured into a graph the launch is always recorded, so that
// a replay rebuilds the tables it reads.
cudaError_t single_trig(sonar_ctx* ctx, const SensorDev& S, bool capturing, cudaStream_t s) {
    if (!capturing && ctx->trig_at == S.trig && ctx->trig_nb == S.nb && ctx->trig_ne == S.ne &&
        ctx->trig_hfov == S.hfov && ctx->trig_vfov == S.vfov)
        return cudaSuccess;
    const cudaError_t e = launch_trig(nullptr, S, 1, S.nb + S.ne, s);
    const bool keep = e == cudaSuccess && !capturing;
    ctx->trig_at = keep ? S.trig : nullptr;
    ctx->trig_nb = S.nb;
    ctx->trig_ne = S.ne;
    ctx->trig_hfov = S.hfov;
    ctx->trig_vfov = S.vfov;
    return e;
}

// Whether the stream is being captured into a graph.  A single-sensor call's later
// kernels are launched early (programmatic dependent launch) only when it is not, so
// that their setup overlaps the kernel before: 32.5 -> 28.8 us a frame of 1,024
// rays, 51.6 -> 42.0 us one of 32,768.
cudaError_t is_capturing(cudaStream_t s, bool* capturing) {
    cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
    const cudaError_t e = cudaStreamIsCapturing(s, &cap);
    *capturing = cap != cudaStreamCaptureStatusNone;
    return e;
}

// Where a single-sensor call keeps its fold's result: the compact lists, or (no
// room for them) P of the bins with returns in the polar image itself.
struct FoldStore {
    float2* vals = nullptr;
    uint2* bands = nullptr;
    float* dense = nullptr;
};

// Trace, fold, noise and row normalisation of one sensor (all offsets 0).
sonar_status single_forward(sonar_ctx* ctx, const SensorDev& S, const SceneDev& sc, const sonar_params* p,
                            const float* d_theta, int32_t n_mat, sonar_hit* hits, const FoldStore& f, float* noised,
                            float* binned, float* polar, uint32_t* gmax, bool capturing, cudaStream_t s) {
    if (p->normalise == 2) CU(cudaMemsetAsync(gmax, 0, sizeof(uint32_t), s), "cudaMemsetAsync");
    CU(single_trig(ctx, S, capturing, s), "trig launch");
    TraceArgs t{};
    t.one = S;
    t.one_scene = sc;
    t.params = *p;
    t.hits = hits;
    t.from_last = S.rot[8] > 0.0f;
    t.err = ctx->d_err;
    CU(launch_trace(t, S.trace_blocks, S.occ, s), "trace launch");
    if (f.dense) CU(cudaMemsetAsync(f.dense, 0, sizeof(float) * (size_t)S.nr * S.naz, s), "cudaMemsetAsync");
    FoldArgs a{};
    a.n_mat = n_mat;
    a.words_per_warp = (int32_t)fold_words(S);
    a.one = S;
    a.one_scene = sc;
    a.theta = d_theta;
    a.sigma_sm = p->sigma_sm;
    a.hits = hits;
    a.vals = f.vals;
    a.bands = f.bands;
    a.dense = f.dense;
    a.err = ctx->d_err;
    int warps = fold_warps(S);
    if (!S.fold_block)
        while (warps > 1 && sizeof(uint32_t) * warps * fold_words(S) > kMaxDynSmem) warps /= 2;
    const size_t smem = sizeof(uint32_t) * fold_words(S) * (S.fold_block ? 1 : warps);
    CU(launch_fold(a, S.fold_block ? S.naz : (S.naz + warps - 1) / warps, 32 * warps, smem, s,
                   !capturing && !f.dense),
       "fold launch");
    RowsArgs r{};
    r.rows_per_block = rows_per_block(S.nr, S.naz, ctx->sm_count);
    r.one = S;
    r.params = *p;
    r.vals = f.vals;
    r.bands = f.bands;
    r.dense = f.dense;
    r.noised = noised;
    r.binned = binned;
    r.polar = polar;
    r.gmax = gmax;
    const bool vec = S.naz % 4 == 0 && aligned16(noised) && aligned16(polar) && aligned16(binned);
    CU(launch_rows(r, (S.nr + r.rows_per_block - 1) / r.rows_per_block, S.naz, staged_naz(S), vec, s, !capturing),
       "row launch");
    return SONAR_OK;
}

// Whole-image normalisation (mode 2) and fan of one sensor (all offsets 0).
sonar_status single_post(sonar_ctx* ctx, const SensorDev& S, int normalise, const float* noised,
                         const uint32_t* gmax, float* polar, float* fan, bool capturing, cudaStream_t s) {
    if (normalise == 2) {
        NormArgs n{};
        n.one = S;
        n.total_rows = S.nr;
        n.noised = noised;
        n.gmax = gmax;
        n.runs = norm_runs(S.naz, S.nr, S.naz % 4 == 0 && aligned16(noised) && aligned16(polar));
        n.polar = polar;
        CU(launch_norm(n, s, !capturing), "normalisation launch");
    }
    if (fan) {
        FanArgs f{};
        f.one = S;
        f.polar = polar;
        f.fan = fan;
        CU(launch_fan_tiles(f, tile_squares(S.fan_w, S.fan_h), s, !capturing), "fan launch");
    }
    return SONAR_OK;
}

// Rays per adjoint work unit: about four units per SM over the whole render,
// a multiple of the block size.
int adj_chunk(int64_t rays, int sm_count, int block) {
    // about 16 units per SM: the per-ray gather is latency-bound and wants
    // many resident blocks
    int64_t c = rays / (16 * (int64_t)sm_count);
    c = (c + block - 1) / block * block;
    return (int)std::max<int64_t>(block, std::min<int64_t>(c, 64ll * block));
}

}  // namespace

extern "C" sonar_status sonar_render(sonar_ctx_t ctx, int32_t scene_id, const sonar_sensor* sensor,
                                     const sonar_params* params, const float* d_theta, int32_t n_mat,
                                     uint64_t seed, uint64_t frame, const sonar_outputs* out,
                                     void* stream) {
    if (!ctx) return SONAR_ERR_ARG;
    sonar_status st;
    if ((st = check_scene(ctx, scene_id)) || (st = check_sensor(ctx, sensor)) || (st = check_params(ctx, params)) ||
        (st = check_nmat(ctx, scene_id, n_mat)))
        return st;
    if (!d_theta) return fail(ctx, SONAR_ERR_ARG, "d_theta is NULL");
    if (!out || !out->polar) return fail(ctx, SONAR_ERR_ARG, "outputs or outputs->polar is NULL");
    if (out->hits && !aligned16(out->hits)) return fail(ctx, SONAR_ERR_ARG, "hits must be 16-byte aligned");
    if (out->fan && (out->fan_w < 1 || out->fan_h < 1)) return fail(ctx, SONAR_ERR_ARG, "fan size must be >= 1");
    cudaStream_t s = (cudaStream_t)stream;
    CU(cudaSetDevice(ctx->device), "cudaSetDevice");
    const Tune t = single_tune(ctx, *sensor);
    SensorDev S = make_sensor(*sensor, seed, frame, t, out->fan ? out->fan_w : 0, out->fan ? out->fan_h : 0);
    S.fold_block = fold_by_block(S, S.naz);
    const int64_t npol = (int64_t)S.nr * S.naz;
    float* noised = out->noised;
    if (!noised) {
        CU(grow(ctx->noised, sizeof(float) * npol, s), "scratch allocation");
        noised = (float*)ctx->noised.p;
    }
    CU(grow(ctx->rowmax, sizeof(uint32_t), s), "scratch allocation");
    sonar_hit* hits = out->hits;
    if (!hits) {
        CU(grow(ctx->hits, sizeof(sonar_hit) * (size_t)S.nb * S.ne, s), "scratch allocation");
        hits = (sonar_hit*)ctx->hits.p;
    }
    CU(grow_trig(ctx, (size_t)(S.nb + S.ne), s), "scratch allocation");
    S.trig = (float4*)ctx->trig.p;
    CU(grow(ctx->vals, sizeof(float2) * (size_t)S.nb * S.ne, s), "scratch allocation");
    CU(grow(ctx->bands, sizeof(uint2) * (size_t)band_count(S) * S.naz, s), "scratch allocation");
    const FoldStore fold{(float2*)ctx->vals.p, (uint2*)ctx->bands.p, nullptr};
    bool capturing = false;
    CU(is_capturing(s, &capturing), "capture status");
    sonar_status st2 = single_forward(ctx, S, scene_dev(ctx->scenes[scene_id]), params, d_theta, n_mat, hits, fold,
                                      noised, out->binned, out->polar, (uint32_t*)ctx->rowmax.p, capturing, s);
    if (st2 != SONAR_OK) return st2;
    return single_post(ctx, S, params->normalise, noised, (const uint32_t*)ctx->rowmax.p, out->polar, out->fan, capturing,
                       s);
}

extern "C" sonar_status sonar_fan_resample(sonar_ctx_t ctx, const sonar_sensor* sensor, const float* d_polar,
                                           int32_t fan_w, int32_t fan_h, float* d_fan, void* stream) {
    if (!ctx) return SONAR_ERR_ARG;
    sonar_status st = check_sensor(ctx, sensor);
    if (st) return st;
    if (!d_polar || !d_fan) return fail(ctx, SONAR_ERR_ARG, "NULL polar or fan");
    if (fan_w < 1 || fan_h < 1) return fail(ctx, SONAR_ERR_ARG, "fan size must be >= 1");
    CU(cudaSetDevice(ctx->device), "cudaSetDevice");
    const SensorDev S = make_sensor(*sensor, 0, 0, Tune{}, fan_w, fan_h);
    FanArgs f{};
    f.one = S;
    f.polar = d_polar;
    f.fan = d_fan;
    CU(launch_fan_tiles(f, tile_squares(S.fan_w, S.fan_h), (cudaStream_t)stream), "fan launch");
    return SONAR_OK;
}

extern "C" sonar_status sonar_render_backward(sonar_ctx_t ctx, int32_t scene_id, const sonar_sensor* sensor,
                                              const sonar_params* params, const float* d_theta, int32_t n_mat,
                                              uint64_t seed, uint64_t frame, const float* d_grad_polar,
                                              const float* d_noised, const sonar_hit* d_hits, float* d_dtheta,
                                              void* stream) {
    if (!ctx) return SONAR_ERR_ARG;
    sonar_status st;
    if ((st = check_scene(ctx, scene_id)) || (st = check_sensor(ctx, sensor)) || (st = check_params(ctx, params)) ||
        (st = check_nmat(ctx, scene_id, n_mat)))
        return st;
    if (!d_theta || !d_grad_polar || !d_noised || !d_dtheta)
        return fail(ctx, SONAR_ERR_ARG, "NULL theta, grad, noised or dtheta");
    if (d_hits && !aligned16(d_hits)) return fail(ctx, SONAR_ERR_ARG, "hits must be 16-byte aligned");
    cudaStream_t s = (cudaStream_t)stream;
    CU(cudaSetDevice(ctx->device), "cudaSetDevice");
    const Tune t = tune_for(ctx, *sensor);
    SensorDev S = make_sensor(*sensor, seed, frame, t, 0, 0);
    const int groups = params->normalise == 1 ? S.nr : 1;
    CU(grow(ctx->rowinfo, sizeof(RowInfo) * groups, s), "scratch allocation");
    bool capturing = false;
    CU(is_capturing(s, &capturing), "capture status");
    const sonar_hit* hits = d_hits;
    if (!hits) {   // recompute the hit records with the ray-cast kernel (bitwise the forward's)
        CU(grow_trig(ctx, (size_t)(S.nb + S.ne), s), "scratch allocation");
        CU(grow(ctx->hits, sizeof(sonar_hit) * (size_t)S.nb * S.ne, s), "scratch allocation");
        S.trig = (float4*)ctx->trig.p;
        S.occ = single_variant(ctx, *sensor, S.tb, S.occ);
        CU(single_trig(ctx, S, capturing, s), "trig launch");
        TraceArgs tr{};
        tr.one = S;
        tr.one_scene = scene_dev(ctx->scenes[scene_id]);
        tr.params = *params;
        tr.hits = (sonar_hit*)ctx->hits.p;
        tr.from_last = S.rot[8] > 0.0f;
        tr.err = ctx->d_err;
        CU(launch_trace(tr, S.trace_blocks, S.occ, s), "trace launch");
        hits = (const sonar_hit*)ctx->hits.p;
    }
    const int nq = n_mat + 2;
    const int64_t rays = (int64_t)S.nb * S.ne;
    const int chunk = adj_chunk(rays, ctx->sm_count, t.block);
    const int n_units = (int)((rays + chunk - 1) / chunk);
    CU(grow(ctx->partials, sizeof(double) * (size_t)n_units * nq, s), "scratch allocation");
    if (params->normalise != 0)
        CU(launch_adj_rows(nullptr, nullptr, S, groups, params->normalise,
                           aligned16(d_noised) && aligned16(d_grad_polar), d_noised, d_grad_polar,
                           (RowInfo*)ctx->rowinfo.p, nullptr, s),
           "adjoint row launch");
    AdjArgs a{};
    a.n_units = n_units;
    a.chunk = chunk;
    a.n_mat = n_mat;
    a.one = S;
    a.one_scene = scene_dev(ctx->scenes[scene_id]);
    a.theta = d_theta;
    a.params = *params;
    a.grad = d_grad_polar;
    a.hits = hits;
    a.rowinfo = (const RowInfo*)ctx->rowinfo.p;
    a.partials = (double*)ctx->partials.p;
    a.err = ctx->d_err;
    const size_t smem = sizeof(double) * (t.block / 32) * n_mat;
    CU(launch_adjoint(a, n_units, t.block, smem, d_dtheta, s, !capturing && params->normalise != 0, !capturing),
       "adjoint launch");
    return SONAR_OK;
}

// ===========================================================================
// batches
// ===========================================================================

struct sonar_batch {
    sonar_ctx* ctx = nullptr;
    std::vector<sonar_batch_item> items;
    std::vector<SensorDev> hs;        // host copy of the descriptors
    std::vector<int4> fold_map;       // per fold block: (sensor, first column, scene, 0)
    std::vector<int2> rows_map;       // per row-kernel block: (sensor, first row)
    std::vector<AdjUnit> adj_units;   // adjoint work list (ray chunks)
    std::vector<int32_t> fan_prefix;  // fan blocks per sensor, prefix
    std::vector<int32_t> trace_prefix;  // trace blocks per sensor, prefix
    int64_t total_rays = 0;
    int64_t total_rows = 0, total_polar = 0;
    int block = 128;
    int plan_occ = 0;                 // the ray-cast variant of the plan
    int trace_occ = 0;                // the one launched: the plan's, as far as the items' scenes allow
    int adj_chunk = 0;
    size_t fold_smem = 0;
    int fold_block = 128, fold_words_per_warp = 0;
    int rows_step = 32, max_naz = 1;
    int max_staged_naz = 0;           // the widest sensor whose column tables the row kernel stages (0: none)
    bool rows_vec = false;            // every row starts on a 16-byte boundary of a 16-byte aligned image
    SensorDev* d_sens = nullptr;
    int4* d_fold_map = nullptr;
    int2* d_rows_map = nullptr;
    float2* d_vals = nullptr;         // the fold's values, a slot per ray
    uint2* d_bands = nullptr;         // the fold's bitmaps
    AdjUnit* d_adj_units = nullptr;
    SceneDev* d_scenes = nullptr;
    int32_t* d_fan_prefix = nullptr;
    int32_t* d_trace_prefix = nullptr;
    int4* d_trace_map = nullptr;      // per trace block: (sensor, tile, scene, 0)
    std::vector<int4> h_trace_map;    // its host copy (an update that moves an item to another scene patches it)
    int2* d_fan_map = nullptr;        // per fan block: (sensor, block)
    int32_t* d_row_map = nullptr;     // per range row: sensor
    // fan coordinate tables: sensors with the same fan geometry share one,
    // filled from the owner's descriptor on every forward replay
    std::vector<int> lut_owner;       // per sensor: owner of its table (-1: none)
    std::vector<uint4*> lut_of;       // per sensor: the table of its owner (nullptr: none)
    uint4* d_fan_lut = nullptr;       // all tables
    uint4** d_luts = nullptr;         // per sensor: its own table when it is an owner
    int2* d_lut_map = nullptr;        // per table block: (owner, block)
    int4* d_group_map = nullptr;      // per grouped fan block: (owner, pixel block, users [m0, m1))
    int32_t* d_members = nullptr;     // users of each table, by owner
    uint32_t* d_fan_stamp = nullptr;  // per table block: the owner's fan_version it was built for
    int lut_blocks = 0, group_blocks = 0;
    int fan_blocks = 0;               // blocks of the per-sensor fan launch
    sonar_hit* d_hits = nullptr;      // hit records when the caller asks for none
    float4* d_trig = nullptr;         // per-sensor exact-ray tables
    uint32_t* d_trig_stamp = nullptr; // per sensor and k_trig block: the version its entries were built for
    int max_angles = 0;
    uint32_t* d_rowmax = nullptr;
    float* d_noised = nullptr;
    RowInfo* d_rowinfo = nullptr;
    double* d_partials = nullptr;
    int32_t* d_counter = nullptr;     // adjoint work
    int n_mat_cap = 0;
    size_t n_scene_table = 0;         // entries in d_scenes
    // host staging for updates (pinned, double-buffered)
    SensorDev* h_stage[2] = {nullptr, nullptr};
    SceneDev* h_stage_sc[2] = {nullptr, nullptr};
    cudaEvent_t stage_ev[2] = {nullptr, nullptr};
    int stage_next = 0;
    // graphs
    cudaStream_t cap = nullptr;
    cudaStream_t side = nullptr;      // the adjoint branch of the combined step graph
    cudaEvent_t fork_ev = nullptr, join_ev = nullptr;
    cudaStream_t mark[2] = {};        // the phase events of the forward and of the adjoint, beside the kernels
    cudaEvent_t mark_ev = nullptr;
    cudaGraphExec_t fwd = nullptr, bwd = nullptr, step = nullptr;
    // the forward without the two table kernels (exact-ray sin/cos, fan
    // coordinates), replayed while the tables are known to be current: no
    // update or plan since a forward that built them was enqueued (the fan
    // coordinates are built only by a forward that writes fans)
    cudaGraphExec_t fwd_lean = nullptr;
    bool trig_current = false, lut_current = false;
    bool lean_last = false;           // the last forward replay was the lean graph
    cudaEvent_t ev[7] = {};           // phase boundaries recorded inside the graphs
    bool ran_fwd = false, ran_bwd = false;
    std::vector<unsigned char> fwd_key, fwd_lean_key, bwd_key, step_key;
    int graphs = 0;
    int fwd_kernels = 0, fwd_lean_kernels = 0, bwd_kernels = 0, step_kernels = 0;   // kernel nodes of the current graphs
};

namespace {

// Drops every captured graph: the next call of each kind captures its launches anew.
void drop_graphs(sonar_batch* b) {
    for (cudaGraphExec_t* g : {&b->fwd, &b->fwd_lean, &b->bwd, &b->step}) {
        if (*g) cudaGraphExecDestroy(*g);
        *g = nullptr;
    }
    b->fwd_key.clear();
    b->fwd_lean_key.clear();
    b->bwd_key.clear();
    b->step_key.clear();
}

void batch_free_device(sonar_batch* b) {
    for (void* p : {(void*)b->d_sens, (void*)b->d_fold_map, (void*)b->d_rows_map, (void*)b->d_vals,
                    (void*)b->d_bands, (void*)b->d_adj_units, (void*)b->d_scenes,
                    (void*)b->d_fan_prefix, (void*)b->d_trace_prefix, (void*)b->d_trace_map,
                    (void*)b->d_fan_map, (void*)b->d_row_map, (void*)b->d_hits, (void*)b->d_trig, (void*)b->d_trig_stamp,
                    (void*)b->d_rowmax,
                    (void*)b->d_noised, (void*)b->d_rowinfo, (void*)b->d_partials, (void*)b->d_counter,
                    (void*)b->d_fan_lut, (void*)b->d_luts, (void*)b->d_lut_map, (void*)b->d_group_map,
                    (void*)b->d_members, (void*)b->d_fan_stamp})
        if (p) cudaFree(p);
    b->d_fan_lut = nullptr;
    b->d_luts = nullptr;
    b->d_lut_map = nullptr;
    b->d_group_map = nullptr;
    b->d_members = nullptr;
    b->d_fan_stamp = nullptr;
    b->lut_blocks = b->group_blocks = b->fan_blocks = 0;
    b->d_trace_prefix = nullptr;
    b->d_trace_map = nullptr;
    b->d_fan_map = nullptr;
    b->d_row_map = nullptr;
    b->d_hits = nullptr;
    b->d_trig = nullptr;
    b->d_trig_stamp = nullptr;
    b->n_mat_cap = 0;
    b->d_fold_map = nullptr; b->d_rows_map = nullptr; b->d_vals = nullptr; b->d_bands = nullptr;
    b->d_sens = nullptr; b->d_adj_units = nullptr; b->d_scenes = nullptr;
    b->d_fan_prefix = nullptr;
    b->d_rowmax = nullptr; b->d_noised = nullptr; b->d_rowinfo = nullptr; b->d_partials = nullptr;
    b->d_counter = nullptr;
    drop_graphs(b);
    b->trig_current = b->lut_current = false;
}

// Fan pixels sample the same bins with the same weights exactly when these agree.
bool same_fan_geometry(const SensorDev& x, const SensorDev& y) {
    auto eq = [](float a, float b) { return memcmp(&a, &b, sizeof a) == 0; };
    return x.nr == y.nr && x.naz == y.naz && x.fan_w == y.fan_w && x.fan_h == y.fan_h && eq(x.hfov, y.hfov) &&
           eq(x.rmin, y.rmin) && eq(x.rmax, y.rmax) && eq(x.inv_dr, y.inv_dr) && eq(x.fan_scale, y.fan_scale);
}

std::vector<SceneDev> scene_table(const sonar_ctx* ctx) {
    std::vector<SceneDev> t(ctx->scenes.size());
    for (size_t k = 0; k < t.size(); ++k) t[k] = scene_dev(ctx->scenes[k]);
    return t;
}

sonar_status check_items(sonar_ctx* ctx, const sonar_batch_item* items, int32_t n) {
    if (!items || n < 1) return fail(ctx, SONAR_ERR_ARG, "batch needs at least one item");
    for (int k = 0; k < n; ++k) {
        sonar_status st;
        if ((st = check_scene(ctx, items[k].scene_id)) || (st = check_sensor(ctx, &items[k].sensor))) {
            ctx->last_error = "item " + std::to_string(k) + ": " + ctx->last_error;
            return st;
        }
        if (items[k].fan_w < 0 || items[k].fan_h < 0 || (items[k].fan_w > 0) != (items[k].fan_h > 0))
            return fail(ctx, SONAR_ERR_ARG, "item " + std::to_string(k) + ": bad fan size");
        if (items[k].polar_offset < 0 || items[k].hits_offset < 0 || items[k].fan_offset < 0)
            return fail(ctx, SONAR_ERR_ARG, "item " + std::to_string(k) + ": negative offset");
    }
    return SONAR_OK;
}

// (Re)builds descriptors, work units and device buffers from b->items.
sonar_status batch_plan(sonar_batch* b) {
    sonar_ctx* ctx = b->ctx;
    batch_free_device(b);
    const int n = (int)b->items.size();
    b->hs.assign(n, SensorDev{});
    b->fold_map.clear();
    b->rows_map.clear();
    b->adj_units.clear();
    b->fan_prefix.assign(n + 1, 0);
    b->trace_prefix.assign(n + 1, 0);
    int64_t rows = 0, polar_end = 0, rays = 0, bands = 0;
    b->max_naz = 1;
    b->max_staged_naz = 0;
    b->rows_vec = true;
    std::map<int, int64_t> block_votes;
    for (int k = 0; k < n; ++k) {
        const sonar_batch_item& it = b->items[k];
        const Tune t = tune_for(ctx, it.sensor);
        SensorDev S = make_sensor(it.sensor, it.seed, it.frame, t, it.fan_w, it.fan_h);
        S.scene = it.scene_id;
        S.polar_off = it.polar_offset;
        S.hits_off = it.hits_offset;
        S.fan_off = it.fan_offset;
        S.rowmax_off = rows;
        S.val_off = rays;
        S.band_off = bands;
        rays += (int64_t)S.nb * S.ne;
        bands += band_count(S) * S.naz;
        b->max_naz = std::max(b->max_naz, S.naz);
        b->max_staged_naz = std::max(b->max_staged_naz, staged_naz(S));
        b->rows_vec = b->rows_vec && S.naz % 4 == 0 && S.polar_off % 4 == 0;
        rows += S.nr;    // room for mode 1; mode 2 uses the first slot of each sensor
        polar_end = std::max<int64_t>(polar_end, it.polar_offset + (int64_t)S.nr * S.naz);
        b->hs[k] = S;
        b->fan_prefix[k + 1] =
            b->fan_prefix[k] + (S.fan_w > 0 ? tile_squares(S.fan_w, S.fan_h) : 0);
        b->trace_prefix[k + 1] = b->trace_prefix[k] + S.trace_blocks;
        block_votes[t.block] += (int64_t)S.nb * S.ne;
    }
    b->block = 128;
    int64_t best = -1;
    for (auto& kv : block_votes)
        if (kv.second > best) { best = kv.second; b->block = kv.first; }
    // the trace launch takes the variant of the sensor shape with most rays; an
    // untuned shape, and a launch small enough for several lanes per ray, the one
    // the launch size calls for; the 8-wide tree only when
    // every scene of the batch has one
    int64_t most = -1;
    int kmost = 0;
    for (int k = 0; k < n; ++k) {
        const SensorDev& S = b->hs[k];
        if ((int64_t)S.nb * S.ne > most) { most = (int64_t)S.nb * S.ne; b->trace_occ = S.occ; kmost = k; }
    }
    if (n > 0) {
        const sonar_sensor& ms = b->items[kmost].sensor;
        if (!ctx->tune.count(ShapeKey{ms.n_beams, ms.n_elev, ms.n_range_bins, ms.n_az_bins}) ||
            group_lanes(ctx, b->trace_prefix[n]))
            b->trace_occ = default_variant(ctx, b->trace_prefix[n]);
        for (const sonar_batch_item& it : b->items)
            if (!ctx->scenes[it.scene_id].nodes8) b->trace_occ &= ~kTraceWide;
    }
    b->plan_occ = b->trace_occ;
    b->total_rows = rows;
    b->total_polar = polar_end;
    int64_t columns = 0;
    for (const SensorDev& S : b->hs) columns += S.naz;
    for (SensorDev& S : b->hs) S.fold_block = fold_by_block(S, columns);
    // the fold's blocks: the warps that the sensor with most rays wants, fewer
    // where the columns of some sensor need more shared memory than that
    int warps = n > 0 ? fold_warps(b->hs[kmost]) : 4;
    int64_t warp_words = 0, block_words = 0;
    for (const SensorDev& S : b->hs) (S.fold_block ? block_words : warp_words) =
        std::max(S.fold_block ? block_words : warp_words, fold_words(S));
    while (warps > 1 && (int64_t)sizeof(uint32_t) * warps * warp_words > (int64_t)kMaxDynSmem) warps /= 2;
    b->fold_block = 32 * warps;
    b->fold_words_per_warp = (int)warp_words;
    b->fold_smem = sizeof(uint32_t) * (size_t)std::max(block_words, warps * warp_words);
    b->rows_step = rows_per_block(rows, b->max_naz, ctx->sm_count);
    for (int k = 0; k < n; ++k) {
        const SensorDev& S = b->hs[k];
        const int step = S.fold_block ? 1 : warps;
        for (int c = 0; c < S.naz; c += step) b->fold_map.push_back(make_int4(k, c, S.scene, 0));
        for (int r = 0; r < S.nr; r += b->rows_step) b->rows_map.push_back(make_int2(k, r));
    }
    int64_t all_rays = 0;
    for (const SensorDev& S : b->hs) all_rays += (int64_t)S.nb * S.ne;
    b->total_rays = all_rays;
    b->adj_chunk = adj_chunk(all_rays, ctx->sm_count, b->block);
    for (int k = 0; k < n; ++k) {
        const int64_t r = (int64_t)b->hs[k].nb * b->hs[k].ne;
        for (int64_t r0 = 0; r0 < r; r0 += b->adj_chunk)
            b->adj_units.push_back(AdjUnit{k, (int32_t)r0, (int32_t)std::min<int64_t>(r, r0 + b->adj_chunk),
                                           b->hs[k].scene});
    }
    const size_t na = b->adj_units.size();
    cudaError_t e = cudaSuccess;
    auto alloc = [&](void** p, size_t bytes) {
        if (e == cudaSuccess) e = cudaMalloc(p, std::max(bytes, (size_t)16));
    };
    alloc((void**)&b->d_sens, sizeof(SensorDev) * n);
    alloc((void**)&b->d_fold_map, sizeof(int4) * b->fold_map.size());
    alloc((void**)&b->d_rows_map, sizeof(int2) * b->rows_map.size());
    alloc((void**)&b->d_vals, sizeof(float2) * rays);
    alloc((void**)&b->d_bands, sizeof(uint2) * bands);
    alloc((void**)&b->d_scenes, sizeof(SceneDev) * std::max<size_t>(1, ctx->scenes.size()));
    b->n_scene_table = ctx->scenes.size();
    alloc((void**)&b->d_adj_units, sizeof(AdjUnit) * na);
    alloc((void**)&b->d_fan_prefix, sizeof(int32_t) * (n + 1));
    alloc((void**)&b->d_trace_prefix, sizeof(int32_t) * (n + 1));
    // fan coordinate tables for geometries that more than one sensor shares
    b->lut_owner.assign(n, -1);
    b->lut_of.assign(n, nullptr);
    std::vector<int> owners;
    std::vector<int> members(n, 0);
    for (int k = 0; k < n; ++k) {
        if (b->hs[k].fan_w <= 0) continue;
        for (int o : owners)
            if (same_fan_geometry(b->hs[k], b->hs[o])) { b->lut_owner[k] = o; ++members[o]; break; }
        if (b->lut_owner[k] < 0) { owners.push_back(k); b->lut_owner[k] = k; members[k] = 1; }
    }
    int64_t lut_px = 0;
    std::vector<int64_t> lut_at(n, -1), stamp_at(n, -1);
    std::vector<int2> lmap;
    for (int o : owners) {
        if (members[o] < 2) continue;
        const int64_t px = (int64_t)b->hs[o].fan_w * b->hs[o].fan_h;
        lut_at[o] = lut_px;
        lut_px += px;
        stamp_at[o] = (int64_t)lmap.size();
        for (int64_t t = 0; t < (px + kFanTile - 1) / kFanTile; ++t) lmap.push_back(make_int2(o, (int)t));
    }
    for (int k = 0; k < n; ++k)
        if (b->lut_owner[k] >= 0 && lut_at[b->lut_owner[k]] < 0) b->lut_owner[k] = -1;
    b->lut_blocks = (int)lmap.size();
    // the fan of a table's users: blocks of (owner, pixel block, run of up to
    // kFanGroup users), so that a table entry serves several frames
    std::vector<int4> gmap;
    std::vector<int32_t> mem;
    for (int o : owners) {
        if (lut_at[o] < 0) continue;
        const int32_t m0 = (int32_t)mem.size();
        for (int k = 0; k < n; ++k)
            if (b->lut_owner[k] == o) mem.push_back(k);
        const int32_t m1 = (int32_t)mem.size();
        for (int32_t a0 = m0; a0 < m1; a0 += kFanGroup)
            for (int t = 0; t < fan_squares(b->hs[o].fan_w, b->hs[o].fan_h); ++t)
                gmap.push_back(make_int4(o, t, a0, std::min(a0 + kFanGroup, m1)));
    }
    b->group_blocks = (int)gmap.size();
    if (lut_px > 0) {
        alloc((void**)&b->d_fan_lut, sizeof(uint4) * lut_px);
        alloc((void**)&b->d_luts, sizeof(uint4*) * n);
        alloc((void**)&b->d_lut_map, sizeof(int2) * lmap.size());
        alloc((void**)&b->d_group_map, sizeof(int4) * gmap.size());
        alloc((void**)&b->d_members, sizeof(int32_t) * mem.size());
        alloc((void**)&b->d_fan_stamp, sizeof(uint32_t) * lmap.size());
        if (e == cudaSuccess) e = cudaMemset(b->d_fan_stamp, 0, sizeof(uint32_t) * lmap.size());
        if (e == cudaSuccess) {
            std::vector<uint4*> own(n, nullptr);
            for (int k = 0; k < n; ++k) {
                const int o = b->lut_owner[k];
                if (o < 0) continue;
                b->lut_of[k] = b->d_fan_lut + lut_at[o];
                b->hs[k].fan_lut = b->lut_of[k];
                if (o == k) {
                    own[k] = b->lut_of[k];
                    b->hs[k].fan_stamp = b->d_fan_stamp + stamp_at[o];   // stamps 0: every block builds once
                    b->hs[k].fan_version = 1;
                }
            }
            e = cudaMemcpy(b->d_luts, own.data(), sizeof(uint4*) * n, cudaMemcpyHostToDevice);
            if (e == cudaSuccess)
                e = cudaMemcpy(b->d_lut_map, lmap.data(), sizeof(int2) * lmap.size(), cudaMemcpyHostToDevice);
            if (e == cudaSuccess)
                e = cudaMemcpy(b->d_group_map, gmap.data(), sizeof(int4) * gmap.size(), cudaMemcpyHostToDevice);
            if (e == cudaSuccess)
                e = cudaMemcpy(b->d_members, mem.data(), sizeof(int32_t) * mem.size(), cudaMemcpyHostToDevice);
        }
    }
    std::vector<int4> tmap;
    std::vector<int2> fmap;
    std::vector<int32_t> rmap;
    // Ray-cast blocks in eight bands of decreasing upward component (world z) of
    // their tile's central ray, sensor by sensor inside a band.  Over a seabed
    // the rays closest to the horizon run farthest, so the longest blocks start
    // first and the launch's tail is short (longest-processing-time-first); the
    // bands keep a sensor's neighbouring tiles together, which share nodes in L2.
    // Results do not depend on the order.
    {
        std::vector<std::pair<float, int64_t>> order;
        for (int k = 0; k < n; ++k) {
            const SensorDev& S = b->hs[k];
            const int tb = S.tb, te = 32 / S.tb, tiles_b = (S.nb + tb - 1) / tb;
            for (int t = 0; t < S.trace_blocks; ++t) {
                const int ty = t / tiles_b, tx = t - ty * tiles_b;
                const double i = std::min(tx * tb + 0.5 * tb, (double)S.nb);
                const double j = std::min(ty * te + 0.5 * te, (double)S.ne);
                const double phi = i * S.hfov / S.nb - 0.5 * S.hfov, th = j * S.vfov / S.ne - 0.5 * S.vfov;
                const double up = S.rot[6] * std::sin(phi) * std::cos(th) + S.rot[7] * std::cos(phi) * std::cos(th) +
                                  S.rot[8] * std::sin(th);
                order.push_back({(float)-up, ((int64_t)k << 32) | (uint32_t)t});
            }
        }
        if (!order.empty()) {
            constexpr int kBands = 8;
            float lo = order[0].first, hi = order[0].first;
            for (const auto& q : order) { lo = std::min(lo, q.first); hi = std::max(hi, q.first); }
            const float width = (hi - lo) / kBands;
            for (auto& q : order)
                q.first = width > 0.0f ? std::min((float)(kBands - 1), std::floor((q.first - lo) / width)) : 0.0f;
        }
        std::stable_sort(order.begin(), order.end(),
                         [](const std::pair<float, int64_t>& x, const std::pair<float, int64_t>& y) {
                             return x.first < y.first;
                         });
        for (const auto& q : order) {
            const int k = (int)(q.second >> 32);
            tmap.push_back(make_int4(k, (int)(q.second & 0xFFFFFFFF), b->hs[k].scene, 0));
        }
    }
    for (int k = 0; k < n; ++k) {
        if (b->lut_owner[k] < 0)   // sensors with a shared table are resampled by the grouped launch
            for (int t = 0; t < b->fan_prefix[k + 1] - b->fan_prefix[k]; ++t) fmap.push_back(make_int2(k, t));
        for (int r = 0; r < b->hs[k].nr; ++r) rmap.push_back(k);
    }
    alloc((void**)&b->d_trace_map, sizeof(int4) * tmap.size());
    alloc((void**)&b->d_fan_map, sizeof(int2) * std::max<size_t>(1, fmap.size()));
    b->fan_blocks = (int)fmap.size();
    alloc((void**)&b->d_row_map, sizeof(int32_t) * rmap.size());
    int64_t angles = 0;
    b->max_angles = 0;
    for (const SensorDev& S : b->hs) {
        angles += S.nb + S.ne;
        b->max_angles = std::max(b->max_angles, S.nb + S.ne);
    }
    alloc((void**)&b->d_trig, sizeof(float4) * angles);
    // per sensor, one stamp per k_trig block (grid x = ceil(max_angles / 128)):
    // stamps 0 and versions 1, so every block builds its entries once
    const int trig_gx = (b->max_angles + 127) / 128;
    alloc((void**)&b->d_trig_stamp, sizeof(uint32_t) * std::max<int64_t>(1, (int64_t)n * trig_gx));
    if (e == cudaSuccess) e = cudaMemset(b->d_trig_stamp, 0, sizeof(uint32_t) * std::max<int64_t>(1, (int64_t)n * trig_gx));
    if (e == cudaSuccess) {
        int64_t off = 0;
        for (int k = 0; k < n; ++k) {
            SensorDev& S = b->hs[k];
            S.trig = b->d_trig + off;
            off += S.nb + S.ne;
            S.trig_stamp = b->d_trig_stamp + (int64_t)k * trig_gx;
            S.trig_version = 1;
        }
    }
    alloc((void**)&b->d_rowmax, sizeof(uint32_t) * rows);
    alloc((void**)&b->d_rowinfo, sizeof(RowInfo) * rows);
    alloc((void**)&b->d_counter, sizeof(int32_t));
    if (e != cudaSuccess) return cuda_fail(ctx, e, "batch allocation");
    const std::vector<SceneDev> table = scene_table(ctx);
    e = cudaMemcpy(b->d_sens, b->hs.data(), sizeof(SensorDev) * n, cudaMemcpyHostToDevice);
    if (e == cudaSuccess)
        e = cudaMemcpy(b->d_fold_map, b->fold_map.data(), sizeof(int4) * b->fold_map.size(), cudaMemcpyHostToDevice);
    if (e == cudaSuccess)
        e = cudaMemcpy(b->d_rows_map, b->rows_map.data(), sizeof(int2) * b->rows_map.size(), cudaMemcpyHostToDevice);
    if (e == cudaSuccess && !table.empty())
        e = cudaMemcpy(b->d_scenes, table.data(), sizeof(SceneDev) * table.size(), cudaMemcpyHostToDevice);
    if (e == cudaSuccess)
        e = cudaMemcpy(b->d_adj_units, b->adj_units.data(), sizeof(AdjUnit) * na, cudaMemcpyHostToDevice);
    if (e == cudaSuccess)
        e = cudaMemcpy(b->d_fan_prefix, b->fan_prefix.data(), sizeof(int32_t) * (n + 1), cudaMemcpyHostToDevice);
    if (e == cudaSuccess)
        e = cudaMemcpy(b->d_trace_prefix, b->trace_prefix.data(), sizeof(int32_t) * (n + 1), cudaMemcpyHostToDevice);
    if (e == cudaSuccess)
        e = cudaMemcpy(b->d_trace_map, tmap.data(), sizeof(int4) * tmap.size(), cudaMemcpyHostToDevice);
    b->h_trace_map = std::move(tmap);
    if (e == cudaSuccess && !fmap.empty())
        e = cudaMemcpy(b->d_fan_map, fmap.data(), sizeof(int2) * fmap.size(), cudaMemcpyHostToDevice);
    if (e == cudaSuccess)
        e = cudaMemcpy(b->d_row_map, rmap.data(), sizeof(int32_t) * rmap.size(), cudaMemcpyHostToDevice);
    if (e != cudaSuccess) return cuda_fail(ctx, e, "batch upload");
    return SONAR_OK;
}

// Scratch for outputs the caller does not want (noised image, hit records),
// allocated before any capture: an allocation inside stream capture fails.
cudaError_t batch_scratch(sonar_batch* b, const sonar_batch_outputs* out) {
    cudaError_t e = cudaSuccess;
    if (!out->noised && !b->d_noised)
        e = cudaMalloc(&b->d_noised, sizeof(float) * std::max<int64_t>(1, b->total_polar));
    if (e == cudaSuccess && !out->hits && !b->d_hits)
        e = cudaMalloc(&b->d_hits, sizeof(sonar_hit) * std::max<int64_t>(1, b->total_rays));
    return e;
}

// Kernel nodes of a captured graph (-1 if the graph cannot be inspected).
int kernel_nodes(cudaGraph_t g) {
    size_t n = 0;
    if (cudaGraphGetNodes(g, nullptr, &n) != cudaSuccess) return -1;
    std::vector<cudaGraphNode_t> nodes(n);
    if (n > 0 && cudaGraphGetNodes(g, nodes.data(), &n) != cudaSuccess) return -1;
    int k = 0;
    for (cudaGraphNode_t v : nodes) {
        cudaGraphNodeType t;
        if (cudaGraphNodeGetType(v, &t) != cudaSuccess) return -1;
        k += t == cudaGraphNodeTypeKernel;
    }
    return k;
}

template <class T>
void append_bytes(std::vector<unsigned char>& v, const T& x) {
    const unsigned char* p = (const unsigned char*)&x;
    v.insert(v.end(), p, p + sizeof(T));
}

// The end of a capture whose launches failed with `st`, already reported.
sonar_status capture_failed(cudaGraph_t g, sonar_status st) {
    if (g) cudaGraphDestroy(g);
    cudaGetLastError();   // what ending the broken capture left
    return st;
}

// Records phase event `ev` after what stream `s` (being captured) holds so far, on
// a branch of its own: the next kernel then follows the last one directly, and
// may start early.
cudaError_t mark_phase(sonar_batch* b, cudaStream_t mark, cudaEvent_t ev, cudaStream_t s) {
    cudaError_t e = cudaEventRecord(b->mark_ev, s);
    if (e == cudaSuccess) e = cudaStreamWaitEvent(mark, b->mark_ev, 0);
    if (e == cudaSuccess) e = cudaEventRecordWithFlags(ev, mark, cudaEventRecordExternal);
    return e;
}

// Joins the branch of phase events back into the captured stream.
cudaError_t join_marks(sonar_batch* b, cudaStream_t mark, cudaStream_t s) {
    const cudaError_t e = cudaEventRecord(b->mark_ev, mark);
    return e == cudaSuccess ? cudaStreamWaitEvent(s, b->mark_ev, 0) : e;
}

// The forward's launches: part 1 up to I~ (trig tables, ray cast, fold, and the
// row kernel, which also normalises by rows), part 2 the whole-image
// normalisation and the fan, part 0 both.
sonar_status batch_forward_launches(sonar_batch* b, const sonar_params* p, const float* d_theta, int32_t n_mat,
                                    const sonar_batch_outputs* out, cudaStream_t s, bool events = false,
                                    int part = 0, bool tables = true) {
    sonar_ctx* ctx = b->ctx;
    if (part != 2) {
        if (p->normalise == 2)
            CU(cudaMemsetAsync(b->d_rowmax, 0, sizeof(uint32_t) * b->total_rows, s), "cudaMemsetAsync");
        sonar_hit* hits = out->hits ? out->hits : b->d_hits;   // scratch allocated by the caller, outside capture
        if (events) CU(mark_phase(b, b->mark[0], b->ev[0], s), "cudaEventRecord");
        if (tables)
            CU(launch_trig(b->d_sens, SensorDev{}, (int)b->items.size(), b->max_angles, s), "batch trig launch");
        TraceArgs t{};
        t.sensors = b->d_sens;
        t.scenes = b->d_scenes;
        t.block_map = b->d_trace_map;
        t.n_sensors = (int32_t)b->items.size();
        t.params = *p;
        t.hits = hits;
        t.err = ctx->d_err;
        CU(launch_trace(t, b->trace_prefix.back(), b->trace_occ, s, tables), "batch trace launch");
        if (events) CU(mark_phase(b, b->mark[0], b->ev[6], s), "cudaEventRecord");
        FoldArgs a{};
        a.sensors = b->d_sens;
        a.scenes = b->d_scenes;
        a.block_map = b->d_fold_map;
        a.n_mat = n_mat;
        a.words_per_warp = b->fold_words_per_warp;
        a.theta = d_theta;
        a.sigma_sm = p->sigma_sm;
        a.hits = hits;
        a.vals = b->d_vals;
        a.bands = b->d_bands;
        a.err = ctx->d_err;
        CU(launch_fold(a, (int)b->fold_map.size(), b->fold_block, b->fold_smem, s, true), "batch fold launch");
        RowsArgs r{};
        r.sensors = b->d_sens;
        r.block_map = b->d_rows_map;
        r.rows_per_block = b->rows_step;
        r.params = *p;
        r.vals = b->d_vals;
        r.bands = b->d_bands;
        r.noised = out->noised ? out->noised : b->d_noised;
        r.binned = out->binned;
        r.polar = out->polar;
        r.gmax = b->d_rowmax;
        const bool vec = b->rows_vec && aligned16(r.noised) && aligned16(r.binned) && aligned16(r.polar);
        CU(launch_rows(r, (int)b->rows_map.size(), b->max_naz, b->max_staged_naz, vec, s, true), "batch row launch");
        if (events) CU(mark_phase(b, b->mark[0], b->ev[1], s), "cudaEventRecord");
    }
    if (part == 1) return SONAR_OK;
    if (p->normalise == 2) {
        NormArgs c{};
        c.sensors = b->d_sens;
        c.row_map = b->d_row_map;
        c.n_sensors = (int32_t)b->items.size();
        c.total_rows = b->total_rows;
        c.noised = out->noised ? out->noised : b->d_noised;
        c.gmax = b->d_rowmax;
        c.runs = norm_runs(b->max_naz, b->total_rows, b->rows_vec && aligned16(c.noised) && aligned16(out->polar));
        c.polar = out->polar;
        CU(launch_norm(c, s, true), "batch normalisation launch");
    }
    if (out->fan) {
        FanArgs f{};
        f.sensors = b->d_sens;
        f.block_map = b->d_fan_map;
        f.n_sensors = (int32_t)b->items.size();
        f.polar = out->polar;
        f.fan = out->fan;
        if (b->lut_blocks > 0) {
            if (tables) {
                FanLutArgs l{b->d_sens, b->d_lut_map, b->d_luts};
                CU(launch_fan_lut(l, b->lut_blocks, s, true), "batch fan table launch");
            }
            FanGroupArgs g{b->d_sens, b->d_group_map, b->d_members, out->polar, out->fan};
            CU(launch_fan_group(g, b->group_blocks, s, true), "batch grouped fan launch");
        }
        CU(launch_fan_tiles(f, b->fan_blocks, s, true), "batch fan launch");
    }
    if (events) CU(mark_phase(b, b->mark[0], b->ev[2], s), "cudaEventRecord");
    return SONAR_OK;
}

}  // namespace

extern "C" sonar_status sonar_batch_create(sonar_ctx_t ctx, const sonar_batch_item* items, int32_t n,
                                           sonar_batch_t* out) {
    if (!ctx || !out) return fail(ctx, SONAR_ERR_ARG, "NULL argument");
    *out = nullptr;
    sonar_status st = check_items(ctx, items, n);
    if (st) return st;
    CU(cudaSetDevice(ctx->device), "cudaSetDevice");
    sonar_batch* b = new sonar_batch();
    b->ctx = ctx;
    b->items.assign(items, items + n);
    st = batch_plan(b);
    cudaError_t e = cudaSuccess;
    for (int k = 0; k < 2 && st == SONAR_OK; ++k) {
        if (e == cudaSuccess) e = cudaMallocHost((void**)&b->h_stage[k], sizeof(SensorDev) * n);
        if (e == cudaSuccess)
            e = cudaMallocHost((void**)&b->h_stage_sc[k], sizeof(SceneDev) * std::max<size_t>(1, 64));
        if (e == cudaSuccess) e = cudaEventCreateWithFlags(&b->stage_ev[k], cudaEventDisableTiming);
    }
    if (st == SONAR_OK && e == cudaSuccess) e = cudaStreamCreateWithFlags(&b->cap, cudaStreamNonBlocking);
    if (st == SONAR_OK && e == cudaSuccess) e = cudaStreamCreateWithFlags(&b->side, cudaStreamNonBlocking);
    for (int k = 0; k < 2 && st == SONAR_OK && e == cudaSuccess; ++k)
        e = cudaStreamCreateWithFlags(&b->mark[k], cudaStreamNonBlocking);
    if (st == SONAR_OK && e == cudaSuccess) e = cudaEventCreateWithFlags(&b->mark_ev, cudaEventDisableTiming);
    if (st == SONAR_OK && e == cudaSuccess) e = cudaEventCreateWithFlags(&b->fork_ev, cudaEventDisableTiming);
    if (st == SONAR_OK && e == cudaSuccess) e = cudaEventCreateWithFlags(&b->join_ev, cudaEventDisableTiming);
    for (int k = 0; k < 7 && st == SONAR_OK && e == cudaSuccess; ++k) e = cudaEventCreate(&b->ev[k]);
    if (st == SONAR_OK && e != cudaSuccess) st = cuda_fail(ctx, e, "batch staging");
    if (st != SONAR_OK) {
        sonar_batch_destroy(b);
        return st;
    }
    *out = b;
    return SONAR_OK;
}

extern "C" sonar_status sonar_batch_update(sonar_batch_t b, const sonar_batch_item* items, int32_t n, void* stream) {
    if (!b) return SONAR_ERR_ARG;
    b->trig_current = b->lut_current = false;   // the next forward replays the table kernels (they skip current entries)
    sonar_ctx* ctx = b->ctx;
    sonar_status st = check_items(ctx, items, n);
    if (st) return st;
    if (n != (int32_t)b->items.size()) return fail(ctx, SONAR_ERR_ARG, "item count differs from the plan");
    for (int k = 0; k < n; ++k) {
        const sonar_batch_item& x = items[k];
        const sonar_batch_item& y = b->items[k];
        if (x.sensor.n_beams != y.sensor.n_beams || x.sensor.n_elev != y.sensor.n_elev ||
            x.sensor.n_range_bins != y.sensor.n_range_bins || x.sensor.n_az_bins != y.sensor.n_az_bins ||
            x.fan_w != y.fan_w || x.fan_h != y.fan_h || x.polar_offset != y.polar_offset ||
            x.hits_offset != y.hits_offset || x.fan_offset != y.fan_offset)
            return fail(ctx, SONAR_ERR_ARG, "item " + std::to_string(k) + ": shape or offsets differ from the plan");
    }
    CU(cudaSetDevice(ctx->device), "cudaSetDevice");
    bool new_scene = false;
    for (int k = 0; k < n; ++k) new_scene |= (size_t)items[k].scene_id >= b->n_scene_table;
    if (new_scene) {
        // a scene uploaded after planning: rebuild the scene table (synchronous)
        CU(cudaStreamSynchronize((cudaStream_t)stream), "stream synchronisation");
        const std::vector<SceneDev> table = scene_table(ctx);
        SceneDev* d = nullptr;
        CU(cudaMalloc(&d, sizeof(SceneDev) * table.size()), "scene table");
        CU(cudaMemcpy(d, table.data(), sizeof(SceneDev) * table.size(), cudaMemcpyHostToDevice), "scene table");
        cudaFree(b->d_scenes);
        b->d_scenes = d;
        b->n_scene_table = table.size();
        drop_graphs(b);   // they hold the old table's address
    }
    // an item may go to a scene whose 8-wide tree was too deep to keep: the launches then
    // walk the 4-wide trees, until an update leads away from it again.  (A scene of
    // one leaf has no nodes to walk, and needs no tree.)
    int occ = b->plan_occ;
    for (int k = 0; k < n; ++k) {
        const SceneStore& sc = ctx->scenes[items[k].scene_id];
        if (sc.root >= 0 && !sc.nodes8) occ &= ~kTraceWide;
    }
    if (occ != b->trace_occ) {
        b->trace_occ = occ;
        drop_graphs(b);
    }
    const int slot = b->stage_next;
    b->stage_next ^= 1;
    CU(cudaEventSynchronize(b->stage_ev[slot]), "staging wait");
    bool scene_moved = false;
    for (int k = 0; k < n; ++k) {
        SensorDev S = b->hs[k];
        scene_moved |= S.scene != items[k].scene_id;
        const sonar_batch_item& it = items[k];
        const SensorDev fresh = make_sensor(it.sensor, it.seed, it.frame, Tune{1, S.tb, b->block, S.occ},
                                            it.fan_w, it.fan_h);
        memcpy(S.pos, fresh.pos, sizeof S.pos);
        memcpy(S.rot, fresh.rot, sizeof S.rot);
        S.hfov = fresh.hfov; S.vfov = fresh.vfov; S.rmin = fresh.rmin; S.rmax = fresh.rmax;
        S.inv_dr = fresh.inv_dr; S.fan_scale = fresh.fan_scale;
        S.seed_lo = fresh.seed_lo; S.seed_hi = fresh.seed_hi; S.frame_lo = fresh.frame_lo; S.frame_hi = fresh.frame_hi;
        S.scene = it.scene_id;
        // an owner's table is rebuilt (inside the graph) once its fan geometry changes
        if (S.fan_stamp && !same_fan_geometry(S, b->hs[k]) && ++S.fan_version == 0) S.fan_version = 1;   // 0: never built
        // and the exact-ray tables once a field of view changes
        if (S.trig_stamp && (S.hfov != b->hs[k].hfov || S.vfov != b->hs[k].vfov) && ++S.trig_version == 0)
            S.trig_version = 1;
        b->hs[k] = S;
        b->items[k] = it;
    }
    for (int k = 0; k < n; ++k) {
        // a sensor keeps its owner's coordinate table only while their fan geometry agrees
        const int o = b->lut_owner.empty() ? -1 : b->lut_owner[k];
        b->hs[k].fan_lut = (o >= 0 && same_fan_geometry(b->hs[k], b->hs[o])) ? b->lut_of[k] : nullptr;
        b->h_stage[slot][k] = b->hs[k];
    }
    cudaStream_t s = (cudaStream_t)stream;
    CU(cudaMemcpyAsync(b->d_sens, b->h_stage[slot], sizeof(SensorDev) * n, cudaMemcpyHostToDevice, s),
       "descriptor upload");
    if (scene_moved) {   // the ray-cast map and the work units carry their scene: patch them (rare, pageable copies)
        for (int4& m : b->h_trace_map) m.z = b->hs[m.x].scene;
        for (int4& m : b->fold_map) m.z = b->hs[m.x].scene;
        for (AdjUnit& x : b->adj_units) x.scene = b->hs[x.sensor].scene;
        CU(cudaMemcpyAsync(b->d_trace_map, b->h_trace_map.data(), sizeof(int4) * b->h_trace_map.size(),
                           cudaMemcpyHostToDevice, s),
           "trace map upload");
        CU(cudaMemcpyAsync(b->d_fold_map, b->fold_map.data(), sizeof(int4) * b->fold_map.size(),
                           cudaMemcpyHostToDevice, s),
           "fold map upload");
        CU(cudaMemcpyAsync(b->d_adj_units, b->adj_units.data(), sizeof(AdjUnit) * b->adj_units.size(),
                           cudaMemcpyHostToDevice, s),
           "unit upload");
    }
    CU(cudaEventRecord(b->stage_ev[slot], s), "cudaEventRecord");
    return SONAR_OK;
}

extern "C" sonar_status sonar_render_batch(sonar_batch_t b, const sonar_params* p, const float* d_theta,
                                           int32_t n_mat, const sonar_batch_outputs* out, void* stream) {
    if (!b) return SONAR_ERR_ARG;
    sonar_ctx* ctx = b->ctx;
    sonar_status st = check_params(ctx, p);
    if (st) return st;
    if (!d_theta || !out || !out->polar) return fail(ctx, SONAR_ERR_ARG, "NULL theta or outputs");
    if (out->hits && !aligned16(out->hits)) return fail(ctx, SONAR_ERR_ARG, "hits must be 16-byte aligned");
    for (const sonar_batch_item& it : b->items)
        if ((st = check_scene(ctx, it.scene_id)) || (st = check_nmat(ctx, it.scene_id, n_mat))) return st;
    CU(cudaSetDevice(ctx->device), "cudaSetDevice");
    cudaStream_t s = (cudaStream_t)stream;
    CU(batch_scratch(b, out), "batch scratch");
    std::vector<unsigned char> key;
    append_bytes(key, *p);
    append_bytes(key, d_theta);
    append_bytes(key, n_mat);
    append_bytes(key, *out);
    // the full forward while a table it reads may be stale, else the lean one
    const bool lean = b->trig_current && (b->lut_current || !out->fan || b->lut_blocks == 0);
    cudaGraphExec_t& exec = lean ? b->fwd_lean : b->fwd;
    std::vector<unsigned char>& exec_key = lean ? b->fwd_lean_key : b->fwd_key;
    if (!exec || key != exec_key) {
        if (exec) cudaGraphExecDestroy(exec);
        exec = nullptr;
        CU(cudaStreamBeginCapture(b->cap, cudaStreamCaptureModeThreadLocal), "graph capture");
        st = batch_forward_launches(b, p, d_theta, n_mat, out, b->cap, true, 0, !lean);
        const cudaError_t ej = join_marks(b, b->mark[0], b->cap);
        cudaGraph_t g = nullptr;
        cudaError_t e = cudaStreamEndCapture(b->cap, &g);
        if (e == cudaSuccess) e = ej;
        if (st != SONAR_OK) return capture_failed(g, st);
        CU(e, "graph capture");
        (lean ? b->fwd_lean_kernels : b->fwd_kernels) = kernel_nodes(g);
        const cudaError_t e2 = cudaGraphInstantiate(&exec, g, 0);
        cudaGraphDestroy(g);
        CU(e2, "graph instantiation");
        exec_key = key;
        ++b->graphs;
    }
    CU(cudaGraphLaunch(exec, s), "graph launch");
    b->trig_current = true;   // built by this replay, in stream order, if they were stale
    if (out->fan) b->lut_current = true;
    b->lean_last = lean;
    b->ran_fwd = true;
    return SONAR_OK;
}

namespace {

sonar_status batch_backward_launches(sonar_batch* b, const sonar_params* p, const float* d_theta, int32_t n_mat,
                                     const float* grad, const float* noised, const sonar_hit* hits, float* dtheta,
                                     cudaStream_t s, bool events = false) {
    sonar_ctx* ctx = b->ctx;
    bool cast = false;   // a kernel of this call precedes the row terms
    // the gather's work counter is cleared by a kernel before it (the ray cast
    // of recomputed records, the row terms), else by a memset
    if (hits && p->normalise == 0)
        CU(cudaMemsetAsync(b->d_counter, 0, sizeof(int32_t), s), "cudaMemsetAsync");
    if (events) CU(mark_phase(b, b->mark[1], b->ev[3], s), "cudaEventRecord");
    if (!hits) {   // recompute the hit records with the ray-cast kernel into the batch scratch
        CU(launch_trig(b->d_sens, SensorDev{}, (int)b->items.size(), b->max_angles, s), "batch trig launch");
        TraceArgs tr{};
        tr.sensors = b->d_sens;
        tr.scenes = b->d_scenes;
        tr.block_map = b->d_trace_map;
        tr.n_sensors = (int32_t)b->items.size();
        tr.params = *p;
        tr.hits = b->d_hits;
        tr.err = ctx->d_err;
        tr.zero_word = b->d_counter;
        CU(launch_trace(tr, b->trace_prefix.back(), b->trace_occ, s, true), "batch trace launch");
        hits = b->d_hits;
        cast = true;
    }
    if (p->normalise != 0)
        CU(launch_adj_rows(b->d_sens, b->d_row_map, SensorDev{},
                           p->normalise == 1 ? b->total_rows : (int64_t)b->items.size(), p->normalise,
                           aligned16(noised) && aligned16(grad), noised, grad, b->d_rowinfo, b->d_counter, s, cast),
           "batch adjoint rows");
    if (events) CU(mark_phase(b, b->mark[1], b->ev[4], s), "cudaEventRecord");
    AdjArgs a{};
    a.sensors = b->d_sens;
    a.units = b->d_adj_units;
    a.scenes = b->d_scenes;
    a.work_counter = b->d_counter;
    a.n_units = (int32_t)b->adj_units.size();
    a.chunk = b->adj_chunk;
    a.n_mat = n_mat;
    a.theta = d_theta;
    a.params = *p;
    a.grad = grad;
    a.hits = hits;
    a.rowinfo = b->d_rowinfo;
    a.partials = b->d_partials;
    a.err = ctx->d_err;
    const size_t smem = sizeof(double) * (b->block / 32) * n_mat;
    const int per_sm = adjoint_blocks_per_sm(b->block, smem);
    const int grid = (int)std::max<int64_t>(1, std::min<int64_t>((int64_t)b->adj_units.size(),
                                                                    (int64_t)ctx->sm_count * per_sm));
    CU(launch_adjoint(a, grid, b->block, smem, dtheta, s, cast || p->normalise != 0, true), "batch adjoint launch");
    if (events) CU(mark_phase(b, b->mark[1], b->ev[5], s), "cudaEventRecord");
    return SONAR_OK;
}

}  // namespace

extern "C" sonar_status sonar_render_batch_backward(sonar_batch_t b, const sonar_params* p, const float* d_theta,
                                                    int32_t n_mat, const float* d_grad, const float* d_noised,
                                                    const sonar_hit* d_hits, float* d_dtheta, void* stream) {
    if (!b) return SONAR_ERR_ARG;
    sonar_ctx* ctx = b->ctx;
    sonar_status st = check_params(ctx, p);
    if (st) return st;
    if (!d_theta || !d_grad || !d_noised || !d_dtheta) return fail(ctx, SONAR_ERR_ARG, "NULL argument");
    if (d_hits && !aligned16(d_hits)) return fail(ctx, SONAR_ERR_ARG, "hits must be 16-byte aligned");
    for (const sonar_batch_item& it : b->items)
        if ((st = check_scene(ctx, it.scene_id)) || (st = check_nmat(ctx, it.scene_id, n_mat))) return st;
    CU(cudaSetDevice(ctx->device), "cudaSetDevice");
    if (!d_hits && !b->d_hits)   // recomputed records need the scratch; allocate outside capture
        CU(cudaMalloc(&b->d_hits, sizeof(sonar_hit) * std::max<int64_t>(1, b->total_rays)), "batch scratch");
    if (n_mat > b->n_mat_cap) {
        if (b->d_partials) cudaFree(b->d_partials);
        b->d_partials = nullptr;
        CU(cudaMalloc(&b->d_partials, sizeof(double) * b->adj_units.size() * (n_mat + 2)), "batch scratch");
        b->n_mat_cap = n_mat;
        if (b->bwd) cudaGraphExecDestroy(b->bwd);
        b->bwd = nullptr;
    }
    std::vector<unsigned char> key;
    append_bytes(key, *p);
    append_bytes(key, d_theta);
    append_bytes(key, n_mat);
    append_bytes(key, d_grad);
    append_bytes(key, d_noised);
    append_bytes(key, d_hits);
    append_bytes(key, d_dtheta);
    if (!b->bwd || key != b->bwd_key) {
        if (b->bwd) cudaGraphExecDestroy(b->bwd);
        b->bwd = nullptr;
        CU(cudaStreamBeginCapture(b->cap, cudaStreamCaptureModeThreadLocal), "graph capture");
        st = batch_backward_launches(b, p, d_theta, n_mat, d_grad, d_noised, d_hits, d_dtheta, b->cap, true);
        const cudaError_t ej = join_marks(b, b->mark[1], b->cap);
        cudaGraph_t g = nullptr;
        cudaError_t e = cudaStreamEndCapture(b->cap, &g);
        if (e == cudaSuccess) e = ej;
        if (st != SONAR_OK) return capture_failed(g, st);
        CU(e, "graph capture");
        b->bwd_kernels = kernel_nodes(g);
        const cudaError_t e2 = cudaGraphInstantiate(&b->bwd, g, 0);
        cudaGraphDestroy(g);
        CU(e2, "graph instantiation");
        b->bwd_key = key;
        ++b->graphs;
    }
    CU(cudaGraphLaunch(b->bwd, (cudaStream_t)stream), "graph launch");
    b->ran_bwd = true;
    return SONAR_OK;
}

extern "C" sonar_status sonar_render_batch_step(sonar_batch_t b, const sonar_params* p, const float* d_theta,
                                                int32_t n_mat, const sonar_batch_outputs* out, const float* d_grad,
                                                float* d_dtheta, void* stream) {
    if (!b) return SONAR_ERR_ARG;
    sonar_ctx* ctx = b->ctx;
    sonar_status st = check_params(ctx, p);
    if (st) return st;
    if (!d_theta || !out || !out->polar || !d_grad || !d_dtheta)
        return fail(ctx, SONAR_ERR_ARG, "NULL theta, outputs, grad or dtheta");
    if (out->hits && !aligned16(out->hits)) return fail(ctx, SONAR_ERR_ARG, "hits must be 16-byte aligned");
    for (const sonar_batch_item& it : b->items)
        if ((st = check_scene(ctx, it.scene_id)) || (st = check_nmat(ctx, it.scene_id, n_mat))) return st;
    CU(cudaSetDevice(ctx->device), "cudaSetDevice");
    CU(batch_scratch(b, out), "batch scratch");
    if (!out->hits && !b->d_hits)   // the adjoint reads the records the forward writes
        CU(cudaMalloc(&b->d_hits, sizeof(sonar_hit) * std::max<int64_t>(1, b->total_rays)), "batch scratch");
    if (n_mat > b->n_mat_cap) {
        if (b->d_partials) cudaFree(b->d_partials);
        b->d_partials = nullptr;
        CU(cudaMalloc(&b->d_partials, sizeof(double) * b->adj_units.size() * (n_mat + 2)), "batch scratch");
        b->n_mat_cap = n_mat;
        if (b->bwd) cudaGraphExecDestroy(b->bwd);
        if (b->step) cudaGraphExecDestroy(b->step);
        b->bwd = b->step = nullptr;
    }
    std::vector<unsigned char> key;
    append_bytes(key, *p);
    append_bytes(key, d_theta);
    append_bytes(key, n_mat);
    append_bytes(key, *out);
    append_bytes(key, d_grad);
    append_bytes(key, d_dtheta);
    if (!b->step || key != b->step_key) {
        if (b->step) cudaGraphExecDestroy(b->step);
        b->step = nullptr;
        const float* noised = out->noised ? out->noised : b->d_noised;
        const sonar_hit* hits = out->hits ? out->hits : b->d_hits;
        // one graph, two branches after the row kernel: the adjoint (which reads I~
        // and the hit records only) beside the fan (and whole-image normalisation)
        CU(cudaStreamBeginCapture(b->cap, cudaStreamCaptureModeThreadLocal), "graph capture");
        st = batch_forward_launches(b, p, d_theta, n_mat, out, b->cap, true, 1);
        cudaError_t e = cudaSuccess;
        bool forked = false;
        if (st == SONAR_OK) {
            e = cudaEventRecord(b->fork_ev, b->cap);
            if (e == cudaSuccess) e = cudaStreamWaitEvent(b->side, b->fork_ev, 0);
            forked = e == cudaSuccess;
        }
        if (st == SONAR_OK && forked)
            st = batch_backward_launches(b, p, d_theta, n_mat, d_grad, noised, hits, d_dtheta, b->side, true);
        if (st == SONAR_OK && forked) st = batch_forward_launches(b, p, d_theta, n_mat, out, b->cap, true, 2);
        if (forked) {   // join the branch whatever happened, so that the capture can end
            const cudaError_t e1 = cudaEventRecord(b->join_ev, b->side);
            const cudaError_t e2 = e1 == cudaSuccess ? cudaStreamWaitEvent(b->cap, b->join_ev, 0) : e1;
            if (e == cudaSuccess) e = e2;
            const cudaError_t e4 = join_marks(b, b->mark[1], b->cap);
            if (e == cudaSuccess) e = e4;
        }
        const cudaError_t e5 = join_marks(b, b->mark[0], b->cap);
        if (e == cudaSuccess) e = e5;
        cudaGraph_t g = nullptr;
        const cudaError_t e3 = cudaStreamEndCapture(b->cap, &g);
        if (st != SONAR_OK) return capture_failed(g, st);
        if (e != cudaSuccess) return capture_failed(g, cuda_fail(ctx, e, "graph fork"));
        CU(e3, "graph capture");
        b->step_kernels = kernel_nodes(g);
        const cudaError_t e6 = cudaGraphInstantiate(&b->step, g, 0);
        cudaGraphDestroy(g);
        CU(e6, "graph instantiation");
        b->step_key = key;
        ++b->graphs;
    }
    CU(cudaGraphLaunch(b->step, (cudaStream_t)stream), "graph launch");
    b->ran_fwd = b->ran_bwd = true;
    return SONAR_OK;
}

extern "C" sonar_status sonar_batch_info(sonar_batch_t b, int64_t out[5]) {
    if (!b || !out) return SONAR_ERR_ARG;
    int64_t rays = 0;
    for (const SensorDev& S : b->hs) rays += (int64_t)S.nb * S.ne;
    out[0] = (int64_t)b->fold_map.size();
    out[1] = rays;
    out[2] = (int64_t)b->fold_map.size();
    out[3] = b->fold_block;
    out[4] = b->graphs;
    return SONAR_OK;
}

extern "C" sonar_status sonar_batch_kernels(sonar_batch_t b, int32_t out[2]) {
    if (!b || !out) return SONAR_ERR_ARG;
    out[0] = b->lean_last ? (b->fwd_lean ? b->fwd_lean_kernels : 0) : (b->fwd ? b->fwd_kernels : 0);
    out[1] = b->bwd ? b->bwd_kernels : 0;
    return SONAR_OK;
}

extern "C" sonar_status sonar_batch_timings(sonar_batch_t b, float ms[5]) {
    if (!b || !ms) return SONAR_ERR_ARG;
    sonar_ctx* ctx = b->ctx;
    for (int k = 0; k < 5; ++k) ms[k] = -1.0f;
    CU(cudaSetDevice(ctx->device), "cudaSetDevice");
    if (b->ran_fwd) {
        CU(cudaEventSynchronize(b->ev[2]), "cudaEventSynchronize");
        CU(cudaEventElapsedTime(&ms[0], b->ev[0], b->ev[6]), "cudaEventElapsedTime");
        CU(cudaEventElapsedTime(&ms[1], b->ev[6], b->ev[1]), "cudaEventElapsedTime");
        CU(cudaEventElapsedTime(&ms[2], b->ev[1], b->ev[2]), "cudaEventElapsedTime");
    }
    if (b->ran_bwd) {
        CU(cudaEventSynchronize(b->ev[5]), "cudaEventSynchronize");
        CU(cudaEventElapsedTime(&ms[3], b->ev[3], b->ev[4]), "cudaEventElapsedTime");
        CU(cudaEventElapsedTime(&ms[4], b->ev[4], b->ev[5]), "cudaEventElapsedTime");
    }
    return SONAR_OK;
}

extern "C" sonar_status sonar_batch_destroy(sonar_batch_t b) {
    if (!b) return SONAR_OK;
    cudaSetDevice(b->ctx->device);
    cudaDeviceSynchronize();
    batch_free_device(b);
    for (cudaEvent_t& e : b->ev)
        if (e) cudaEventDestroy(e);
    for (int k = 0; k < 2; ++k) {
        if (b->h_stage[k]) cudaFreeHost(b->h_stage[k]);
        if (b->h_stage_sc[k]) cudaFreeHost(b->h_stage_sc[k]);
        if (b->stage_ev[k]) cudaEventDestroy(b->stage_ev[k]);
    }
    if (b->cap) cudaStreamDestroy(b->cap);
    if (b->side) cudaStreamDestroy(b->side);
    for (cudaStream_t& m : b->mark)
        if (m) cudaStreamDestroy(m);
    if (b->mark_ev) cudaEventDestroy(b->mark_ev);
    if (b->fork_ev) cudaEventDestroy(b->fork_ev);
    if (b->join_ev) cudaEventDestroy(b->join_ev);
    delete b;
    return SONAR_OK;
}

// ===========================================================================
// autotuner
// ===========================================================================

namespace {

// Times the batch's forward launches, and its adjoint launches when `grad` is
// given (no graph): the best over `rounds` of the mean of `reps` back-to-back
// passes, after one warm-up pass; 1e30 when a launch sequence fails.
float time_batch(sonar_batch* b, const sonar_params* p, const float* d_theta, int32_t n_mat,
                 const sonar_batch_outputs* out, const float* grad, float* dtheta, cudaStream_t s, int reps,
                 int rounds) {
    cudaEvent_t e0, e1;
    cudaEventCreate(&e0);
    cudaEventCreate(&e1);
    bool ok = true;
    auto pass = [&] {
        ok = ok && batch_forward_launches(b, p, d_theta, n_mat, out, s) == SONAR_OK;
        if (grad)
            ok = ok && batch_backward_launches(b, p, d_theta, n_mat, grad, out->noised, out->hits, dtheta, s) ==
                           SONAR_OK;
    };
    pass();
    float best = 1e30f;
    for (int k = 0; k < rounds && ok; ++k) {
        cudaEventRecord(e0, s);
        for (int r = 0; r < reps; ++r) pass();
        cudaEventRecord(e1, s);
        cudaEventSynchronize(e1);
        float ms = 0.0f;
        cudaEventElapsedTime(&ms, e0, e1);
        best = std::min(best, ms / reps);
    }
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
    return ok ? best : 1e30f;   // a candidate whose launches failed is never chosen
}

}  // namespace

extern "C" sonar_status sonar_autotune(sonar_batch_t b, const sonar_params* p, const float* d_theta, int32_t n_mat,
                                       const sonar_batch_outputs* out, void* stream) {
    if (!b) return SONAR_ERR_ARG;
    sonar_ctx* ctx = b->ctx;
    sonar_status st = check_params(ctx, p);
    if (st) return st;
    if (!d_theta || !out || !out->polar) return fail(ctx, SONAR_ERR_ARG, "NULL theta or outputs");
    for (const sonar_batch_item& it : b->items)
        if ((st = check_scene(ctx, it.scene_id)) || (st = check_nmat(ctx, it.scene_id, n_mat))) return st;
    CU(cudaSetDevice(ctx->device), "cudaSetDevice");
    cudaStream_t s = (cudaStream_t)stream;
    CU(batch_scratch(b, out), "batch scratch");
    std::vector<ShapeKey> shapes;
    for (const sonar_batch_item& it : b->items) {
        const ShapeKey k{it.sensor.n_beams, it.sensor.n_elev, it.sensor.n_range_bins, it.sensor.n_az_bins};
        if (std::find(shapes.begin(), shapes.end(), k) == shapes.end()) shapes.push_back(k);
    }
    const std::vector<sonar_batch_item> all = b->items;
    // an upstream gradient for timing the adjoint: every element the float
    // with bytes 0x3A (about 7e-4)
    float* adj_grad = nullptr;
    float* adj_dtheta = nullptr;
    if (out->hits && out->noised) {
        if (cudaMalloc(&adj_grad, sizeof(float) * std::max<int64_t>(1, b->total_polar)) != cudaSuccess ||
            cudaMalloc(&adj_dtheta, sizeof(float) * (n_mat + 2)) != cudaSuccess ||
            cudaMemsetAsync(adj_grad, 0x3A, sizeof(float) * std::max<int64_t>(1, b->total_polar), s) != cudaSuccess) {
            if (adj_grad) cudaFree(adj_grad);
            if (adj_dtheta) cudaFree(adj_dtheta);
            return fail(ctx, SONAR_ERR_OOM, "autotune scratch");
        }
    }
    // per shape, timed on that shape's items alone
    for (const ShapeKey& k : shapes) {
        std::vector<sonar_batch_item> sub;
        for (const sonar_batch_item& it : all)
            if (ShapeKey{it.sensor.n_beams, it.sensor.n_elev, it.sensor.n_range_bins, it.sensor.n_az_bins} == k)
                sub.push_back(it);
        b->items = sub;
        Tune best;
        best.block = 128;
        float best_ms = 1e30f;
        // the trace warp tile (beams x elevations per warp) and register budget,
        // with default binning shapes
        for (int occ : {0, kTraceCap, kTraceWide, kTraceCap | kTraceWide}) {
            for (int tb : {1, 2, 4, 8, 16, 32}) {
                ctx->tune[k] = Tune{1, tb, 128, occ};
                if ((st = batch_plan(b)) != SONAR_OK) goto restore;
                // a launch small enough for several lanes per ray does not go by the row's
                // variant: four equal launches would leave it to noise.  The row, which
                // later and larger batches of the shape go by, keeps the variant that
                // those default to
                if (occ != kTraceCap && group_lanes(ctx, b->trace_prefix.back())) continue;
                if (batch_scratch(b, out) != cudaSuccess) { st = fail(ctx, SONAR_ERR_OOM, "batch scratch"); goto restore; }
                const float ms = time_batch(b, p, d_theta, n_mat, out, nullptr, nullptr, s, 3, 3);
                if (cudaGetLastError() != cudaSuccess) continue;
                if (ms < best_ms) { best_ms = ms; best.tb = tb; best.occ = occ; }
            }
        }
        // then the adjoint's block size (which also sets its ray chunks), when the
        // caller's outputs hold the hit records and I~ that its timing needs: the
        // forward and the adjoint of a constant upstream gradient
        best_ms = 1e30f;
        const int tb = best.tb, occ = best.occ;
        for (int block : {64, 128, 256}) {
            if (!adj_grad) break;
            ctx->tune[k] = Tune{1, tb, block, occ};
            if ((st = batch_plan(b)) != SONAR_OK) goto restore;
            if (batch_scratch(b, out) != cudaSuccess) { st = fail(ctx, SONAR_ERR_OOM, "batch scratch"); goto restore; }
            if (cudaMalloc(&b->d_partials, sizeof(double) * b->adj_units.size() * (n_mat + 2)) != cudaSuccess) {
                st = fail(ctx, SONAR_ERR_OOM, "batch scratch");
                goto restore;
            }
            b->n_mat_cap = n_mat;
            const float ms = time_batch(b, p, d_theta, n_mat, out, adj_grad, adj_dtheta, s, 3, 3);
            if (cudaGetLastError() != cudaSuccess) continue;
            if (ms < best_ms) { best_ms = ms; best = Tune{1, tb, block, occ}; }
        }
        ctx->tune[k] = best;
    }
restore:
    b->items = all;
    if (adj_grad) cudaFree(adj_grad);
    if (adj_dtheta) cudaFree(adj_dtheta);
    {
        const sonar_status st2 = batch_plan(b);
        if (st == SONAR_OK) st = st2;
    }
    CU(cudaStreamSynchronize(s), "autotune synchronisation");
    return st;
}

extern "C" sonar_status sonar_tune_get(sonar_ctx_t ctx, int32_t* rows, int32_t cap, int32_t* count) {
    if (!ctx || !count) return SONAR_ERR_ARG;
    int k = 0;
    for (auto& kv : ctx->tune) {
        if (rows && k < cap) {
            int32_t* r = rows + 8 * k;
            r[0] = kv.first[0]; r[1] = kv.first[1]; r[2] = kv.first[2]; r[3] = kv.first[3];
            r[4] = kv.second.cols; r[5] = kv.second.tb; r[6] = kv.second.block; r[7] = kv.second.occ;
        }
        ++k;
    }
    *count = k;
    return SONAR_OK;
}

extern "C" sonar_status sonar_tune_set(sonar_ctx_t ctx, const int32_t* rows, int32_t count) {
    if (!ctx || (!rows && count > 0) || count < 0) return fail(ctx, SONAR_ERR_ARG, "bad tune rows");
    for (int k = 0; k < count; ++k) {
        const int32_t* r = rows + 8 * k;
        if (r[0] < 1 || r[1] < 1 || r[2] < 1 || r[3] < 1 || r[4] < 1 || r[5] < 1 || r[5] > 32 ||
            (r[5] & (r[5] - 1)) || r[6] < 32 || r[6] > 512 || (r[6] & 31) || (r[7] & ~(kTraceCap | kTraceWide)))
            return fail(ctx, SONAR_ERR_ARG, "bad tune row " + std::to_string(k));
        ctx->tune[ShapeKey{r[0], r[1], r[2], r[3]}] = Tune{r[4], r[5], r[6], r[7]};
    }
    return SONAR_OK;
}

// ===========================================================================
// counters
// ===========================================================================

extern "C" sonar_status sonar_uw_image(sonar_ctx_t ctx, const float* d_J, const float* d_depth, int64_t n_pixels,
                                       const float coef[9], float* d_I, void* stream) {
    if (!ctx) return SONAR_ERR_ARG;
    if (n_pixels < 0) return fail(ctx, SONAR_ERR_ARG, "n_pixels < 0");
    if (!coef) return fail(ctx, SONAR_ERR_ARG, "coef is NULL");
    for (int c = 0; c < 9; ++c) {
        if (!std::isfinite(coef[c])) return fail(ctx, SONAR_ERR_ARG, "coefficients must be finite");
        if (c < 6 && coef[c] < 0.0f) return fail(ctx, SONAR_ERR_ARG, "attenuation and backscatter must be >= 0");
    }
    if (n_pixels == 0) return SONAR_OK;
    if (!d_J || !d_depth || !d_I) return fail(ctx, SONAR_ERR_ARG, "NULL image buffer");
    CU(cudaSetDevice(ctx->device), "cudaSetDevice");
    UwCoef k;
    for (int c = 0; c < 3; ++c) {
        k.b_attn[c] = coef[c];
        k.b_bs[c] = coef[3 + c];
        k.b_inf[c] = coef[6 + c];
    }
    CU(launch_uw_image(d_J, d_depth, n_pixels, k, d_I, ctx->sm_count, (cudaStream_t)stream), "image launch");
    return SONAR_OK;
}

extern "C" sonar_status sonar_dvl(sonar_ctx_t ctx, int32_t scene_id, const float* d_poses, const float* d_vel,
                                  int64_t n, const sonar_dvl_params* p, uint64_t seed, float* d_ranges,
                                  float* d_vel_out, int32_t* d_flags, float* d_period, void* stream) {
    if (!ctx) return SONAR_ERR_ARG;
    if (!p) return fail(ctx, SONAR_ERR_ARG, "params is NULL");
    if (n < 0) return fail(ctx, SONAR_ERR_ARG, "n < 0");
    sonar_status st;
    if ((st = check_scene(ctx, scene_id))) return st;
    const float vals[] = {p->tilt, p->r_min, p->r_max, p->sigma_b, p->t0, p->t1, p->t_lost};
    for (float v : vals)
        if (!std::isfinite(v)) return fail(ctx, SONAR_ERR_ARG, "DVL parameters must be finite");
    if (!(p->tilt > 0.0f && p->tilt < 1.5707963f)) return fail(ctx, SONAR_ERR_ARG, "tilt must lie in (0, pi/2)");
    if (!(p->r_min >= 0.0f && p->r_max > p->r_min)) return fail(ctx, SONAR_ERR_ARG, "need 0 <= r_min < r_max");
    if (p->min_beams != 3 && p->min_beams != 4) return fail(ctx, SONAR_ERR_ARG, "min_beams must be 3 or 4");
    if (p->sigma_b < 0.0f || p->t0 < 0.0f || p->t1 < 0.0f || !(p->t_lost > 0.0f))
        return fail(ctx, SONAR_ERR_ARG, "need sigma_b, t0, t1 >= 0 and t_lost > 0");
    if (n == 0) return SONAR_OK;
    if (!d_poses || !d_vel || !d_ranges || !d_vel_out || !d_flags || !d_period)
        return fail(ctx, SONAR_ERR_ARG, "NULL buffer");
    CU(cudaSetDevice(ctx->device), "cudaSetDevice");
    DvlArgs a{};
    a.scene = scene_dev(ctx->scenes[scene_id]);
    a.pose = d_poses;
    a.vel_world = d_vel;
    a.n = n;
    for (int k = 0; k < 4; ++k) {
        const double az = M_PI / 4.0 + k * (M_PI / 2.0);
        a.beam[k][0] = (float)(std::sin((double)p->tilt) * std::cos(az));
        a.beam[k][1] = (float)(std::sin((double)p->tilt) * std::sin(az));
        a.beam[k][2] = (float)(-std::cos((double)p->tilt));
    }
    a.r_min = p->r_min;
    a.r_max = p->r_max;
    a.sigma_b = p->sigma_b;
    a.t0 = p->t0;
    a.t1 = p->t1;
    a.t_lost = p->t_lost;
    a.min_beams = p->min_beams;
    a.seed_lo = (uint32_t)seed;
    a.seed_hi = (uint32_t)(seed >> 32);
    a.ranges = d_ranges;
    a.vel = d_vel_out;
    a.flags = d_flags;
    a.period = d_period;
    a.err = ctx->d_err;
    CU(launch_dvl(a, (cudaStream_t)stream), "DVL launch");
    return SONAR_OK;
}

extern "C" sonar_status sonar_dvl_schedule(sonar_ctx_t ctx, const float* d_period, int64_t n_veh, int64_t n_steps,
                                           float dt, int32_t* d_emit, void* stream) {
    if (!ctx) return SONAR_ERR_ARG;
    if (n_veh < 0 || n_steps < 0) return fail(ctx, SONAR_ERR_ARG, "negative count");
    if (!(dt > 0.0f) || !std::isfinite(dt)) return fail(ctx, SONAR_ERR_ARG, "dt must be finite and > 0");
    if (n_veh == 0 || n_steps == 0) return SONAR_OK;
    if (!d_period || !d_emit) return fail(ctx, SONAR_ERR_ARG, "NULL buffer");
    CU(cudaSetDevice(ctx->device), "cudaSetDevice");
    CU(launch_dvl_schedule(d_period, n_veh, n_steps, dt, d_emit, (cudaStream_t)stream), "DVL schedule launch");
    return SONAR_OK;
}

extern "C" sonar_status sonar_trace_stats(sonar_ctx_t ctx, int32_t scene_id, const sonar_sensor* sensor,
                                          const sonar_params* params, void* stream, int64_t out[6]) {
    if (!ctx || !out) return fail(ctx, SONAR_ERR_ARG, "NULL argument");
    sonar_status st;
    if ((st = check_scene(ctx, scene_id)) || (st = check_sensor(ctx, sensor)) || (st = check_params(ctx, params)))
        return st;
    CU(cudaSetDevice(ctx->device), "cudaSetDevice");
    cudaStream_t s = (cudaStream_t)stream;
    const SceneStore& sc = ctx->scenes[scene_id];
    const int64_t node_words = sc.n_pairs / 32 + 1, tri_words = sc.n_tris / 32 + 1;
    unsigned long long* cnt = nullptr;
    uint32_t *nb = nullptr, *tb = nullptr;
    CU(cudaMalloc(&cnt, sizeof(unsigned long long) * 8), "stats allocation");
    cudaError_t e = cudaMalloc(&nb, sizeof(uint32_t) * node_words);
    if (e == cudaSuccess) e = cudaMalloc(&tb, sizeof(uint32_t) * tri_words);
    if (e == cudaSuccess) e = cudaMemsetAsync(cnt, 0, sizeof(unsigned long long) * 8, s);
    if (e == cudaSuccess) e = cudaMemsetAsync(nb, 0, sizeof(uint32_t) * node_words, s);
    if (e == cudaSuccess) e = cudaMemsetAsync(tb, 0, sizeof(uint32_t) * tri_words, s);
    TraceCounters tc{cnt, cnt + 1, cnt + 2, nb, tb};
    // the tuned warp tiles of this sensor shape: a lane's visits depend a little
    // on its warp's rays (leaves are parked until the whole warp holds one)
    const Tune t = tune_for(ctx, *sensor);
    SensorDev S = make_sensor(*sensor, 0, 0, t, 0, 0);
    float4* trig = nullptr;
    if (e == cudaSuccess) e = cudaMalloc(&trig, sizeof(float4) * (S.nb + S.ne));
    S.trig = trig;
    if (e == cudaSuccess) e = launch_trig(nullptr, S, 1, S.nb + S.ne, s);
    if (e == cudaSuccess) e = launch_stats(S, scene_dev(sc), *params, tc, ctx->d_err, s);
    if (e == cudaSuccess) e = launch_popcount(nb, node_words, cnt + 3, s);
    if (e == cudaSuccess) e = launch_popcount(tb, tri_words, cnt + 4, s);
    unsigned long long h[8] = {};
    if (e == cudaSuccess) e = cudaMemcpyAsync(h, cnt, sizeof h, cudaMemcpyDeviceToHost, s);
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);
    cudaFree(cnt);
    cudaFree(nb);
    cudaFree(tb);
    cudaFree(trig);
    if (e != cudaSuccess) return cuda_fail(ctx, e, "trace statistics");
    out[0] = (int64_t)h[0];
    out[1] = (int64_t)h[1];
    out[2] = (int64_t)h[3];
    out[3] = (int64_t)h[4];
    out[4] = (int64_t)S.nb * S.ne;
    out[5] = (int64_t)h[2];
    return SONAR_OK;
}

extern "C" sonar_status sonar_philox(sonar_ctx_t ctx, const uint32_t* d_counters, int64_t n, uint64_t seed,
                                     uint32_t* d_out, void* stream) {
    if (!ctx) return SONAR_ERR_ARG;
    if (n < 0) return fail(ctx, SONAR_ERR_ARG, "n < 0");
    if (n == 0) return SONAR_OK;
    if (!d_counters || !d_out) return fail(ctx, SONAR_ERR_ARG, "NULL buffer");
    if (!aligned16(d_counters) || !aligned16(d_out)) return fail(ctx, SONAR_ERR_ARG, "buffers must be 16-byte aligned");
    CU(cudaSetDevice(ctx->device), "cudaSetDevice");
    CU(launch_philox(d_counters, n, (uint32_t)seed, (uint32_t)(seed >> 32), d_out, (cudaStream_t)stream),
       "philox launch");
    return SONAR_OK;
}

extern "C" sonar_status sonar_probe_l2_read(sonar_ctx_t ctx, const void* d_buf, int64_t bytes, int32_t passes,
                                            float* d_block_sums, int32_t n_blocks, void* stream) {
    if (!ctx) return SONAR_ERR_ARG;
    if (!d_buf || !d_block_sums) return fail(ctx, SONAR_ERR_ARG, "NULL buffer");
    if (bytes <= 0 || bytes % 16 != 0) return fail(ctx, SONAR_ERR_ARG, "bytes must be a positive multiple of 16");
    if (reinterpret_cast<uintptr_t>(d_buf) % 16 != 0) return fail(ctx, SONAR_ERR_ARG, "buffer not 16-byte aligned");
    if (passes < 1) return fail(ctx, SONAR_ERR_ARG, "passes < 1");
    if (n_blocks < 1 || n_blocks > 65535) return fail(ctx, SONAR_ERR_ARG, "n_blocks outside [1, 65535]");
    CU(cudaSetDevice(ctx->device), "cudaSetDevice");
    CU(launch_l2_read(d_buf, bytes, passes, d_block_sums, n_blocks, (cudaStream_t)stream), "probe launch");
    return SONAR_OK;
}

// ===========================================================================
// rendering without device allocation
// ===========================================================================

namespace {

// The scratch of sonar_render_noalloc: a fixed array in the library's device
// image, resident on every device that loads the library until the process
// exits.  Host code cannot use the symbol as a pointer; each device's address
// comes from cudaGetSymbolAddress.
static __device__ __align__(256) float g_noalloc_scratch[SONAR_NOALLOC_SCRATCH_WORDS];

std::mutex g_noalloc_mutex;
std::map<unsigned long long, void*> g_noalloc_addr;   // by context id (unique for the process)

// The unique id of the calling thread's current context (cuCtxGetCurrent and
// cuCtxGetId, through the runtime's driver entry points); false when the
// driver does not offer them.
bool current_context_id(unsigned long long* id) {
    typedef int (*get_current_t)(void**);
    typedef int (*get_id_t)(void*, unsigned long long*);
    static get_current_t get_current = nullptr;
    static get_id_t get_id = nullptr;
    static bool looked_up = false;
    if (!looked_up) {
        void* f = nullptr;
        void* g = nullptr;
        cudaDriverEntryPointQueryResult q1, q2;
        if (cudaGetDriverEntryPointByVersion("cuCtxGetCurrent", &f, 12000, cudaEnableDefault, &q1) == cudaSuccess &&
            cudaGetDriverEntryPointByVersion("cuCtxGetId", &g, 12000, cudaEnableDefault, &q2) == cudaSuccess &&
            q1 == cudaDriverEntryPointSuccess && q2 == cudaDriverEntryPointSuccess) {
            get_current = (get_current_t)f;
            get_id = (get_id_t)g;
        }
        looked_up = true;
    }
    void* ctx = nullptr;
    return get_current && get_id && get_current(&ctx) == 0 && ctx && get_id(ctx, id) == 0;
}

// Device address of the scratch array in the current context (the caller has
// made the context's device current).  Looked up once per context: a context
// that is destroyed and created again (cudaDeviceReset) reloads the library's
// device code, the array may move, and the new context has a new id.  Where
// the driver cannot name the context, the address is looked up on every call
// (a host-side lookup once the device code is loaded).
cudaError_t noalloc_scratch(void** out) {
    std::lock_guard<std::mutex> lock(g_noalloc_mutex);
    unsigned long long id = 0;
    const bool keyed = current_context_id(&id);
    if (keyed) {
        auto it = g_noalloc_addr.find(id);
        if (it != g_noalloc_addr.end()) {
            *out = it->second;
            return cudaSuccess;
        }
    }
    void* p = nullptr;
    const cudaError_t e = cudaGetSymbolAddress(&p, g_noalloc_scratch);
    if (e != cudaSuccess) return e;
    if (keyed) g_noalloc_addr[id] = p;
    *out = p;
    return cudaSuccess;
}

}  // namespace

extern "C" sonar_status sonar_render_noalloc(sonar_ctx_t ctx, int32_t scene_id, const sonar_sensor* sensor,
                                             const sonar_params* params, const float* d_theta, int32_t n_mat,
                                             uint64_t seed, uint64_t frame, const sonar_outputs* out,
                                             void* stream) {
    if (!ctx) return SONAR_ERR_ARG;
    sonar_status st;
    if ((st = check_scene(ctx, scene_id)) || (st = check_sensor(ctx, sensor)) || (st = check_params(ctx, params)) ||
        (st = check_nmat(ctx, scene_id, n_mat)))
        return st;
    if (!d_theta) return fail(ctx, SONAR_ERR_ARG, "d_theta is NULL");
    if (!out || !out->polar) return fail(ctx, SONAR_ERR_ARG, "outputs or outputs->polar is NULL");
    if (out->hits && !aligned16(out->hits)) return fail(ctx, SONAR_ERR_ARG, "hits must be 16-byte aligned");
    if (out->fan && (out->fan_w < 1 || out->fan_h < 1)) return fail(ctx, SONAR_ERR_ARG, "fan size must be >= 1");
    // scratch layout (words): the image maximum at 0; from 64 the exact-ray
    // tables (4 words a beam and an elevation); then, each at a 256-byte
    // boundary, the hit records (4 words a ray) and the noised image unless the
    // caller passes them
    const int64_t npol = (int64_t)sensor->n_range_bins * sensor->n_az_bins;
    const int64_t trig_words = 4 * ((int64_t)sensor->n_beams + sensor->n_elev);
    const int64_t hits_at = 64 + (trig_words + 63) / 64 * 64;
    const int64_t hit_words = out->hits ? 0 : 4 * (int64_t)sensor->n_beams * sensor->n_elev;
    const int64_t noised_at = hits_at + (hit_words + 63) / 64 * 64;
    const int64_t need = out->noised ? noised_at : noised_at + npol;
    // the fold's compact lists (2 words a ray, 2 a column and band of 32 rows)
    // where the array has room for them too; else it writes P into the polar
    // image, which holds it until the row kernel overwrites it (same images)
    const int64_t vals_at = (need + 63) / 64 * 64;
    const int64_t bands_at = vals_at + (2 * (int64_t)sensor->n_beams * sensor->n_elev + 63) / 64 * 64;
    const int64_t fold_end = bands_at + 2 * (((int64_t)sensor->n_range_bins + 31) / 32) * sensor->n_az_bins;
    if (need > (int64_t)SONAR_NOALLOC_SCRATCH_WORDS)
        return fail(ctx, SONAR_ERR_ARG, "sonar_render_noalloc: frame needs " + std::to_string(need) +
                                            " scratch words, the fixed scratch holds " +
                                            std::to_string(SONAR_NOALLOC_SCRATCH_WORDS) +
                                            " (pass outputs->hits and outputs->noised to need fewer)");
    cudaStream_t s = (cudaStream_t)stream;
    CU(cudaSetDevice(ctx->device), "cudaSetDevice");
    void* base = nullptr;
    CU(noalloc_scratch(&base), "cudaGetSymbolAddress of the fixed scratch");
    uint32_t* rowmax = (uint32_t*)base;
    sonar_hit* hits = out->hits ? out->hits : (sonar_hit*)((float*)base + hits_at);
    float* noised = out->noised ? out->noised : (float*)base + noised_at;
    const Tune t = single_tune(ctx, *sensor);
    SensorDev S = make_sensor(*sensor, seed, frame, t, out->fan ? out->fan_w : 0, out->fan ? out->fan_h : 0);
    S.fold_block = fold_by_block(S, S.naz);
    S.trig = (float4*)((float*)base + 64);
    // single_forward clears the maximum (the array still holds the previous
    // call's values); hit records and the noised image are fully overwritten
    FoldStore fold;
    if (fold_end <= (int64_t)SONAR_NOALLOC_SCRATCH_WORDS) {
        fold.vals = (float2*)((float*)base + vals_at);
        fold.bands = (uint2*)((float*)base + bands_at);
    } else {
        fold.dense = out->polar;
    }
    bool capturing = false;
    CU(is_capturing(s, &capturing), "capture status");
    st = single_forward(ctx, S, scene_dev(ctx->scenes[scene_id]), params, d_theta, n_mat, hits, fold, noised,
                        out->binned, out->polar, rowmax, capturing, s);
    if (st != SONAR_OK) return st;
    return single_post(ctx, S, params->normalise, noised, rowmax, out->polar, out->fan, capturing, s);
}

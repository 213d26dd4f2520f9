// sj_api.cu -- C ABI of libsj.so (declared in include/sj.h): argument checks,
// layer construction (validation, MBBs, candidate lists) and the join
// pipelines (bucketing -> work items -> refinement), all stream-ordered.
#include <cuda_runtime.h>
#include <stdint.h>
#include <string.h>

#include <atomic>
#include <cmath>
#include <mutex>
#include <string>
#include <utility>
#include <vector>

#include "sj_host.hpp"

namespace sj {
cudaError_t launch_check_offsets(const int64_t *off, int64_t n, int64_t min_size, int64_t first, int64_t last, int *out,
                                 int *bad, cudaStream_t s);
cudaError_t launch_check_finite(const double2 *v, int n, int *bad, cudaStream_t s);
cudaError_t launch_pip_topology(const int *ring_off, int R, const int *poly_ring_off, int P, int V, int *poly_voff,
                                int *nxt, int *prv, int *owner, cudaStream_t s);
cudaError_t launch_split(const double2 *v, int n, float4 *vs, cudaStream_t s);
cudaError_t launch_seg_table(const double2 *v, const int *line_off, int L, int V, double2 *e64, double *inv64,
                             float4 *seg32, cudaStream_t s);
cudaError_t launch_mbb(const LayerBuildArgs &a, cudaStream_t s);
cudaError_t launch_raster_count(const LayerBuildArgs &a, unsigned long long *total, cudaStream_t s);
cudaError_t launch_raster_emit(const LayerBuildArgs &a, int2 *pairs, int M, int *cand_ids, cudaStream_t s);
cudaError_t launch_segcell_count(const LayerBuildArgs &a, const float4 *seg32, const double2 *e64, int *seg_off,
                                 unsigned long long *total, cudaStream_t s);
cudaError_t launch_segcell_emit(const LayerBuildArgs &a, const float4 *seg32, const double2 *e64, const int *seg_off,
                                int2 *pairs, int MS, const int *cand_ids, int *cseg_start, int *cseg_ids,
                                int *cell_algo, cudaStream_t s);
cudaError_t launch_prow_count(const LayerBuildArgs &a, int *prow_base, int *prow_r0, unsigned long long *total,
                              cudaStream_t s);
cudaError_t launch_cseg_records(const int *cseg_start, const int *cseg_ids, const GridDev &g, const float *frame_x,
                                const float *frame_y, const float4 *vsplit, const float4 *seg32, float4 *rec,
                                cudaStream_t s);
cudaError_t launch_offsets(const int *cnt, int n, int *out, int2 *block_sums, size_t cap, int *totals,
                           cudaStream_t s);
cudaError_t launch_sum64(const int *cnt, int n, unsigned long long *total, cudaStream_t s);
cudaError_t launch_thresholds(const GridDev &g, unsigned long long *kx, unsigned long long *ky, cudaStream_t s);
cudaError_t launch_frames(const GridDev &g, float *fx, float *fy, cudaStream_t s);
int p2p_blocks_per_sm(int form);
}  // namespace sj

using namespace sj;


// ------------------------------------------------------------------ errors

static thread_local std::string g_err;

sj_status sj::fail(sj_status st, const std::string &msg) {
    g_err = msg;
    return st;
}

sj_status sj::cuda_fail(cudaError_t e, const char *what) {
    return fail(e == cudaErrorMemoryAllocation ? SJ_ERR_OOM : SJ_ERR_CUDA,
                std::string(what) + ": " + cudaGetErrorString(e));
}

// ------------------------------------------------------------------ bounds-checked build

// After a join of a build compiled with SJ_CHECK_BOUNDS: synchronise the
// stream and read the kernels' error words; a guard that fired (an index out
// of range, skipped on the device) makes the call fail with SJ_ERR_CUDA.  In
// normal builds: nothing.
static sj_status check_bounds(cudaStream_t s) {
#ifdef SJ_CHECK_BOUNDS
    CUDA_TRY(cudaStreamSynchronize(s));
    const unsigned v = bounds_take_filter() | bounds_take_p2p() | bounds_take_pip();
    if (v) return fail(SJ_ERR_CUDA, "bounds check: out-of-range device accesses skipped, guard codes " +
                                        std::to_string(v));
#else
    (void)s;
#endif
    return SJ_OK;
}

extern "C" int32_t sj_bounds_checked(void) {
#ifdef SJ_CHECK_BOUNDS
    return 1;
#else
    return 0;
#endif
}

// ------------------------------------------------------------------ fault injection

static std::mutex g_fault_mu;
static int g_fault_kind = SJ_FAULT_NONE, g_fault_after = 0, g_fault_count = 0;

bool sj::fault_fires(int kind) {
    std::lock_guard<std::mutex> lk(g_fault_mu);
    if (g_fault_kind != kind || g_fault_count <= 0) return false;
    if (g_fault_after > 0) {
        --g_fault_after;
        return false;
    }
    if (--g_fault_count == 0) g_fault_kind = SJ_FAULT_NONE;
    return true;
}

cudaError_t sj::dev_malloc(void **p, size_t bytes) {
    if (fault_fires(SJ_FAULT_ALLOC)) return cudaErrorMemoryAllocation;
    return cudaMalloc(p, bytes);
}

cudaError_t sj::dev_malloc_async(void **p, size_t bytes, cudaStream_t s) {
    if (fault_fires(SJ_FAULT_ALLOC)) return cudaErrorMemoryAllocation;
    return cudaMallocAsync(p, bytes, s);
}

extern "C" sj_status sj_fault_inject(int32_t kind, int32_t after, int32_t count) {
    if (kind != SJ_FAULT_NONE && kind != SJ_FAULT_ALLOC && kind != SJ_FAULT_ADMIT)
        return fail(SJ_ERR_INVALID, "unknown fault kind");
    if (after < 0 || count < 0) return fail(SJ_ERR_INVALID, "after and count must be >= 0");
    std::lock_guard<std::mutex> lk(g_fault_mu);
    g_fault_kind = count > 0 ? kind : SJ_FAULT_NONE;
    g_fault_after = after;
    g_fault_count = count;
    return SJ_OK;
}

extern "C" int32_t sj_fault_pending(void) {
    std::lock_guard<std::mutex> lk(g_fault_mu);
    return g_fault_kind == SJ_FAULT_NONE ? 0 : g_fault_count;
}

// ------------------------------------------------------------------ device info

static DevInfo g_dev[64];
static std::mutex g_dev_mu;

sj_status sj::device_info(int dev, DevInfo **out) {
    if (dev < 0 || dev >= 64) return fail(SJ_ERR_INVALID, "device index out of range");
    std::lock_guard<std::mutex> lk(g_dev_mu);
    DevInfo &d = g_dev[dev];
    if (!d.init) {
        CUDA_TRY(cudaDeviceGetAttribute(&d.sms, cudaDevAttrMultiProcessorCount, dev));
        for (int f = 0; f < 2; ++f) d.p2p_bps[f] = p2p_blocks_per_sm(f);
        // keep freed stream-ordered scratch in the pool for the next call
        cudaMemPool_t pool;
        if (cudaDeviceGetDefaultMemPool(&pool, dev) == cudaSuccess) {
            uint64_t thr = UINT64_MAX;
            cudaMemPoolSetAttribute(pool, cudaMemPoolAttrReleaseThreshold, &thr);
        }
        for (cudaStream_t &hs : d.hstream) CUDA_TRY(cudaStreamCreateWithFlags(&hs, cudaStreamNonBlocking));
        d.init = true;
    }
    *out = &d;
    return SJ_OK;
}

static bool grid_ok(const sj_grid *g) {
    if (!g) return false;
    if (!(g->nx >= 1 && g->ny >= 1)) return false;
    if (g->nx > (1 << 20) || g->ny > (1 << 20)) return false;
    if ((int64_t)g->nx * (int64_t)g->ny > MAX_COUNT) return false;
    if (!(std::isfinite(g->x0) && std::isfinite(g->x1) && std::isfinite(g->y0) && std::isfinite(g->y1))) return false;
    return g->x1 > g->x0 && g->y1 > g->y0;
}

// Bound of axis_estimate's error, in cells: |v - fl(v)| < 2u |v| (truncation) or
// 2^-126 (flushed to zero), |x0f - x0| <= u |x0|, the difference's rounding u per
// cell index, 1 / w rounded (2u) and the product (u): at most (3u max|x| + 2^-126)
// / w + 4u n cells, times 1.5.  Beyond 1e37 the estimate is never certain: from
// 3.4e38 on approx_float clamps, and 1 / w leaves the FP32 normal range at 8.5e37.
// Below, a clamped value maps past the grid's end.  Nor is it with cells below
// 1e-37: from 2.9e-39 on 1 / w is infinite, and every point seems far outside.
static float estimate_tol(double lo, double hi, double w, int n) {
    const double u = 5.9604644775390625e-08, m = std::max(std::fabs(lo), std::fabs(hi));
    if (!(m <= 1e37 && w >= 1e-37)) return INFINITY;
    return (float)(1.5 * ((3.0 * u * m + 1.1754943508222875e-38) / w + 4.0 * u * n));
}

static GridDev make_grid(const sj_grid *g) {
    GridDev d;
    d.x0 = g->x0; d.y0 = g->y0; d.x1 = g->x1; d.y1 = g->y1;
    d.nx = g->nx; d.ny = g->ny;
    d.G = g->nx * g->ny;
    volatile double cw = (g->x1 - g->x0) / (double)g->nx;   // one IEEE division each
    volatile double ch = (g->y1 - g->y0) / (double)g->ny;
    d.cw = cw; d.ch = ch;
    d.x0f = (float)g->x0; d.y0f = (float)g->y0;
    d.icwf = (float)(1.0 / cw); d.ichf = (float)(1.0 / ch);
    d.tolx = estimate_tol(g->x0, g->x1, cw, g->nx);
    d.toly = estimate_tol(g->y0, g->y1, ch, g->ny);
    d.kx = d.ky = nullptr;
    return d;
}

// Threshold tables of point_cell for the grid of layer L (computed on the GPU
// with the FP64 cell rule itself).
static sj_status layer_tables(sj_layer *L, cudaStream_t s) {
    CUDA_TRY(dev_malloc((void **)&L->cell_keys, sizeof(unsigned long long) * ((size_t)L->g.nx + L->g.ny + 2)));
    CUDA_TRY(launch_thresholds(L->g, L->cell_keys, L->cell_keys + L->g.nx + 1, s));
    L->g.kx = L->cell_keys;
    L->g.ky = L->cell_keys + L->g.nx + 1;
    CUDA_TRY(dev_malloc((void **)&L->frames, sizeof(float) * ((size_t)L->g.nx + L->g.ny)));
    CUDA_TRY(launch_frames(L->g, L->frames, L->frames + L->g.nx, s));
    L->xmax = std::max(std::max(std::fabs(L->grid.x0), std::fabs(L->grid.x1)),
                       std::max(std::fabs(L->grid.y0), std::fabs(L->grid.y1)));
    return SJ_OK;
}

// FP32 float at or below (down) / at or above (up) the double x.
static float float_down(double x) {
    float f = (float)x;
    return ((double)f > x) ? std::nextafter(f, -INFINITY) : f;
}
static float float_up(double x) {
    float f = (float)x;
    return ((double)f < x) ? std::nextafter(f, INFINITY) : f;
}

// Layer-dependent fields of the P2P refinement arguments.
void sj::fill_refine(const sj_layer *L, RefineArgs &ra) {
    ra.g = L->g;
    ra.seg = SegArgs{L->verts, L->seg_e64, L->seg_inv64, L->seg32};
    ra.cseg_start = L->cseg_start;
    ra.cseg_ids = L->cseg_ids;
    ra.cseg_rec = L->cseg_rec;
    ra.D = L->D;
    ra.Df = L->Df;
    ra.Ddn = L->Ddn;
    ra.Dup = L->Dup;
    ra.eps_abs = L->eps_abs;
    // where the squares of coordinates or the FP32 inverse lengths could leave
    // the FP32 range, an infinite bound sends every point to the FP64 recheck
    if (!(L->xmax <= 1e15 && L->xmax >= 1e-6)) ra.eps_abs = INFINITY;
    ra.frame_x = L->frames;
    ra.frame_y = L->frames + L->g.nx;
    ra.stats = L->stats;
}

// Arguments of the PIP join of a polygon layer.  Beyond the FP32 range the
// cell-relative coordinates mean nothing: an infinite rounding bound sends
// every test to the FP64 rule.
PipArgs sj::pip_args(const sj_layer *L) {
    PipArgs a{};
    a.g = L->g;
    a.cells = L->cells;
    a.units = L->units;
    a.units_n = (int)L->units_n;
    a.verts = L->verts;
    a.nxt = L->nxt;
    a.frame_x = L->frames;
    a.frame_y = L->frames + L->g.nx;
    a.eps = L->xmax > 1e30 ? INFINITY : L->eps_abs;
    a.search = PIP_SEARCH;
    a.stats = L->stats;
    return a;
}

// ------------------------------------------------------------------ layers

// Sum and destroy the pending timing events (the device must be idle).
static void resolve_events(const sj_layer *L) {
    std::lock_guard<std::mutex> lk(L->ev_mu);
    for (auto &p : L->ev_pending) {
        float ms = 0.0f;
        if (cudaEventElapsedTime(&ms, p.first, p.second) == cudaSuccess) {
            L->refine_ms += ms;
            L->refine_launches += 1;
        }
        cudaEventDestroy(p.first);
        cudaEventDestroy(p.second);
    }
    L->ev_pending.clear();
}

static void layer_free(sj_layer *L) {
    resolve_events(L);
    void *ptrs[] = {L->verts, L->vsplit, L->obj_voff, L->nxt, L->ring_off, L->poly_ring_off, L->seg_e64,
                    L->seg_inv64, L->seg32, L->mbb, L->cand_start, L->cand_ids, L->stats, L->cell_keys,
                    L->frames, L->cseg_start, L->cseg_ids, L->cell_algo, L->cseg_rec, L->prow_base, L->prow_r0,
                    L->prow_start, L->pedge_ids, L->cell_work, L->cells, L->units};
    for (void *p : ptrs)
        if (p) cudaFree(p);
    delete L;
}

struct LayerGuard {
    sj_layer *L;
    ~LayerGuard() {
        if (L) layer_free(L);
    }
};

template <class T>
static cudaError_t dalloc(T **p, size_t n) {
    return dev_malloc((void **)p, (n ? n : 1) * sizeof(T));
}

static sj_status read_flag(int *dflag, cudaStream_t s, int *out) {
    CUDA_TRY(cudaMemcpyAsync(out, dflag, sizeof(int), cudaMemcpyDeviceToHost, s));
    CUDA_TRY(cudaStreamSynchronize(s));
    return SJ_OK;
}

// What a layer's build leaves reserved in the stream-ordered pool: what was
// reserved before, or BUILD_KEEP; the rest goes back to the device when this object,
// declared before the scratch, ends.  Kept for the next build, which would map it
// again: with nothing kept the 40,000 tiles take 2.65 instead of 2.19 ms to build,
// the heavy-tail tiling (850 MB of scratch) 10.1 instead of 7.8.  1 GB of the
// device's 280, so that what is sized from the free memory hardly shrinks.
constexpr uint64_t BUILD_KEEP = 1u << 30;
struct BuildPool {
    cudaStream_t s;
    cudaMemPool_t pool = nullptr;
    uint64_t keep = BUILD_KEEP;
    BuildPool(int dev, cudaStream_t st) : s(st) {
        uint64_t r = 0;
        if (cudaDeviceGetDefaultMemPool(&pool, dev) != cudaSuccess) pool = nullptr;
        else if (cudaMemPoolGetAttribute(pool, cudaMemPoolAttrReservedMemCurrent, &r) == cudaSuccess && r > keep) keep = r;
    }
    ~BuildPool() {
        uint64_t r = 0;
        if (!pool || cudaMemPoolGetAttribute(pool, cudaMemPoolAttrReservedMemCurrent, &r) != cudaSuccess || r <= keep) return;
        cudaStreamSynchronize(s);   // the scratch has been given back by then
        cudaMemPoolTrimTo(pool, keep);
    }
};

// Build scratch: stream-ordered allocations, freed with the object.
struct BuildTmp {
    cudaStream_t s;
    std::vector<void *> ptrs;
    explicit BuildTmp(cudaStream_t st) : s(st) {}
    ~BuildTmp() {
        for (void *p : ptrs) cudaFreeAsync(p, s);
    }
    template <class T>
    cudaError_t take(T **p, size_t n) {
        void *q = nullptr;
        cudaError_t e = dev_malloc_async(&q, (n ? n : 1) * sizeof(T), s);
        if (e == cudaSuccess) {
            ptrs.push_back(q);
            *p = (T *)q;
        }
        return e;
    }
};

// Shared tail of both layer builders: MBB, cover check, rasterisation, CSR.
static sj_status build_candidates(sj_layer *L, int *dbad, cudaStream_t s) {
    LayerBuildArgs a{};
    a.g = L->g;
    a.kind = L->kind;
    a.D = L->D;
    a.nobj = L->nobj;
    a.V = L->V;
    a.verts = L->verts;
    a.obj_voff = L->obj_voff;
    a.bad = dbad;
    CUDA_TRY(dalloc(&L->mbb, (size_t)L->nobj));
    CUDA_TRY(dalloc(&L->cand_start, (size_t)L->g.G + 1));
    a.mbb = L->mbb;
    a.cand_start = L->cand_start;

    int *cell_cnt = nullptr, *cursor = nullptr, *obj_cells = nullptr, *totals = nullptr;
    int2 *block_sums = nullptr, *pairs = nullptr;
    unsigned long long *total = nullptr;
    size_t nbs = bucket_scan_blocks(std::max(L->g.G, L->nobj));
    BuildTmp tmp(s);
    CUDA_TRY(tmp.take(&cell_cnt, (size_t)L->g.G + 1));
    CUDA_TRY(tmp.take(&cursor, (size_t)L->g.G));
    CUDA_TRY(tmp.take(&obj_cells, (size_t)L->nobj + 1));
    CUDA_TRY(tmp.take(&block_sums, nbs));
    CUDA_TRY(tmp.take(&totals, 4));
    CUDA_TRY(tmp.take(&total, 1));
    CUDA_TRY(cudaMemsetAsync(cell_cnt, 0, sizeof(int) * ((size_t)L->g.G + 1), s));
    CUDA_TRY(cudaMemsetAsync(cursor, 0, sizeof(int) * (size_t)L->g.G, s));
    CUDA_TRY(cudaMemsetAsync(total, 0, sizeof(unsigned long long), s));
    a.cell_cnt = cell_cnt;
    a.cursor = cursor;
    a.obj_cells = obj_cells;
    a.block_sums = block_sums;
    a.bs_cap = nbs;
    a.totals = totals;

    if (L->nobj > 0) {
        CUDA_TRY(launch_mbb(a, s));
        int bad = 0;
        sj_status st = read_flag(dbad, s, &bad);
        if (st != SJ_OK) return st;
        if (bad & 2) return fail(SJ_ERR_GRID_COVER, "an object's MBB is not inside the closed grid box");
        CUDA_TRY(launch_raster_count(a, total, s));
    }
    unsigned long long M = 0;
    CUDA_TRY(cudaMemcpyAsync(&M, total, sizeof(M), cudaMemcpyDeviceToHost, s));
    CUDA_TRY(cudaStreamSynchronize(s));
    if (M > (unsigned long long)MAX_COUNT) return fail(SJ_ERR_INVALID, "more than 2^31 - 2^22 (cell, object) candidate pairs");
    L->M = (int64_t)M;
    CUDA_TRY(dalloc(&L->cand_ids, (size_t)M));
    if (L->nobj > 0) {
        CUDA_TRY(tmp.take(&pairs, (size_t)M));
        CUDA_TRY(launch_raster_emit(a, pairs, (int)M, L->cand_ids, s));
    } else {
        CUDA_TRY(cudaMemsetAsync(L->cand_start, 0, sizeof(int) * ((size_t)L->g.G + 1), s));
    }
    CUDA_TRY(cudaStreamSynchronize(s));
    // The cell-relative coordinate rel = fl32(fl32(hi - o) + lo) of any value v
    // in the grid box satisfies |rel - (v - o)| <= 2.0001 u |rel| + eps_abs with
    // eps_abs = 6.0001 u^2 max|coordinate| (the truncation remainder |lo| is
    // below 2u |v|, rounded once more by the conversion); 8 u^2 is used.
    double u = 5.9604644775390625e-08;
    L->eps_abs = (float)(8.0 * u * u * L->xmax * (1.0 + 1e-6)) + 1e-30f;
    L->Df = (float)L->D;
    L->Ddn = float_down(L->D * (1.0 - 1e-12));
    L->Dup = float_up(L->D * (1.0 + 1e-12) + 1e-300);
    return SJ_OK;
}

// P2P per-cell segment lists (after build_candidates): every segment whose box
// widened by D meets a cell is listed under that cell, sorted by segment index.
static sj_status build_seg_lists(sj_layer *L, cudaStream_t s) {
    const int G = L->g.G, V = L->V;
    CUDA_TRY(dalloc(&L->cseg_start, (size_t)G + 1));
    CUDA_TRY(dalloc(&L->cell_algo, (size_t)G));
    if (V == 0) {
        L->MS = 0;
        CUDA_TRY(dalloc(&L->cseg_ids, 0));
        CUDA_TRY(dalloc(&L->cseg_rec, 0));
        CUDA_TRY(dalloc(&L->cell_work, (size_t)G));
        CUDA_TRY(cudaMemsetAsync(L->cseg_start, 0, sizeof(int) * ((size_t)G + 1), s));
        CUDA_TRY(cudaMemsetAsync(L->cell_algo, 0, sizeof(int) * (size_t)G, s));
        CUDA_TRY(cudaMemsetAsync(L->cell_work, 0, sizeof(int) * (size_t)G, s));
        CUDA_TRY(cudaStreamSynchronize(s));
        return SJ_OK;
    }
    LayerBuildArgs a{};
    a.g = L->g;
    a.kind = KIND_P2P;
    a.D = L->D;
    a.nobj = L->nobj;
    a.V = V;
    a.verts = L->verts;
    a.obj_voff = L->obj_voff;
    a.cand_start = L->cand_start;
    BuildTmp tmp(s);
    int *seg_off = nullptr;
    int2 *pairs = nullptr;
    unsigned long long *total = nullptr;
    const size_t nbs = bucket_scan_blocks(std::max(G, V));
    CUDA_TRY(tmp.take(&a.cell_cnt, (size_t)G + 1));
    CUDA_TRY(tmp.take(&a.cursor, (size_t)G));
    CUDA_TRY(tmp.take(&seg_off, (size_t)V + 1));
    CUDA_TRY(tmp.take(&a.block_sums, nbs));
    a.bs_cap = nbs;
    CUDA_TRY(tmp.take(&a.totals, 4));
    CUDA_TRY(tmp.take(&total, 1));
    CUDA_TRY(cudaMemsetAsync(a.cell_cnt, 0, sizeof(int) * ((size_t)G + 1), s));
    CUDA_TRY(cudaMemsetAsync(a.cursor, 0, sizeof(int) * (size_t)G, s));
    CUDA_TRY(cudaMemsetAsync(total, 0, sizeof(unsigned long long), s));
    CUDA_TRY(launch_segcell_count(a, L->seg32, L->seg_e64, seg_off, total, s));
    unsigned long long MS = 0;
    CUDA_TRY(cudaMemcpyAsync(&MS, total, sizeof(MS), cudaMemcpyDeviceToHost, s));
    CUDA_TRY(cudaStreamSynchronize(s));
    if (MS > (unsigned long long)MAX_COUNT) return fail(SJ_ERR_INVALID, "more than 2^31 - 2^22 (cell, segment) pairs");
    L->MS = (int64_t)MS;
    CUDA_TRY(dalloc(&L->cseg_ids, (size_t)MS));
    CUDA_TRY(tmp.take(&pairs, (size_t)MS));
    CUDA_TRY(launch_segcell_emit(a, L->seg32, L->seg_e64, seg_off, pairs, (int)MS, L->cand_ids, L->cseg_start,
                                 L->cseg_ids, L->cell_algo, s));
    CUDA_TRY(dalloc(&L->cseg_rec, 2 * (size_t)MS));
    CUDA_TRY(launch_cseg_records(L->cseg_start, L->cseg_ids, L->g, L->frames, L->frames + L->g.nx, L->vsplit,
                                 L->seg32, L->cseg_rec, s));
    CUDA_TRY(dalloc(&L->cell_work, (size_t)G));
    CUDA_TRY(launch_cell_work_p2p(L->cseg_start, G, L->cell_work, s));
    CUDA_TRY(cudaStreamSynchronize(s));
    return SJ_OK;
}

// 64-bit counters on the device, read back.
static sj_status read_totals(const unsigned long long *d, unsigned long long *h, int n, cudaStream_t s) {
    CUDA_TRY(cudaMemcpyAsync(h, d, sizeof(*h) * (size_t)n, cudaMemcpyDeviceToHost, s));
    CUDA_TRY(cudaStreamSynchronize(s));
    return SJ_OK;
}

// PIP cell records (after build_candidates): per-(polygon, row) edge lists,
// what each candidate entry holds, the cells' codes and records (sj_pip.cu).
// prv and owner (per vertex) are the caller's.
static sj_status build_pip_records(sj_layer *L, const int *prv, const int *owner, cudaStream_t s) {
    const int P = L->nobj, G = L->g.G, V = L->V, M = (int)L->M;
    CUDA_TRY(dalloc(&L->prow_base, (size_t)P + 1));
    CUDA_TRY(dalloc(&L->prow_r0, (size_t)P));
    CUDA_TRY(dalloc(&L->cells, (size_t)G));
    if (P == 0) {
        L->MR = L->ME = L->units_n = 0;
        CUDA_TRY(dalloc(&L->prow_start, 1));
        CUDA_TRY(dalloc(&L->pedge_ids, 0));
        CUDA_TRY(dalloc(&L->units, 0));
        CUDA_TRY(cudaMemsetAsync(L->cells, 0xff, sizeof(int4) * (size_t)G, s));   // -1: no candidates
        CUDA_TRY(cudaMemsetAsync(L->prow_base, 0, sizeof(int), s));
        CUDA_TRY(cudaMemsetAsync(L->prow_start, 0, sizeof(int), s));
        CUDA_TRY(cudaStreamSynchronize(s));
        return SJ_OK;
    }
    BuildTmp tmp(s);
    unsigned long long *total = nullptr, h[4] = {};
    int *totals = nullptr;
    CUDA_TRY(tmp.take(&total, 4));
    CUDA_TRY(tmp.take(&totals, 4));
    CUDA_TRY(cudaMemsetAsync(total, 0, 4 * sizeof(unsigned long long), s));

    // rows of each polygon, then its (polygon, row) edge lists
    LayerBuildArgs a{};
    a.g = L->g;
    a.kind = KIND_PIP;
    a.nobj = P;
    a.V = V;
    a.verts = L->verts;
    a.obj_voff = L->obj_voff;
    a.mbb = L->mbb;
    a.totals = totals;
    a.bs_cap = bucket_scan_blocks(P);
    CUDA_TRY(tmp.take(&a.block_sums, a.bs_cap));
    CUDA_TRY(launch_prow_count(a, L->prow_base, L->prow_r0, total, s));
    PipBuildArgs b{};
    b.g = L->g;
    b.V = V;
    b.M = M;
    b.verts = L->verts;
    b.nxt = L->nxt;
    b.prv = prv;
    b.owner = owner;
    b.obj_voff = L->obj_voff;
    b.cand_start = L->cand_start;
    b.cand_ids = L->cand_ids;
    b.prow_base = L->prow_base;
    b.prow_r0 = L->prow_r0;
    b.frame_x = L->frames;
    b.frame_y = L->frames + L->g.nx;
    CUDA_TRY(tmp.take(&b.e.rows, (size_t)V));
    CUDA_TRY(tmp.take(&b.e.xr, (size_t)V));
    CUDA_TRY(tmp.take(&b.e.kind, (size_t)V));
    CUDA_TRY(launch_pip_edges(b, s));
    sj_status st = read_totals(total, h, 1, s);
    if (st != SJ_OK) return st;
    if (h[0] > (unsigned long long)MAX_COUNT) return fail(SJ_ERR_INVALID, "more than 2^31 - 2^22 (polygon, row) slots");
    L->MR = (int64_t)h[0];
    int *cnt = nullptr, *cursor = nullptr;
    int2 *bs = nullptr;
    const size_t slots_cap = bucket_scan_blocks((int)L->MR);
    CUDA_TRY(tmp.take(&cnt, (size_t)L->MR));
    CUDA_TRY(tmp.take(&cursor, (size_t)L->MR));
    CUDA_TRY(tmp.take(&bs, slots_cap));
    CUDA_TRY(cudaMemsetAsync(cnt, 0, sizeof(int) * (size_t)L->MR, s));
    CUDA_TRY(cudaMemsetAsync(cursor, 0, sizeof(int) * (size_t)L->MR, s));
    CUDA_TRY(launch_prow_edges(b, cnt, total + 1, nullptr, nullptr, nullptr, s));
    // pairs of equal edges, while the list sizes travel
    {
        size_t slots = 64;
        while (slots < 2 * (size_t)V && slots < ((size_t)1 << 31)) slots <<= 1;
        int *table = nullptr;
        CUDA_TRY(tmp.take(&table, slots));
        CUDA_TRY(tmp.take(&b.twin, (size_t)V));
        CUDA_TRY(launch_pip_twins(b, table, (unsigned)slots, s));
    }
    st = read_totals(total + 1, h, 1, s);
    if (st != SJ_OK) return st;
    if (h[0] > (unsigned long long)MAX_COUNT) return fail(SJ_ERR_INVALID, "more than 2^31 - 2^22 (polygon, row, edge) entries");
    L->ME = (int64_t)h[0];
    CUDA_TRY(dalloc(&L->prow_start, (size_t)L->MR + 1));
    CUDA_TRY(dalloc(&L->pedge_ids, (size_t)L->ME));
    CUDA_TRY(launch_offsets(cnt, (int)L->MR, L->prow_start, bs, slots_cap, totals, s));
    PipRow *rows = nullptr;
    CUDA_TRY(tmp.take(&rows, (size_t)L->ME));
    CUDA_TRY(launch_prow_edges(b, cursor, nullptr, L->prow_start, L->pedge_ids, rows, s));
    b.prow_start = L->prow_start;
    b.rows = rows;

    // what each entry and cell holds; delta = 1e-7 of the largest grid coordinate
    // (0.01 m at 1e5 m) is far above FP64 rounding and far below a cell
    const double delta = 1e-7 * L->xmax + 1e-300;
    int *at[3] = {};
    CUDA_TRY(tmp.take(&b.col, (size_t)L->g.nx));
    CUDA_TRY(tmp.take(&b.entry_cell, (size_t)M));
    CUDA_TRY(tmp.take(&b.ord, (size_t)M));
    CUDA_TRY(tmp.take(&b.edge_at, (size_t)M));
    CUDA_TRY(tmp.take(&b.flip_at, (size_t)M));
    CUDA_TRY(tmp.take(&b.ent, (size_t)M));
    int **of[3] = {&b.units_of, &b.edges_of, &b.flips_of};
    for (int q = 0; q < 3; ++q) {
        CUDA_TRY(tmp.take(of[q], (size_t)G));
        CUDA_TRY(tmp.take(&at[q], (size_t)G + 1));
    }
    b.cells = L->cells;
    // sub-cell classes: margin for delta, for twice the error of a point's place in
    // its cell (the place and the cell's edge), and for the frame origin's rounding
    // and the box's own; none where it would fill the sub-cell
    b.cwf = (float)L->g.cw;
    b.chf = (float)L->g.ch;
    b.eps = pip_args(L).eps;
    const double u = 5.9604644775390625e-08, rest = delta + 4.0 * u * L->xmax;
    const double mx = 1.01 * (rest + (2.0 * L->g.tolx + 8.0 * u) * L->g.cw);
    const double my = 1.01 * (rest + (2.0 * L->g.toly + 8.0 * u) * L->g.ch);
    const bool subs = mx < L->g.cw / 32 && my < L->g.ch / 32 && L->xmax <= 1e15 && L->xmax >= 1e-6;
    b.sub_mx = subs ? float_up(mx) : -1.0f;
    b.sub_my = subs ? float_up(my) : -1.0f;
    CUDA_TRY(launch_pip_count(b, delta, s));
    int2 *bs2 = nullptr;
    const size_t cells_cap = bucket_scan_blocks(G);
    CUDA_TRY(tmp.take(&bs2, cells_cap));
    CUDA_TRY(cudaMemsetAsync(total, 0, 3 * sizeof(unsigned long long), s));
    for (int q = 0; q < 3; ++q) {
        CUDA_TRY(launch_sum64(*of[q], G, total + q, s));
        CUDA_TRY(launch_offsets(*of[q], G, at[q], bs2, cells_cap, totals, s));
    }
    st = read_totals(total, h, 3, s);
    if (st != SJ_OK) return st;
    for (int q = 0; q < 3; ++q)
        if (h[q] > (unsigned long long)MAX_COUNT) return fail(SJ_ERR_INVALID, "cell records exceed 2^31 - 2^22 entries");
    L->units_n = (int64_t)h[0];
    CUDA_TRY(dalloc(&L->units, 2 * ((size_t)h[0] + 2)));   // the join reads two units past a header
    CUDA_TRY(cudaMemsetAsync(L->units + 2 * (size_t)h[0], 0, 4 * sizeof(int4), s));
    CUDA_TRY(tmp.take(&b.tmp_edge, (size_t)h[1]));
    CUDA_TRY(tmp.take(&b.tmp_rel, (size_t)h[1]));
    CUDA_TRY(tmp.take(&b.tmp_flip, (size_t)h[2]));
    CUDA_TRY(tmp.take(&b.long_list, (size_t)((h[1] + h[2]) / PIP_LONG_MIN) + 1));
    CUDA_TRY(tmp.take(&b.long_n, 1));
    CUDA_TRY(cudaMemsetAsync(b.long_n, 0, sizeof(int), s));
    b.units_at = at[0];
    b.edges_at = at[1];
    b.flips_at = at[2];
    b.units = L->units;
    CUDA_TRY(launch_pip_records(b, s));
    CUDA_TRY(cudaStreamSynchronize(s));
    return SJ_OK;
}

static sj_status layer_common_checks(const double *verts, int64_t V, const sj_grid *g, void *stream,
                                     sj_layer **out, DevInfo **di) {
    if (!out) return fail(SJ_ERR_INVALID, "out is NULL");
    *out = nullptr;
    if (!grid_ok(g)) return fail(SJ_ERR_INVALID, "invalid grid");
    if (V < 0 || V > MAX_COUNT) return fail(SJ_ERR_INVALID, "vertex count out of range (at most 2^31 - 2^22)");
    if (V > 0 && (!verts || !aligned16(verts))) return fail(SJ_ERR_INVALID, "verts NULL or not 16-byte aligned");
    (void)stream;
    int dev = 0;
    CUDA_TRY(cudaGetDevice(&dev));
    return device_info(dev, di);
}

extern "C" sj_status sj_pip_layer_create(const double *verts, int64_t V, const int64_t *ring_off, int64_t R,
                                         const int64_t *poly_ring_off, int32_t P, const sj_grid *g, void *stream,
                                         sj_layer **out) {
    DevInfo *di;
    sj_status st = layer_common_checks(verts, V, g, stream, out, &di);
    if (st != SJ_OK) return st;
    if (P < 0 || R < 0 || R > MAX_COUNT) return fail(SJ_ERR_INVALID, "ring or polygon count out of range");
    if (!ring_off || !poly_ring_off) return fail(SJ_ERR_INVALID, "offset array is NULL");
    cudaStream_t s = (cudaStream_t)stream;
    LayerGuard guard{new sj_layer()};
    sj_layer *L = guard.L;
    L->kind = KIND_PIP;
    CUDA_TRY(cudaGetDevice(&L->device));
    BuildPool bounded(L->device, s);
    L->grid = *g;
    L->g = make_grid(g);
    {
        sj_status ts = layer_tables(L, s);
        if (ts != SJ_OK) return ts;
    }
    L->nobj = P;
    L->V = (int)V;
    L->R = R;
    int *dbad = nullptr;
    CUDA_TRY(dalloc(&dbad, 1));
    struct F { int *p; ~F() { cudaFree(p); } } fbad{dbad};
    CUDA_TRY(cudaMemsetAsync(dbad, 0, sizeof(int), s));
    CUDA_TRY(dalloc(&L->ring_off, (size_t)R + 1));
    CUDA_TRY(dalloc(&L->poly_ring_off, (size_t)P + 1));
    CUDA_TRY(launch_check_offsets(ring_off, R, 3, 0, V, L->ring_off, dbad, s));
    CUDA_TRY(launch_check_offsets(poly_ring_off, P, 1, 0, R, L->poly_ring_off, dbad, s));
    CUDA_TRY(dalloc(&L->verts, (size_t)V));
    if (V > 0) {
        CUDA_TRY(cudaMemcpyAsync(L->verts, verts, sizeof(double2) * (size_t)V, cudaMemcpyDeviceToDevice, s));
        CUDA_TRY(launch_check_finite(L->verts, (int)V, dbad, s));
    }
    int bad = 0;
    st = read_flag(dbad, s, &bad);
    if (st != SJ_OK) return st;
    if (bad) return fail(SJ_ERR_INVALID, "invalid polygon layer (offsets, ring sizes or non-finite vertex)");
    CUDA_TRY(dalloc(&L->obj_voff, (size_t)P + 1));
    CUDA_TRY(dalloc(&L->nxt, (size_t)V));
    BuildTmp tmp(s);
    int *prv = nullptr, *owner = nullptr;
    CUDA_TRY(tmp.take(&prv, (size_t)V));
    CUDA_TRY(tmp.take(&owner, (size_t)V));
    CUDA_TRY(launch_pip_topology(L->ring_off, (int)R, L->poly_ring_off, P, (int)V, L->obj_voff, L->nxt, prv, owner, s));
    CUDA_TRY(dalloc(&L->stats, ST_N));
    CUDA_TRY(cudaMemsetAsync(L->stats, 0, sizeof(unsigned long long) * ST_N, s));
    st = build_candidates(L, dbad, s);
    if (st != SJ_OK) return st;
    st = build_pip_records(L, prv, owner, s);
    if (st != SJ_OK) return st;
    *out = L;
    guard.L = nullptr;
    return SJ_OK;
}

extern "C" sj_status sj_p2p_layer_create(const double *verts, int64_t V, const int64_t *line_off, int32_t Lc, double D,
                                         const sj_grid *g, void *stream, sj_layer **out) {
    DevInfo *di;
    sj_status st = layer_common_checks(verts, V, g, stream, out, &di);
    if (st != SJ_OK) return st;
    if (Lc < 0) return fail(SJ_ERR_INVALID, "polyline count out of range");
    if (!line_off) return fail(SJ_ERR_INVALID, "line_off is NULL");
    if (!(std::isfinite(D) && D >= 0.0)) return fail(SJ_ERR_INVALID, "D must be finite and >= 0");
    cudaStream_t s = (cudaStream_t)stream;
    LayerGuard guard{new sj_layer()};
    sj_layer *L = guard.L;
    L->kind = KIND_P2P;
    CUDA_TRY(cudaGetDevice(&L->device));
    BuildPool bounded(L->device, s);
    L->grid = *g;
    L->g = make_grid(g);
    {
        sj_status ts = layer_tables(L, s);
        if (ts != SJ_OK) return ts;
    }
    L->nobj = Lc;
    L->V = (int)V;
    L->R = Lc;
    L->D = D;
    int *dbad = nullptr;
    CUDA_TRY(dalloc(&dbad, 1));
    struct F { int *p; ~F() { cudaFree(p); } } fbad{dbad};
    CUDA_TRY(cudaMemsetAsync(dbad, 0, sizeof(int), s));
    CUDA_TRY(dalloc(&L->obj_voff, (size_t)Lc + 1));
    CUDA_TRY(launch_check_offsets(line_off, Lc, 1, 0, V, L->obj_voff, dbad, s));
    CUDA_TRY(dalloc(&L->verts, (size_t)V));
    if (V > 0) {
        CUDA_TRY(cudaMemcpyAsync(L->verts, verts, sizeof(double2) * (size_t)V, cudaMemcpyDeviceToDevice, s));
        CUDA_TRY(launch_check_finite(L->verts, (int)V, dbad, s));
    }
    int bad = 0;
    st = read_flag(dbad, s, &bad);
    if (st != SJ_OK) return st;
    if (bad) return fail(SJ_ERR_INVALID, "invalid polyline layer (offsets or non-finite vertex)");
    CUDA_TRY(dalloc(&L->vsplit, (size_t)V));
    CUDA_TRY(dalloc(&L->seg_e64, (size_t)V));
    CUDA_TRY(dalloc(&L->seg_inv64, (size_t)V));
    CUDA_TRY(dalloc(&L->seg32, (size_t)V));
    if (V > 0) {
        CUDA_TRY(launch_split(L->verts, (int)V, L->vsplit, s));
        CUDA_TRY(launch_seg_table(L->verts, L->obj_voff, Lc, (int)V, L->seg_e64, L->seg_inv64, L->seg32, s));
    }
    CUDA_TRY(dalloc(&L->stats, ST_N));
    CUDA_TRY(cudaMemsetAsync(L->stats, 0, sizeof(unsigned long long) * ST_N, s));
    st = build_candidates(L, dbad, s);
    if (st != SJ_OK) return st;
    st = build_seg_lists(L, s);
    if (st != SJ_OK) return st;
    *out = L;
    guard.L = nullptr;
    return SJ_OK;
}

extern "C" sj_status sj_layer_destroy(sj_layer *L) {
    if (!L) return SJ_OK;
    cudaDeviceSynchronize();
    layer_free(L);
    return SJ_OK;
}

extern "C" sj_status sj_layer_get_info(const sj_layer *L, sj_layer_info *out) {
    if (!L || !out) return fail(SJ_ERR_INVALID, "NULL argument");
    out->kind = L->kind;
    out->n_objects = L->nobj;
    out->n_vertices = L->V;
    out->n_rings = L->R;
    out->n_cells = L->g.G;
    out->n_candidates = L->M;
    out->D = L->D;
    return SJ_OK;
}

extern "C" sj_status sj_layer_get_candidates(const sj_layer *L, int32_t *cand_start, int32_t *cand_ids) {
    if (!L || !cand_start || (!cand_ids && L->M > 0)) return fail(SJ_ERR_INVALID, "NULL argument");
    CUDA_TRY(cudaMemcpy(cand_start, L->cand_start, sizeof(int) * ((size_t)L->g.G + 1), cudaMemcpyDeviceToHost));
    if (L->M > 0) CUDA_TRY(cudaMemcpy(cand_ids, L->cand_ids, sizeof(int) * (size_t)L->M, cudaMemcpyDeviceToHost));
    return SJ_OK;
}

extern "C" sj_status sj_layer_get_stats(const sj_layer *L, sj_run_stats *out) {
    if (!L || !out) return fail(SJ_ERR_INVALID, "NULL argument");
    unsigned long long h[ST_N];
    CUDA_TRY(cudaDeviceSynchronize());
    CUDA_TRY(cudaMemcpy(h, L->stats, sizeof(h), cudaMemcpyDeviceToHost));
    resolve_events(L);
    out->refine_launches = L->refine_launches;
    out->refine_ms = L->refine_ms;
    out->joins = L->joins.load();
    out->points = L->points.load();
    out->items = (int64_t)h[ST_ITEMS];
    out->pairs = (int64_t)h[ST_PAIRS];
    out->edge_tests = (int64_t)h[ST_TESTS];
    out->fallbacks = (int64_t)h[ST_FALLBACK];
    out->hits = (int64_t)h[ST_HITS];
    out->algo_tests = (int64_t)h[ST_ALGO];
    out->resolved = (int64_t)h[ST_RESOLVED];
    out->census_tests = L->census_tests.load();
    out->census_straddles = L->census_straddles.load();
    return SJ_OK;
}

extern "C" sj_status sj_layer_reset_stats(sj_layer *L) {
    if (!L) return fail(SJ_ERR_INVALID, "NULL argument");
    CUDA_TRY(cudaDeviceSynchronize());
    CUDA_TRY(cudaMemset(L->stats, 0, sizeof(unsigned long long) * ST_N));
    resolve_events(L);
    L->refine_ms = 0.0;
    L->refine_launches = 0;
    L->joins = 0;
    L->points = 0;
    L->census_tests = 0;
    L->census_straddles = 0;
    return SJ_OK;
}

// ------------------------------------------------------------------ joins

struct JoinBufs {
    int *cnt, *cell_start, *perm, *totals, *pos, *cell_base, *sub_start;
    int2 *key_rank, *items, *block_sums, *fb;
};

// Scratch of a P2P join.  The slots' result records take the place of key_rank,
// which the scatter has used up (P2PRec has its size).  to_input: with the
// slot of each input point (pos), for outputs written in input order.
// ch_min: the smallest work item (cell_chunk's floor when items are split by
// edge budget, else ch).
static void carve(Scratch &s, JoinBufs &b, int64_t N, int G, int ch, bool to_input, int lS = 0, int ch_min = 0) {
    size_t max_items = (size_t)(N / (ch_min > 0 ? ch_min : ch)) + (size_t)std::min<int64_t>(G, N) + 1;
    b.cnt = s.take<int>(((size_t)G << lS) + 1);
    b.sub_start = lS ? s.take<int>((size_t)G << lS) : nullptr;
    b.cell_start = s.take<int>((size_t)G + 1);
    b.totals = s.take<int>(4);
    b.key_rank = s.take<int2>((size_t)N);
    b.perm = s.take<int>((size_t)N);
    b.items = s.take<int2>(max_items);
    b.block_sums = s.take<int2>(bucket_scan_blocks(G));
    b.fb = s.take<int2>((size_t)N);
    b.pos = to_input ? s.take<int>((size_t)N) : nullptr;
    b.cell_base = to_input ? s.take<int>((size_t)G) : nullptr;
}
static_assert(sizeof(P2PRec) == sizeof(int2), "");

// CUDA events around the launches of a span (SJ_FLAG_TIME_REFINE), kept with the
// layer once recorded; an error sets e.
struct TimedSpan {
    const sj_layer *L;
    cudaStream_t s;
    cudaEvent_t ev0 = nullptr, ev1 = nullptr;
    TimedSpan(const sj_layer *layer, bool on, cudaStream_t stream, cudaError_t &e) : L(layer), s(stream) {
        if (!on || e != cudaSuccess) return;
        e = cudaEventCreate(&ev0);
        if (e == cudaSuccess) e = cudaEventCreate(&ev1);
        if (e == cudaSuccess) e = cudaEventRecord(ev0, s);
    }
    void stop(cudaError_t &e) {
        if (!ev1) return;
        if (e == cudaSuccess) e = cudaEventRecord(ev1, s);
        std::lock_guard<std::mutex> lk(L->ev_mu);
        L->ev_pending.emplace_back(ev0, ev1);
    }
};

static DirectArgs direct_args(const sj_layer *L, int32_t *out_id, double *out_d) {
    DirectArgs g{};
    g.cand_start = L->cand_start;
    g.cell_algo = L->cell_algo;
    // a point lies within its cell, the cell's FP32 frame origin within u xmax of
    // its corner, and the coordinate's own rounding adds 2u of it
    g.cell_mag = float_up((std::max(L->g.cw, L->g.ch) + 1.2e-7 * L->xmax) * (1.0 + 1e-6));
    g.out_id = out_id;
    g.out_d = out_d;
    return g;
}

// window < 0: the layer's D; else a P2P window 0 <= window <= D for this call
// alone (the layer's lists, built for D, hold every segment within any smaller
// window, so the same kernels apply with the window's thresholds).
static sj_status join_impl(const sj_layer *L, int kind, const double *pts, int64_t N, int32_t *out_id, double *out_d,
                           const sj_opts *o, void *stream, double window = -1.0) {
    if (!L) return fail(SJ_ERR_INVALID, "layer is NULL");
    if (L->kind != kind) return fail(SJ_ERR_INVALID, kind == KIND_PIP ? "not a polygon layer" : "not a polyline layer");
    if (window >= 0.0 && !(window <= L->D)) return fail(SJ_ERR_INVALID, "window must lie in [0, layer D]");
    if (N < 0 || N > MAX_COUNT) return fail(SJ_ERR_INVALID, "N out of range (at most 2^31 - 2^22)");
    if (N > 0 && (!pts || !out_id)) return fail(SJ_ERR_INVALID, "NULL buffer");
    if (N > 0 && !aligned16(pts)) return fail(SJ_ERR_INVALID, "pts not 16-byte aligned");
    int form = o ? o->form : SJ_FP64;
    if (form != SJ_FP64 && form != SJ_FP32X) return fail(SJ_ERR_INVALID, "unknown form");
    int launch = o ? o->launch : SJ_PER_REQUEST;
    if (launch != SJ_PER_REQUEST && launch != SJ_PERSISTENT) return fail(SJ_ERR_INVALID, "unknown launch form");
    if (form == SJ_FP32X && L->xmax > 1e30)
        return fail(SJ_ERR_INVALID, "SJ_FP32X needs grid coordinates below 1e30 in magnitude; use SJ_FP64");
    int ch = (o && o->pts_per_item) ? o->pts_per_item : 128;
    if (ch < 1 || ch > MAX_CH) return fail(SJ_ERR_INVALID, "pts_per_item must be in 1..128");
    const int nw = (o && o->block) ? o->block : 4;
    if (nw != 2 && nw != 4 && nw != 8) return fail(SJ_ERR_INVALID, "block must be 0, 2, 4 or 8 (warps per block)");
    int budget = o ? o->edges_per_chunk : 0;
    if (budget < 0) return fail(SJ_ERR_INVALID, "edges_per_chunk must be >= 0");
    // default: no split (no setting was faster on the walks)
    int dev = 0;
    CUDA_TRY(cudaGetDevice(&dev));
    if (dev != L->device) return fail(SJ_ERR_INVALID, "layer belongs to another device");
    DevInfo *di;
    sj_status st = device_info(dev, &di);
    if (st != SJ_OK) return st;
    L->joins++;
    L->points += N;
    if (N == 0) return SJ_OK;
    cudaStream_t s = (cudaStream_t)stream;
    const bool timed = o && (o->flags & SJ_FLAG_TIME_REFINE);
    const bool subcells = o && (o->flags & SJ_FLAG_SUBCELL_ON) && !(o->flags & SJ_FLAG_SUBCELL_OFF);
    if (kind == KIND_PIP) {   // one kernel over the points in input order (sj_pip.cu)
        PipArgs pa = pip_args(L);
        if (subcells) pa.search = PIP_SEARCH_MIN;
        cudaError_t e = cudaSuccess;
        unsigned *lists = nullptr;
        const size_t nl = (size_t)pip_list_ints(N, di->sms);
        if (nl) CUDA_TRY(dev_malloc_async((void **)&lists, sizeof(unsigned) * nl, s));
        TimedSpan span(L, timed, s, e);
        if (e == cudaSuccess) e = launch_pip_join(pa, (const double2 *)pts, (int)N, out_id, lists, di->sms, s);
        span.stop(e);
        if (lists) {
            cudaError_t e2 = cudaFreeAsync(lists, s);
            if (e == cudaSuccess) e = e2;
        }
        if (e != cudaSuccess) return cuda_fail(e, "join launch");
        return check_bounds(s);
    }
    RefineArgs ra{};
    fill_refine(L, ra);
    if (window >= 0.0) {
        ra.D = window;
        ra.Df = (float)window;
        ra.Ddn = float_down(window * (1.0 - 1e-12));
        ra.Dup = float_up(window * (1.0 + 1e-12) + 1e-300);
    }
    ra.pts = (const double2 *)pts;
    ra.npts = (int)N;
    // Few points: no bucketing (see k_p2p_direct).  Calls that shape their work
    // items or order their points keep the path that has them.
    // The line is by points alone: list lengths do not move it (measured there) but
    // for points that crowd into a small part of a cell with a long list, where an
    // item drops the segments far from its points.  60,000 walks on 16 x 16 cells
    // (lists of some 5,000 segments), all points within 100 m, us bucketed / direct:
    // FP32X 5,000 points 82 / 83, 32,000 197 / 327, FP64 131,000 312 / 1,262.  As many
    // points spread over the cells take 813 / 157, 1,464 / 586 and 3,577 / 1,694, and
    // no rule on sizes tells the two apart.  With lists of some 1,000 (32 x 32 cells)
    // crowded points draw at 20,000 to 32,000 points (FP64 73 / 71, FP32X 110 / 103).
    if (N <= (form == SJ_FP32X ? P2P_DIRECT_FP32X : P2P_DIRECT_FP64) && !(o && o->pts_per_item) && budget == 0 &&
        !subcells) {
        cudaError_t e = cudaSuccess;
        if (form == SJ_FP64) CUDA_TRY(dev_malloc_async((void **)&ra.rec, sizeof(P2PRec) * (size_t)N, s));
        TimedSpan span(L, timed, s, e);
        if (e == cudaSuccess) e = launch_p2p_direct(ra, direct_args(L, out_id, out_d), form, (int)N, di->sms, s);
        span.stop(e);
        if (form == SJ_FP64) {
            if (e == cudaSuccess) e = launch_p2p_finish(ra, form, nullptr, (int)N, out_id, out_d, s);
            cudaError_t e2 = cudaFreeAsync(ra.rec, s);
            if (e == cudaSuccess) e = e2;
        }
        if (e != cudaSuccess) return cuda_fail(e, "join launch");
        return check_bounds(s);
    }
    const int G = L->g.G;
    // Sub-cell order of the points inside their cells (see BucketArgs), on
    // request (SJ_FLAG_SUBCELL_ON): each work item of a dense cell then covers
    // a compact part of it and the exact per-item prune (the box distance)
    // drops more of the staged segments -- 40 % fewer tests at 170 M points --
    // but the per-sub-cell start table (G x S entries, read at random by the
    // scatter) costs more than that saves on the workloads measured, so
    // arrival order is the default.  4 x 4 sub-cells in Z-order.
    int sub_lx = subcells ? 2 : 0, sub_ly = sub_lx;
    if (((long long)G << (sub_lx + sub_ly)) > MAX_COUNT) sub_lx = sub_ly = 0;
    const int lS = sub_lx + sub_ly;

    JoinBufs b;
    const bool split = budget > 0;   // items sized by the cells' edge work
    const int ch_min = split ? std::min(ch, 8) : ch;
    size_t bytes = measure([&](Scratch &sc) { carve(sc, b, N, G, ch, true, lS, ch_min); });
    Scratch sc;
    CUDA_TRY(dev_malloc_async((void **)&sc.base, bytes, s));
    carve(sc, b, N, G, ch, true, lS, ch_min);
    cudaError_t e = cudaMemsetAsync(b.cnt, 0, sizeof(int) * (((size_t)G << lS) + 1), s);
    if (e == cudaSuccess) e = cudaMemsetAsync(b.totals, 0, sizeof(int) * 4, s);

    BucketArgs ba{};
    ba.g = L->g;
    ba.pts = (const double2 *)pts;
    ba.n = (int)N;
    ba.cnt = b.cnt;
    ba.key_rank = b.key_rank;
    ba.cell_start = b.cell_start;
    ba.perm = b.perm;
    ba.cand_start = L->cand_start;
    ba.cell_algo = L->cell_algo;
    ba.stats = L->stats;
    ba.ch = ch;
    ba.cell_work = split ? L->cell_work : nullptr;
    ba.budget = split ? budget : 0;
    ba.items = b.items;
    ba.block_sums = b.block_sums;
    ba.bs_cap = bucket_scan_blocks(G);
    ba.totals = b.totals;
    ba.pos = b.pos;
    ba.cell_base = b.cell_base;
    ba.sub_lx = sub_lx;
    ba.sub_ly = sub_ly;
    ba.sub_start = b.sub_start;
    if (e == cudaSuccess) e = launch_bucket(ba, s);

    ra.items = b.items;
    ra.n_items = b.totals + 1;
    ra.work_next = b.totals + 3;   // zeroed with the totals at the start of the join
    // Items a warp takes per counter update.  On dense grids (two or more
    // items per cell on average): two consecutive items, mostly two chunks of
    // one cell, whose second reads the cell's records from L1 and halves the
    // counter traffic (170 M points, 512^2 grid, D = 50 m: refine 5.35 ->
    // 4.21 ms; D = 100 m unchanged); sparse grids keep one (the 10 M point
    // join is 1 % slower with two).
    ra.claim = (N >= 2LL * ch * (long long)G) ? 2 : 1;
    ra.cell_start = b.cell_start;
    ra.perm = b.perm;
    ra.ch = ch;
    ra.cell_work = ba.cell_work;
    ra.budget = ba.budget;
    ra.rec = reinterpret_cast<P2PRec *>(b.key_rank);   // every slot of a refined cell written
    ra.fb = b.fb;
    ra.n_fb = b.totals + 2;
    TimedSpan span(L, timed, s, e);   // the refinement launch alone
    if (e == cudaSuccess) e = launch_p2p_refine(ra, form, nw, di->sms * di->p2p_bps[form], s);
    span.stop(e);
    if (e == cudaSuccess) e = launch_p2p_recheck(ra, form, di->sms * 4, s);
    if (e == cudaSuccess) e = launch_p2p_finish(ra, form, b.pos, (int)N, out_id, out_d, s);   // a8
    cudaError_t e2 = cudaFreeAsync(sc.base, s);
    if (e != cudaSuccess) return cuda_fail(e, "join launch");
    if (e2 != cudaSuccess) return cuda_fail(e2, "cudaFreeAsync");
    return check_bounds(s);
}

extern "C" sj_status sj_pip_join(const sj_layer *L, const double *pts, int64_t N, int32_t *out_id, const sj_opts *o,
                                 void *stream) {
    return join_impl(L, KIND_PIP, pts, N, out_id, nullptr, o, stream);
}

extern "C" sj_status sj_p2p_join(const sj_layer *L, const double *pts, int64_t N, int32_t *out_id, double *out_d,
                                 const sj_opts *o, void *stream) {
    return join_impl(L, KIND_P2P, pts, N, out_id, out_d, o, stream);
}

extern "C" sj_status sj_p2p_join_window(const sj_layer *L, const double *pts, int64_t N, double window,
                                        int32_t *out_id, double *out_d, const sj_opts *o, void *stream) {
    if (!(window >= 0.0)) return fail(SJ_ERR_INVALID, "window must lie in [0, layer D]");   // NaN too
    return join_impl(L, KIND_P2P, pts, N, out_id, out_d, o, stream, window);
}

// Host-buffer join, pipelined in three stages on library streams: chunks of
// the points are copied in on one stream, joined on a second (each waiting for
// its chunk's copy) and their results copied out on a third (each waiting for
// its chunk's join), so that copies in, joins and copies out of different
// chunks overlap (both copy directions and the SMs work at once).  Each chunk
// is an independent join (a point's result does not depend on the other
// points), so the outputs equal those of one join over all N points.  P2P: at most
// three chunks: every chunk is a full join with fixed costs (scans over every
// cell, sparser work items), so four quarter joins were measured slower.  PIP:
// a join costs its points and a launch, so chunks of about HOST_PIP_CHUNK points
// keep the first join's wait and the last copy out short (5 M points: 585 us with
// two chunks, 535 / 517 / 526 with chunks of 0.5 / 1 / 2 M).
constexpr int64_t HOST_PIP_CHUNK = 1 << 20, HOST_MAX_CHUNKS = 16;
static sj_status join_host(const sj_layer *L, int kind, const double *pts, int64_t N, int32_t *out_id, double *out_d,
                           const sj_opts *o, void *stream, double window = -1.0) {
    if (N < 0 || N > MAX_COUNT) return fail(SJ_ERR_INVALID, "N out of range (at most 2^31 - 2^22)");
    if (N > 0 && (!pts || !out_id)) return fail(SJ_ERR_INVALID, "NULL buffer");
    if (!L) return fail(SJ_ERR_INVALID, "layer is NULL");
    cudaStream_t s = (cudaStream_t)stream;
    if (N == 0) return join_impl(L, kind, nullptr, 0, nullptr, nullptr, o, stream, window);
    int dev = 0;
    CUDA_TRY(cudaGetDevice(&dev));
    DevInfo *di;
    sj_status st = device_info(dev, &di);
    if (st != SJ_OK) return st;
    cudaStream_t t_in = di->hstream[0], t_cmp = di->hstream[1], t_out = di->hstream[2];
    // chunk bounds, P2P: one chunk up to 2 M points, halves up to 8 M, else quarter /
    // half / quarter (a short first chunk starts the joins early, a short last
    // one keeps the final copy out short)
    int64_t bound[HOST_MAX_CHUNKS + 1] = {0, N, N, N};
    int nchunks = 1;
    if (kind == KIND_PIP) {
        nchunks = (int)std::min<int64_t>(HOST_MAX_CHUNKS, (N + HOST_PIP_CHUNK - 1) / HOST_PIP_CHUNK);
        // equal chunks of an even number of points (the device results of each
        // start aligned)
        const int64_t size = ((N + nchunks - 1) / nchunks + 63) & ~(int64_t)63;
        for (int c = 1; c <= nchunks; ++c) bound[c] = std::min(N, size * c);
    } else if (N > (int64_t)8 << 20) {
        bound[1] = N / 4;
        bound[2] = N - N / 4;
        nchunks = 3;
    } else if (N > (int64_t)2 << 20) {
        bound[1] = N / 2;
        nchunks = 2;
    }
    char *d = nullptr;
    size_t bp = (size_t)N * 16, bi = ((size_t)N * 4 + 255) & ~(size_t)255, bd = out_d ? (size_t)N * 8 : 0;
    CUDA_TRY(dev_malloc_async((void **)&d, bp + bi + bd, s));
    double *dp = (double *)d;
    int32_t *dI = (int32_t *)(d + bp);
    double *dD = out_d ? (double *)(d + bp + bi) : nullptr;
    std::vector<cudaEvent_t> evs(2 * (size_t)nchunks + 3, nullptr);
    cudaError_t e = cudaSuccess;
    for (auto &ev : evs)
        if (e == cudaSuccess) e = cudaEventCreateWithFlags(&ev, cudaEventDisableTiming);
    cudaEvent_t ev_start = evs[0], ev_done = evs[1];
    // every stage starts after the caller's stream (its prior work and the allocation)
    if (e == cudaSuccess) e = cudaEventRecord(ev_start, s);
    for (cudaStream_t t : {t_in, t_cmp, t_out})
        if (e == cudaSuccess) e = cudaStreamWaitEvent(t, ev_start, 0);
    for (int c = 0; c < nchunks && e == cudaSuccess && st == SJ_OK; ++c) {
        cudaEvent_t copied = evs[2 + 2 * c], joined = evs[3 + 2 * c];
        const int64_t off = bound[c], n = bound[c + 1] - off;
        if (n == 0) continue;
        e = cudaMemcpyAsync(dp + 2 * off, pts + 2 * off, (size_t)n * 16, cudaMemcpyHostToDevice, t_in);
        if (e == cudaSuccess) e = cudaEventRecord(copied, t_in);
        if (e == cudaSuccess) e = cudaStreamWaitEvent(t_cmp, copied, 0);
        if (e != cudaSuccess) break;
        st = join_impl(L, kind, dp + 2 * off, n, dI + off, dD ? dD + off : nullptr, o, t_cmp, window);
        if (st != SJ_OK) break;
        e = cudaEventRecord(joined, t_cmp);
        if (e == cudaSuccess) e = cudaStreamWaitEvent(t_out, joined, 0);
        if (e == cudaSuccess) e = cudaMemcpyAsync(out_id + off, dI + off, (size_t)n * 4, cudaMemcpyDeviceToHost, t_out);
        if (e == cudaSuccess && out_d)
            e = cudaMemcpyAsync(out_d + off, dD + off, (size_t)n * 8, cudaMemcpyDeviceToHost, t_out);
    }
    // the caller's stream waits for the join and copy-out stages (the copy-in
    // stage is behind both), then frees the buffer
    cudaError_t e2 = cudaEventRecord(ev_done, t_out);
    if (e2 == cudaSuccess) e2 = cudaStreamWaitEvent(s, ev_done, 0);
    if (e2 == cudaSuccess) e2 = cudaEventRecord(evs.back(), t_cmp);
    if (e2 == cudaSuccess) e2 = cudaStreamWaitEvent(s, evs.back(), 0);
    cudaFreeAsync(d, s);
    cudaError_t e3 = cudaStreamSynchronize(s);
    for (cudaEvent_t ev : evs)
        if (ev) cudaEventDestroy(ev);
    if (st != SJ_OK) return st;
    if (e != cudaSuccess) return cuda_fail(e, "host join copy");
    if (e2 != cudaSuccess) return cuda_fail(e2, "host join streams");
    if (e3 != cudaSuccess) return cuda_fail(e3, "cudaStreamSynchronize");
    return SJ_OK;
}

extern "C" sj_status sj_pip_join_host(const sj_layer *L, const double *pts, int64_t N, int32_t *out_id,
                                      const sj_opts *o, void *stream) {
    return join_host(L, KIND_PIP, pts, N, out_id, nullptr, o, stream);
}

extern "C" sj_status sj_p2p_join_host(const sj_layer *L, const double *pts, int64_t N, int32_t *out_id, double *out_d,
                                      const sj_opts *o, void *stream) {
    return join_host(L, KIND_P2P, pts, N, out_id, out_d, o, stream);
}

extern "C" sj_status sj_p2p_join_window_host(const sj_layer *L, const double *pts, int64_t N, double window,
                                             int32_t *out_id, double *out_d, const sj_opts *o, void *stream) {
    if (!(window >= 0.0)) return fail(SJ_ERR_INVALID, "window must lie in [0, layer D]");   // NaN too
    if (L && L->kind == KIND_P2P && !(window <= L->D)) return fail(SJ_ERR_INVALID, "window must lie in [0, layer D]");
    return join_host(L, KIND_P2P, pts, N, out_id, out_d, o, stream, window);
}

extern "C" sj_status sj_bucket_points(const double *pts, int64_t N, const sj_grid *g, int32_t *cell_start, int32_t *perm,
                                      void *stream) {
    if (!grid_ok(g)) return fail(SJ_ERR_INVALID, "invalid grid");
    if (N < 0 || N > MAX_COUNT) return fail(SJ_ERR_INVALID, "N out of range (at most 2^31 - 2^22)");
    if (!cell_start || (N > 0 && (!pts || !perm))) return fail(SJ_ERR_INVALID, "NULL buffer");
    if (N > 0 && !aligned16(pts)) return fail(SJ_ERR_INVALID, "pts not 16-byte aligned");
    cudaStream_t s = (cudaStream_t)stream;
    GridDev gd = make_grid(g);
    Scratch sc;
    auto lay = [&](Scratch &x, int **cnt, int **totals, int2 **kr, int2 **bs, unsigned long long **keys) {
        *cnt = x.take<int>((size_t)gd.G + 1);
        *totals = x.take<int>(4);
        *kr = x.take<int2>((size_t)N);
        *bs = x.take<int2>(bucket_scan_blocks(gd.G));
        *keys = x.take<unsigned long long>((size_t)gd.nx + gd.ny + 2);
    };
    int *cnt, *totals;
    int2 *kr, *bs;
    unsigned long long *keys;
    size_t bytes = measure([&](Scratch &x) { lay(x, &cnt, &totals, &kr, &bs, &keys); });
    CUDA_TRY(dev_malloc_async((void **)&sc.base, bytes, s));
    lay(sc, &cnt, &totals, &kr, &bs, &keys);
    gd.kx = keys;
    gd.ky = keys + gd.nx + 1;
    BucketArgs ba{};
    ba.g = gd;
    ba.pts = (const double2 *)pts;
    ba.n = (int)N;
    ba.cnt = cnt;
    ba.key_rank = kr;
    ba.cell_start = cell_start;
    ba.perm = perm;
    ba.block_sums = bs;
    ba.bs_cap = bucket_scan_blocks(gd.G);
    ba.totals = totals;
    ba.ch = 1;
    cudaError_t e = cudaMemsetAsync(cnt, 0, sizeof(int) * ((size_t)gd.G + 1), s);
    if (e == cudaSuccess) e = launch_thresholds(gd, keys, keys + gd.nx + 1, s);
    if (e == cudaSuccess) e = launch_bucket(ba, s);
    cudaError_t e2 = cudaFreeAsync(sc.base, s);
    if (e != cudaSuccess) return cuda_fail(e, "bucket launch");
    if (e2 != cudaSuccess) return cuda_fail(e2, "cudaFreeAsync");
    return SJ_OK;
}

extern "C" sj_status sj_pip_census(const sj_layer *L, const double *pts, int64_t N, int64_t *out, void *stream) {
    if (!L || !out) return fail(SJ_ERR_INVALID, "NULL argument");
    if (L->kind != KIND_PIP) return fail(SJ_ERR_INVALID, "not a polygon layer");
    if (N < 0 || N > MAX_COUNT) return fail(SJ_ERR_INVALID, "N out of range (at most 2^31 - 2^22)");
    if (N > 0 && (!pts || !aligned16(pts))) return fail(SJ_ERR_INVALID, "pts NULL or not 16-byte aligned");
    out[0] = out[1] = 0;
    if (N == 0) return SJ_OK;
    cudaStream_t s = (cudaStream_t)stream;
    unsigned long long *d = nullptr, h[2] = {0, 0};
    CUDA_TRY(dev_malloc_async((void **)&d, sizeof(h), s));
    CensusArgs ca{L->g,          L->cand_start, L->cand_ids,  L->obj_voff, L->prow_base,
                  L->prow_r0,    L->prow_start, L->pedge_ids, L->nxt,      L->verts};
    cudaError_t e = cudaMemsetAsync(d, 0, sizeof(h), s);
    if (e == cudaSuccess) e = launch_pip_census(ca, (const double2 *)pts, (int)N, d, s);
    if (e == cudaSuccess) e = cudaMemcpyAsync(h, d, sizeof(h), cudaMemcpyDeviceToHost, s);
    cudaError_t e2 = cudaFreeAsync(d, s);
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);
    if (e != cudaSuccess) return cuda_fail(e, "census");
    if (e2 != cudaSuccess) return cuda_fail(e2, "cudaFreeAsync");
    out[0] = (int64_t)h[0];
    out[1] = (int64_t)h[1];
    L->census_tests += out[0];
    L->census_straddles += out[1];
    return SJ_OK;
}

extern "C" const char *sj_last_error(void) { return g_err.c_str(); }

extern "C" const char *sj_version(void) { return "sj 0.1 (sm_103a)"; }

// ------------------------------------------------------------------ P2P join without allocation
//
// Some callers cannot allocate device memory at the moment they join: code on
// a hard latency budget (a device allocation can stall for milliseconds),
// code that runs inside a pre-sized memory arena or a fixed memory budget, and
// hosts where another component owns the CUDA allocator and forbids
// allocations from libraries.  sj_p2p_join_noalloc runs the same kernels as
// sj_p2p_join but takes all of its scratch from one file-scope device array
// of fixed size, so it calls no allocator at all.
//
// The array is part of this module's device image: every GPU that loads the
// module holds it until the process exits.  All calls share it, so two calls
// whose kernels overlap on the GPU race on it; callers must serialise them
// (one stream, or events between streams).  It keeps the previous call's
// contents, so the counters that must start at zero are cleared on the
// caller's stream at the start of every call.

namespace {

constexpr int64_t NOALLOC_MAX_POINTS = SJ_NOALLOC_MAX_POINTS;
constexpr int64_t NOALLOC_MAX_CELLS = SJ_NOALLOC_MAX_CELLS;
constexpr int NOALLOC_CH = 64;
constexpr size_t NOALLOC_BYTES = 32u << 20;   // holds carve() at the two limits above (about 27 MB)

__device__ __align__(256) unsigned char g_noalloc_scratch[NOALLOC_BYTES];

void *g_noalloc_ptr[64];
std::mutex g_noalloc_mu;

// Device address of the array on the current device, looked up once per
// device (host code cannot use the symbol itself: on the host it names a
// stand-in, not device memory).
sj_status noalloc_scratch(int dev, char **out) {
    std::lock_guard<std::mutex> lk(g_noalloc_mu);
    if (!g_noalloc_ptr[dev]) {
        void *p = nullptr;
        cudaError_t e = cudaGetSymbolAddress(&p, g_noalloc_scratch);
        if (e != cudaSuccess) return cuda_fail(e, "cudaGetSymbolAddress(noalloc scratch)");
        g_noalloc_ptr[dev] = p;
    }
    *out = (char *)g_noalloc_ptr[dev];
    return SJ_OK;
}

}  // namespace

extern "C" sj_status sj_p2p_join_noalloc(const sj_layer *L, const double *pts, int64_t N, int32_t *out_id,
                                         double *out_d, const sj_opts *o, void *stream) {
    if (!L) return fail(SJ_ERR_INVALID, "layer is NULL");
    if (L->kind != KIND_P2P) return fail(SJ_ERR_INVALID, "not a polyline layer");
    if (N < 0 || N > NOALLOC_MAX_POINTS)
        return fail(SJ_ERR_INVALID, "sj_p2p_join_noalloc: N must be in 0.." + std::to_string(NOALLOC_MAX_POINTS) +
                                        " (fixed scratch size); use sj_p2p_join for larger batches");
    if ((int64_t)L->g.G > NOALLOC_MAX_CELLS)
        return fail(SJ_ERR_INVALID, "sj_p2p_join_noalloc: the layer's grid has more than " +
                                        std::to_string(NOALLOC_MAX_CELLS) + " cells (fixed scratch size)");
    if (N > 0 && (!pts || !out_id)) return fail(SJ_ERR_INVALID, "NULL buffer");
    if (N > 0 && !aligned16(pts)) return fail(SJ_ERR_INVALID, "pts not 16-byte aligned");
    const int form = o ? o->form : SJ_FP64;
    if (form != SJ_FP64 && form != SJ_FP32X) return fail(SJ_ERR_INVALID, "unknown form");
    if (form == SJ_FP32X && L->xmax > 1e30)
        return fail(SJ_ERR_INVALID, "SJ_FP32X needs grid coordinates below 1e30 in magnitude; use SJ_FP64");
    int dev = 0;
    CUDA_TRY(cudaGetDevice(&dev));
    if (dev != L->device) return fail(SJ_ERR_INVALID, "layer belongs to another device");
    if (dev < 0 || dev >= 64) return fail(SJ_ERR_INVALID, "device index out of range");
    DevInfo *di;
    sj_status st = device_info(dev, &di);
    if (st != SJ_OK) return st;
    char *base = nullptr;
    st = noalloc_scratch(dev, &base);
    if (st != SJ_OK) return st;
    L->joins++;
    L->points += N;
    if (N == 0) return SJ_OK;
    cudaStream_t s = (cudaStream_t)stream;
    const int G = L->g.G;
    if (N <= (form == SJ_FP32X ? P2P_DIRECT_FP32X : P2P_DIRECT_FP64)) {   // as join_impl
        RefineArgs ra{};
        fill_refine(L, ra);
        ra.pts = (const double2 *)pts;
        ra.npts = (int)N;
        ra.rec = reinterpret_cast<P2PRec *>(base);
        CUDA_TRY(launch_p2p_direct(ra, direct_args(L, out_id, out_d), form, (int)N, di->sms, s));
        if (form == SJ_FP64) CUDA_TRY(launch_p2p_finish(ra, form, nullptr, (int)N, out_id, out_d, s));
        return check_bounds(s);
    }
    JoinBufs b;
    size_t bytes = measure([&](Scratch &sc) { carve(sc, b, N, G, NOALLOC_CH, false); });
    if (bytes > NOALLOC_BYTES) return fail(SJ_ERR_INVALID, "sj_p2p_join_noalloc: scratch does not fit");
    Scratch sc;
    sc.base = base;
    carve(sc, b, N, G, NOALLOC_CH, false);
    CUDA_TRY(cudaMemsetAsync(b.cnt, 0, sizeof(int) * ((size_t)G + 1), s));
    CUDA_TRY(cudaMemsetAsync(b.totals, 0, sizeof(int) * 4, s));

    BucketArgs ba{};
    ba.g = L->g;
    ba.pts = (const double2 *)pts;
    ba.n = (int)N;
    ba.cnt = b.cnt;
    ba.key_rank = b.key_rank;
    ba.cell_start = b.cell_start;
    ba.perm = b.perm;
    ba.cand_start = L->cand_start;
    ba.cell_algo = L->cell_algo;
    ba.stats = L->stats;
    ba.ch = NOALLOC_CH;
    ba.items = b.items;
    ba.block_sums = b.block_sums;
    ba.bs_cap = bucket_scan_blocks(G);
    ba.totals = b.totals;
    ba.out_id = out_id;
    ba.out_d = out_d;
    CUDA_TRY(launch_bucket(ba, s));
    // slots of cells without candidates are not refined: no polyline
    CUDA_TRY(cudaMemsetAsync(b.key_rank, 0xff, sizeof(int2) * (size_t)N, s));

    RefineArgs ra{};
    fill_refine(L, ra);
    ra.items = b.items;
    ra.n_items = b.totals + 1;
    ra.cell_start = b.cell_start;
    ra.perm = b.perm;
    ra.pts = (const double2 *)pts;
    ra.ch = NOALLOC_CH;
    ra.npts = (int)N;
    ra.rec = reinterpret_cast<P2PRec *>(b.key_rank);
    ra.fb = b.fb;
    ra.n_fb = b.totals + 2;
    // items from the device counter, as in join_impl (totals[3], zeroed above)
    ra.work_next = b.totals + 3;
    ra.claim = (N >= 2LL * NOALLOC_CH * (long long)G) ? 2 : 1;
    CUDA_TRY(launch_p2p_refine(ra, form, 4, di->sms * di->p2p_bps[form], s));
    CUDA_TRY(launch_p2p_recheck(ra, form, di->sms * 4, s));
    CUDA_TRY(launch_p2p_finish_slots(ra, form, b.totals, (int)N, out_id, out_d, s));
    return check_bounds(s);
}

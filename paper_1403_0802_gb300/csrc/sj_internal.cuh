// sj_internal.cuh -- device-side building blocks shared by the CUDA
// translation units of libsj.so (not part of the public ABI).
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "sj.h"

namespace sj {

constexpr unsigned FULL = 0xffffffffu;
constexpr int MAX_CH = 128;        // largest point chunk per work item
// Largest element count of any array the kernels index with 32-bit ints
// (points, vertices, candidate and list entries): every grid-stride loop with
// a 32-bit index advances by at most 2^22 (grids are capped below that), so an
// index i < MAX_COUNT never passes 2^31 - 1 when it advances; loops with a
// larger step (the unrolled bucketing and finishing kernels) count in unsigned 32 or 64 bits.
constexpr long long MAX_COUNT = (1LL << 31) - (1LL << 22);
constexpr float U32 = 5.9604644775390625e-08f;   // 2^-24, unit roundoff of FP32

// Grid with derived cell sizes (computed once on the host, FP64, rounded) and
// the per-axis threshold tables of point_cell.
struct GridDev {
    double x0, y0, x1, y1;
    double cw, ch;     // (x1 - x0) / nx, (y1 - y0) / ny
    int nx, ny, G;
    const unsigned long long *kx;   // [nx + 1] order keys of the x thresholds
    const unsigned long long *ky;   // [ny + 1]
    float x0f, y0f, icwf, ichf;     // FP32 estimates of x0, y0, 1 / cw, 1 / ch
    float tolx, toly;               // bounds of the error of axis_estimate, in cells
};

// Cell of one coordinate: floor((v - lo) / w) as a double (may be out of range
// or NaN).  Every operation is a single IEEE round-to-nearest step.
__device__ __forceinline__ double axis_floor(double v, double lo, double w) {
    return floor(__ddiv_rn(__dsub_rn(v, lo), w));
}

// Order-preserving map of a double to an unsigned 64-bit key (x < y iff
// key(x) < key(y) for non-NaN values; -0 sorts just below +0).
__device__ __forceinline__ unsigned long long order_key(double v) {
    unsigned long long b = (unsigned long long)__double_as_longlong(v);
    return (b >> 63) ? ~b : (b | 0x8000000000000000ULL);
}
__device__ __forceinline__ double key_value(unsigned long long k) {
    return __longlong_as_double((long long)((k >> 63) ? (k & 0x7fffffffffffffffULL) : ~k));
}

// FP32 value of a finite double, truncated, from its bit pattern with integer
// operations only (no FP64 instruction); magnitudes outside the FP32 normal
// range are clamped.  Only used as an estimate.
__device__ __forceinline__ float approx_float(double v) {
    unsigned long long b = (unsigned long long)__double_as_longlong(v);
    unsigned hi = (unsigned)(b >> 32);
    int e = (int)((hi >> 20) & 0x7ff) - 896;          // FP32 biased exponent
    unsigned m = (unsigned)(b >> 29) & 0x7fffffu;
    unsigned bits = (e <= 0) ? 0u : (e >= 255 ? 0x7f7fffffu : (((unsigned)e << 23) | m));
    return __uint_as_float(bits | (hi & 0x80000000u));
}

// Split a finite double v into FP32 hi + lo with integer and FP32 operations
// only: hi = v truncated toward zero to FP32 (a monotone map), lo = fl32(v - hi)
// (the 29 mantissa bits the truncation drops, converted and scaled by a power
// of two).  |v - hi| < ulp32(hi) <= 2^-23 |v|; magnitudes below 2^-126 give
// hi = lo = 0 and magnitudes beyond the FP32 range are clamped (callers keep
// coordinates below 1e30).
__device__ __forceinline__ void split_double(double v, float &hi, float &lo) {
    const unsigned long long b = (unsigned long long)__double_as_longlong(v);
    hi = approx_float(v);
    const int pe = (int)((b >> 52) & 0x7ff) - 948;   // FP32 biased exponent of 2^(e - 52)
    const float scale = (pe >= 1 && pe <= 254) ? __int_as_float(pe << 23) : 0.0f;
    const float l = __uint2float_rn((unsigned)(b & 0x1fffffffULL)) * scale;
    lo = (b >> 63) ? -l : l;
}

// Cell-relative FP32 coordinate (hi - origin) + lo of a split value.
__device__ __forceinline__ float rel_coord(float hi, float lo, float origin) {
    return __fadd_rn(__fsub_rn(hi, origin), lo);
}

// Bit pattern of the double equal to a float (exact widening) with integer
// operations only; finite normal or zero inputs, infinities kept.
__device__ __forceinline__ double widen(float f) {
    const unsigned u = __float_as_uint(f);
    const unsigned long long s = (unsigned long long)(u & 0x80000000u) << 32;
    const unsigned e = (u >> 23) & 0xff, m = u & 0x7fffffu;
    unsigned long long bits;
    if (e == 0) bits = s;                                        // zero (FP32 subnormals flushed)
    else if (e == 0xff) bits = s | 0x7ff0000000000000ULL | ((unsigned long long)m << 29);
    else bits = s | ((unsigned long long)(e + 896) << 52) | ((unsigned long long)m << 29);
    return __longlong_as_double((long long)bits);
}

// Cell index along one axis by threshold table: keys[k] is the order key of the
// smallest double whose cell, floor(fl(fl(v - lo) / w)), is >= k, so the cell
// of v is the k with keys[k] <= key(v) < keys[k + 1] (exactly the FP64 rule:
// the rule is monotone in v).  An FP32 estimate picks the start; integer key
// compares walk to the exact cell.  Returns -1 outside [keys[0], keys[n]).
__device__ __forceinline__ int axis_cell(double v, const unsigned long long *keys, int n, float lof, float iwf) {
    const unsigned long long k = order_key(v);
    if (k < keys[0] || k >= keys[n]) return -1;
    float t = floorf((approx_float(v) - lof) * iwf);
    int i = (t >= (float)(n - 1)) ? n - 1 : (t > 0.0f ? (int)t : 0);
    while (k < keys[i]) --i;          // keys[0] <= k, so this stops at i >= 0
    while (k >= keys[i + 1]) ++i;     // k < keys[n], so this stops at i <= n - 1
    return i;
}

// Cell index along one axis from FP32 alone: true when the estimate lies
// farther than its error bound tol from every cell boundary and inside the
// grid, so that i is certain; r is then the place within the cell, 0 to 1, off
// by at most tol.  The bound (estimate_tol) covers the truncation of v to FP32
// (subnormals to zero), the rounding of lo and 1 / w, and the two operations; it
// is infinite for grids that leave the FP32 range.  NaN, infinite and far outside
// values are never certain.
__device__ __forceinline__ bool axis_estimate(double v, float lof, float iwf, float tol, int n, int &i, float &r) {
    const float t = __fmul_rn(__fsub_rn(approx_float(v), lof), iwf);
    const float f = floorf(t);
    r = t - f;
    i = (int)f;
    return r > tol && r < 1.0f - tol && t > 0.0f && t < (float)n;
}
__device__ __forceinline__ bool axis_estimate(double v, float lof, float iwf, float tol, int n, int &i) {
    float r;
    return axis_estimate(v, lof, iwf, tol, n, i, r);
}

// Whether a point certainly lies outside the grid box (NaN and infinite
// coordinates among them, which approx_float clamps): the estimate is monotone in
// v, so where it is farther than twice its bound from the grid's range, v is
// farther than the bound from it, hence no rounding of the exact rule puts it in.
// (Left to the exact rule such points wait in the PIP join's lists: 5 M points,
// 15 of 16 outside the stars' 64 x 64 grid, 160 us against 49; the 100 M points
// of the tilings, of which a few are outside, 1,211 against 1,138 us.)
__device__ __forceinline__ bool axis_outside(double v, float lof, float iwf, float tol, int n) {
    const float t = __fmul_rn(__fsub_rn(approx_float(v), lof), iwf);
    return t < -2.0f * tol || t > (float)n + 2.0f * tol;
}
__device__ __forceinline__ bool point_outside(const GridDev &g, double x, double y) {
    return axis_outside(x, g.x0f, g.icwf, g.tolx, g.nx) || axis_outside(y, g.y0f, g.ichf, g.toly, g.ny);
}

// Column and row of a point, (-1 in an axis) outside the half-open grid box or
// with a NaN or infinite coordinate.
__device__ __forceinline__ int2 point_cell_exact(const GridDev &g, double x, double y) {
    const unsigned long long EXP = 0x7ff0000000000000ULL;
    int2 r = make_int2(-1, -1);
    if (((unsigned long long)__double_as_longlong(x) & EXP) != EXP &&
        ((unsigned long long)__double_as_longlong(y) & EXP) != EXP) {
        r.x = axis_cell(x, g.kx, g.nx, g.x0f, g.icwf);
        r.y = axis_cell(y, g.ky, g.ny, g.y0f, g.ichf);
    }
    return r;
}

// Cell id of a point (Sec. III.A), G when it lies outside the half-open grid
// box or has a NaN or infinite coordinate; (ix, iy) its column and row.  The
// estimate settles all but the points near a cell boundary (0.1 % at 512 cells
// per axis); the tables' four 8-byte loads per axis at random places were most
// of the cell-id pass's L1 traffic (170 M points: the join 12.39 -> 12.21 ms, the
// pass's atomics bound it now).
__device__ __forceinline__ int point_cell_xy(const GridDev &g, double x, double y, int &ix, int &iy) {
    const bool sx = axis_estimate(x, g.x0f, g.icwf, g.tolx, g.nx, ix);
    const bool sy = axis_estimate(y, g.y0f, g.ichf, g.toly, g.ny, iy);
    if (!(sx && sy)) {
        const int2 e = point_cell_exact(g, x, y);
        ix = e.x;
        iy = e.y;
        if (ix < 0 || iy < 0) return g.G;
    }
    return iy * g.nx + ix;
}
__device__ __forceinline__ int point_cell(const GridDev &g, double x, double y) {
    int ix, iy;
    return point_cell_xy(g, x, y, ix, iy);
}

// floor((v - lo) / w) clamped to [0, n - 1] (rasterisation of MBB corners).
__device__ __forceinline__ int clamped_axis(double v, double lo, double w, int n) {
    double f = axis_floor(v, lo, w);
    if (!(f >= 0.0)) return 0;
    if (f > (double)(n - 1)) return n - 1;
    return (int)f;
}

// FP32 frame origin of cell c: the lower-left corner x0 + ix * cw rounded to
// FP32, read from per-axis tables built with the layer (frame_x[nx], frame_y[ny]).
__device__ __forceinline__ float2 cell_frame(const float *fx, const float *fy, int nx, int c) {
    const int iy = c / nx;
    return make_float2(fx[c - iy * nx], fy[iy]);
}

__device__ __forceinline__ int lane_id() { return threadIdx.x & 31; }

// Bounds-checked builds (compiled with -DSJ_CHECK_BOUNDS): a guarded access
// first tests its index; out of range, it is skipped and the guard's code is
// OR-ed into this translation unit's error word, which the host reads back
// after the call (bounds_take()) -- no trap, the context stays usable.  In
// normal builds a guard is `true` and costs nothing.
enum {
    BND_BUCKET = 1, BND_SCATTER = 2, BND_UNSORT = 4, BND_P2P_POINT = 8, BND_P2P_REC = 16, BND_P2P_RES = 32,
    BND_PIP_POINT = 64, BND_PIP_REC = 128, BND_PIP_RES = 256
};
#ifdef SJ_CHECK_BOUNDS
static __device__ unsigned g_bounds_err;
#define SJ_IN_BOUNDS(cond, code) ((cond) || (atomicOr(&g_bounds_err, (unsigned)(code)), false))
// This translation unit's error word, read and cleared (host).
static inline unsigned bounds_take() {
    unsigned v = 0, z = 0;
    if (cudaMemcpyFromSymbol(&v, g_bounds_err, sizeof(v)) != cudaSuccess) return 0x80000000u;
    cudaMemcpyToSymbol(g_bounds_err, &z, sizeof(z));
    return v;
}
#else
#define SJ_IN_BOUNDS(cond, code) true
static inline unsigned bounds_take() { return 0; }
#endif

// 16-byte asynchronous copy global -> shared (cp.async), cached in L2 only:
// the copied data is read once, from shared memory, and allocating it in L1
// would evict the segment records that consecutive items of a cell re-read
// (P2P refine at 170 M points: 4.72 -> 4.23 ms).  Both addresses 16-byte
// aligned.  The copying thread sees the data after copy_async_wait_all().
__device__ __forceinline__ void copy16_async(void *smem_dst, const void *gmem_src) {
    const unsigned d = (unsigned)__cvta_generic_to_shared(smem_dst);
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(d), "l"(gmem_src) : "memory");
}
__device__ __forceinline__ void copy_async_wait_all() {
    asm volatile("cp.async.commit_group;\ncp.async.wait_group 0;\n" ::: "memory");
}

// Points per work item of cell c: the join's chunk size ch, reduced for cells
// whose points each test many edges / segments (work = the cell's list
// length) so that points x work stays within ch x budget -- the work queue is
// split by candidate-edge count, heavy cells yielding more, smaller items --
// but never below min(ch, 8) points (budget 0: ch for every cell).
__host__ __device__ __forceinline__ int cell_chunk(int ch, int work, int budget) {
    if (budget <= 0 || work <= budget) return ch;
    const long long c = (long long)ch * budget / work;
    const int lo = ch < 8 ? ch : 8;
    return c < lo ? lo : (c > ch ? ch : (int)c);
}

// clamped_axis without FP64 for all but the values near a cell boundary or the
// grid's ends: the FP32 estimate with four times its error bound (the values of
// interest reach one cell beyond the grid, where the bound's max |v| may treble).
__device__ __forceinline__ int clamped_cell(double v, double lo, double w, int n, float lof, float iwf, float tol) {
    const float t = __fmul_rn(__fsub_rn(approx_float(v), lof), iwf);
    const float f = floorf(t), r = t - f, e = 4.0f * tol;
    if (r > e && r < 1.0f - e && t > -1.0f && t < (float)n + 1.0f) return min(max((int)f, 0), n - 1);
    return clamped_axis(v, lo, w, n);
}
__device__ __forceinline__ int clamped_col(const GridDev &g, double x) {
    return clamped_cell(x, g.x0, g.cw, g.nx, g.x0f, g.icwf, g.tolx);
}
__device__ __forceinline__ int clamped_row(const GridDev &g, double y) {
    return clamped_cell(y, g.y0, g.ch, g.ny, g.y0f, g.ichf, g.toly);
}

// Minimum bounding box of an object.
struct Box {
    double xmin, ymin, xmax, ymax;
};

// Layer kinds.
enum { KIND_PIP = 0, KIND_P2P = 1 };

// Per-layer device counters (index into sj_run_stats order after `joins`).
enum { ST_POINTS = 0, ST_ITEMS, ST_PAIRS, ST_TESTS, ST_FALLBACK, ST_HITS, ST_ALGO, ST_RESOLVED, ST_N };

// Adds counters to the layer's statistics with one global atomic per counter
// and block: every lane 0 of the block's NW warps passes its warp's values
// (others pass anything), which are summed over the block's shared memory.
// Every thread of the block must call it (it synchronises the block).
// Thousands of warps adding to the same few addresses would otherwise queue at
// the L2; a shared 64-bit atomic per counter and warp instead of the plain
// stores cost a small call 1 us.
template <int NW>
__device__ __forceinline__ void flush_stats(unsigned long long *stats, const unsigned long long *v) {
    __shared__ unsigned long long blk[NW][ST_N];
    if ((threadIdx.x & 31) == 0)
#pragma unroll
        for (int k = 0; k < ST_N; ++k) blk[threadIdx.x >> 5][k] = v[k];
    __syncthreads();
    if (threadIdx.x < ST_N) {
        unsigned long long t = 0;
#pragma unroll
        for (int w = 0; w < NW; ++w) t += blk[w][threadIdx.x];
        if (t) atomicAdd(&stats[threadIdx.x], t);
    }
}

// Sum of the lanes' counters: in 32 bits while they are small.
__device__ __forceinline__ unsigned long long warp_sum(unsigned long long v) {
    if (!__any_sync(FULL, (v >> 26) != 0)) return __reduce_add_sync(FULL, (unsigned)v);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(FULL, v, o);
    return v;
}

// What the P2P refinement leaves in a slot, for the finishing kernels.
//   FP32X: id >= 0: the polyline, aux = the bits of its certified FP32 distance;
//          id < -1: the nearest segment is -2 - id (FP64 distance to be taken).
//   FP64:  id >= 0: a segment, aux >= 0: a second one; the nearest is among them.
//   id == -1: no polyline within the window.
struct alignas(8) P2PRec {
    int id, aux;
};

// Segment tables: the segment that starts at vertex i.
struct SegArgs {
    const double2 *verts;    // [V] FP64 vertices
    const double2 *seg_e64;  // [V] b - a
    const double *seg_inv64; // [V] 1 / |b - a|^2 (0 for a degenerate segment)
    const float4 *seg32;     // [V] (fl32(ex), fl32(ey), fl32(1 / |e|^2), owner polyline id bits)
};

// Arguments of the P2P refinement kernels.
struct RefineArgs {
    GridDev g;
    const int2 *items;       // (cell, first point of the chunk within the cell)
    const int *n_items;      // device count
    int *work_next;          // zeroed device counter handing out items (or null: fixed stride)
    int claim;               // consecutive items a warp takes per counter update (>= 1)
    const int *cell_start;   // [G + 1] sorted point ranges
    const int *perm;         // sorted slot -> input index
    const double2 *spts;     // sorted points (FP64), or null: the point of slot j is pts[perm[j]]
    const double2 *pts;      // input points (used when spts is null)
    SegArgs seg;
    const int *cseg_start;   // [G + 1] per-cell segment lists
    const int *cseg_ids;     //      segment (= first vertex) indices, ascending per cell
    const float4 *cseg_rec;  //      [2 MS] staging records of the list entries (see sj_filter.cu)
    double D;                // window
    float Ddn, Dup;          // FP32 D rounded down / up with a 1e-12 relative margin
    float Df;                // D rounded to FP32 (staging prune)
    // per-point windows (batched rounds whose requests ask for windows below
    // D): when win_on and *win_on != 0, point slot j is joined within win[j]
    // (<= D) instead of D; the lists and the staging prune stay those of D
    const double *win;
    const int *win_on;
    float eps_abs;           // absolute term of the split-coordinate rounding bound
    const float *frame_x;    // [nx] FP32 cell frame origins along x
    const float *frame_y;    // [ny]
    int npts;                // input points (slot indices and perm values stay below it)
    int ch;                  // points per work item (at most; see cell_chunk)
    const int *cell_work;    // [G] per-point edge / segment work of each cell (or null)
    int budget;              // edge budget per point of an item (0: none)
    P2PRec *rec;             // [n] per slot
    int2 *fb;                // points to redo in FP64 (sorted slot, cell)
    int *n_fb;
    unsigned long long *stats;
};

// FP64 point of sorted slot j.
__device__ __forceinline__ double2 slot_point(const RefineArgs &a, int j) {
    return a.spts ? a.spts[j] : a.pts[a.perm[j]];
}

// One request of a batched round as the kernels see it.
struct RoundReq {
    const double2 *pts;
    int *out_id;
    double *out_d;
    double window;   // P2P window of this request (the layer's D when none is asked)
    int off;         // first global point index
    int n;
};

// The request that holds global point i: the last one whose offset is <= i.
__device__ __forceinline__ int find_request(const RoundReq *r, int nr, int i) {
    int lo = 0, hi = nr;
    while (hi - lo > 1) {
        const int mid = (lo + hi) >> 1;
        if (r[mid].off <= i) lo = mid; else hi = mid;
    }
    return lo;
}

// Order key of a y-value with -0 folded onto +0 (IEEE compares treat them as
// equal; the order key alone would not).
__device__ __forceinline__ unsigned long long y_key(double v) { return order_key(v == 0.0 ? 0.0 : v); }

// Near-edge lists longer than PIP_SEARCH are searched by y instead of scanned
// (with the sub-cell flag: longer than PIP_SEARCH_MIN).  A scan stops early, so
// up to about 32 edges it costs what the two dependent binary searches do.
constexpr int PIP_SEARCH = 32, PIP_SEARCH_MIN = 16;

// Arguments of the PIP join (the records are described in sj_pip.cu).
struct PipArgs {
    GridDev g;
    const int4 *cells;       // [G] code (result of a classified cell, else -2 - first unit of its
                             //     record), sub-cell classes, the ids of classes 1 and 2
    const int4 *units;       // [2 per 32-byte unit]
    int units_n;
    const double2 *verts;
    const int *nxt;          // next vertex of the same ring
    const float *frame_x, *frame_y;
    float eps;               // absolute term of the split-coordinate rounding bound
    int search;              // lists longer than this are searched by y
    unsigned long long *stats;
};
// Scratch of the lists of a join's or a round's points, in 4-byte integers (0 for
// small calls: lists null).
long long pip_list_ints(long long n, int sms);
long long pip_round_list_ints(long long max_points, int sms);
cudaError_t launch_pip_join(const PipArgs &a, const double2 *pts, int n, int *out, unsigned *lists, int sms,
                            cudaStream_t s);
cudaError_t launch_pip_round(const PipArgs &a, const RoundReq *reqs, const int *meta, long long max_points,
                             unsigned *lists, int sms, cudaStream_t s);

// PIP layer build: per edge its rows (of the lower and the upper end), x-range
// and kind (bit 0: the first end is the lower one; bit 1: horizontal).
struct PipEdges {
    int2 *rows;
    float2 *xr;
    unsigned char *kind;
};
// A row list's entry, with what the cells' entries need to know of its edge.
struct alignas(32) PipRow {
    int edge;         // first vertex
    float x0, x1;     // x-range, rounded outward
    int lo, hi;       // rows of the lower and the upper end
    int kind;         // as PipEdges::kind
    int twin;         // polygon of the edge with the same end points, or -1
    int pad;
};
struct alignas(16) PipFlipTmp {
    unsigned long long key;
    unsigned mask;
    int pad;
};
struct PipBuildArgs {
    GridDev g;
    int V, M;
    const double2 *verts;
    const int *nxt, *prv, *owner, *obj_voff;
    PipEdges e;
    int *twin;                                  // [V] edge with the same end points in another place, or -1
    const int *cand_start, *cand_ids;
    const int *prow_base, *prow_r0, *prow_start;
    const PipRow *rows;                         // [ME] the row lists' records
    float2 *col;                                // [nx] column limits widened by delta
    int *entry_cell, *ord, *edge_at, *flip_at;  // [M]
    int2 *ent;                                  // [M] near edges, (flips << 3 | horizontal << 2 | base parity << 1 | any)
    int4 *cells;                                // [G] as PipArgs
    float cwf, chf;                             // cell size
    float sub_mx, sub_my;                       // margins of the sub-cell classes (< 0: none)
    float eps;                                  // as PipArgs
    int *units_of, *edges_of, *flips_of;        // [G]
    const int *units_at, *edges_at, *flips_at;  // [G + 1] their exclusive sums
    int4 *units;
    int2 *tmp_edge;                             // (edge, mask) of every record's near edges
    float4 *tmp_rel;                            // their cell-relative ends
    PipFlipTmp *tmp_flip;
    int4 *long_list;                            // groups ordered by a whole block
    int *long_n;
    const float *frame_x, *frame_y;
};
cudaError_t launch_pip_edges(const PipBuildArgs &b, cudaStream_t s);
cudaError_t launch_pip_twins(const PipBuildArgs &b, int *table, unsigned slots, cudaStream_t s);
cudaError_t launch_prow_edges(const PipBuildArgs &b, int *cnt, unsigned long long *total, const int *start, int *ids,
                              PipRow *rows, cudaStream_t s);
cudaError_t launch_pip_count(const PipBuildArgs &b, double delta, cudaStream_t s);
cudaError_t launch_pip_records(const PipBuildArgs &b, cudaStream_t s);
constexpr int PIP_LONG_MIN = 256;   // records of more elements may be listed in long_list

// Arguments of the PIP work census.
struct CensusArgs {
    GridDev g;
    const int *cand_start, *cand_ids, *obj_voff;
    const int *prow_base, *prow_r0, *prow_start, *pedge_ids, *nxt;
    const double2 *verts;
};

cudaError_t launch_cell_work_p2p(const int *cseg_start, int G, int *work, cudaStream_t s);

// The error words of the bounds-checked build, per translation unit, read
// and cleared (0 in normal builds).
unsigned bounds_take_filter();
unsigned bounds_take_p2p();
unsigned bounds_take_pip();

// Host-side launchers (defined in the .cu files).
cudaError_t launch_p2p_refine(const RefineArgs &a, int form, int warps_per_block, int blocks, cudaStream_t s);
cudaError_t launch_p2p_recheck(const RefineArgs &a, int form, int blocks, cudaStream_t s);
// A small call without bucketing (FP32X: n <= P2P_DIRECT_FP32X; FP64 leaves a.rec by input point).
struct DirectArgs {
    const int *cand_start, *cell_algo;   // statistics
    float cell_mag;    // no point of a cell has a larger |cell-relative coordinate|
    int *out_id;       // FP32X
    double *out_d;     //   (may be null)
};
constexpr int P2P_DIRECT_FP32X = 32768, P2P_DIRECT_FP64 = 131072;
constexpr int DIRECT_WARPS = 8;   // of a block
constexpr int DIRECT_OPEN = 64;   // FP32X: points of a block whose work item matters, at most
// Blocks of a direct call: a warp per point up to eight blocks an SM, then
// several points a warp, but (a part of a GPU with few SMs) no block more points
// than it can leave open.
constexpr int p2p_direct_blocks(int n, int sms) {
    const int most = (n + DIRECT_WARPS - 1) / DIRECT_WARPS, least = (n + DIRECT_OPEN - 1) / DIRECT_OPEN;
    const int blocks = most < sms * 8 ? most : (least > sms * 8 ? least : sms * 8);
    return blocks > 1 ? blocks : 1;
}
cudaError_t launch_p2p_direct(const RefineArgs &a, const DirectArgs &g, int form, int n, int sms, cudaStream_t s);
cudaError_t launch_p2p_finish(const RefineArgs &a, int form, const int *pos, int n, int *out_id, double *out_d,
                              cudaStream_t s);
cudaError_t launch_p2p_finish_slots(const RefineArgs &a, int form, const int *in_grid, int n, int *out_id,
                                    double *out_d, cudaStream_t s);
cudaError_t launch_p2p_finish_round(const RefineArgs &a, int form, const RoundReq *reqs, const int *meta,
                                    const int *pos, long long n_max, cudaStream_t s);
cudaError_t launch_pip_census(const CensusArgs &a, const double2 *pts, int n, unsigned long long *out,
                              cudaStream_t s);

struct BucketArgs {
    GridDev g;
    const double2 *pts;
    int n;
    int *cnt;            // [G + 1] zeroed
    int2 *key_rank;      // [n] (cell, rank within cell)
    int *cell_start;     // [G + 1]
    int *perm;           // [n]
    const int *cand_start;  // layer candidates (null: no work items)
    int ch;
    const int *cell_work;   // with budget > 0: work items of cell_chunk(ch, cell_work[c], budget) points
    int budget;
    int2 *items;         // work items or null
    int2 *block_sums;    // scan scratch
    size_t bs_cap;       // its capacity in int2 (launches fail when it is too small)
    int *totals;         // [2]: in-grid points, items
    const int *cell_algo;        // with stats: [G] segments of the cell's candidate polylines
    unsigned long long *stats;   // ST_PAIRS, ST_ALGO of the points of cells with candidates (or null)
    int *out_id;         // initialised to -1 (or null)
    double *out_d;       // initialised to +inf (or null)
    int *pos;            // [n] sorted slot of each input point, -1 when its cell has no
                         //     candidates or it lies outside the grid (or null)
    int *cell_base;      // [G] with pos: cell_start of cells that yield work items, else -1
    // Sub-cell order (sub_lx + sub_ly > 0): inside each cell the points are
    // ordered by sub-cell, 2^sub_lx x 2^sub_ly sub-cells in Z-order, so that
    // consecutive points of a cell -- one work item -- cover a compact part of
    // it.  cnt then holds G * S + 1 counters (S = 2^(sub_lx + sub_ly)) and
    // sub_start [G * S] the first slot of each sub-cell (-1 with pos for cells
    // without work items).  The order is a pure permutation within cells: no
    // result depends on it.
    int sub_lx, sub_ly;
    int *sub_start;
};

// Z-order index of sub-cell (sx, sy) with lx / ly bits per axis (at most 3).
__device__ __forceinline__ int sub_index(int sx, int sy, int lx, int ly) {
    int sub = 0, bit = 0;
#pragma unroll
    for (int b = 0; b < 3; ++b) {
        if (b < lx) sub |= ((sx >> b) & 1) << bit++;
        if (b < ly) sub |= ((sy >> b) & 1) << bit++;
    }
    return sub;
}
size_t bucket_scan_blocks(int G);
cudaError_t launch_bucket(const BucketArgs &a, cudaStream_t s);
struct LayerBuildArgs {
    GridDev g;
    int kind;
    double D;
    int nobj, V;
    const double2 *verts;
    const int *obj_voff;     // [nobj + 1]
    Box *mbb;                // [nobj]
    int *cell_cnt;           // [G + 1] zeroed
    int *cand_start;         // [G + 1]
    int *cursor;             // [G] zeroed
    int *obj_cells;          // [nobj + 1]
    int2 *block_sums;
    size_t bs_cap;           // capacity of block_sums in int2
    int *totals;
    int *bad;                // validation flags
};

}  // namespace sj

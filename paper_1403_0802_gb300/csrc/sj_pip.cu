// sj_pip.cu -- PIP join (Sec. III.C, Fig. 3): ray-crossing parity of each point
// against every ring of each candidate polygon of its cell; the result is the
// smallest candidate id with odd parity.
//
// The paper refines (cell, points) pairs against whole candidate polygons; here
// all that a point of a cell needs is laid out once with the layer, in one
// contiguous record per grid cell, so the join is one kernel over the points in
// input order: no bucketing, one coalesced read of the points and one coalesced
// write of the ids.
//
// Per cell (PipArgs::cells), a code:
//   >= -1   the result of every point of the cell (no candidate's edge comes
//           near the cell, so each candidate holds all of it or none of it);
//   <= -2   -2 - (first 32-byte unit of the cell's record),
// and for the latter the class of each of 4 x 4 sub-cells, two bits: 1 or 2 -- no
// near edge meets the sub-cell widened by a margin, and its points' result is
// the cell's first or second id --, 3 -- the same with no polygon --, or 0: the
// record decides.  One 16-byte read answers four of five points of the cells
// that edges pass (the tiles: 36 % of the points are in such cells, 8 % in a
// sub-cell that an edge meets).
// A record is a chain of groups of up to 32 relevant candidates in id order (a
// candidate that holds none of the cell is left out, and so is every candidate
// after one that holds all of it): a header, the near edges, the flips.  For a
// candidate of the cell (column [X0, X1), row r) the edges whose y-range
// reaches row r -- no other edge can straddle a point of the row -- split
// three ways by their x-range against the column widened by delta:
//   left:  farther than delta left of every point, so the FP64 rule never
//          counts a crossing -- dropped;
//   far:   farther than delta right of every point, so the FP64 rule counts a
//          crossing exactly when the edge straddles the point's y.  Their
//          parity is the parity of the number of their end y-values at or
//          below y: ends below the row give the group's base mask, ends inside
//          the row are "flips" (sorted by y, each with the mask that holds
//          from it on; an end shared by two far edges of the ring cancels);
//   near:  the rest, tested point by point.  Horizontal edges never straddle
//          and are left out.  An edge shared by two candidates (the common
//          side of two tiles: equal end points) is kept once, with the bits of
//          both, since the rule depends on the two end points only.
// Near edges are ordered by their lower y: a scan stops at the first edge above
// the point, and long lists are searched.
//
// Arithmetic: the straddle test and the orientation are evaluated in FP32 on
// cell-relative coordinates (from the (hi, lo) split of the FP64 inputs) with
// forward error bounds (Shewchuk's orient2d bound plus the input-rounding
// terms); whatever is not certain is redone with the FP64 rule on the original
// vertices.  The result is the FP64 rule's, bit for bit, in both forms.
#include <cuda_runtime.h>

#include <algorithm>

#include "sj_host.hpp"

namespace sj {

unsigned bounds_take_pip() { return bounds_take(); }

// ------------------------------------------------------------------ the crossing rule

// The crossing rule in FP64: straddle iff (a.y > p.y) != (b.y > p.y); with lo
// the end at or below p.y, count iff (hi.x-lo.x)(p.y-lo.y) - (hi.y-lo.y)(p.x-lo.x) > 0.
__device__ __forceinline__ int cross64(double px, double py, double ax, double ay, double bx, double by) {
    bool a_up = ay > py, b_up = by > py;
    if (a_up == b_up) return 0;
    double lx = a_up ? bx : ax, ly = a_up ? by : ay;
    double hx = a_up ? ax : bx, hy = a_up ? ay : by;
    double d = __dsub_rn(__dmul_rn(__dsub_rn(hx, lx), __dsub_rn(py, ly)),
                         __dmul_rn(__dsub_rn(hy, ly), __dsub_rn(px, lx)));
    return d > 0.0;
}

// Sign of the orientation d = A*B - C*D on cell-relative FP32 inputs, certified
// against the FP64 rule.  Every input coordinate c carries the rounding bound
// KV |c| + eps of the (hi, lo) split.  Returns false when |d| does not exceed
// E = errA + errIn + err64:
//   errA  = 3.0001 u (|AB| + |CD|)          FP32 rounding of d (Shewchuk orient2d)
//   errIn = first-order input perturbation plus cross terms, x (1 + 4u)
//   err64 = 4e-16 (|A||B| + |C||D|)         FP64 rounding of the reference rule
// E is inflated by (1 + 16u) for the FP32 evaluation of the bound itself.
__device__ __forceinline__ bool orient32(float px, float py, float lx, float ly, float hx, float hy, float eps,
                                         bool &pos) {
    const float KV = 2.0001f * U32;
    float A = __fsub_rn(hx, lx), B = __fsub_rn(py, ly);
    float C = __fsub_rn(hy, ly), Dd = __fsub_rn(px, lx);
    float AB = __fmul_rn(A, B), CD = __fmul_rn(C, Dd);
    float d = __fsub_rn(AB, CD);
    float dhx = fmaf(KV, fabsf(hx), eps), dhy = fmaf(KV, fabsf(hy), eps);
    float dlx = fmaf(KV, fabsf(lx), eps), dly = fmaf(KV, fabsf(ly), eps);
    float dpx = fmaf(KV, fabsf(px), eps), dpy = fmaf(KV, fabsf(py), eps);
    float dA = dhx + dlx, dB = dpy + dly, dC = dhy + dly, dD = dpx + dlx;
    float aA = fabsf(A), aB = fabsf(B), aC = fabsf(C), aD = fabsf(Dd);
    float errIn = (dA * aB + aA * dB + dA * dB + dC * aD + aC * dD + dC * dD) * (1.0f + 4.0f * U32);
    float errA = (3.0001f * U32) * (fabsf(AB) + fabsf(CD));
    float err64 = 4e-16f * ((aA + dA) * (aB + dB) + (aC + dC) * (aD + dD));
    float E = (errA + errIn + err64) * (1.0f + 16.0f * U32) + 1e-30f;
    pos = d > 0.0f;
    return fabsf(d) > E;
}

// Bound of the error of fl(a - b) against the difference of the two values
// whose cell-relative forms a and b are (2.0001 u |.| + eps each, plus the
// subtraction's own rounding): 3.01 u (|a| + |b|) + 2 eps.
__device__ __forceinline__ float diff_bound(float a, float b, float eps) {
    return fmaf(3.01f * U32, fabsf(a) + fabsf(b), 2.0f * eps);
}

// ------------------------------------------------------------------ cell records

// A group of a cell's record, in 32-byte units: header, n near edges, then (16
// bytes each) nf flips and, with PIP_EXT, the ids of its candidates.
constexpr int PIP_MORE = 1 << 30;      // another group follows
constexpr int PIP_EXT = 1 << 29;       // ids follow the flips; id[1] holds the float bits of h
constexpr int PIP_INLINE_IDS = 3;

struct alignas(16) PipHead {
    int n, nf;
    unsigned base;     // parity mask below the row's flips
    int ncand;         // candidates of the cell (statistics), with the PIP_* bits
    int id[3];         // ids of candidates 0..2; with PIP_EXT: candidates in the group, h, unused
    int algo;          // edges of the cell's candidate polygons (statistics)
};
struct alignas(16) PipEdge {
    float lx, ly, hx, hy;   // cell-relative ends, lower y first
    int vid;                // edge (= first vertex) index, for the FP64 rule
    unsigned mask;          // bits of the candidates it belongs to
    int pad[2];
};
struct alignas(16) PipFlip {
    float y;                    // cell-relative
    unsigned mask;              // parity mask from this y on
    unsigned long long key;     // y_key of the exact value
};
static_assert(sizeof(PipHead) == 32 && sizeof(PipEdge) == 32 && sizeof(PipFlip) == 16, "");

__host__ __device__ __forceinline__ long long group_units(int n, int nf, int ng) {
    const int ids = (ng > PIP_INLINE_IDS || n > PIP_SEARCH_MIN) ? (ng + 3) / 4 : 0;
    return 1LL + n + ((long long)nf + ids + 1) / 2;
}

// ------------------------------------------------------------------ the join

// Where a join's points come from and its ids go, and the scratch of the lists of
// points that wait (pip_list_ints; null: in shared memory).
struct OneSource {
    const double2 *pts;
    int *out;
    unsigned *lists;
    int n;
    __device__ __forceinline__ int count() const { return n; }
    __device__ __forceinline__ double2 point(unsigned i) const { return __ldcs(pts + i); }
    __device__ __forceinline__ void put(unsigned i, int id) const { out[i] = id; }
};
// Many requests as one point set (batched rounds).
struct RoundSource {
    const RoundReq *reqs;
    const int *meta;   // requests, points
    unsigned *lists;
    __device__ __forceinline__ int count() const { return meta[1]; }
    __device__ __forceinline__ const RoundReq &find(unsigned i) const {
        return reqs[find_request(reqs, meta[0], (int)i)];
    }
    __device__ __forceinline__ double2 point(unsigned i) const {
        const RoundReq &r = find(i);
        return __ldcs(r.pts + (i - r.off));
    }
    __device__ __forceinline__ void put(unsigned i, int id) const {
        const RoundReq &r = find(i);
        r.out_id[i - r.off] = id;
    }
};

// Warps per block and blocks per SM: bound by the latency of its gathers, the
// join is fastest at the most warps whose 64 registers hold the loop without
// spills: 10 M points on the heavy-tail tiles 458 / 430 / 445 us with 7 / 8 / 10
// blocks (48 registers, spilled), 100 M on the 40,000 tiles 1.12 / 1.14 / 1.32 ms.
constexpr int PIP_WARPS = 4, PIP_BLOCKS = 8;
// Code of a queued point whose cell the FP32 estimate leaves open (no record
// starts there: units are fewer than 2^31 - 2^22).
constexpr int PIP_UNSURE = -2147483647 - 1;
constexpr int PIP_SCAN_FLIPS = 8;   // flips scanned one by one by pip_short

// A lane's counters of the points refined.  In shared memory: the refinement
// has no registers for three 64-bit sums.
struct PipSums {
    unsigned long long tests, pairs, algo;
};

// Points of a tile with one point per lane: 32, but calls and rounds of fewer tiles
// than there are warps take tiles of 16, 8 or 4 points, since a warp refines two of
// the points that wait at a time (1,003 points in cells of some 500 edges, stars on
// a 16 x 16 grid: 70 / 39 / 23 / 14 / 10 us with 32 / 16 / 8 / 4 / 1; on the 40,000
// tiles 8.2 / 6.9 / 6.2 / 6.2 / 6.2).
__host__ __device__ __forceinline__ unsigned tile_points(unsigned n, unsigned warps) {
    unsigned per = 32;
    while (per > 4 && (n + per / 2 - 1) / (per / 2) <= warps) per /= 2;
    return per;
}

// A point that waits for its refinement.
struct PipQueued {
    double2 p;
    int i, code, ix, iy;   // point index, cell code, column, row
};
static_assert(sizeof(PipQueued) == 32, "");

// Whether a near edge counts for the point (px, py): 1 yes, 0 no, -1 not
// certain in FP32.
__device__ __forceinline__ int edge_cross(float px, float py, const float4 r, float eps) {
    const float sl = __fsub_rn(py, r.y), sh = __fsub_rn(py, r.w);
    const float el = diff_bound(py, r.y, eps), eh = diff_bound(py, r.w, eps);
    if (sl < -el || sh > eh) return 0;                      // certainly does not straddle
    bool pos = false;
    const bool sure = sl > el && sh < -eh && orient32(px, py, r.x, r.y, r.z, r.w, eps, pos);
    return sure ? (int)pos : -1;
}

// The same for edge i by the FP64 rule on the original vertices.
__device__ __forceinline__ int edge_cross64(const PipArgs &a, double2 p, int i) {
    const double2 A = a.verts[i], B = a.verts[a.nxt[i]];
    return cross64(p.x, p.y, A.x, A.y, B.x, B.y);
}

__device__ __forceinline__ float2 point_rel(const PipArgs &a, const PipQueued &q) {
    float hx, lx, hy, ly;
    split_double(q.p.x, hx, lx);
    split_double(q.p.y, hy, ly);
    return make_float2(rel_coord(hx, lx, a.frame_x[q.ix]), rel_coord(hy, ly, a.frame_y[q.iy]));
}

// Results of up to 32 points, one per lane, whose records are short: n <= a.search
// near edges, the id in the first group.  Returns false for a point that needs
// pip_hard, otherwise its id in res.  EXACT: tests that FP32 leaves open are redone
// with the FP64 rule (fb counts them); else such a point returns false too.
template <bool EXACT>
__device__ __forceinline__ bool pip_short(const PipArgs &a, const PipQueued &q, PipSums &sum, int &res, unsigned &fb) {
    res = -1;
    if (!EXACT && q.code == PIP_UNSURE) return false;
    const int off = -2 - q.code;
    if (!SJ_IN_BOUNDS(off < a.units_n, BND_PIP_REC)) return true;
    const int4 *u = a.units + 2 * (size_t)off;
    const int4 h0 = __ldg(u), h1 = __ldg(u + 1);   // n, nf, base, ncand; ids, algo (PipHead)
    const PipEdge *E = reinterpret_cast<const PipEdge *>(u + 2);
    // the first two edges travel with the header (a record ends at least two
    // units before the end of the array), the next ones two tests ahead
    float4 e0 = __ldg(reinterpret_cast<const float4 *>(E)), e1 = __ldg(reinterpret_cast<const float4 *>(E + 1));
    const int n = h0.x, nf = h0.y;
    if (n > a.search || nf > PIP_SCAN_FLIPS) return false;
    const PipFlip *F = reinterpret_cast<const PipFlip *>(E + n);
    const float2 r = point_rel(a, q);
    bool unsure = false;
    unsigned m = (unsigned)h0.z, redone = 0;
    if (EXACT) {
        const unsigned long long ky = y_key(q.p.y);
        for (int f = 0; f < nf && F[f].key <= ky; ++f) m = F[f].mask;
    }
    for (int f = 0; !EXACT && f < nf; ++f) {   // flips at or below y
        const float4 v = __ldg(reinterpret_cast<const float4 *>(F + f));
        const float d = __fsub_rn(r.y, v.x);
        unsure |= !(fabsf(d) > diff_bound(r.y, v.x, a.eps));
        if (!(d > 0.0f)) break;
        m = __float_as_uint(v.y);
    }
    int t = 0;
    for (; t < n; ++t) {
        const float4 e = e0;
        e0 = e1;
        if (t + 2 < n) e1 = __ldg(reinterpret_cast<const float4 *>(E + t + 2));
        // lower ends ascend: from the first edge wholly above y on, none straddles
        if (__fsub_rn(e.y, r.y) > diff_bound(r.y, e.y, a.eps)) break;
        int x = edge_cross(r.x, r.y, e, a.eps);
        if (EXACT && x < 0) {
            x = edge_cross64(a, q.p, E[t].vid);
            ++redone;
        }
        unsure |= x < 0;
        if (x > 0) m ^= __ldg(&E[t].mask);
    }
    if (unsure || (!m && (h0.w & PIP_MORE))) return false;
    sum.tests += (unsigned)t;
    sum.pairs += (unsigned)(h0.w & (PIP_EXT - 1));
    sum.algo += (unsigned)h1.w;
    fb += redone;
    if (m) {
        const int k = __ffs(m) - 1;
        if (h0.w & PIP_EXT) res = __ldg(reinterpret_cast<const int *>(F + nf) + k);
        else res = k == 0 ? h1.x : (k == 1 ? h1.y : h1.z);
    }
    return true;
}

// The general case, one point by HARD lanes (lane: 0 .. HARD - 1, mask gm): any
// number of groups, long lists searched by y, tests that FP32 leaves open redone
// with the FP64 rule.
constexpr int HARD = 16;   // 4 / 8 / 16 / 32: 506 / 420 / 401 / 425 us on the heavy-tail tiles (lists of 30 to 3,000 edges)
__device__ __forceinline__ int pip_hard(const PipArgs &a, const PipQueued &q, PipSums &sum, int lane, unsigned gm,
                                        unsigned &fb) {
    const double2 p = q.p;
    const float2 r = point_rel(a, q);
    const unsigned long long ky = y_key(p.y);
    int off = -2 - q.code, res = -1;
    unsigned tests = 0;
    bool first = true;
    while (SJ_IN_BOUNDS(off < a.units_n, BND_PIP_REC)) {
        const int4 *u = a.units + 2 * (size_t)off;
        const int4 h0 = u[0], h1 = u[1];
        const int n = h0.x, nf = h0.y;
        const PipEdge *E = reinterpret_cast<const PipEdge *>(u + 2);
        const PipFlip *F = reinterpret_cast<const PipFlip *>(E + n);
        if (first && lane == 0) {
            sum.pairs += (unsigned)(h0.w & (PIP_EXT - 1));
            sum.algo += (unsigned)h1.w;
        }
        first = false;
        unsigned m = (unsigned)h0.z;
        for (int f0 = 0, f1 = nf; f0 < f1;) {   // the last flip at or below y
            const int mid = (f0 + f1) >> 1;
            if (F[mid].key <= ky) {
                m = F[mid].mask;
                f0 = mid + 1;
            } else {
                f1 = mid;
            }
        }
        int lo = 0, hi = n;
        if (n > a.search) {
            // edges that can straddle y: lower ends within [y - h, y], widened
            // by the rounding bounds; both predicates are monotone in ly
            const float hh = __int_as_float(h1.y), ep = diff_bound(r.y, r.y, a.eps);
            int b1 = n;
            while (lo < b1) {
                const int mid = (lo + b1) >> 1;
                if (__fadd_ru(E[mid].ly, hh) < __fsub_rd(r.y, ep)) lo = mid + 1; else b1 = mid;
            }
            hi = lo;
            b1 = n;
            while (hi < b1) {
                const int mid = (hi + b1) >> 1;
                const float ly = E[mid].ly;
                if (fmaf(-3.01f * U32, fabsf(ly), ly) > __fadd_ru(r.y, ep)) b1 = mid; else hi = mid + 1;
            }
        }
        unsigned mm = 0;
        for (int t = lo + lane; t < hi; t += 4 * HARD) {   // four loads in flight per lane
            float4 e[4];
#pragma unroll
            for (int k = 0; k < 4; ++k)
                if (t + HARD * k < hi) e[k] = __ldg(reinterpret_cast<const float4 *>(E + t + HARD * k));
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                if (t + HARD * k >= hi) break;
                int x = edge_cross(r.x, r.y, e[k], a.eps);
                if (x < 0) {
                    x = edge_cross64(a, p, E[t + HARD * k].vid);
                    ++fb;
                }
                if (x) mm ^= E[t + HARD * k].mask;
            }
        }
        m ^= __reduce_xor_sync(gm, mm);
        tests += (unsigned)(hi - lo);
        if (m) {
            const int k = __ffs(m) - 1;
            if (h0.w & PIP_EXT) res = reinterpret_cast<const int *>(F + nf)[k];
            else res = k == 0 ? h1.x : (k == 1 ? h1.y : h1.z);
            break;
        }
        if (!(h0.w & PIP_MORE)) break;
        off += (int)group_units(n, nf, h1.x);   // a group before another holds 32 ids: PIP_EXT
    }
    if (lane == 0) sum.tests += tests;
    return res;
}

// One warp takes tiles of 32 U consecutive points.  A point whose cell is
// certain and classified is answered at once.  The others are queued in shared
// memory and refined 32 at a time, so that the refinement runs with full warps
// although only some of a tile's points (6 - 54 %) need it.  The few that this
// cannot finish wait until the warp has seen its last tile, in the warp's list (in
// scratch, or while it is short in shared memory); by then their general,
// register-hungry code costs the loop nothing (with a call to it inside the loop the
// 100 M point join took 2.3 - 4.5 ms instead of 1.6; with lists of up to 64 points in
// shared memory, refined whenever 32 wait, 1.31 instead of 1.22 ms, and 10 M points on
// the heavy-tail tiles 433 instead of 396 us).  Not in the output, threaded through
// the points' own places: requests and streams may share an output, and a list lost
// there takes other requests' points with it.
//
// Bound by the latency and the L1 wavefronts of the random reads of the cell
// table and the records, both L2-resident (ncu at 20 M points on the tiles: issue
// slots half busy, long-scoreboard the top stall, DRAM 14 % of peak).  Measured, us
// a join, against bucketing the points and refining (cell, point-chunk) items,
// then without and with the sub-cell classes: 1,003 points 53 -> 11 -> 11, 1 M on
// the stars (FP64 form) 119 -> 29 -> 21, 10 M on the heavy-tail tiles 2,450 -> 536
// -> 426 (401 with HARD = 16), 100 M on the 40,000 tiles 4,486 -> 1,590 -> 1,130.
// room: points of a warp's list at most.
template <int U, class Src>
__global__ void __launch_bounds__(PIP_WARPS * 32, PIP_BLOCKS) k_pip_join(PipArgs a, Src src, unsigned room) {
    __shared__ PipQueued queue[PIP_WARPS][32 * (U + 1)];
    extern __shared__ unsigned short_lists[];
    __shared__ PipSums sums[PIP_WARPS * 32];
    const int lane = lane_id(), w = threadIdx.x >> 5;
    const unsigned lt = (1u << lane) - 1u;
    const unsigned n = (unsigned)src.count(), step = U == 1 ? tile_points(n, gridDim.x * PIP_WARPS) : 32u * U;
    const unsigned tiles = (n + step - 1u) / step;
    unsigned items = 0, resolved = 0, hits = 0, fb = 0;
    sums[threadIdx.x] = PipSums{0, 0, 0};
    int qn = 0, wn = 0;   // points queued, points that wait
    for (unsigned t = blockIdx.x * PIP_WARPS + w;; t += gridDim.x * PIP_WARPS) {
        const bool more = t < tiles;   // else: the points left in the queues
        if (more) {
            const unsigned i0 = t * step + lane, end = U == 1 && (unsigned)lane >= step ? 0u : n;
            double2 p[U];
            int code[U], ix[U], iy[U];
#pragma unroll
            for (int u = 0; u < U; ++u)
                if (i0 + 32u * u < end) p[u] = src.point(i0 + 32u * u);
#pragma unroll
            for (int u = 0; u < U; ++u) {
                code[u] = -1;
                if (i0 + 32u * u < end) {
                    float rx, ry;
                    const bool sx = axis_estimate(p[u].x, a.g.x0f, a.g.icwf, a.g.tolx, a.g.nx, ix[u], rx);
                    const bool sy = axis_estimate(p[u].y, a.g.y0f, a.g.ichf, a.g.toly, a.g.ny, iy[u], ry);
                    code[u] = PIP_UNSURE;
                    if (sx && sy) {
                        const int4 c = __ldg(a.cells + iy[u] * a.g.nx + ix[u]);
                        code[u] = c.x;
                        if (c.x < -1) {
                            const int k = (int)(ry * 4.0f) * 4 + (int)(rx * 4.0f);
                            const unsigned cls = ((unsigned)c.y >> (2 * k)) & 3u;
                            if (cls) code[u] = cls == 1 ? c.z : (cls == 2 ? c.w : -1);
                        }
                        resolved += code[u] >= -1;
                    } else if (point_outside(a.g, p[u].x, p[u].y)) {
                        code[u] = -1;
                    }
                }
            }
#pragma unroll
            for (int u = 0; u < U; ++u) {
                const unsigned i = i0 + 32u * u;
                const bool q = i < end && code[u] < -1;
                if (i < end && !q) {
                    src.put(i, code[u]);
                    hits += code[u] >= 0;
                }
                const unsigned bal = __ballot_sync(FULL, q);
                if (q) queue[w][qn + __popc(bal & lt)] = PipQueued{p[u], (int)i, code[u], ix[u], iy[u]};
                qn += __popc(bal);
            }
            __syncwarp();
        }
        while (more ? qn >= 32 : qn > 0) {
            const int cnt = min(qn, 32);
            qn -= cnt;
            bool wait = false;
            unsigned i = 0;
            if (lane < cnt) {
                const PipQueued q = queue[w][qn + lane];
                i = (unsigned)q.i;
                int res;
                const bool done = pip_short<false>(a, q, sums[threadIdx.x], res, fb);
                if (SJ_IN_BOUNDS(i < n, BND_PIP_RES)) {
                    if (done) src.put(i, res);
                    hits += done && res >= 0;
                    wait = !done;
                }
            }
            const unsigned bal = __ballot_sync(FULL, wait);
            if (wait) {   // (a pointer to the list kept through the loop would cost it two registers)
                const unsigned k = (unsigned)(wn + __popc(bal & lt));
                if (src.lists) src.lists[(size_t)(blockIdx.x * PIP_WARPS + w) * room + k] = i;
                else short_lists[w * room + k] = i;
            }
            wn += __popc(bal);
            ++items;
        }
        if (!more) break;
        __syncwarp();
    }
    __syncwarp();
    // The points that wait, one per lane: those of short records end here (5 M points
    // on the sides of 500 m squares, all of whose tests FP64 decides: 2,100 us with
    // all of them by pip_hard, 310 - 390 so).
    for (int k0 = 0; k0 < wn; k0 += 32) {
        PipQueued q;
        bool act = k0 + lane < wn;
        int res = -1;
        if (act) {
            const unsigned k = (unsigned)(k0 + lane);
            q.i = (int)(src.lists ? src.lists[(size_t)(blockIdx.x * PIP_WARPS + w) * room + k] : short_lists[w * room + k]);
            q.p = src.point((unsigned)q.i);
            const int2 e = point_cell_exact(a.g, q.p.x, q.p.y);
            const int code = e.x >= 0 && e.y >= 0 ? a.cells[e.y * a.g.nx + e.x].x : -1;
            q.ix = e.x;
            q.iy = e.y;
            q.code = code;
            bool done = code >= -1;
            res = code;
            if (done) resolved += e.x >= 0 && e.y >= 0;
            else done = pip_short<true>(a, q, sums[threadIdx.x], res, fb);
            if (done) {
                src.put((unsigned)q.i, res);
                hits += res >= 0;
                act = false;
            }
        }
        const int sub = lane & (HARD - 1), grp = lane / HARD;
        const unsigned gm = (HARD == 32 ? FULL : (1u << (HARD & 31)) - 1u) << (lane & ~(HARD - 1));
        for (unsigned left = __ballot_sync(FULL, act); left;) {   // a point for each group of lanes
            int j = -1;
#pragma unroll
            for (int k = 0; k < 32 / HARD; ++k) {
                if (grp == k && left) j = __ffs(left) - 1;
                left &= left - 1;
            }
            const int from = j < 0 ? lane : j;
            PipQueued r;
            r.p = make_double2(__shfl_sync(FULL, q.p.x, from), __shfl_sync(FULL, q.p.y, from));
            r.i = __shfl_sync(FULL, q.i, from);
            r.code = __shfl_sync(FULL, q.code, from);
            r.ix = __shfl_sync(FULL, q.ix, from);
            r.iy = __shfl_sync(FULL, q.iy, from);
            if (j >= 0) {
                const int id = pip_hard(a, r, sums[threadIdx.x], sub, gm, fb);
                if (sub == 0) {
                    src.put((unsigned)r.i, id);
                    hits += id >= 0;
                }
            }
            __syncwarp();
        }
        if (__any_sync(FULL, act)) ++items;
    }
    if (a.stats) {
        unsigned long long v[ST_N] = {};
        const PipSums s = sums[threadIdx.x];
        v[ST_ITEMS] = items;
        v[ST_PAIRS] = warp_sum(s.pairs);
        v[ST_TESTS] = warp_sum(s.tests);
        v[ST_ALGO] = warp_sum(s.algo);
        v[ST_RESOLVED] = __reduce_add_sync(FULL, resolved);
        v[ST_FALLBACK] = __reduce_add_sync(FULL, fb);
        v[ST_HITS] = __reduce_add_sync(FULL, hits);
        flush_stats<PIP_WARPS>(a.stats, v);
    }
}

// Points per lane and tile: two once that still gives every SM all its warps
// twice over (100 M points: 1.32 / 1.14 / 1.13 / 1.38 ms with 1 / 2 / 3 / 4); smaller
// calls spread over more warps, one point per lane.
constexpr int PIP_U = 2;

// Points per lane of a call's tiles.
static int pip_unroll(long long n, int sms) { return n >= sms * PIP_WARPS * PIP_BLOCKS * 32LL * 2 * PIP_U ? PIP_U : 1; }

static int pip_per(int U, long long n, int sms) {
    return U == 1 ? (int)tile_points((unsigned)n, (unsigned)(sms * PIP_BLOCKS * PIP_WARPS)) : 32 * U;
}

static int pip_blocks(int per, long long n, int sms) {
    const long long tiles = (n + per - 1) / per;
    return (int)std::max(1LL, std::min((tiles + PIP_WARPS - 1) / PIP_WARPS, (long long)sms * PIP_BLOCKS));
}

// Points of a call's warps at most (a call of fewer points on the same grid: no more).
static long long pip_room(int per, long long n, int sms) {
    const long long tiles = (n + per - 1) / per, warps = (long long)pip_blocks(per, n, sms) * PIP_WARPS;
    return (tiles + warps - 1) / warps * per;
}

// Lists of up to this many points are held in shared memory (calls of up to 1.2 M
// points: the stream-ordered allocation of scratch takes 2 us of a call).
constexpr int PIP_SHORT = 256;

static long long list_ints(int per, long long n, int sms) {
    const long long room = pip_room(per, n, sms);
    return room <= PIP_SHORT ? 0 : room * pip_blocks(per, n, sms) * PIP_WARPS;
}
long long pip_list_ints(long long n, int sms) { return list_ints(pip_per(pip_unroll(n, sms), n, sms), n, sms); }
long long pip_round_list_ints(long long max_points, int sms) { return list_ints(pip_per(1, max_points, sms), max_points, sms); }

template <int U, class Src>
static cudaError_t pip_launch(const PipArgs &a, const Src &src, int per, long long n, int sms, cudaStream_t s) {
    if (!src.lists && list_ints(per, n, sms) > 0) return cudaErrorInvalidValue;
    const unsigned room = (unsigned)pip_room(per, n, sms);
    const size_t smem = src.lists ? 0 : sizeof(unsigned) * PIP_WARPS * room;
    k_pip_join<U><<<pip_blocks(per, n, sms), PIP_WARPS * 32, smem, s>>>(a, src, room);
    return cudaGetLastError();
}

cudaError_t launch_pip_join(const PipArgs &a, const double2 *pts, int n, int *out, unsigned *lists, int sms,
                            cudaStream_t s) {
    const OneSource src{pts, out, lists, n};
    const int U = pip_unroll(n, sms), per = pip_per(U, n, sms);
    return U == PIP_U ? pip_launch<PIP_U>(a, src, per, n, sms, s) : pip_launch<1>(a, src, per, n, sms, s);
}

cudaError_t launch_pip_round(const PipArgs &a, const RoundReq *reqs, const int *meta, long long max_points,
                             unsigned *lists, int sms, cudaStream_t s) {
    return pip_launch<1>(a, RoundSource{reqs, meta, lists}, pip_per(1, max_points, sms), max_points, sms, s);
}

// ------------------------------------------------------------------ layer build

// Where a layer's edges lie (PipEdges), one thread per edge (vertex i -> nxt[i]):
// its grid rows under the cell rule, its x-range rounded outward to FP32, and
// which end is the lower one.
__global__ void k_pip_edges(GridDev g, const double2 *verts, const int *nxt, int V, PipEdges e) {
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < V; i += gridDim.x * blockDim.x) {
        const double2 A = verts[i], B = verts[nxt[i]];
        const bool up = A.y <= B.y;
        e.rows[i] = make_int2(clamped_row(g, up ? A.y : B.y), clamped_row(g, up ? B.y : A.y));
        e.xr[i] = make_float2(__double2float_rd(fmin(A.x, B.x)), __double2float_ru(fmax(A.x, B.x)));
        e.kind[i] = (up ? 1 : 0) | (A.y == B.y ? 2 : 0);
    }
}

// Edges with equal end points (the common side of two polygons), paired
// through an open-addressing table of edge indices.  Pairs only: a third copy
// of an edge, or one that finds no slot within a few probes, stays single,
// which costs a test and changes no result.
__device__ __forceinline__ unsigned edge_hash(double2 l, double2 h) {
    unsigned long long v = (unsigned long long)__double_as_longlong(l.x) * 0x9E3779B97F4A7C15ULL;
    v = (v ^ (v >> 32) ^ (unsigned long long)__double_as_longlong(l.y)) * 0xC2B2AE3D27D4EB4FULL;
    v = (v ^ (v >> 29) ^ (unsigned long long)__double_as_longlong(h.x)) * 0x9E3779B97F4A7C15ULL;
    v = (v ^ (v >> 32) ^ (unsigned long long)__double_as_longlong(h.y)) * 0xC2B2AE3D27D4EB4FULL;
    return (unsigned)(v >> 32);
}

__global__ void k_pip_twins(const double2 *verts, const int *nxt, const unsigned char *kind, int V, int *table,
                            unsigned slots_mask, int *twin) {
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < V; i += gridDim.x * blockDim.x) {
        if (kind[i] & 2) continue;   // horizontal: never listed
        const bool up = kind[i] & 1;
        const double2 A = verts[i], B = verts[nxt[i]];
        const double2 l = up ? A : B, h = up ? B : A;
        unsigned at = edge_hash(l, h);
        for (int probe = 0; probe < 16; ++probe, ++at) {
            const int j = atomicCAS(&table[at & slots_mask], -1, i);
            if (j == -1) break;
            const bool uj = kind[j] & 1;
            const double2 Aj = verts[j], Bj = verts[nxt[j]];
            const double2 lj = uj ? Aj : Bj, hj = uj ? Bj : Aj;
            if (l.x == lj.x && l.y == lj.y && h.x == hj.x && h.y == hj.y) {
                if (atomicCAS(&twin[j], -1, i) == -1) twin[i] = j;
                break;
            }
        }
    }
}

// Row lists: for each (polygon, row of its MBB) the edges whose rows include
// it.  One thread per edge.  Count (ids == nullptr), then emit, with the records
// that k_pip_entries reads in list order.
__global__ void k_prow_edges(PipBuildArgs b, int *cnt, unsigned long long *total, const int *start, int *ids,
                             PipRow *out) {
    unsigned long long n = 0;
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < b.V; i += gridDim.x * blockDim.x) {
        const int P = b.owner[i], base = b.prow_base[P] - b.prow_r0[P];
        const int2 r = b.e.rows[i];
        PipRow q{};
        if (ids) {
            const float2 x = b.e.xr[i];
            const int t = b.twin[i];
            q = PipRow{i, x.x, x.y, r.x, r.y, b.e.kind[i], t >= 0 ? b.owner[t] : -1, 0};
        }
        for (int y = r.x; y <= r.y; ++y) {
            const int k = atomicAdd(&cnt[base + y], 1);
            if (ids) {
                ids[start[base + y] + k] = i;
                out[start[base + y] + k] = q;
            }
        }
        n += (unsigned long long)(r.y - r.x + 1);
    }
    if (!ids) {
        for (int o = 16; o > 0; o >>= 1) n += __shfl_xor_sync(FULL, n, o);
        if (lane_id() == 0 && n) atomicAdd(total, n);
    }
}

// x-limits of each column widened by delta, rounded outward.
__global__ void k_pip_columns(GridDev g, double delta, float2 *col) {
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < g.nx; i += gridDim.x * blockDim.x)
        col[i] = make_float2(__double2float_rd(key_value(g.kx[i]) - delta), __double2float_ru(key_value(g.kx[i + 1]) + delta));
}

// Cell of each candidate entry.
__global__ void k_pip_entry_cells(const int *cand_start, int G, int *cell) {
    for (int c = blockIdx.x * blockDim.x + threadIdx.x; c < G; c += gridDim.x * blockDim.x)
        for (int k = cand_start[c]; k < cand_start[c + 1]; ++k) cell[k] = c;
}

// The candidate entry of polygon Q in cell c when the cell has few enough
// candidates to form one group, else -1.
__device__ __forceinline__ int entry_of(const PipBuildArgs &b, int k0, int k1, int Q) {
    if (k1 - k0 > 32) return -1;
    for (int k = k0; k < k1; ++k)
        if (b.cand_ids[k] == Q) return k;
    return -1;
}

// Candidate entries, a warp each.  Count pass: near edges (a shared edge
// counted with its polygon of smaller id), flips, base parity and whether the
// entry has any near edge or flip, and whether a horizontal edge is near (ent[k]
// = near, flips << 3 | horizontal << 2 | base << 1 | any).
// Emit pass: the near edges (vid, mask) and flips (key, bit) of the relevant
// entries, unordered, at edge_at[k] / flip_at[k] in the temporary units.
// A whole warp although a (polygon, row) list holds 5 - 60 edges on average: the
// lists of thousands of a few large polygons set the time (the two passes on the
// 40,000 tiles at 768 x 768: 286 + 507 us with eight lanes an entry, 240 + 234 with
// 32; the layer build of the heavy-tail tiling 17.2 ms with 8, 9.7 with 16, 7.5
// with 32).
template <bool EMIT>
__global__ void __launch_bounds__(256) k_pip_entries(PipBuildArgs b) {
    const int lane = lane_id();
    const unsigned lt = (1u << lane) - 1u;
    const long long T = (long long)gridDim.x * blockDim.x;
    for (long long kk = ((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5; kk < b.M; kk += T >> 5) {
        const int k = (int)kk;
        const int bit = EMIT ? b.ord[k] : 0;
        if (EMIT && bit < 0) continue;
        const int c = b.entry_cell[k];
        const int iy = c / b.g.nx, ix = c - iy * b.g.nx;
        const float2 col = b.col[ix];
        const int P = b.cand_ids[k];
        const int slot = b.prow_base[P] + (iy - b.prow_r0[P]);
        const int e0 = b.prow_start[slot], e1 = b.prow_start[slot + 1];
        const int k0 = b.cand_start[c], k1 = b.cand_start[c + 1];
        const unsigned own = EMIT ? 1u << (bit & 31) : 0u;
        int n = 0, nf = 0, par = 0;
        bool any = false, level = false;
        for (int base = e0; base < e1; base += 32) {
            const int t = base + lane;
            bool is_near = false, mine = false, fl = false, fh = false, up = false;
            int i = 0, tk = -1;
            if (t < e1) {
                const PipRow q = b.rows[t];
                i = q.edge;
                up = q.kind & 1;
                if (q.x0 > col.y) {   // far
                    par ^= q.lo < iy;
                    if (q.lo == iy || q.hi == iy) {
                        // the ends inside the row, unless shared with another far edge
                        const bool a_far = b.e.xr[b.prv[i]].x > col.y, b_far = b.e.xr[b.nxt[i]].x > col.y;
                        fl = q.lo == iy && !(up ? a_far : b_far);
                        fh = q.hi == iy && !(up ? b_far : a_far);
                    }
                } else if (!(q.x1 < col.x) && (q.kind & 2)) {    // near, horizontal
                    level = true;
                } else if (!(q.x1 < col.x)) {   // near
                    is_near = mine = true;
                    if (q.twin >= 0 && q.twin != P) {
                        tk = entry_of(b, k0, k1, q.twin);
                        if (tk >= 0 && q.twin < P) mine = false;
                    }
                }
            }
            const unsigned bn = __ballot_sync(FULL, mine);
            const unsigned bl = __ballot_sync(FULL, fl), bh = __ballot_sync(FULL, fh);
            any |= __any_sync(FULL, is_near) || bl || bh;
            if (EMIT) {
                if (mine) {
                    unsigned m = own;
                    if (tk >= 0 && b.ord[tk] >= 0) m |= 1u << (b.ord[tk] & 31);
                    b.tmp_edge[b.edge_at[k] + n + __popc(bn & lt)] = make_int2(i, (int)m);
                }
                if (fl || fh) {
                    const int j = b.nxt[i];
                    PipFlipTmp *f = b.tmp_flip + b.flip_at[k] + nf + __popc(bl & lt) + __popc(bh & lt);
                    if (fl) *f++ = PipFlipTmp{y_key(b.verts[up ? i : j].y), own, 0};
                    if (fh) *f = PipFlipTmp{y_key(b.verts[up ? j : i].y), own, 0};
                }
            }
            n += __popc(bn);
            nf += __popc(bl) + __popc(bh);
        }
        if (!EMIT) {
            par = (int)__popc(__ballot_sync(FULL, par & 1)) & 1;
            level = __any_sync(FULL, level);
            if (lane == 0) b.ent[k] = make_int2(n, (nf << 3) | (level ? 4 : 0) | (par << 1) | (any ? 1 : 0));
        }
    }
}

// Cells, one thread each: the relevant candidates (ord[k] = place among them,
// or -1), the cell's code when every candidate is classified, else the size of
// its record in units, near edges and flips (for the temporary lists).
__global__ void k_pip_cells(PipBuildArgs b) {
    for (int c = blockIdx.x * blockDim.x + threadIdx.x; c < b.g.G; c += gridDim.x * blockDim.x) {
        const int k0 = b.cand_start[c], k1 = b.cand_start[c + 1];
        int rel = 0, code = -1;
        bool done = false, any = false, level = false;
        long long units = 0, tn = 0, tf = 0;
        int n = 0, nf = 0, ng = 0;
        for (int k = k0; k < k1; ++k) {
            const int2 e = b.ent[k];
            const bool bd = e.y & 1, base = e.y & 2;
            if (done || (!bd && !base)) {
                b.ord[k] = -1;
                continue;
            }
            if (!bd) {
                if (rel == 0) code = b.cand_ids[k];
                done = true;
            }
            any |= bd;
            level |= (e.y & 4) != 0;
            b.ord[k] = rel++;
            n += e.x;
            nf += e.y >> 3;
            if (++ng == 32) {
                units += group_units(n, nf, ng);
                tn += n;
                tf += nf;
                n = nf = ng = 0;
            }
        }
        if (ng) units += group_units(n, nf, ng);
        tn += n;
        tf += nf;
        if (!any) {   // classified: no record
            for (int k = k0; k < k1; ++k) b.ord[k] = -1;
            units = tn = tf = 0;
        } else {
            code = -2;
        }
        b.cells[c] = make_int4(code, level ? -1 : 0, -1, -1);   // -1: no sub-cell classes (k_pip_order)
        b.units_of[c] = (int)min(units, 2147483647LL);
        b.edges_of[c] = (int)min(tn, 2147483647LL);
        b.flips_of[c] = (int)min(tf, 2147483647LL);
    }
}

// Headers, ids and the entries' places in the temporary lists, one thread per cell.
__global__ void k_pip_heads(PipBuildArgs b) {
    for (int c = blockIdx.x * blockDim.x + threadIdx.x; c < b.g.G; c += gridDim.x * blockDim.x) {
        if (b.cells[c].x != -2) continue;
        const int k0 = b.cand_start[c], k1 = b.cand_start[c + 1];
        int off = b.units_at[c], te = b.edges_at[c], tf = b.flips_at[c];
        b.cells[c].x = -2 - off;
        long long algo = 0;
        int last = k0;   // last relevant entry
        for (int k = k0; k < k1; ++k) {
            algo += b.obj_voff[b.cand_ids[k] + 1] - b.obj_voff[b.cand_ids[k]];
            if (b.ord[k] >= 0) last = k;
        }
        for (int k = k0; k <= last;) {   // a group
            PipHead h;
            h.n = h.nf = 0;
            h.base = 0;
            h.id[0] = h.id[1] = h.id[2] = 0;
            int ng = 0, q = k;
            for (; q <= last && ng < 32; ++q) {
                if (b.ord[q] < 0) continue;
                const int2 e = b.ent[q];
                b.edge_at[q] = te + h.n;
                b.flip_at[q] = tf + h.nf;
                if (e.y & 2) h.base |= 1u << ng;
                if (ng < PIP_INLINE_IDS) h.id[ng] = b.cand_ids[q];
                h.n += e.x;
                h.nf += e.y >> 3;
                ++ng;
            }
            int4 *u = b.units + 2 * (size_t)off;
            h.ncand = min(k1 - k0, PIP_EXT - 1);
            if (ng > PIP_INLINE_IDS || h.n > PIP_SEARCH_MIN) {
                h.ncand |= PIP_EXT;
                int *ids = reinterpret_cast<int *>(u + 2 + 2 * (size_t)h.n + h.nf);
                for (int r = k, t = 0; r < q; ++r)
                    if (b.ord[r] >= 0) ids[t++] = b.cand_ids[r];
                h.id[0] = ng;
            }
            if (q <= last) h.ncand |= PIP_MORE;
            h.algo = (int)min(algo, 2147483647LL);
            u[0] = make_int4(h.n, h.nf, (int)h.base, h.ncand);
            u[1] = make_int4(h.id[0], h.id[1], h.id[2], h.algo);
            off += (int)group_units(h.n, h.nf, ng);
            te += h.n;
            tf += h.nf;
            k = q;
        }
    }
}

// The order of a near edge in its list (a NaN, possible only beyond the FP32
// range where every test goes to the FP64 rule, must not break the ranks).
__device__ __forceinline__ float list_key(float ly) { return ly == ly ? ly : 0.0f; }

__device__ __forceinline__ float4 edge_rel(const PipBuildArgs &b, int i, float2 fo) {
    const double2 A = b.verts[i], B = b.verts[b.nxt[i]];
    const bool up = b.e.kind[i] & 1;
    const double2 l = up ? A : B, h = up ? B : A;
    float a, c;
    float4 r;
    split_double(l.x, a, c); r.x = rel_coord(a, c, fo.x);
    split_double(l.y, a, c); r.y = rel_coord(a, c, fo.y);
    split_double(h.x, a, c); r.z = rel_coord(a, c, fo.x);
    split_double(h.y, a, c); r.w = rel_coord(a, c, fo.y);
    return r;
}
// An upper bound of hi.y - lo.y with both ends' rounding bounds (the search window).
__device__ __forceinline__ float edge_height(float4 r) {
    return __fadd_ru(__fsub_ru(r.w, r.y), __fmul_ru(8.0f * U32, fabsf(r.w) + fabsf(r.y)));
}
__device__ __forceinline__ float key_rel(unsigned long long key, float fo) {
    float a, c;
    split_double(key_value(key), a, c);
    return rel_coord(a, c, fo);
}

// Classes of a cell's 4 x 4 sub-cells (see the top of the file), by a warp: lane
// l takes sub-cell l & 15 with every second edge.  The sub-cell's box in cell-
// relative coordinates is widened by the margins (the classes' delta, the error
// of a point's estimated place, that of the frame origin); where an edge may
// meet it (separating axes, rounding included) or the parity at its centre is
// not certain in FP32, the class is 0.  Elsewhere every point of the sub-cell
// has the centre's result, by the argument for whole cells -- which needs every
// edge near the cell: a cell with a near horizontal edge (not in its record) has
// no classes, nor has one whose record has several groups or a long list.
template <class EdgeAt>
__device__ __forceinline__ void pip_sub_classes(const PipBuildArgs &b, int c, const int4 u0, const int4 *u, EdgeAt edge_at,
                                                float eps, int lane) {
    const int n = u0.x, nf = u0.y, sub = lane & 15;
    const float qx = 0.25f * b.cwf, qy = 0.25f * b.chf;
    const float cx = ((float)(sub & 3) + 0.5f) * qx, cy = ((float)(sub >> 2) + 0.5f) * qy;
    unsigned m = lane < 16 ? (unsigned)u0.z : 0u;
    bool bad = false;
    if (lane < 16) {   // flips at or below the centre
        const PipFlip *F = reinterpret_cast<const PipFlip *>(reinterpret_cast<const PipEdge *>(u + 2) + n);
        for (int f = 0; f < nf; ++f) {
            const float d = __fsub_rn(cy, F[f].y);
            bad |= !(fabsf(d) > diff_bound(cy, F[f].y, eps));
            if (!(d > 0.0f)) break;
            m = F[f].mask;
        }
    }
    for (int j = 0; j < n; j += 2) {
        unsigned mask;
        const float4 e = edge_at(min(j + (lane >> 4), n - 1), mask);
        if (j + (lane >> 4) >= n) continue;
        const float mag = fmaxf(fmaxf(fabsf(e.x), fabsf(e.z)), fmaxf(fabsf(e.y), fabsf(e.w)));
        const float hx = 0.5f * qx + b.sub_mx + fmaf(8.0f * U32, mag, 2.0f * eps);
        const float hy = 0.5f * qy + b.sub_my + fmaf(8.0f * U32, mag, 2.0f * eps);
        const bool box = !(fminf(e.x, e.z) > cx + hx || fmaxf(e.x, e.z) < cx - hx || e.y > cy + hy || e.w < cy - hy);
        const float dx = e.z - e.x, dy = e.w - e.y;
        const float p1 = dx * (cy - e.y), p2 = dy * (cx - e.x);
        bad |= box && !(fabsf(p1 - p2) > (fabsf(dx) * hy + fabsf(dy) * hx) + 16.0f * U32 * (fabsf(p1) + fabsf(p2)));
        const int x = bad ? 0 : edge_cross(cx, cy, e, eps);
        bad |= x < 0;
        if (x > 0) m ^= mask;
    }
    m ^= __shfl_xor_sync(FULL, m, 16);
    bad = ((__ballot_sync(FULL, bad) >> sub) & 0x10001u) != 0;
    // ids of the lowest set bits; the first two that occur get classes 1 and 2
    int id = -1;
    if (!bad && m) {
        const int k = __ffs(m) - 1;
        const int4 u1 = u[1];
        if (u0.w & PIP_EXT) id = reinterpret_cast<const int *>(u + 2 + 2 * (size_t)n + nf)[k];
        else id = k == 0 ? u1.x : (k == 1 ? u1.y : u1.z);
    }
    const unsigned some = __ballot_sync(FULL, !bad && id >= 0);
    const int id1 = some ? __shfl_sync(FULL, id, __ffs(some) - 1) : -1;
    const unsigned more = __ballot_sync(FULL, !bad && id >= 0 && id != id1);
    const int id2 = more ? __shfl_sync(FULL, id, __ffs(more) - 1) : -1;
    const unsigned cls = bad ? 0u : (id < 0 ? 3u : (id == id1 ? 1u : (id == id2 ? 2u : 0u)));
    const unsigned all = __reduce_or_sync(FULL, lane < 16 ? cls << (2 * sub) : 0u);
    if (lane == 0) {
        b.cells[c].y = (int)all;
        b.cells[c].z = id1;
        b.cells[c].w = id2;
    }
}

// Record groups larger than this are ordered by a whole block (k_pip_order_long).
constexpr int PIP_LONG = PIP_LONG_MIN;

// The records' edges (ordered by lower y) and flips (ordered by key, masks
// accumulated), a warp per cell: each element's place is its rank.
__global__ void __launch_bounds__(256) k_pip_order(PipBuildArgs b) {
    const int lane = lane_id();
    const long long T = (long long)gridDim.x * blockDim.x;
    for (long long cc = ((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5; cc < b.g.G; cc += T >> 5) {
        const int c = (int)cc;
        const int2 cell = *reinterpret_cast<const int2 *>(&b.cells[c]);   // code, -1: a horizontal edge
        const int code = cell.x;
        if (code >= -1) continue;
        const float2 fo = cell_frame(b.frame_x, b.frame_y, b.g.nx, c);
        int off = -2 - code, te = b.edges_at[c], tf = b.flips_at[c];
        __syncwarp();
        if (cell.y && lane == 0) b.cells[c].y = 0;
        while (true) {
            int4 *u = b.units + 2 * (size_t)off;
            const int4 u0 = u[0];
            const int n = u0.x, nf = u0.y;
            if (n > PIP_LONG || nf > PIP_LONG) {
                if (lane == 0) b.long_list[atomicAdd(b.long_n, 1)] = make_int4(off, c, te, tf);
            } else {
                PipEdge *E = reinterpret_cast<PipEdge *>(u + 2);
                float hmax = 0.0f;
                int2 v = make_int2(0, 0);
                float4 r = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
                if (n <= 32) {   // in registers
                    if (lane < n) {
                        v = b.tmp_edge[te + lane];
                        r = edge_rel(b, v.x, fo);
                        hmax = edge_height(r);
                    }
                    const float key = list_key(r.y);
                    int rank = 0;
                    for (int j = 0; j < n; ++j) {
                        const float kj = __shfl_sync(FULL, key, j);
                        rank += kj < key || (kj == key && j < lane);
                    }
                    if (lane < n) {
                        reinterpret_cast<float4 *>(E + rank)[0] = r;
                        reinterpret_cast<int4 *>(E + rank)[1] = make_int4(v.x, v.y, 0, 0);
                    }
                } else {
                    for (int i = lane; i < n; i += 32) {
                        const float4 r = edge_rel(b, b.tmp_edge[te + i].x, fo);
                        b.tmp_rel[te + i] = r;
                        hmax = fmaxf(hmax, edge_height(r));
                    }
                    __syncwarp();
                    for (int i = lane; i < n; i += 32) {
                        const float4 r = b.tmp_rel[te + i];
                        const int2 v = b.tmp_edge[te + i];
                        const float key = list_key(r.y);
                        int rank = 0;
#pragma unroll 4
                        for (int j = 0; j < n; ++j) {
                            const float kj = list_key(b.tmp_rel[te + j].y);
                            rank += kj < key || (kj == key && j < i);
                        }
                        reinterpret_cast<float4 *>(E + rank)[0] = r;
                        reinterpret_cast<int4 *>(E + rank)[1] = make_int4(v.x, v.y, 0, 0);
                    }
                }
                if (u0.w & PIP_EXT) {
                    for (int o = 16; o > 0; o >>= 1) hmax = fmaxf(hmax, __shfl_xor_sync(FULL, hmax, o));
                    if (lane == 0) reinterpret_cast<int *>(u)[5] = __float_as_int(hmax);
                }
                PipFlip *F = reinterpret_cast<PipFlip *>(E + n);
                for (int i = lane; i < nf; i += 32) {
                    const PipFlipTmp v = b.tmp_flip[tf + i];
                    int rank = 0;
                    unsigned m = (unsigned)u0.z;
                    for (int j = 0; j < nf; ++j) {
                        const PipFlipTmp w = b.tmp_flip[tf + j];
                        const bool before = w.key < v.key || (w.key == v.key && j <= i);
                        rank += before;
                        if (before) m ^= w.mask;
                    }
                    F[rank - 1] = PipFlip{key_rel(v.key, fo.y), m, v.key};
                }
                if (b.sub_mx >= 0.0f && cell.y == 0 && !(u0.w & PIP_MORE) && off == -2 - code) {   // one group
                    __syncwarp();
                    if (n <= 32) {
                        pip_sub_classes(b, c, u0, u, [&](int j, unsigned &mask) {
                            mask = (unsigned)__shfl_sync(FULL, v.y, j);
                            return make_float4(__shfl_sync(FULL, r.x, j), __shfl_sync(FULL, r.y, j),
                                               __shfl_sync(FULL, r.z, j), __shfl_sync(FULL, r.w, j));
                        }, b.eps, lane);
                    } else {
                        pip_sub_classes(b, c, u0, u, [&](int j, unsigned &mask) {
                            mask = (unsigned)b.tmp_edge[te + j].y;
                            return b.tmp_rel[te + j];
                        }, b.eps, lane);
                    }
                }
            }
            if (!(u0.w & PIP_MORE)) break;
            off += (int)group_units(n, nf, u[1].x);
            te += n;
            tf += nf;
        }
    }
}

// Sort of n elements by a block, in place: the bitonic network in the form
// whose compare-exchanges all put the smaller element first, which sorts any n
// when partners beyond n are skipped.
template <class Less, class Swap>
__device__ __forceinline__ void block_sort(int n, Less less, Swap swap) {
    auto pass = [&](auto partner) {
        for (long long i = threadIdx.x; i < n; i += blockDim.x) {
            const long long j = partner(i);
            if (j > i && j < n && less((int)j, (int)i)) swap((int)i, (int)j);
        }
        __syncthreads();
    };
    for (long long k = 2; k < 2LL * n; k <<= 1) {
        pass([&](long long i) { return i ^ (k - 1); });
        for (long long h = k >> 2; h > 0; h >>= 1) pass([&](long long i) { return i ^ h; });
    }
}

__global__ void __launch_bounds__(512) k_pip_order_long(PipBuildArgs b) {
    __shared__ int hbits;
    const int total = *b.long_n;
    for (int g = blockIdx.x; g < total; g += gridDim.x) {
        const int4 q = b.long_list[g];
        const float2 fo = cell_frame(b.frame_x, b.frame_y, b.g.nx, q.y);
        int4 *u = b.units + 2 * (size_t)q.x;
        const int4 u0 = u[0];
        const int n = u0.x, nf = u0.y;
        PipEdge *E = reinterpret_cast<PipEdge *>(u + 2);
        PipFlip *F = reinterpret_cast<PipFlip *>(E + n);
        float4 *rel = b.tmp_rel + q.z;
        int2 *tv = b.tmp_edge + q.z;
        PipFlipTmp *fl = b.tmp_flip + q.w;
        if (threadIdx.x == 0) hbits = 0;
        __syncthreads();
        float hmax = 0.0f;
        for (int i = threadIdx.x; i < n; i += blockDim.x) {
            rel[i] = edge_rel(b, tv[i].x, fo);
            hmax = fmaxf(hmax, edge_height(rel[i]));
        }
        if (hmax > 0.0f) atomicMax(&hbits, __float_as_int(hmax));   // positive floats order as ints
        __syncthreads();
        block_sort(n, [&](int i, int j) { return list_key(rel[i].y) < list_key(rel[j].y); },
                   [&](int i, int j) {
                       const float4 r = rel[i]; rel[i] = rel[j]; rel[j] = r;
                       const int2 v = tv[i]; tv[i] = tv[j]; tv[j] = v;
                   });
        block_sort(nf, [&](int i, int j) { return fl[i].key < fl[j].key; },
                   [&](int i, int j) { const PipFlipTmp v = fl[i]; fl[i] = fl[j]; fl[j] = v; });
        for (int i = threadIdx.x; i < n; i += blockDim.x) {
            reinterpret_cast<float4 *>(E + i)[0] = rel[i];
            reinterpret_cast<int4 *>(E + i)[1] = make_int4(tv[i].x, tv[i].y, 0, 0);
        }
        if (threadIdx.x == 0) {
            if (u0.w & PIP_EXT) reinterpret_cast<int *>(u)[5] = hbits;
            unsigned m = (unsigned)u0.z;
            for (int i = 0; i < nf; ++i) {
                m ^= fl[i].mask;
                F[i] = PipFlip{key_rel(fl[i].key, fo.y), m, fl[i].key};
            }
        }
        __syncthreads();
    }
}

static int grid_for(long long n, int per, int cap) {
    return (int)std::max(1LL, std::min((n + per - 1) / per, (long long)cap));
}

cudaError_t launch_pip_edges(const PipBuildArgs &b, cudaStream_t s) {
    k_pip_edges<<<grid_for(b.V, 256, 8192), 256, 0, s>>>(b.g, b.verts, b.nxt, b.V, b.e);
    return cudaGetLastError();
}
cudaError_t launch_pip_twins(const PipBuildArgs &b, int *table, unsigned slots, cudaStream_t s) {
    cudaError_t e = cudaMemsetAsync(table, 0xff, sizeof(int) * (size_t)slots, s);
    if (e == cudaSuccess) e = cudaMemsetAsync(b.twin, 0xff, sizeof(int) * (size_t)b.V, s);
    if (e != cudaSuccess) return e;
    k_pip_twins<<<grid_for(b.V, 256, 8192), 256, 0, s>>>(b.verts, b.nxt, b.e.kind, b.V, table, slots - 1, b.twin);
    return cudaGetLastError();
}
cudaError_t launch_prow_edges(const PipBuildArgs &b, int *cnt, unsigned long long *total, const int *start, int *ids,
                              PipRow *rows, cudaStream_t s) {
    k_prow_edges<<<grid_for(b.V, 256, 8192), 256, 0, s>>>(b, cnt, total, start, ids, rows);
    return cudaGetLastError();
}
// Step 1: what each candidate entry and cell holds.
cudaError_t launch_pip_count(const PipBuildArgs &b, double delta, cudaStream_t s) {
    k_pip_columns<<<grid_for(b.g.nx, 256, 4096), 256, 0, s>>>(b.g, delta, b.col);
    k_pip_entry_cells<<<grid_for(b.g.G, 256, 8192), 256, 0, s>>>(b.cand_start, b.g.G, b.entry_cell);
    k_pip_entries<false><<<grid_for(32LL * b.M, 256, 32768), 256, 0, s>>>(b);
    k_pip_cells<<<grid_for(b.g.G, 256, 8192), 256, 0, s>>>(b);
    return cudaGetLastError();
}
// Step 2: the records (units, temporary lists and offsets allocated).
cudaError_t launch_pip_records(const PipBuildArgs &b, cudaStream_t s) {
    k_pip_heads<<<grid_for(b.g.G, 256, 8192), 256, 0, s>>>(b);
    k_pip_entries<true><<<grid_for(32LL * b.M, 256, 32768), 256, 0, s>>>(b);
    k_pip_order<<<grid_for(32LL * b.g.G, 256, 32768), 256, 0, s>>>(b);
    k_pip_order_long<<<152 * 2, 512, 0, s>>>(b);
    return cudaGetLastError();
}

// ------------------------------------------------------------------ census

// Census of the algorithmic PIP work (a measurement pass, not part of a
// join): for every in-grid point, out[0] += the edges of its cell's candidate
// polygons (every ring), out[1] += how many of them straddle the point's y
// under the crossing rule's straddle test (Sec. III.C).  Only an edge of a
// candidate's list for the point's grid row can straddle it (the row lists are
// exact), so the straddles are counted over those lists.  One thread per point.
__global__ void k_pip_census(CensusArgs a, const double2 *pts, int n, unsigned long long *out) {
    unsigned long long e = 0, st = 0;
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
        const double2 p = pts[i];
        const int c = point_cell(a.g, p.x, p.y);
        if (c >= a.g.G) continue;
        const int iy = c / a.g.nx;
        for (int k = a.cand_start[c]; k < a.cand_start[c + 1]; ++k) {
            const int P = a.cand_ids[k];
            e += (unsigned long long)(a.obj_voff[P + 1] - a.obj_voff[P]);
            const int slot = a.prow_base[P] + (iy - a.prow_r0[P]);
            for (int t = a.prow_start[slot]; t < a.prow_start[slot + 1]; ++t) {
                const int v = a.pedge_ids[t];
                st += (unsigned long long)((a.verts[v].y > p.y) != (a.verts[a.nxt[v]].y > p.y));
            }
        }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        e += __shfl_xor_sync(FULL, e, o);
        st += __shfl_xor_sync(FULL, st, o);
    }
    if (lane_id() == 0) {
        atomicAdd(&out[0], e);
        atomicAdd(&out[1], st);
    }
}

cudaError_t launch_pip_census(const CensusArgs &a, const double2 *pts, int n, unsigned long long *out,
                              cudaStream_t s) {
    const int nb = std::max(1, std::min((n + 255) / 256, 152 * 16));
    k_pip_census<<<nb, 256, 0, s>>>(a, pts, n, out);
    return cudaGetLastError();
}

}  // namespace sj

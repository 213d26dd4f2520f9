// sj_p2p.cu -- P2P refinement (Sec. III.B, Fig. 2): for every point of a work
// item, the candidate polyline at the smallest distance, accepted when the
// distance is within the window D.
//
// Work decomposition: one warp per (cell, point-chunk) item.
//   1. The item's points are converted to cell-relative coordinates and their
//      bounding box is reduced across the warp.
//   2. The cell's segment list -- every segment of the candidate polylines
//      whose box widened by D meets the cell, built with the layer; the others
//      are farther than D from every point of the cell -- is read 32 entries
//      at a time, one per lane, as records prepared with the layer (the
//      segment relative to this cell's FP32 frame, its owner and magnitude).
//   3. Staging: a segment whose bounding box is farther than D (plus a
//      rounding slack) from the points' box cannot be within D of any point of
//      the item and is dropped (exact: it cannot change any result); the others
//      are compacted into shared memory (a, e = b - a, 1 / |e|^2, a tag) with a
//      ballot.
//   4. The warp takes the item's points in rounds.  Each splits the lanes into
//      point groups of SG lanes (SG so that the round's points fill the warp);
//      each lane strides over the staged segments keeping the smallest squared
//      distances of its point, and the SG lanes of a group fold theirs with
//      shuffles (the cross-lane min of the vertex-per-lane alternative of
//      Sec. III.B); the point's record is made from the fold in registers.  The
//      few lists that fill the staging area more than once are staged part by
//      part in every round, so no state of a point lives in shared memory: what
//      the kernel does not take there is L1, which holds the records that the
//      items of a cell share.
//
// The point-to-segment distance is the two-case distance of Fig. 2 written as
// the clamped projection: t = clamp(((p - a) . e) / |e|^2, 0, 1) and
// d^2 = |p - a - t e|^2 (t = 0 or 1 gives the nearer end, 0 < t < 1 the
// perpendicular foot; a zero-length segment has 1 / |e|^2 = 0, hence t = 0).
//
// Both forms test the segments in FP32 on cell-relative coordinates (from the
// (hi, lo) split of the FP64 inputs): every distance carries the bound
// E = 64 u M + 4 eps (u = 2^-24, M the largest |coordinate| of the point and of
// the item's staged segments).
//   FP32X  -- keeps the best polyline and the best distance of any other one
//             (tag: polyline id).  A point is final only when its best polyline
//             is ahead of the runner-up by more than 2E and its distance
//             differs from D by more than E; the result is the FP32 distance.
//   FP64   -- keeps the best two segments and the third-best distance (tag:
//             segment).  A segment more than 2E behind the best cannot hold the
//             smallest FP64 distance, so the FP64 formula is evaluated for the
//             best one, for the second when it is within 2E (the two segments
//             of a vertex), and the result is the smallest (d^2, id) of all
//             segments in FP64 arithmetic, bit for bit.
// A point that this does not settle (FP32X: not certified; FP64: three
// segments within 2E) is queued and redone in FP64 over its cell's whole list
// (k_p2p_recheck).  Either way the point's slot ends up with an 8-byte record
// (P2PRec), from which k_p2p_finish* makes the outputs in input order.
//
// FP64 arithmetic runs at 1/64 of the FP32 rate (a warp instruction holds the
// SM's FP64 pipe for 16 cycles), which is what the FP64 form is bound by: all
// tests in FP64 took 3.33 ms for 3 M points on the 100,000 walks (106 M tests).
// The one or two evaluations that a point needs are left to the finishing
// kernel, whose warps are full of points: made at the end of each item, with
// half of the lanes idle, they still took most of the refinement (0.43 ms).
// Now the FP64 form's refinement takes 0.27 ms and its finishing 0.13 ms there,
// the join 0.50 ms instead of 3.50.
#include <cuda_runtime.h>

#include <algorithm>

#include "sj_internal.cuh"

namespace sj {

unsigned bounds_take_p2p() { return bounds_take(); }

constexpr int P2P_WARPS = 4;

// Staging holds segments in pairs (2k, 2k + 1), each quantity of the
// pair side by side, so that one lane evaluates both with the packed FP32
// instructions (FADD2 / FMUL2 / FFMA2: two IEEE round-to-nearest operations
// each, the same roundings as the scalar ones).  The stored values are
// negated (-a, -e, -1 / |e|^2), which keeps every packed operation an add or
// a fused multiply-add of the stored operands; the arithmetic is the clamped
// projection below, operation for operation.
template <bool F64>
struct Best;
// FP32X: smallest squared distance, its polyline, smallest of any other polyline.
template <>
struct Best<false> {
    float b1, b2;
    int i1;
};
// FP64: the two smallest with their segments, and the third.
template <>
struct Best<true> {
    float b1, b2, b3;
    int i1, i2;
};

struct P2PSmem {
    static constexpr int SMAX = 128;   // even
    float4 sa[SMAX / 2];     // (-ax, -ax', -ay, -ay') cell-relative
    float4 se[SMAX / 2];     // (-ex, -ex', -ey, -ey')
    float4 si[SMAX / 2];     // (-1 / |e|^2, -1 / |e'|^2, tag, tag')
    float2 pt[MAX_CH];
};

// Squared distance from p to the segment (a, a + e) by the clamped projection:
// d = p - a, t = clamp((e . d) / |e|^2, 0, 1), |d - t e|^2, each operation
// rounded once (FP64 here; the loop in p2p_compute evaluates the same
// operations in FP32 on segment pairs).
__device__ __forceinline__ double seg_d2(double px, double py, double ax, double ay, double ex, double ey,
                                         double inv) {
    double dx = __dsub_rn(px, ax), dy = __dsub_rn(py, ay);
    double t = __dmul_rn(__fma_rn(ex, dx, __dmul_rn(ey, dy)), inv);
    t = fmin(fmax(t, 0.0), 1.0);
    double qx = __fma_rn(-t, ex, dx), qy = __fma_rn(-t, ey, dy);
    return __fma_rn(qx, qx, __dmul_rn(qy, qy));
}

__device__ __forceinline__ Best<false> best_none(Best<false> *) {
    const float INF = __int_as_float(0x7f800000);
    return Best<false>{INF, INF, -1};
}
__device__ __forceinline__ Best<true> best_none(Best<true> *) {
    const float INF = __int_as_float(0x7f800000);
    return Best<true>{INF, INF, INF, -1, -1};
}

// A further segment at squared distance d with tag l.
__device__ __forceinline__ void consider(Best<false> &s, float d, int l) {
    // b1 <= b2 always; the runner-up becomes max(d, b1) when l is another
    // polyline (whichever of the old best and d is not the new best).
    const bool lt = d < s.b1;
    const float nb2 = (l == s.i1) ? s.b2 : fminf(s.b2, fmaxf(d, s.b1));
    s.b1 = fminf(s.b1, d);
    s.i1 = lt ? l : s.i1;
    s.b2 = nb2;
}
__device__ __forceinline__ void consider(Best<true> &s, float d, int l) {
    const bool lt1 = d < s.b1, lt2 = d < s.b2;
    s.b3 = fminf(s.b3, fmaxf(d, s.b2));
    s.b2 = fminf(s.b2, fmaxf(d, s.b1));
    s.b1 = fminf(s.b1, d);
    s.i2 = lt1 ? s.i1 : (lt2 ? l : s.i2);
    s.i1 = lt1 ? l : s.i1;
}

// Result over the union of two disjoint segment sets (commutative and associative).
__device__ __forceinline__ Best<false> merge(Best<false> A, Best<false> B) {
    Best<false> r;
    if (A.i1 == B.i1) {
        r.b1 = fminf(A.b1, B.b1); r.i1 = A.i1; r.b2 = fminf(A.b2, B.b2);
    } else if (B.b1 < A.b1 || (B.b1 == A.b1 && B.i1 < A.i1)) {
        r.b1 = B.b1; r.i1 = B.i1; r.b2 = fminf(B.b2, A.b1);
    } else {
        r.b1 = A.b1; r.i1 = A.i1; r.b2 = fminf(A.b2, B.b1);
    }
    return r;
}
__device__ __forceinline__ Best<true> merge(Best<true> A, Best<true> B) {
    consider(A, B.b1, B.i1);
    consider(A, B.b2, B.i2);
    A.b3 = fminf(A.b3, B.b3);
    return A;
}
__device__ __forceinline__ Best<false> shfl_best(const Best<false> &s, int o) {
    return Best<false>{__shfl_xor_sync(FULL, s.b1, o), __shfl_xor_sync(FULL, s.b2, o), __shfl_xor_sync(FULL, s.i1, o)};
}
__device__ __forceinline__ Best<true> shfl_best(const Best<true> &s, int o) {
    return Best<true>{__shfl_xor_sync(FULL, s.b1, o), __shfl_xor_sync(FULL, s.b2, o), __shfl_xor_sync(FULL, s.b3, o),
                      __shfl_xor_sync(FULL, s.i1, o), __shfl_xor_sync(FULL, s.i2, o)};
}

// FP64 result of one point over some segments: the smallest (squared distance,
// polyline id), and a segment that has it.
struct Best64 {
    double d2;
    int id, seg;
};
__device__ __forceinline__ void consider64(Best64 &s, double d2, int id, int seg) {
    if (d2 < s.d2 || (d2 == s.d2 && id < s.id)) s = Best64{d2, id, seg};
}
// Squared distance from p to segment i, FP64.
__device__ __forceinline__ double seg_d2(const SegArgs &a, double2 p, int i) {
    const double2 v = a.verts[i], e = a.seg_e64[i];
    return seg_d2(p.x, p.y, v.x, v.y, e.x, e.y, a.seg_inv64[i]);
}
__device__ __forceinline__ int seg_owner(const SegArgs &a, int i) { return __float_as_int(a.seg32[i].w); }

// A window w in FP32, rounded down / up with the same 1e-12 relative margin
// the layer's D gets on the host (explicit roundings, no contraction).
__device__ __forceinline__ void window_f32(double w, float &dn, float &up) {
    dn = __double2float_rd(__dmul_rn(w, 1.0 - 1e-12));
    up = __double2float_ru(__dadd_rn(__dmul_rn(w, 1.0 + 1e-12), 1e-300));
}

// Warp-wide min / max of a float (no NaN) in one integer reduction: flipping
// the magnitude bits of negative floats makes signed-integer order equal
// float order (-0 sorts just below +0).
__device__ __forceinline__ int float_key(float v) {
    const int i = __float_as_int(v);
    return i ^ ((i >> 31) & 0x7fffffff);
}
__device__ __forceinline__ float key_float(int k) { return __int_as_float(k ^ ((k >> 31) & 0x7fffffff)); }
__device__ __forceinline__ float warp_min(float v) { return key_float(__reduce_min_sync(FULL, float_key(v))); }
__device__ __forceinline__ float warp_max(float v) { return key_float(__reduce_max_sync(FULL, float_key(v))); }

// What one point's result needs besides its fold.
struct P2PItem {
    int c;          // cell
    float mag;      // largest |cell-relative coordinate| of the item's points and staged segments
};

// The record of slot j (point pt, cell-relative) from its complete fold; a
// point that it does not settle is queued for the FP64 recheck.
template <bool F64, bool PW>
__device__ __forceinline__ void p2p_result(const RefineArgs &a, const P2PItem &it, int j, float2 pt, const Best<F64> &st,
                                           bool pw, unsigned &c_fb, unsigned &c_hits) {
    const float d = sqrtf(st.b1), d2 = sqrtf(st.b2);
    const float e = fmaf(64.0f * U32, fmaxf(it.mag, fmaxf(fabsf(pt.x), fabsf(pt.y))), 4.0f * a.eps_abs) *
                    (1.0f + 8.0f * U32);
    const float sep = 2.0f * e * (1.0f + 4.0f * U32);
    float Ddn = a.Ddn, Dup = a.Dup;
    if (PW && pw) window_f32(a.win[j], Ddn, Dup);
    P2PRec r{-1, -1};
    bool redo = false;
    // e infinite: coordinates beyond the range of the bound (every point is redone)
    if (!(e < __int_as_float(0x7f800000))) {
        redo = true;
    } else if (st.i1 >= 0 && !((d - e) * (1.0f - 4.0f * U32) > Dup)) {   // not certainly outside the window
        const bool alone = (d2 - d) * (1.0f - 4.0f * U32) > sep;         // no other one within 2E
        if constexpr (F64) {
            redo = !((sqrtf(st.b3) - d) * (1.0f - 4.0f * U32) > sep);
            r = P2PRec{st.i1, alone ? -1 : st.i2};
        } else {
            const bool in_window = (d + e) * (1.0f + 4.0f * U32) < Ddn;
            redo = !(in_window && alone);
            r = P2PRec{st.i1, __float_as_int(d)};
        }
    }
    if (redo) {
        const int slot = atomicAdd(a.n_fb, 1);
        a.fb[slot] = make_int2(j, it.c);
        ++c_fb;
    } else if (SJ_IN_BOUNDS(j < a.npts, BND_P2P_RES)) {
        a.rec[j] = r;
        if (!F64) c_hits += r.id >= 0;
    }
}

// PW: per-point windows (a.win_on set; batched rounds).  The direct joins use
// PW = false, whose code has no window load at all.  32 warps per SM: 64
// registers without spills.
template <bool F64, bool PW, int NW>
__global__ void __launch_bounds__(NW * 32, 32 / NW) k_p2p_refine(RefineArgs a) {
    constexpr int SMAX = P2PSmem::SMAX;
    extern __shared__ __align__(16) unsigned char p2p_smem_raw[];
    const int lane = lane_id(), w = threadIdx.x >> 5;
    P2PSmem &s = reinterpret_cast<P2PSmem *>(p2p_smem_raw)[w];
    const int n_items = *a.n_items;
    const float FINF = __int_as_float(0x7f800000);
    const unsigned lt_mask = (1u << lane) - 1u;
    unsigned long long c_tests = 0, c_items = 0;
    unsigned c_fb = 0, c_hits = 0;
    const bool pw = PW && *a.win_on;   // per-point windows in this launch (uniform)

    // Items come from a device counter when a.work_next is set (the next index
    // is fetched at the start of an item, so its latency hides behind the
    // item), else in a fixed stride.
    // The next item's record and its cell's point range are loaded while the
    // current item is refined, off the per-item chain of dependent loads.
    // A warp takes a.claim consecutive items per counter update: consecutive
    // items are mostly chunks of one cell, whose segment records are then
    // still in L1 for the second chunk.
    const int claim = a.claim > 1 ? a.claim : 1;
    int it = blockIdx.x * NW + w, it_end = it + 1;
    if (a.work_next) {
        int t0 = 0;
        if (lane == 0) t0 = atomicAdd(a.work_next, claim);
        it = __shfl_sync(FULL, t0, 0);
        it_end = it + claim;
    }
    int2 item = make_int2(0, 0);
    int cs0 = 0, cs1 = 0;
    if (it < n_items) {
        item = a.items[it];
        cs0 = a.cell_start[item.x];
        cs1 = a.cell_start[item.x + 1];
    }
    while (it < n_items) {
        int it_next = it + gridDim.x * NW;
        const bool in_claim = it + 1 < it_end;
        if (a.work_next) {
            if (in_claim) it_next = it + 1;
            else if (lane == 0) it_next = atomicAdd(a.work_next, claim);
        }
        ++c_items;
        const int c = item.x;
        const int j0 = cs0 + item.y;
        const int np = min(cell_chunk(a.ch, a.budget > 0 ? a.cell_work[c] : 0, a.budget), cs1 - j0);
        const float2 fo = cell_frame(a.frame_x, a.frame_y, a.g.nx, c);

        // 1. points: cell-relative FP32 coordinates, their box and magnitude
        float bxlo = FINF, bxhi = -FINF, bylo = FINF, byhi = -FINF;
        // The (up to MAX_CH / 32) point loads of a lane are issued together --
        // every slot index, then every point as an asynchronous copy into the
        // (idle) staging area -- so that their latencies overlap instead of
        // forming one chain per point.
        constexpr int PQ = MAX_CH / 32;
        static_assert(sizeof(P2PSmem::sa) + sizeof(P2PSmem::se) >= MAX_CH * sizeof(double2), "");
        double2 *pbuf = reinterpret_cast<double2 *>(&s.sa[0]);   // sa and se, contiguous
        {
            int src[PQ];
#pragma unroll
            for (int u = 0; u < PQ; ++u) {
                const int q = lane + 32 * u;
                src[u] = (q < np && SJ_IN_BOUNDS(j0 + q < a.npts, BND_P2P_POINT)) ? (a.spts ? j0 + q : a.perm[j0 + q])
                                                                                 : -1;
            }
#pragma unroll
            for (int u = 0; u < PQ; ++u)
                if (src[u] >= 0 && SJ_IN_BOUNDS(src[u] < a.npts, BND_P2P_POINT))
                    copy16_async(pbuf + lane + 32 * u, a.spts ? a.spts + src[u] : a.pts + src[u]);
            copy_async_wait_all();
        }
        for (int q = lane; q < np; q += 32) {
            const double2 p = pbuf[q];
            float hx, lx, hy, ly;
            split_double(p.x, hx, lx);
            split_double(p.y, hy, ly);
            const float rx = rel_coord(hx, lx, fo.x), ry = rel_coord(hy, ly, fo.y);
            s.pt[q] = make_float2(rx, ry);
            bxlo = fminf(bxlo, rx); bxhi = fmaxf(bxhi, rx);
            bylo = fminf(bylo, ry); byhi = fmaxf(byhi, ry);
        }
        __syncwarp();   // every lane is done with the point buffer before staging reuses it
        bxlo = warp_min(bxlo); bylo = warp_min(bylo);
        bxhi = warp_max(bxhi); byhi = warp_max(byhi);
        // largest |coordinate| of the points: the larger magnitude of the box's ends
        const float pmag = fmaxf(fmaxf(fabsf(bxlo), fabsf(bxhi)), fmaxf(fabsf(bylo), fabsf(byhi)));
        if (a.work_next) it_next = __shfl_sync(FULL, it_next, 0);
        const int end_next = in_claim ? it_end : it_next + (a.work_next ? claim : 1);
        int2 item_n = make_int2(0, 0);
        if (it_next < n_items) item_n = a.items[it_next];
        float mag = pmag;   // largest |cell-relative coordinate| refined for this item

        // 2. the cell's segment list, 32 segments at a time (one per lane),
        // 3. staging with the exact distance prune, 4. rounds of points
        const int g0 = a.cseg_start[c], g1 = a.cseg_start[c + 1];
        int base = g0, nst = 0, q0 = 0, sg = 0;
        bool fill = true, parts = false;
        Best<F64> st = best_none((Best<F64> *)nullptr);
        while (true) {
            if (fill) {
                __syncwarp();   // no lane still reads what the fill overwrites
                nst = 0;
                while (base < g1 && nst <= SMAX - 32) {
                    const int g = base + lane;
                    bool keep = false;
                    int tag = 0;
                    float ax = 0.0f, ay = 0.0f, ex = 0.0f, ey = 0.0f, inv = 0.0f, smag = 0.0f;
                    if (g < g1 && SJ_IN_BOUNDS(g < a.cseg_start[a.g.G], BND_P2P_REC)) {
                        const float4 r0 = a.cseg_rec[2 * (size_t)g], r1 = a.cseg_rec[2 * (size_t)g + 1];
                        ax = r0.x;
                        ay = r0.y;
                        ex = r0.z;
                        ey = r0.w;
                        inv = r1.x;
                        tag = __float_as_int(F64 ? r1.w : r1.y);   // segment or polyline
                        smag = r1.z;
                        const float bx = ax + ex, by = ay + ey;
                        const float gx = fmaxf(0.0f, fmaxf(fminf(ax, bx) - bxhi, bxlo - fmaxf(ax, bx)));
                        const float gy = fmaxf(0.0f, fmaxf(fminf(ay, by) - byhi, bylo - fmaxf(ay, by)));
                        // rounding slack of the relative coordinates of both boxes (far above it)
                        const float lim = a.Df * (1.0f + 1e-6f) + 8.0f * U32 * (smag + pmag) + 8.0f * a.eps_abs;
                        keep = gx * gx + gy * gy <= lim * lim * (1.0f + 8.0f * U32);
                    }
                    const unsigned bal = __ballot_sync(FULL, keep);
                    if (keep) {
                        const int pos = nst + __popc(bal & lt_mask);
                        const int k = pos >> 1, h = pos & 1;
                        float *A = reinterpret_cast<float *>(&s.sa[k]);
                        float *E = reinterpret_cast<float *>(&s.se[k]);
                        float *I = reinterpret_cast<float *>(&s.si[k]);
                        A[h] = -ax; A[2 + h] = -ay;
                        E[h] = -ex; E[2 + h] = -ey;
                        I[h] = -inv; I[2 + h] = __int_as_float(tag);
                        mag = fmaxf(mag, smag);
                    }
                    nst += __popc(bal);
                    base += 32;
                }
                // an odd count: the pair's second slot gets a segment at
                // infinite distance (a far point, zero length), which never
                // changes a point's fold
                if ((nst & 1) && lane == 0) {
                    const int k = nst >> 1;
                    reinterpret_cast<float *>(&s.sa[k])[1] = -3.0e38f;
                    reinterpret_cast<float *>(&s.sa[k])[3] = -3.0e38f;
                    reinterpret_cast<float *>(&s.se[k])[1] = 0.0f;
                    reinterpret_cast<float *>(&s.se[k])[3] = 0.0f;
                    reinterpret_cast<float *>(&s.si[k])[1] = 0.0f;
                    reinterpret_cast<float *>(&s.si[k])[3] = __int_as_float(-2);
                }
                __syncwarp();
                parts |= base < g1;
            }
            const int ns = (nst + 1) >> 1, rem = np - q0;
            if (sg == 0) {   // a round begins: one lane per point while 32 remain, then groups that fill the warp
                sg = rem > 16 ? 1 : min(1 << (__clz(rem - 1) - 27), parts ? 32 : 1 << (32 - __clz(max(ns, 1) - 1)));
            }
            const int lg = __ffs(sg) - 1;
            const int sub = lane & (sg - 1), q = q0 + (lane >> lg);
            const float2 p = s.pt[min(q, np - 1)];
            if (q < np) {
                // the squared distances of the pair by the clamped projection
                // in FP32: dx = px - ax, t = sat(fma(ex, dx, ey * dy) / |e|^2),
                // q = fma(-t, e, d), |q|^2 = fma(qx, qx, qy * qy), written with
                // the negated operands (p + (-a) = p - a, fma(-ex, dx, -ey * dy)
                // * (-1 / |e|^2) = (e . d) / |e|^2, fma(t, -e, d) = d - t e:
                // each rounding the same as the unnegated one)
                const float2 px = make_float2(p.x, p.x), py = make_float2(p.y, p.y);
#pragma unroll 1
                for (int t = sub; t < ns; t += sg) {
                    const float4 A = s.sa[t], E = s.se[t], I = s.si[t];
                    const float2 nex = make_float2(E.x, E.y), ney = make_float2(E.z, E.w);
                    const float2 dx = __fadd2_rn(px, make_float2(A.x, A.y));
                    const float2 dy = __fadd2_rn(py, make_float2(A.z, A.w));
                    const float2 w2 = __ffma2_rn(nex, dx, __fmul2_rn(ney, dy));
                    const float2 tt =
                        make_float2(__saturatef(__fmul_rn(w2.x, I.x)), __saturatef(__fmul_rn(w2.y, I.y)));
                    const float2 qx = __ffma2_rn(tt, nex, dx), qy = __ffma2_rn(tt, ney, dy);
                    const float2 d = __ffma2_rn(qx, qx, __fmul2_rn(qy, qy));
                    consider(st, d.x, __float_as_int(I.z));
                    consider(st, d.y, __float_as_int(I.w));
                }
            }
            const int pg = 32 >> lg;
            c_tests += (unsigned long long)min(rem, pg) * (unsigned long long)nst;
            if (base < g1) {   // the list's next part
                fill = true;
                continue;
            }
            for (int o = sg >> 1; o > 0; o >>= 1) st = merge(st, shfl_best(st, o));
            const float m = warp_max(mag);
            if (sub == 0 && q < np) p2p_result<F64, PW>(a, P2PItem{c, m}, j0 + q, p, st, pw, c_fb, c_hits);
            q0 += pg;
            if (q0 >= np) break;
            sg = 0;
            st = best_none((Best<F64> *)nullptr);
            fill = parts;
            if (parts) base = g0;
        }
        int cs0n = 0, cs1n = 0;
        if (it_next < n_items) {
            cs0n = a.cell_start[item_n.x];
            cs1n = a.cell_start[item_n.x + 1];
        }
        __syncwarp();
        it = it_next;
        it_end = end_next;
        item = item_n;
        cs0 = cs0n;
        cs1 = cs1n;
    }
    if (a.stats) {
        unsigned long long v[ST_N] = {};
        v[ST_ITEMS] = c_items;
        v[ST_TESTS] = c_tests;
        v[ST_FALLBACK] = __reduce_add_sync(FULL, c_fb);
        v[ST_HITS] = __reduce_add_sync(FULL, c_hits);
        flush_stats<NW>(a.stats, v);
    }
}

// Squared FP32 distance to a list entry: the arithmetic of the staged loop.
__device__ __forceinline__ float rec_d2(float2 p, const float4 r0, float inv) {
    const float dx = __fsub_rn(p.x, r0.x), dy = __fsub_rn(p.y, r0.y);
    const float t = __saturatef(__fmul_rn(__fmaf_rn(r0.z, dx, __fmul_rn(r0.w, dy)), inv));
    const float qx = __fmaf_rn(-t, r0.z, dx), qy = __fmaf_rn(-t, r0.w, dy);
    return __fmaf_rn(qx, qx, __fmul_rn(qy, qy));
}

// Smallest of the lanes' non-negative floats (their bits order as integers).
__device__ __forceinline__ float warp_min_pos(float v) {
    return __uint_as_float(__reduce_min_sync(FULL, __float_as_uint(v)));
}

__device__ __forceinline__ Best64 warp_fold64(Best64 st) {
    for (int o = 16; o > 0; o >>= 1)
        consider64(st, __shfl_xor_sync(FULL, st.d2, o), __shfl_xor_sync(FULL, st.id, o),
                   __shfl_xor_sync(FULL, st.seg, o));
    return st;
}

// The smallest FP64 (squared distance, id) over a cell's list, by a warp.
__device__ __forceinline__ Best64 list_best64(const RefineArgs &a, int g0, int g1, double2 p, int lane) {
    Best64 st{__longlong_as_double(0x7ff0000000000000LL), 0x7fffffff, -1};
    for (int g = g0 + lane; g < g1; g += 32) {
        const int i = a.cseg_ids[g];
        consider64(st, seg_d2(a.seg, p, i), seg_owner(a.seg, i), i);
    }
    return warp_fold64(st);
}

// The segments of a cell's list [g0, g1) that can be the nearest to point p (pt
// cell-relative) in FP64, by a warp: those that FP32 finds within 2E of its nearest.
// The first 32 and their polylines go to seg and own (shared memory); the result is
// their number, or more than 32.  The caller synchronises the warp.
__device__ __forceinline__ int near_segments(const RefineArgs &a, int g0, int g1, float2 pt, int *seg, int *own, int lane) {
    float mag = fmaxf(fabsf(pt.x), fabsf(pt.y)), d = __int_as_float(0x7f800000);
    for (int g = g0 + lane; g < g1; g += 32) {
        const float4 r0 = __ldg(a.cseg_rec + 2 * (size_t)g), r1 = __ldg(a.cseg_rec + 2 * (size_t)g + 1);
        d = fminf(d, rec_d2(pt, r0, r1.x));
        mag = fmaxf(mag, r1.z);
    }
    d = sqrtf(warp_min_pos(d));
    const float bound = fmaf(64.0f * U32, warp_max(mag), 4.0f * a.eps_abs) * (1.0f + 8.0f * U32);
    const float sep = 2.0f * bound * (1.0f + 4.0f * U32);
    int cnt = 0;
    __syncwarp();   // a point of more than 32 leaves seg and own as it filled them: orders the writes
    for (int b = g0; b < g1 && cnt <= 32; b += 32) {
        const int g = b + lane;
        bool near = false;
        float4 r1 = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
        if (g < g1) {
            r1 = __ldg(a.cseg_rec + 2 * (size_t)g + 1);
            near = !((sqrtf(rec_d2(pt, __ldg(a.cseg_rec + 2 * (size_t)g), r1.x)) - d) * (1.0f - 4.0f * U32) > sep);
        }
        const unsigned bal = __ballot_sync(FULL, near);
        const int at = cnt + __popc(bal & ((1u << lane) - 1u));
        if (near && at < 32) {
            seg[at] = __float_as_int(r1.w);
            own[at] = __float_as_int(r1.y);
        }
        cnt += __popc(bal);
    }
    return cnt;
}

// FP64 result of one point, by a warp (seg and own as near_segments).
__device__ __forceinline__ Best64 point_best64(const RefineArgs &a, int g0, int g1, double2 p, float2 pt, int *seg, int *own,
                                               int lane) {
    const int cnt = near_segments(a, g0, g1, pt, seg, own, lane);
    if (cnt > 32) return list_best64(a, g0, g1, p, lane);
    Best64 st{__longlong_as_double(0x7ff0000000000000LL), 0x7fffffff, -1};
    __syncwarp();
    if (lane < cnt) consider64(st, seg_d2(a.seg, p, seg[lane]), own[lane], seg[lane]);
    __syncwarp();
    return warp_fold64(st);
}

// FP64 recomputation of the points that the FP32 pass did not settle, a warp per
// point: the lanes test the cell's list in FP32, the segments within 2E of the
// nearest (E as above, M over the whole list) are queued, and FP64 distances are
// taken for a queue of several points with full warps, lane k keeping the smallest
// (squared distance, polyline id) of the queue's k-th point.  What is more than 2E
// behind cannot be the nearest in FP64 arithmetic.  A point with more such segments
// than a warp has lanes (all of them, where E is infinite) takes its whole list in
// FP64.  The record is left as the segment found, for the finishing kernel.
// Bound by the FP32 tests and the latency of the records; with every list entry
// in FP64 it was bound by that pipe (the join of 3 M points with 50,000 walks given
// three times each, FP64 form: 4,852 us then, 1,220 now).
constexpr int RECHECK_WARPS = 8, RECHECK_QUEUE = 64;

template <bool F64>
__global__ void __launch_bounds__(RECHECK_WARPS * 32) k_p2p_recheck(RefineArgs a) {
    __shared__ int seg[RECHECK_WARPS][RECHECK_QUEUE], owner[RECHECK_WARPS][RECHECK_QUEUE];
    __shared__ unsigned char place[RECHECK_WARPS][RECHECK_QUEUE];   // of the segment's point
    __shared__ double dist[RECHECK_WARPS][RECHECK_QUEUE];
    const int lane = lane_id(), w = threadIdx.x >> 5;
    const int nwarps = gridDim.x * RECHECK_WARPS;
    const int n = *a.n_fb;
    const double INF = __longlong_as_double(0x7ff0000000000000LL);
    const bool pw = a.win_on && *a.win_on;
    unsigned c_hits = 0;
    int np = 0, nq = 0;                  // points and segments in the queue
    int slot = -1, q0 = 0, q1 = 0;       // of the queue's lane-th point, its segments
    double2 mine = make_double2(0.0, 0.0);
    auto put = [&](int j, const Best64 &st) {   // one lane
        const bool hit = st.seg >= 0 && sqrt(st.d2) <= (pw ? a.win[j] : a.D);
        a.rec[j] = !hit ? P2PRec{-1, -1} : (F64 ? P2PRec{st.seg, -1} : P2PRec{-2 - st.seg, 0});
        c_hits += hit;
    };
    for (int f = blockIdx.x * RECHECK_WARPS + w;; f += nwarps) {
        if (np > 0 && (f >= n || np == 32 || nq > RECHECK_QUEUE - 32)) {
            __syncwarp();
            for (int k = 0; k < nq; k += 32) {
                const bool one = k + lane < nq;
                const int from = one ? place[w][k + lane] : 0;
                const double2 p = make_double2(__shfl_sync(FULL, mine.x, from), __shfl_sync(FULL, mine.y, from));
                if (one) dist[w][k + lane] = seg_d2(a.seg, p, seg[w][k + lane]);
            }
            __syncwarp();
            if (lane < np) {
                Best64 st{INF, 0x7fffffff, -1};
                for (int k = q0; k < q1; ++k) consider64(st, dist[w][k], owner[w][k], seg[w][k]);
                put(slot, st);
            }
            __syncwarp();
            np = nq = 0;
        }
        if (f >= n) break;
        const int2 e = a.fb[f];
        const int j = e.x, c = e.y, g0 = a.cseg_start[c], g1 = a.cseg_start[c + 1];
        const double2 p = slot_point(a, j);
        const float2 fo = cell_frame(a.frame_x, a.frame_y, a.g.nx, c);
        float hx, lx, hy, ly;
        split_double(p.x, hx, lx);
        split_double(p.y, hy, ly);
        const float2 pt = make_float2(rel_coord(hx, lx, fo.x), rel_coord(hy, ly, fo.y));
        const int cnt = near_segments(a, g0, g1, pt, &seg[w][nq], &owner[w][nq], lane);
        if (cnt > 32) {
            const Best64 st = list_best64(a, g0, g1, p, lane);
            if (lane == 0) put(j, st);
        } else {   // at least the nearest
            if (lane == np) {
                slot = j;
                q0 = nq;
                q1 = nq + cnt;
                mine = p;
            }
            if (lane < cnt) place[w][nq + lane] = (unsigned char)np;
            ++np;
            nq += cnt;
        }
    }
    if (!F64 && a.stats) {   // F64: the finishing kernel counts the hits
        c_hits = __reduce_add_sync(FULL, c_hits);
        if (lane == 0 && c_hits) atomicAdd(&a.stats[ST_HITS], (unsigned long long)c_hits);
    }
}

// ------------------------------------------------------------------ small calls
//
// A call of few points spends its time on the grid, not on the points: counters
// of every cell are cleared, counted into and scanned.  Here a warp takes each
// point straight from the input: its cell, then the cell's segment list with the
// lanes over the segments.  Every list entry is tested once per point and the
// points of a cell share nothing, so the cost grows with the points, where
// bucketing pays for the grid.  us a join, bucketed against direct, 512 x 512
// grid, 150,000 walks, D = 100 m: FP32X 1,000 points 51 / 11, 32,000 73 / 27;
// FP64 1,000 59 / 19, 64,000 102 / 53, 131,000 134 / 93.  The lines
// (P2P_DIRECT_*) lie where direct wins on every layer tried but two, by 6 % (FP64), and
// where looking up a point's cell (below) stays a few us (FP32X).  Longer lists do
// not move them: bucketed work items test their lists once per point as well.
// 150,000 walks on coarser grids, bucketed / direct: FP32X 32,000 points 77 / 44
// (128 x 128 cells), 107 / 99 (64 x 64), 303 / 214 (32 x 32); FP64 131,000 points
// 118 / 126, 220 / 233, 786 / 627, and 5,000 walks on 4 x 4 cells 2,599 / 934.
//
// FP64 leaves each point's record for k_p2p_finish_fp64.  FP32X answers as the
// bucketed refinement would with all of the call's points of a cell in one work
// item (which it is up to 128 of them; beyond, ids still agree, and a point at the
// edge of the certificate can have its FP32 distance on one path and its FP64
// distance on the other).  The refinement's certificate takes the
// magnitude M and the tested segments from the point's work item.  Both only
// grow with the item, and with them the chance
// that the point is redone: so they are bounded from below by those of the
// point alone and from above by those of the whole cell.  Where both agree, the
// item does not matter; for the others (one point in 10^4) the block looks up
// the cell's other points in the input.

// Decision for a point's fold under a certificate: 0 outside the window, 1
// final, 2 to be redone in FP64.
__device__ __forceinline__ int fp32x_decide(const RefineArgs &a, const Best<false> &st, float mag) {
    const float d = sqrtf(st.b1), d2 = sqrtf(st.b2);
    const float e = fmaf(64.0f * U32, mag, 4.0f * a.eps_abs) * (1.0f + 8.0f * U32);
    if (!(e < __int_as_float(0x7f800000))) return 2;   // as in p2p_result
    if (st.i1 < 0 || (d - e) * (1.0f - 4.0f * U32) > a.Dup) return 0;
    const bool in_window = (d + e) * (1.0f + 4.0f * U32) < a.Ddn;
    const bool separated = (d2 - d) * (1.0f - 4.0f * U32) > 2.0f * e * (1.0f + 4.0f * U32);
    return in_window && separated ? 1 : 2;
}

// The staged loop's prune: whether the entry's box comes within D of the box.
__device__ __forceinline__ bool rec_near(const RefineArgs &a, const float4 r0, float smag, float4 box, float pmag) {
    const float bx = r0.x + r0.z, by = r0.y + r0.w;
    const float gx = fmaxf(0.0f, fmaxf(fminf(r0.x, bx) - box.y, box.x - fmaxf(r0.x, bx)));
    const float gy = fmaxf(0.0f, fmaxf(fminf(r0.y, by) - box.w, box.z - fmaxf(r0.y, by)));
    const float lim = a.Df * (1.0f + 1e-6f) + 8.0f * U32 * (smag + pmag) + 8.0f * a.eps_abs;
    return gx * gx + gy * gy <= lim * lim * (1.0f + 8.0f * U32);
}

// FP32X fold of the lanes' folds: the best polyline, and the best distance of
// any other (a lane's own runner-up where its best is that polyline).  Equal
// best distances of two polylines give b2 = b1, which is never final.
__device__ __forceinline__ Best<false> warp_best(const Best<false> &s) {
    Best<false> r;
    r.b1 = warp_min_pos(s.b1);
    r.i1 = __shfl_sync(FULL, s.i1, __ffs(__ballot_sync(FULL, s.b1 == r.b1)) - 1);
    r.b2 = warp_min_pos(s.i1 == r.i1 ? s.b2 : s.b1);
    return r;
}

// Registers for 5 blocks per SM (FP64: 61 registers without the bound, 60,007 points
// 61.6 us a call instead of 59.6) and 4 (FP32X).
template <bool F64>
__global__ void __launch_bounds__(DIRECT_WARPS * 32, F64 ? 5 : 4) k_p2p_direct(RefineArgs a, DirectArgs g, int n) {
    __shared__ int open[DIRECT_OPEN], open_n, box[4], near_seg[DIRECT_WARPS][32], near_own[DIRECT_WARPS][32];
    const int lane = lane_id(), w = threadIdx.x >> 5;
    const double INF = __longlong_as_double(0x7ff0000000000000LL);
    const float FINF = __int_as_float(0x7f800000);
    unsigned long long c_tests = 0, c_pairs = 0, c_algo = 0;
    unsigned c_items = 0, c_fb = 0, c_hits = 0;
    if (!F64) {
        if (threadIdx.x == 0) open_n = 0;
        __syncthreads();
    }
    auto put = [&](int i, int id, double d) {   // one lane
        g.out_id[i] = id;
        if (g.out_d) g.out_d[i] = d;
        c_hits += id >= 0;
    };
    auto redo = [&](int i, int g0, int g1, double2 p, float2 pt) {
        Best64 st;
        if constexpr (F64) st = point_best64(a, g0, g1, p, pt, near_seg[w], near_own[w], lane);
        else st = list_best64(a, g0, g1, p, lane);   // few points, and no registers for more
        const double d = sqrt(st.d2);
        const bool hit = st.seg >= 0 && d <= a.D;
        if (lane == 0) {
            ++c_fb;
            if (F64) a.rec[i] = hit ? P2PRec{st.seg, -1} : P2PRec{-1, -1};
            else put(i, hit ? st.id : -1, hit ? d : INF);
        }
    };
    for (int i = blockIdx.x * DIRECT_WARPS + w; i < n; i += gridDim.x * DIRECT_WARPS) {
        const double2 p = a.pts[i];
        int ix, iy, g0 = 0, g1 = 0;
        const int c = point_cell_xy(a.g, p.x, p.y, ix, iy);
        if (c < a.g.G) {
            g0 = a.cseg_start[c];
            g1 = a.cseg_start[c + 1];
            if (lane == 0) {
                const int nc = g.cand_start[c + 1] - g.cand_start[c];
                c_items += nc > 0;
                c_pairs += nc;
                c_algo += nc > 0 ? g.cell_algo[c] : 0;
            }
        }
        if (g0 == g1) {
            if (lane == 0) {
                if (F64) a.rec[i] = P2PRec{-1, -1};
                else put(i, -1, INF);
            }
            continue;
        }
        float hx, lx, hy, ly;
        split_double(p.x, hx, lx);
        split_double(p.y, hy, ly);
        const float2 pt = make_float2(rel_coord(hx, lx, a.frame_x[ix]), rel_coord(hy, ly, a.frame_y[iy]));
        const float pmag = fmaxf(fabsf(pt.x), fabsf(pt.y));
        const float4 own = make_float4(pt.x, pt.x, pt.y, pt.y);
        Best<F64> all = best_none((Best<F64> *)nullptr), kept = all;
        float mag_all = F64 ? pmag : g.cell_mag, mag = pmag;
        int tests = 0;
        for (int b = g0; b < g1; b += 32) {
            const int k = b + lane;
            bool keep = false;
            if (k < g1 && SJ_IN_BOUNDS(k < a.cseg_start[a.g.G], BND_P2P_REC)) {
                const float4 r0 = __ldg(a.cseg_rec + 2 * (size_t)k), r1 = __ldg(a.cseg_rec + 2 * (size_t)k + 1);
                const float d = rec_d2(pt, r0, r1.x);
                const int tag = __float_as_int(F64 ? r1.w : r1.y);
                keep = rec_near(a, r0, r1.z, own, pmag);
                consider(all, d, tag);
                mag_all = fmaxf(mag_all, r1.z);
                if (!F64 && keep) {
                    consider(kept, d, tag);
                    mag = fmaxf(mag, r1.z);
                }
            }
            tests += __popc(__ballot_sync(FULL, keep));
        }
        c_tests += lane == 0 ? tests : 0;
        mag_all = warp_max(mag_all);
        if constexpr (F64) {
            // segments within 2E of the best: a record for one or two of them
            const float e = fmaf(64.0f * U32, mag_all, 4.0f * a.eps_abs) * (1.0f + 8.0f * U32);
            const float d = sqrtf(warp_min_pos(all.b1)), sep = 2.0f * e * (1.0f + 4.0f * U32);
            const bool n1 = !((sqrtf(all.b1) - d) * (1.0f - 4.0f * U32) > sep);
            const bool n2 = !((sqrtf(all.b2) - d) * (1.0f - 4.0f * U32) > sep);
            const bool n3 = !((sqrtf(all.b3) - d) * (1.0f - 4.0f * U32) > sep);
            const unsigned m1 = __ballot_sync(FULL, n1), m2 = __ballot_sync(FULL, n2);
            const bool three = __any_sync(FULL, n3) || __popc(m1) + __popc(m2) > 2;
            const int l1 = __ffs(m1) - 1, l2 = m2 ? l1 : 31 - __clz(m1);
            P2PRec r;
            r.id = __shfl_sync(FULL, all.i1, max(l1, 0));
            r.aux = __shfl_sync(FULL, m2 ? all.i2 : all.i1, max(l2, 0));
            if (__popc(m1) + __popc(m2) < 2) r.aux = -1;
            const bool out = (d - e) * (1.0f - 4.0f * U32) > a.Dup;
            if (!(e < FINF) || (!out && three)) redo(i, g0, g1, p, pt);
            else if (lane == 0) a.rec[i] = out ? P2PRec{-1, -1} : r;
        } else {
            all = warp_best(all);
            kept = warp_best(kept);
            mag = warp_max(mag);
            const int low = fp32x_decide(a, kept, mag);   // outside: nothing nearer was left out
            if (low == 2) {
                redo(i, g0, g1, p, pt);
            } else if (low == 0) {
                if (lane == 0) put(i, -1, INF);
            } else if (fp32x_decide(a, all, mag_all) == 1) {
                if (lane == 0) put(i, kept.i1, widen(sqrtf(kept.b1)));
            } else if (lane == 0) {
                const int o = atomicAdd(&open_n, 1);
                if (SJ_IN_BOUNDS(o < DIRECT_OPEN, BND_P2P_RES)) open[o] = i;
            }
        }
    }
    if (!F64) {
        __syncthreads();
        const int m = min(open_n, DIRECT_OPEN);
        for (int k = 0; k < m; ++k) {
            const int i = open[k];
            const double2 p = a.pts[i];
            int ix, iy;
            const int c = point_cell_xy(a.g, p.x, p.y, ix, iy);
            const float2 fo = make_float2(a.frame_x[ix], a.frame_y[iy]);
            __syncthreads();
            if (threadIdx.x < 4) box[threadIdx.x] = float_key((threadIdx.x & 1) ? -FINF : FINF);
            __syncthreads();
            for (int j0 = threadIdx.x; j0 < n; j0 += 8 * DIRECT_WARPS * 32) {
                double2 r[8];
#pragma unroll
                for (int u = 0; u < 8; ++u) {
                    const int j = j0 + u * DIRECT_WARPS * 32;
                    r[u] = j < n ? a.pts[j] : make_double2(INF, INF);
                }
#pragma unroll
                for (int u = 0; u < 8; ++u) {
                    int x, y;
                    // within one column and row by the estimate, then exactly
                    axis_estimate(r[u].x, a.g.x0f, a.g.icwf, a.g.tolx, a.g.nx, x);
                    axis_estimate(r[u].y, a.g.y0f, a.g.ichf, a.g.toly, a.g.ny, y);
                    if (a.g.tolx < 0.5f && a.g.toly < 0.5f && (abs(x - ix) > 1 || abs(y - iy) > 1)) continue;
                    if (point_cell(a.g, r[u].x, r[u].y) != c) continue;
                    float ax, bx, ay, by;
                    split_double(r[u].x, ax, bx);
                    split_double(r[u].y, ay, by);
                    const int kx = float_key(rel_coord(ax, bx, fo.x)), ky = float_key(rel_coord(ay, by, fo.y));
                    atomicMin(&box[0], kx);
                    atomicMax(&box[1], kx);
                    atomicMin(&box[2], ky);
                    atomicMax(&box[3], ky);
                }
            }
            __syncthreads();
            if (w == 0) {
                const int g0 = a.cseg_start[c], g1 = a.cseg_start[c + 1];
                const float4 item = make_float4(key_float(box[0]), key_float(box[1]), key_float(box[2]), key_float(box[3]));
                const float pmag = fmaxf(fmaxf(fabsf(item.x), fabsf(item.y)), fmaxf(fabsf(item.z), fabsf(item.w)));
                float hx, lx, hy, ly;
                split_double(p.x, hx, lx);
                split_double(p.y, hy, ly);
                const float2 pt = make_float2(rel_coord(hx, lx, fo.x), rel_coord(hy, ly, fo.y));
                Best<false> st = best_none((Best<false> *)nullptr);
                float mag = pmag;
                for (int q = g0 + lane; q < g1; q += 32) {
                    const float4 r0 = a.cseg_rec[2 * (size_t)q], r1 = a.cseg_rec[2 * (size_t)q + 1];
                    if (!rec_near(a, r0, r1.z, item, pmag)) continue;
                    consider(st, rec_d2(pt, r0, r1.x), __float_as_int(r1.y));
                    mag = fmaxf(mag, r1.z);
                }
                __syncwarp();
                st = warp_best(st);
                mag = warp_max(mag);
                if (fp32x_decide(a, st, mag) == 1) {
                    if (lane == 0) put(i, st.i1, widen(sqrtf(st.b1)));
                } else {
                    redo(i, g0, g1, p, pt);
                }
            }
        }
        __syncthreads();
    }
    if (a.stats) {
        unsigned long long v[ST_N] = {};
        v[ST_ITEMS] = __shfl_sync(FULL, c_items, 0);
        v[ST_PAIRS] = c_pairs;
        v[ST_TESTS] = c_tests;
        v[ST_ALGO] = c_algo;
        v[ST_FALLBACK] = c_fb;
        v[ST_HITS] = c_hits;
        flush_stats<DIRECT_WARPS>(a.stats, v);   // lane 0's
    }
}

cudaError_t launch_p2p_direct(const RefineArgs &a, const DirectArgs &g, int form, int n, int sms, cudaStream_t s) {
    const int blocks = p2p_direct_blocks(n, sms);
    if (form == SJ_FP32X) k_p2p_direct<false><<<blocks, DIRECT_WARPS * 32, 0, s>>>(a, g, n);
    else k_p2p_direct<true><<<blocks, DIRECT_WARPS * 32, 0, s>>>(a, g, n);
    return cudaGetLastError();
}

// ------------------------------------------------------------------ outputs in input order

// FP32X: out[i] from the record of i's slot (pos[i], -1: no slot): the id and
// the FP32 distance, widened exactly, or the FP64 distance to the segment that
// the recheck found.
__device__ __forceinline__ void fp32x_output(const SegArgs &a, const P2PRec r, double2 p, int &id, double &d) {
    id = r.id;
    d = r.id >= 0 ? widen(__int_as_float(r.aux)) : __longlong_as_double(0x7ff0000000000000LL);
    if (r.id < -1) {
        id = seg_owner(a, -2 - r.id);
        d = sqrt(seg_d2(a, p, -2 - r.id));
    }
}

// Points (pairs of points) per thread in the finishing kernels: four in flight
// once the call fills the GPU that way, else one, over four times the blocks
// (whole FP64 calls, four against one: 60,007 points 63.0 and 58.4 us, 131,000
// points 92.0 and 90.0, 400,000 points 194.8 and 197.3).
constexpr int FIN_U = 4;
constexpr long long FIN_MANY = 152LL * 2048;
// Blocks of k_p2p_finish_pairs at most: one tile each, in input order, for all
// but the largest calls.  Blocks that each walk the whole input (16 per SM)
// gather their records from all over the array at once: whole calls, 16 and 512
// blocks per SM, 170 M points 12.23 and 12.12 ms, 10 M points 746 and 741 us.
constexpr int PAIRS_MAX = 152 * 512;

// One request, two consecutive points per thread and step (one 8-byte load of
// their slots, 8- and 16-byte stores): half the memory instructions of one
// point at a time, whose load / store queue fills first.  out_id 8-byte and
// out_d 16-byte aligned, n even or odd.
template <int U>
__global__ void k_p2p_finish_pairs(SegArgs a, const int *pos, const P2PRec *rec, const double2 *pts, int n, int *out_id,
                                   double *out_d) {
    const unsigned T = gridDim.x * blockDim.x;
    const unsigned pairs = ((unsigned)n + 1u) / 2u;
    for (unsigned p0 = blockIdx.x * blockDim.x + threadIdx.x; p0 < pairs; p0 += U * T) {
        int2 j[U];
        P2PRec r0[U], r1[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const unsigned p = p0 + u * T, i = 2u * p;
            j[u] = make_int2(-1, -1);
            if (p < pairs) {
                if (i + 1u < (unsigned)n) j[u] = *reinterpret_cast<const int2 *>(pos + i);
                else j[u].x = pos[i];
            }
        }
#pragma unroll
        for (int u = 0; u < U; ++u) {
            if (j[u].x >= 0 && !SJ_IN_BOUNDS(j[u].x < n, BND_UNSORT)) j[u].x = -1;
            if (j[u].y >= 0 && !SJ_IN_BOUNDS(j[u].y < n, BND_UNSORT)) j[u].y = -1;
            r0[u] = j[u].x >= 0 ? rec[j[u].x] : P2PRec{-1, -1};
            r1[u] = j[u].y >= 0 ? rec[j[u].y] : P2PRec{-1, -1};
        }
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const unsigned p = p0 + u * T, i = 2u * p;
            if (p >= pairs) continue;
            const bool two = i + 1u < (unsigned)n;
            int id0, id1;
            double d0, d1;
            fp32x_output(a, r0[u], r0[u].id < -1 ? pts[i] : make_double2(0.0, 0.0), id0, d0);
            fp32x_output(a, r1[u], r1[u].id < -1 ? pts[i + 1u] : make_double2(0.0, 0.0), id1, d1);
            if (two) {
                *reinterpret_cast<int2 *>(out_id + i) = make_int2(id0, id1);
                if (out_d) *reinterpret_cast<double2 *>(out_d + i) = make_double2(d0, d1);
            } else {
                out_id[i] = id0;
                if (out_d) out_d[i] = d0;
            }
        }
    }
}

// Where a finishing kernel's points come from: a call's points in input order,
// a call's slots (no scratch for pos), or the requests of a batched round.
struct FinOne {
    const int *pos;
    const double2 *pts;
    int *out_id;
    double *out_d;
    int n;
    double window;
    __device__ __forceinline__ int count() const { return n; }
    __device__ __forceinline__ int slot(int i) const { return pos ? pos[i] : i; }   // no pos: records by point
    __device__ __forceinline__ double2 point(int i) const { return pts[i]; }
    __device__ __forceinline__ double win(int) const { return window; }
    __device__ __forceinline__ void put(int i, int id, double d) const {
        out_id[i] = id;
        if (out_d) out_d[i] = d;
    }
};
struct FinSlots {
    const int *perm, *in_grid;   // in_grid: device count of slots
    const double2 *pts;
    int *out_id;
    double *out_d;
    double window;
    __device__ __forceinline__ int count() const { return *in_grid; }
    __device__ __forceinline__ int slot(int i) const { return i; }
    __device__ __forceinline__ double2 point(int i) const { return pts[perm[i]]; }
    __device__ __forceinline__ double win(int) const { return window; }
    __device__ __forceinline__ void put(int i, int id, double d) const {
        const int k = perm[i];
        out_id[k] = id;
        if (out_d) out_d[k] = d;
    }
};
struct FinRound {
    const RoundReq *reqs;
    const int *meta, *pos;
    __device__ __forceinline__ const RoundReq &find(int i) const { return reqs[find_request(reqs, meta[0], i)]; }
    __device__ __forceinline__ int count() const { return meta[1]; }
    __device__ __forceinline__ int slot(int i) const { return pos[i]; }
    __device__ __forceinline__ double2 point(int i) const {
        const RoundReq &r = find(i);
        return r.pts[i - r.off];
    }
    __device__ __forceinline__ double win(int i) const { return find(i).window; }
    __device__ __forceinline__ void put(int i, int id, double d) const {
        const RoundReq &r = find(i);
        r.out_id[i - r.off] = id;
        if (r.out_d) r.out_d[i - r.off] = d;
    }
};

template <class Src>
__global__ void k_p2p_finish_fp32x(SegArgs a, const P2PRec *rec, Src src) {
    const int n = src.count();
    for (long long k = blockIdx.x * (long long)blockDim.x + threadIdx.x; k < n; k += (long long)gridDim.x * blockDim.x) {
        const int i = (int)k, j = src.slot(i);
        const P2PRec r = j >= 0 ? rec[j] : P2PRec{-1, -1};
        int id;
        double d;
        fp32x_output(a, r, r.id < -1 ? src.point(i) : make_double2(0.0, 0.0), id, d);
        src.put(i, id, d);
    }
}

// FP64: the FP64 distances to the one or two segments of each point's record.
// A warp takes U x 32 points; the second segments, which about a third of
// the points have, are gathered in shared memory and evaluated with full warps,
// since the FP64 pipe takes as long for one lane as for 32.  The compares of
// the (non-negative, finite) distances and of t are made on their bit patterns,
// off that pipe.
__device__ __forceinline__ double clamp01(double t) {
    const long long b = __double_as_longlong(t);   // a NaN (0 times an infinite 1 / |e|^2) gives 0, as fmax does
    return (b <= 0 || b > 0x7ff0000000000000LL) ? 0.0 : (b > 0x3ff0000000000000LL ? 1.0 : t);
}
__device__ __forceinline__ double seg_d2_finite(const SegArgs &a, double2 p, int i) {
    const double2 v = a.verts[i], e = a.seg_e64[i];
    const double dx = __dsub_rn(p.x, v.x), dy = __dsub_rn(p.y, v.y);
    const double t = clamp01(__dmul_rn(__fma_rn(e.x, dx, __dmul_rn(e.y, dy)), a.seg_inv64[i]));
    const double qx = __fma_rn(-t, e.x, dx), qy = __fma_rn(-t, e.y, dy);
    return __fma_rn(qx, qx, __dmul_rn(qy, qy));
}

constexpr int FIN_WARPS = 8;

template <int U, class Src>
__global__ void __launch_bounds__(FIN_WARPS * 32) k_p2p_finish_fp64(SegArgs a, const P2PRec *rec, Src src,
                                                                    unsigned long long *stats) {
    __shared__ int2 q[FIN_WARPS][32 * U];        // (point of the tile, second segment)
    __shared__ double d2s[FIN_WARPS][32 * U];
    const double INF = __longlong_as_double(0x7ff0000000000000LL);
    const int lane = lane_id(), w = threadIdx.x >> 5;
    const unsigned lt = (1u << lane) - 1u;
    const long long n = src.count();
    unsigned hits = 0;
    for (long long base = (blockIdx.x * (long long)FIN_WARPS + w) * (32 * U); base < n;
         base += (long long)gridDim.x * FIN_WARPS * (32 * U)) {
        P2PRec r[U];
        double d2[U];
        int nq = 0;
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const long long i = base + 32 * u + lane;
            const int j = i < n ? src.slot((int)i) : -1;
            r[u] = j >= 0 ? rec[j] : P2PRec{-1, -1};
        }
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const bool two = r[u].id >= 0 && r[u].aux >= 0;
            const unsigned bal = __ballot_sync(FULL, two);
            if (two) q[w][nq + __popc(bal & lt)] = make_int2(32 * u + lane, r[u].aux);
            nq += __popc(bal);
            d2[u] = r[u].id >= 0 ? seg_d2_finite(a, src.point((int)(base + 32 * u + lane)), r[u].id) : INF;
        }
        __syncwarp();
        for (int k = lane; k < nq; k += 32) {
            const int2 e = q[w][k];
            d2s[w][e.x] = seg_d2_finite(a, src.point((int)(base + e.x)), e.y);
        }
        __syncwarp();
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const long long i = base + 32 * u + lane;
            if (i >= n) continue;
            int id = -1;
            double d = INF;
            if (r[u].id >= 0) {
                int oid = seg_owner(a, r[u].id);
                if (r[u].aux >= 0) {   // the smaller (squared distance, id)
                    const double e2 = d2s[w][32 * u + lane];
                    const long long x = __double_as_longlong(d2[u]), y = __double_as_longlong(e2);
                    const int o2 = seg_owner(a, r[u].aux);
                    if (y < x || (y == x && o2 < oid)) {
                        d2[u] = e2;
                        oid = o2;
                    }
                }
                const double s = sqrt(d2[u]);
                if (s <= src.win((int)i)) {
                    id = oid;
                    d = s;
                }
            }
            src.put((int)i, id, d);
            hits += id >= 0;
        }
        __syncwarp();
    }
    if (stats) {
        unsigned long long v[ST_N] = {};
        v[ST_HITS] = __reduce_add_sync(FULL, hits);
        flush_stats<FIN_WARPS>(stats, v);
    }
}

static int fin_blocks(long long n, int per_block, int cap) {
    const long long b = (n + per_block - 1) / per_block;
    return (int)(b < 1 ? 1 : (b > cap ? cap : b));
}

template <class Src>
static void finish(const RefineArgs &a, int form, const Src &src, long long n_max, cudaStream_t s) {
    if (form == SJ_FP32X)
        k_p2p_finish_fp32x<Src><<<fin_blocks(n_max, 256, 152 * 16), 256, 0, s>>>(a.seg, a.rec, src);
    else
        (n_max >= FIN_MANY ? k_p2p_finish_fp64<FIN_U, Src> : k_p2p_finish_fp64<1, Src>)<<<
            fin_blocks(n_max, 32 * FIN_WARPS * (n_max >= FIN_MANY ? FIN_U : 1), 152 * 16), FIN_WARPS * 32, 0, s>>>(
            a.seg, a.rec, src, a.stats);
}

// a8: outputs in input order from the slots' records (pos: slot of each input
// point or -1; null: the records are by input point).
cudaError_t launch_p2p_finish(const RefineArgs &a, int form, const int *pos, int n, int *out_id, double *out_d,
                              cudaStream_t s) {
    if (form == SJ_FP32X && pos && ((uintptr_t)out_id & 7) == 0 && ((uintptr_t)out_d & 15) == 0)
        (n >= FIN_MANY ? k_p2p_finish_pairs<FIN_U> : k_p2p_finish_pairs<1>)<<<
            fin_blocks((n + 1LL) / 2, 256 * (n >= FIN_MANY ? FIN_U : 1), PAIRS_MAX), 256, 0, s>>>(a.seg, pos, a.rec, a.pts, n,
                                                                                            out_id, out_d);
    else
        finish(a, form, FinOne{pos, a.pts, out_id, out_d, n, a.D}, n, s);
    return cudaGetLastError();
}
// The same slot by slot through perm (in_grid: device count of slots).
cudaError_t launch_p2p_finish_slots(const RefineArgs &a, int form, const int *in_grid, int n, int *out_id,
                                    double *out_d, cudaStream_t s) {
    finish(a, form, FinSlots{a.perm, in_grid, a.pts, out_id, out_d, a.D}, n, s);
    return cudaGetLastError();
}
cudaError_t launch_p2p_finish_round(const RefineArgs &a, int form, const RoundReq *reqs, const int *meta,
                                    const int *pos, long long n_max, cudaStream_t s) {
    finish(a, form, FinRound{reqs, meta, pos}, n_max, s);
    return cudaGetLastError();
}

// ------------------------------------------------------------------ launches

template <bool F64, bool PW, int NW>
static cudaError_t p2p_prepare() {
    static bool done = false;   // per process; the attribute is per function
    if (!done) {
        cudaError_t e = cudaFuncSetAttribute(k_p2p_refine<F64, PW, NW>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                             (int)sizeof(P2PSmem) * NW);
        if (e != cudaSuccess) return e;
        done = true;
    }
    return cudaSuccess;
}

template <bool F64, bool PW, int NW>
static cudaError_t p2p_launch(const RefineArgs &a, int blocks, cudaStream_t s) {
    cudaError_t e = p2p_prepare<F64, PW, NW>();
    if (e != cudaSuccess) return e;
    k_p2p_refine<F64, PW, NW><<<blocks, NW * 32, sizeof(P2PSmem) * NW, s>>>(a);
    return cudaGetLastError();
}

template <bool F64, bool PW>
static cudaError_t p2p_launch_nw(const RefineArgs &a, int nw, int blocks, cudaStream_t s) {
    if (nw == 2) return p2p_launch<F64, PW, 2>(a, blocks, s);
    if (nw == 8) return p2p_launch<F64, PW, 8>(a, blocks, s);
    return p2p_launch<F64, PW, P2P_WARPS>(a, blocks, s);
}

// blocks: the grid for blocks of P2P_WARPS warps (resident blocks x SMs); a
// block of warps_per_block (2, 4 or 8) warps gets the same number of warps.
cudaError_t launch_p2p_refine(const RefineArgs &a, int form, int warps_per_block, int blocks, cudaStream_t s) {
    const int nw = (warps_per_block == 2 || warps_per_block == 8) ? warps_per_block : P2P_WARPS;
    blocks = (int)(((long long)blocks * P2P_WARPS + nw - 1) / nw);
    const bool pw = a.win && a.win_on;
    if (form == SJ_FP32X) return pw ? p2p_launch_nw<false, true>(a, nw, blocks, s) : p2p_launch_nw<false, false>(a, nw, blocks, s);
    return pw ? p2p_launch_nw<true, true>(a, nw, blocks, s) : p2p_launch_nw<true, false>(a, nw, blocks, s);
}

cudaError_t launch_p2p_recheck(const RefineArgs &a, int form, int blocks, cudaStream_t s) {
    if (form == SJ_FP32X) k_p2p_recheck<false><<<blocks, RECHECK_WARPS * 32, 0, s>>>(a);
    else k_p2p_recheck<true><<<blocks, RECHECK_WARPS * 32, 0, s>>>(a);
    return cudaGetLastError();
}

int p2p_blocks_per_sm(int form) {
    int n = 0;
    if (form == SJ_FP32X) {
        if (p2p_prepare<false, false, P2P_WARPS>() != cudaSuccess) return 1;
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, k_p2p_refine<false, false, P2P_WARPS>, P2P_WARPS * 32,
                                                      sizeof(P2PSmem) * P2P_WARPS);
    } else {
        if (p2p_prepare<true, false, P2P_WARPS>() != cudaSuccess) return 1;
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, k_p2p_refine<true, false, P2P_WARPS>, P2P_WARPS * 32,
                                                      sizeof(P2PSmem) * P2P_WARPS);
    }
    return n > 0 ? n : 1;
}

}  // namespace sj

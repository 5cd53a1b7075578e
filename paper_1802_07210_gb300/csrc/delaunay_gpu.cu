// Delaunay triangulation of the support points on the GPU (Sec. III.A: the
// mesh of the support points; the paper keeps this step on a CPU and finds it
// dominates its run time, Sec. VII).
//
// The triangulation wanted is the unique one of the symbolically perturbed
// point set (lifted heights |p_i|^2 + eps_i, eps_0 >> eps_1 >> ..., i = list
// index), the same one the host routine builds.  Here every point builds its
// own star (the triangles around it) by gift-wrapping: the third vertex of a
// directed edge (p, a) is the point on its left that no other such point lies
// inside the circle through p, a and it (a strict total order with the
// symbolic tie-break, so a warp reduction finds it).  A triangle is emitted
// once, by its lowest-index vertex, so of a star only the fan of triangles
// that p owns and one more on either side are needed (dt_warp_star).
//   1. Warp pass: one warp per point, the points within 24 pixels from a
//      16-pixel grid; a star counts when the circles of its triangles fit
//      that disc (2r <= R, so no farther point can matter), 93-95 % of them.
//   2. Middle pass (batches): the others again, with 64 pixels.
//   3. CTA pass: one CTA per star left (the hull, the rims of empty areas):
//      the star over the points within 96 pixels, then scans of the cells
//      that its wide circles meet until they are empty (dt_block_item).
// The output order is deterministic: an exclusive scan of the per-point
// counts, and within a star counter-clockwise from the nearest neighbour (an
// open star then clockwise from it).
//
// One step of the earlier design (4 or 16 lanes per star, the whole star,
// 64-bit key comparisons, one region scan per step of a wide star) against
// this one: 640x480 172 -> 96 us, 1920x1080 590 -> 276 us, 64 x 1242x375
// 3.44 -> 1.82 ms for all triangulation kernels.
#include "launch.cuh"

namespace elas {

constexpr int kDtCell = 16;

__device__ __forceinline__ int dt_ncell(const DtArgs &a) { return a.gw * a.gh; }

__device__ __forceinline__ int dt_cell(const DtArgs &a, int x, int y) {
    const int cx = min(max(x, 0) / kDtCell, a.gw - 1), cy = min(max(y, 0) / kDtCell, a.gh - 1);
    return cy * a.gw + cx;
}

// -------------------------------------------------------------------------
// Grid build
// -------------------------------------------------------------------------

__device__ __forceinline__ void dt_points_body(const DtArgs &a, const VB &vb) {
    const DtSide S = vb.y ? a.s[1] : a.s[0];
    const int n = min(max(*a.count, 0), a.cap);
    for (int i = vb.x * blockDim.x + threadIdx.x; i < n; i += vb.gx * blockDim.x) {
        const int u = a.list[3 * i], v = a.list[3 * i + 1], d = a.list[3 * i + 2];
        const int x = S.right ? u - d : u;
        S.X[i] = x;
        S.Y[i] = v;
        S.owned[i] = 0;
        if (i > 0 && a.list[3 * i - 2] > v) atomicOr(S.err, 8);  // not in raster order
        atomicAdd(S.cell_cnt + dt_cell(a, x, v), 1);
        if (v >= 0 && v < a.h) {
            atomicMin(S.rowmin + v, x);
            atomicMax(S.rowmax + v, x);
        }
    }
}

__global__ void dt_points_kernel(DtArgs a) { dt_points_body(a, vb_single()); }
__global__ void dt_points_kernel_b(const DtArgs *__restrict__ tab, VMap vm) {
    const VB vb = vb_batch(vm);
    dt_points_body(slot_entry(tab, vm.stride, vb.slot), vb);
}

// One CTA per side: exclusive scan of the cell counts, each thread taking
// kCellScanItems consecutive cells of a chunk (their loads go out together).
__device__ __forceinline__ void dt_cell_scan_body(const DtArgs &a, const VB &vb) {
    constexpr int kCellScanItems = 4;
    __shared__ int s_w[32];
    __shared__ int s_carry;
    const DtSide S = vb.y ? a.s[1] : a.s[0];
    const int ncell = dt_ncell(a);
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    const int chunk = kCellScanItems * (int)blockDim.x;
    if (tid == 0) s_carry = 0;
    __syncthreads();
    for (int base = 0; base <= ncell; base += chunk) {
        const int i0 = base + kCellScanItems * tid;
        int v[kCellScanItems];
#pragma unroll
        for (int k = 0; k < kCellScanItems; ++k) v[k] = i0 + k < ncell ? S.cell_cnt[i0 + k] : 0;
        int tot = 0;
#pragma unroll
        for (int k = 0; k < kCellScanItems; ++k) tot += v[k];
        int incl = tot;
        for (int o = 1; o < 32; o <<= 1) {
            const int y = __shfl_up_sync(0xFFFFFFFFu, incl, o);
            if (lane >= o) incl += y;
        }
        if (lane == 31) s_w[wid] = incl;
        __syncthreads();
        if (wid == 0) {
            int x = lane < (int)(blockDim.x >> 5) ? s_w[lane] : 0;
            for (int o = 1; o < 32; o <<= 1) {
                const int y = __shfl_up_sync(0xFFFFFFFFu, x, o);
                if (lane >= o) x += y;
            }
            s_w[lane] = x;
        }
        __syncthreads();
        int excl = s_carry + (wid ? s_w[wid - 1] : 0) + incl - tot;
#pragma unroll
        for (int k = 0; k < kCellScanItems; ++k) {
            if (i0 + k <= ncell) {  // entry ncell receives the total
                S.cell_start[i0 + k] = excl;
                S.cell_fill[i0 + k] = excl;
            }
            excl += v[k];
        }
        __syncthreads();
        if (tid == 0) s_carry += s_w[31];
        __syncthreads();
    }
}

__global__ void __launch_bounds__(1024) dt_cell_scan_kernel(DtArgs a) { dt_cell_scan_body(a, vb_single()); }
__global__ void __launch_bounds__(1024) dt_cell_scan_kernel_b(const DtArgs *__restrict__ tab, VMap vm) {
    const VB vb = vb_batch(vm);
    dt_cell_scan_body(slot_entry(tab, vm.stride, vb.slot), vb);
}

__device__ __forceinline__ void dt_scatter_body(const DtArgs &a, const VB &vb) {
    const DtSide S = vb.y ? a.s[1] : a.s[0];
    const int n = min(max(*a.count, 0), a.cap);
    for (int i = vb.x * blockDim.x + threadIdx.x; i < n; i += vb.gx * blockDim.x) {
        const int x = S.X[i], y = S.Y[i];
        const int k = atomicAdd(S.cell_fill + dt_cell(a, x, y), 1);
        S.pts[k] = make_int4(x, y, i, 1);
        S.slot[i] = k;
    }
}

__global__ void dt_scatter_kernel(DtArgs a) { dt_scatter_body(a, vb_single()); }
__global__ void dt_scatter_kernel_b(const DtArgs *__restrict__ tab, VMap vm) {
    const VB vb = vb_batch(vm);
    dt_scatter_body(slot_entry(tab, vm.stride, vb.slot), vb);
}

// Coincident points (right coordinates only) keep the lowest list index.
__device__ __forceinline__ void dt_dedup_body(const DtArgs &a, const VB &vb) {
    const DtSide S = vb.y ? a.s[1] : a.s[0];
    const int n = min(max(*a.count, 0), a.cap);
    for (int i = vb.x * blockDim.x + threadIdx.x; i < n; i += vb.gx * blockDim.x) {
        const int x = S.X[i], y = S.Y[i];
        const int c = dt_cell(a, x, y);
        bool dup = false;
        for (int k = S.cell_start[c]; k < S.cell_start[c + 1]; ++k) {
            const int4 q = S.pts[k];
            if (q.x == x && q.y == y && q.z < i) dup = true;
        }
        if (dup) S.pts[S.slot[i]].w = 0;
    }
}

__global__ void dt_dedup_kernel(DtArgs a) { dt_dedup_body(a, vb_single()); }
__global__ void dt_dedup_kernel_b(const DtArgs *__restrict__ tab, VMap vm) {
    const VB vb = vb_batch(vm);
    dt_dedup_body(slot_entry(tab, vm.stride, vb.slot), vb);
}

// -------------------------------------------------------------------------
// Stars
// -------------------------------------------------------------------------

constexpr int kDtSlots = 16;       // owned triangles kept per point; larger fans go to the pool
constexpr int kDtRadius = 24;      // warp pass: candidates within this many pixels
constexpr int kDtListCap = 128;    // its list (a radius-24 disc holds about 75 points of a full step-5 lattice)
constexpr int kDtRadiusM = 64;     // middle pass (batches)
constexpr int kDtListCapM = 640;   // a radius-64 disc holds about 520 lattice points
constexpr int kDtWarps = 8;        // stars per CTA of the warp pass
constexpr int kDtWarpsM = 4;       // stars per CTA of the middle pass
constexpr float kDtInf = 3.402823466e38f;  // "no candidate" key (every real key is far below)

__device__ __forceinline__ float dt_warp_min(float v) {
    float r;
    asm volatile("redux.sync.min.f32 %0, %1, 0xffffffff;" : "=f"(r) : "f"(v));
    return r;
}

// The Delaunay third vertex of directed edge (p, e) on side s (+1 left, -1
// right) is the candidate c with s*cross(e, c) > 0 (coordinates relative to
// p) that minimises t(c) = N/D, N = |c|^2 - e.c, D = s*cross(e, c): the
// circles through p and e are nested on each side in the order of t.  Every
// step below finds the least t in FP32 (one approximate division per
// candidate, one warp reduction), takes the candidates within a band that
// covers the rounding, and, when the band has several members, orders those
// exactly in integers.
//
// Equal t means that p, e and both candidates are cocircular: of the four,
// the one with the lowest list index (raised the most by the symbolic
// perturbation) gets the ear, so the diagonal joins its two neighbours on
// the circle.  With x the first candidate after e (going round from p over
// e) and y the second, y wins iff the lowest index is p's or x's.
// Does the second candidate beat the first?  o = s*cross(c1, c2).
__device__ __forceinline__ bool dt_tie_second(int pz, int ez, int z1, int z2, bool first_is_x) {
    const int xz = first_is_x ? z1 : z2, yz = first_is_x ? z2 : z1;
    const bool ywins = min(pz, xz) < min(ez, yz);
    return first_is_x == ywins;
}

// Is the circle through the origin, a and b no wider than R (2r <= R)?
// |a|^2 |b|^2 |a-b|^2 <= R^2 cross(a, b)^2, in FP32 with a margin far above
// its rounding: a false answer only sends a star to the next pass.
__device__ __forceinline__ bool dt_small_circle(int ax, int ay, int bx, int by, float R2) {
    const float pa = (float)(ax * ax + ay * ay), pb = (float)(bx * bx + by * by);
    const int dx = bx - ax, dy = by - ay;
    const float ab = (float)dx * (float)dx + (float)dy * (float)dy, ar = (float)(ax * by - ay * bx);
    return pa * pb * ab * 1.00001f <= R2 * ar * ar;
}

struct DtPt {
    int x, y, z;  // relative to the star's point; list index
};

// Candidates of a star as packed relative coordinates and list index.
struct DtListSrc {
    const int2 *list;
    int k;
    __device__ __forceinline__ DtPt get(int c) const {
        const int2 v = list[c];
        return DtPt{(int)(int16_t)(v.x & 0xFFFF), v.x >> 16, v.y};
    }
};
__device__ __forceinline__ int2 dt_pack(int x, int y, int z) { return make_int2((y << 16) | (x & 0xFFFF), z); }

// A quarter of the grid-sorted points (the exact pass over every point).
struct DtAllSrc {
    const int4 *pts;
    int k, part, px, py, pz;
    __device__ __forceinline__ DtPt get(int c) const {
        const int4 q = pts[4 * c + part];
        if (!q.w || q.z == pz) return DtPt{0, 0, pz};  // D = 0: never a candidate
        return DtPt{q.x - px, q.y - py, q.z};
    }
};

// Does c2 beat c1 for edge (p, e) on `side`, exactly?
__device__ __forceinline__ bool dt_beats(const DtPt &e, int pz, const DtPt &c1, const DtPt &c2, int side) {
    const int D1 = side * (e.x * c1.y - e.y * c1.x), D2 = side * (e.x * c2.y - e.y * c2.x);
    const int N1 = c1.x * c1.x + c1.y * c1.y - (e.x * c1.x + e.y * c1.y);
    const int N2 = c2.x * c2.x + c2.y * c2.y - (e.x * c2.x + e.y * c2.y);
    const int64_t l = (int64_t)N2 * D1, r = (int64_t)N1 * D2;
    if (l != r) return l < r;
    if (c1.z == c2.z) return false;
    return dt_tie_second(pz, e.z, c1.z, c2.z, side * ((int64_t)c1.x * c2.y - (int64_t)c1.y * c2.x) > 0);
}

// One wrap step by a warp over src's candidates, exact while every
// coordinate difference stays below 2^14.5 (N and D fit 32 bits; their
// rounding to FP32 and the division leave a relative error below 2^-20).
template <class Src>
__device__ __forceinline__ bool dt_step(const Src &src, int lane, const DtPt &e, int pz, int side, DtPt &w) {
    float f1 = kDtInf, f2 = kDtInf;
    int c1 = 0;
    const int sx = side * e.x, sy = side * e.y;
#pragma unroll 4
    for (int c = lane; c < src.k; c += 32) {
        const DtPt q = src.get(c);
        const int D = sx * q.y - sy * q.x, N = q.x * q.x + q.y * q.y - (e.x * q.x + e.y * q.y);
        const float f = D > 0 ? __fdividef((float)N, (float)D) : kDtInf;
        f2 = fminf(f2, fmaxf(f1, f));
        if (f < f1) {
            f1 = f;
            c1 = c;
        }
    }
    const float fm = dt_warp_min(f1);
    if (fm == kDtInf) return false;
    const float thr = fm + 0x1p-17f * fabsf(fm);
    bool in = f1 <= thr;
    if (in && f2 <= thr) {  // several of this lane's candidates: keep the exact best
        int best = -1;
        DtPt bq{0, 0, 0};
        for (int c = lane; c < src.k; c += 32) {
            const DtPt q = src.get(c);
            const int D = sx * q.y - sy * q.x, N = q.x * q.x + q.y * q.y - (e.x * q.x + e.y * q.y);
            if (D <= 0 || __fdividef((float)N, (float)D) > thr) continue;
            if (best < 0 || dt_beats(e, pz, bq, q, side)) {
                best = c;
                bq = q;
            }
        }
        c1 = best;
    }
    unsigned b = __ballot_sync(0xFFFFFFFFu, in);
    int ch = __shfl_sync(0xFFFFFFFFu, c1, __ffs(b) - 1);
    w = src.get(ch);
    if (b & (b - 1)) {
        const DtPt mine = in ? src.get(c1) : w;
        while (b & (b - 1)) {
            in = in && c1 != ch && dt_beats(e, pz, w, mine, side);
            b = __ballot_sync(0xFFFFFFFFu, in);
            if (!b) break;
            ch = __shfl_sync(0xFFFFFFFFu, c1, __ffs(b) - 1);
            w = src.get(ch);
        }
    }
    return true;
}

// First vertex of a fan (see dt_warp_star): the candidate below p (y > 0)
// that a circle through p growing straight down touches first, least
// |c|^2 / y; of several on that circle the first one counter-clockwise.
template <class Src> __device__ __forceinline__ bool dt_fan_start(const Src &src, int lane, DtPt &w) {
    auto better = [](const DtPt &c1, const DtPt &c2) {  // c2 before c1
        const int64_t l = (int64_t)(c2.x * c2.x + c2.y * c2.y) * c1.y, r = (int64_t)(c1.x * c1.x + c1.y * c1.y) * c2.y;
        if (l != r) return l < r;
        return (int64_t)c2.x * c1.y - (int64_t)c2.y * c1.x > 0;
    };
    float f1 = kDtInf, f2 = kDtInf;
    int c1 = 0;
    for (int c = lane; c < src.k; c += 32) {
        const DtPt q = src.get(c);
        const float f = q.y > 0 ? __fdividef((float)(q.x * q.x + q.y * q.y), (float)q.y) : kDtInf;
        f2 = fminf(f2, fmaxf(f1, f));
        if (f < f1) {
            f1 = f;
            c1 = c;
        }
    }
    const float fm = dt_warp_min(f1);
    if (fm == kDtInf) return false;
    const float thr = fm + 0x1p-17f * fm;
    bool in = f1 <= thr;
    if (in && f2 <= thr) {
        DtPt bq = src.get(c1);
        for (int c = lane; c < src.k; c += 32) {
            const DtPt q = src.get(c);
            if (q.y > 0 && better(bq, q)) {
                bq = q;
                c1 = c;
            }
        }
    }
    unsigned b = __ballot_sync(0xFFFFFFFFu, in);
    int ch = __shfl_sync(0xFFFFFFFFu, c1, __ffs(b) - 1);
    w = src.get(ch);
    if (b & (b - 1)) {
        const DtPt mine = in ? src.get(c1) : w;
        while (b & (b - 1)) {
            in = in && c1 != ch && better(w, mine);
            b = __ballot_sync(0xFFFFFFFFu, in);
            if (!b) break;
            ch = __shfl_sync(0xFFFFFFFFu, c1, __ffs(b) - 1);
            w = src.get(ch);
        }
    }
    return true;
}

// The warp pass's candidates: within 24 pixels of p, so every key is a small
// integer and FP32 arithmetic on it is exact (N and D below 2^11, their
// cross products below 2^24).  Each lane keeps two of them (x, y, |c|^2,
// index) in registers; a list of more than 64 reads the rest from shared
// memory.
struct DtNearSrc {
    const float4 *list;
    int k;
    float4 c0, c1;

    __device__ __forceinline__ void load(int lane) {
        const float4 none = make_float4(0.0f, 0.0f, 0.0f, 0.0f);  // D = 0 and y = 0: never a candidate
        c0 = lane < k ? list[lane] : none;
        c1 = lane + 32 < k ? list[lane + 32] : none;
    }
    __device__ __forceinline__ float4 far_cand(int c) const {
        return c < k ? list[c] : make_float4(0.0f, 0.0f, 0.0f, 0.0f);
    }
    __device__ __forceinline__ DtPt point(const float4 &v) const {
        return DtPt{(int)v.x, (int)v.y, __float_as_int(v.z == 0.0f ? 0.0f : v.w)};
    }
    // Least key over the slots, then the exact order among its band:
    // key(c) (kDtInf: not a candidate), beats(c1, c2): c2 before c1.
    template <class Key, class Beats>
    __device__ __forceinline__ bool select(int lane, Key key, Beats beats, float4 &w) const {
        const float f0 = key(c0), f1 = key(c1);
        float f2 = kDtInf, f3 = kDtInf;
        if (k > 64) {
            f2 = key(far_cand(lane + 64));
            f3 = key(far_cand(lane + 96));
        }
        const float fm = dt_warp_min(fminf(fminf(f0, f1), fminf(f2, f3)));
        if (fm == kDtInf) return false;
        const float thr = fm + 0x1p-18f * fabsf(fm);
        unsigned b0 = __ballot_sync(0xFFFFFFFFu, f0 <= thr), b1 = __ballot_sync(0xFFFFFFFFu, f1 <= thr);
        unsigned b2 = 0, b3 = 0;
        if (k > 64) {
            b2 = __ballot_sync(0xFFFFFFFFu, f2 <= thr);
            b3 = __ballot_sync(0xFFFFFFFFu, f3 <= thr);
        }
        for (;;) {
            const int ch = b0   ? __ffs(b0) - 1
                           : b1 ? __ffs(b1) + 31
                           : b2 ? __ffs(b2) + 63
                                : __ffs(b3) + 95;
            w = list[ch];
            if (__popc(b0) + __popc(b1) + __popc(b2) + __popc(b3) == 1) return true;
            const unsigned me = 1u << lane;
            // the champion itself never beats itself
            const unsigned n0 = __ballot_sync(0xFFFFFFFFu, (b0 & me) && beats(w, c0));
            const unsigned n1 = __ballot_sync(0xFFFFFFFFu, (b1 & me) && beats(w, c1));
            unsigned n2 = 0, n3 = 0;
            if (k > 64) {
                n2 = __ballot_sync(0xFFFFFFFFu, (b2 & me) && beats(w, far_cand(lane + 64)));
                n3 = __ballot_sync(0xFFFFFFFFu, (b3 & me) && beats(w, far_cand(lane + 96)));
            }
            if (!(n0 | n1 | n2 | n3)) return true;
            b0 = n0;
            b1 = n1;
            b2 = n2;
            b3 = n3;
        }
    }
};

__device__ __forceinline__ bool dt_step(const DtNearSrc &src, int lane, const float4 &e, int pz, float side,
                                        float4 &w) {
    const float sx = side * e.x, sy = side * e.y;
    auto dkey = [&](const float4 &c) { return __fmaf_rn(sx, c.y, -(sy * c.x)); };
    auto nkey = [&](const float4 &c) { return __fmaf_rn(-e.x, c.x, __fmaf_rn(-e.y, c.y, c.z)); };
    return src.select(
        lane,
        [&](const float4 &c) {
            const float D = dkey(c);
            return D > 0.0f ? __fdividef(nkey(c), D) : kDtInf;
        },
        [&](const float4 &c1, const float4 &c2) {
            const float l = nkey(c2) * dkey(c1), r = nkey(c1) * dkey(c2);
            if (l != r) return l < r;
            const int z1 = __float_as_int(c1.w), z2 = __float_as_int(c2.w);
            return z1 != z2 &&
                   dt_tie_second(pz, __float_as_int(e.w), z1, z2, side * (c1.x * c2.y - c1.y * c2.x) > 0.0f);
        },
        w);
}

__device__ __forceinline__ bool dt_fan_start(const DtNearSrc &src, int lane, float4 &w) {
    return src.select(
        lane, [&](const float4 &c) { return c.y > 0.0f ? __fdividef(c.z, c.y) : kDtInf; },
        [&](const float4 &c1, const float4 &c2) {
            const float l = c2.z * c1.y, r = c1.z * c2.y;
            if (l != r) return l < r;
            return c2.x * c1.y - c2.y * c1.x > 0.0f;
        },
        w);
}

// Views of a candidate for the star driver.
__device__ __forceinline__ int dt_z(const DtPt &c) { return c.z; }
__device__ __forceinline__ int dt_z(const float4 &c) { return __float_as_int(c.w); }
__device__ __forceinline__ int dt_ix(const DtPt &c) { return c.x; }
__device__ __forceinline__ int dt_ix(const float4 &c) { return (int)c.x; }
__device__ __forceinline__ int dt_iy(const DtPt &c) { return c.y; }
__device__ __forceinline__ int dt_iy(const float4 &c) { return (int)c.y; }

// Nearest candidate (least |c|^2, then least index) and the open quadrants
// that hold candidates (bit 2*(y>0) + (x>0)).
__device__ __forceinline__ unsigned dt_quadrant(int x, int y) {
    return x && y ? 1u << ((x > 0) | ((y > 0) << 1)) : 0u;
}
__device__ __forceinline__ float4 dt_nearest(const DtNearSrc &src, int lane, unsigned &quads) {
    unsigned d = 0x7FFFFFFFu, q = 0;
    int z = 0x7FFFFFFF, c = 0;
    auto offer = [&](const float4 &v, int at) {
        if (v.z == 0.0f) return;
        const unsigned vd = __float_as_uint(v.z);  // positive: ordered as integers
        const int vz = __float_as_int(v.w);
        if (vd < d || (vd == d && vz < z)) {
            d = vd;
            z = vz;
            c = at;
        }
        q |= dt_quadrant((int)v.x, (int)v.y);
    };
    offer(src.c0, lane);
    offer(src.c1, lane + 32);
    if (src.k > 64) {
        offer(src.far_cand(lane + 64), lane + 64);
        offer(src.far_cand(lane + 96), lane + 96);
    }
    quads = __reduce_or_sync(0xFFFFFFFFu, q);
    const unsigned dm = __reduce_min_sync(0xFFFFFFFFu, d);
    const int zm = __reduce_min_sync(0xFFFFFFFFu, d == dm ? z : 0x7FFFFFFF);
    const unsigned b = __ballot_sync(0xFFFFFFFFu, d == dm && z == zm);
    return src.list[__shfl_sync(0xFFFFFFFFu, c, __ffs(b) - 1)];
}
__device__ __forceinline__ DtPt dt_nearest(const DtListSrc &src, int lane, unsigned &quads) {
    unsigned d = 0xFFFFFFFFu, q = 0;
    int z = 0x7FFFFFFF, c = 0;
    for (int j = lane; j < src.k; j += 32) {
        const DtPt v = src.get(j);
        const unsigned vd = (unsigned)(v.x * v.x + v.y * v.y);
        if (vd < d || (vd == d && v.z < z)) {
            d = vd;
            z = v.z;
            c = j;
        }
        q |= dt_quadrant(v.x, v.y);
    }
    quads = __reduce_or_sync(0xFFFFFFFFu, q);
    const unsigned dm = __reduce_min_sync(0xFFFFFFFFu, d);
    const int zm = __reduce_min_sync(0xFFFFFFFFu, d == dm ? z : 0x7FFFFFFF);
    const unsigned b = __ballot_sync(0xFFFFFFFFu, d == dm && z == zm);
    return src.get(__shfl_sync(0xFFFFFFFFu, c, __ffs(b) - 1));
}

// Where triangle t of a fan of m goes in the output: the owned triangles of a
// star are written counter-clockwise from its nearest neighbour, which is
// vertex r of the fan (0 when it is none of its vertices).
__device__ __forceinline__ int dt_fan_pos(int t, int m, int r) { return t >= r ? t - r : t + m - r; }

// The owned triangles of a star whose vertices sit one per lane: a[0..na]
// counter-clockwise from the first vertex, b[0..nb] clockwise from it.
__device__ __forceinline__ void dt_warp_write(const DtSide &S, int pz, int lane, bool fan, int va, int vb, int na,
                                              int nb, int nnz) {
    const int va1 = __shfl_down_sync(0xFFFFFFFFu, va, 1), vb1 = __shfl_down_sync(0xFFFFFFFFu, vb, 1);
    const bool oa = lane < na && pz < va && pz < va1, ob = lane < nb && pz < vb && pz < vb1;
    const unsigned ba = __ballot_sync(0xFFFFFFFFu, oa), bb = __ballot_sync(0xFFFFFFFFu, ob);
    const int ma = __popc(ba), mb = __popc(bb), m = ma + mb;
    int pa = __popc(ba & ((1u << lane) - 1u)), pb = ma + __popc(bb & ((1u << lane) - 1u));
    if (fan) {
        const unsigned ra = __ballot_sync(0xFFFFFFFFu, lane <= ma && va == nnz);
        const unsigned rb = __ballot_sync(0xFFFFFFFFu, lane <= mb && vb == nnz);
        const int r = ra ? mb + __ffs(ra) - 1 : (rb ? mb - (__ffs(rb) - 1) : 0);
        pa = dt_fan_pos(mb + lane, m, r);
        pb = dt_fan_pos(mb - 1 - lane, m, r);
    }
    int2 *out = S.slots + (size_t)pz * kDtSlots;
    if (m > kDtSlots) {
        int base = 0;
        if (lane == 0) {
            base = atomicAdd(S.npool, m);
            *out = make_int2(base, 0);
        }
        out = S.pool + __shfl_sync(0xFFFFFFFFu, base, 0);
    }
    if (oa) out[pa] = make_int2(va, va1);
    if (ob) out[pb] = make_int2(vb1, vb);
    if (lane == 0) S.owned[pz] = m;
}

// One star by a warp over the candidates within R of p; true if it came out
// certified (its owned triangles are then written).
//
// Triangles are emitted by their lowest-index vertex.  A list in raster order
// (v never decreases) puts the two others of an owned triangle level with p
// or below it, so the owned triangles are one run of consecutive sectors in
// the lower half of the star, and only that fan is wrapped: from the vertex
// that the circle growing straight down from p meets first, both ways until
// a vertex is not below p.  That is 4 steps per star on average instead of
// the whole star's 6.  It needs p strictly inside the hull (candidates in all
// four open quadrants show that); other stars, and every star of an
// unordered list, are wrapped whole from the nearest neighbour,
// counter-clockwise and, when that meets the hull, clockwise from it again.
//
// A triangle is certain when its circle, which passes through p, is no wider
// than R: no point farther than R from p is inside it.  Where a whole star
// stays open (p on the hull), nothing may lie beyond either open edge, tested
// against the extreme points of every image row.
template <class Src>
__device__ __forceinline__ bool dt_warp_star(const DtArgs &a, const DtSide &S, const int4 &p, const Src &src, int R,
                                             bool ordered, int lane) {
    unsigned quads;
    auto nn = dt_nearest(src, lane, quads);
    auto first = nn;
    const bool fan = ordered && quads == 15u;
    if (fan && !dt_fan_start(src, lane, first)) return false;
    const float R2 = (float)(R * R);
    int va = dt_z(first), vb = va, na = 0, nb = 0;
    bool closed = false, open_l = false, open_r = false;
    auto cur = first;
    for (;;) {  // counter-clockwise
        auto w = cur;
        if (!dt_step(src, lane, cur, p.z, 1, w)) {
            open_l = true;
            break;
        }
        if (na == 30 || !dt_small_circle(dt_ix(cur), dt_iy(cur), dt_ix(w), dt_iy(w), R2)) return false;
        ++na;
        if (lane == na) va = dt_z(w);
        if (fan && dt_iy(w) <= 0) break;
        if (!fan && dt_z(w) == dt_z(first)) {
            closed = true;
            break;
        }
        cur = w;
    }
    if (fan && open_l) return false;
    const auto e_l = cur;
    cur = first;
    while (!closed) {  // clockwise
        auto w = cur;
        if (!dt_step(src, lane, cur, p.z, -1, w)) {
            open_r = true;
            break;
        }
        if (nb == 30 || !dt_small_circle(dt_ix(w), dt_iy(w), dt_ix(cur), dt_iy(cur), R2)) return false;
        ++nb;
        if (lane == nb) vb = dt_z(w);
        if (fan && dt_iy(w) <= 0) break;
        cur = w;
    }
    if (fan && open_r) return false;
    if (open_l || open_r) {
        const int lx = dt_ix(e_l), ly = dt_iy(e_l), rx = dt_ix(cur), ry = dt_iy(cur);
        bool bad = false;
        for (int y = lane; y < a.h; y += 32) {
            const int x0 = S.rowmin[y], x1 = S.rowmax[y];
            if (x0 > x1) continue;
            const int dy = y - p.y, d0 = x0 - p.x, d1 = x1 - p.x;
            bad |= lx * dy - ly * d0 > 0 || lx * dy - ly * d1 > 0;
            bad |= rx * dy - ry * d0 < 0 || rx * dy - ry * d1 < 0;
        }
        if (__any_sync(0xFFFFFFFFu, bad)) return false;
    }
    dt_warp_write(S, p.z, lane, fan, va, vb, na, nb, dt_z(nn));
    return true;
}

// Calls visit(q, inside) for the points of the grid cells that the square of
// half-size R around p meets, 32 at a time: the cell rows' ranges, up to
// 2^LOG2 of them, are walked as one index space (a binary search over the
// lanes' prefix sums), two loads in flight.
template <int LOG2, class Visit>
__device__ __forceinline__ void dt_warp_window(const DtArgs &a, const DtSide &S, const int4 &p, int R, int lane,
                                               Visit visit) {
    const int cx0 = min(a.gw - 1, max(0, p.x - R) / kDtCell), cx1 = min(a.gw - 1, max(0, p.x + R) / kDtCell);
    const int cy0 = max(0, p.y - R) / kDtCell, cy1 = min(a.gh - 1, max(0, p.y + R) / kDtCell);
    int rs = 0, len = 0;
    if (lane <= cy1 - cy0) {
        const int *row = S.cell_start + (cy0 + lane) * a.gw;
        rs = row[cx0];
        len = row[cx1 + 1] - rs;
    }
    int incl = len;
#pragma unroll
    for (int o = 1; o < (1 << LOG2); o <<= 1) {
        const int y = __shfl_up_sync(0xFFFFFFFFu, incl, o);
        if (lane >= o) incl += y;
    }
    const int total = __shfl_sync(0xFFFFFFFFu, incl, (1 << LOG2) - 1);
    const int excl = incl - len, off = rs - excl;
    for (int t0 = 0; t0 < total; t0 += 64) {
        int4 q[2];
        bool in[2];
#pragma unroll
        for (int u = 0; u < 2; ++u) {
            const int t = t0 + 32 * u + lane;
            int lo = 0;
#pragma unroll
            for (int s = 1 << (LOG2 - 1); s > 0; s >>= 1)
                if (t >= __shfl_sync(0xFFFFFFFFu, excl, lo + s)) lo += s;
            in[u] = t < total;
            const int at = t + __shfl_sync(0xFFFFFFFFu, off, lo);
            q[u] = in[u] ? S.pts[at] : make_int4(0, 0, 0, 0);
        }
        visit(q[0], in[0]);
        if (t0 + 32 < total) visit(q[1], in[1]);
    }
}

// Warp pass: one warp per point, the candidates within 24 pixels (12 or 6
// where the list is full).  Bound by instruction issue: about 400 warp
// instructions per star.
__device__ __forceinline__ void dt_pass1_body(const DtArgs &a, const VB &vb) {
    __shared__ float4 s_list[kDtWarps][kDtListCap];
    const DtSide &S = a.s[vb.y];
    const int n = min(max(*a.count, 0), a.cap);
    const int lane = threadIdx.x & 31;
    float4 *list = s_list[threadIdx.x >> 5];
    const bool ordered = !(*S.err & 8);
    for (int j = vb.x * kDtWarps + (threadIdx.x >> 5); j < n; j += vb.gx * kDtWarps) {
        const int4 p = S.pts[j];
        if (!p.w) continue;
        int k = 0;
        auto gather = [&](int R) {
            k = 0;
            dt_warp_window<2>(a, S, p, R, lane, [&](const int4 &q, bool inside) {
                const int dx = q.x - p.x, dy = q.y - p.y, d2 = dx * dx + dy * dy;
                const bool take = inside && q.w && q.z != p.z && d2 <= R * R;
                const unsigned b = __ballot_sync(0xFFFFFFFFu, take);
                const int pos = k + __popc(b & ((1u << lane) - 1u));
                if (take && pos < kDtListCap)
                    list[pos] = make_float4((float)dx, (float)dy, (float)d2, __int_as_float(q.z));
                k += __popc(b);
            });
        };
        int R = kDtRadius;
        gather(R);
        while (k > kDtListCap && R > 6) {
            R >>= 1;
            __syncwarp();
            gather(R);
        }
        __syncwarp();
        bool done = false;
        if (k > 0 && k <= kDtListCap) {
            DtNearSrc src{list, k};
            src.load(lane);
            done = dt_warp_star(a, S, p, src, R, ordered, lane);
        }
        if (!done && lane == 0) S.pending[atomicAdd(S.npending, 1)] = p.z;
        __syncwarp();
    }
}

__global__ void __launch_bounds__(kDtWarps * 32, 5) dt_pass1_kernel(DtArgs a) { dt_pass1_body(a, vb_single()); }
__global__ void __launch_bounds__(kDtWarps * 32, 5) dt_pass1_kernel_b(const DtArgs *__restrict__ tab, VMap vm) {
    const VB vb = vb_batch(vm);
    dt_pass1_body(slot_entry(tab, vm.stride, vb.slot), vb);
}

// Middle pass (batches): the stars left by the warp pass, again a warp each,
// with the candidates within 64 pixels.
__device__ __forceinline__ void dt_pass1m_body(const DtArgs &a, const VB &vb) {
    __shared__ int2 s_list[kDtWarpsM][kDtListCapM];
    const DtSide &S = a.s[vb.y];
    const int lane = threadIdx.x & 31;
    int2 *list = s_list[threadIdx.x >> 5];
    const bool ordered = !(*S.err & 8);
    const int njobs = *S.npending;
    for (int j = vb.x * kDtWarpsM + (threadIdx.x >> 5); j < njobs; j += vb.gx * kDtWarpsM) {
        const int4 p = S.pts[S.slot[S.pending[j]]];
        int k = 0;
        dt_warp_window<4>(a, S, p, kDtRadiusM, lane, [&](const int4 &q, bool inside) {
            const int dx = q.x - p.x, dy = q.y - p.y;
            const bool take = inside && q.w && q.z != p.z && dx * dx + dy * dy <= kDtRadiusM * kDtRadiusM;
            const unsigned b = __ballot_sync(0xFFFFFFFFu, take);
            const int pos = k + __popc(b & ((1u << lane) - 1u));
            if (take && pos < kDtListCapM) list[pos] = dt_pack(dx, dy, q.z);
            k += __popc(b);
        });
        __syncwarp();
        bool done = false;
        if (k > 0 && k <= kDtListCapM) {
            const DtListSrc src{list, k};
            done = dt_warp_star(a, S, p, src, kDtRadiusM, ordered, lane);
        }
        if (!done && lane == 0) S.pending2[atomicAdd(S.npending2, 1)] = p.z;
        __syncwarp();
    }
}
static_assert(2 * kDtRadius / kDtCell + 1 <= 4 && 2 * kDtRadiusM / kDtCell + 2 <= 16, "cell rows of a disc");

__global__ void __launch_bounds__(kDtWarpsM * 32) dt_pass1m_kernel_b(const DtArgs *__restrict__ tab, VMap vm) {
    const VB vb = vb_batch(vm);
    dt_pass1m_body(slot_entry(tab, vm.stride, vb.slot), vb);
}

// -------------------------------------------------------------------------
// CTA pass: the stars whose circles do not fit the listed discs (the hull,
// the rims of empty areas)
// -------------------------------------------------------------------------
// One CTA per star.  The points within kDtRadiusC are cached in shared
// memory and the star is wrapped over the cache (warp 0 counter-clockwise,
// warp 1 clockwise).  Triangles whose circle is no wider than the disc are
// certain; for all the others at once the CTA scans the grid cells that their
// circles (and, at an open end, the half-plane beyond the edge) meet, adds
// every point found inside to the cache, and the star is wrapped again.  The
// star is done when a scan finds no point: each of its triangles then has an
// empty circle.  Most stars take one scan, the widest three; a step-by-step
// search would scan once per triangle (up to 50).  A large region is first
// scanned with a stride, which finds points that shrink the circles to a
// small part of it.  A full cache keeps only the star's own vertices and
// goes on with the whole star (its region can only shrink, so that ends).
constexpr int kDtRadiusC = 96;
constexpr int kDtCacheCap = 2048;   // cached points (16 KB)
constexpr int kDtBlockThreads = 128;
constexpr int kDtBlocksPerSM = 8;
constexpr int kDtVertCap = 256;     // star vertices per direction
constexpr int kDtBadCap = 32;       // circles scanned for at a time (a warp's triangles)
constexpr int kDtMaxRounds = 64;
constexpr int kDtSampleMin = 2048;  // regions of more points are sampled first

// Triangle (p, a, b), counter-clockwise, coordinates relative to p: q lies
// inside its circle iff |q|^2 W - U q.x - V q.y < 0 (below 2^60).
struct DtCircle {
    DtPt a, b;
    int W;
    int64_t U, V;
};

__device__ __forceinline__ DtCircle dt_circle(const DtPt &a, const DtPt &b) {
    DtCircle c;
    c.a = a;
    c.b = b;
    const int64_t a2 = a.x * a.x + a.y * a.y, b2 = b.x * b.x + b.y * b.y;
    c.W = a.x * b.y - a.y * b.x;
    c.U = b.y * a2 - a.y * b2;
    c.V = a.x * b2 - b.x * a2;
    return c;
}

// Does q invalidate the triangle: inside its circle or, on it, favoured by
// the symbolic order?  On the circle the triangle stays iff the lowest index
// of the four is q's or that of the vertex opposite to it (the diagonal then
// joins the two others).
__device__ __forceinline__ bool dt_violates(const DtCircle &c, int pz, const DtPt &q) {
    const int64_t q2 = q.x * q.x + q.y * q.y;
    const int64_t s = q2 * c.W - c.U * q.x - c.V * q.y;
    if (s != 0) return s < 0;
    if (q.z == pz || q.z == c.a.z || q.z == c.b.z) return false;
    const int64_t oa = (int64_t)c.a.x * q.y - (int64_t)c.a.y * q.x, ob = (int64_t)c.b.x * q.y - (int64_t)c.b.y * q.x;
    const int opp = oa < 0 ? c.b.z : (ob > 0 ? c.a.z : pz);
    const int m1 = oa < 0 || ob > 0 ? pz : c.a.z, m2 = oa < 0 ? c.a.z : c.b.z;
    return min(m1, m2) < min(opp, q.z);
}

struct DtStarShared {
    DtCircle bad[kDtBadCap];
    int2 vert[2][kDtVertCap];  // the star: counter-clockwise, clockwise from the first vertex
    int nv[2];                 // triangles in each direction
    int open[2];
    int over;                  // more vertices than the lists hold
    int closed;
    unsigned long long nn;     // |c|^2 and index of the nearest point
    unsigned quads;
    int k, nbad, next, found, total;
    int rs[16], rlen[16];
    DtPt win[4];
    int won[4];
};

// Cell range of image rows [cy*16, cy*16+15] that a region meets, widened so
// that FP32 rounding cannot lose a cell (two pixels in y, one cell and more
// in x).  A disc (rad >= 0) or the half-plane nx*x + ny*y >= 0 about (x0, y0).
__device__ __forceinline__ bool dt_row_range(int cy, float x0, float y0, float rad, float nx, float ny, int gw,
                                             int &c0, int &c1) {
    const float ya = (float)(cy * kDtCell - 2) - y0, yb = (float)(cy * kDtCell + kDtCell + 1) - y0;
    float xlo = -1e9f, xhi = 1e9f;
    if (rad >= 0.0f) {
        const float dy = ya > 0.0f ? ya : (yb < 0.0f ? -yb : 0.0f);
        if (dy > rad) return false;
        const float hc = sqrtf(rad * rad - dy * dy) + 2.0f;
        xlo = x0 - hc;
        xhi = x0 + hc;
    } else {
        // x >= or <= the boundary of the band's more permissive edge, 4 pixels wider
        const float m = fmaxf(ny * ya, ny * yb) + 4.0f;
        if (fabsf(nx) < 1e-4f) {
            if (m < -4.0f) return false;
        } else if (nx > 0.0f) {
            xlo = x0 - m / nx - 4.0f;
        } else {
            xhi = x0 - m / nx + 4.0f;
        }
    }
    c0 = (int)fmaxf(0.0f, fminf((float)(gw - 1), floorf(xlo / kDtCell) - 1.0f));
    c1 = (int)fmaxf(0.0f, fminf((float)(gw - 1), floorf(xhi / kDtCell) + 1.0f));
    return true;
}

// Gathers the points within R of p into the cache (their number, even past
// the capacity, in sh.k), with the nearest one and the quadrants.
__device__ __forceinline__ void dt_block_gather(const DtArgs &a, const DtSide &S, const int4 &p, int R, int2 *cand,
                                                DtStarShared &sh) {
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int cx0 = min(a.gw - 1, max(0, p.x - R) / kDtCell), cx1 = min(a.gw - 1, max(0, p.x + R) / kDtCell);
    const int cy0 = max(0, p.y - R) / kDtCell, cy1 = min(a.gh - 1, max(0, p.y + R) / kDtCell);
    const int nrows = cy1 - cy0 + 1;
    __syncthreads();
    if (tid < nrows) {
        const int *row = S.cell_start + (cy0 + tid) * a.gw;
        const int r0 = row[cx0], r1 = row[cx1 + 1];
        sh.rs[tid] = r0;
        sh.rlen[tid] = r1 - r0;
    }
    if (tid == 0) {
        sh.k = 0;
        sh.nn = ~0ull;
        sh.quads = 0;
    }
    __syncthreads();
    unsigned long long nn = ~0ull;
    unsigned quads = 0;
    for (int r = warp; r < nrows; r += kDtBlockThreads / 32) {
        const int s0 = sh.rs[r], len = sh.rlen[r];
        for (int j0 = 0; j0 < len; j0 += 64) {
            int4 q[2];
#pragma unroll
            for (int u = 0; u < 2; ++u) {
                const int j = j0 + 32 * u + lane;
                q[u] = j < len ? S.pts[s0 + j] : make_int4(0, 0, 0, 0);
            }
#pragma unroll
            for (int u = 0; u < 2; ++u) {
                const int dx = q[u].x - p.x, dy = q[u].y - p.y, d2 = dx * dx + dy * dy;
                const bool take = q[u].w && q[u].z != p.z && abs(dx) <= R && abs(dy) <= R && d2 <= R * R;
                const unsigned m = __ballot_sync(0xFFFFFFFFu, take);
                int base = 0;
                if (lane == 0 && m) base = atomicAdd(&sh.k, __popc(m));
                const int pos = __shfl_sync(0xFFFFFFFFu, base, 0) + __popc(m & ((1u << lane) - 1u));
                if (take) {
                    if (pos < kDtCacheCap) cand[pos] = dt_pack(dx, dy, q[u].z);
                    nn = min(nn, ((unsigned long long)d2 << 32) | (unsigned)q[u].z);
                    quads |= dt_quadrant(dx, dy);
                }
            }
        }
    }
    if (nn != ~0ull) {
        atomicMin(&sh.nn, nn);
        atomicOr(&sh.quads, quads);
    }
    __syncthreads();
}
static_assert(2 * kDtRadiusC / kDtCell + 2 <= 16, "cell rows of the cached disc");

// Wraps the star over the cache: warp 0 counter-clockwise, warp 1 clockwise.
__device__ __forceinline__ void dt_block_wrap(const int2 *cand, int k, int pz, bool fan, const DtPt &nn,
                                              DtStarShared &sh) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    __syncthreads();
    if (warp < 2) {
        const DtListSrc src{cand, k};
        const int side = warp ? -1 : 1;
        DtPt first = nn;
        bool ok = !fan || dt_fan_start(src, lane, first);
        DtPt cur = first;
        int nv = 0;
        bool open = false, closed = false;
        if (lane == 0) sh.vert[warp][0] = dt_pack(first.x, first.y, first.z);
        while (ok) {
            DtPt w;
            if (!dt_step(src, lane, cur, pz, side, w)) {
                open = true;
                break;
            }
            if (nv == kDtVertCap - 1) {
                ok = false;
                break;
            }
            ++nv;
            if (lane == 0) sh.vert[warp][nv] = dt_pack(w.x, w.y, w.z);
            if (fan && w.y <= 0) break;
            if (!fan && w.z == first.z) {
                closed = true;
                break;
            }
            cur = w;
        }
        if (lane == 0) {
            sh.nv[warp] = nv;
            sh.open[warp] = open;
            if (!ok || (fan && open)) sh.over = 1;
            if (closed) sh.closed = 1;  // both warps meet the first vertex again
        }
    }
    __syncthreads();
    if (threadIdx.x == 0 && sh.closed) sh.nv[1] = 0;
    __syncthreads();
}

// Triangle t of the star in sh (counter-clockwise run first), as (a, b).
__device__ __forceinline__ void dt_star_tri(const DtStarShared &sh, int t, DtPt &a, DtPt &b) {
    const int na = sh.nv[0];
    const DtListSrc src{sh.vert[t < na ? 0 : 1] + (t < na ? t : t - na), 2};
    a = src.get(t < na ? 0 : 1);
    b = src.get(t < na ? 1 : 0);
}

// Writes the owned triangles of the star in sh (warp 0).
__device__ __forceinline__ void dt_block_write(const DtSide &S, int pz, bool fan, int nnz, const DtStarShared &sh) {
    const int lane = threadIdx.x & 31;
    const int na = sh.nv[0], nt = na + sh.nv[1];
    int ma = 0, mb = 0, r = -1;
    for (int t0 = 0; t0 < nt; t0 += 32) {
        DtPt u{0, 0, 0}, v{0, 0, 0};
        if (t0 + lane < nt) dt_star_tri(sh, t0 + lane, u, v);
        const bool own = t0 + lane < nt && pz < u.z && pz < v.z;
        ma += __popc(__ballot_sync(0xFFFFFFFFu, own && t0 + lane < na));
        mb += __popc(__ballot_sync(0xFFFFFFFFu, own && t0 + lane >= na));
    }
    const int m = ma + mb;
    if (fan) {
        for (int i = lane; i <= ma; i += 32)
            if (sh.vert[0][i].y == nnz) r = mb + i;
        for (int i = lane; i <= mb; i += 32)
            if (sh.vert[1][i].y == nnz) r = mb - i;
        r = max(0, __reduce_max_sync(0xFFFFFFFFu, r));
    }
    int2 *out = S.slots + (size_t)pz * kDtSlots;
    if (m > kDtSlots) {
        int base = 0;
        if (lane == 0) {
            base = atomicAdd(S.npool, m);
            *out = make_int2(base, 0);
        }
        out = S.pool + __shfl_sync(0xFFFFFFFFu, base, 0);
    }
    int done = 0;
    for (int t0 = 0; t0 < nt; t0 += 32) {
        const int t = t0 + lane;
        DtPt u{0, 0, 0}, v{0, 0, 0};
        if (t < nt) dt_star_tri(sh, t, u, v);
        const bool own = t < nt && pz < u.z && pz < v.z;
        const unsigned b = __ballot_sync(0xFFFFFFFFu, own);
        int pos = done + __popc(b & ((1u << lane) - 1u));
        if (fan) pos = dt_fan_pos(t < na ? mb + t : mb - 1 - (t - na), m, r);
        if (own) out[pos] = make_int2(u.z, v.z);
        done += __popc(b);
    }
    if (lane == 0) S.owned[pz] = m;
}

// The whole star of p over every point, one exact step after the other (more
// vertices than the lists hold, e.g. the apex of a huge fan): counted first,
// then written.
__device__ void dt_block_star_all(const DtSide &S, const int4 &p, int n, const DtPt &nn, DtStarShared &sh) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    int2 *out = nullptr;
    int m = 0;
    for (int pass = 0; pass < 2; ++pass) {
        int written = 0;
        bool closed = false;
        for (int side = 1; side >= -1 && !closed; side -= 2) {
            DtPt cur = nn;
            for (int step = 0; step <= n; ++step) {
                const DtAllSrc src{S.pts, (n - warp + 3) / 4, warp, p.x, p.y, p.z};
                DtPt w{0, 0, 0};
                const bool any = dt_step(src, lane, cur, p.z, side, w);
                __syncthreads();
                if (lane == 0) {
                    sh.win[warp] = w;
                    sh.won[warp] = any;
                }
                __syncthreads();
                bool got = false;
                for (int i = 0; i < 4; ++i)
                    if (sh.won[i] && (!got || dt_beats(cur, p.z, w, sh.win[i], side))) {
                        w = sh.win[i];
                        got = true;
                    }
                if (!got) break;
                if (p.z < cur.z && p.z < w.z) {
                    if (out && threadIdx.x == 0) out[written] = side > 0 ? make_int2(cur.z, w.z) : make_int2(w.z, cur.z);
                    ++written;
                }
                if (w.z == nn.z) {
                    closed = true;
                    break;
                }
                cur = w;
            }
        }
        if (pass == 0) {
            m = written;
            out = S.slots + (size_t)p.z * kDtSlots;
            if (m > kDtSlots) {
                if (threadIdx.x == 0) {
                    sh.total = atomicAdd(S.npool, m);
                    *out = make_int2(sh.total, 0);
                }
                __syncthreads();
                out = S.pool + sh.total;
            }
        }
    }
    if (threadIdx.x == 0) S.owned[p.z] = m;
    __syncthreads();
}

__device__ __forceinline__ void dt_block_item(const DtArgs &a, const DtSide &S, int i, int n, bool ordered,
                                              int2 *cand, int *r_start, int *r_len, DtStarShared &sh) {
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int4 p = S.pts[S.slot[i]];
    int R = kDtRadiusC;
    dt_block_gather(a, S, p, R, cand, sh);
    while (sh.k > kDtCacheCap && R > 1) {
        R >>= 1;
        dt_block_gather(a, S, p, R, cand, sh);
    }
    int k = sh.k;
    if (k == 0) {  // nothing near: the nearest of all points
        unsigned long long key = ~0ull;
        for (int j = tid; j < n; j += kDtBlockThreads) {
            const int4 q = S.pts[j];
            const int64_t dx = q.x - p.x, dy = q.y - p.y;
            if (q.w && q.z != p.z) key = min(key, ((unsigned long long)(dx * dx + dy * dy) << 32) | (unsigned)q.z);
        }
        if (key != ~0ull) atomicMin(&sh.nn, key);
        __syncthreads();
        if (sh.nn == ~0ull) {  // p is the only point
            if (tid == 0) S.owned[p.z] = 0;
            __syncthreads();
            return;
        }
    }
    const int4 nq = S.pts[S.slot[(int)(unsigned)(sh.nn & 0xFFFFFFFFu)]];
    const DtPt nn{nq.x - p.x, nq.y - p.y, nq.z};
    bool fan = ordered && sh.quads == 15u;
    if (k == 0) {
        if (tid == 0) cand[0] = dt_pack(nn.x, nn.y, nn.z);
        k = 1;
    }
    for (int round = 0;; ++round) {
        if (tid == 0) {
            sh.over = 0;
            sh.closed = 0;
            sh.found = 0;
        }
        dt_block_wrap(cand, k, p.z, fan, nn, sh);
        if (sh.over || round == kDtMaxRounds) {
            dt_block_star_all(S, p, n, nn, sh);
            return;
        }
        const int nt = sh.nv[0] + sh.nv[1];
        const bool open_l = sh.open[0], open_r = !sh.closed && sh.open[1];
        const float R2 = (float)(R * R);
        bool first = true;  // the open ends go with the first group of circles
        int found = 0;
        for (int t0 = 0; t0 < nt || first;) {
            // the next circles that the disc does not certify
            __syncthreads();
            if (warp == 0) {
                int nb = 0;
                for (; t0 < nt && nb == 0; t0 += 32) {
                    DtPt u{0, 0, 0}, v{0, 0, 0};
                    if (t0 + lane < nt) dt_star_tri(sh, t0 + lane, u, v);
                    const bool bad = t0 + lane < nt && !dt_small_circle(u.x, u.y, v.x, v.y, R2);
                    const unsigned b = __ballot_sync(0xFFFFFFFFu, bad);
                    if (bad) sh.bad[__popc(b & ((1u << lane) - 1u))] = dt_circle(u, v);
                    nb = __popc(b);
                }
                if (lane == 0) {
                    sh.nbad = nb;
                    sh.next = t0;
                    sh.total = 0;
                }
            }
            const bool ends = first && (open_l || open_r);
            first = false;
            __syncthreads();
            const int nbad = sh.nbad;
            t0 = sh.next;
            if (nbad == 0 && !ends) continue;
            const DtListSrc v0{sh.vert[0], 0}, v1{sh.vert[1], 0};
            const DtPt el = v0.get(sh.nv[0]), er = v1.get(sh.nv[1]);
            int tot = 0;
            for (int cy = tid; cy < a.gh; cy += kDtBlockThreads) {
                int lo = a.gw, hi = -1, c0, c1;
                for (int b = 0; b < nbad; ++b) {
                    const DtCircle &c = sh.bad[b];
                    const float U = (float)c.U, V = (float)c.V, W2 = 2.0f * (float)c.W;
                    const float ux = U / W2, uy = V / W2, r = sqrtf(ux * ux + uy * uy);
                    bool any;
                    if (r <= 1e6f) {
                        any = dt_row_range(cy, (float)p.x + ux, (float)p.y + uy, r * 1.0001f + 4.0f, 0.0f, 0.0f, a.gw,
                                           c0, c1);
                    } else {  // the half-plane beyond the circle's tangent at p holds the disc
                        const float l = rsqrtf(U * U + V * V);
                        any = dt_row_range(cy, (float)p.x, (float)p.y, -1.0f, U * l, V * l, a.gw, c0, c1);
                    }
                    if (any) {
                        lo = min(lo, c0);
                        hi = max(hi, c1);
                    }
                }
                if (ends) {
                    for (int s = 0; s < 2; ++s) {
                        if (!(s ? open_r : open_l)) continue;
                        const float ex = (float)(s ? -er.x : el.x), ey = (float)(s ? -er.y : el.y);
                        const float l = rsqrtf(ex * ex + ey * ey);
                        if (dt_row_range(cy, (float)p.x, (float)p.y, -1.0f, -ey * l, ex * l, a.gw, c0, c1)) {
                            lo = min(lo, c0);
                            hi = max(hi, c1);
                        }
                    }
                }
                const int *row = S.cell_start + cy * a.gw;
                const int s0 = lo <= hi ? row[lo] : 0, e0 = lo <= hi ? row[hi + 1] : 0;
                r_start[cy] = s0;
                r_len[cy] = e0 - s0;
                tot += e0 - s0;
            }
            tot = __reduce_add_sync(0xFFFFFFFFu, tot);
            if (lane == 0 && tot) atomicAdd(&sh.total, tot);
            __syncthreads();
            int stride = sh.total > kDtSampleMin && round < 4 ? sh.total / (kDtSampleMin / 4) : 1;
            for (;;) {
                for (int cy = warp; cy < a.gh; cy += kDtBlockThreads / 32) {
                    const int s0 = r_start[cy], len = r_len[cy];
                    for (int j0 = stride > 1 ? (cy * 5) % stride : 0; j0 < len; j0 += 32 * stride) {
                        const int j = j0 + lane * stride;
                        bool hit = false;
                        DtPt q{0, 0, 0};
                        if (j < len) {
                            const int4 t = S.pts[s0 + j];
                            if (t.w && t.z != p.z) {
                                q = DtPt{t.x - p.x, t.y - p.y, t.z};
                                for (int b = 0; b < nbad && !hit; ++b) hit = dt_violates(sh.bad[b], p.z, q);
                                if (ends) {
                                    hit = hit || (open_l && el.x * q.y - el.y * q.x > 0);
                                    hit = hit || (open_r && er.x * q.y - er.y * q.x < 0);
                                }
                            }
                        }
                        const unsigned m = __ballot_sync(0xFFFFFFFFu, hit);
                        if (!m) continue;
                        int base = 0;
                        if (lane == 0) base = atomicAdd(&sh.found, __popc(m));
                        const int pos = k + __shfl_sync(0xFFFFFFFFu, base, 0) + __popc(m & ((1u << lane) - 1u));
                        if (hit && pos < kDtCacheCap) cand[pos] = dt_pack(q.x, q.y, q.z);
                    }
                }
                __syncthreads();
                found = sh.found;
                __syncthreads();
                if (stride == 1 || found > 0) break;
                stride = 1;
            }
            if (found) break;  // wrap again before the other circles
        }
        if (found == 0) break;
        if (k + found <= kDtCacheCap) {
            k += found;
            continue;
        }
        // full: wrap the whole star over the cache and keep only its vertices
        // (no disc certifies its circles any more)
        fan = false;
        R = 0;
        if (tid == 0) {
            sh.over = 0;
            sh.closed = 0;
        }
        dt_block_wrap(cand, kDtCacheCap, p.z, false, nn, sh);
        if (sh.over) {
            dt_block_star_all(S, p, n, nn, sh);
            return;
        }
        const int na = sh.nv[0] + (sh.closed ? 0 : 1);
        for (int j = tid; j < na; j += kDtBlockThreads) cand[j] = sh.vert[0][j];
        for (int j = tid; j < sh.nv[1]; j += kDtBlockThreads) cand[na + j] = sh.vert[1][j + 1];
        k = na + sh.nv[1];
        __syncthreads();
    }
    if (warp == 0) dt_block_write(S, p.z, fan, nn.z, sh);
    __syncthreads();
}

// One pair, persistent (every CTA resident): the CTAs take the stars of
// both sides' queues from one atomic counter, the two queues interleaved so
// that both sides' stars start in the first wave (the pass lasts as long as
// its longest star, so none should wait behind the other side's).  The
// counter is side 0's npending2, which dt_init_kernel zeroes and the one-pair
// passes leave unused.
__global__ void __launch_bounds__(kDtBlockThreads, kDtBlocksPerSM) dt_pass_block_kernel(DtArgs a, int nsides) {
    extern __shared__ int2 s_cand[];  // [kDtCacheCap], then the region rows
    __shared__ DtStarShared sh;
    __shared__ int s_item;
    int *r_start = reinterpret_cast<int *>(s_cand + kDtCacheCap);
    const int n = min(max(*a.count, 0), a.cap);
    const int nq0 = *a.s[0].npending, nq1 = nsides > 1 ? *a.s[1].npending : 0;
    const int m = min(nq0, nq1), total = nq0 + nq1;
    int32_t *counter = a.s[0].npending2;
    for (;;) {
        if (threadIdx.x == 0) s_item = atomicAdd(counter, 1);
        __syncthreads();
        const int item = s_item;
        __syncthreads();
        if (item >= total) break;
        const bool two = item < 2 * m;
        const int side = two ? (item & 1) : (nq0 > nq1 ? 0 : 1);
        const int idx = two ? (item >> 1) : item - m;
        const DtSide &S = a.s[side];
        dt_block_item(a, S, S.pending[idx], n, !(*S.err & 8), s_cand, r_start, r_start + a.gh, sh);
    }
}

// Many pairs, persistent: the queues of every (pair, side) of the launch are
// concatenated in launch order and the CTAs take their entries one at a
// time from one atomic counter (zeroed by dt_init_kernel_b), so the long
// stars of one pair overlap the work of all the others.  second: the middle
// pass's queues; else the warp pass's (a batch of one pair, which skips the
// middle pass).
__global__ void __launch_bounds__(kDtBlockThreads, kDtBlocksPerSM)
    dt_pass_block_kernel_b(const DtArgs *__restrict__ tab, VMap vm, int nsides, int32_t *counter, int second) {
    extern __shared__ int2 s_cand[];
    __shared__ DtStarShared sh;
    __shared__ int s_pre[2 * kMaxBatch + 1];
    __shared__ int s_item;
    const int tid = threadIdx.x, lane = tid & 31;
    const int nq_all = vm.n * nsides;
    // exclusive prefix of the queue lengths (warp 0; nq_all <= 2 * kMaxBatch)
    if (tid < 32) {
        constexpr int kPer = (2 * kMaxBatch + 31) / 32;
        int v[kPer], sum = 0;
#pragma unroll
        for (int j = 0; j < kPer; ++j) {
            const int q = lane * kPer + j;
            v[j] = 0;
            if (q < nq_all) {
                const DtSide &Q = slot_entry(tab, vm.stride, vm.slot[q / nsides]).s[q % nsides];
                v[j] = max(0, second ? *Q.npending2 : *Q.npending);
            }
            sum += v[j];
        }
        int incl = sum;
        for (int o = 1; o < 32; o <<= 1) {
            const int y = __shfl_up_sync(0xFFFFFFFFu, incl, o);
            if (lane >= o) incl += y;
        }
        int run = incl - sum;
#pragma unroll
        for (int j = 0; j < kPer; ++j) {
            const int q = lane * kPer + j;
            if (q <= nq_all) s_pre[q] = run;
            run += v[j];
        }
        if (lane == 31 && nq_all == 32 * kPer) s_pre[nq_all] = incl;
    }
    __syncthreads();
    const int total = s_pre[nq_all];
    int *r_start = reinterpret_cast<int *>(s_cand + kDtCacheCap);
    for (;;) {
        if (tid == 0) s_item = atomicAdd(counter, 1);
        __syncthreads();
        const int item = s_item;
        __syncthreads();
        if (item >= total) break;
        // last queue whose start is <= item
        int lo = 0, hi = nq_all - 1;
        while (lo < hi) {
            const int mid = (lo + hi + 1) >> 1;
            if (s_pre[mid] <= item)
                lo = mid;
            else
                hi = mid - 1;
        }
        const DtArgs &a = slot_entry(tab, vm.stride, vm.slot[lo / nsides]);
        const DtSide &S = a.s[lo % nsides];
        const int n = min(max(*a.count, 0), a.cap);
        const int i = (second ? S.pending2 : S.pending)[item - s_pre[lo]];
        dt_block_item(a, S, i, n, !(*S.err & 8), s_cand, r_start, r_start + a.gh, sh);
    }
}

// One CTA per side: exclusive scan of the owned counts, total = ntri.
__device__ __forceinline__ void dt_tri_scan_body(const DtArgs &a, const VB &vb) {
    // each thread scans kScanItems consecutive counts of a chunk (their loads
    // go out together), then the threads' totals are scanned across the CTA
    constexpr int kScanItems = 8;
    __shared__ int s_w[32];
    __shared__ int s_carry;
    const DtSide S = vb.y ? a.s[1] : a.s[0];
    const int n = min(max(*a.count, 0), a.cap);
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    const int chunk = kScanItems * (int)blockDim.x;
    if (tid == 0) s_carry = 0;
    __syncthreads();
    for (int base = 0; base < n; base += chunk) {
        const int i0 = base + kScanItems * tid;
        int v[kScanItems];
#pragma unroll
        for (int k = 0; k < kScanItems; ++k) v[k] = i0 + k < n ? S.owned[i0 + k] : 0;
        int tot = 0;
#pragma unroll
        for (int k = 0; k < kScanItems; ++k) tot += v[k];
        int incl = tot;
        for (int o = 1; o < 32; o <<= 1) {
            const int y = __shfl_up_sync(0xFFFFFFFFu, incl, o);
            if (lane >= o) incl += y;
        }
        if (lane == 31) s_w[wid] = incl;
        __syncthreads();
        if (wid == 0) {
            int x = lane < (int)(blockDim.x >> 5) ? s_w[lane] : 0;
            for (int o = 1; o < 32; o <<= 1) {
                const int y = __shfl_up_sync(0xFFFFFFFFu, x, o);
                if (lane >= o) x += y;
            }
            s_w[lane] = x;
        }
        __syncthreads();
        int run = s_carry + (wid ? s_w[wid - 1] : 0) + incl - tot;
#pragma unroll
        for (int k = 0; k < kScanItems; ++k) {
            if (i0 + k < n) S.offset[i0 + k] = run;
            run += v[k];
        }
        __syncthreads();
        if (tid == 0) s_carry += s_w[31];
        __syncthreads();
    }
    if (tid == 0) {
        if (s_carry > a.cap_tri) atomicOr(S.err, 2);
        *S.ntri = (*S.err & 2) ? -1 : s_carry;  // -1: the triangulation failed
    }
}

__global__ void __launch_bounds__(1024) dt_tri_scan_kernel(DtArgs a) { dt_tri_scan_body(a, vb_single()); }
__global__ void __launch_bounds__(1024) dt_tri_scan_kernel_b(const DtArgs *__restrict__ tab, VMap vm) {
    const VB vb = vb_batch(vm);
    dt_tri_scan_body(slot_entry(tab, vm.stride, vb.slot), vb);
}

// One thread per point: copy the owned triangles to their offset.
__device__ __forceinline__ void dt_emit_body(const DtArgs &a, const VB &vb) {
    const DtSide &S = a.s[vb.y];
    const int n = min(max(*a.count, 0), a.cap);
    if (*S.ntri < 0) return;
    for (int i = vb.x * blockDim.x + threadIdx.x; i < n; i += vb.gx * blockDim.x) {
        const int m = S.owned[i];
        int32_t *out = S.tri + 3 * (size_t)S.offset[i];
        const int2 *sl = S.slots + (size_t)i * kDtSlots;
        if (m > kDtSlots) sl = S.pool + sl->x;
        for (int k = 0; k < m; ++k) {
            const int2 t = sl[k];
            out[3 * k + 0] = i;
            out[3 * k + 1] = t.x;
            out[3 * k + 2] = t.y;
        }
    }
}

__global__ void dt_emit_kernel(DtArgs a) { dt_emit_body(a, vb_single()); }
__global__ void dt_emit_kernel_b(const DtArgs *__restrict__ tab, VMap vm) {
    const VB vb = vb_batch(vm);
    dt_emit_body(slot_entry(tab, vm.stride, vb.slot), vb);
}

// -------------------------------------------------------------------------
// Host side
// -------------------------------------------------------------------------

constexpr int kDtCounters = 4;  // err, npending, npending2, npool

static void dt_geom(int w, int h, int &gw, int &gh) {
    gw = (w + kDtCell - 1) / kDtCell;
    gh = (h + kDtCell - 1) / kDtCell;
}

size_t dt_side_bytes(int cap, int w, int h) {
    int gw, gh;
    dt_geom(w, h, gw, gh);
    const size_t c = (size_t)(cap > 0 ? cap : 1);
    const size_t cells = (size_t)gw * gh + 1;
    return 2 * align_up(c * 4, 256) + align_up(c * 16, 256) + align_up(c * 4, 256) + 3 * align_up(cells * 4, 256) +
           2 * align_up(c * 4, 256) + align_up(c * kDtSlots * 8, 256) + align_up(2 * c * 8, 256) +
           2 * align_up(c * 4, 256) + 2 * align_up((size_t)h * 4, 256) + align_up(kDtCounters * 4, 256);
}

static DtSide dt_carve(void *ws, int cap, int w, int h) {
    int gw, gh;
    dt_geom(w, h, gw, gh);
    const size_t c = (size_t)(cap > 0 ? cap : 1);
    const size_t cells = (size_t)gw * gh + 1;
    char *b = reinterpret_cast<char *>(ws);
    DtSide s{};
    auto take = [&](size_t bytes) {
        char *r = b;
        b += align_up(bytes, 256);
        return r;
    };
    s.X = reinterpret_cast<int32_t *>(take(c * 4));
    s.Y = reinterpret_cast<int32_t *>(take(c * 4));
    s.pts = reinterpret_cast<int4 *>(take(c * 16));
    s.slot = reinterpret_cast<int32_t *>(take(c * 4));
    s.cell_cnt = reinterpret_cast<int32_t *>(take(cells * 4));
    s.cell_start = reinterpret_cast<int32_t *>(take(cells * 4));
    s.cell_fill = reinterpret_cast<int32_t *>(take(cells * 4));
    s.owned = reinterpret_cast<int32_t *>(take(c * 4));
    s.offset = reinterpret_cast<int32_t *>(take(c * 4));
    s.slots = reinterpret_cast<int2 *>(take(c * kDtSlots * 8));
    s.pool = reinterpret_cast<int2 *>(take(2 * c * 8));  // a mesh has fewer than 2n triangles
    s.pending = reinterpret_cast<int32_t *>(take(c * 4));
    s.pending2 = reinterpret_cast<int32_t *>(take(c * 4));
    s.rowmin = reinterpret_cast<int32_t *>(take((size_t)h * 4));
    s.rowmax = reinterpret_cast<int32_t *>(take((size_t)h * 4));
    int32_t *counters = reinterpret_cast<int32_t *>(take(kDtCounters * 4));
    s.err = counters;
    s.npending = counters + 1;
    s.npending2 = counters + 2;
    s.npool = counters + 3;
    return s;
}

__global__ void __launch_bounds__(256) dt_init_kernel(DtArgs a);

// Triangulates one or both sides.  sides[i] = right flag; tri/ntri per side.
elas_status launch_triangulate_device(const int16_t *list, const int32_t *count, int cap, int w, int h, int nsides,
                                      const int *rights, int32_t *const *tri, int32_t *const *ntri, int cap_tri,
                                      void *ws, cudaStream_t st) {
    DtArgs a{};
    a.list = list;
    a.count = count;
    a.cap = cap;
    a.cap_tri = cap_tri;
    a.w = w;
    a.h = h;
    dt_geom(w, h, a.gw, a.gh);
    const size_t side_bytes = dt_side_bytes(cap, w, h);
    for (int i = 0; i < nsides; ++i) {
        a.s[i] = dt_carve(reinterpret_cast<char *>(ws) + i * side_bytes, cap, w, h);
        a.s[i].right = rights[i];
        a.s[i].tri = tri[i];
        a.s[i].ntri = ntri[i];
    }
    // counters, cell counts and row extremes of both sides: one kernel
    const int nall = a.gw * a.gh + 1 + 2 * h + kDtCounters;
    dt_init_kernel<<<dim3((nall + 255) / 256, nsides), 256, 0, st>>>(a);
    const int tb = 256;
    const int pblocks = max(1, min((cap + tb - 1) / tb, sm_count() * 8));
    dt_points_kernel<<<dim3(pblocks, nsides), tb, 0, st>>>(a);
    dt_cell_scan_kernel<<<dim3(1, nsides), 1024, 0, st>>>(a);
    dt_scatter_kernel<<<dim3(pblocks, nsides), tb, 0, st>>>(a);
    dt_dedup_kernel<<<dim3(pblocks, nsides), tb, 0, st>>>(a);
    // one pair: the CTA pass takes the warp pass's queue directly (its time is
    // that of its longest star, which a middle pass would not shorten)
    dt_pass1_kernel<<<dim3(max(1, min((cap + kDtWarps - 1) / kDtWarps, sm_count() * 16)), nsides), kDtWarps * 32, 0,
                      st>>>(a);
    const int smem = kDtCacheCap * (int)sizeof(int2) + 2 * a.gh * (int)sizeof(int);
    if (cudaFuncSetAttribute(dt_pass_block_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, smem) != cudaSuccess)
        return launch_status("dt_pass_block_kernel shared memory attribute");
    dt_pass_block_kernel<<<sm_count() * kDtBlocksPerSM, kDtBlockThreads, smem, st>>>(a, nsides);
    dt_tri_scan_kernel<<<dim3(1, nsides), 1024, 0, st>>>(a);
    dt_emit_kernel<<<dim3(pblocks, nsides), tb, 0, st>>>(a);
    return launch_status("triangulation kernels");
}

// Batched launches keep no memsets: this kernel clears the counters and the
// row extremes of every (pair, side), and the CTA pass's queue counter.
__device__ __forceinline__ void dt_init_body(const DtArgs &a, const VB &vb, int32_t *counter) {
    const DtSide &S = a.s[vb.y];
    const int ncell1 = a.gw * a.gh + 1;
    const int nall = ncell1 + 2 * a.h + kDtCounters;
    if (counter && blockIdx.x == 0 && threadIdx.x == 0) *counter = 0;
    for (int k = vb.x * blockDim.x + threadIdx.x; k < nall; k += vb.gx * blockDim.x) {
        if (k < ncell1)
            S.cell_cnt[k] = 0;
        else if (k < ncell1 + a.h)
            S.rowmin[k - ncell1] = 0x7F7F7F7F;
        else if (k < ncell1 + 2 * a.h)
            S.rowmax[k - ncell1 - a.h] = (int32_t)0x80808080u;
        else
            S.err[k - ncell1 - 2 * a.h] = 0;
    }
}

__global__ void __launch_bounds__(256) dt_init_kernel(DtArgs a) { dt_init_body(a, vb_single(), nullptr); }
__global__ void __launch_bounds__(256) dt_init_kernel_b(const DtArgs *__restrict__ tab, VMap vm, int32_t *counter) {
    const VB vb = vb_batch(vm);
    dt_init_body(slot_entry(tab, vm.stride, vb.slot), vb, counter);
}

static int dt_point_blocks(int cap, int threads, int npairs) {
    // grid-stride kernels: about a third of the capacity per sweep in a
    // batch (the support list holds a fraction of the lattice), capped
    const int full = (cap + threads - 1) / threads;
    if (npairs <= 1) return max(1, min(full, sm_count() * 8));
    return max(1, min((full + 2) / 3, sm_count() * 8));
}

elas_status launch_triangulate_b(const DtArgs *tab, const DtArgs *host, const VMap &pairs, int nsides,
                                 int32_t *counter, cudaStream_t st) {
    if (pairs.n == 0) return ELAS_OK;
    if (nsides < 1 || nsides > 2) return fail(ELAS_ERR_INVALID_ARG, "nsides %d", nsides);
    VMap m_init, m_pts, m_scan, m_grp, m_grp2;
    vmap_clear(m_init, pairs.stride);
    vmap_clear(m_pts, pairs.stride);
    vmap_clear(m_scan, pairs.stride);
    vmap_clear(m_grp, pairs.stride);
    vmap_clear(m_grp2, pairs.stride);
    int max_gh = 1;
    for (int i = 0; i < pairs.n; ++i) {
        const int slot = pairs.slot[i];
        const DtArgs &a = slot_entry(host, pairs.stride, slot);
        const int nall = a.gw * a.gh + 1 + 2 * a.h + kDtCounters;
        vmap_add(m_init, slot, dim3((nall + 255) / 256, nsides));
        vmap_add(m_pts, slot, dim3(dt_point_blocks(a.cap, 256, pairs.n), nsides));
        vmap_add(m_scan, slot, dim3(1, nsides));
        vmap_add(m_grp, slot, dim3(dt_point_blocks(a.cap, kDtWarps, pairs.n), nsides));
        // the middle pass gets a few percent of the points (grid-stride over
        // the queue)
        vmap_add(m_grp2, slot, dim3(max(1, min(sm_count(), a.cap / 128)), nsides));
        max_gh = max(max_gh, a.gh);
    }
    const int smem = kDtCacheCap * (int)sizeof(int2) + 2 * max_gh * (int)sizeof(int);
    if (cudaFuncSetAttribute(dt_pass_block_kernel_b, cudaFuncAttributeMaxDynamicSharedMemorySize, smem) != cudaSuccess)
        return launch_status("dt_pass_block_kernel_b shared memory attribute");
    dt_init_kernel_b<<<vmap_total(m_init), 256, 0, st>>>(tab, m_init, counter);
    dt_points_kernel_b<<<vmap_total(m_pts), 256, 0, st>>>(tab, m_pts);
    dt_cell_scan_kernel_b<<<vmap_total(m_scan), 1024, 0, st>>>(tab, m_scan);
    dt_scatter_kernel_b<<<vmap_total(m_pts), 256, 0, st>>>(tab, m_pts);
    dt_dedup_kernel_b<<<vmap_total(m_pts), 256, 0, st>>>(tab, m_pts);
    dt_pass1_kernel_b<<<vmap_total(m_grp), kDtWarps * 32, 0, st>>>(tab, m_grp);
    const int middle = pairs.n > 1;
    if (middle) dt_pass1m_kernel_b<<<vmap_total(m_grp2), kDtWarpsM * 32, 0, st>>>(tab, m_grp2);
    dt_pass_block_kernel_b<<<sm_count() * kDtBlocksPerSM, kDtBlockThreads, smem, st>>>(tab, pairs, nsides, counter,
                                                                                       middle);
    dt_tri_scan_kernel_b<<<vmap_total(m_scan), 1024, 0, st>>>(tab, m_scan);
    dt_emit_kernel_b<<<vmap_total(m_pts), 256, 0, st>>>(tab, m_pts);
    return launch_status("batched triangulation kernels");
}

// Argument block of one pair's triangulation (both sides), for the tables
// of batched launches.
DtArgs triangulate_args(const int16_t *list, const int32_t *count, int cap, int w, int h, int32_t *const *tri,
                        int32_t *const *ntri, int cap_tri, void *ws) {
    DtArgs a{};
    a.list = list;
    a.count = count;
    a.cap = cap;
    a.cap_tri = cap_tri;
    a.w = w;
    a.h = h;
    dt_geom(w, h, a.gw, a.gh);
    const size_t side_bytes = dt_side_bytes(cap, w, h);
    for (int i = 0; i < 2; ++i) {
        a.s[i] = dt_carve(reinterpret_cast<char *>(ws) + i * side_bytes, cap, w, h);
        a.s[i].right = i;
        a.s[i].tri = tri[i];
        a.s[i].ntri = ntri[i];
    }
    return a;
}

size_t triangulate_device_workspace(int cap, int w, int h, int nsides) { return nsides * dt_side_bytes(cap, w, h); }

}  // namespace elas

extern "C" size_t elas_triangulate_device_workspace_bytes(int32_t cap, int32_t w, int32_t h) {
    if (cap < 0 || w < 1 || h < 1) return 0;
    return elas::triangulate_device_workspace(cap, w, h, 1);
}

extern "C" elas_status elas_triangulate_device(const int16_t *list, const int32_t *count, int32_t cap, int32_t w,
                                               int32_t h, int32_t right, int32_t *tri, int32_t cap_tri,
                                               int32_t *ntri, void *workspace, size_t workspace_bytes,
                                               elas_stream stream) {
    using namespace elas;
    if (w < 1 || h < 1 || w > 16383 || h > 16383) return fail(ELAS_ERR_INVALID_ARG, "image size %dx%d", w, h);
    if (!list || !count || !tri || !ntri || !workspace) return fail(ELAS_ERR_INVALID_ARG, "NULL buffer");
    if (cap < 0 || cap_tri < 2 * cap + 8)
        return fail(ELAS_ERR_CAPACITY, "triangle capacity %d below 2*cap+8 = %d", cap_tri, 2 * cap + 8);
    if (!aligned(workspace, 256)) return fail(ELAS_ERR_INVALID_ARG, "workspace not 256-byte aligned");
    if (workspace_bytes < triangulate_device_workspace(cap, w, h, 1))
        return fail(ELAS_ERR_CAPACITY, "workspace %zu < %zu bytes", workspace_bytes,
                    triangulate_device_workspace(cap, w, h, 1));
    const int rights[1] = {right ? 1 : 0};
    int32_t *tris[1] = {tri};
    int32_t *nts[1] = {ntri};
    return launch_triangulate_device(list, count, cap, w, h, 1, rights, tris, nts, cap_tri, workspace,
                                     to_stream(stream));
}

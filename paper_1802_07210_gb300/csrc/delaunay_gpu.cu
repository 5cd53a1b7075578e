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
//   2. Middle pass (batches): the others again, with 48 pixels.
//   3. CTA pass: one CTA per star left (the hull, the rims of empty areas):
//      the star over the points within 48 pixels, then scans of the cells
//      that its wide circles meet until they are empty (dt_block_item).
// The output order is deterministic: an exclusive scan of the per-point
// counts, and within a star counter-clockwise from the nearest neighbour (an
// open star then clockwise from it).
//
// The earlier design (4 or 16 lanes per star, the whole star, 64-bit key
// comparisons, one region scan per step of a wide star) against this one, all
// triangulation kernels: 640x480 172 -> 69 us, 1920x1080 590 -> 207 us,
// 64 x 1242x375 3.44 -> 1.33 ms.  Sound with the limits below: the extents
// that the integer steps hold, and the room in the pool.
#include <climits>

#include "launch.cuh"
#include "elas_probe.h"

namespace elas {

constexpr int kDtCell = 16;

// Bits of DtSide::err.  Pool and range: the triangulation fails (ntri = -1).
constexpr int kDtErrPool = 4;    // the pool has no room for a fan
constexpr int kDtErrOrder = 8;   // the list is not in raster order
constexpr int kDtErrBox = 16;    // a point lies outside the box below
constexpr int kDtErrRange = 32;  // the points lie too far apart for the integer steps

// The integer steps are exact, and so the stars agree with one another, while
// X^2 + Y^2 < 2^31 for the extents X and Y of the points: |N| = |c.(c - e)| and
// |c|^2 are at most that, D at most X Y.  Points inside this box meet it, and
// it holds every point of an image and its disparities; the extents are only
// taken (dt_scatter_body) when a point lies outside.
constexpr int kDtBoxX0 = -8192, kDtBoxX1 = 32767, kDtBoxY0 = -4096, kDtBoxY1 = 17407;
static_assert((int64_t)(kDtBoxX1 - kDtBoxX0) * (kDtBoxX1 - kDtBoxX0) +
                      (int64_t)(kDtBoxY1 - kDtBoxY0) * (kDtBoxY1 - kDtBoxY0) < (int64_t)1 << 31,
              "points of the box meet the integer steps' range");

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
        if (i > 0 && a.list[3 * i - 2] > v) atomicOr(S.err, kDtErrOrder);
        if (x < kDtBoxX0 || x > kDtBoxX1 || v < kDtBoxY0 || v > kDtBoxY1) atomicOr(S.err, kDtErrBox);
        atomicAdd(S.cell_cnt + dt_cell(a, x, v), 1);
        // the lanes of one image row (a run of the raster-ordered list) take
        // its extremes with one atomic each
        const unsigned row = __match_any_sync(__activemask(), v);
        const int x0 = __reduce_min_sync(row, x), x1 = __reduce_max_sync(row, x);
        if (v >= 0 && v < a.h && (threadIdx.x & 31) == __ffs(row) - 1) {
            atomicMin(S.rowmin + v, x0);
            atomicMax(S.rowmax + v, x1);
        }
    }
}

__global__ void dt_points_kernel(DtArgs a) {
    after_previous();
    dt_points_body(a, vb_single());
}
__global__ void dt_points_kernel_b(const DtArgs *__restrict__ tab, VMap vm) {
    const VB vb = vb_batch(vm);
    dt_points_body(slot_entry(tab, vm.stride, vb.slot), vb);
}

// Exclusive scan of v[0..n-1] (16-byte aligned) by one CTA of up to 32 warps;
// put(i, four sums) for every fourth i (entries past n are to be dropped);
// returns the total.  Each warp takes one contiguous part and reads it twice
// (sums, then prefixes), four values a lane and the next ones in flight, so
// the CTA meets only once: a chunk of the whole CTA at a time, with two
// barriers each, took 32.7 us instead of 10.6 for the 41,000 points of a
// 1920x1080 pair.
template <class Put> __device__ __forceinline__ int dt_block_scan(const int32_t *v, int n, Put put) {
    __shared__ int s_sum[32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    const int part = ((n + nw - 1) / nw + 127) & ~127;
    const int i0 = min(n, warp * part), i1 = min(n, i0 + part);
    auto load = [&](int i) {
        int4 q = make_int4(0, 0, 0, 0);
        if (i < i1) {
            q = *reinterpret_cast<const int4 *>(v + i);
            if (i + 1 >= i1) q.y = 0;
            if (i + 2 >= i1) q.z = 0;
            if (i + 3 >= i1) q.w = 0;
        }
        return q;
    };
    int sum = 0;
#pragma unroll 4
    for (int i = i0 + 4 * lane; i < i1; i += 128) {
        const int4 q = load(i);
        sum += q.x + q.y + q.z + q.w;
    }
    sum = __reduce_add_sync(0xFFFFFFFFu, sum);
    if (lane == 0) s_sum[warp] = sum;
    __syncthreads();
    const int mine = lane < nw ? s_sum[lane] : 0;
    int run = __reduce_add_sync(0xFFFFFFFFu, lane < warp ? mine : 0);
    const int total = __reduce_add_sync(0xFFFFFFFFu, mine);
    int4 next = load(i0 + 4 * lane);
    for (int i = i0 + 4 * lane; i - 4 * lane < i1; i += 128) {
        const int4 q = next;
        next = load(i + 128);
        const int own = q.x + q.y + q.z + q.w;
        int incl = own;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int y = __shfl_up_sync(0xFFFFFFFFu, incl, o);
            if (lane >= o) incl += y;
        }
        const int x = run + incl - own;
        if (i < i1) put(i, make_int4(x, x + q.x, x + q.x + q.y, x + q.x + q.y + q.z));
        run += __shfl_sync(0xFFFFFFFFu, incl, 31);
    }
    return total;
}

// One CTA per side: where each cell's points start; entry ncell is the total
// (its own count stays 0).  The arrays are padded to 16 bytes.
__device__ __forceinline__ void dt_cell_scan_body(const DtArgs &a, const VB &vb) {
    const DtSide &S = a.s[vb.y];
    dt_block_scan(S.cell_cnt, dt_ncell(a) + 1, [&](int i, const int4 &before) {
        *reinterpret_cast<int4 *>(S.cell_start + i) = before;
        *reinterpret_cast<int4 *>(S.cell_fill + i) = before;
    });
}

__global__ void __launch_bounds__(1024) dt_cell_scan_kernel(DtArgs a) {
    after_previous();
    dt_cell_scan_body(a, vb_single());
}
__global__ void __launch_bounds__(1024) dt_cell_scan_kernel_b(const DtArgs *__restrict__ tab, VMap vm) {
    const VB vb = vb_batch(vm);
    dt_cell_scan_body(slot_entry(tab, vm.stride, vb.slot), vb);
}

// Sets kDtErrRange when the points' extents are beyond the integer steps.
__device__ __noinline__ void dt_check_extents(const int32_t *X, const int32_t *Y, int n, int32_t *err) {
    __shared__ int s_ext[4];
    if (threadIdx.x < 4) s_ext[threadIdx.x] = threadIdx.x & 1 ? INT_MIN : INT_MAX;
    __syncthreads();
    int x0 = INT_MAX, x1 = INT_MIN, y0 = INT_MAX, y1 = INT_MIN;
    for (int i = threadIdx.x; i < n; i += blockDim.x) {
        x0 = min(x0, X[i]);
        x1 = max(x1, X[i]);
        y0 = min(y0, Y[i]);
        y1 = max(y1, Y[i]);
    }
    atomicMin(&s_ext[0], x0);
    atomicMax(&s_ext[1], x1);
    atomicMin(&s_ext[2], y0);
    atomicMax(&s_ext[3], y1);
    __syncthreads();
    const int64_t ex = (int64_t)s_ext[1] - s_ext[0], ey = (int64_t)s_ext[3] - s_ext[2];
    if (threadIdx.x == 0 && ex * ex + ey * ey >= (int64_t)1 << 31) atomicOr(err, kDtErrRange);
}

__device__ __forceinline__ void dt_scatter_body(const DtArgs &a, const VB &vb) {
    const DtSide S = vb.y ? a.s[1] : a.s[0];
    const int n = min(max(*a.count, 0), a.cap);
    const int err = vb.x == 0 ? *S.err : 0;
    for (int i = vb.x * blockDim.x + threadIdx.x; i < n; i += vb.gx * blockDim.x) {
        const int x = S.X[i], y = S.Y[i];
        const int k = atomicAdd(S.cell_fill + dt_cell(a, x, y), 1);
        S.pts[k] = make_int4(x, y, i, 1);
        S.slot[i] = k;
    }
    if (err & kDtErrBox) dt_check_extents(S.X, S.Y, n, S.err);
}

__global__ void dt_scatter_kernel(DtArgs a) {
    after_previous();
    dt_scatter_body(a, vb_single());
}
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
        const int k0 = S.cell_start[c], k1 = S.cell_start[c + 1];
        for (int k = k0; k < k1; k += 4) {  // four loads in flight
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const int4 q = S.pts[min(k + u, k1 - 1)];
                dup |= q.x == x && q.y == y && q.z < i;
            }
        }
        if (dup) S.pts[S.slot[i]].w = 0;
    }
}

__global__ void dt_dedup_kernel(DtArgs a) {
    after_previous();
    dt_dedup_body(a, vb_single());
}
__global__ void dt_dedup_kernel_b(const DtArgs *__restrict__ tab, VMap vm) {
    const VB vb = vb_batch(vm);
    dt_dedup_body(slot_entry(tab, vm.stride, vb.slot), vb);
}

// -------------------------------------------------------------------------
// Stars
// -------------------------------------------------------------------------

constexpr int kDtSlots = 16;       // owned triangles kept per point; larger fans go to the pool
constexpr int kDtRadius = 24;      // warp pass: candidates within this many pixels
constexpr int kDtNearCap = 64;     // and at most this many, two per lane (else the nearer ones of 16 or 8 pixels)
constexpr int kDtRadiusM = 48;     // middle pass
constexpr int kDtListCapM = 320;   // a radius-48 disc holds about 290 points of a full step-5 lattice
constexpr float kDtWideMax = 96.0f;  // the middle pass searches circles up to this radius
constexpr int kDtWarps = 8;        // stars per CTA of the warp pass
constexpr int kDtWarpsM = 4;       // stars per CTA of the middle pass
constexpr float kDtInf = 3.402823466e38f;  // "no candidate" key (every real key is far below)

__device__ __forceinline__ float dt_warp_min(float v) {
    float r;
    asm volatile("redux.sync.min.f32 %0, %1, 0xffffffff;" : "=f"(r) : "f"(v));
    return r;
}

// n / d for an integer-valued d >= 1, off by at most 2^-22.4 (relatively).
__device__ __forceinline__ float dt_div(float n, float d) {
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(d));
    return n * r;
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

// Is the circle of edge (p, e) with pencil parameter t no wider than R
// (2r <= R)?  Its centre lies |e|/2 along the edge and t |e|/2 off it, so
// 4 r^2 = |e|^2 (1 + t^2); with a margin far above the FP32 rounding of t (a
// false answer only sends a star to the next pass).
__device__ __forceinline__ bool dt_small_circle(float e2, float t, float R2) {
    return e2 * __fmaf_rn(t, t, 1.0f) * 1.0001f <= R2;
}

struct DtPt {
    int x, y, z;  // relative to the star's point; list index
};

// Candidates are (x, y, |c|^2, index) in FP32, coordinates relative to p.
__device__ __forceinline__ float4 dt_cand(int x, int y, int z) {
    return make_float4((float)x, (float)y, (float)(x * x + y * y), __int_as_float(z));
}
__device__ __forceinline__ DtPt dt_point(const float4 &v) {
    return DtPt{(int)v.x, (int)v.y, __float_as_int(v.w)};
}
__device__ __forceinline__ float4 dt_no_cand() {  // D = 0 and y = 0: never a candidate
    return make_float4(0.0f, 0.0f, 0.0f, 0.0f);
}

// N and D of candidate c; exact in FP32 while every coordinate is below 2048
// (all values then stay below 2^24).
constexpr int kDtNearMax = 2048;
__device__ __forceinline__ float dt_n(const float4 &e, const float4 &c) {
    return __fmaf_rn(-e.x, c.x, __fmaf_rn(-e.y, c.y, c.z));
}
__device__ __forceinline__ float dt_d(const float4 &e, const float4 &c, float side) {
    return side * __fmaf_rn(e.x, c.y, -(e.y * c.x));
}

// Does c2 beat c1 for edge (p, e) on `side`, exactly (coordinates below
// 2048)?  The cross products N2 D1 and N1 D2 compare by their rounded values
// (rounding is monotone) and, when those are equal, by their exact errors.
__device__ __forceinline__ bool dt_beats(const float4 &e, int pz, const float4 &c1, const float4 &c2, float side) {
    const float N1 = dt_n(e, c1), D1 = dt_d(e, c1, side), N2 = dt_n(e, c2), D2 = dt_d(e, c2, side);
    const float l = N2 * D1, r = N1 * D2;
    if (l != r) return l < r;
    const float le = __fmaf_rn(N2, D1, -l), re = __fmaf_rn(N1, D2, -r);
    if (le != re) return le < re;
    const int z1 = __float_as_int(c1.w), z2 = __float_as_int(c2.w);
    return z1 != z2 && dt_tie_second(pz, __float_as_int(e.w), z1, z2, side * (c1.x * c2.y - c1.y * c2.x) > 0.0f);
}

// The same in integers, for coordinate differences below 2^14.5 (N and D fit
// 32 bits).
__device__ __forceinline__ bool dt_beats(const DtPt &e, int pz, const DtPt &c1, const DtPt &c2, int side) {
    const int D1 = side * (e.x * c1.y - e.y * c1.x), D2 = side * (e.x * c2.y - e.y * c2.x);
    const int N1 = c1.x * c1.x + c1.y * c1.y - (e.x * c1.x + e.y * c1.y);
    const int N2 = c2.x * c2.x + c2.y * c2.y - (e.x * c2.x + e.y * c2.y);
    const int64_t l = (int64_t)N2 * D1, r = (int64_t)N1 * D2;
    if (l != r) return l < r;
    if (c1.z == c2.z) return false;
    return dt_tie_second(pz, e.z, c1.z, c2.z, side * ((int64_t)c1.x * c2.y - (int64_t)c1.y * c2.x) > 0);
}

// Winner of a warp's lanes, those with `in` offering candidate own(at): the
// band's members ordered exactly, champion against challengers.  get(at) on
// every lane: the candidate that some lane offered.
template <class Pt, class Get, class Own, class Beats>
__device__ __forceinline__ int dt_champion(bool in, int at, Get get, Own own, Beats beats, Pt &w) {
    unsigned b = __ballot_sync(0xFFFFFFFFu, in);
    int ch = __shfl_sync(0xFFFFFFFFu, at, __ffs(b) - 1);
    w = get(ch);
    if (b & (b - 1)) {
        const Pt mine = own(at);
        do {
            in = in && at != ch && beats(w, mine);
            b = __ballot_sync(0xFFFFFFFFu, in);
            if (!b) break;
            ch = __shfl_sync(0xFFFFFFFFu, at, __ffs(b) - 1);
            w = get(ch);
        } while (b & (b - 1));
    }
    return ch;
}

// One wrap step by a warp over points given as integers by get(0..k-1)
// (coordinate differences below 2^14.5; the keys' rounding to FP32 and the
// division leave a relative error below 2^-20).  The winner's position in at.
// Four points in flight, and no second walk while a lane's second least key
// lies outside the band: an apex of 3,000 neighbours takes 29.8 ms, 66.8
// without (the earlier pass with twice the threads 54.1).
template <class Get>
__device__ __forceinline__ bool dt_step_int(Get get, int k, int lane, const DtPt &e, int pz, int side, DtPt &w,
                                            int &at) {
    auto key = [&](const DtPt &q) {
        const int D = side * (e.x * q.y - e.y * q.x), N = q.x * q.x + q.y * q.y - (e.x * q.x + e.y * q.y);
        return D > 0 ? dt_div((float)N, (float)D) : kDtInf;
    };
    float f1 = kDtInf, f2 = kDtInf;  // least and second least key of the lane
    int c1 = -1;
#pragma unroll 4
    for (int c = lane; c < k; c += 32) {
        const float f = key(get(c));
        f2 = fminf(f2, fmaxf(f1, f));
        if (f < f1) {
            f1 = f;
            c1 = c;
        }
    }
    const float fm = dt_warp_min(f1);
    if (fm == kDtInf) return false;
    const float thr = fm + 0x1p-17f * fabsf(fm);
    const bool in = f1 <= thr;
    if (in && f2 <= thr) {  // several of this lane's candidates: its exact best
        DtPt bq = get(c1);
        for (int c = lane; c < k; c += 32) {
            const DtPt q = get(c);
            if (c == c1 || key(q) > thr || !dt_beats(e, pz, bq, q, side)) continue;
            c1 = c;
            bq = q;
        }
    }
    at = dt_champion(
        in, c1, get, [&](int c) { return get(max(0, c)); },
        [&](const DtPt &a, const DtPt &b) { return dt_beats(e, pz, a, b, side); }, w);
    return true;
}

// A star's candidates in shared memory.  near: all below 2048, so that the
// FP32 arithmetic is exact but for the division.
struct DtListSrc {
    const float4 *list;
    int k;
    bool near;
    __device__ __forceinline__ DtListSrc(const float4 *l, int n, bool exact, int) : list(l), k(n), near(exact) {}

    // Least key over the list (kDtInf: no candidate) and the winner, the
    // keys' band (2^-17, far above the division's error) ordered by beats.
    // Four candidates a lane at a time, so that their latencies overlap.
    template <class Key, class Beats>
    __device__ __forceinline__ float select(int lane, Key key, Beats beats, float4 &w, int &at) const {
        float f1 = kDtInf, f2 = kDtInf;
        int c1 = 0;
        for (int c0 = lane; c0 - lane < k; c0 += 128) {
            float f[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) f[u] = key(list[min(c0 + 32 * u, k - 1)]);
#pragma unroll
            for (int u = 0; u < 4; ++u)
                if (c0 + 32 * u >= k) f[u] = kDtInf;
            const float fa = fminf(f[0], f[1]), fb = fminf(f[2], f[3]), g = fminf(fa, fb);
            const float second = fminf(fmaxf(fa, fb), fa < fb ? fmaxf(f[0], f[1]) : fmaxf(f[2], f[3]));
            f2 = fminf(f2, fminf(second, fmaxf(f1, g)));
            if (g < f1) {
                f1 = g;
                c1 = c0 + (g == f[0] ? 0 : g == f[1] ? 32 : g == f[2] ? 64 : 96);
            }
        }
        const float fm = dt_warp_min(f1);
        if (fm == kDtInf) return fm;
        const float thr = __fmaf_rn(fabsf(fm), 0x1p-17f, fm);
        const bool in = f1 <= thr;
        const unsigned b = __ballot_sync(0xFFFFFFFFu, in);
        const unsigned more = __ballot_sync(0xFFFFFFFFu, f2 <= thr);
        if (!(more | (b & (b - 1)))) {
            at = __shfl_sync(0xFFFFFFFFu, c1, __ffs(b) - 1);
            w = list[at];
            return fm;
        }
        if (in && f2 <= thr) {  // several of this lane's candidates: its exact best
            float4 bq = list[c1];
            for (int c = lane; c < k; c += 32) {
                const float4 q = list[c];
                if (c == c1 || key(q) > thr || !beats(bq, q)) continue;
                c1 = c;
                bq = q;
            }
        }
        at = dt_champion(
            in, c1, [&](int c) { return list[c]; }, [&](int c) { return list[c]; }, beats, w);
        return fm;
    }
};

__device__ __noinline__ bool dt_step_far(const float4 *list, int k, int lane, const float4 &e, int pz, int side,
                                         float4 &w, int &at) {
    DtPt wi;
    const bool any = dt_step_int([&](int c) { return dt_point(list[c]); }, k, lane, dt_point(e), pz, side, wi, at);
    if (any) w = list[at];
    return any;
}

// One wrap step over a list; t: the winner's pencil parameter (near lists),
// at: its place in the list.
__device__ __forceinline__ bool dt_step(const DtListSrc &src, int lane, const float4 &e, int pz, int side, float4 &w,
                                        float &t, int &at) {
    if (!src.near) {
        t = kDtInf;
        return dt_step_far(src.list, src.k, lane, e, pz, side, w, at);
    }
    const float sd = (float)side, sx = sd * e.x, sy = sd * e.y;
    t = src.select(
        lane,
        [&](const float4 &c) {
            const float D = __fmaf_rn(sx, c.y, -(sy * c.x));
            return D > 0.0f ? dt_div(dt_n(e, c), D) : kDtInf;
        },
        [&](const float4 &c1, const float4 &c2) { return dt_beats(e, pz, c1, c2, sd); }, w, at);
    return t != kDtInf;
}

// First vertex of a fan (see dt_warp_star): the candidate below p (y > 0)
// that a circle through p growing straight down touches first, least
// |c|^2 / y; of several on that circle the first one counter-clockwise.
__device__ __forceinline__ bool dt_fan_start(const DtListSrc &src, int lane, float4 &w, int &at) {
    return src.select(
               lane, [](const float4 &c) { return c.y > 0.0f ? dt_div(c.z, c.y) : kDtInf; },
               [](const float4 &c1, const float4 &c2) {
                   const DtPt a = dt_point(c1), b = dt_point(c2);
                   const int64_t l = (int64_t)(b.x * b.x + b.y * b.y) * a.y, r = (int64_t)(a.x * a.x + a.y * a.y) * b.y;
                   if (l != r) return l < r;
                   return (int64_t)b.x * a.y - (int64_t)b.y * a.x > 0;
               },
               w, at) != kDtInf;
}

// The warp pass's candidates: at most 64 within 24 pixels of p, two per lane
// in registers as (x, y, |c|^2, index), the list in shared memory for the
// winners.  All their arithmetic is exact in FP32 but the keys' division:
// |N| <= 1152 and D <= 576, so two different keys lie at least 2^-19.3 apart
// (relatively: 1 / (|N| D)), while a computed key is off by at most 2^-22.4.  The keys within 2^-20.35 of the least one are
// therefore exactly those equal to it: the band holds ties only.
struct DtNearSrc {
    const float4 *list;
    float4 c0, c1;

    __device__ __forceinline__ DtNearSrc(const float4 *l, int k, int lane) : list(l) {
        c0 = lane < k ? list[lane] : dt_no_cand();
        c1 = lane + 32 < k ? list[lane + 32] : dt_no_cand();
    }
    // The winner of keys f0, f1 (least value fm): with ties, champion and
    // challenger in turn, beats(c1, c2): c2 before c1.
    template <class Beats>
    __device__ __forceinline__ float4 pick(float f0, float f1, float fm, Beats beats) const {
        const float thr = __fmaf_rn(fabsf(fm), 7.5e-7f, fm);
        unsigned b0 = __ballot_sync(0xFFFFFFFFu, f0 <= thr), b1 = __ballot_sync(0xFFFFFFFFu, f1 <= thr);
        auto next = [&]() {
            const float4 *l = b0 ? list : list + 32;
            const unsigned b = b0 ? b0 : b1;
            if (b0)
                b0 &= b0 - 1;
            else
                b1 &= b1 - 1;
            return l[__ffs(b) - 1];
        };
        float4 w = next();
        while (b0 | b1) {
            const float4 q = next();
            if (beats(w, q)) w = q;
        }
        return w;
    }
};

// One wrap step; t: the winner's pencil parameter.
__device__ __forceinline__ bool dt_step(const DtNearSrc &src, int, const float4 &e, int pz, int side, float4 &w,
                                        float &t, int &) {
    const float sx = side > 0 ? e.x : -e.x, sy = side > 0 ? e.y : -e.y;
    auto key = [&](const float4 &c) {
        const float D = __fmaf_rn(sx, c.y, -(sy * c.x));
        const float N = __fmaf_rn(-e.x, c.x, __fmaf_rn(-e.y, c.y, c.z));
        return D > 0.0f ? dt_div(N, D) : kDtInf;
    };
    const float f0 = key(src.c0), f1 = key(src.c1);
    t = dt_warp_min(fminf(f0, f1));
    if (t == kDtInf) return false;
    w = src.pick(f0, f1, t, [&](const float4 &c1, const float4 &c2) {
        const float o = c1.x * c2.y - c1.y * c2.x;
        return dt_tie_second(pz, __float_as_int(e.w), __float_as_int(c1.w), __float_as_int(c2.w),
                             side > 0 ? o > 0.0f : o < 0.0f);
    });
    return true;
}

__device__ __forceinline__ bool dt_fan_start(const DtNearSrc &src, int, float4 &w, int &) {
    const float f0 = src.c0.y > 0.0f ? dt_div(src.c0.z, src.c0.y) : kDtInf;
    const float f1 = src.c1.y > 0.0f ? dt_div(src.c1.z, src.c1.y) : kDtInf;
    const float fm = dt_warp_min(fminf(f0, f1));
    if (fm == kDtInf) return false;
    w = src.pick(f0, f1, fm, [](const float4 &c1, const float4 &c2) { return c2.x * c1.y - c2.y * c1.x > 0.0f; });
    return true;
}

// Nearest candidate (least |c|^2, then least index) and the open quadrants
// that hold candidates (bit 2*(y>0) + (x>0)).
__device__ __forceinline__ unsigned dt_quadrant(int x, int y) {
    return x && y ? 1u << ((x > 0) | ((y > 0) << 1)) : 0u;
}
__device__ __forceinline__ float4 dt_nearest(const DtNearSrc &src, int lane, unsigned &quads) {
    auto quad = [](const float4 &c) {
        return c.x != 0.0f && c.y != 0.0f ? 1u << ((c.x > 0.0f ? 1 : 0) | (c.y > 0.0f ? 2 : 0)) : 0u;
    };
    quads = __reduce_or_sync(0xFFFFFFFFu, quad(src.c0) | quad(src.c1));
    const float d0 = src.c0.z > 0.0f ? src.c0.z : kDtInf, d1 = src.c1.z > 0.0f ? src.c1.z : kDtInf;
    const float dm = dt_warp_min(fminf(d0, d1));
    const unsigned z = min(d0 == dm ? __float_as_uint(src.c0.w) : 0xFFFFFFFFu,
                           d1 == dm ? __float_as_uint(src.c1.w) : 0xFFFFFFFFu);
    const unsigned zm = __reduce_min_sync(0xFFFFFFFFu, z);
    const unsigned b = __ballot_sync(0xFFFFFFFFu, z == zm);
    const int at = __ffs(b) - 1;
    const float4 w = src.list[at];
    if (__float_as_uint(w.w) == zm) return w;
    return src.list[at + 32];
}
__device__ __forceinline__ float4 dt_nearest(const DtListSrc &src, int lane, unsigned &quads) {
    float d = kDtInf;
    unsigned q = 0, z = 0xFFFFFFFFu;
    int c = 0;
    for (int j = lane; j < src.k; j += 32) {
        const float4 v = src.list[j];
        const unsigned vz = __float_as_uint(v.w);
        if (v.z < d || (v.z == d && vz < z)) {
            d = v.z;
            z = vz;
            c = j;
        }
        q |= dt_quadrant((int)v.x, (int)v.y);
    }
    quads = __reduce_or_sync(0xFFFFFFFFu, q);
    const float dm = dt_warp_min(d);
    const unsigned zm = __reduce_min_sync(0xFFFFFFFFu, d == dm ? z : 0xFFFFFFFFu);
    const unsigned b = __ballot_sync(0xFFFFFFFFu, d == dm && z == zm);
    return src.list[__shfl_sync(0xFFFFFFFFu, c, __ffs(b) - 1)];
}

// Calls visit(q, inside) for the points of the cells [c0, c1] of consecutive
// cell rows from cy0 on, one row per lane (up to 16; c0 > c1: none), 32 at a
// time and two loads in flight: the rows' ranges are walked as one index
// space (a binary search over the lanes' prefix sums).
template <class Visit>
__device__ __forceinline__ void dt_warp_rows(const DtArgs &a, const DtSide &S, int cy0, int nrows, int c0, int c1,
                                             int lane, Visit visit) {
    int rs = 0, len = 0;
    if (lane < nrows && c0 <= c1) {
        const int *row = S.cell_start + (cy0 + lane) * a.gw;
        rs = row[c0];
        len = row[c1 + 1] - rs;
    }
    int incl = len;
#pragma unroll
    for (int o = 1; o < 16; o <<= 1) {
        const int y = __shfl_up_sync(0xFFFFFFFFu, incl, o);
        if (lane >= o) incl += y;
    }
    const int total = __shfl_sync(0xFFFFFFFFu, incl, 15);
    const int excl = incl - len, off = rs - excl;
    for (int t0 = 0; t0 < total; t0 += 64) {
        int4 q[2];
        bool in[2];
#pragma unroll
        for (int u = 0; u < 2; ++u) {
            const int t = t0 + 32 * u + lane;
            int lo = 0;
#pragma unroll
            for (int s = 8; s > 0; s >>= 1)
                if (t >= __shfl_sync(0xFFFFFFFFu, excl, lo + s)) lo += s;
            in[u] = t < total;
            const int at = t + __shfl_sync(0xFFFFFFFFu, off, lo);
            q[u] = in[u] ? S.pts[at] : make_int4(0, 0, 0, 0);
        }
        visit(q[0], in[0]);
        if (t0 + 32 < total) visit(q[1], in[1]);
    }
}

// A step whose circle the near list does not certify: w (parameter t) is the
// best listed third vertex of edge (p, e), so the true one is w or lies inside
// their circle (centre e/2 + side t perp(e)/2).  Every point of the cells that
// the circle meets is offered; each lane keeps its exact best, and the lanes'
// bests are ordered like dt_step's.  False: the circle is too wide.
__device__ __forceinline__ bool dt_wide_step(const DtArgs &a, const DtSide &S, const int4 &p, const float4 &e, int side,
                                             float t, int lane, float4 &w) {
    const float r = 0.5f * sqrtf(e.z * __fmaf_rn(t, t, 1.0f));
    if (!(r <= kDtWideMax)) return false;
    const float st = side > 0 ? t : -t;
    const float X = (float)p.x + 0.5f * (e.x - st * e.y), Y = (float)p.y + 0.5f * (e.y + st * e.x);
    const float rr = r * 1.001f + 1.0f;  // padded for the rounding of t and the centre
    const int cy0 = (int)fmaxf(0.0f, floorf((Y - rr) / kDtCell));
    const int cy1 = min(a.gh - 1, (int)fmaxf(0.0f, floorf((Y + rr) / kDtCell)));
    const float ya = (float)((cy0 + lane) * kDtCell) - Y, yb = ya + (float)(kDtCell - 1);
    const float dy = ya > 0.0f ? ya : (yb < 0.0f ? -yb : 0.0f);
    int c0 = 1, c1 = 0;
    if (dy <= rr) {
        const float hc = sqrtf(rr * rr - dy * dy);
        // points left of the image are in the first cell of their row
        c0 = min(a.gw - 1, (int)fmaxf(0.0f, floorf((X - hc) / kDtCell)));
        c1 = min(a.gw - 1, (int)fmaxf(0.0f, floorf((X + hc) / kDtCell)));
    }
    const float sd = (float)side, most = __fmaf_rn(fabsf(t), 0x1p-16f, t);
    float fl = kDtInf;
    float4 best = dt_no_cand();
    dt_warp_rows(a, S, cy0, cy1 - cy0 + 1, c0, c1, lane, [&](const int4 &q, bool inside) {
        const float x = (float)(q.x - p.x), y = (float)(q.y - p.y);
        const float4 c = make_float4(x, y, __fmaf_rn(x, x, y * y), __int_as_float(q.z));
        const float D = dt_d(e, c, sd);
        const float f = inside && q.w && D > 0.0f ? dt_div(dt_n(e, c), D) : kDtInf;
        if (f > most) return;
        const float band = 0x1p-17f * fabsf(f);
        if (f < fl - band || (f <= fl + band && dt_beats(e, p.z, best, c, sd))) {
            fl = f;
            best = c;
        }
    });
    const float fm = dt_warp_min(fl);
    if (fm == kDtInf) return false;
    dt_champion(
        fl <= __fmaf_rn(fabsf(fm), 0x1p-17f, fm), lane,
        [&](int src) {
            return make_float4(__shfl_sync(0xFFFFFFFFu, best.x, src), __shfl_sync(0xFFFFFFFFu, best.y, src),
                               __shfl_sync(0xFFFFFFFFu, best.z, src), __shfl_sync(0xFFFFFFFFu, best.w, src));
        },
        [&](int) { return best; },
        [&](const float4 &c1, const float4 &c2) { return dt_beats(e, p.z, c1, c2, sd); }, w);
    return true;
}

// Where triangle t of a fan of m goes in the output: the owned triangles of a
// star are written counter-clockwise from its nearest neighbour, which is
// vertex r of the fan (0 when it is none of its vertices).
__device__ __forceinline__ int dt_fan_pos(int t, int m, int r) { return t >= r ? t - r : t + m - r; }

// The owned triangles of a star whose vertices sit one per lane: a[0..na]
// counter-clockwise from the first vertex, b[0..nb] clockwise from it.  False:
// more than the point's slots hold, which the CTA pass takes to the pool (the
// pool's bound in this function took the middle pass of 64 x 1242x375 from 230
// to 241 us).
__device__ __forceinline__ bool dt_warp_write(const DtSide &S, int pz, int lane, bool fan, int va, int vb, int na,
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
    if (m > kDtSlots) return false;
    int2 *out = S.slots + (size_t)pz * kDtSlots;
    if (oa) out[pa] = make_int2(va, va1);
    if (ob) out[pb] = make_int2(vb1, vb);
    if (lane == 0) S.owned[pz] = m;
    return true;
}

// One star by a warp over the candidates within R of p; true if it came out
// certain (its owned triangles are then written).
//
// Triangles are emitted by their lowest-index vertex.  A list in raster order
// (v never decreases) puts the two others of an owned triangle level with p
// or below it, so the owned triangles are one run of consecutive sectors in
// the lower half of the star, and only that fan is wrapped: from the vertex
// that the circle growing straight down from p meets first, both ways until
// a vertex is not below p.  That is 4 steps per star on average instead of
// the whole star's 6.  It needs p strictly inside the hull (candidates in all
// four open quadrants show that) and a certain first vertex; other stars, and
// every star of an unordered list, are wrapped whole from the nearest neighbour,
// counter-clockwise and, when that meets the hull, clockwise from it again.
//
// A triangle is certain when its circle, which passes through p, is no wider
// than R (no point farther than R from p is inside it), or when its third
// vertex came from a search of the circle (WIDE: dt_wide_step).  Where a whole star
// stays open (p on the hull), nothing may lie beyond either open edge, tested
// against the extreme points of every image row.
template <bool WIDE, class Src>
__device__ __forceinline__ bool dt_warp_star(const DtArgs &a, const DtSide &S, const int4 &p, const Src &src, int R,
                                             bool ordered, int lane) {
    unsigned quads;
    const float4 nn = dt_nearest(src, lane, quads);
    bool fan = ordered && quads == 15u;
    float4 first = nn;
    if (fan) {
        int at;
        dt_fan_start(src, lane, first, at);
        // certain only when the touching circle (diameter |c|^2 / y) fits the disc
        fan = first.z <= (float)R * first.y;
        if (!fan) first = nn;
    }
    const float R2 = (float)(R * R);
    const int z0 = __float_as_int(first.w);
    int va = z0, vb = z0, na = 0, nb = 0, at;
    float4 cur = first, w;
    float t;
    bool closed = false, open = false;
    for (;;) {  // counter-clockwise
        if (!dt_step(src, lane, cur, p.z, 1, w, t, at)) {
            open = true;
            break;
        }
        if (!dt_small_circle(cur.z, t, R2)) {
            if constexpr (!WIDE) return false;
            if (!dt_wide_step(a, S, p, cur, 1, t, lane, w)) return false;
        }
        if (na == 30) return false;
        ++na;
        const int z = __float_as_int(w.w);
        if (lane == na) va = z;
        if (fan) {
            if (!(w.y > 0.0f)) break;
        } else if (z == z0) {
            closed = true;
            break;
        }
        cur = w;
    }
    if (fan && open) return false;
    const float lx = cur.x, ly = cur.y;
    cur = first;
    while (!closed) {  // clockwise
        if (!dt_step(src, lane, cur, p.z, -1, w, t, at)) {
            open = true;
            break;
        }
        if (!dt_small_circle(cur.z, t, R2)) {
            if constexpr (!WIDE) return false;
            if (!dt_wide_step(a, S, p, cur, -1, t, lane, w)) return false;
        }
        if (nb == 30) return false;
        ++nb;
        if (lane == nb) vb = __float_as_int(w.w);
        if (fan && !(w.y > 0.0f)) break;
        cur = w;
    }
    if (fan && open) return false;
    if (open) {
        const int ax = (int)lx, ay = (int)ly, bx = (int)cur.x, by = (int)cur.y;
        bool bad = false;
        for (int y = lane; y < a.h; y += 32) {
            const int x0 = S.rowmin[y], x1 = S.rowmax[y];
            if (x0 > x1) continue;
            const int dy = y - p.y, d0 = x0 - p.x, d1 = x1 - p.x;
            bad |= ax * dy - ay * d0 > 0 || ax * dy - ay * d1 > 0;
            bad |= bx * dy - by * d0 < 0 || bx * dy - by * d1 < 0;
        }
        if (__any_sync(0xFFFFFFFFu, bad)) return false;
    }
    return dt_warp_write(S, p.z, lane, fan, va, vb, na, nb, __float_as_int(nn.w));
}

// Warp pass: one warp per point, the candidates within 24 pixels (16 or 8
// where there are more than 64).  Bound by instruction issue; 64 x 1242x375
// 685 us for 0.77 M stars, 640x480 10 (whole stars by 4 or 16 lanes each: 1,590
// and 47), 1920x1080 67.
__device__ __forceinline__ void dt_pass1_body(const DtArgs &a, const VB &vb) {
    constexpr int kRows = 2 * kDtRadius / kDtCell + 1;  // cell rows (and columns) the disc's square meets
    static_assert(2 * kDtRadius % kDtCell == 0, "the square of a disc spans kRows rows wherever it lies");
    __shared__ float4 s_list[kDtWarps][kDtNearCap];
    const DtSide &S = a.s[vb.y];
    const int n = min(max(*a.count, 0), a.cap);
    const int lane = threadIdx.x & 31;
    float4 *list = s_list[threadIdx.x >> 5];
    const int err = *S.err;
    const bool ordered = !(err & kDtErrOrder);
    for (int j = vb.x * kDtWarps + (threadIdx.x >> 5); j < n; j += vb.gx * kDtWarps) {
        const int4 p = S.pts[j];
        // out of range: no star is built, the later passes find empty queues
        if (!p.w || (err & kDtErrRange)) continue;
        const int cx0 = min(a.gw - 1, max(0, p.x - kDtRadius) / kDtCell);
        const int cx1 = min(a.gw - 1, max(0, p.x + kDtRadius) / kDtCell);
        const int cy0 = max(0, p.y - kDtRadius) / kDtCell, cy1 = min(a.gh - 1, (p.y + kDtRadius) / kDtCell);
        int rs = 0, len = 0;
        if (lane <= cy1 - cy0) {
            const int *row = S.cell_start + (cy0 + lane) * a.gw;
            rs = row[cx0];
            len = row[cx1 + 1] - rs;
        }
        const int most = __reduce_max_sync(0xFFFFFFFFu, len);
        int R = kDtRadius, k;
        for (;;) {
            const float R2 = (float)(R * R);
            k = 0;
            for (int c0 = 0; c0 < most; c0 += 32) {
                int4 q[kRows];  // a chunk of every row, the loads together
#pragma unroll
                for (int r = 0; r < kRows; ++r) {
                    const int s0 = __shfl_sync(0xFFFFFFFFu, rs, r), l = __shfl_sync(0xFFFFFFFFu, len, r);
                    q[r] = c0 + lane < l ? S.pts[s0 + c0 + lane] : make_int4(0, 0, p.z, 0);
                }
#pragma unroll
                for (int r = 0; r < kRows; ++r) {
                    const float dx = (float)(q[r].x - p.x), dy = (float)(q[r].y - p.y);
                    const float d2 = __fmaf_rn(dx, dx, dy * dy);
                    const bool take = q[r].w && q[r].z != p.z && d2 <= R2;
                    const unsigned b = __ballot_sync(0xFFFFFFFFu, take);
                    const int pos = k + __popc(b & ((1u << lane) - 1u));
                    if (take && pos < kDtNearCap) list[pos] = make_float4(dx, dy, d2, __int_as_float(q[r].z));
                    k += __popc(b);
                }
            }
            if (k <= kDtNearCap || R <= 8) break;
            R -= 8;
            __syncwarp();
        }
        __syncwarp();
        bool done = false;
        if (k > 0 && k <= kDtNearCap) done = dt_warp_star<false>(a, S, p, DtNearSrc(list, k, lane), R, ordered, lane);
        if (!done && lane == 0) S.pending[atomicAdd(S.npending, 1)] = j;
        __syncwarp();
    }
}

__global__ void __launch_bounds__(kDtWarps * 32, 4) dt_pass1_kernel(const __grid_constant__ DtArgs a) {
    after_previous();
    dt_pass1_body(a, vb_single());
}
__global__ void __launch_bounds__(kDtWarps * 32, 4) dt_pass1_kernel_b(const DtArgs *__restrict__ tab, VMap vm) {
    const VB vb = vb_batch(vm);
    dt_pass1_body(slot_entry(tab, vm.stride, vb.slot), vb);
}

// Middle pass (batches): the stars left by the warp pass, again a warp each, with the
// candidates within 48 pixels and searches of wider circles.
__device__ __forceinline__ void dt_pass2_body(const DtArgs &a, const VB &vb) {
    __shared__ float4 s_list[kDtWarpsM][kDtListCapM];
    const DtSide &S = a.s[vb.y];
    const int lane = threadIdx.x & 31;
    float4 *list = s_list[threadIdx.x >> 5];
    const bool ordered = !(*S.err & kDtErrOrder);
    const int njobs = *S.npending;
    for (int j = vb.x * kDtWarpsM + (threadIdx.x >> 5); j < njobs; j += vb.gx * kDtWarpsM) {
        const int at = S.pending[j];
        const int4 p = S.pts[at];
        const int cx0 = min(a.gw - 1, max(0, p.x - kDtRadiusM) / kDtCell);
        const int cx1 = min(a.gw - 1, max(0, p.x + kDtRadiusM) / kDtCell);
        const int cy0 = max(0, p.y - kDtRadiusM) / kDtCell, cy1 = min(a.gh - 1, (p.y + kDtRadiusM) / kDtCell);
        int R = kDtRadiusM, k;
        for (;;) {
            k = 0;
            dt_warp_rows(a, S, cy0, cy1 - cy0 + 1, cx0, cx1, lane, [&](const int4 &q, bool inside) {
                const int dx = q.x - p.x, dy = q.y - p.y;
                const bool take = inside && q.w && q.z != p.z && dx * dx + dy * dy <= R * R;
                const unsigned b = __ballot_sync(0xFFFFFFFFu, take);
                const int pos = k + __popc(b & ((1u << lane) - 1u));
                if (take && pos < kDtListCapM) list[pos] = dt_cand(dx, dy, q.z);
                k += __popc(b);
            });
            if (k <= kDtListCapM || R <= 8) break;
            R >>= 1;
            __syncwarp();
        }
        __syncwarp();
        bool done = false;
        if (k > 0 && k <= kDtListCapM)
            done = dt_warp_star<true>(a, S, p, DtListSrc(list, k, true, lane), R, ordered, lane);
        if (!done && lane == 0) S.pending2[atomicAdd(S.npending2, 1)] = at;
        __syncwarp();
    }
}

__global__ void __launch_bounds__(kDtWarpsM * 32, 7) dt_pass2_kernel_b(const DtArgs *__restrict__ tab, VMap vm) {
    const VB vb = vb_batch(vm);
    dt_pass2_body(slot_entry(tab, vm.stride, vb.slot), vb);
}

// -------------------------------------------------------------------------
// CTA pass: the stars whose circles do not fit the listed discs (the hull,
// the rims of empty areas)
// -------------------------------------------------------------------------
// One CTA per star.  The points within kDtRadiusC are cached in shared
// memory and the star is wrapped over the cache (warp 0 counter-clockwise,
// warp 1 clockwise).  Triangles whose circle is no wider than the disc are
// certain; for all the others at once the CTA scans the grid cells that their
// circles (and, at an open end, the half-plane beyond the edge) meet and adds
// every point found inside to the cache.  Then the star is wrapped again:
// triangles that no point was found in stay, the gaps are stepped over anew.
// The star is done when a scan finds no point: each of its triangles then has
// an empty circle.  Most stars take one or two scans; a step-by-step search
// would scan once per triangle (up to 50).  A large region is first scanned
// with a stride, which finds points that shrink the circles to a small part
// of it.  A full cache keeps only the star's own vertices and goes on with
// the whole star (its region can only shrink, so that ends).
//
// Bound by the latency of the stars' own chains (a step over the cache is
// about 800 cycles, two warps of the CTA at work; a scan 5,000 to 20,000) and,
// from several thousand stars on, by issue: 640x480 94 -> 38 us with 1,050
// stars, one for each resident CTA, the longest 39 us; 1920x1080 5,500 stars,
// 110 us; 64 x 1242x375 after the middle pass 920 -> 325 us.
constexpr int kDtRadiusC = 48;
constexpr int kDtSamples = 64;     // points of the whole set cached too
constexpr int kDtCacheCap = 1024;   // cached points (16 KB)
constexpr int kDtBlockThreads = 128;
constexpr int kDtBlockWarps = kDtBlockThreads / 32;
constexpr int kDtBlocksPerSM = 8;   // 256 threads and 4 are slower (1920x1080 triangulation 227 against 218 us)
constexpr int kDtVertCap = 256;     // star vertices per direction
constexpr int kDtBadCap = 32;       // circles scanned for at a time (a warp's triangles)
constexpr int kDtMaxRounds = 64;
constexpr int kDtSampleMin = 512;   // regions of more points are sampled first

// Is the circle through the origin, a and b no wider than R (2r <= R)?
// |a|^2 |b|^2 |a-b|^2 <= R^2 cross(a, b)^2, in FP32 with a margin (a false
// answer only has the circle scanned).
__device__ __forceinline__ bool dt_small_circle(const DtPt &a, const DtPt &b, float R2) {
    const float pa = (float)(a.x * a.x + a.y * a.y), pb = (float)(b.x * b.x + b.y * b.y);
    const float dx = (float)(b.x - a.x), dy = (float)(b.y - a.y);
    const float ab = dx * dx + dy * dy, ar = (float)(a.x * b.y - a.y * b.x);
    return pa * pb * ab * 1.00001f <= R2 * ar * ar;
}

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

// The region of a circle, relative to p: a disc (x, y, r padded for the FP32
// rounding of the centre) or, past 1e6 pixels, the half-plane beyond its
// tangent at p, which holds it (unit normal x, y; r < 0).
__device__ __forceinline__ float3 dt_region(const DtCircle &c) {
    const float U = (float)c.U, V = (float)c.V, w = 0.5f * dt_div(1.0f, (float)c.W);
    const float ux = U * w, uy = V * w, r = sqrtf(ux * ux + uy * uy);
    if (r <= 1e6f) return make_float3(ux, uy, r * 1.0001f + 1.0f);
    const float l = rsqrtf(U * U + V * V);
    return make_float3(U * l, V * l, -1.0f);
}

// A star over the cache: per direction the vertices' places in it and the
// state of the triangle that follows each.
enum { kDtOpenCircle = 0, kDtEmpty = 1, kDtHit = 2 };
struct DtStarList {
    uint16_t v[2][kDtVertCap];
    uint8_t state[2][kDtVertCap];
    int n[2];     // triangles in each direction
    int open[2];  // the direction ends at the hull of the cache
};

struct DtStarShared {
    DtStarList star[2];            // the star and the one before it
    DtCircle bad[kDtBadCap];
    float3 region[kDtBadCap + 2];  // of the circles, then of the open ends
    uint16_t tri[kDtBadCap];       // direction << 15 | triangle
    int over;                      // more vertices than the lists hold
    int closed;
    unsigned long long nn;         // |c|^2 and index of the nearest point
    int nearest;                   // its place in the cache
    unsigned quads;
    int far;                       // a cached point lies 2048 pixels or more from p
    int k, nbad, next, found, total, row0, row1;
    int rs[16], rpre[17];
    DtPt win[kDtBlockWarps];
    int won[kDtBlockWarps];
};

// Cells [c0, c1] that a region (about (x0, y0), padded for the FP32 rounding)
// meets in cell row cy.  False: none.
__device__ __forceinline__ bool dt_row_range(int cy, float x0, float y0, const float3 &g, int gw, int &c0, int &c1) {
    const float ya = (float)(cy * kDtCell) - y0, yb = (float)(cy * kDtCell + kDtCell - 1) - y0;
    float xlo = -1e9f, xhi = 1e9f;
    if (g.z >= 0.0f) {
        const float a = ya - g.y, b = yb - g.y;
        const float dy = a > 0.0f ? a : (b < 0.0f ? -b : 0.0f);
        if (dy > g.z) return false;
        const float h2 = g.z * g.z - dy * dy, hc = h2 * rsqrtf(fmaxf(h2, 1e-6f)) * 1.0001f + 1.0f;
        xlo = x0 + g.x - hc;
        xhi = x0 + g.x + hc;
    } else {
        // the boundary at the band's more permissive edge, 4 pixels wider
        const float m = fmaxf(g.y * ya, g.y * yb) + 4.0f;
        if (fabsf(g.x) < 1e-4f) {
            if (m < -4.0f) return false;
        } else if (g.x > 0.0f) {
            xlo = x0 - __fdividef(m, g.x) - 4.0f;
        } else {
            xhi = x0 - __fdividef(m, g.x) + 4.0f;
        }
    }
    c0 = (int)fmaxf(0.0f, fminf((float)(gw - 1), floorf(xlo * (1.0f / kDtCell))));
    c1 = (int)fmaxf(0.0f, fminf((float)(gw - 1), floorf(xhi * (1.0f / kDtCell))));
    return true;
}

// Gathers the points within R of p into the cache (their number, even past
// the capacity, in sh.k), with the nearest one and the quadrants.
__device__ __forceinline__ void dt_block_gather(const DtArgs &a, const DtSide &S, const int4 &p, int R, float4 *cand,
                                                DtStarShared &sh) {
    const int tid = threadIdx.x, lane = tid & 31;
    const int cx0 = min(a.gw - 1, max(0, p.x - R) / kDtCell), cx1 = min(a.gw - 1, max(0, p.x + R) / kDtCell);
    const int cy0 = max(0, p.y - R) / kDtCell, cy1 = min(a.gh - 1, max(0, p.y + R) / kDtCell);
    const int nrows = cy1 - cy0 + 1;
    __syncthreads();
    if (tid < 32) {
        int r0 = 0, len = 0;
        if (lane < nrows) {
            const int *row = S.cell_start + (cy0 + lane) * a.gw;
            r0 = row[cx0];
            len = row[cx1 + 1] - r0;
        }
        int incl = len;
#pragma unroll
        for (int o = 1; o < 16; o <<= 1) {
            const int y = __shfl_up_sync(0xFFFFFFFFu, incl, o);
            if (lane >= o) incl += y;
        }
        if (lane < 16) {
            sh.rs[lane] = r0 - (incl - len);
            sh.rpre[lane] = incl - len;
            if (lane == 15) sh.rpre[16] = incl;
        }
        if (lane == 0) {
            sh.k = 0;
            sh.nn = ~0ull;
            sh.quads = 0;
        }
    }
    __syncthreads();
    const int total = sh.rpre[16];
    unsigned long long nn = ~0ull;
    unsigned quads = 0;
    int at = 0;
    for (int t0 = 0; t0 < total; t0 += 4 * kDtBlockThreads) {  // four loads in flight
        int4 q[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const int t = t0 + u * kDtBlockThreads + tid;
            int r = 0;
#pragma unroll
            for (int s = 8; s > 0; s >>= 1)
                if (t >= sh.rpre[r + s]) r += s;
            q[u] = t < total ? S.pts[sh.rs[r] + t] : make_int4(0, 0, 0, 0);
        }
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            if (t0 + u * kDtBlockThreads >= total) break;
            const int dx = q[u].x - p.x, dy = q[u].y - p.y, d2 = dx * dx + dy * dy;
            const bool take = q[u].w && q[u].z != p.z && abs(dx) <= R && abs(dy) <= R && d2 <= R * R;
            const unsigned m = __ballot_sync(0xFFFFFFFFu, take);
            int base = 0;
            if (lane == 0 && m) base = atomicAdd(&sh.k, __popc(m));
            const int pos = __shfl_sync(0xFFFFFFFFu, base, 0) + __popc(m & ((1u << lane) - 1u));
            if (take) {
                if (pos < kDtCacheCap) cand[pos] = dt_cand(dx, dy, q[u].z);
                const unsigned long long key = ((unsigned long long)d2 << 32) | (unsigned)q[u].z;
                if (key < nn) {
                    nn = key;
                    at = pos;
                }
                quads |= dt_quadrant(dx, dy);
            }
        }
    }
    if (nn != ~0ull) {
        atomicMin(&sh.nn, nn);
        atomicOr(&sh.quads, quads);
    }
    __syncthreads();
    if (nn != ~0ull && nn == sh.nn) sh.nearest = at;
    __syncthreads();
}
static_assert(2 * kDtRadiusC / kDtCell + 2 <= 16, "cell rows of the cached disc");

// Wraps the star over the cache into sh.star[cur] (warp 0 counter-clockwise,
// warp 1 clockwise from the first vertex).  again: sh.star[cur ^ 1] is the
// star before the last points were added, its hit triangles marked: the
// others stay triangles of the star, so only the gaps are stepped over.
__device__ __forceinline__ void dt_block_wrap(const float4 *cand, int k, int pz, bool fan, bool again, int cur,
                                              DtStarShared &sh) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const DtStarList &old = sh.star[cur ^ 1];
    DtStarList &star = sh.star[cur];
    __syncthreads();
    if (warp < 2) {
        const DtListSrc src(cand, k, !sh.far, lane);
        // a fan's first vertex is certain while a triangle beside it is
        if (again && fan && old.state[0][0] == kDtHit && old.state[1][0] == kDtHit) again = false;
        const int side = warp ? -1 : 1, nold = again ? old.n[warp] : 0;
        int first = again ? old.v[warp][0] : sh.nearest, n = 0;
        float4 e;
        bool ok = again || !fan || dt_fan_start(src, lane, e, first);
        bool open = false;
        const bool skip = warp == 1 && again && sh.closed;  // the other direction has the whole star
        e = cand[first];
        const int z0 = __float_as_int(e.w);
        if (lane == 0) star.v[warp][0] = first;
        int i = 0;        // the last vertex of the old star met
        bool on = again;  // e is that vertex
        while (ok && !skip) {
            int at;
            uint8_t state = kDtOpenCircle;
            float4 w;
            if (on && i < nold && old.state[warp][i] != kDtHit) {  // this triangle stays
                state = old.state[warp][i];
                at = old.v[warp][++i];
                w = cand[at];
            } else {
                float t;
                if (!dt_step(src, lane, e, pz, side, w, t, at)) {
                    open = true;
                    break;
                }
                on = false;
                for (int j0 = i; j0 <= nold && !on && nold > 0; j0 += 32) {
                    const unsigned b = __ballot_sync(0xFFFFFFFFu, j0 + lane <= nold && old.v[warp][j0 + lane] == at);
                    if (b) {
                        i = j0 + __ffs(b) - 1;
                        on = true;
                    }
                }
            }
            if (n == kDtVertCap - 1) {
                ok = false;
                break;
            }
            if (lane == 0) {
                star.v[warp][n + 1] = at;
                star.state[warp][n] = state;
            }
            ++n;
            if (fan) {
                if (!(w.y > 0.0f)) break;
            } else if (__float_as_int(w.w) == z0) {
                if (lane == 0) sh.closed = 1;
                break;
            }
            e = w;
        }
        if (lane == 0) {
            star.n[warp] = skip ? 0 : n;
            star.open[warp] = open;
            if (!ok || (fan && open)) sh.over = 1;
        }
    }
    __syncthreads();
    // a closed star is the counter-clockwise run alone
    if (threadIdx.x == 0 && sh.closed) star.n[1] = star.open[1] = 0;
    __syncthreads();
}

// Triangle t of a star (counter-clockwise run first), as (a, b).
__device__ __forceinline__ void dt_star_tri(const DtStarList &star, const float4 *cand, int t, float4 &a, float4 &b) {
    const int na = star.n[0];
    const uint16_t *v = t < na ? star.v[0] + t : star.v[1] + (t - na);
    a = cand[v[t < na ? 0 : 1]];
    b = cand[v[t < na ? 1 : 0]];
}

// Room in the pool for the m > kDtSlots owned triangles of point pz (one
// thread): their first entry, which the point's slots then name, or -1 when
// there is none and the triangulation fails.  Stars that agree own fewer than
// two triangles a point in all, which the pool holds.
__device__ __noinline__ int dt_pool_room(const DtSide &S, int pz, int m) {
    const int base = atomicAdd(S.npool, m);
    if (base < 0 || m > S.pool_cap - base) {
        atomicOr(S.err, kDtErrPool);
        return -1;
    }
    S.slots[(size_t)pz * kDtSlots] = make_int2(base, 0);
    return base;
}

// Writes the owned triangles of a star (warp 0).
__device__ __forceinline__ void dt_block_write(const DtSide &S, int pz, bool fan, const float4 *cand,
                                               const DtStarList &star, int nearest) {
    const int lane = threadIdx.x & 31;
    const int na = star.n[0], nt = na + star.n[1];
    auto owned = [&](int t, float4 &u, float4 &v) {
        if (t >= nt) return false;
        dt_star_tri(star, cand, t, u, v);
        return pz < __float_as_int(u.w) && pz < __float_as_int(v.w);
    };
    int ma = 0, mb = 0, r = -1;
    for (int t0 = 0; t0 < nt; t0 += 32) {
        float4 u, v;
        const bool own = owned(t0 + lane, u, v);
        ma += __popc(__ballot_sync(0xFFFFFFFFu, own && t0 + lane < na));
        mb += __popc(__ballot_sync(0xFFFFFFFFu, own && t0 + lane >= na));
    }
    const int m = ma + mb;
    if (fan) {
        for (int i = lane; i <= ma; i += 32)
            if (star.v[0][i] == nearest) r = mb + i;
        for (int i = lane; i <= mb; i += 32)
            if (star.v[1][i] == nearest) r = mb - i;
        r = max(0, __reduce_max_sync(0xFFFFFFFFu, r));
    }
    int2 *out = S.slots + (size_t)pz * kDtSlots;
    if (m > kDtSlots) {
        int base = 0;
        if (lane == 0) base = dt_pool_room(S, pz, m);
        base = __shfl_sync(0xFFFFFFFFu, base, 0);
        if (base < 0) return;
        out = S.pool + base;
    }
    int done = 0;
    for (int t0 = 0; t0 < nt; t0 += 32) {
        const int t = t0 + lane;
        float4 u, v;
        const bool own = owned(t, u, v);
        const unsigned b = __ballot_sync(0xFFFFFFFFu, own);
        int pos = done + __popc(b & ((1u << lane) - 1u));
        if (fan) pos = dt_fan_pos(t < na ? mb + t : mb - 1 - (t - na), m, r);
        if (own) out[pos] = make_int2(__float_as_int(u.w), __float_as_int(v.w));
        done += __popc(b);
    }
    if (lane == 0) S.owned[pz] = m;
}

// The whole star of p over every point, one exact step after the other (more
// vertices than the lists hold, e.g. the apex of a huge fan): counted first,
// then written.
__device__ __noinline__ void dt_block_star_all(const DtSide &S, const int4 &p, int n, const DtPt &nn, DtStarShared &sh) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    int2 *out = nullptr;
    int m = 0;
    for (int pass = 0; pass < 2; ++pass) {
        int written = 0;
        bool closed = false;
        for (int side = 1; side >= -1 && !closed; side -= 2) {
            DtPt cur = nn;
            for (int step = 0; step <= n; ++step) {
                DtPt w{0, 0, 0};
                int at;
                const bool any = dt_step_int(
                    [&](int c) {  // this warp's quarter of the points
                        const int4 q = S.pts[kDtBlockWarps * c + warp];
                        // D = 0: never a candidate
                        return q.w && q.z != p.z ? DtPt{q.x - p.x, q.y - p.y, q.z} : DtPt{0, 0, p.z};
                    },
                    (n - warp + kDtBlockWarps - 1) / kDtBlockWarps, lane, cur, p.z, side, w, at);
                __syncthreads();
                if (lane == 0) {
                    sh.win[warp] = w;
                    sh.won[warp] = any;
                }
                __syncthreads();
                bool got = false;
                for (int i = 0; i < kDtBlockWarps; ++i)
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
                if (threadIdx.x == 0) sh.total = dt_pool_room(S, p.z, m);
                __syncthreads();
                if (sh.total < 0) return;
                out = S.pool + sh.total;
            }
        }
    }
    if (threadIdx.x == 0) S.owned[p.z] = m;
    __syncthreads();
}

__device__ __forceinline__ void dt_block_item(const DtArgs &a, const DtSide &S, int at, int n, bool ordered,
                                              float4 *cand, int *r_start, int *r_len, DtStarShared &sh) {
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int4 p = S.pts[at];
    int R = 2 * kDtRadiusC;
    do {
        R >>= 1;
        dt_block_gather(a, S, p, R, cand, sh);
    } while (sh.k > kDtCacheCap - kDtSamples && R > 1);
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
        if (tid == 0) {
            const int4 q = S.pts[S.slot[(int)(unsigned)(sh.nn & 0xFFFFFFFFu)]];
            cand[0] = dt_cand(q.x - p.x, q.y - p.y, q.z);
            sh.nearest = 0;
        }
        k = 1;
        __syncthreads();
    }
    const bool ring = ordered && sh.quads == 15u;  // a fan already (dt_warp_star)
    if (tid == 0) {
        sh.far = max(fabsf(cand[sh.nearest].x), fabsf(cand[sh.nearest].y)) >= (float)kDtNearMax;
        sh.k = k;
    }
    __syncthreads();
    // points spread over the whole set, so that the first circles are not
    // far wider than the star's (a point with neighbours all around has none
    // that wide, and would only step over the samples too: 1920x1080 pass
    // 124 -> 112 us with this and the circles' regions below)
    if (tid < kDtSamples && !ring) {
        const int4 q = S.pts[(int)((int64_t)tid * n / kDtSamples)];
        const int dx = q.x - p.x, dy = q.y - p.y, nz = __float_as_int(cand[sh.nearest].w);
        if (q.w && q.z != p.z && q.z != nz && (max(abs(dx), abs(dy)) > R || dx * dx + dy * dy > R * R)) {
            cand[atomicAdd(&sh.k, 1)] = dt_cand(dx, dy, q.z);
            if (max(abs(dx), abs(dy)) >= kDtNearMax) sh.far = 1;
            atomicOr(&sh.quads, dt_quadrant(dx, dy));
        }
    }
    __syncthreads();
    k = sh.k;
    bool fan = ordered && sh.quads == 15u;
    bool again = false, compact = false;
    int cur = 0;
    for (int round = 0;; ++round) {
        if (tid == 0) {
            sh.over = 0;
            if (!again) sh.closed = 0;
        }
        dt_block_wrap(cand, k, p.z, fan, again, cur, sh);
        DtStarList &star = sh.star[cur];
        if (sh.over || round == kDtMaxRounds) {
            dt_block_star_all(S, p, n, dt_point(cand[sh.nearest]), sh);
            return;
        }
        if (compact) {
            // full cache: keep only the whole star's vertices (no disc
            // certifies its circles any more)
            const int na = star.n[0] + (sh.closed ? 0 : 1), nv = na + star.n[1];
            float4 keep[2 * kDtVertCap / kDtBlockThreads];
#pragma unroll
            for (int u = 0; u < 2 * kDtVertCap / kDtBlockThreads; ++u) {
                const int j = u * kDtBlockThreads + tid;
                if (j < nv) keep[u] = cand[j < na ? star.v[0][j] : star.v[1][j - na + 1]];
            }
            __syncthreads();
#pragma unroll
            for (int u = 0; u < 2 * kDtVertCap / kDtBlockThreads; ++u) {
                const int j = u * kDtBlockThreads + tid;
                if (j < nv) cand[j] = keep[u];
            }
            k = nv;
            if (tid == 0) sh.nearest = 0;  // the first vertex
            compact = false;
            __syncthreads();
            continue;
        }
        const int nt = star.n[0] + star.n[1];
        const bool open_l = star.open[0], open_r = star.open[1];
        const float R2 = (float)(R * R);
        bool first = true;  // the open ends go with the first group of circles
        int found = 0;
        for (int t0 = 0; t0 < nt || first;) {
            // the next circles that neither the disc nor a scan certifies
            __syncthreads();
            if (warp == 0) {
                int nb = 0;
                for (; t0 < nt && nb == 0; t0 += 32) {
                    const int t = t0 + lane, dir = t < star.n[0] ? 0 : 1, i = dir ? t - star.n[0] : t;
                    bool bad = false;
                    DtPt u{0, 0, 0}, v{0, 0, 0};
                    if (t < nt && star.state[dir][i] != kDtEmpty) {
                        float4 uf, vf;
                        dt_star_tri(star, cand, t, uf, vf);
                        u = dt_point(uf);
                        v = dt_point(vf);
                        bad = !dt_small_circle(u, v, R2);
                    }
                    const unsigned b = __ballot_sync(0xFFFFFFFFu, bad);
                    if (bad) {
                        const int to = __popc(b & ((1u << lane) - 1u));
                        sh.bad[to] = dt_circle(u, v);
                        sh.region[to] = dt_region(sh.bad[to]);
                        sh.tri[to] = (uint16_t)(dir << 15 | i);
                    }
                    nb = __popc(b);
                }
                if (lane < 2 && first && (lane ? open_r : open_l)) {  // beyond the open edge
                    const float4 e = cand[star.v[lane][star.n[lane]]];
                    const float ex = lane ? -e.x : e.x, ey = lane ? -e.y : e.y, l = rsqrtf(ex * ex + ey * ey);
                    sh.region[kDtBadCap + lane] = make_float3(-ey * l, ex * l, -1.0f);
                }
                if (lane == 0) {
                    sh.nbad = nb;
                    sh.next = t0;
                    sh.total = 0;
                    sh.found = 0;
                    sh.row0 = a.gh;
                    sh.row1 = -1;
                }
            } else {
                for (int cy = tid - 32; cy < a.gh; cy += kDtBlockThreads - 32) {
                    r_start[cy] = a.gw;
                    r_len[cy] = -1;
                }
            }
            const bool ends = first && (open_l || open_r);
            __syncthreads();
            const int nbad = sh.nbad;
            t0 = sh.next;
            first = false;
            if (nbad == 0 && !ends) continue;
            const DtPt el = dt_point(cand[star.v[0][star.n[0]]]), er = dt_point(cand[star.v[1][star.n[1]]]);
            // cell ranges: each warp takes regions, its lanes their cell rows
            for (int b = warp; b < kDtBadCap + 2; b += kDtBlockWarps) {
                if (b < kDtBadCap ? b >= nbad : !(ends && (b == kDtBadCap ? open_l : open_r))) continue;
                const float3 g = sh.region[b];
                int y0 = 0, y1 = a.gh - 1;
                if (g.z >= 0.0f) {
                    y0 = (int)fmaxf(0.0f, ((float)p.y + g.y - g.z - 2.0f) * (1.0f / kDtCell));
                    y1 = (int)fminf((float)y1, ((float)p.y + g.y + g.z + 2.0f) * (1.0f / kDtCell));
                }
                for (int cy = y0 + lane; cy <= y1; cy += 32) {
                    int c0, c1;
                    if (dt_row_range(cy, (float)p.x, (float)p.y, g, a.gw, c0, c1)) {
                        atomicMin(&r_start[cy], c0);
                        atomicMax(&r_len[cy], c1);
                    }
                }
            }
            __syncthreads();
            int tot = 0, row0 = a.gh, row1 = -1;
            for (int cy = tid; cy < a.gh; cy += kDtBlockThreads) {
                const int lo = r_start[cy], hi = r_len[cy];
                const int *row = S.cell_start + cy * a.gw;
                const int s0 = lo <= hi ? row[lo] : 0, len = lo <= hi ? row[hi + 1] - s0 : 0;
                r_start[cy] = s0;
                r_len[cy] = len;
                tot += len;
                if (len) {
                    row0 = min(row0, cy);
                    row1 = cy;
                }
            }
            tot = __reduce_add_sync(0xFFFFFFFFu, tot);
            row0 = __reduce_min_sync(0xFFFFFFFFu, row0);
            row1 = __reduce_max_sync(0xFFFFFFFFu, row1);
            if (lane == 0 && tot) {
                atomicAdd(&sh.total, tot);
                atomicMin(&sh.row0, row0);
                atomicMax(&sh.row1, row1);
            }
            __syncthreads();
            row0 = sh.row0;
            row1 = sh.row1;
            int stride = sh.total > kDtSampleMin && round < 4 ? sh.total / (kDtSampleMin / 2) : 1;
            for (;;) {
                // 32 rows at a time as one index space, which the warps share
                // out evenly (a hull point's region is often one long row)
                for (int cy0 = row0; cy0 <= row1; cy0 += 32) {
                    const int cy = cy0 + lane;
                    const int len = cy <= row1 ? r_len[cy] : 0;
                    int incl = len;
#pragma unroll
                    for (int o = 1; o < 32; o <<= 1) {
                        const int y = __shfl_up_sync(0xFFFFFFFFu, incl, o);
                        if (lane >= o) incl += y;
                    }
                    const int all = __shfl_sync(0xFFFFFFFFu, incl, 31), excl = incl - len;
                    const int off = (cy <= row1 ? r_start[cy] : 0) - excl;
                    auto load = [&](int j) {
                        int r = 0;
#pragma unroll
                        for (int h = 16; h > 0; h >>= 1)
                            if (j >= __shfl_sync(0xFFFFFFFFu, excl, r + h)) r += h;
                        const int src = __shfl_sync(0xFFFFFFFFu, off, r) + j;
                        return j < all ? S.pts[src] : make_int4(0, 0, 0, 0);
                    };
                    int4 next = load(tid * stride);
                    for (int j0 = 32 * warp * stride; j0 < all; j0 += kDtBlockThreads * stride) {
                        const int4 t = next;
                        if (j0 + kDtBlockThreads * stride < all) next = load(j0 + (kDtBlockThreads + lane) * stride);
                        const DtPt q{t.x - p.x, t.y - p.y, t.z};
                        const float qx = (float)q.x, qy = (float)q.y;
                        // the circles that need the exact test: all whose
                        // padded region holds the point
                        unsigned need = 0;
                        for (int b = 0; b < nbad; ++b) {
                            const float3 g = sh.region[b];
                            const float dx = qx - g.x, dy = qy - g.y;
                            const bool in = g.z >= 0.0f ? dx * dx + dy * dy <= g.z * g.z
                                                        : g.x * qx + g.y * qy >= -1.0f;
                            need |= (unsigned)in << b;
                        }
                        const bool some = t.w && t.z != p.z;
                        bool hit = false;
                        if (ends && some)
                            hit = (open_l && el.x * q.y - el.y * q.x > 0) || (open_r && er.x * q.y - er.y * q.x < 0);
                        if (!some) need = 0;
                        for (; need; need &= need - 1) {
                            const int b = __ffs(need) - 1;
                            if (!dt_violates(sh.bad[b], p.z, q)) continue;
                            hit = true;
                            star.state[sh.tri[b] >> 15][sh.tri[b] & 0x7FFF] = kDtHit;
                        }
                        const unsigned m = __ballot_sync(0xFFFFFFFFu, hit);
                        if (!m) continue;
                        int base = 0;
                        if (lane == 0) base = atomicAdd(&sh.found, __popc(m));
                        const int pos = k + __shfl_sync(0xFFFFFFFFu, base, 0) + __popc(m & ((1u << lane) - 1u));
                        if (hit && pos < kDtCacheCap) cand[pos] = dt_cand(q.x, q.y, q.z);
                        if (hit && max(abs(q.x), abs(q.y)) >= kDtNearMax) sh.far = 1;
                    }
                }
                __syncthreads();
                found = sh.found;
                if (stride == 1 && tid < nbad) {
                    uint8_t &st = star.state[sh.tri[tid] >> 15][sh.tri[tid] & 0x7FFF];
                    if (st != kDtHit) st = kDtEmpty;
                }
                __syncthreads();
                if (stride == 1 || found > 0) break;
                stride = 1;
            }
            if (found) break;  // wrap again before the other circles
        }
        if (found == 0) break;
        if (k + found <= kDtCacheCap) {
            k += found;
            again = true;
            cur ^= 1;
        } else {
            k = kDtCacheCap;
            fan = again = false;
            compact = true;
            R = 0;
        }
    }
    if (warp == 0) dt_block_write(S, p.z, fan, cand, sh.star[cur], sh.nearest);
    __syncthreads();
}

// One pair, persistent (every CTA resident): the CTAs take the stars of
// both sides' queues from one atomic counter, the two queues interleaved so
// that both sides' stars start in the first wave (the pass lasts as long as
// its longest star, so none should wait behind the other side's).  The
// counter is side 0's nwork, which dt_init_kernel zeroes and the one-pair
// passes leave unused.
__global__ void __launch_bounds__(kDtBlockThreads, kDtBlocksPerSM) dt_pass_block_kernel(const __grid_constant__ DtArgs a,
                                                                                             int nsides) {
    after_previous();
    extern __shared__ float4 s_cand[];  // [kDtCacheCap], then the region rows
    __shared__ DtStarShared sh;
    __shared__ int s_item;
    int *r_start = reinterpret_cast<int *>(s_cand + kDtCacheCap);
    const int n = min(max(*a.count, 0), a.cap);
    const int nq0 = *a.s[0].npending, nq1 = nsides > 1 ? *a.s[1].npending : 0;
    const int m = min(nq0, nq1), total = nq0 + nq1;
    int32_t *counter = a.s[0].nwork;
    int next = threadIdx.x == 0 ? atomicAdd(counter, 1) : 0;  // fetched while the item before is worked on
    for (;;) {
        if (threadIdx.x == 0) s_item = next;
        __syncthreads();
        const int item = s_item;
        __syncthreads();
        if (item >= total) break;
        if (threadIdx.x == 0) next = atomicAdd(counter, 1);
        const bool two = item < 2 * m;
        const int side = two ? (item & 1) : (nq0 > nq1 ? 0 : 1);
        const int idx = two ? (item >> 1) : item - m;
        const DtSide &S = a.s[side];
        dt_block_item(a, S, S.pending[idx], n, !(*S.err & kDtErrOrder), s_cand, r_start, r_start + a.gh, sh);
    }
}

// Many pairs, persistent: the queues of every (pair, side) of the launch are
// concatenated in launch order and the CTAs take their entries one at a
// time from one atomic counter (zeroed by dt_init_kernel_b), so the long
// stars of one pair overlap the work of all the others.  second: the middle
// pass's queues, else the warp pass's (a batch of one pair, which skips the
// middle pass).
__global__ void __launch_bounds__(kDtBlockThreads, kDtBlocksPerSM)
    dt_pass_block_kernel_b(const DtArgs *__restrict__ tab, VMap vm, int nsides, int32_t *counter, int second) {
    extern __shared__ float4 s_cand[];
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
    int next = tid == 0 ? atomicAdd(counter, 1) : 0;  // fetched while the item before is worked on
    for (;;) {
        if (tid == 0) s_item = next;
        __syncthreads();
        const int item = s_item;
        __syncthreads();
        if (item >= total) break;
        if (tid == 0) next = atomicAdd(counter, 1);
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
        const int at = (second ? S.pending2 : S.pending)[item - s_pre[lo]];
        dt_block_item(a, S, at, n, !(*S.err & kDtErrOrder), s_cand, r_start, r_start + a.gh, sh);
    }
}

// One CTA per side: exclusive scan of the owned counts, total = ntri.
__device__ __forceinline__ void dt_tri_scan_body(const DtArgs &a, const VB &vb) {
    const DtSide &S = a.s[vb.y];
    const int total = dt_block_scan(S.owned, min(max(*a.count, 0), a.cap), [&](int i, const int4 &before) {
        *reinterpret_cast<int4 *>(S.offset + i) = before;
    });
    const bool failed = total > a.cap_tri || *S.err & (kDtErrPool | kDtErrRange);
    if (threadIdx.x == 0) *S.ntri = failed ? -1 : total;
}

__global__ void __launch_bounds__(1024) dt_tri_scan_kernel(DtArgs a) {
    after_previous();
    dt_tri_scan_body(a, vb_single());
}
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

__global__ void dt_emit_kernel(DtArgs a) {
    after_previous();
    dt_emit_body(a, vb_single());
}
__global__ void dt_emit_kernel_b(const DtArgs *__restrict__ tab, VMap vm) {
    const VB vb = vb_batch(vm);
    dt_emit_body(slot_entry(tab, vm.stride, vb.slot), vb);
}

// -------------------------------------------------------------------------
// Host side
// -------------------------------------------------------------------------

constexpr int kDtCounters = 5;  // err, npending, npending2, nwork, npool

// Dynamic shared memory of the CTA pass for images of up to gh cell rows.
static constexpr int dt_block_smem(int gh) { return kDtCacheCap * (int)sizeof(float4) + 2 * gh * (int)sizeof(int); }
static_assert(dt_block_smem(16384 / kDtCell) + sizeof(DtStarShared) + (2 * kMaxBatch + 2) * sizeof(int) <= kSmemNoLeave,
              "the CTA pass needs no leave for its shared memory at any size");

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

static int dt_pool_cap(int cap) { return 2 * (cap > 0 ? cap : 1); }  // a mesh has fewer than 2n triangles

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
    s.pool = reinterpret_cast<int2 *>(take((size_t)dt_pool_cap(cap) * 8));
    s.pool_cap = dt_pool_cap(cap);
    s.pending = reinterpret_cast<int32_t *>(take(c * 4));
    s.pending2 = reinterpret_cast<int32_t *>(take(c * 4));
    s.rowmin = reinterpret_cast<int32_t *>(take((size_t)h * 4));
    s.rowmax = reinterpret_cast<int32_t *>(take((size_t)h * 4));
    int32_t *counters = reinterpret_cast<int32_t *>(take(kDtCounters * 4));
    s.err = counters;
    s.npending = counters + 1;
    s.npending2 = counters + 2;
    s.nwork = counters + 3;
    s.npool = counters + 4;
    return s;
}

__global__ void __launch_bounds__(256) dt_init_kernel(DtArgs a);

// Triangulates one or both sides.  sides[i] = right flag; tri/ntri per side.
elas_status launch_triangulate_device(const int16_t *list, const int32_t *count, int cap, int w, int h, int nsides,
                                      const int *rights, int32_t *const *tri, int32_t *const *ntri, int cap_tri,
                                      void *ws, cudaStream_t st, int pool_cap) {
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
        if (pool_cap >= 0) a.s[i].pool_cap = min(pool_cap, a.s[i].pool_cap);
    }
    // counters, cell counts and row extremes of both sides: one kernel
    const int nall = a.gw * a.gh + 1 + 2 * h + kDtCounters;
    launch_after(dt_init_kernel, dim3((nall + 255) / 256, nsides), 256, 0, st, a);
    const int tb = 256;
    const int pblocks = max(1, min((cap + tb - 1) / tb, sm_count() * 8));
    launch_after(dt_points_kernel, dim3(pblocks, nsides), tb, 0, st, a);
    launch_after(dt_cell_scan_kernel, dim3(1, nsides), 1024, 0, st, a);
    launch_after(dt_scatter_kernel, dim3(pblocks, nsides), tb, 0, st, a);
    launch_after(dt_dedup_kernel, dim3(pblocks, nsides), tb, 0, st, a);
    launch_after(dt_pass1_kernel, dim3(max(1, min((cap + kDtWarps - 1) / kDtWarps, sm_count() * 16)), nsides), kDtWarps * 32, 0, st, a);

    // no middle pass: it would add its longest star's time to the CTA pass's
    // (640x480 38 us alone, 37 + 37 with it; 1920x1080 126 and 52 + 74)
    const int smem = dt_block_smem(a.gh);
    launch_after(dt_pass_block_kernel, sm_count() * kDtBlocksPerSM, kDtBlockThreads, smem, st, a, nsides);
    launch_after(dt_tri_scan_kernel, dim3(1, nsides), 1024, 0, st, a);
    launch_after(dt_emit_kernel, dim3(pblocks, nsides), tb, 0, st, a);
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

__global__ void __launch_bounds__(256) dt_init_kernel(DtArgs a) {
    after_previous();
    dt_init_body(a, vb_single(), nullptr);
}
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
    // the star passes' warps take their points in turn: with a CTA for every
    // eight points of the capacity, finding its pair and loading the argument
    // block cost a warp 140 instructions for little more than one star (a
    // third of the pass)
    long long caps = 0;
    for (int i = 0; i < pairs.n; ++i) caps += slot_entry(host, pairs.stride, pairs.slot[i]).cap;
    for (int i = 0; i < pairs.n; ++i) {
        const int slot = pairs.slot[i];
        const DtArgs &a = slot_entry(host, pairs.stride, slot);
        const int nall = a.gw * a.gh + 1 + 2 * a.h + kDtCounters;
        vmap_add(m_init, slot, dim3((nall + 255) / 256, nsides));
        vmap_add(m_pts, slot, dim3(dt_point_blocks(a.cap, 256, pairs.n), nsides));
        vmap_add(m_scan, slot, dim3(1, nsides));
        vmap_add(m_grp, slot, dim3(vmap_share(a.cap, caps, sm_count() * 4 * 8 / nsides), nsides));
        vmap_add(m_grp2, slot, dim3(vmap_share(a.cap, caps, sm_count() * 7 * 4 / nsides), nsides));
        max_gh = max(max_gh, a.gh);
    }
    const int smem = dt_block_smem(max_gh);
    dt_init_kernel_b<<<vmap_total(m_init), 256, 0, st>>>(tab, m_init, counter);
    dt_points_kernel_b<<<vmap_total(m_pts), 256, 0, st>>>(tab, m_pts);
    dt_cell_scan_kernel_b<<<vmap_total(m_scan), 1024, 0, st>>>(tab, m_scan);
    dt_scatter_kernel_b<<<vmap_total(m_pts), 256, 0, st>>>(tab, m_pts);
    dt_dedup_kernel_b<<<vmap_total(m_pts), 256, 0, st>>>(tab, m_pts);
    dt_pass1_kernel_b<<<vmap_total(m_grp), kDtWarps * 32, 0, st>>>(tab, m_grp);
    const int middle = pairs.n > 1;
    if (middle) dt_pass2_kernel_b<<<vmap_total(m_grp2), kDtWarpsM * 32, 0, st>>>(tab, m_grp2);
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

namespace elas {
// The C entry; pool_cap >= 0: room for only so many triangles of large fans.
static elas_status triangulate_entry(const int16_t *list, const int32_t *count, int32_t cap, int32_t w, int32_t h,
                                     int32_t right, int32_t *tri, int32_t cap_tri, int32_t *ntri, void *workspace,
                                     size_t workspace_bytes, int32_t pool_cap, elas_stream stream) {
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
                                     to_stream(stream), pool_cap);
}
}  // namespace elas

extern "C" elas_status elas_triangulate_device(const int16_t *list, const int32_t *count, int32_t cap, int32_t w,
                                               int32_t h, int32_t right, int32_t *tri, int32_t cap_tri,
                                               int32_t *ntri, void *workspace, size_t workspace_bytes,
                                               elas_stream stream) {
    return elas::triangulate_entry(list, count, cap, w, h, right, tri, cap_tri, ntri, workspace, workspace_bytes, -1,
                                   stream);
}

extern "C" elas_status elas_probe_triangulate_pool(const int16_t *list, const int32_t *count, int32_t cap, int32_t w,
                                                   int32_t h, int32_t right, int32_t *tri, int32_t cap_tri,
                                                   int32_t *ntri, void *workspace, size_t workspace_bytes,
                                                   int32_t pool, elas_stream stream) {
    if (pool < 0) return elas::fail(ELAS_ERR_INVALID_ARG, "pool of %d triangles", pool);
    return elas::triangulate_entry(list, count, cap, w, h, right, tri, cap_tri, ntri, workspace, workspace_bytes, pool,
                                   stream);
}

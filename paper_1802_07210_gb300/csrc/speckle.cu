// Small-segment (speckle) removal, ELAS post-processing: two 4-neighbouring
// valid pixels are linked iff their disparities differ by at most
// sim_threshold; segments (connected components of the links) with fewer
// than min_size pixels are invalidated.
//
// Connected components by union-find over pixel indices, every parent index
// below its child's, so a root is the least pixel index of its tree:
//   speckle_local_kernel   one CTA per 64x32 or 64x16 tile: union-find of the links
//                          inside the tile in shared memory.  A tile-local
//                          root's label is its own global index and its size
//                          entry its pixel count in the tile; another pixel's
//                          label names its tile-local root (as -2 - index,
//                          -1: invalid), and its size entry is not used.
//   speckle_border_kernel  one thread per link across a tile's right or
//                          bottom edge: union in global memory (atomicMin on
//                          roots).
//   speckle_resolve_kernel each tile-local root finds its final root, points
//                          its label there and adds its count to the root's
//                          (one atomic per tile-local segment).
//   speckle_apply_kernel   two hops (pixel -> tile-local root -> final root)
//                          give the segment size: out = d if large enough,
//                          else -1.
// The partition is unique, so the output is too.  Every loop is bounded by
// the pixel count (each step moves to a strictly smaller index); a loop that
// reaches its bound sets the status word instead of spinning on.
#include "launch.cuh"

namespace elas {

// Tiles of 64 x TY pixels, 16 warps each.  Taller tiles have fewer links
// across edges and fewer tile-local roots that those link, shorter ones more
// CTAs, each with less to walk: 32 rows from a tile for every SM on, else 16
// (local and border pass: 1920x1080 27.0 us with 32 rows, 29.2 with 16;
// 320x240 11.8 and 10.9; with 32x16 tiles 39 and 10.9).
constexpr int kSpTX = 64, kSpWarps = 16, kSpMaxCells = kSpTX * 32;

struct SpeckleArgs {
    const int16_t *d;
    int16_t *out;
    int32_t *label;   // [h][w]: tile-local roots: parent; else -2 - the tile-local root, -1 for invalid pixels
    int32_t *size;    // [h][w]: tile-local roots: pixel count
    int32_t *status;  // 0, or 1 if a loop bound was reached
    int w, h, thr, min_size;
};

__device__ __forceinline__ bool sp_linked(int a, int b, int thr) { return a >= 0 && b >= 0 && abs(a - b) <= thr; }

__device__ __forceinline__ int sp_tile_root(const int32_t *L, int i) {
    const int v = __ldcg(L + i);
    return v < -1 ? -2 - v : i;
}

// Root of x in a forest whose parents are strictly smaller indices; reads
// through L2 (`ld.cg`) because other CTAs relink roots during the kernel.
// Path halving: a visited non-root is pointed at its grandparent (an
// ancestor, so the forest stays valid; roots are only changed by unions).
__device__ __forceinline__ int sp_find_global(int32_t *L, int x, int limit) {
    for (int it = 0; it < limit; ++it) {
        const int p = __ldcg(L + x);
        if (p == x) return x;
        const int g = __ldcg(L + p);
        if (g != p) __stcg(L + x, g);
        x = g;
    }
    return -1;
}

// Joins the trees of a and b: the larger root is linked under the smaller
// one with atomicMin; if that root was relinked meanwhile, the returned old
// parent (a smaller index) is where the walk resumes.  The larger tile-local
// root is linked so at once, before any walk: mostly it is a root still, and a
// walk up a chain that other links are just growing costs an L2 round trip a
// step (a segment winding through a map of 100x3000: 196 us with walks first,
// 34 now; 1920x1080 of diagonals 52.8 and 41.3, a scene's map 44.1 and 42.6).
__device__ void sp_unite_global(int32_t *L, int a, int b, int limit, int32_t *status) {
    a = sp_tile_root(L, a);
    b = sp_tile_root(L, b);
    if (a == b) return;
    if (a > b) {
        const int t = a;
        a = b;
        b = t;
    }
    const int was = atomicMin(L + b, a);
    if (was == b) return;
    b = was;
    for (int it = 0; it < limit; ++it) {
        a = sp_find_global(L, a, limit);
        b = sp_find_global(L, b, limit);
        if (a < 0 || b < 0) break;
        if (a == b) return;
        if (a > b) {
            const int t = a;
            a = b;
            b = t;
        }
        const int old = atomicMin(L + b, a);
        if (old == b) return;
        b = old;
    }
    atomicExch(status, 1);
}

// The same walk without writes: after the unions, each tile-local root's
// label is set to its final root by that root's own thread alone, which a
// halving write from another walk could overwrite with an intermediate root.
__device__ __forceinline__ int sp_find_readonly(const int32_t *L, int x, int limit) {
    for (int it = 0; it < limit; ++it) {
        const int p = __ldcg(L + x);
        if (p == x) return x;
        x = p;
    }
    return -1;
}

__device__ __forceinline__ int sp_find_shared(volatile int *L, int x) {
    for (int it = 0; it < kSpMaxCells; ++it) {
        const int p = L[x];
        if (p == x) return x;
        const int g = L[p];
        if (g != p) L[x] = g;
        x = g;
    }
    return -1;
}

// Without writes, as sp_find_readonly and for the same reason.
__device__ __forceinline__ int sp_find_shared_readonly(const volatile int *L, int x) {
    for (int it = 0; it < kSpMaxCells; ++it) {
        const int p = L[x];
        if (p == x) return x;
        x = p;
    }
    return -1;
}

__device__ void sp_unite_shared(int *L, int a, int b, int32_t *status) {
    for (int it = 0; it < kSpMaxCells; ++it) {
        a = sp_find_shared(L, a);
        b = sp_find_shared(L, b);
        if (a < 0 || b < 0) break;
        if (a == b) return;
        if (a > b) {
            const int t = a;
            a = b;
            b = t;
        }
        const int old = atomicMin(L + b, a);
        if (old == b) return;
        b = old;
    }
    atomicExch(status, 1);
}

// A warp takes whole tile rows, a lane the pixels lane and lane + 32 of each:
// the horizontal links of a row become runs from two ballots (a pixel's run
// root is the nearest run start at or left of it), so union-find only joins
// runs through vertical links, and a vertical link is skipped where the link
// to its left, with the two horizontal links beside it, already connects the
// same pixels (those links are processed or skipped for the same reason
// further left, ending at a processed one).  Bound by instruction issue, most
// of it in the walks, which few lanes of a row have: the links left and the
// run starts are listed, so that whole warps walk, and a run adds its length
// to its root's count once (1920x1080: 24.7 us with a thread for each pixel's
// link and addition, 23.7 with the additions of runs, 16.8 with the lists).
template <int TY>
__global__ void __launch_bounds__(32 * kSpWarps, 2048 / (32 * kSpWarps)) speckle_local_kernel(SpeckleArgs a) {
    constexpr int kSpTY = TY, kSpCells = kSpTX * TY, kSpRows = TY / kSpWarps;
    after_previous();
    __shared__ int sL[kSpCells];
    __shared__ int sC[kSpCells];  // run starts: the run's length, then roots: the segment's pixels
    __shared__ int16_t sD[kSpCells];
    __shared__ uint16_t sLink[kSpCells], sRun[kSpCells];
    __shared__ int s_links, s_runs;
    const int lane = threadIdx.x & 31, row0 = (threadIdx.x >> 5) * kSpRows;
    const int x0 = blockIdx.x * kSpTX, y0 = blockIdx.y * kSpTY;
    const unsigned upto = 0xFFFFFFFFu >> (31 - lane), below = upto >> 1;
    int16_t dv[2 * kSpRows];
#pragma unroll
    for (int k = 0; k < 2 * kSpRows; ++k) {
        const int x = x0 + lane + 32 * (k & 1), y = y0 + row0 + (k >> 1);
        dv[k] = x < a.w && y < a.h ? a.d[(size_t)y * a.w + x] : (int16_t)-1;
    }
#pragma unroll
    for (int k = 0; k < 2 * kSpRows; ++k) sD[row0 * kSpTX + 32 * k + lane] = dv[k];
    if (threadIdx.x == 0) s_links = s_runs = 0;
    __syncthreads();
#pragma unroll
    for (int r = 0; r < kSpRows; ++r) {
        const int c = (row0 + r) * kSpTX + lane, d0 = dv[2 * r], d1 = dv[2 * r + 1];
        const bool l0 = lane > 0 && sp_linked(sD[c - (lane > 0)], d0, a.thr), l1 = sp_linked(sD[c + 31], d1, a.thr);
        const unsigned s0 = ~__ballot_sync(0xFFFFFFFFu, l0);  // run starts (pixel 0 of the row always)
        const unsigned s1 = ~__ballot_sync(0xFFFFFFFFu, l1);
        const int first = c - lane;
        sL[c] = d0 >= 0 ? first + 31 - __clz(s0 & upto) : -1;
        sL[c + 32] = d1 >= 0 ? first + (s1 & upto ? 63 - __clz(s1 & upto) : 31 - __clz(s0)) : -1;
        auto link = [&](int e, int d, bool left) {
            if (row0 + r + 1 == kSpTY) return false;
            const int q = sD[e + kSpTX];
            if (!sp_linked(d, q, a.thr)) return false;
            if (!left) return true;
            const int v = sD[e - 1 + kSpTX];
            return !(sp_linked(sD[e - 1], v, a.thr) && sp_linked(v, q, a.thr));
        };
        const bool k0 = link(c, d0, l0), k1 = link(c + 32, d1, l1);
        const unsigned m0 = __ballot_sync(0xFFFFFFFFu, k0), m1 = __ballot_sync(0xFFFFFFFFu, k1);
        const unsigned h0 = s0 & __ballot_sync(0xFFFFFFFFu, d0 >= 0), h1 = s1 & __ballot_sync(0xFFFFFFFFu, d1 >= 0);
        int at = 0;
        if (lane == 0) at = atomicAdd(&s_links, __popc(m0) + __popc(m1));
        if (lane == 1) at = atomicAdd(&s_runs, __popc(h0) + __popc(h1));
        const int lk = __shfl_sync(0xFFFFFFFFu, at, 0), rn = __shfl_sync(0xFFFFFFFFu, at, 1);
        if (k0) sLink[lk + __popc(m0 & below)] = (uint16_t)c;
        if (k1) sLink[lk + __popc(m0) + __popc(m1 & below)] = (uint16_t)(c + 32);
        if (h0 >> lane & 1u) {
            const unsigned after = s0 & ~upto;
            sRun[rn + __popc(h0 & below)] = (uint16_t)c;
            sC[c] = (after ? __ffs(after) - 1 : s1 ? 31 + __ffs(s1) : 64) - lane;
        }
        if (h1 >> lane & 1u) {
            const unsigned after = s1 & ~upto;
            sRun[rn + __popc(h0) + __popc(h1 & below)] = (uint16_t)(c + 32);
            sC[c + 32] = (after ? __ffs(after) - 1 : 32) - lane;
        }
    }
    __syncthreads();
    const int links = s_links, runs = s_runs;
    for (int q = threadIdx.x; q < links; q += 32 * kSpWarps) sp_unite_shared(sL, sLink[q], sLink[q] + kSpTX, a.status);
    __syncthreads();
    for (int q = threadIdx.x; q < runs; q += 32 * kSpWarps) {
        const int c = sRun[q];
        int root = sp_find_shared_readonly(sL, c);
        if (root < 0) {
            atomicExch(a.status, 1);
            root = c;
        }
        if (root == c) continue;
        sL[c] = root;                 // an ancestor: the forest stays valid
        atomicAdd(sC + root, sC[c]);  // lengths are added to roots alone
    }
    __syncthreads();
#pragma unroll
    for (int k = 0; k < 2 * kSpRows; ++k) {
        const int x = x0 + lane + 32 * (k & 1), y = y0 + row0 + (k >> 1), c = row0 * kSpTX + 32 * k + lane;
        if (x >= a.w || y >= a.h) continue;
        const int i = y * a.w + x;
        int label = -1;
        if (dv[k] >= 0) {
            // a pixel's parent is a run's first pixel, whose parent is the
            // root.  The root's global index is at most i: local order is
            // raster order inside the tile
            const int root = sL[sL[c]];
            label = root == c ? i : -2 - ((y0 + root / kSpTX) * a.w + x0 + root % kSpTX);
            if (root == c) a.size[i] = sC[c];
        }
        a.label[i] = label;
    }
}

// Links across tile edges: first every right edge (x = 64k + 63, k =
// 0..ntx-2) of every row, then every bottom edge (y = TY k + TY - 1) of every
// column.  A right-edge link is skipped where the link above it and the two
// vertical links beside it connect the same pixels and those vertical links
// lie inside a tile (not on a tile's first row); a bottom-edge link likewise
// with the link to its left and horizontal links inside a tile.  Each skip
// rests on a link one row up or one column left, so the chain ends at a
// processed link and no component loses a connection.
template <int kSpTY> __global__ void __launch_bounds__(256) speckle_border_kernel(SpeckleArgs a) {
    after_previous();
    const int ntx = (a.w + kSpTX - 1) / kSpTX, nty = (a.h + kSpTY - 1) / kSpTY;
    const int nr = (ntx - 1) * a.h, nb = (nty - 1) * a.w;
    const int n = a.w * a.h, w = a.w, thr = a.thr;
    const int16_t *d = a.d;
    for (int k = blockIdx.x * blockDim.x + threadIdx.x; k < nr + nb; k += gridDim.x * blockDim.x) {
        int i, j;
        bool redundant;
        if (k < nr) {
            const int y = k / (ntx - 1), e = k - y * (ntx - 1);
            i = y * w + e * kSpTX + kSpTX - 1;
            j = i + 1;
            if (!sp_linked(d[i], d[j], thr)) continue;
            redundant = (y % kSpTY) != 0 && sp_linked(d[i - w], d[j - w], thr) && sp_linked(d[i - w], d[i], thr) &&
                        sp_linked(d[j - w], d[j], thr);
        } else {
            const int kb = k - nr, e = kb / w, x = kb - e * w;
            i = (e * kSpTY + kSpTY - 1) * w + x;
            j = i + w;
            if (!sp_linked(d[i], d[j], thr)) continue;
            redundant = (x % kSpTX) != 0 && sp_linked(d[i - 1], d[j - 1], thr) && sp_linked(d[i - 1], d[i], thr) &&
                        sp_linked(d[j - 1], d[j], thr);
        }
        if (!redundant) sp_unite_global(a.label, i, j, n, a.status);
    }
}

__global__ void __launch_bounds__(256) speckle_resolve_kernel(SpeckleArgs a) {
    after_previous();
    const int n = a.w * a.h;
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
        const int l = __ldcg(a.label + i);
        if (l < 0 || l == i) continue;  // not a tile-local root, or a final root
        const int root = sp_find_readonly(a.label, l, n);
        if (root < 0) {
            atomicExch(a.status, 1);
            continue;
        }
        __stcg(a.label + i, root);            // an ancestor: the forest stays valid
        atomicAdd(a.size + root, a.size[i]);  // counts are added to final roots alone
    }
}

__global__ void __launch_bounds__(256) speckle_apply_kernel(SpeckleArgs a) {
    after_previous();
    const int n = a.w * a.h;
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
        int r = a.label[i];
        const int16_t dv = a.d[i];
        if (r < -1) r = a.label[-2 - r];  // the tile-local root's final root (itself if it is one)
        a.out[i] = r >= 0 && a.size[r] >= a.min_size ? dv : (int16_t)-1;
    }
}

size_t speckle_workspace(int w, int h) {
    return align_up(16, 256) + 2 * align_up((size_t)w * h * sizeof(int32_t), 256);
}

elas_status launch_speckle(const int16_t *d, int w, int h, int thr, int min_size, int16_t *out, void *ws,
                           cudaStream_t st) {
    SpeckleArgs a;
    char *b = reinterpret_cast<char *>(ws);
    a.status = reinterpret_cast<int32_t *>(b);
    a.label = reinterpret_cast<int32_t *>(b + align_up(16, 256));
    a.size = reinterpret_cast<int32_t *>(b + align_up(16, 256) + align_up((size_t)w * h * sizeof(int32_t), 256));
    a.d = d;
    a.out = out;
    a.w = w;
    a.h = h;
    a.thr = thr;
    a.min_size = min_size;
    if (cudaMemsetAsync(a.status, 0, sizeof(int32_t), st) != cudaSuccess) return launch_status("speckle status");
    const int ntx = (w + kSpTX - 1) / kSpTX;
    const int ty = ntx * ((h + 31) / 32) >= sm_count() ? 32 : 16, nty = (h + ty - 1) / ty;
    launch_after(ty == 32 ? speckle_local_kernel<32> : speckle_local_kernel<16>, dim3(ntx, nty), 32 * kSpWarps, 0, st,
                 a);
    elas_status s = launch_status("speckle_local_kernel");
    if (s != ELAS_OK) return s;
    const int cap = sm_count() * 8, links = (ntx - 1) * h + (nty - 1) * w;
    if (links > 0) {
        launch_after(ty == 32 ? speckle_border_kernel<32> : speckle_border_kernel<16>, min((links + 255) / 256, cap),
                     256, 0, st, a);
        if ((s = launch_status("speckle_border_kernel")) != ELAS_OK) return s;
    }
    const int blocks = min((w * h + 255) / 256, cap);
    launch_after(speckle_resolve_kernel, blocks, 256, 0, st, a);
    if ((s = launch_status("speckle_resolve_kernel")) != ELAS_OK) return s;
    launch_after(speckle_apply_kernel, blocks, 256, 0, st, a);
    return launch_status("speckle_apply_kernel");
}

}  // namespace elas

extern "C" size_t elas_speckle_workspace_bytes(int32_t w, int32_t h) {
    if (w < 1 || h < 1 || w > 16383 || h > 16383) return 0;
    return elas::speckle_workspace(w, h);
}

extern "C" elas_status elas_speckle(const int16_t *d, int32_t w, int32_t h, int32_t sim_threshold,
                                    int32_t min_size, int16_t *out, void *workspace, size_t workspace_bytes,
                                    elas_stream stream) {
    using namespace elas;
    if (w < 1 || h < 1 || w > 16383 || h > 16383) return fail(ELAS_ERR_INVALID_ARG, "map size %dx%d", w, h);
    if (sim_threshold < 0) return fail(ELAS_ERR_INVALID_ARG, "sim_threshold %d < 0", sim_threshold);
    if (!d || !out || !workspace) return fail(ELAS_ERR_INVALID_ARG, "NULL buffer");
    if (!aligned(workspace, 256)) return fail(ELAS_ERR_INVALID_ARG, "workspace not 256-byte aligned");
    if (workspace_bytes < speckle_workspace(w, h))
        return fail(ELAS_ERR_CAPACITY, "workspace %zu < %zu bytes", workspace_bytes, speckle_workspace(w, h));
    return launch_speckle(d, w, h, sim_threshold, min_size, out, workspace, to_stream(stream));
}

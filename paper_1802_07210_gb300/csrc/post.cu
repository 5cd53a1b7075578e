// Left-right consistency check and post-processing (Sec. III.A, Fig. 1(i)).
//
// lr_check_kernel   one CTA per image row; both rows are staged in shared
//                   memory before any write, so the in-place update reads
//                   only unmodified values (rows are independent).
// post_pass_kernel  one pass per launch, one thread per pixel: gap
//                   interpolation along rows or columns (the maximal invalid
//                   run through a pixel is found by scanning at most
//                   ipol_gap_width steps each way), the adaptive mean along
//                   rows or columns (taps in ascending offset order, FP32
//                   without contraction), or the copy to float.
#include "launch.cuh"

namespace elas {

// V pixels (2 V bytes) as one word.
template <int V> struct LrVec;
template <> struct LrVec<2> { using T = uint32_t; };
template <> struct LrVec<1> { using T = uint16_t; };

// One row of both maps, V pixels per access.
template <int V> __device__ __forceinline__ void lr_check_row(const LrArgs &a, size_t row, int16_t *sL, int16_t *sR) {
    using T = typename LrVec<V>::T;
    union Px {
        T v;
        int16_t d[V];
    };
    const int w = a.w, thr = a.thr, n = w / V;
    T *gL = reinterpret_cast<T *>(a.dL + row), *gR = reinterpret_cast<T *>(a.dR + row);
    constexpr int kAhead = 3;  // loads of each map in flight
    for (int c0 = threadIdx.x; c0 < n; c0 += kAhead * blockDim.x) {
        T l[kAhead], r[kAhead];
#pragma unroll
        for (int k = 0; k < kAhead; ++k) {
            const int c = c0 + k * blockDim.x;
            if (c < n) l[k] = gL[c], r[k] = gR[c];
        }
#pragma unroll
        for (int k = 0; k < kAhead; ++k) {
            const int c = c0 + k * blockDim.x;
            if (c < n) reinterpret_cast<T *>(sL)[c] = l[k], reinterpret_cast<T *>(sR)[c] = r[k];
        }
    }
    __syncthreads();
    uint8_t *maskL = a.maskL, *maskR = a.maskR;
    for (int c = threadIdx.x; c < n; c += blockDim.x) {
        Px l, r;
        l.v = reinterpret_cast<const T *>(sL)[c];
        r.v = reinterpret_cast<const T *>(sR)[c];
#pragma unroll
        for (int k = 0; k < V; ++k) {
            const int u = V * c + k, d = l.d[k], e = r.d[k];
            const int dr = d >= 0 && d <= u ? sR[u - d] : -1;
            const int dl = e >= 0 && e < w - u ? sL[u + e] : -1;
            const bool kl = dr >= 0 && abs(d - dr) <= thr, kr = dl >= 0 && abs(e - dl) <= thr;
            if (!kl) l.d[k] = -1;
            if (!kr) r.d[k] = -1;
            if (maskL) maskL[row + u] = kl;
            if (maskR) maskR[row + u] = kr;
        }
        gL[c] = l.v;
        gR[c] = r.v;
    }
}

// Two pixels an access where every row of both maps is 4-byte aligned (wider
// ones conflict in the gathers' banks), three accesses of each map in flight
// and 32 registers: 64 x 1242x375 123 -> 90 us (one pixel an access and one
// in flight before).
__device__ __forceinline__ void lr_check_body(const LrArgs &a, const VB &vb) {
    extern __shared__ __align__(16) int16_t s_rows[];
    int16_t *sL = s_rows, *sR = s_rows + ((a.w + 7) & ~7);
    const size_t row = (size_t)vb.x * a.w;
    const unsigned al = (unsigned)(2 * a.w) | (unsigned)reinterpret_cast<uintptr_t>(a.dL) |
                        (unsigned)reinterpret_cast<uintptr_t>(a.dR);
    if (!(al & 3))
        lr_check_row<2>(a, row, sL, sR);
    else
        lr_check_row<1>(a, row, sL, sR);
}

__global__ void __launch_bounds__(256, 8) lr_check_kernel(LrArgs a) {
    after_previous();
    lr_check_body(a, vb_single());
}
__global__ void __launch_bounds__(256, 8) lr_check_kernel_b(const LrArgs *__restrict__ tab, VMap vm) {
    const VB vb = vb_batch(vm);
    lr_check_body(slot_entry(tab, vm.stride, vb.slot), vb);
}

// Gap interpolation along a row or a column at element k of a line of
// length len (stride es from base); In is LineIn (global maps, size_t
// indices).
template <class In, class I>
__device__ __forceinline__ float gap_at(const In &in, I base, I es, int k, int len, int gap) {
    const float x = in.at(base + (I)k * es);
    float res = x;
    if (x < 0.0f) {
        // nearest valid element on each side within gap steps
        int l = -1, r = -1;
        for (int s = 1; s <= gap && k - s >= 0; ++s)
            if (in.at(base + (I)(k - s) * es) >= 0.0f) { l = k - s; break; }
        for (int s = 1; s <= gap && k + s < len; ++s)
            if (in.at(base + (I)(k + s) * es) >= 0.0f) { r = k + s; break; }
        if (l >= 0 && r >= 0 && r - l - 1 <= gap) {
            const float d1 = in.at(base + (I)l * es), d2 = in.at(base + (I)r * es);
            res = fabsf(__fsub_rn(d1, d2)) < 3.0f ? __fmul_rn(__fadd_rn(d1, d2), 0.5f) : fminf(d1, d2);
        }
    }
    return res;
}

constexpr int kMeanRadius = 3;

// Adaptive mean along a line: taps in ascending offset order, FP32 without
// contraction.
template <class In, class I>
__device__ __forceinline__ float mean_at(const In &in, I base, I es, int k, int len) {
    const float d0 = in.at(base + (I)k * es);
    float res = d0;
    if (d0 >= 0.0f) {
        float sw = 0.0f, swd = 0.0f;
#pragma unroll
        for (int o = -kMeanRadius; o <= kMeanRadius; ++o) {
            const int m = k + o;
            if (m < 0 || m >= len) continue;
            const float di = in.at(base + (I)m * es);
            if (di < 0.0f) continue;
            const float wgt = __fsub_rn(4.0f, fabsf(__fsub_rn(di, d0)));
            if (wgt > 0.0f) {
                sw = __fadd_rn(sw, wgt);
                swd = __fadd_rn(swd, __fmul_rn(wgt, di));
            }
        }
        res = __fdiv_rn(swd, sw);
    }
    return res;
}

// One pass of post-processing over a 32x8 pixel tile: gap interpolation or
// adaptive mean along rows or columns, or the int16 -> float copy.
__device__ __forceinline__ void post_pass_body(const PostArgs &a, const VB &vb) {
    const int w = a.w, h = a.h;
    const int u = vb.x * blockDim.x + threadIdx.x;
    const int v = vb.y * blockDim.y + threadIdx.y;
    if (u >= w || v >= h) return;
    const int kind = a.kind;
    float res;
    if (kind == kPostCopy) {
        res = a.in.at((size_t)v * w + u);
    } else {
        const int vertical = kind == kPostGapCols || kind == kPostMeanCols;
        const int len = vertical ? h : w;
        const int k = vertical ? v : u;
        const size_t base = vertical ? (size_t)u : (size_t)v * w;
        const size_t es = vertical ? (size_t)w : 1;
        res = kind <= kPostGapCols ? gap_at(a.in, base, es, k, len, a.gap) : mean_at(a.in, base, es, k, len);
    }
    a.out[(size_t)v * w + u] = res;
}

__global__ void __launch_bounds__(256) post_pass_kernel(PostArgs a) {
    after_previous();
    post_pass_body(a, vb_single());
}
__global__ void __launch_bounds__(256) post_pass_kernel_b(const PostArgs *__restrict__ tab, VMap vm) {
    const VB vb = vb_batch(vm);
    post_pass_body(slot_entry(tab, vm.stride, vb.slot), vb);
}

// ---------------------------------------------------------------------------
// Fused post-processing: the four passes on one 32 x 24 tile in shared memory.
//
// The output tile needs the vertical mean over rows +-3 (r), which needs the
// horizontal mean over columns +-3, which needs the column gap pass over
// rows +-g (g = ipol_gap_width), which needs the row gap pass over columns
// +-g: the tile is loaded with a halo H = r + g, pixels outside the image
// read -1.  That is the same as the per-pass kernels, whose searches stop at
// the image border, because a -1 is never taken as a valid neighbour or a
// tap.  Each pass runs over exactly the region the next one reads, with the
// same arithmetic as the per-pass kernels.  Regions are walked as one linear
// index split into row and column by a multiply-high; the means take four
// outputs along their line per thread (ten values in registers instead of 28
// reads) and no branch: an invalid tap is far below every disparity, so its
// weight is zero, and adding a zero leaves the sums as they are.  Bound by
// instruction issue (400 thread instructions a pixel; 720 with a branch per
// tap, searches that stop early and one output per thread): 1920x1080 map 43
// -> 28 us, 640x480 pair's LR check and post-processing 21 -> 17 us.
// ---------------------------------------------------------------------------
constexpr int kFusedTX = 32;  // tile width (one warp across)
constexpr int kFusedTY = 24;  // (24 + 2 * 3) rows * 8 four-pixel groups: 240 of the CTA's 256 threads
constexpr float kFusedInvalid = -1e4f;
constexpr int kFusedMaxGap = 16;
constexpr int kFusedHalo = kFusedMaxGap + kMeanRadius;

// Row of element i of a region w wide: floor(i / w) = umulhi(i, m) with
// m = floor((2^32 - 1) / w) + 1, exact for i < 2^32 / w (here i < 2^13).
struct RowSplit {
    unsigned w, m;
    __device__ __forceinline__ explicit RowSplit(int width) : w((unsigned)width), m(0xFFFFFFFFu / (unsigned)width + 1u) {}
    __device__ __forceinline__ void at(int i, int &row, int &col) const {
        const unsigned q = w == 1u ? (unsigned)i : __umulhi((unsigned)i, m);
        row = (int)q;
        col = i - (int)(q * w);
    }
};

// gap_at for an element of the tile whose gap neighbours on either side lie
// inside it.  G: the gap width when known at compile time; 0: both sides a step
// at a time; -1 (kFusedWideGap and more): one side after the other, four values
// at a time, the second only as far as the gap allows.  A wide gap's search is a
// chain of loads, which few CTAs of a small map do not hide: 640x480, gap 16,
// in steps 28.7 us, in fours 19.4 (1920x1080 66.0 and 60.6; gap 8 45.3 and
// 45.1, gap 5 38.1 and 41.7).
constexpr int kFusedWideGap = 8;
template <int G> __device__ __forceinline__ float tile_gap(const float *v, int es, int gap) {
    const float x = v[0];
    if (x >= 0.0f) return x;
    int l = 0, r = 0;  // distance of the nearest valid element on each side
    float d1 = 0.0f, d2 = 0.0f;
    if constexpr (G > 0) {
#pragma unroll
        for (int s = G; s >= 1; --s) {
            const float a = v[-s * es], b = v[s * es];
            if (a >= 0.0f) l = s, d1 = a;
            if (b >= 0.0f) r = s, d2 = b;
        }
    } else if constexpr (G == 0) {
        for (int s = 1; s <= gap && !(l && r); ++s) {
            const float a = v[-s * es], b = v[s * es];
            if (!l && a >= 0.0f) l = s, d1 = a;
            if (!r && b >= 0.0f) r = s, d2 = b;
        }
    } else {
        auto nearest = [&](int dir, int most, float &d) {
            int at = 0;
            for (int s = 1; s <= most && !at; s += 4) {
                float a[4];
#pragma unroll
                for (int j = 0; j < 4; ++j) a[j] = s + j <= most ? v[dir * (s + j)] : kFusedInvalid;
#pragma unroll
                for (int j = 3; j >= 0; --j)
                    if (a[j] >= 0.0f) at = s + j, d = a[j];
            }
            return at;
        };
        l = nearest(-es, gap, d1);
        if (!l) return x;
        r = nearest(es, gap + 1 - l, d2);
    }
    if (!l || !r || l + r - 1 > gap) return x;
    return fabsf(__fsub_rn(d1, d2)) < 3.0f ? __fmul_rn(__fadd_rn(d1, d2), 0.5f) : fminf(d1, d2);
}

// Both gap passes of the tile: rows into nxt, then columns back into cur.
template <int G>
__device__ __forceinline__ void tile_gaps(float *cur, float *nxt, int PX, int PY, int g, const RowSplit &inner) {
    const int cw = PX - 2 * g;
    // rows: every row, the columns the later passes read
    for (int i = threadIdx.x; i < cw * PY; i += blockDim.x) {
        int yy, c;
        inner.at(i, yy, c);
        const int at = yy * PX + g + c;
        nxt[at] = tile_gap<G>(cur + at, 1, g);
    }
    __syncthreads();
    // columns: those columns, the rows the means read
    for (int i = threadIdx.x; i < cw * (PY - 2 * g); i += blockDim.x) {
        int rr, c;
        inner.at(i, rr, c);
        const int at = (g + rr) * PX + g + c;
        cur[at] = tile_gap<G>(nxt + at, PX, g);
    }
    __syncthreads();
}

// Adaptive means of v[3..6] over their seven-value windows.
__device__ __forceinline__ void mean4(const float *v, float *out) {
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        const float d0 = v[j + kMeanRadius];
        float sw = 0.0f, swd = 0.0f;
#pragma unroll
        for (int o = 0; o <= 2 * kMeanRadius; ++o) {
            const float di = v[j + o];
            const float wgt = fmaxf(__fsub_rn(4.0f, fabsf(__fsub_rn(di, d0))), 0.0f);
            sw = __fadd_rn(sw, wgt);
            swd = __fadd_rn(swd, __fmul_rn(wgt, di));
        }
        out[j] = d0 >= 0.0f ? __fdiv_rn(swd, sw) : d0;
    }
}

__device__ __forceinline__ void fused_post_body(const FusedPostArgs &a, const VB &vb) {
    constexpr int TX = kFusedTX, TY = kFusedTY;
    __shared__ float s_a[(TY + 2 * kFusedHalo) * (TX + 2 * kFusedHalo)];
    __shared__ float s_b[(TY + 2 * kFusedHalo) * (TX + 2 * kFusedHalo)];
    const int w = a.w, h = a.h;
    const int g = a.gap, r = a.mean ? kMeanRadius : 0, H = g + r;
    const int PX = TX + 2 * H, PY = TY + 2 * H;  // tile pitch and rows
    const int x0 = vb.x * TX - H, y0 = vb.y * TY - H;
    const int tid = threadIdx.x, nth = blockDim.x;
    if (H == 0) {  // no pass: the map as floats
        for (int i = tid; i < TX * TY; i += nth) {
            const int gx = x0 + i % TX, gy = y0 + i / TX;
            if (gx < w && gy < h) a.out[(size_t)gy * w + gx] = (float)a.d[(size_t)gy * w + gx];
        }
        return;
    }
    const RowSplit full(PX), inner(PX - 2 * g);
    for (int i = tid; i < PX * PY; i += nth) {
        int yy, xx;
        full.at(i, yy, xx);
        const int gx = x0 + xx, gy = y0 + yy;
        const int d = gx >= 0 && gx < w && gy >= 0 && gy < h ? a.d[(size_t)gy * w + gx] : -1;
        s_a[i] = d >= 0 ? (float)d : kFusedInvalid;
    }
    __syncthreads();
    float *cur = s_a, *nxt = s_b;
    if (g == 3)  // the default width
        tile_gaps<3>(cur, nxt, PX, PY, g, inner);
    else if (g >= kFusedWideGap)
        tile_gaps<-1>(cur, nxt, PX, PY, g, inner);
    else if (g > 0)
        tile_gaps<0>(cur, nxt, PX, PY, g, inner);
    // an invalid pixel that no pass filled keeps the map's own value
    auto put = [&](int xx, int yy, float v) {
        const int gx = x0 + xx, gy = y0 + yy;
        if (gx >= w || gy >= h) return;
        const size_t at = (size_t)gy * w + gx;
        a.out[at] = v >= 0.0f ? v : (float)a.d[at];
    };
    if (r == 0) {
        for (int i = tid; i < TX * TY; i += nth) put(H + i % TX, H + i / TX, cur[(H + i / TX) * PX + H + i % TX]);
        return;
    }
    // horizontal mean: the output columns, rows +-r
    float v[4 + 2 * kMeanRadius], m[4];
    for (int i = tid; i < TX / 4 * (TY + 2 * kMeanRadius); i += nth) {
        const int at = (g + i / (TX / 4)) * PX + H + 4 * (i % (TX / 4));
#pragma unroll
        for (int k = 0; k < 4 + 2 * kMeanRadius; ++k) v[k] = cur[at + k - kMeanRadius];
        mean4(v, m);
#pragma unroll
        for (int k = 0; k < 4; ++k) nxt[at + k] = m[k];
    }
    __syncthreads();
    // vertical mean
    for (int i = tid; i < TX * TY / 4; i += nth) {
        const int xx = H + i % TX, yy = H + 4 * (i / TX);
#pragma unroll
        for (int k = 0; k < 4 + 2 * kMeanRadius; ++k) v[k] = nxt[(yy + k - kMeanRadius) * PX + xx];
        mean4(v, m);
#pragma unroll
        for (int k = 0; k < 4; ++k) put(xx, yy + k, m[k]);
    }
}

__global__ void __launch_bounds__(256) fused_post_kernel(FusedPostArgs a) {
    after_previous();
    fused_post_body(a, vb_single());
}
__global__ void __launch_bounds__(256) fused_post_kernel_b(const FusedPostArgs *__restrict__ tab, VMap vm) {
    const VB vb = vb_batch(vm);
    fused_post_body(slot_entry(tab, vm.stride, vb.slot), vb);
}

bool post_fusable(const elas_params *p) { return p->ipol_gap_width <= kFusedMaxGap; }

FusedPostArgs fused_post_args(const int16_t *d, int w, int h, const elas_params *p, float *out) {
    return FusedPostArgs{d, out, w, h, p->ipol_gap_width > 0 ? p->ipol_gap_width : 0,
                         p->filter_adaptive_mean ? 1 : 0};
}

dim3 fused_post_grid(int w, int h) {
    return dim3((w + kFusedTX - 1) / kFusedTX, (h + kFusedTY - 1) / kFusedTY);
}

size_t post_workspace(int w, int h) { return 2 * align_up((size_t)w * h * sizeof(float), 256); }

size_t lr_smem(int w) { return 2 * (size_t)((w + 7) & ~7) * sizeof(int16_t); }

static elas_status lr_smem_attr(const void *fn, size_t smem) {
    return allow_smem(fn, smem, lr_smem(16383), "lr_check smem attribute");  // the widest map
}

elas_status launch_lr_check(int16_t *dL, int16_t *dR, int w, int h, int thr, uint8_t *maskL, uint8_t *maskR,
                            cudaStream_t st) {
    const size_t smem = lr_smem(w);
    elas_status s = lr_smem_attr((const void *)lr_check_kernel, smem);
    if (s != ELAS_OK) return s;
    launch_after(lr_check_kernel, h, 256, smem, st, LrArgs{dL, dR, w, h, thr, maskL, maskR});
    return launch_status("lr_check_kernel");
}

// The ordered passes of post-processing for one map: gap interpolation
// (rows, then columns) and the adaptive mean (rows, then columns); the last
// pass writes `out`, the others alternate between the two scratch maps.  With
// no pass enabled the one pass is the copy to float.
int post_passes(const int16_t *d, int w, int h, const elas_params *p, float *out, void *ws, PostArgs *passes) {
    float *A = reinterpret_cast<float *>(ws);
    float *B = reinterpret_cast<float *>(reinterpret_cast<char *>(ws) + align_up((size_t)w * h * sizeof(float), 256));
    int kinds[4], np = 0;
    if (p->ipol_gap_width > 0) {
        kinds[np++] = kPostGapRows;
        kinds[np++] = kPostGapCols;
    }
    if (p->filter_adaptive_mean) {
        kinds[np++] = kPostMeanRows;
        kinds[np++] = kPostMeanCols;
    }
    if (np == 0) kinds[np++] = kPostCopy;
    LineIn in{d, nullptr};
    for (int i = 0; i < np; ++i) {
        float *dst = (i == np - 1) ? out : ((i & 1) ? B : A);
        passes[i] = PostArgs{in, dst, w, h, kinds[i], p->ipol_gap_width};
        in = LineIn{nullptr, dst};
    }
    return np;
}

dim3 post_grid(int w, int h) { return dim3((w + 31) / 32, (h + 7) / 8); }

elas_status launch_post(const int16_t *d, int w, int h, const elas_params *p, float *out, void *ws, cudaStream_t st) {
    if (post_fusable(p)) {
        launch_after(fused_post_kernel, fused_post_grid(w, h), 256, 0, st, fused_post_args(d, w, h, p, out));
        return launch_status("fused_post_kernel");
    }
    PostArgs passes[4];
    const int np = post_passes(d, w, h, p, out, ws, passes);
    for (int i = 0; i < np; ++i) {
        launch_after(post_pass_kernel, post_grid(w, h), dim3(32, 8), 0, st, passes[i]);
        elas_status s = launch_status("post_pass_kernel");
        if (s != ELAS_OK) return s;
    }
    return ELAS_OK;
}

// Batched LR check and post-processing.  Pairs with fused[i] run the fused
// kernel (table fused_tab); the others run npass[i] separate passes, pass k
// from table post_tab[k] (npass 0 and not fused: no post-processing).
elas_status launch_lr_post_b(const LrArgs *lr_tab, const LrArgs *host_lr, const PostArgs *const *post_tab,
                             const int *npass, const FusedPostArgs *fused_tab, const int *fused, const VMap &pairs,
                             cudaStream_t st) {
    if (pairs.n == 0) return ELAS_OK;
    VMap m_lr;
    vmap_clear(m_lr, pairs.stride);
    int maxw = 1, maxp = 0;
    for (int i = 0; i < pairs.n; ++i) {
        const LrArgs &l = slot_entry(host_lr, pairs.stride, pairs.slot[i]);
        vmap_add(m_lr, pairs.slot[i], dim3(l.h));
        maxw = max(maxw, l.w);
        maxp = max(maxp, npass[i]);
    }
    const size_t smem = lr_smem(maxw);
    elas_status s = lr_smem_attr((const void *)lr_check_kernel_b, smem);
    if (s != ELAS_OK) return s;
    lr_check_kernel_b<<<vmap_total(m_lr), 256, smem, st>>>(lr_tab, m_lr);
    if ((s = launch_status("lr_check_kernel_b")) != ELAS_OK) return s;
    VMap m_f;
    vmap_clear(m_f, pairs.stride);
    for (int i = 0; i < pairs.n; ++i) {
        const LrArgs &l = slot_entry(host_lr, pairs.stride, pairs.slot[i]);
        vmap_add(m_f, pairs.slot[i], fused[i] ? fused_post_grid(l.w, l.h) : dim3(0));
    }
    if (vmap_total(m_f) > 0) {
        fused_post_kernel_b<<<vmap_total(m_f), 256, 0, st>>>(fused_tab, m_f);
        if ((s = launch_status("fused_post_kernel_b")) != ELAS_OK) return s;
    }
    for (int k = 0; k < maxp && k < 4; ++k) {
        VMap m;
        vmap_clear(m, pairs.stride);
        for (int i = 0; i < pairs.n; ++i) {
            const LrArgs &l = slot_entry(host_lr, pairs.stride, pairs.slot[i]);
            vmap_add(m, pairs.slot[i], k < npass[i] ? post_grid(l.w, l.h) : dim3(0));
        }
        if (vmap_total(m) == 0) continue;
        post_pass_kernel_b<<<vmap_total(m), dim3(32, 8), 0, st>>>(post_tab[k], m);
        if ((s = launch_status("post_pass_kernel_b")) != ELAS_OK) return s;
    }
    return ELAS_OK;
}

}  // namespace elas

extern "C" elas_status elas_lr_check(int16_t *dL, int16_t *dR, int32_t w, int32_t h, int32_t lr_threshold,
                                     uint8_t *maskL, uint8_t *maskR, elas_stream stream) {
    using namespace elas;
    if (w < 1 || h < 1 || w > 16383 || h > 16383) return fail(ELAS_ERR_INVALID_ARG, "image size %dx%d", w, h);
    if (!dL || !dR) return fail(ELAS_ERR_INVALID_ARG, "NULL disparity map");
    if (lr_threshold < 0) return fail(ELAS_ERR_INVALID_ARG, "lr_threshold %d", lr_threshold);
    return launch_lr_check(dL, dR, w, h, lr_threshold, maskL, maskR, to_stream(stream));
}

extern "C" size_t elas_postprocess_workspace_bytes(int32_t w, int32_t h) {
    if (w < 1 || h < 1) return 0;
    return elas::post_workspace(w, h);
}

extern "C" elas_status elas_postprocess(const int16_t *d, int32_t w, int32_t h, const elas_params *p, float *out,
                                        void *workspace, size_t workspace_bytes, elas_stream stream) {
    using namespace elas;
    elas_status s = check_params(p, w, h);
    if (s != ELAS_OK) return s;
    if (!d || !out || !workspace) return fail(ELAS_ERR_INVALID_ARG, "NULL buffer");
    if (!aligned(workspace, 256)) return fail(ELAS_ERR_INVALID_ARG, "workspace not 256-byte aligned");
    if (workspace_bytes < post_workspace(w, h))
        return fail(ELAS_ERR_CAPACITY, "workspace %zu < %zu bytes", workspace_bytes, post_workspace(w, h));
    return launch_post(d, w, h, p, out, workspace, to_stream(stream));
}

// ---------------------------------------------------------------------------
// Median filter (Sec. VII, the refinement applied for the comparison with
// CSM; the paper gives no size).  Every valid pixel takes the median of the
// valid disparities in its (2r+1) x (2r+1) window clipped to the image (the
// lower median, element (n-1)/2 in sorted order, for an even count n);
// invalid pixels stay -1.  A tile with its halo in shared memory (cells
// outside the image read -1, so they drop out as invalid values).  The 3x3
// window has a kernel of its own (median3_kernel); for the larger ones the
// window is loaded into registers and the median is selected bit by bit:
// disparities are below 1024, so from bit 9 down, the count of valid values
// that share the bits chosen so far and have a 0 at the current bit decides
// that bit of the k-th smallest value (k = (n-1)/2).
// ---------------------------------------------------------------------------
namespace elas {

constexpr int kMedTX = 32, kMedTY = 8, kMedMaxR = 3;

template <int R> __device__ __forceinline__ int median_select(const int16_t *c, int SW) {
    constexpr int N = (2 * R + 1) * (2 * R + 1);
    int v[N];
    int n = 0;
#pragma unroll
    for (int j = 0; j < N; ++j) {
        v[j] = c[(j / (2 * R + 1) - R) * SW + (j % (2 * R + 1) - R)];
        n += v[j] >= 0;
    }
    int k = (n - 1) / 2, val = 0;
#pragma unroll
    for (int b = 9; b >= 0; --b) {
        int cnt = 0;
#pragma unroll
        for (int j = 0; j < N; ++j) cnt += (v[j] >= 0) & ((v[j] >> b) == (val >> b));
        if (k >= cnt) {
            k -= cnt;
            val |= 1 << b;
        }
    }
    return val;
}

__global__ void __launch_bounds__(kMedTX *kMedTY) median_kernel(const int16_t *__restrict__ d, int w, int h, int r,
                                                                int16_t *__restrict__ out) {
    __shared__ int16_t s[(kMedTY + 2 * kMedMaxR) * (kMedTX + 2 * kMedMaxR)];
    const int SW = kMedTX + 2 * r, SH = kMedTY + 2 * r;
    const int x0 = blockIdx.x * kMedTX - r, y0 = blockIdx.y * kMedTY - r;
    const int tid = threadIdx.y * kMedTX + threadIdx.x;
    for (int k = tid; k < SW * SH; k += kMedTX * kMedTY) {
        const int x = x0 + k % SW, y = y0 + k / SW;
        s[k] = (x >= 0 && x < w && y >= 0 && y < h) ? d[(size_t)y * w + x] : (int16_t)-1;
    }
    __syncthreads();
    const int x = blockIdx.x * kMedTX + threadIdx.x, y = blockIdx.y * kMedTY + threadIdx.y;
    if (x >= w || y >= h) return;
    const int16_t *c = s + (threadIdx.y + r) * SW + threadIdx.x + r;
    int res = -1;
    if (c[0] >= 0) {
        res = r == 0 ? c[0] : (r == 2 ? median_select<2>(c, SW) : median_select<3>(c, SW));
    }
    out[(size_t)y * w + x] = (int16_t)res;
}

// 3x3.  Bound by the integer pipe, so two neighbouring pixels are worked on
// as the halves of one word (packed 16-bit min and max), in two rows a
// thread, and the columns of three are sorted once for the three windows
// they lie in.  With the sorted columns' low, middle and high values sorted
// again each, the five largest of the nine come from a short network.  With
// `bad` invalid values (negative, so they sort first) the median is the value
// of rank 4 + bad / 2.  One pixel a thread, sorted by odd-even transposition,
// took 24.1 us at 1920x1080, this 8.6 us.
constexpr int kMed3TX = 64, kMed3TY = 16, kMed3W = kMed3TX / 2 + 2;

__device__ __forceinline__ void med3_sort(uint32_t &a, uint32_t &b) {
    const uint32_t lo = __vmins2(a, b);
    b = __vmaxs2(a, b);
    a = lo;
}

// (high half of a, low half of b): the pair of pixels between two pairs.
__device__ __forceinline__ uint32_t med3_between(uint32_t a, uint32_t b) { return __byte_perm(a, b, 0x5432); }

// kWide: an even width and 4-byte aligned maps, read and written by words.
template <bool kWide>
__global__ void __launch_bounds__(256) median3_kernel(const int16_t *__restrict__ d, int w, int h,
                                                      int16_t *__restrict__ out) {
    // a row holds the pixels x0 - 2 .. x0 + kMed3TX + 1
    __shared__ uint32_t s[kMed3TY + 2][kMed3W];
    after_previous();
    d = settled(d);
    const int tid = threadIdx.x, tx = tid & 31, ty = tid >> 5;
    const int x0 = blockIdx.x * kMed3TX, y0 = blockIdx.y * kMed3TY;
    if (kWide) {
        for (int k = tid; k < (kMed3TY + 2) * kMed3W; k += 256) {
            const int r = k / kMed3W, c = k - r * kMed3W, x = x0 - 2 + 2 * c, y = y0 - 1 + r;
            s[r][c] = x >= 0 && x < w && y >= 0 && y < h
                          ? *reinterpret_cast<const uint32_t *>(d + (size_t)y * w + x)
                          : 0xFFFFFFFFu;
        }
    } else {
        for (int k = tid; k < (kMed3TY + 2) * 2 * kMed3W; k += 256) {
            const int r = k / (2 * kMed3W), c = k - r * 2 * kMed3W, x = x0 - 2 + c, y = y0 - 1 + r;
            reinterpret_cast<int16_t *>(s[r])[c] =
                x >= 0 && x < w && y >= 0 && y < h ? d[(size_t)y * w + x] : (int16_t)-1;
        }
    }
    __syncthreads();
    uint32_t A[4], B[4], C[4], neg = 0;
#pragma unroll
    for (int r = 0; r < 4; ++r) {
        const uint32_t *q = s[2 * ty + r] + tx;
        B[r] = q[1];
        A[r] = med3_between(q[0], B[r]);
        C[r] = med3_between(B[r], q[2]);
        neg |= A[r] | C[r];
    }
    const bool holes = (neg & 0x80008000u) != 0;
    uint32_t la = A[1], ha = A[2], lc = C[1], hc = C[2];  // the two rows that both windows share
    med3_sort(la, ha);
    med3_sort(lc, hc);
#pragma unroll
    for (int o = 0; o < 2; ++o) {
        const int x = x0 + 2 * tx, y = y0 + 2 * ty + o;
        if (x >= w || y >= h) return;
        // sorted columns x - 1 and x + 1 (their halves), x between them
        uint32_t l0 = A[3 * o], m0 = la, h0 = ha, l2 = C[3 * o], m2 = lc, h2 = hc;
        med3_sort(l0, m0);
        med3_sort(m0, h0);
        med3_sort(l2, m2);
        med3_sort(m2, h2);
        uint32_t l1 = med3_between(l0, l2), m1 = med3_between(m0, m2), h1 = med3_between(h0, h2);
        med3_sort(l0, l1);
        med3_sort(l1, l2);
        med3_sort(l0, l1);
        med3_sort(m0, m1);
        med3_sort(m1, m2);
        med3_sort(m0, m1);
        med3_sort(h0, h1);
        med3_sort(h1, h2);
        med3_sort(h0, h1);
        // h2 is the largest; then m2 and h1; then l2, p and h0; ...
        const uint32_t r8 = h2, r7 = __vmaxs2(m2, h1);
        uint32_t p = __vmins2(m2, h1);
        med3_sort(l2, p);
        med3_sort(p, h0);
        med3_sort(l2, p);
        const uint32_t r6 = h0, r5 = __vmaxs2(m1, p);
        const uint32_t r4 = __vmaxs2(__vmaxs2(__vmins2(m1, p), l2), __vmaxs2(l1, m0));
        uint32_t res = r4;
        if (holes) {
            uint32_t na = 0, nc = 0;
#pragma unroll
            for (int r = o; r < o + 3; ++r) {
                na += (A[r] >> 15) & 0x00010001u;
                nc += (C[r] >> 15) & 0x00010001u;
            }
            const uint32_t bad = na + nc + med3_between(na, nc);
            uint32_t half[2];
#pragma unroll
            for (int k = 0; k < 2; ++k) {
                const uint32_t nb = (bad >> (16 * k)) & 15u;
                half[k] = (nb < 2 ? r4 : nb < 4 ? r5 : nb < 6 ? r6 : nb < 8 ? r7 : r8) >> (16 * k) & 0xFFFFu;
                if (B[o + 1] >> (16 * k) & 0x8000u) half[k] = 0xFFFFu;
            }
            res = half[0] | half[1] << 16;
        }
        int16_t *to = out + (size_t)y * w + x;
        if (kWide) {
            *reinterpret_cast<uint32_t *>(to) = res;
        } else {
            to[0] = (int16_t)(res & 0xFFFFu);
            if (x + 1 < w) to[1] = (int16_t)(res >> 16);
        }
    }
}

}  // namespace elas

extern "C" elas_status elas_median(const int16_t *d, int32_t w, int32_t h, int32_t radius, int16_t *out,
                                   elas_stream stream) {
    using namespace elas;
    if (w < 1 || h < 1 || w > 16383 || h > 16383) return fail(ELAS_ERR_INVALID_ARG, "image size %dx%d", w, h);
    if (radius < 0 || radius > kMedMaxR) return fail(ELAS_ERR_INVALID_ARG, "median radius %d (0..%d)", radius, kMedMaxR);
    if (!d || !out) return fail(ELAS_ERR_INVALID_ARG, "NULL buffer");
    if (d == out) return fail(ELAS_ERR_INVALID_ARG, "median output must not alias its input");
    if (radius == 1) {
        const dim3 tiles((w + kMed3TX - 1) / kMed3TX, (h + kMed3TY - 1) / kMed3TY);
        if (w % 2 == 0 && aligned(d, 4) && aligned(out, 4))
            launch_after(median3_kernel<true>, tiles, 256, 0, to_stream(stream), d, w, h, out);
        else
            launch_after(median3_kernel<false>, tiles, 256, 0, to_stream(stream), d, w, h, out);
        return launch_status("median3_kernel");
    }
    const dim3 grid((w + kMedTX - 1) / kMedTX, (h + kMedTY - 1) / kMedTY);
    median_kernel<<<grid, dim3(kMedTX, kMedTY), 0, to_stream(stream)>>>(d, w, h, radius, out);
    return launch_status("median_kernel");
}

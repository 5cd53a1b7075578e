// Internal helpers shared by the CUDA translation units of libelas_gb300.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "elas_gb300.h"

namespace elas {

// Thread-local error text behind elas_last_error().
void set_error(const char *fmt, ...);
elas_status fail(elas_status st, const char *fmt, ...);
// Converts a pending launch error into ELAS_ERR_CUDA.
elas_status launch_status(const char *what);
// Validates the parameter block against the image size.
elas_status check_params(const elas_params *p, int32_t w, int32_t h);
// Streaming multiprocessors of the current device (queried once per device;
// launch grids are sized in multiples of it).
int sm_count();

inline cudaStream_t to_stream(elas_stream s) { return reinterpret_cast<cudaStream_t>(s); }

// Records a timing mark on st; while st is being captured into a graph the
// record becomes an event-record node of the graph.
inline cudaError_t record_mark(cudaEvent_t e, cudaStream_t st) {
    cudaStreamCaptureStatus cs = cudaStreamCaptureStatusNone;
    if (cudaStreamIsCapturing(st, &cs) != cudaSuccess) return cudaGetLastError();
    return cs == cudaStreamCaptureStatusActive ? cudaEventRecordWithFlags(e, st, cudaEventRecordExternal)
                                               : cudaEventRecord(e, st);
}
inline bool aligned(const void *p, size_t a) { return (reinterpret_cast<uintptr_t>(p) % a) == 0; }
inline size_t align_up(size_t x, size_t a) { return (x + a - 1) / a * a; }

constexpr int kMaxSradius = 15;
constexpr int kMaxDisp = 1023;

// Grid-vector geometry.
struct GridGeom {
    int gw, gh, nw;  // cells across, cells down, 32-bit words per cell
};
inline GridGeom grid_geom(int w, int h, const elas_params *p) {
    GridGeom g;
    g.gw = (w + p->grid_size - 1) / p->grid_size;
    g.gh = (h + p->grid_size - 1) / p->grid_size;
    g.nw = (p->disp_max + 1 + 31) / 32;
    return g;
}

// Prior table P[0..sradius] from the parameters (host, double precision).
void prior_table(const elas_params *p, int32_t *P);

// Launch of a kernel that begins with after_previous(): its CTAs may take
// their places while the last ones of the kernel before it in the stream
// still run, so the launch's own latency is hidden behind that kernel (the
// triangulation is nine kernels of 1 to 40 us: 1242x375, both sides one call
// each, 180 -> 151 us; LR check to speckle removal of 1920x1080 91 -> 80).  A
// kernel launched without it, a copy or an event waits for the whole kernel
// as ever.  Under capture it is an ordinary launch: a graph's own edges are as
// quick (640x480, twenty kernels: 143 us with them, 140 to 150 with early
// starts).
template <class... P, class... A>
inline void launch_after(void (*kernel)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t st, A... args) {
    cudaLaunchAttribute early{};
    early.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    early.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cfg.attrs = &early;
    cudaStreamCaptureStatus cs = cudaStreamCaptureStatusNone;
    if (cudaStreamIsCapturing(st, &cs) != cudaSuccess) {
        (void)cudaGetLastError();  // the launch reports what is wrong
        cs = cudaStreamCaptureStatusActive;
    }
    cfg.numAttrs = cs == cudaStreamCaptureStatusNone ? 1 : 0;
    cudaLaunchKernelEx(&cfg, kernel, P(args)...);  // errors: launch_status
}

// ---------------------------------------------------------------------------
// Device helpers
// ---------------------------------------------------------------------------

// Lets the next kernel of the stream take its places as soon as every CTA of
// this one has started.
__device__ __forceinline__ void let_next_in() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

// First statement of a kernel launched by launch_after: waits until the
// kernel before it in the stream (so, in turn, all before that) is complete
// and its writes are visible; no global memory is touched earlier.
__device__ __forceinline__ void after_previous() {
    let_next_in();
    asm volatile("griddepcontrol.wait;" ::: "memory");
}

// p, not known to the compiler before this point: a read-only load (__ldg, or
// one that a `const __restrict__` pointer allows) through it cannot be moved
// above after_previous().  Every such pointer of a kernel launched by
// launch_after goes through this, or does without the qualifier: the compiler
// no longer knows p for a global address, so plain loads through it keep their
// order with shared memory's (redundancy filter of odd lattice widths, 1739x627:
// 11.6 us, 16.6 with p settled).
template <class T> __device__ __forceinline__ T *settled(T *p) {
    asm volatile("" : "+l"(p)::"memory");
    return p;
}

// Sum of |a_i - b_i| over the 4 bytes of a and b, added to acc.
__device__ __forceinline__ uint32_t sad4_acc(uint32_t a, uint32_t b, uint32_t acc) {
    return __dp4a(__vabsdiffu4(a, b), 0x01010101u, acc);
}

// The same sum with the byte-SIMD absolute difference and its accumulating
// merge (one instruction per 4 bytes): the matchers' form (measured faster
// than the dp4a form in both).
__device__ __forceinline__ uint32_t sad4_vacc(uint32_t a, uint32_t b, uint32_t acc) {
    uint32_t r = acc;
    asm("vabsdiff4.u32.u32.u32.add %0, %1, %2, %0;" : "+r"(r) : "r"(a), "r"(b));
    return r;
}

__device__ __forceinline__ uint32_t sad16_vacc(const uint4 &a, const uint4 &b) {
    uint32_t s = sad4_vacc(a.x, b.x, 0u);
    s = sad4_vacc(a.y, b.y, s);
    s = sad4_vacc(a.z, b.z, s);
    return sad4_vacc(a.w, b.w, s);
}

// Texture of a descriptor: sum of |b - 128| over its 16 bytes.
__device__ __forceinline__ uint32_t texture16(const uint4 &a) {
    const uint32_t m = 0x80808080u;
    uint32_t s = sad4_acc(a.x, m, 0u);
    s = sad4_acc(a.y, m, s);
    s = sad4_acc(a.z, m, s);
    return sad4_acc(a.w, m, s);
}

// Hamming distance of two 128-bit census strings (Sec. VI.A).
__device__ __forceinline__ uint32_t ham16(const uint4 &a, const uint4 &b) {
    return __popc(a.x ^ b.x) + __popc(a.y ^ b.y) + __popc(a.z ^ b.z) + __popc(a.w ^ b.w);
}

}  // namespace elas

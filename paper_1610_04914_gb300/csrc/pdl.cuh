// Programmatic dependent launch: a kernel launched with launch_pdl may start
// while the kernel before it on the stream drains (or, where that one calls
// pdl_go, as soon as all of its blocks have started); it calls pdl_wait before
// it touches memory that an earlier kernel writes or reads.  pdl_wait returns
// when the kernel before has finished and its writes are visible.  Nothing that
// an earlier kernel on the stream writes may be relied on before that, not even
// what the kernel before the last one wrote (some kernels call pdl_go before
// their own pdl_wait).  Such data is read by plain loads: __ldg and
// const __restrict__ parameters tell the compiler that it does not change while
// the kernel runs, so that a load may move ahead of the wait.
//
// In interval graphs the kernels get ordinary edges, with one exception.
// Programmatic edges between graph nodes gained nothing or cost time (an interval of 96 replicas 2048 -> 2133 us, RK5 at 128^3 1108 -> 1148,
// 10 FP64 steps at 16^3 243 -> 244, 2 FP64 Heun steps at 41x11x101 59 -> 66)
// but for the pulse and the observables of FP32 lattices up to about 2^20
// sites (64^3 particle, 20 RK2 steps 500 -> 477; 45x37x27 RK4 260 -> 250;
// 128^3 513 -> 514).  On a stream every kernel gains: the first, uncaptured
// interval at 128^3 575 -> 535 us; batched steps keep ordinary launches, whose
// tiling is tuned on them.
#pragma once
#include <cuda_runtime.h>

namespace spin {

__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;\n" ::: "memory"); }
__device__ __forceinline__ void pdl_go() { asm volatile("griddepcontrol.launch_dependents;\n" ::: "memory"); }

// A word that an earlier kernel on the stream writes, read without the
// non-coherent cache.  Before pdl_wait its value may be an old one.
__device__ __forceinline__ unsigned long long load_shared_word(const long long* p) {
    unsigned long long v;
    asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];\n" : "=l"(v) : "l"(p) : "memory");
    return v;
}

constexpr long long kPdlGraphSites = 1LL << 20;

// Where a launch goes: to a stream, into a handle's own interval graph, or into
// a graph that the caller captures.  The last gets ordinary launches only: a
// caller may ask for the edges of its graph, or add to the capture, by calls
// that refuse edges with data.
enum LaunchInto { kStream = 0, kIntervalGraph = 1, kCallersGraph = 2 };
inline int launch_into(cudaStream_t st) {
    cudaStreamCaptureStatus s = cudaStreamCaptureStatusNone;
    return cudaStreamIsCapturing(st, &s) == cudaSuccess && s != cudaStreamCaptureStatusNone ? kCallersGraph : kStream;
}
// The pulse and the observables (elt: bytes of a component).
inline bool pdl_after_step(int into, int elt, long long N) {
    return into == kStream || (into == kIntervalGraph && elt == 4 && N <= kPdlGraphSites);
}

// pdl = false: an ordinary launch.
template <typename Kern, typename... Args>
cudaError_t launch_pdl(bool pdl, Kern kernel, dim3 grid, dim3 block, size_t smem, cudaStream_t st, const Args&... args) {
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = at;
    cfg.numAttrs = pdl ? 1 : 0;
    return cudaLaunchKernelEx(&cfg, kernel, args...);
}

}  // namespace spin

// Kernels that start while the one before them on the stream drains (programmatic dependent launch).
//
// Every kernel of this library calls previous_grid_done() before its first access to global memory and next_grid_may_start()
// behind it, so that nothing it reads or writes can meet the previous kernel's accesses, while launch latency, barrier
// set-up and the allocation of tensor memory lie under the previous kernel's tail.  The completion of a kernel implies that
// of all before it (its own wait has passed), so the order of the stream is kept as a whole.  A kernel launched without the
// attribute passes the wait at once: it starts behind the previous one anyway.
//
// A kernel with tensor memory lets the next one start only when its CTA holds its columns: allocation, __syncthreads(), then
// next_grid_may_start().  The allocation blocks while too few columns of the SM are free.  If the next kernel's CTA could
// take them first, it would hold them in its wait for this kernel, which would wait for them.  As it is, a CTA that
// waits with columns in its hands waits only for grids whose CTAs have theirs.
// No kernel launched this way reads global memory through the read-only path (__restrict__ const parameters, __ldg): such
// loads may be moved ahead of the wait.
#pragma once
#include <cuda_runtime.h>

#include <utility>

namespace ckpt {

__device__ __forceinline__ void previous_grid_done() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void next_grid_may_start() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

// EARLY: a kernel whose CTAs take most of an SM each.  ON_STREAMS: only where a launch goes to the stream itself, not into a
// recording: several small CTAs per SM that arrive early crowd on the SMs that drain first, while all that a replayed
// graph leaves to hide is some 0.3 us per kernel (us, none -> whole-SM kernels -> all, replayed: 32 units of 64 channels 2862 ->
// 2757 -> 2830, VGG-16 with 48 channels 1044 -> 1011 -> 1070, a float32 VGG-16 1351 -> 1351 -> 1440; launched one by one, where a
// launch takes 2 us: VGG-16 in three units per layer 2039 -> 1910 -> 1717, eight 16-channel float32 units 566 -> 558 -> 407,
// ResNet-50 at batch 128 13240 -> 12690 with all).
enum class Start { EARLY, ON_STREAMS };

inline bool starts_early(Start s, cudaStream_t st) {
    if (s == Start::EARLY) return true;
    cudaStreamCaptureStatus status = cudaStreamCaptureStatusNone;
    if (cudaStreamIsCapturing(st, &status) != cudaSuccess) { cudaGetLastError(); return false; }
    return status == cudaStreamCaptureStatusNone;
}

// Adds the attribute to a launch configuration whose attribute array has room for one more.
inline void start_early(cudaLaunchConfig_t* cfg, cudaLaunchAttribute* attrs, Start s) {
    if (!starts_early(s, cfg->stream)) return;
    attrs[cfg->numAttrs].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attrs[cfg->numAttrs].val.programmaticStreamSerializationAllowed = 1;
    cfg->attrs = attrs;
    ++cfg->numAttrs;
}

// kernel<<<grid, block, smem, stream>>>(args...), early.  (A failure is left to cudaGetLastError, as by that syntax.)
template <typename... P, typename... A>
void launch(Start s, void (*kernel)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t st, A&&... args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid; cfg.blockDim = block; cfg.dynamicSmemBytes = smem; cfg.stream = st;
    cudaLaunchAttribute attr[1];
    start_early(&cfg, attr, s);
    (void)cudaLaunchKernelEx(&cfg, kernel, std::forward<A>(args)...);
}

}  // namespace ckpt

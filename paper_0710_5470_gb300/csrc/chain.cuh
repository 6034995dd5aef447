// Launches of kernels that follow one another on a stream, with the start of one
// under the end of the other (programmatic stream serialisation).
//
// A chained kernel's launch is processed while its predecessor runs; its CTAs start as
// soon as the predecessor's last CTA has left, and wait in chain_begin() until that
// kernel's writes are visible, where an ordinary launch begins only then.  Small steps
// are bound by this gap.  us per step on a GB300, ordinary -> chained launches: D2Q9
// 100^2 float64 forcing 7.52 -> 6.86, float32 3.03 -> 2.52, 512^2 float32 6.03 -> 5.16,
// 1024^2 fp16 equilibrium 12.6 -> 11.8; D3Q19 forcing in two passes 64^3 17.0 -> 13.7,
// 101 x 75 x 53 25.2 -> 23.5; 128^3 float32 equilibrium 74.0 -> 72.1, fp16 forcing
// 66.6 -> 65.1; a sweep of 24 fp16 lattices 41 -> 38.4.  Figures elsewhere that do not
// say so were taken with ordinary launches on both sides.
//
// The predecessor does not ask for the launch any earlier
// (griddepcontrol.launch_dependents): CTAs that come while it still runs take the
// slots that happen to be free and lie unevenly over the SMs: 64^3 as above 19.0 us,
// 512^2 float32 5.62, 128^3 float32 equilibrium 76.0.
#pragma once
#include <cuda_runtime.h>

namespace lbk {

// First statement of a kernel launched by launch_chained: nothing is read or written
// before it, and no thread leaves before it, so that a kernel that has ended has seen
// the end of every kernel before it.  Not for kernels with read-only loads (__ldg), which
// the compiler may move above it.
__device__ __forceinline__ void chain_begin() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

// Launches a kernel that begins with chain_begin().
template <class... P, class... A>
cudaError_t launch_chained(void (*kernel)(P...), dim3 grid, unsigned threads, size_t smem, cudaStream_t st, A&&... args) {
    cudaLaunchAttribute attr{};
    attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = grid;
    cfg.blockDim = dim3(threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cfg.attrs = &attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kernel, P(args)...);
}

}  // namespace lbk

// Instantiations of the marching float32 D3Q19 binary step (binary3d_march.cuh).
#include "binary3d_march.cuh"
#include "binary_launch.h"

namespace lbb {

namespace {

constexpr int TX3 = 32, TY3 = 8;
using Lay3 = LayoutMarch3<TX3, TY3>;
static_assert(Lay3::bytes(true) <= 48 * 1024, "fits without opting in to more shared memory");

using Kernel = void (*)(const March3Args);
Kernel kernel(bool forcing, int nx) {
    if (forcing) return nx % 2 == 0 ? binary_step_kernel3_march<true, TX3, TY3, true> : binary_step_kernel3_march<true, TX3, TY3, false>;
    return nx % 2 == 0 ? binary_step_kernel3_march<false, TX3, TY3, true> : binary_step_kernel3_march<false, TX3, TY3, false>;
}

}  // namespace

int binary_march3_ctas(bool forcing, int nx) {
    int occ = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, reinterpret_cast<const void*>(kernel(forcing, nx)), Lay3::NTH,
                                                      Lay3::bytes(forcing)) != cudaSuccess || occ < 1)
        occ = 1;
    cudaGetLastError();
    return occ;
}

cudaError_t binary_march3(bool forcing, const StepArgs<float>& a, const int4* work, int ctas, cudaStream_t st) {
    return lbk::launch_chained(kernel(forcing, a.nx), ctas, Lay3::NTH, Lay3::bytes(forcing), st, March3Args{a, work});
}

}  // namespace lbb

// First recorded index violation of this unit's kernels (checked builds; see bounds.cuh).
LB_BOUNDS_READER(lbk_bounds_b3march)

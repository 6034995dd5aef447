// Instantiations of the two-pass D3Q19 forcing step (step3d_fd.cuh).
#include <cstdlib>

#include "dispatch.h"
#include "step3d_fd.cuh"

using namespace lbk;

namespace {

template <class S, bool AOS, bool AL>
struct FDLaunch {
    static constexpr int TX = 32, TY = 8;
    using Lay = LayoutFD<TX, TY>;
    static_assert(Lay::BYTES <= 48 * 1024, "fits without opting in to more shared memory");
    static const void* fn() { return reinterpret_cast<const void*>(step_kernel3d_fd<S, TX, TY, 3, AOS, AL>); }
    static cudaError_t step(const StepArgs& a, dim3 grid, cudaStream_t st) {
        const unsigned pairs = (unsigned(a.nx) * unsigned(a.ny) * unsigned(a.nz) + 1u) / 2u;
        const cudaError_t e = launch_chained(density_pairs<S, AOS>, (pairs + 255u) / 256u, 256, 0, st, a, pairs);
        return e != cudaSuccess ? e
                                : launch_chained(step_kernel3d_fd<S, TX, TY, 3, AOS, AL>, grid, Lay::NTH, Lay::BYTES, st, a);
    }
    static LbKernelSet apply(LbKernelSet k, const char* name) {
        k.tx = TX;
        k.ty = TY;
        k.threads = Lay::NTH;
        k.smem = Lay::BYTES;
        k.step_fn = fn();
        k.step = &step;
        k.step_pair_needs_even_nx = false;
        k.name = name;
        k.aos = AOS;
        return k;
    }
};

template <class S>
LbKernelSet pick(int nx, LbKernelSet k) {
    if constexpr (PairIO<S>::RAW16)
        if (nx % AOS_SITES == 0) return FDLaunch<S, true, true>::apply(k, "pairs 32x8, density field, interleaved blocks");
    return nx % 2 == 0 ? FDLaunch<S, false, true>::apply(k, "pairs 32x8, density field")
                       : FDLaunch<S, false, false>::apply(k, "pairs 32x8, density field, site by site");
}

}  // namespace

// Whether a lattice runs the two-pass form (LB_D3_FIELD=0 / 1 forces it, for
// comparisons).  us per step on a GB300, fused -> two passes:
//   float32, even nx: the fused kernel holds two CTAs per SM (82 KB of shared
//     memory).  48^3 11.8 -> 12.5 (the second launch), 64^3 17.2 -> 15.9, 96^3
//     44.1 -> 35.1, 128^3 93.4 -> 82.6, 256^3 729 -> 675, 320^3 1347 -> 1294, 384^3
//     2342 -> 2409 (HBM);
//   odd nx: the fused form is the one-site tile kernel.  fp16 deviations 33 x 40 x
//     25 17.4 -> 16.3, 101 x 75 x 53 30.7 -> 26.3, 97 x 101 x 103 63.3 -> 51.0, 201 x
//     190 x 180 348 -> 347; float32 17.3 -> 14.4, 31.9 -> 25.2, 71.8 -> 55.1, 372 -> 385;
//   16-bit, even nx, one array per population: 24^3 12.9 -> 11.8, 100 x 76 x 54
//     25.3 -> 23.4, 200 x 190 x 180 252 -> 232;
//   16-bit, interleaved blocks: 64^3 16.1 -> 15.7, 96^3 34.0 -> 30.7, then even:
//     128^3 66.4 -> 66.8 (both buffers no longer fit the L2), 512^3 3570 -> 3585.
bool lbk_fd_wanted(int storage, int nx, size_t sites) {
    if (const char* e = std::getenv("LB_D3_FIELD")) return std::atoi(e) != 0;
    const double n = double(sites);
    if (nx % 2 != 0) return n <= (storage == 1 ? 4e6 : 7e6);
    if (storage == 1) return n >= 1.5e5 && n <= 4e7;
    return nx % AOS_SITES != 0 || n <= 1.6e6;
}

LbKernelSet lbk_fd_forcing(int storage, int nx, LbKernelSet k) {
    switch (storage) {
        case 2: return pick<StF16>(nx, k);
        case 3: return pick<StBF16>(nx, k);
        default: return pick<StF32>(nx, k);
    }
}

// First recorded index violation of this unit's kernels (checked builds; see bounds.cuh).
LB_BOUNDS_READER(lbk_bounds_d3fd)

// Instantiations of the two-pass D3Q19 forcing step (step3d_fd.cuh).
#include <cstdlib>

#include "dispatch.h"
#include "step3d_fd.cuh"

using namespace lbk;

namespace {

cudaError_t density(const StepArgs& a, cudaStream_t st, void (*kernel)(const StepArgs, unsigned)) {
    const unsigned pairs = (unsigned(a.nx) * unsigned(a.ny) * unsigned(a.nz) + 1u) / 2u;
    return launch_chained(kernel, (pairs + 255u) / 256u, 256, 0, st, a, pairs);
}

template <class S, bool AOS>
struct FDLaunch {
    static constexpr int TX = 32, TY = 8;
    using Lay = LayoutFD<TX, TY>;
    static_assert(Lay::BYTES <= 48 * 1024, "fits without opting in to more shared memory");
    static const void* fn() { return reinterpret_cast<const void*>(step_kernel3d_fd<S, TX, TY, 3, AOS>); }
    static cudaError_t step(const StepArgs& a, dim3 grid, cudaStream_t st) {
        const cudaError_t e = density(a, st, density_pairs<S, AOS, PairIO<S>::RAW16>);
        return e != cudaSuccess ? e
                                : launch_chained(step_kernel3d_fd<S, TX, TY, 3, AOS>, grid, Lay::NTH, Lay::BYTES, st, a);
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

// Odd nx: one site per thread.
template <class S>
struct FD1Launch {
    static constexpr int TX = 32, TY = 4, MINB = 4;
    static const void* fn() { return reinterpret_cast<const void*>(step_kernel3d_fd1<S, TX, TY, MINB>); }
    static cudaError_t step(const StepArgs& a, dim3 grid, cudaStream_t st) {
        const cudaError_t e = density(a, st, density_pairs<S, false, false>);
        return e != cudaSuccess ? e : launch_chained(step_kernel3d_fd1<S, TX, TY, MINB>, grid, TX * TY, 0, st, a);
    }
    static LbKernelSet apply(LbKernelSet k) {
        k.tx = TX;
        k.ty = TY;
        k.threads = TX * TY;
        k.smem = 0;
        k.step_fn = fn();
        k.step = &step;
        k.step_pair_needs_even_nx = false;
        k.name = "32x4, density field, one site per thread";
        k.aos = false;
        return k;
    }
};

template <class S>
LbKernelSet pick(int nx, LbKernelSet k) {
    if constexpr (PairIO<S>::RAW16)
        if (nx % AOS_SITES == 0) return FDLaunch<S, true>::apply(k, "pairs 32x8, density field, interleaved blocks");
    return nx % 2 == 0 ? FDLaunch<S, false>::apply(k, "pairs 32x8, density field") : FD1Launch<S>::apply(k);
}

}  // namespace

// Whether a lattice runs the two-pass form (LB_D3_FIELD=0 / 1 forces it, for
// comparisons).  us per step on a GB300, fused -> two passes:
//   odd nx: both forms take one site per thread; the fused one keeps a stash and two
//     CTAs per SM.  fp16 deviations 9 x 10 x 11 16.8 -> 8.4, 33 x 40 x 25 15.8 -> 8.1, 101 x
//     75 x 53 29.1 -> 20.6, 97 x 101 x 103 61.5 -> 44.7, 201 x 190 x 180 347 -> 262, 301 x 300 x
//     300 1143 -> 907, 481 x 480 x 480 4832 -> 3612; float32 16.2 -> 8.6, 15.9 -> 8.4, 30.7 ->
//     22.0, 70.6 -> 50.0, 370 -> 319, 1285 -> 1207, 5341 -> 5197: at every size, where the field can
//     be had;
//   float32, even nx: the fused kernel holds two CTAs per SM (82 KB of shared memory), the two
//     passes move 236 bytes per site and are bound by HBM where the lattice exceeds the L2.
//     Rows of whole 32-byte sectors (nx a multiple of 8) up to 4e7 sites: 16^3 9.5 -> 8.7, 64^3
//     15.8 -> 13.4, 128^3 92.2 -> 79.8, 200^3 370 -> 347, 256^3 728 -> 673, 320^3 1345 -> 1287, 336^3 1694 ->
//     1579; 384^3 2342 -> 2397; others up to 1e7: 130^3 107 -> 100, 190^3 286 -> 284, 210^3 414 -> 397,
//     220^3 438 -> 446, 250^3 660 -> 714, 310^3 1221 -> 1386.  Where the tiles' halo in x is the own tile
//     or the neighbour's (up to 32 and, full, to 64 columns) the fused kernel finds it in the L1: 24 x
//     200 x 200 41.1 -> 40.1, 24 x 300 x 300 82.2 -> 92.6, 32 x 120 x 120 18.8 -> 17.2, 32 x 200 x 200 44.1 ->
//     46.6, 32 x 600 x 600 330 -> 411 (1e6; up to 16 columns, half a tile, 3e6: 16 x 430 x 430 153 ->
//     151), 62 x 130 x 130 48.0 -> 41.7, 64 x 120 x 120 38.8 -> 34.5, 64 x 200 x 200 94.5 -> 99.0, 62 x 330 x 330
//     266 -> 276 (1.6e6), but 56 x 330 x 330 251 -> 244;
//   16-bit, even nx, one array per population: 24^3 11.3 -> 9.1, 100 x 76 x 54 23.9 -> 20.4, 200 x
//     190 x 180 251 -> 230, 300^3 924 -> 822, 500^3 4026 -> 3710; as above not from 1.6e6 sites on with 26
//     to 32 columns (30 x 200 x 200 38.7 -> 37.3, 30 x 300 x 300 76.5 -> 82.3; 24 x 430 x 430 151 -> 150) and 38
//     to 64 (56 x 130 x 130 37.8 -> 34.5, 52 x 330 x 330 190 -> 195; 34 x 430 x 430 309 -> 302);
//   16-bit, interleaved blocks: 32^3 10.3 -> 9.4, 64^3 15.1 -> 13.0, 96^3 32.9 -> 28.2,
//     then near even up to 3.4e6 sites: 128^3 65.2 -> 63.8 (both buffers no longer fit the L2), 160 x
//     160 x 128 99.3 -> 98.5; 128 x 220 x 220 177 -> 183, 512^3 3554 -> 3569; 32 and 64 columns as above
//     (64 x 120 x 120 31.0 -> 28.9, 64 x 200 x 200 71.9 -> 77.8, 32 x 300 x 300 75.1 -> 84.1).
bool lbk_fd_wanted(int storage, int nx, size_t sites) {
    if (const char* e = std::getenv("LB_D3_FIELD")) return std::atoi(e) != 0;
    const double n = double(sites);
    if (nx % 2 != 0) return true;
    if (storage == 1) {
        if (nx <= 32) return n <= (nx <= 16 ? 3e6 : 1e6);
        if (nx > 56 && nx <= 64) return n <= 1.6e6;
        return n <= (nx % 8 == 0 ? 4e7 : 1e7);
    }
    if ((nx > 24 && nx <= 32) || (nx > 36 && nx <= 64)) return n <= 1.6e6;
    return nx % AOS_SITES != 0 || n <= 3.4e6;
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

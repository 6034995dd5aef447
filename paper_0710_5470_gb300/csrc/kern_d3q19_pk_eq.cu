// Instantiations of the two-sites-per-thread D3Q19 equilibrium-scheme step
// (step3d_pk_eq.cuh).
#include <cstdlib>

#include "dispatch.h"
#include "step3d_pk_eq.cuh"

using namespace lbk;

namespace {

template <class S, int TX, int TY, int MINB, bool AOS, bool HPF = true>
struct PKELaunch {
    using Lay = LayoutPKE<TX, TY, PairIO<S>::RAW16>;
    static const void* fn() { return reinterpret_cast<const void*>(step_kernel3d_pk_eq<S, TX, TY, MINB, AOS, HPF>); }
    static cudaError_t step(const StepArgs& a, dim3 grid, cudaStream_t st) {
        static int attr_done = 0;
        if (!attr_done) {
            cudaError_t e = cudaFuncSetAttribute(fn(), cudaFuncAttributeMaxDynamicSharedMemorySize, int(Lay::BYTES));
            if (e != cudaSuccess) return e;
            attr_done = 1;
        }
        return launch_chained(step_kernel3d_pk_eq<S, TX, TY, MINB, AOS, HPF>, grid, Lay::NTH, Lay::BYTES, st, a);
    }
    static void apply(LbKernelSet& k, const char* name) {
        k.tx = TX;
        k.ty = TY;
        k.threads = Lay::NTH;
        k.smem = Lay::BYTES;
        k.step_fn = fn();
        k.step = &step;
        k.step_pair_needs_even_nx = true;
        k.name = name;
        k.aos = AOS;
    }
};

}  // namespace

bool lbk_wide(int nx, int ny, int ty) {
    if (const char* e = std::getenv("LB_WIDE")) return std::atoi(e) != 0;
    const auto pad = [](long long n, int t) { return (n + t - 1) / t * t; };
    return double(pad(nx, 64)) * double(pad(ny, ty)) <= 1.2 * double(pad(nx, 32)) * double(pad(ny, 8));
}

// The pair kernel of the equilibrium scheme (step3d_pk_eq.cuh) for 32-bit
// arithmetic storage in place of `step` of `base` (an even nx is required;
// base.step1 stays the fallback; measured on GB300 at 128^3 / 512^3: fp16
// deviations 43.5 / 50.2 GLUPS against 37.7 / 43.1 for the tile kernel,
// float32 28.7 / 29.8 against 28.0 / 28.6).  LB_D3_VARIANT=0 keeps the tile kernel.
// Tiles of 64 x 4 sites where lbk_wide() allows, us per step, 32 x 8 -> 64 x 4: fp16
// deviations 64^3 9.7 -> 9.1, 100 x 76 x 54 15.4 -> 13.1, 128^3 48.0 -> 42.6, 256^3 361 -> 322
// (96^3, not allowed: 22.4 -> 24.5).  In float32 the halo's populations are loaded when
// they are summed and not a plane ahead, which leaves registers for three CTAs per SM
// instead of two: 100 x 76 x 54 17.5 -> 15.6, 128^3 72.2 -> 63.2 (5.0 TB/s), 256^3 559 -> 482
// (with the halo a plane ahead, two CTAs: 66.2 and 483); from 2.5e5 sites on, since a
// small lattice waits for those loads (48^3 7.2 -> 8.3, 64^3 10.2 -> 10.1).
LbKernelSet lbk_pk_equilibrium(int storage, int nx, int ny, int nz, LbKernelSet k) {
    const char* env = std::getenv("LB_D3_VARIANT");
    const int v = env ? std::atoi(env) : -1;
    if (v == 0) return k;
    const bool aos = nx % AOS_SITES == 0;
    const bool wide = nx % 2 == 0 && lbk_wide(nx, ny, 4) && (storage != 1 || double(nx) * ny * nz >= 2.5e5 || std::getenv("LB_WIDE"));
    if (wide) {
        if (storage == 2) {
            if (aos) PKELaunch<StF16, 64, 4, 3, true>::apply(k, "pairs 64x4, equilibrium, interleaved blocks");
            else PKELaunch<StF16, 64, 4, 3, false>::apply(k, "pairs 64x4, equilibrium");
        } else if (storage == 3) {
            if (aos) PKELaunch<StBF16, 64, 4, 3, true>::apply(k, "pairs 64x4, equilibrium, interleaved blocks");
            else PKELaunch<StBF16, 64, 4, 3, false>::apply(k, "pairs 64x4, equilibrium");
        } else if (storage == 1) {
            PKELaunch<StF32, 64, 4, 3, false, false>::apply(k, "pairs 64x4, equilibrium");
        }
        return k;
    }
    if (storage == 2) {
        if (aos) PKELaunch<StF16, 32, 8, 3, true>::apply(k, "pairs 32x8, equilibrium, interleaved blocks");
        else PKELaunch<StF16, 32, 8, 3, false>::apply(k, "pairs 32x8, equilibrium");
    } else if (storage == 3) {
        if (aos) PKELaunch<StBF16, 32, 8, 3, true>::apply(k, "pairs 32x8, equilibrium, interleaved blocks");
        else PKELaunch<StBF16, 32, 8, 3, false>::apply(k, "pairs 32x8, equilibrium");
    } else if (storage == 1) {
        PKELaunch<StF32, 32, 8, 2, false>::apply(k, "pairs 32x8, equilibrium");
    }
    return k;
}

// First recorded index violation of this unit's kernels (checked builds; see bounds.cuh).
LB_BOUNDS_READER(lbk_bounds_d3pke)

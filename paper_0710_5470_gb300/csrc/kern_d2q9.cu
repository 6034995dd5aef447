// Kernel instantiations for the D2Q9 lattice.
#include "kernels_impl.cuh"

using namespace lbk;

// The float64 step on another tile than the 32 x 8 of Launchers.
template <bool F, int TX, int TY, int NTH>
static LbKernelSet f64_tile(LbKernelSet k) {
    using Lay = Layout64<F, TX, TY, NTH>;
    static_assert(Lay::BYTES <= 48 * 1024, "fits without opting in to more shared memory");
    k.tx = TX;
    k.ty = TY;
    k.threads = NTH;
    k.smem = Lay::BYTES;
    k.step_fn = reinterpret_cast<const void*>(step_kernel2d_f64<F, TX, TY, NTH>);
    k.step = [](const StepArgs& a, dim3 grid, cudaStream_t st) -> cudaError_t {
        return launch_chained(step_kernel2d_f64<F, TX, TY, NTH>, grid, NTH, Lay::BYTES, st, tile2d_args(a),
                              consts64(a.a, a.b, a.T, a.kappa, a.omega, a.nu));
    };
    return k;
}

// Tiles of the float64 step by the sites an SM gets.  A small lattice leaves
// SMs and schedulers idle with 32 x 8 tiles (100^2: 52 CTAs on 152 SMs), and a
// warp's own chain of float64 instructions is what a step takes, so small tiles
// win until their halo (8 x 4, forcing: 3 densities and 1.9 gradients per site)
// costs more than the idle pipes.  us per step on a GB300, forcing scheme,
// 8 x 4 / 8 x 8 / 32 x 8: 100^2 7.5 / 8.9 / 13.2, 160^2 12.0 / 12.0 / 13.2, 200^2
// 17.4 / 17.5 / 23.3, 256^2 26.5 / 23.4 / 23.3, 400^2 55.5 / 52.7 / 55.3, 512^2 86.9 /
// 84.3 / 76.4; equilibrium scheme (one halo row less), 8 x 4 / 32 x 8: 100^2 6.5 /
// 11.1, 200^2 13.5 / 19.4, 400^2 41.6 / 45.3, 512^2 64.5 / 62.5.
template <bool F>
static LbKernelSet pick_f64(int nx, int ny, int sms) {
    const LbKernelSet k = Launchers<D2Q9, F, StF64, 32, 8>::make();
    const double per_sm = double(nx) * ny / (sms > 0 ? sms : 1);
    if constexpr (F) {
        if (per_sm <= 215) return f64_tile<F, 8, 4, 128>(k);
        if (per_sm <= 1300) return f64_tile<F, 8, 8, 64>(k);
    } else {
        if (per_sm <= 1300) return f64_tile<F, 8, 4, 64>(k);
    }
    return k;
}

template <bool F>
static LbKernelSet pick(int storage, int nx, int ny, int sms) {
    switch (storage) {
        case 0: return pick_f64<F>(nx, ny, sms);
        case 1: return Launchers<D2Q9, F, StF32, 32, 8>::make();
        case 2: return Launchers<D2Q9, F, StF16, 32, 8>::make();
        case 3: return Launchers<D2Q9, F, StBF16, 32, 8>::make();
    }
    return LbKernelSet{};
}

LbKernelSet lbk_pk2d(int scheme, int storage, LbKernelSet k, int nx, int ny, int sms);

LbKernelSet lbk_kernels_d2q9(int scheme, int storage, int nx, int ny, int sms) {
    return lbk_pk2d(scheme, storage, scheme == 1 ? pick<true>(storage, nx, ny, sms) : pick<false>(storage, nx, ny, sms),
                    nx, ny, sms);
}

// First recorded index violation of this unit's kernels (checked builds; see bounds.cuh).
LB_BOUNDS_READER(lbk_bounds_d2q9)

// Instantiations of the two-sites-per-thread D3Q19 equilibrium-scheme step
// (step3d_pk_eq.cuh).
#include <algorithm>
#include <cstdlib>
#include <vector>

#include "../../include/lb.h"
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

// Estimated time of a step with tiles of tx x ty sites and occ resident CTAs per SM: the work
// list in waves of resident CTAs, each as long as its longest chunk and three planes of halo,
// filling and draining, a plane taking c0 + the SM's CTAs.
double waves(int sms, int occ, double c0, int nx, int ny, int nz, int tx, int ty) {
    int n = 0;
    if (lb_work_list(sms, occ, nx, ny, nz, tx, ty, nullptr, 0, &n) != LB_OK) return 0.0;
    std::vector<int> list;
    try {
        list.resize(4 * size_t(n));
    } catch (...) {
        return 0.0;
    }
    lb_work_list(sms, occ, nx, ny, nz, tx, ty, list.data(), n, &n);
    double t = 0.0;
    for (long long k = 0; k < n; k += (long long)sms * occ) {
        const long long ctas = std::min<long long>(n - k, (long long)sms * occ);
        t += (list[4 * k + 3] - list[4 * k + 2] + 3) * (c0 + double((ctas + sms - 1) / sms));
    }
    return t;
}

// Whether the pair kernel takes tiles of 64 x 4 sites in place of 32 x 8 (LB_WIDE=0 / 1
// forces it, for comparisons).  A warp of a 64-wide tile stores whole rows, and a row pushed
// one site aside touches one more sector per 64 sites instead of one per 32: a tenth less
// time where the work list is the same.  Against that stand its overhang over the lattice and
// longer waves (E: ratio of the estimates).  Measured at 151 (16-bit) and 122 (float32) lattices; us
// per step, 32 x 8 -> 64 x 4:
//   16-bit: E up to 1.1, for lattices of less than a tile's eight rows up to 0.95, and more than
//     32 columns (a warp's width).  128^3 (E 1) 47.8 -> 42.5, 100 x 76 x 54 15.3 -> 12.9, 224^3 257 ->
//     235, 288^3 505 -> 472, 512^3 2674 -> 2393, 512 x 4 x 256 (0.62) 17.7 -> 12.9; 288 x 200 x 100 (1.30)
//     120 -> 129, 160^3 88.9 -> 94.4, 144^3 74.6 -> 80.0, 138 x 158 x 13 10.6 -> 12.6, 200 x 5 x 84 (1.5)
//     6.5 -> 8.5, 510 x 6 x 177 (1.0) 16.1 -> 17.0, 32 x 4 x 4096 16.3 -> 18.8;
//   float32 (three CTAs per SM instead of two, for which the halo's loads come late: small
//     lattices, one CTA per SM either way, wait for them): E up to 0.95, of less than eight rows
//     0.9, of an overhang more than 1.15 times as large 0.85; from 1.3e6 sites on up to 1.0 with an
//     overhang up to 1.2 times.  128^3 71.9 -> 63.0, 144^3 (0.96) 114 -> 105, 288^3 830 -> 739, 146 x 246 x
//     39 (0.69) 74.8 -> 52.8, 224 x 176 x 12 24.9 -> 16.8; 48^3 (1.0) 7.0 -> 8.0, 64^3 (1.0) 10.1 -> 9.9,
//     160^3 (1.25) 137 -> 144, 138 x 158 x 13 11.7 -> 15.1, 160 x 25 x 68 11.6 -> 13.8, 138 x 97 x 48 (0.92,
//     overhang 1.154) 24.0 -> 25.2, 510 x 6 x 177 (0.96) 17.6 -> 20.5.
bool wide_tiles(int storage, int nx, int ny, int nz, int sms) {
    if (nx % 2 != 0) return false;
    if (const char* e = std::getenv("LB_WIDE")) return std::atoi(e) != 0;
    const bool f32 = storage == 1;
    if (!f32 && nx <= 32) return false;
    const double c0 = f32 ? 2.0 : 1.0;
    const double E = waves(sms, 3, c0, nx, ny, nz, 64, 4) / waves(sms, f32 ? 2 : 3, c0, nx, ny, nz, 32, 8);
    if (!f32) return E <= (ny < 8 ? 0.95 : 1.1);
    const auto pad = [](int n, int t) { return double((n + t - 1) / t) * t; };
    const double overhang = pad(nx, 64) * pad(ny, 4) / (pad(nx, 32) * pad(ny, 8));
    if (double(nx) * ny * nz >= 1.3e6 && overhang <= 1.2) return E <= 1.0;
    return E <= (overhang > 1.15 ? 0.85 : (ny < 8 ? 0.9 : 0.95));
}

}  // namespace

// The pair kernel of the equilibrium scheme (step3d_pk_eq.cuh) for 32-bit
// arithmetic storage in place of `step` of `base` (an even nx is required;
// base.step1 stays the fallback; measured on GB300 at 128^3 / 512^3: fp16
// deviations 43.5 / 50.2 GLUPS against 37.7 / 43.1 for the tile kernel,
// float32 28.7 / 29.8 against 28.0 / 28.6).  LB_D3_VARIANT=0 keeps the tile kernel.
// Tiles of 64 x 4 sites where wide_tiles() says so.  In float32 the halo's populations are
// then loaded when they are summed and not a plane ahead, which leaves registers for three
// CTAs per SM instead of two: 100 x 76 x 54 17.4 -> 15.6 us, 128^3 71.9 -> 63.0 (5.0 TB/s), 256^3 559
// -> 482 (with the halo a plane ahead, two CTAs: 66.2 and 483).
LbKernelSet lbk_pk_equilibrium(int storage, int nx, int ny, int nz, int sms, LbKernelSet k) {
    const char* env = std::getenv("LB_D3_VARIANT");
    const int v = env ? std::atoi(env) : -1;
    if (v == 0) return k;
    const bool aos = nx % AOS_SITES == 0;
    if (wide_tiles(storage, nx, ny, nz, sms)) {
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

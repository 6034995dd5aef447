// Float64 D3Q19 step in passes (step3d_f64.cuh): workspace, slabs and launches.
#include <algorithm>
#include <cstdlib>

#include "dispatch.h"
#include "step3d_f64.cuh"

using namespace lbk;

namespace {

constexpr int THREADS = THREADS64;
constexpr size_t WORKSPACE_LIMIT = size_t(1) << 30;
constexpr int MIN_SLAB = 8;   // fewer planes than this would recompute too many halo planes

int fields(bool forcing) { return forcing ? 11 : 1; }   // float64 fields of the workspace
int halo(bool forcing) { return forcing ? 2 : 1; }

template <class K>
cudaError_t run(K kernel, Args64x3 a, int first, int planes, cudaStream_t st) {
    a.first = first;
    a.planes = planes;
    const unsigned n = unsigned(a.nx) * unsigned(a.ny) * unsigned(planes);
    return launch_chained(kernel, (n + THREADS - 1) / THREADS, THREADS, 0, st, a);
}

template <bool F>
cudaError_t step(const StepArgs& s, dim3, cudaStream_t st) {
    Args64x3 a{};
    a.src = reinterpret_cast<const double*>(s.src_base);
    a.dst = reinterpret_cast<double*>(s.dst_base);
    a.pitch = s.pitch;
    a.nx = s.nx;
    a.ny = s.ny;
    a.nz = s.nz;
    a.status = s.status;
    a.k = Consts64x3{s.a, s.b, s.T, s.omega, 1.0 - s.omega, s.omega * s.nu / 12.0, s.omega * s.nu / 4.0,
                     s.omega * s.a * s.nu / 2.0, s.kappa / 6.0,
                     s.kappa / 1728.0, s.omega * s.kappa / 144.0};
    const bool whole = s.lz >= s.nz;
    const int H = whole ? 0 : halo(F);
    a.halo = H;
    a.wrap_planes = whole ? s.nz : 0;
    a.field = (long long)s.nx * s.ny * (whole ? s.nz : s.lz + 2 * H);
    a.rho = s.work64;
    a.G = s.work64 + a.field;
    a.M = s.work64 + 5 * a.field;
    for (int z0 = 0; z0 < s.nz; z0 += s.lz) {
        const int n = std::min(s.lz, s.nz - z0);
        a.z0 = z0;
        cudaError_t e = run(density3_f64, a, -H, n + 2 * H, st);
        if (F && e == cudaSuccess) e = run(mprime3_f64, a, whole ? 0 : -1, whole ? n : n + 2, st);
        if (e == cudaSuccess) e = run(collide3_f64<F>, a, 0, n, st);
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

}  // namespace

// LB_F64_SLAB=n: slabs of n planes (0: the fused kernel), for comparisons.
int lbk_f64_slab(int scheme, int nx, int ny, int nz, size_t* bytes) {
    const bool f = scheme == 1;
    const size_t plane = size_t(nx) * ny * fields(f) * sizeof(double);
    int slab = nz;
    if (const char* e = std::getenv("LB_F64_SLAB")) {
        slab = std::min(nz, std::max(0, std::atoi(e)));
    } else if (plane * nz > WORKSPACE_LIMIT) {
        slab = int(std::min<size_t>(nz, WORKSPACE_LIMIT / plane)) - 2 * halo(f);
        if (slab < MIN_SLAB) return 0;
    }
    *bytes = plane * (slab >= nz ? nz : slab + 2 * halo(f));
    return slab;
}

LbKernelSet lbk_f64_passes(int scheme, LbKernelSet k) {
    k.tx = THREADS;
    k.ty = 1;
    k.threads = THREADS;
    k.smem = 0;
    k.name = scheme == 1 ? "three passes, one site per thread" : "two passes, one site per thread";
    k.step_fn = scheme == 1 ? reinterpret_cast<const void*>(collide3_f64<true>)
                            : reinterpret_cast<const void*>(collide3_f64<false>);
    k.step = scheme == 1 ? &step<true> : &step<false>;
    k.step_pair_needs_even_nx = false;
    return k;
}

// First recorded index violation of this unit's kernels (checked builds; see bounds.cuh).
LB_BOUNDS_READER(lbk_bounds_d3f64)

// Instantiations of the two-sites-per-thread D2Q9 step (step2d_pk.cuh) for
// single lattices.
#include <algorithm>
#include <cstdlib>

#include "dispatch.h"
#include "step2d_march.cuh"

using namespace lbk;

namespace {

template <bool F, class S, int TX, int TY>
struct PK2Launch {
    using Lay = Layout2PK<F, TX, TY, PairIO<S>::RAW16 ? 3 : 2>;
    static const void* fn() { return reinterpret_cast<const void*>(step_kernel2d_pk<F, S, TX, TY>); }
    static cudaError_t step(const StepArgs& a, dim3 grid, cudaStream_t st) {
        static int attr_done = 0;
        if (!attr_done) {
            cudaError_t e = cudaFuncSetAttribute(fn(), cudaFuncAttributeMaxDynamicSharedMemorySize, int(Lay::BYTES));
            if (e != cudaSuccess) return e;
            attr_done = 1;
        }
        Tile2DArgs t{a.src_base, a.dst_base, a.pitch, a.nx, a.ny, a.pair2d, a.a, a.b, a.T, a.kappa, a.omega,
                     a.nu, a.fa, a.fb, a.fT, a.fkappa, a.fomega, a.fnu, a.pref, a.rsum, a.status};
        return launch_chained(step_kernel2d_pk<F, S, TX, TY>, grid, Lay::NTH, Lay::BYTES, st, t);
    }
    static void apply(LbKernelSet& k, const char* name) {
        k.tx = TX;
        k.ty = TY;
        k.threads = Lay::NTH;
        k.smem = Lay::BYTES;
        k.step_fn = fn();
        k.step = &step;
        k.step_pair_needs_even_nx = false;   // odd nx: every site of a pair loaded on its own
        k.name = name;
    }
};

// The marching form (step2d_march.cuh): equilibrium scheme, 16-bit storage, even nx.
template <class S>
struct MarchLaunch {
    static const void* fn() { return reinterpret_cast<const void*>(step_kernel2d_march<S>); }
    static cudaError_t step(const StepArgs& a, dim3 grid, cudaStream_t st) {   // a.lz: rows of a chunk
        Tile2DArgs t{a.src_base, a.dst_base, a.pitch, a.nx, a.ny, a.pair2d, a.a, a.b, a.T, a.kappa, a.omega,
                     a.nu, a.fa, a.fb, a.fT, a.fkappa, a.fomega, a.fnu, a.pref, a.rsum, a.status};
        const int strips = (a.nx + MARCH_COLS - 1) / MARCH_COLS, chunks = (a.ny + a.lz - 1) / a.lz;
        return launch_chained(step_kernel2d_march<S>, grid, 32 * MARCH_WARPS, 0, st, t, strips, a.lz, strips * chunks);
    }
    static LbKernelSet make(LbKernelSet k, int rows) {
        k.tx = MARCH_COLS;
        k.ty = rows;
        k.threads = 32 * MARCH_WARPS;
        k.smem = 0;
        k.step_fn = fn();
        k.step = &step;
        k.march_warps = MARCH_WARPS;
        k.name = "pairs, marching strips of 60 columns, mixed adds";
        return k;
    }
};

template <bool F>
LbKernelSet pick(int storage, LbKernelSet k) {
    switch (storage) {
        case 1: PK2Launch<F, StF32, 32, 8>::apply(k, "pairs 32x8"); break;
        case 2: PK2Launch<F, StF16, 32, 8>::apply(k, "pairs 32x8, mixed adds"); break;
        case 3: PK2Launch<F, StBF16, 32, 8>::apply(k, "pairs 32x8, mixed adds"); break;
        default: break;
    }
    return k;
}

}  // namespace

// Rows of a marching warp's chunk, 0: the lattice keeps the tiles (LB_D2_ROWS=n
// forces n, for comparisons).  A warp passes through rows + 2 rows and about two more in
// filling and draining, each in a time of 1.2 + its SM's CTAs, of which four are
// resident (12 rows: 12.4 us with up to three per SM, 15.3 with four; 14 rows 14.0 and
// 17.4); the rows with the least time over all waves are taken: 2048^2 30 rows (one wave of
// 604 CTAs) 37.6 us, 28 rows (two waves) 46.2, 32 rows 39.5, 40 rows 39.4.  From 7,200 sites
// per SM on, where a wave of a dozen rows and more fills the chip, tiles -> strips, chained
// launches: 1100^2 13.8 -> 12.5, 1200 x 1100 14.6 -> 13.3, 700 x 2000 15.7 -> 14.1, 3000 x 400
// 13.4 -> 12.4, 1500 x 1400 22.4 -> 18.6; 1024^2 (6,900 per SM) 11.8 -> 12.4, 800^2 8.1 -> 9.5.
// Not where the strips overhang the lattice by a fifth more than tiles of 32 columns do; at
// 4.2e6 sites, by the columns and the ratio of the overhangs: 62 (1.88) 43.4 -> 65.6, 64 (1.88) 41.7
// -> 63.3, 128 (1.41) 43.3 -> 49.0, 192 (1.25) 44.0 -> 44.0, 96 (1.25) 42.6 -> 44.1, 250 (1.17)
// 46.0 -> 42.7, 160 (1.13) 43.5 -> 40.5, 120 (0.94) 46.2 -> 36.8.  Nor where the least time of the
// strips (0.184 us a unit below 2e6 sites) is above what tiles take, 0.75 us and 1.55 ns for each
// site of theirs per SM: 40000 x 30 13.7 -> 14.7, 80000 x 15 13.8 -> 14.7; 100000 x 12 15.8 -> 12.3,
// 60000 x 20 14.7 -> 14.4, 20000 x 64 13.9 -> 13.1.  Tiles have no launch for more than 65535 of
// their rows: such a lattice keeps the strips.
int march_rows(int nx, int ny, int sms) {
    if (const char* e = std::getenv("LB_D2_ROWS")) return std::min(ny, std::max(0, std::atoi(e)));
    if (nx % 2 != 0 || double(nx) * ny < 7.2e3 * sms) return 0;
    const long long strips = (nx + MARCH_COLS - 1) / MARCH_COLS;
    const double tile_x = 32.0 * ((nx + 31) / 32), tile_y = 8.0 * ((ny + 7) / 8);
    const bool tiles = tile_y <= 8.0 * 65535;
    if (tiles && double(strips * MARCH_COLS) > 1.2 * tile_x) return 0;
    int best = 0;
    double cost = 0;
    for (int r = 12; r <= 64 && r <= ny; ++r) {
        const long long ctas = (strips * ((ny + r - 1) / r) + MARCH_WARPS - 1) / MARCH_WARPS, last = ctas % (4LL * sms);
        const double c = (r + 4) * (5.2 * double(ctas / (4LL * sms)) + (last ? 1.2 + double((last + sms - 1) / sms) : 0.0));
        if (best == 0 || c < cost) {
            best = r;
            cost = c;
        }
    }
    return tiles && 0.184 * cost > 0.75 + 1.55e-3 * tile_x * tile_y / sms ? 0 : best;
}

// The pair kernel for D2Q9 with 32-bit arithmetic (storage 1, 2, 3) in place
// of `step` of `base` (float64 keeps the tile kernel: its arithmetic bounds
// it).  LB_D2_VARIANT=0 keeps the tile kernel for comparisons.
LbKernelSet lbk_pk2d(int scheme, int storage, LbKernelSet k, int nx, int ny, int sms) {
    const char* env = std::getenv("LB_D2_VARIANT");
    if (env && std::atoi(env) == 0) return k;
    if (scheme != 1 && (storage == 2 || storage == 3) && nx % 2 == 0 && !std::getenv("LB_NO_PAIR")) {
        const int rows = march_rows(nx, ny, sms);
        if (rows > 0) return storage == 2 ? MarchLaunch<StF16>::make(k, rows) : MarchLaunch<StBF16>::make(k, rows);
    }
    return scheme == 1 ? pick<true>(storage, k) : pick<false>(storage, k);
}

// First recorded index violation of this unit's kernels (checked builds; see bounds.cuh).
LB_BOUNDS_READER(lbk_bounds_d2pk)

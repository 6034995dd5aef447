// D2Q9 equilibrium-scheme time step in 16-bit storage: a warp marches up a strip
// of columns.
//
// The same step as step2d_pair_tile (step2d_pk.cuh), with its arithmetic and bits.  A
// warp holds 64 adjacent columns, one aligned pair of sites per lane (even nx), and
// moves through a chunk of rows.  Per row it sums its pairs' densities and takes the
// x neighbours from the adjacent lanes by shuffles; the rows of the stencils (Eq. 32)
// and a row's raw populations until its collision, one row later, stay in registers.
// The first and the last lane are halo: lanes 1..30 collide and push 60 columns.
//
// A tile of 32 x 8 sites sums the densities of 1.41 sites per site and waits at its
// barrier for one wave of loads; a strip sums 64/60 x (rows + 2)/rows of them, has no
// barrier and no shared memory, and has the loads of two rows in flight while it works
// on a third: 197 instructions per site against about 330.  A row takes a warp half a
// microsecond however few there are, so the form is for lattices that fill the chip
// with chunks of a dozen rows and more (march_rows in kern_d2q9_pk.cu).  Measured on
// a GB300, us per step, tiles -> strips, fp16 deviations: 2048^2 44.4 -> 37.6 (4.5 TB/s),
// 4096^2 164.4 -> 137.6 (4.9 TB/s), 1500 x 1400 22.4 -> 18.6, 600 x 5000 32.6 -> 27.0; 1024^2
// 11.8 -> 12.4 (chained launches).  Rows in flight 1 / 2 / 3 at 2048^2 and 32 rows: 41.3 / 40.5 / 50 (168
// registers).
#pragma once
#include "chain.cuh"
#include "step2d_pk.cuh"

namespace lbk {

constexpr int MARCH_COLS = 60;    // columns a warp collides
constexpr int MARCH_WARPS = 4;    // warps per CTA, four CTAs per SM
constexpr int MARCH_AHEAD = 2;    // rows in flight

// Neighbours of a row held as one pair per lane: the values at x - 1 and at x + 1 of both sites.
__device__ __forceinline__ void row_neighbours(P2 c, P2& xm, P2& xp) {
    const float l = __shfl_up_sync(0xffffffffu, c.v.y, 1), r = __shfl_down_sync(0xffffffffu, c.v.x, 1);
    xm = pp(l, c.v.x);
    xp = pp(c.v.y, r);
}

// One step of the sites [x0, x0 + 60) x [y0, y1) of a lattice with an even nx, by one warp.
template <class S>
__device__ __forceinline__ void step2d_march(const Tile2DArgs& args, int x0, int y0, int y1) {
    using L = D2Q9;
    using IO = PairIO<S>;
    static_assert(IO::RAW16, "16-bit storage");
    constexpr int NR = 2 + MARCH_AHEAD;    // rows held: the one collided, the newest, those in flight
    const int nx = args.nx, ny = args.ny;
#ifdef LB_DEBUG_BOUNDS
    const unsigned nsites = unsigned(nx) * unsigned(ny);
#endif
    const int lane = threadIdx.x % 32;
    const PairPhys ph{args.fa, args.fb, args.fT, args.fkappa, args.fomega, args.fnu, args.pref, args.rsum};
    const char* src = args.src;
    char* dst = args.dst;
    const long long pitch = args.pitch;
    const int xo = x0 - 2 + 2 * lane;      // column of the pair's site 0
    const bool own = lane >= 1 && lane <= 30 && xo < nx;
    const unsigned xc = unsigned(wrap_near(xo, nx)), xm1 = unsigned(wrap_near(xo - 1, nx)),
                   xp2 = unsigned(wrap_near(xo + 2, nx));

    struct Row {
        float2 f0;
        unsigned w[8];
    } raw[NR];
    auto load = [&](Row& r, unsigned row) {   // row: site index of the lattice row's first site
        const unsigned q = row + xc;
        LB_GUARD(q + 1 < nsites, BK_2D_LOAD, q, r.f0 = make_float2(0.f, 0.f); for (int i = 0; i < 8; ++i) r.w[i] = 0u; return)
        r.f0 = reinterpret_cast<const float2*>(src)[q >> 1];
        static_for<1, 9>([&](auto I) {
            constexpr int i = decltype(I)::value;
            r.w[i - 1] = IO::ld(src + S::pop_offset(i, pitch), q);
        });
    };

    const P2 third = pp(1.0f / 3.0f), twelfth = pp(1.0f / 12.0f);
    const unsigned unx = unsigned(nx), area = unx * unsigned(ny);
    // first sites of the row loaded next and of the row collided next
    unsigned lrow = unsigned(wrap_near(y0 - 1, ny)) * unx, crow = unsigned(y0) * unx;
    auto up = [&](unsigned row) { return row + unx == area ? 0u : row + unx; };
    auto down = [&](unsigned row) { return row == 0u ? area - unx : row - unx; };
    const int nrows = y1 - y0 + 2;         // rows passed through
#pragma unroll
    for (int k = 0; k < MARCH_AHEAD; ++k) {
        if (k < nrows) load(raw[k], lrow);
        lrow = up(lrow);
    }
    // density and its x difference and sum, one and two rows back
    P2 c1 = pp(0.f), d1 = c1, s1 = c1, c2 = c1, d2 = c1, s2 = c1;
    for (int k = 0;;) {
#pragma unroll
        for (int m = 0; m < NR; ++m, ++k) {
            // row k of the march is in raw[k % NR]
            if (k + MARCH_AHEAD < nrows) {
                load(raw[(m + MARCH_AHEAD) % NR], lrow);
                lrow = up(lrow);
            }
            const P2 c = pair_rho9<S>(raw[m].f0, raw[m].w, ph.rsum);
            P2 xm, xp;
            row_neighbours(c, xm, xp);
            const P2 d = xp - xm, s = xp + xm;
            if (k >= 2) {
                // gradient and Laplacian of row k - 1 (Eq. 32), the sums of pair_stencil9
                const P2 G[2] = {fma(third, d1, twelfth * (d + d2)), fma(third, c - c2, twelfth * (s - s2))};
                const P2 lap = pp(2.0f) * (fma(third, s1 + (c + c2), twelfth * (s + s2)) - pp(5.0f / 3.0f) * c1);
                const Row& old = raw[(m + NR - 1) % NR];
                P2 j[2];
                pair_momentum9<S>(old.w, j);
                if (own && (!(c1.v.x > 0.f) || !(c1.v.x < 1e30f) || !(c1.v.y > 0.f) || !(c1.v.y < 1e30f)))
                    atomicOr(args.status, 1u);
                PairColl2D<false> K;
                const P2 none[2] = {pp(0.f), pp(0.f)};
                K.prep(c1, j, G, lap, none, ph);
                const unsigned yr[3] = {down(crow), crow, up(crow)};
                if (own) {
                    LB_GUARD(crow + xc + 1 < nsites, BK_2D_STORE, crow + xc, return)
                    reinterpret_cast<float2*>(dst)[(crow + xc) >> 1] = fma(K.omw, P2{old.f0}, K.c0).v;
                    auto store = [&](auto I, P2 v) {
                        constexpr int i = decltype(I)::value;
                        constexpr int ex = L::ex(i), ey = L::ey(i);
                        char* p = dst + S::pop_offset(i, pitch);
                        const unsigned row = yr[1 + ey];
                        LB_GUARD(row + xm1 < nsites && row + xp2 < nsites, BK_2D_STORE, row, return)
                        if constexpr (ex == 0) {
                            IO::st2(p, row + xc, v);
                        } else {
                            IO::st1(p, row + (ex > 0 ? xc + 1 : xm1), v.v.x);
                            IO::st1(p, row + (ex > 0 ? xp2 : xc), v.v.y);
                        }
                    };
                    static_for<1, 9>([&](auto I) {
                        constexpr int i = decltype(I)::value;
                        constexpr int o = opposite<L>(i);
                        if constexpr (i < o) {
                            P2 oi, on;
                            K.template out<i>(IO::dec(old.w[i - 1]), IO::dec(old.w[o - 1]), oi, on);
                            store(std::integral_constant<int, i>{}, oi);
                            store(std::integral_constant<int, o>{}, on);
                        }
                    });
                }
                crow = yr[2];
            }
            c2 = c1;
            d2 = d1;
            s2 = s1;
            c1 = c;
            d1 = d;
            s1 = s;
            if (k + 1 == nrows) return;
        }
    }
}

// One step of a single D2Q9 lattice: a warp per (strip, chunk of `rows` rows), the strips side by side.
template <class S>
__global__ void __launch_bounds__(32 * MARCH_WARPS, 4) step_kernel2d_march(const Tile2DArgs args, int strips, int rows,
                                                                          int items) {
    chain_begin();
    const int item = blockIdx.x * MARCH_WARPS + threadIdx.x / 32;
    if (item >= items) return;
    const int x0 = (item % strips) * MARCH_COLS, y0 = (item / strips) * rows;
    step2d_march<S>(args, x0, y0, min(y0 + rows, args.ny));
}

}  // namespace lbk

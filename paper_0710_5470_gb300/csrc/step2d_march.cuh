// D2Q9 time step of 32-bit arithmetic: a warp marches up a strip of columns.
//
// The same step as step2d_tile (step_kernel.cuh) on the arithmetic of
// step2d_pk.cuh.  A warp holds 64 adjacent columns, one pair of sites per lane,
// and moves through a chunk of rows.  Per row it loads its pairs, sums their
// densities and takes the x neighbours from the adjacent lanes by shuffles; the
// rows of the stencils (Eq. 32) and, in the forcing scheme, of div M' (Eq. 28)
// are carried in registers from one row to the next, as is the row's raw
// populations until its collision (one row later, two in the forcing scheme).
// The first and the last lane are halo: lanes 1..30 collide and push 60
// columns.
//
//   * A tile of 32 x 8 sites recomputes the densities of 1.69 sites per site
//     (forcing) and waits at two barriers for one wave of loads; a strip
//     recomputes 64/60 x (rows + 4)/rows, has no barrier and no shared memory,
//     and has the loads of the next row in flight while it works on this one.
//   * Every site's arithmetic is the same wherever the strips and chunks are
//     cut, so a batch and a single lattice agree bit for bit.
//
// AL: nx even, so every pair is one aligned 2-vector in every population array
// and never split by the periodic wrap; otherwise (odd nx) every site of a
// pair is loaded and stored on its own, wrapped on its own.
#pragma once
#include "step2d_pk.cuh"

namespace lbk {

constexpr int MARCH_COLS = 60;   // columns a warp collides

// Neighbours of a row held as one pair per lane: (value at x - 1, value at x + 1) of both sites.
__device__ __forceinline__ void row_neighbours(P2 c, P2& xm, P2& xp) {
    const float l = __shfl_up_sync(0xffffffffu, c.v.y, 1), r = __shfl_down_sync(0xffffffffu, c.v.x, 1);
    xm = pp(l, c.v.x);
    xp = pp(c.v.y, r);
}

// One step of the sites [x0, x0 + 60) x [y0, y1) of a lattice, by one warp.
template <bool FORCING, class S, bool AL, int PD>
__device__ __forceinline__ void step2d_march(const Tile2DArgs& args, int x0, int y0, int y1) {
    using L = D2Q9;
    using IO = PairIO<S>;
    using Wd = typename IO::W;
    constexpr int H = FORCING ? 2 : 1;     // rows above and below that the collision needs
    constexpr int NR = H + 1 + PD;         // rows held: the one collided .. the one being loaded
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
    const bool mine = lane >= 1 && lane <= 30;
    const bool v0 = mine && xo < nx, v1 = mine && xo + 1 < nx;
    const unsigned xa = unsigned(wrap_near(xo, nx)), xb = unsigned(wrap_near(xo + 1, nx));

    struct Row {
        float2 f0;
        Wd w[8];
    } raw[NR];
    auto load = [&](Row& r, unsigned row) {   // row: site index of the lattice row's first site
        LB_GUARD(row + xa < nsites && row + xb < nsites, BK_2D_LOAD, row, r.f0 = make_float2(0.f, 0.f);
                 for (int i = 0; i < 8; ++i) r.w[i] = Wd{}; return)
        if constexpr (AL) {
            const unsigned q = row + xa;
            r.f0 = reinterpret_cast<const float2*>(src)[q >> 1];
            static_for<1, 9>([&](auto I) {
                constexpr int i = decltype(I)::value;
                r.w[i - 1] = IO::ld(src + S::pop_offset(i, pitch), q);
            });
        } else {
            const float* f = reinterpret_cast<const float*>(src);
            r.f0 = make_float2(f[row + xa], f[row + xb]);
            static_for<1, 9>([&](auto I) {
                constexpr int i = decltype(I)::value;
                r.w[i - 1] = ld_split<S>(src + S::pop_offset(i, pitch), row + xa, row + xb);
            });
        }
    };

    const P2 third = pp(1.0f / 3.0f), twelfth = pp(1.0f / 12.0f);
    const unsigned unx = unsigned(nx), area = unx * unsigned(ny);
    // site index of the first site of the row being loaded, and of the row about to be collided
    unsigned lrow = unsigned(wrap_near(y0 - H, ny)) * unx;
    unsigned crow = unsigned(y0) * unx;
    auto up = [&](unsigned row) { return row + unx == area ? 0u : row + unx; };
    auto down = [&](unsigned row) { return row == 0u ? area - unx : row - unx; };
#pragma unroll
    for (int k = 0; k < PD; ++k) {
        load(raw[k], lrow);
        lrow = up(lrow);
    }
    // carried: density and its x difference / sum one and two rows back; forcing: the
    // partial sums of -g two rows back (all but the newest row's part) and one row back
    // (the oldest row's part), gradient and Laplacian of the row to collide
    P2 c1 = pp(0.f), d1 = c1, s1 = c1, c2 = c1, d2 = c1, s2 = c1;
    P2 gx2 = c1, gy2 = c1, gx1 = c1, gy1 = c1, G1x = c1, G1y = c1, lap1 = c1;
    const int nrows = y1 - y0 + 2 * H;     // rows passed through
    int k = 0;
    for (;;) {
#pragma unroll
        for (int ph_ = 0; ph_ < NR; ++ph_, ++k) {
            // row k of the march is in raw[k % NR]; the row loaded now goes where row k + PD belongs
            if (k + PD < nrows) {
                load(raw[(ph_ + PD) % NR], lrow);
                lrow = up(lrow);
            }
            const Row& now = raw[ph_];
            const P2 c = pair_rho9<S>(now.f0, now.w, ph.rsum);
            P2 xm, xp;
            row_neighbours(c, xm, xp);
            const P2 d = xp - xm, s = xp + xm;
            // gradient and Laplacian of row k - 1 (Eq. 32)
            P2 G[2], lap;
            G[0] = fma(third, d1, twelfth * (d + d2));
            G[1] = fma(third, c - c2, twelfth * (s - s2));
            lap = pp(2.0f) * (fma(third, s1 + (c + c2), twelfth * (s + s2)) - pp(5.0f / 3.0f) * c1);
            const P2 rho = FORCING ? c2 : c1;
            P2 g[2] = {pp(0.f), pp(0.f)};
            P2 Gc[2] = {G[0], G[1]}, lapc = lap;
            if constexpr (FORCING) {
                // M' of row k - 1: M'_xx = -M'_yy = D, M'_xy = O; its parts of -g in rows k - 2, k - 1, k
                const P2 kap = pp(ph.kappa), hk = pp(0.5f * ph.kappa);
                const P2 D = hk * fma(G[0], G[0], -(G[1] * G[1])), O = kap * (G[0] * G[1]);
                P2 Dm, Dp, Om, Op;
                row_neighbours(D, Dm, Dp);
                row_neighbours(O, Om, Op);
                const P2 dD = Dp - Dm, sD = Dp + Dm, dO = Op - Om, sO = Op + Om;
                const P2 ax = twelfth * dD, bx = fma(third, O, twelfth * sO);
                const P2 ay = twelfth * dO, by = fma(third, D, twelfth * sD);
                // -g_x = d_x D + d_y O, -g_y = d_x O - d_y D (Eq. 28)
                g[0] = -(gx2 + (ax + bx));
                g[1] = -(gy2 + (ay - by));
                gx2 = gx1 + third * dD;
                gy2 = gy1 + third * dO;
                gx1 = ax - bx;
                gy1 = ay + by;
                Gc[0] = G1x;
                Gc[1] = G1y;
                lapc = lap1;
                G1x = G[0];
                G1y = G[1];
                lap1 = lap;
            }
            if (k >= 2 * H) {
                const Row& old = raw[(ph_ + NR - H) % NR];
                P2 j[2];
                pair_momentum9<S>(old.w, j);
                if ((v0 && (!(rho.v.x > 0.f) || !(rho.v.x < 1e30f))) || (v1 && (!(rho.v.y > 0.f) || !(rho.v.y < 1e30f))))
                    atomicOr(args.status, 1u);
                PairColl2D<FORCING> K;
                K.prep(rho, j, Gc, lapc, g, ph);
                const P2 o0 = fma(K.omw, P2{old.f0}, K.c0);
                const unsigned yr[3] = {down(crow), crow, up(crow)};
                // destination column of site s moved by ex (site 0 at xa, site 1 at xb)
                const unsigned col[2][3] = {{unsigned(wrap_near(xo - 1, nx)), xa, xb},
                                            {xa, xb, unsigned(wrap_near(xo + 2, nx))}};
                auto store = [&](auto I, P2 v) {
                    constexpr int i = decltype(I)::value;
                    constexpr int ex = L::ex(i), ey = L::ey(i);
                    char* p = dst + S::pop_offset(i, pitch);
                    const unsigned row = yr[1 + ey];
#ifdef LB_DEBUG_BOUNDS
                    LB_GUARD(row + col[0][1 + ex] < nsites && row + col[1][1 + ex] < nsites, BK_2D_STORE, row, return)
#endif
                    if constexpr (AL && ex == 0) {
                        if (v0) IO::st2(p, row + xa, v);
                    } else {
                        if (v0) IO::st1(p, row + col[0][1 + ex], v.v.x);
                        if (v1) IO::st1(p, row + col[1][1 + ex], v.v.y);
                    }
                };
                if (v0) {
                    float* f0d = reinterpret_cast<float*>(dst);
                    if constexpr (AL) {
                        reinterpret_cast<float2*>(dst)[(crow + xa) >> 1] = o0.v;
                    } else {
                        f0d[crow + xa] = o0.v.x;
                        if (v1) f0d[crow + xb] = o0.v.y;
                    }
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

// One step of a single D2Q9 lattice: a warp per (strip, chunk of `rows` rows), strips side by side first.
template <bool FORCING, class S>
struct MarchForm {
    static constexpr int PD = 1;
    static constexpr int WARPS = 4;                                     // per CTA
    static constexpr int CTAS = PairIO<S>::RAW16 ? 4 : 3;               // resident CTAs per SM
};
template <bool FORCING, class S>
__global__ void __launch_bounds__(32 * MarchForm<FORCING, S>::WARPS, MarchForm<FORCING, S>::CTAS)
    step_kernel2d_march(const Tile2DArgs args, int strips, int rows, int items) {
    using F = MarchForm<FORCING, S>;
    const int item = blockIdx.x * F::WARPS + threadIdx.x / 32;
    if (item >= items) return;
    const int x0 = (item % strips) * MARCH_COLS, y0 = (item / strips) * rows;
    const int y1 = min(y0 + rows, args.ny);
    if (args.pair) step2d_march<FORCING, S, true, F::PD>(args, x0, y0, y1);
    else step2d_march<FORCING, S, false, F::PD>(args, x0, y0, y1);
}

}  // namespace lbk

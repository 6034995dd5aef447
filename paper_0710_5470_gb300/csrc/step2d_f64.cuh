// Fused D2Q9 time step in float64, one site per thread.
//
// The step of step2d_tile (step_kernel.cuh) for the arithmetic that the FP64
// pipe bounds: a GB300 SM completes two float64 lanes per clock, so a warp's
// instruction holds its scheduler for 64 clocks and every addition,
// multiplication and FMA counts alike, while loads, shared memory and integer
// work are free beside them.  Hence
//   * the stencils, the body force and the collision are written for the fewest
//     operations (138 per site and step in the forcing scheme where the
//     lattice-generic form took about 230): common differences are shared, the
//     factors 1/12 and 1/6 of the stencils go into constants of the host, M'
//     has two components (M'_xx = -M'_yy), one division gives both reciprocals;
//   * a thread keeps its own site's populations, gradient and Laplacian in
//     registers, and the halo sites go to the threads beyond the tile's (NTH >
//     TX * TY) first, which sit on other schedulers;
//   * the tile is chosen by the lattice's size (kern_d2q9.cu).
// Measured on a GB300 (us per step, forcing / equilibrium scheme, the
// lattice-generic kernel on 32 x 8 tiles -> now, launches chained): 100^2 18.2 -> 6.9 /
// 13.6 -> 5.8, 200^2 33.4 -> 17.2 / 24.6 -> 13.1, 512^2 113 -> 76 / 82 -> 63, 1024^2 432 ->
// 292 / 313 -> 239 (3.6 G sites/s; with 157 operations per site, halo included, 90% of
// the FP64 pipe).
#pragma once
#include "chain.cuh"
#include "step_kernel.cuh"

namespace lbk {

// Host-side constants of the float64 step.  G' = 12 grad rho and lap' = 6 lap
// rho are the unscaled stencil sums.
struct Consts64 {
    double a, b, T, omega, omw;        // omw = 1 - omega
    double nu12, nu12x3, nu12x6a;      // nu/12, 3 nu/12, 6 a nu/12: lambda/12 of Eq. 36 from T ib^2 and rho
    double kap6;                       // kappa/6: kappa rho lap = (kappa/6) rho lap'
    double kD, kO;                     // kappa/3456, kappa/1728: M'_xx / 12 and M'_xy / 12 from G'
    double kM;                         // omega kappa/144: omega M_ab from G' (equilibrium scheme)
};
inline Consts64 consts64(double a, double b, double T, double kappa, double omega, double nu) {
    return Consts64{a, b, T, omega, 1.0 - omega, nu / 12.0, nu / 4.0, a * nu / 2.0, kappa / 6.0, kappa / 3456.0,
                    kappa / 1728.0, omega * kappa / 144.0};
}

// Unscaled stencil sums at index c of a field with row stride RX: with A =
// f_NE - f_SW and B = f_SE - f_NW, 12 d_x f = 4 (f_E - f_W) + (A + B) and 12 d_y
// f = 4 (f_N - f_S) + (A - B); 6 lap f = 4 faces + diagonals - 20 f (Eq. 32).
struct Stencil9 {
    double gx, gy, lap;
};
__device__ __forceinline__ void gradient9_f64(const double* f, int c, int RX, double& gx, double& gy) {
    const double A = f[c + RX + 1] - f[c - RX - 1], B = f[c - RX + 1] - f[c + RX - 1];
    gx = fma(4.0, f[c + 1] - f[c - 1], A + B);
    gy = fma(4.0, f[c + RX] - f[c - RX], A - B);
}
__device__ __forceinline__ Stencil9 stencil9_f64(const double* f, int c, int RX) {
    Stencil9 s;
    gradient9_f64(f, c, RX, s.gx, s.gy);
    const double faces = (f[c + 1] + f[c - 1]) + (f[c + RX] + f[c - RX]);
    const double diag = (f[c + RX + 1] + f[c - RX - 1]) + (f[c - RX + 1] + f[c + RX - 1]);
    s.lap = fma(4.0, faces, fma(-20.0, f[c], diag));
    return s;
}

// Body force (Eq. 28) from D = M'_xx / 12 = -M'_yy / 12 and O = M'_xy / 12:
// g_x = -(d_x D + d_y O), g_y = -(d_x O - d_y D).
__device__ __forceinline__ void body_force9_f64(const double* D, const double* O, int c, int SX, double& gx, double& gy) {
    const double AD = D[c + SX + 1] - D[c - SX - 1], BD = D[c - SX + 1] - D[c + SX - 1];
    const double AO = O[c + SX + 1] - O[c - SX - 1], BO = O[c - SX + 1] - O[c + SX - 1];
    const double fx = (D[c + 1] - D[c - 1]) + (O[c + SX] - O[c - SX]);
    const double fy = (O[c + 1] - O[c - 1]) - (D[c + SX] - D[c - SX]);
    gx = -fma(4.0, fx, (AD + BD) + (AO - BO));
    gy = -fma(4.0, fy, (AO + BO) - (AD - BD));
}

// collide() of step_kernel.cuh for D2Q9 float64 from G', lap' and the force g:
// the same quadratic form in e_i, with S_ab = omega Q_ab + u_a g_b + u_b g_a, so
// that the even part of the axis pairs is Aw/3 + S_cc/2 and that of the diagonal
// pairs Aw/12 + (S_xx + S_yy)/8 +- S_xy/4.
template <bool FORCING>
__device__ __forceinline__ void collide9_f64(const double (&f)[9], double rho, double gx_, double gy_, double lap,
                                             double gx, double gy, const Consts64& k, double (&out)[9]) {
    const double a1 = f[1] - f[2], a3 = f[3] - f[4], a5 = f[5] - f[6], a7 = f[7] - f[8];
    const double jx = a1 + (a5 - a7), jy = a3 + (a5 + a7);
    const double ob = fma(-k.b, rho, 1.0);
    const double r = 1.0 / (rho * ob);
    const double irho = r * ob, ib = r * rho;
    const double ux = jx * irho, uy = jy * irho;
    // T / (1 - b rho) to half a unit (one Newton step): p0 multiplies its error several times (collide19_f64)
    const double Tib0 = k.T * ib, Tib = fma(ib, fma(-ob, Tib0, k.T), Tib0);
    const double p0 = rho * fma(-k.a, rho, Tib);                                      // Eq. 2
    const double lam12 = fma(-k.nu12x3, Tib * ib, fma(k.nu12x6a, rho, k.nu12));       // Eq. 36, over 12
    const double lx = lam12 * ux, ly = lam12 * uy;
    const double hx = lx * gx_, hy = ly * gy_, hh = hx + hy;
    const double qxx = fma(jx, ux, fma(2.0, hx, hh)), qyy = fma(jy, uy, fma(2.0, hy, hh));
    const double qxy = fma(jx, uy, fma(lx, gy_, ly * gx_));
    double Sxx, Syy, Sxy, Jx, Jy;
    double Aw = fma(-0.5, qxx + qyy, fma(-(k.kap6 * rho), lap, p0));
    if constexpr (FORCING) {
        const double mx = ux * gx, my = uy * gy;
        Sxx = fma(2.0, mx, k.omega * qxx);
        Syy = fma(2.0, my, k.omega * qyy);
        Sxy = fma(k.omega, qxy, fma(ux, gy, uy * gx));
        Aw = fma(k.omega, Aw, -(mx + my));
        Jx = fma(k.omega, jx, gx);
        Jy = fma(k.omega, jy, gy);
    } else {
        Sxx = k.omega * qxx;
        Syy = k.omega * qyy;
        Sxy = k.omega * qxy;
        Aw = k.omega * Aw;
        Jx = k.omega * jx;
        Jy = k.omega * jy;
    }
    const double third = 1.0 / 3.0;
    const double A3 = Aw * third;
    double Ex = fma(0.5, Sxx, A3), Ey = fma(0.5, Syy, A3);
    double P = fma(0.125, Sxx + Syy, 0.25 * A3);
    if constexpr (!FORCING) {
        // omega w^ab kappa d_a rho d_b rho: 1/3 and -1/6 on the axes, -1/24 and +-1/4 on the diagonals
        const double mx = k.kM * gx_, Mxx = mx * gx_, Myy = (k.kM * gy_) * gy_;
        Ex = fma(third, Mxx, fma(-1.0 / 6.0, Myy, Ex));
        Ey = fma(third, Myy, fma(-1.0 / 6.0, Mxx, Ey));
        P = fma(-1.0 / 24.0, Mxx + Myy, P);
        Sxy = fma(mx, gy_, Sxy);
    }
    const double Dp = fma(0.25, Sxy, P), Dm = fma(-0.25, Sxy, P);
    const double X = Jx * third, Y = Jy * third, d1 = X + Y, d2 = Y - X;
    out[0] = fma(k.omw, f[0], fma(-2.0, fma(2.0, P, Ex + Ey), k.omega * rho));   // Eq. 6 and sum_i F_i = 0
    out[1] = fma(k.omw, f[1], Ex + X);
    out[2] = fma(k.omw, f[2], Ex - X);
    out[3] = fma(k.omw, f[3], Ey + Y);
    out[4] = fma(k.omw, f[4], Ey - Y);
    out[5] = fma(k.omw, f[5], fma(0.25, d1, Dp));
    out[6] = fma(k.omw, f[6], fma(-0.25, d1, Dp));
    out[7] = fma(k.omw, f[7], fma(0.25, d2, Dm));
    out[8] = fma(k.omw, f[8], fma(-0.25, d2, Dm));
}

template <bool FORCING, int TX, int TY, int NTH>
struct Layout64 {
    static constexpr int H = FORCING ? 2 : 1;                     // density halo
    static constexpr int RX = TX + 2 * H, RY = TY + 2 * H, RN = RX * RY;
    static constexpr int SX = TX + 2, SY = TY + 2, SN = SX * SY;  // tile + one ring
    static constexpr int NT = TX * TY;
    static constexpr int NHALO = RN - NT, NRING = SN - NT;
    static constexpr size_t BYTES = size_t(RN + (FORCING ? 2 * SN : 0)) * sizeof(double);
    static_assert(NTH >= NT, "one thread per site at least");
};

// Site index of the n-th site of the frame of width W around a TX x TY tile, n
// in row order: the W full rows below, the side columns, the rows above.
template <int TX, int TY, int W>
__device__ __forceinline__ void frame_site(int n, int& x, int& y) {
    constexpr int FX = TX + 2 * W, BELOW = W * FX, SIDES = 2 * W * TY;
    if (n < BELOW) {
        x = n % FX;
        y = n / FX;
    } else if (n < BELOW + SIDES) {
        const int m = n - BELOW, s = m % (2 * W);
        y = W + m / (2 * W);
        x = s < W ? s : TX + s;
    } else {
        const int m = n - BELOW - SIDES;
        x = m % FX;
        y = W + TY + m / FX;
    }
}

// One D2Q9 time step of the TX x TY tile at (x0, y0) (Eq. 4) by NTH threads.
template <bool FORCING, int TX, int TY, int NTH>
__device__ __forceinline__ void step2d_tile_f64(const Tile2DArgs& args, const Consts64& k, int x0, int y0, double* sm) {
    using L = D2Q9;
    using Lay = Layout64<FORCING, TX, TY, NTH>;
    constexpr int H = Lay::H, NT = Lay::NT, RX = Lay::RX, SX = Lay::SX, SN = Lay::SN;
    double* rho_s = sm;
    double* D_s = sm + Lay::RN;
    double* O_s = D_s + SN;
    const int nx = args.nx, ny = args.ny, tid = threadIdx.x;
    const int tx = tid % TX, ty = tid / TX;
    const bool owner = NTH == NT || tid < NT;
    const double* src = reinterpret_cast<const double*>(args.src);
    const long long pitch = args.pitch;
    auto density = [&](const double (&f)[9]) {
        return f[0] + (((f[1] + f[2]) + (f[3] + f[4])) + ((f[5] + f[6]) + (f[7] + f[8])));
    };
    auto load = [&](int x, int y, double (&f)[9]) {
        const size_t q = size_t(wrap_near(y, ny)) * nx + wrap_near(x, nx);
        LB_GUARD(q < size_t(nx) * ny, BK_2D_LOAD, q, for (int i = 0; i < 9; ++i) f[i] = 0.0; return)
#pragma unroll
        for (int i = 0; i < 9; ++i) f[i] = src[i * pitch + q];
    };

    // ---------------- stage A: density of the tile and its halo
    double f[9];
    double rho = 0.0;
    const int rc = (ty + H) * RX + tx + H;
    if (owner) {
        load(x0 + tx, y0 + ty, f);
        rho = density(f);
        rho_s[rc] = rho;
    }
    // the threads without a site take the first halo sites
    const int first = tid >= NT ? tid - NT : tid + (NTH - NT);
#pragma unroll
    for (int n = first; n < Lay::NHALO; n += NTH) {
        int rx, ry;
        frame_site<TX, TY, H>(n, rx, ry);
        double h[9];
        load(x0 - H + rx, y0 - H + ry, h);
        rho_s[ry * RX + rx] = density(h);
    }
    __syncthreads();

    // ---------------- stage B: gradient, Laplacian; forcing: M' on the tile + 1 ring
    Stencil9 st{0.0, 0.0, 0.0};
    if (owner) st = stencil9_f64(rho_s, rc, RX);
    double gx = 0.0, gy = 0.0;
    if constexpr (FORCING) {
        auto put = [&](int at, double a, double b) {
            D_s[at] = k.kD * fma(a, a, -(b * b));
            O_s[at] = k.kO * (a * b);
        };
        const int kc = (ty + 1) * SX + tx + 1;
        if (owner) put(kc, st.gx, st.gy);
#pragma unroll
        for (int n = first; n < Lay::NRING; n += NTH) {
            int sx, sy;
            frame_site<TX, TY, 1>(n, sx, sy);
            double a, b;
            gradient9_f64(rho_s, (sy + H - 1) * RX + sx + H - 1, RX, a, b);
            put(sy * SX + sx, a, b);
        }
        __syncthreads();
        if (owner) body_force9_f64(D_s, O_s, kc, SX, gx, gy);
    }

    // ---------------- stage C: collide and push
    const int xs = x0 + tx, ys = y0 + ty;
    if (owner && xs < nx && ys < ny) {
        if (!(rho > 0.0) || !(rho < 1e30)) atomicOr(args.status, 1u);
        double out[9];
        collide9_f64<FORCING>(f, rho, st.gx, st.gy, st.lap, gx, gy, k, out);
        const int xw[3] = {wrap_near(xs - 1, nx), xs, wrap_near(xs + 1, nx)};
        const size_t yr[3] = {size_t(wrap_near(ys - 1, ny)) * nx, size_t(ys) * nx, size_t(wrap_near(ys + 1, ny)) * nx};
        double* dst = reinterpret_cast<double*>(args.dst);
        static_for<0, 9>([&](auto I) {
            constexpr int i = decltype(I)::value;
            const size_t idx = yr[1 + L::ey(i)] + xw[1 + L::ex(i)];
            LB_GUARD(idx < size_t(nx) * ny, BK_2D_STORE, idx, return)
            dst[i * pitch + idx] = out[i];
        });
    }
}

// One step of a single D2Q9 lattice: one CTA per tile.
template <bool FORCING, int TX, int TY, int NTH>
__global__ void __launch_bounds__(NTH) step_kernel2d_f64(const Tile2DArgs args, const Consts64 k) {
    chain_begin();
    extern __shared__ __align__(16) unsigned char smem_raw[];
    step2d_tile_f64<FORCING, TX, TY, NTH>(args, k, blockIdx.x * TX, blockIdx.y * TY, reinterpret_cast<double*>(smem_raw));
}

}  // namespace lbk

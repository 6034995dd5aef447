// D3Q19 time step in float64: two or three passes over one-site threads.
//
// What bounds float64 on a GB300 is the FP64 pipe (two lanes per clock and SM):
// at 301 operations per site the forcing step needs 0.48 ns of the whole chip
// per site, while its 600 bytes of traffic need 0.09 ns.  So the step is cut
// where that removes operations, and moves the intermediate fields through
// memory (mostly L2) instead of recomputing them:
//   density3_f64   rho = sum_i f_i (Eq. 3): 18 operations;
//   mprime3_f64    (forcing) G' = 12 grad rho, lap' = 6 lap rho (Eq. 29) and
//                  M'_ab - delta_ab M'_cc / 2 over 12: 52;
//   collide3_f64   the force -div M' (Eq. 28), the collision (Eqs. 2-6, 27, 36)
//                  and the push (Eq. 4): 231; (equilibrium) its own G', lap'.
// The fused kernel of step3d.cuh, which marches 32 x 4 tiles through z,
// recomputed the densities of 2.25 and the M' of 1.6 sites per site and spent
// about 520 operations, in one long chain per CTA.  Measured, us per step, fused
// -> passes, forcing and equilibrium scheme (launches chained): 32^3 96 -> 23.6 and 51 ->
// 17.5, 64^3 263 -> 159 and 164 -> 119, 128^3 1884 -> 1198 and 1305 -> 898 (1.75 and 2.34
// G sites/s, the FP64 pipe 85% busy).
//
// The fields live in a workspace of the context: the whole lattice where that
// fits its limit, else slabs of planes with two (forcing) or one halo planes on
// either side, computed one slab after the other (kern_d3q19_f64.cu).
#pragma once
#include "chain.cuh"
#include "bounds.cuh"
#include "step_kernel.cuh"

namespace lbk {

// Threads per CTA: one warp, so that a lattice of a few hundred warps spreads
// over all schedulers (32^3 forcing 26.7 us against 30.1 with 128 threads; the
// same from 48^3 on).
constexpr int THREADS64 = 32;

struct Consts64x3 {
    double a, b, T, omega, omw;         // omw = 1 - omega
    double onu12, onu12x3, onu12x6a;    // omega nu/12 (x 3, x 6 a): omega lambda/12 of Eq. 36 from T ib^2 and rho
    double kap6;                        // kappa/6: kappa rho lap = (kappa/6) rho lap'
    double k1728;                       // kappa/(144 12): M' over 12 from G'
    double kM;                          // omega kappa/144: omega M_ab from G' (equilibrium scheme)
};

struct Args64x3 {
    const double* src;
    double* dst;
    long long pitch;       // elements per population array
    double* rho;           // workspace: [plane][site of the plane]
    double* G;             // (G'_x, G'_y, G'_z, lap'), one field each, `field` elements apart
    double* M;             // (xx, yy, zz, xy, yz, xz) likewise
    long long field;
    int nx, ny, nz;
    int z0;                // lattice plane of local plane 0
    int first, planes;     // local planes of this launch: [first, first + planes)
    int halo;              // workspace plane of local plane p: p + halo
    int wrap_planes;       // > 0: the workspace holds the whole lattice, periodic in so many planes
    Consts64x3 k;
    unsigned* status;
};

// A thread's site: place in its plane, lattice and workspace indices of the
// plane's first site, and the neighbours' offsets.
struct Site3 {
    int x, y, z;
    unsigned wp[3];        // workspace planes below, own, above: index of the first site
    unsigned row[3];       // y - 1, y, y + 1 within a plane
    unsigned col[3];
    // index of the neighbour (dx, dy, dz)
    __device__ __forceinline__ unsigned at(int dx, int dy, int dz) const { return wp[1 + dz] + row[1 + dy] + col[1 + dx]; }
};

__device__ __forceinline__ bool site3(const Args64x3& a, Site3& s) {
    const unsigned area = unsigned(a.nx) * unsigned(a.ny);
    const unsigned t = blockIdx.x * blockDim.x + threadIdx.x;
    const unsigned p = t / area;
    if (p >= unsigned(a.planes)) return false;
    const unsigned q = t - p * area;
    s.y = int(q / unsigned(a.nx));
    s.x = int(q - unsigned(s.y) * unsigned(a.nx));
    const int lp = a.first + int(p);
    s.z = wrapi(a.z0 + lp, a.nz);
    const int w = lp + a.halo;
    const int up = a.wrap_planes > 0 && w + 1 == a.wrap_planes ? 0 : w + 1;
    const int dn = a.wrap_planes > 0 && w == 0 ? a.wrap_planes - 1 : w - 1;
    s.wp[0] = unsigned(dn) * area;
    s.wp[1] = unsigned(w) * area;
    s.wp[2] = unsigned(up) * area;
    const unsigned nx = unsigned(a.nx);
    s.row[0] = unsigned(s.y == 0 ? a.ny - 1 : s.y - 1) * nx;
    s.row[1] = unsigned(s.y) * nx;
    s.row[2] = unsigned(s.y == a.ny - 1 ? 0 : s.y + 1) * nx;
    s.col[0] = unsigned(s.x == 0 ? a.nx - 1 : s.x - 1);
    s.col[1] = unsigned(s.x);
    s.col[2] = unsigned(s.x == a.nx - 1 ? 0 : s.x + 1);
    return true;
}

// Whether the workspace planes lo..hi beside the site's lie in the workspace (checked builds).
__device__ __forceinline__ bool planes_inside(const Args64x3& a, const Site3& s, int lo, int hi) {
    for (int d = lo; d <= hi; ++d)
        if ((long long)s.wp[1 + d] + (long long)a.nx * a.ny > a.field) return false;
    return true;
}

// Sum of the 19 populations in pairs of opposite velocities.
__device__ __forceinline__ double density19_f64(const double (&f)[19]) {
    return f[0] + tree_sum<1, 19>(f);
}

__global__ void __launch_bounds__(THREADS64) density3_f64(const Args64x3 a) {
    chain_begin();
    Site3 s;
    if (!site3(a, s)) return;
    const size_t q = (size_t(s.z) * a.ny + s.y) * a.nx + s.x;
    LB_GUARD(q < size_t(a.nx) * a.ny * a.nz, BK_3D_LOAD, q, return)
    LB_GUARD(planes_inside(a, s, 0, 0), BK_WORK, s.wp[1], return)
    double f[19];
#pragma unroll
    for (int i = 0; i < 19; ++i) f[i] = a.src[i * a.pitch + q];
    a.rho[s.at(0, 0, 0)] = density19_f64(f);
}

// 12 grad and 6 lap of rho at a site (Eq. 29: 12 d_x = 2 (E - W) + diagonals, 6
// lap = 2 faces + diagonals - 24 rho).  The difference of two opposite diagonal
// neighbours serves both gradients of its plane: 21 + 18 operations.
__device__ __forceinline__ void stencil19_f64(const double* rho, const Site3& s, double c, double (&g)[3], double& lap) {
    const double e = rho[s.at(1, 0, 0)], w = rho[s.at(-1, 0, 0)], n = rho[s.at(0, 1, 0)], o = rho[s.at(0, -1, 0)];
    const double u = rho[s.at(0, 0, 1)], d = rho[s.at(0, 0, -1)];
    double faces = ((e + w) + (n + o)) + (u + d);
    double pp = rho[s.at(1, 1, 0)], mm = rho[s.at(-1, -1, 0)], pm = rho[s.at(1, -1, 0)], mp = rho[s.at(-1, 1, 0)];
    double A = pp - mm, B = pm - mp, diag = (pp + mm) + (pm + mp);
    double gx = A + B, gy = A - B;
    pp = rho[s.at(1, 0, 1)], mm = rho[s.at(-1, 0, -1)], pm = rho[s.at(1, 0, -1)], mp = rho[s.at(-1, 0, 1)];
    A = pp - mm, B = pm - mp;
    diag += (pp + mm) + (pm + mp);
    gx += A + B;
    double gz = A - B;
    pp = rho[s.at(0, 1, 1)], mm = rho[s.at(0, -1, -1)], pm = rho[s.at(0, 1, -1)], mp = rho[s.at(0, -1, 1)];
    A = pp - mm, B = pm - mp;
    diag += (pp + mm) + (pm + mp);
    gy += A + B;
    gz += A - B;
    g[0] = fma(2.0, e - w, gx);
    g[1] = fma(2.0, n - o, gy);
    g[2] = fma(2.0, u - d, gz);
    lap = fma(2.0, faces, fma(-24.0, c, diag));
}

__global__ void __launch_bounds__(THREADS64) mprime3_f64(const Args64x3 a) {
    chain_begin();
    Site3 s;
    if (!site3(a, s)) return;
    const unsigned at = s.at(0, 0, 0);
    LB_GUARD(planes_inside(a, s, -1, 1), BK_WORK, at, return)
    double g[3], lap;
    stencil19_f64(a.rho, s, a.rho[at], g, lap);
#pragma unroll
    for (int c = 0; c < 3; ++c) a.G[c * a.field + at] = g[c];
    a.G[3 * a.field + at] = lap;
    const double kx = a.k.k1728 * g[0], ky = a.k.k1728 * g[1], kz = a.k.k1728 * g[2];
    const double h = -0.5 * fma(kx, g[0], fma(ky, g[1], kz * g[2]));
    a.M[at] = fma(kx, g[0], h);
    a.M[a.field + at] = fma(ky, g[1], h);
    a.M[2 * a.field + at] = fma(kz, g[2], h);
    a.M[3 * a.field + at] = kx * g[1];
    a.M[4 * a.field + at] = ky * g[2];
    a.M[5 * a.field + at] = kx * g[2];
}

// g = -div M' (Eq. 28, read in 3D) from the six fields over 12.  In the plane
// of axes p and q a diagonal neighbour pair contributes (A + B) of M_cp and (A -
// B) of M_cq to component c, A and B the differences of the two opposite
// diagonals: 81 operations.
__device__ __forceinline__ void body_force19_f64(const double* M, long long field, const Site3& s, double (&g)[3]) {
    const double *xx = M, *yy = M + field, *zz = M + 2 * field, *xy = M + 3 * field, *yz = M + 4 * field,
                 *xz = M + 5 * field;
    double ax[3];
    {
        const unsigned e = s.at(1, 0, 0), w = s.at(-1, 0, 0), n = s.at(0, 1, 0), o = s.at(0, -1, 0), u = s.at(0, 0, 1),
                       d = s.at(0, 0, -1);
        ax[0] = ((xx[e] - xx[w]) + (xy[n] - xy[o])) + (xz[u] - xz[d]);
        ax[1] = ((xy[e] - xy[w]) + (yy[n] - yy[o])) + (yz[u] - yz[d]);
        ax[2] = ((xz[e] - xz[w]) + (yz[n] - yz[o])) + (zz[u] - zz[d]);
    }
    double dg[3];
    auto plane = [&](unsigned pp, unsigned mm, unsigned pm, unsigned mp, const double* cp, const double* cq, auto add) {
        // contribution of M_cp (p: first axis of the plane) and M_cq to a component
        const double Ap = cp[pp] - cp[mm], Bp = cp[pm] - cp[mp], Aq = cq[pp] - cq[mm], Bq = cq[pm] - cq[mp];
        add(Ap, Bp, Aq, Bq);
    };
    {   // xy: M_xx, M_xy | M_xy, M_yy | M_xz, M_yz
        const unsigned pp = s.at(1, 1, 0), mm = s.at(-1, -1, 0), pm = s.at(1, -1, 0), mp = s.at(-1, 1, 0);
        plane(pp, mm, pm, mp, xx, yy, [&](double Axx, double Bxx, double Ayy, double Byy) {
            const double A = xy[pp] - xy[mm], B = xy[pm] - xy[mp];
            dg[0] = (Axx + Bxx) + (A - B);
            dg[1] = (A + B) + (Ayy - Byy);
        });
        plane(pp, mm, pm, mp, xz, yz, [&](double Ap, double Bp, double Aq, double Bq) { dg[2] = (Ap + Bp) + (Aq - Bq); });
    }
    {   // xz: M_xx, M_xz | M_xy, M_yz | M_xz, M_zz
        const unsigned pp = s.at(1, 0, 1), mm = s.at(-1, 0, -1), pm = s.at(1, 0, -1), mp = s.at(-1, 0, 1);
        plane(pp, mm, pm, mp, xx, zz, [&](double Axx, double Bxx, double Azz, double Bzz) {
            const double A = xz[pp] - xz[mm], B = xz[pm] - xz[mp];
            dg[0] += (Axx + Bxx) + (A - B);
            dg[2] += (A + B) + (Azz - Bzz);
        });
        plane(pp, mm, pm, mp, xy, yz, [&](double Ap, double Bp, double Aq, double Bq) { dg[1] += (Ap + Bp) + (Aq - Bq); });
    }
    {   // yz: M_xy, M_xz | M_yy, M_yz | M_yz, M_zz
        const unsigned pp = s.at(0, 1, 1), mm = s.at(0, -1, -1), pm = s.at(0, 1, -1), mp = s.at(0, -1, 1);
        plane(pp, mm, pm, mp, yy, zz, [&](double Ayy, double Byy, double Azz, double Bzz) {
            const double A = yz[pp] - yz[mm], B = yz[pm] - yz[mp];
            dg[1] += (Ayy + Byy) + (A - B);
            dg[2] += (A + B) + (Azz - Bzz);
        });
        plane(pp, mm, pm, mp, xy, xz, [&](double Ap, double Bp, double Aq, double Bq) { dg[0] += (Ap + Bp) + (Aq - Bq); });
    }
#pragma unroll
    for (int c = 0; c < 3; ++c) g[c] = -fma(2.0, ax[c], dg[c]);
}

// collide() of step_kernel.cuh for D3Q19 float64 from G', lap' and the force g:
// the same quadratic form in e_i, with S_ab = omega Q_ab + u_a g_b + u_b g_a; the
// even part of an axis pair is E_c = Aw/6 + S_cc/4, that of a diagonal pair
// Aw/12 + (S_cc + S_dd)/8 +- S_cd/4.  152 operations.
template <bool FORCING, class Push>
__device__ __forceinline__ void collide19_f64(const double (&f)[19], double rho, const double (&G)[3], double lap,
                                              const double (&g)[3], const Consts64x3& k, Push&& push) {
    using L = D3Q19;
    double j[3];
    {
        const double Axy = f[7] - f[10], Bxy = f[9] - f[8], Ayz = f[11] - f[14], Byz = f[13] - f[12];
        const double Axz = f[15] - f[18], Bxz = f[17] - f[16];
        j[0] = (f[1] - f[2]) + ((Axy + Bxy) + (Axz + Bxz));
        j[1] = (f[3] - f[4]) + ((Axy - Bxy) + (Ayz + Byz));
        j[2] = (f[5] - f[6]) + ((Axz - Bxz) + (Ayz - Byz));
    }
    const double ob = fma(-k.b, rho, 1.0);
    const double r = 1.0 / (rho * ob);
    const double irho = r * ob, ib = r * rho;
    // T / (1 - b rho) to half a unit: p0 is a small difference of it and a rho, which multiplies its
    // error several times (one Newton step, two operations; without it the populations' error against
    // exact arithmetic was 7 - 17% larger, 20 steps of a drop)
    const double Tib0 = k.T * ib, Tib = fma(ib, fma(-ob, Tib0, k.T), Tib0);
    const double p0 = rho * fma(-k.a, rho, Tib);                                     // Eq. 2
    const double olam = fma(-k.onu12x3, Tib * ib, fma(k.onu12x6a, rho, k.onu12));    // omega lambda/12, Eq. 36
    // omega Q_ab + u_a g_b + u_b g_a = omega j_a u_b + u_a w_b + u_b w_a + delta_ab omega lambda u.G
    // with w = g + omega lambda G
    double u[3], oj[3], w[3], X[3];
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        u[c] = j[c] * irho;
        oj[c] = k.omega * j[c];
        w[c] = FORCING ? fma(olam, G[c], g[c]) : olam * G[c];
        X[c] = (FORCING ? oj[c] + g[c] : oj[c]) * (1.0 / 6.0);
    }
    const double ohh = olam * fma(u[0], G[0], fma(u[1], G[1], u[2] * G[2]));
    double S[3][3];
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        S[c][c] = fma(u[c], fma(2.0, w[c], oj[c]), ohh);
#pragma unroll
        for (int d = c + 1; d < 3; ++d) S[c][d] = fma(oj[c], u[d], fma(u[c], w[d], u[d] * w[c]));
    }
    // omega (p0 - kappa rho lap - tr Q / 2) - u.g, tr Q = j.u + 5 lambda u.G
    double Aw = fma(-0.5, fma(oj[0], u[0], fma(oj[1], u[1], oj[2] * u[2])), k.omega * fma(-(k.kap6 * rho), lap, p0));
    Aw = fma(-2.5, ohh, Aw);
    if constexpr (FORCING) Aw -= fma(u[0], g[0], fma(u[1], g[1], u[2] * g[2]));
    const double A6 = Aw * (1.0 / 6.0), hA = 0.5 * A6;
    double E[3], P[3][3];
#pragma unroll
    for (int c = 0; c < 3; ++c) E[c] = fma(0.25, S[c][c], A6);
#pragma unroll
    for (int c = 0; c < 3; ++c)
#pragma unroll
        for (int d = c + 1; d < 3; ++d) P[c][d] = fma(0.125, S[c][c] + S[d][d], hA);
    if constexpr (!FORCING) {
        // omega w^ab kappa d_a rho d_b rho: on an axis 5/12 of its own diagonal term and -1/3 of
        // the others; on a diagonal -1/24 of the two it touches, 1/12 of the third and +-1/4 of M_cd
        double M[3];
        double kg[3];
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            kg[c] = k.kM * G[c];
            M[c] = kg[c] * G[c];
        }
        const double t3 = ((M[0] + M[1]) + M[2]) * (-1.0 / 3.0);
        const double t24 = t3 * 0.125;                       // -(1/24) sum
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            E[c] += fma(0.75, M[c], t3);                     // 5/12 + 1/3 = 3/4
#pragma unroll
            for (int d = c + 1; d < 3; ++d) {
                P[c][d] += fma(0.125, M[3 - c - d], t24);    // 1/12 + 1/24 = 1/8
                S[c][d] = fma(kg[c], G[d], S[c][d]);
            }
        }
    }
    push(std::integral_constant<int, 0>{},
         fma(k.omw, f[0], fma(-2.0, fma(2.0, (P[0][1] + P[0][2]) + P[1][2], (E[0] + E[1]) + E[2]), k.omega * rho)));
    static_for<1, 19>([&](auto I) {
        constexpr int i = decltype(I)::value, o = opposite<L>(i);
        if constexpr (i < o) {
            constexpr int c = first_axis<L>(i), d = second_axis<L>(i);
            constexpr int ec = e_comp<L>(i, c);
            double vi, vo;   // even +- odd part of the pair
            if constexpr (d < 0) {
                vi = ec > 0 ? E[c] + X[c] : E[c] - X[c];
                vo = ec > 0 ? E[c] - X[c] : E[c] + X[c];
            } else {
                constexpr int ed = e_comp<L>(i, d);
                const double ev = fma(ec * ed > 0 ? 0.25 : -0.25, S[c][d], P[c][d]);
                const double od = (ec > 0 ? X[c] : -X[c]) + (ed > 0 ? X[d] : -X[d]);
                vi = fma(0.5, od, ev);
                vo = fma(-0.5, od, ev);
            }
            push(I, fma(k.omw, f[i], vi));
            push(std::integral_constant<int, o>{}, fma(k.omw, f[o], vo));
        }
    });
}

template <bool FORCING>
__global__ void __launch_bounds__(THREADS64, 16) collide3_f64(const Args64x3 a) {
    chain_begin();
    using L = D3Q19;
    Site3 s;
    if (!site3(a, s)) return;
    const unsigned area = unsigned(a.nx) * unsigned(a.ny), at = s.at(0, 0, 0);
    // lattice planes below, own, above
    const unsigned lp[3] = {unsigned(s.z == 0 ? a.nz - 1 : s.z - 1) * area, unsigned(s.z) * area,
                            unsigned(s.z == a.nz - 1 ? 0 : s.z + 1) * area};
    const unsigned q = lp[1] + s.row[1] + s.col[1];
    LB_GUARD(q < area * unsigned(a.nz), BK_3D_LOAD, q, return)
    LB_GUARD(planes_inside(a, s, -1, 1), BK_WORK, at, return)
    double f[19];
#pragma unroll
    for (int i = 0; i < 19; ++i) f[i] = a.src[i * a.pitch + q];
    const double rho = a.rho[at];
    double G[3], lap, g[3] = {0.0, 0.0, 0.0};
    if constexpr (FORCING) {
        body_force19_f64(a.M, a.field, s, g);
#pragma unroll
        for (int c = 0; c < 3; ++c) G[c] = a.G[c * a.field + at];
        lap = a.G[3 * a.field + at];
    } else {
        stencil19_f64(a.rho, s, rho, G, lap);
    }
    if (!(rho > 0.0) || !(rho < 1e30)) atomicOr(a.status, 1u);
    collide19_f64<FORCING>(f, rho, G, lap, g, a.k, [&](auto I, double v) {
        constexpr int i = decltype(I)::value;
        const unsigned idx = lp[1 + L::ez(i)] + s.row[1 + L::ey(i)] + s.col[1 + L::ex(i)];
        LB_GUARD(idx < area * unsigned(a.nz), BK_3D_STORE, idx, return)
        a.dst[i * a.pitch + idx] = v;
    });
}

}  // namespace lbk

// Binary-fluid D3Q19 step in float32, two adjacent x sites per thread, marching
// through z planes of the phi field (binary_phi_kernel).
//
// A CTA owns a 32 x 8 column tile and a chunk of planes, as the liquid-gas kernels
// do (step3d_fd.cuh): per plane it takes phi on the tile and its halo from the field
// into shared memory, forms the z-split parts of the gradient and Laplacian
// (Eq. 29), in the forcing scheme M'_ab - delta_ab M'_cc / 2 on the tile plus one
// ring and the z-split parts of its divergence (reading R7), and collides the plane
// two (equilibrium scheme: one) behind as packed float32 pairs: f with the binary
// pressure, g with phi v for the momentum and Gamma mu for the pressure, by the same
// quadratic form.
// The brick kernel of binary3d.cu (one site per thread, 32 x 4 x 2 sites) formed M'
// on 3.2 and the stencils anew on every site: 1680 instructions per site in the
// forcing scheme, bound by issue; this one has 640 and is bound by the loads of the
// 38 populations.  Measured on a GB300, us per step with the phi pass (27 us at
// 128^3), bricks -> march:
// 64^3 forcing 24.3 -> 19.7, 101 x 75 x 53 45.4 -> 36.7, 128^3 189 -> 146 (388 bytes
// per site at 82% of the copy bandwidth), 256^3 1459 -> 1288; equilibrium 64^3 17.2
// -> 15.7, 128^3 152 -> 131, 256^3 1263 -> 1179 (launches chained).
//
// AL: nx even, so that pairs are aligned 2-vectors and never split by the periodic
// wrap; otherwise every site of a pair is loaded and stored on its own.
#pragma once
#include "binary_common.cuh"
#include "chain.cuh"
#include "step3d_pk_eq.cuh"

namespace lbb {

using lbk::fma;
using lbk::BK_B3_LOAD;
using lbk::BK_B3_STORE;

struct March3Args {
    StepArgs<float> s;
    const int4* work;    // per CTA (x0, y0, z0, z1)
};

template <int TX, int TY>
struct LayoutMarch3 {
    using PK = lbk::LayoutPK<TX, TY, true>;
    static constexpr int NTH = PK::NTH, RX = PK::RX, RN = PK::RN, SN = PK::SN;
    static constexpr size_t OFF_MPA = (size_t(2) * RN * 4 + 15) / 16 * 16;
    static constexpr size_t OFF_MPB = OFF_MPA + size_t(SN) * 16;
    static constexpr size_t bytes(bool forcing) { return forcing ? OFF_MPB + size_t(SN) * 8 : OFF_MPA; }
};

// The relaxation of one distribution as a quadratic form in e_i (PairColl of
// step3d_pk.cuh with lambda = 0): relaxation rate om, momentum m, velocity u,
// isotropic part iso and, with FORCE, the force g of Eq. 27.  A population moves by
// om (feq - f) + F as one small number added to it, as the brick kernel adds it: (1 -
// om) f + om feq rounds twice at the size of f.
struct Form {
    P2 Jw[3];            // om m + g
    P2 EA[3];            // even part of the axis pairs, weighted
    P2 WE[3], WO[3];     // diagonal planes xy, xz, yz: even part WE +- WO, weighted
    P2 mom, lost;        // -om; sum of f_i - f*_i over the populations 1.. relaxed so far

    template <bool FORCE, bool MTERMS>
    __device__ __forceinline__ void prep(float om, const P2 (&m)[3], const P2 (&u)[3], P2 iso,
                                         const P2 (&g)[3], float kappa, const P2 (&G)[3]) {
        const P2 w15 = pp(1.5f * om), w3 = pp(3.0f * om), o = pp(om);
        constexpr int cc[3] = {0, 0, 1}, dd[3] = {1, 2, 2};
        constexpr float wax = 1.0f / 6.0f, wdg = 1.0f / 12.0f;
        P2 q[3], Td[3];
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            q[c] = m[c] * u[c];
            Td[c] = FORCE ? fma(w15, q[c], pp(3.0f) * (u[c] * g[c])) : w15 * q[c];
            Jw[c] = FORCE ? fma(o, m[c], g[c]) : o * m[c];
        }
        P2 Aw = o * fma(pp(-0.5f), (q[0] + q[1]) + q[2], iso);
        if constexpr (FORCE) Aw -= fma(u[0], g[0], fma(u[1], g[1], u[2] * g[2]));
#pragma unroll
        for (int c = 0; c < 3; ++c) EA[c] = pp(wax) * (Aw + Td[c]);
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            const int c = cc[k], e = dd[k];
            const P2 x = w3 * (m[c] * u[e]);
            WE[k] = pp(wdg) * ((Aw + Td[c]) + Td[e]);
            WO[k] = pp(wdg) * (FORCE ? fma(pp(3.0f), fma(u[c], g[e], u[e] * g[c]), x) : x);
        }
        if constexpr (MTERMS) {
            // w^ab om kappa d_a phi d_b phi: axis 3/4 M_cc - 1/3 sum, diagonal 1/12 sum -
            // 1/8 (M_cc + M_dd) +- 1/4 M_cd (PairCollEq::prep)
            const P2 ok = pp(om * kappa);
            P2 M[3];
#pragma unroll
            for (int c = 0; c < 3; ++c) M[c] = ok * G[c] * G[c];
            const P2 Ms = (M[0] + M[1]) + M[2];
#pragma unroll
            for (int c = 0; c < 3; ++c) EA[c] += fma(pp(0.75f), M[c], pp(-1.0f / 3.0f) * Ms);
#pragma unroll
            for (int k = 0; k < 3; ++k) {
                WE[k] += fma(pp(wdg), Ms, pp(-0.125f) * (M[cc[k]] + M[dd[k]]));
                WO[k] = fma(pp(0.25f) * ok, G[cc[k]] * G[dd[k]], WO[k]);
            }
        }
        mom = pp(-om);
        lost = pp(0.0f);
    }

    __device__ __forceinline__ P2 relax(P2 f, P2 gain) const { return f + fma(mom, f, gain); }

    // Population 0, after the others.  The relaxation conserves the density (Eq. 6, sum F_i =
    // 0), so population 0 takes what the others lost as they were rounded: differences of
    // nearby numbers, exact or nearly so, where om feq_0 from a sum of populations would
    // round it at the size of the density every step.
    __device__ __forceinline__ P2 rest(P2 f0) const { return f0 + lost; }

    // the relaxed opposite pair (i, o), i < o
    template <int i>
    __device__ __forceinline__ void out(P2 fi, P2 fo, P2& oi, P2& oo) {
        using L = D3Q19;
        constexpr int c = lbk::first_axis<L>(i), e2 = lbk::second_axis<L>(i);
        P2 odd, ev;
        if constexpr (e2 < 0) {
            odd = lbk::e_comp<L>(i, c) > 0 ? Jw[c] : -Jw[c];
            ev = EA[c];
        } else {
            constexpr int sc = lbk::e_comp<L>(i, c), se = lbk::e_comp<L>(i, e2);
            constexpr int k = (c == 0 && e2 == 1) ? 0 : ((c == 0 && e2 == 2) ? 1 : 2);
            odd = (sc > 0 ? Jw[c] : -Jw[c]) + (se > 0 ? Jw[e2] : -Jw[e2]);
            ev = sc * se > 0 ? WE[k] + WO[k] : WE[k] - WO[k];
        }
        const P2 w = pp(float(lbk::w_vel<L>(i)));
        const P2 gi = fma(w, odd, ev), go = fma(-w, odd, ev);
        oi = relax(fi, gi);
        oo = relax(fo, go);
        lost += (fi - oi) + (fo - oo);
    }
};

// Three CTAs per SM (168 registers); with two the step took 9% longer at 128^3, at
// four (128 registers, spills) 25%.
template <bool FORCING, int TX, int TY, bool AL>
__global__ void __launch_bounds__((TX / 2) * TY, 3) binary_step_kernel3_march(const March3Args args) {
    lbk::chain_begin();
    using L = D3Q19;
    using Lay = lbk::LayoutPK<TX, TY, true>;
    using LF = LayoutMarch3<TX, TY>;
    constexpr int H = Lay::H, HX = Lay::HX, TXP = Lay::TXP, NTH = Lay::NTH, RX = Lay::RX, SX = Lay::SX;
    constexpr int NBR = Lay::NBR, LAG = FORCING ? 2 : 1;
    const StepArgs<float>& a = args.s;

    extern __shared__ __align__(16) unsigned char smem_raw[];
    float* phi_s = reinterpret_cast<float*>(smem_raw);
    float4* mpA = reinterpret_cast<float4*>(smem_raw + LF::OFF_MPA);   // (Mxx, Mxy, Mxz, Myy)
    float2* mpB = reinterpret_cast<float2*>(smem_raw + LF::OFF_MPB);   // (Myz, Mzz)

    const int nx = a.nx, ny = a.ny, nz = a.nz;
    const int tid = threadIdx.x, px = tid % TXP, py = tid / TXP;
    const int4 wk = args.work[blockIdx.x];
    const int x0 = wk.x, y0 = wk.y, z0 = wk.z, z1 = wk.w;
    const unsigned plane = unsigned(nx) * unsigned(ny), vol = plane * unsigned(nz), pitch = a.pitch;
    const float pk = a.kappa;
    const float* src = a.src;
    float* dst = a.dst;

    // region items of phi: pairs (AL) or single sites
    constexpr int W = AL ? 2 : 1, NIT = Lay::RN / W, NA = (NIT + NTH - 1) / NTH, RXW = RX / W;
    unsigned a_in[NA];
#pragma unroll
    for (int m = 0; m < NA; ++m) {
        const int k = tid + m * NTH;
        a_in[m] = k < NIT ? unsigned(wrapc(y0 - H + k / RXW, ny)) * unsigned(nx) + unsigned(wrapc(x0 - HX + (k % RXW) * W, nx)) : 0u;
    }
    const int xo = x0 + 2 * px, yo = y0 + py;
    const bool own = xo < nx && yo < ny, own1 = own && (AL || xo + 1 < nx);
    int b_rc = -1, b_mp = 0;                  // ring site of stage B: region index and M' index
    if constexpr (FORCING) {
        static_assert(NBR == 1, "one ring site per thread");
        int sx, sy;
        if (tid < 2 * SX) {
            sx = tid % SX;
            sy = tid < SX ? 0 : Lay::SY - 1;
        } else {
            const int k = tid - 2 * SX;
            sy = 1 + (k >> 1);
            sx = (k & 1) ? SX - 1 : 0;
        }
        if (tid < Lay::NRING) {
            b_rc = (sy + H - 1) * RX + (sx + HX - 1);
            b_mp = Lay::mp_index(sx, sy);
        }
    }
    const int rc = (py + H) * RX + 2 * px + HX;
    const int mp0 = Lay::mp_index(2 * px + 1, py + 1), mp1 = Lay::mp_index(2 * px + 2, py + 1);
    const unsigned xm1 = unsigned(wrapc(xo - 1, nx)), xc = unsigned(wrapc(xo, nx));
    const unsigned xp1 = AL ? xc + 1 : unsigned(wrapc(xo + 1, nx)), xp2 = unsigned(wrapc(xo + 2, nx));
    const unsigned yr[3] = {unsigned(wrapc(yo - 1, ny)) * unsigned(nx), unsigned(wrapc(yo, ny)) * unsigned(nx),
                            unsigned(wrapc(yo + 1, ny)) * unsigned(nx)};

    unsigned ld_off = unsigned(wrapc(z0 - LAG, nz)) * plane;
    unsigned zr[3] = {unsigned(wrapc(z0 - 1, nz)) * plane, unsigned(wrapc(z0, nz)) * plane,
                      unsigned(wrapc(z0 + 1, nz)) * plane};
    auto advance = [&](unsigned& v) {
        v += plane;
        if (v == vol) v = 0;
    };
    float2 rn[NA];
    auto issue = [&]() {
#pragma unroll
        for (int m = 0; m < NA; ++m) {
            if (tid + m * NTH < NIT) {
                const unsigned q = ld_off + a_in[m];
                LB_GUARD(q + W - 1 < vol, BK_B3_LOAD, q, rn[m] = make_float2(0.f, 0.f); continue)
                if constexpr (AL) rn[m] = reinterpret_cast<const float2*>(a.phi)[q >> 1];
                else rn[m].x = a.phi[q];
            }
        }
        advance(ld_off);
    };
    issue();
    // population k (f_0..f_18, g_0..g_18) of the own pair of the plane collided next
    auto load = [&](int k) -> P2 {
        const unsigned q = unsigned(k) * pitch + zr[1] + yr[1];
        LB_GUARD(zr[1] + yr[1] + xc < vol && zr[1] + yr[1] + xp1 < vol, BK_B3_LOAD, zr[1] + yr[1] + xc, return pp(0.f))
        if constexpr (AL) return P2{reinterpret_cast<const float2*>(src)[(q + xc) >> 1]};
        else return pp(src[q + xc], src[q + xp1]);
    };

    lbk::StencilAcc<float> acc{0, 0, 0, 0, 0, 0, 0};
    lbk::StencilAcc2 acc2{pp(0.f), pp(0.f), pp(0.f), pp(0.f), pp(0.f), pp(0.f), pp(0.f)};
    P2 gacc1[3] = {pp(0.f), pp(0.f), pp(0.f)}, gacc2[3] = {pp(0.f), pp(0.f), pp(0.f)};
    P2 Gc[3] = {pp(0.f), pp(0.f), pp(0.f)}, lapc = pp(0.f), c1 = pp(0.f), c2 = pp(0.f);
    bool bad = false;

    for (int p = z0 - LAG; p < z1 + LAG; ++p) {
        const int it = p - (z0 - LAG), s = p - LAG;
        float* phi_p = phi_s + (it & 1) * Lay::RN;
#pragma unroll
        for (int m = 0; m < NA; ++m) {
            const int k = tid + m * NTH;
            if (k < NIT) {
                if constexpr (AL) *reinterpret_cast<float2*>(phi_p + 2 * k) = rn[m];
                else phi_p[k] = rn[m].x;
            }
        }
        if (p + 1 < z1 + LAG) issue();
        P2 f[19];
        if (s >= z0) {
#pragma unroll
            for (int i = 0; i < 19; ++i) f[i] = load(i);
        }
        __syncthreads();

        // stencil parts of plane p; gradient, Laplacian and M' of plane p - 1
        const bool assemble = it >= 2;
        P2 Gn[3], lapn, cn;
        {
            const lbk::PlaneParts2 cur = lbk::plane_parts2(phi_p, rc, RX);
            cn = cur.c;
            if (assemble) {
                lbk::finish2(acc2, cur, Gn, lapn);
                if constexpr (FORCING) {
#pragma unroll
                    for (int m = 0; m < 2; ++m) {
                        const float gx = m ? Gn[0].v.y : Gn[0].v.x, gy = m ? Gn[1].v.y : Gn[1].v.x,
                                    gz = m ? Gn[2].v.y : Gn[2].v.x;
                        const float hk = 0.5f * pk * (gx * gx + gy * gy + gz * gz);
                        const int at = m ? mp1 : mp0;
                        mpA[at] = make_float4(pk * gx * gx - hk, pk * gx * gy, pk * gx * gz, pk * gy * gy - hk);
                        mpB[at] = make_float2(pk * gy * gz, pk * gz * gz - hk);
                    }
                }
            }
            lbk::start2(acc2, cur);
            if constexpr (FORCING) {
                if (b_rc >= 0) {
                    const lbk::PlaneParts<float> cr = lbk::plane_parts(phi_p, b_rc, RX);
                    if (assemble) {
                        float G[3], lap;
                        lbk::finish(acc, cr, G, lap);
                        const float hk = 0.5f * pk * (G[0] * G[0] + G[1] * G[1] + G[2] * G[2]);
                        mpA[b_mp] = make_float4(pk * G[0] * G[0] - hk, pk * G[0] * G[1], pk * G[0] * G[2],
                                                pk * G[1] * G[1] - hk);
                        mpB[b_mp] = make_float2(pk * G[1] * G[2], pk * G[2] * G[2] - hk);
                    }
                    lbk::start(acc, cr);
                }
            }
        }
        P2 gf[3] = {pp(0.f), pp(0.f), pp(0.f)};
        if constexpr (FORCING) {
            __syncthreads();
            if (assemble) lbk::pair_force_parts<Lay>(mpA, mpB, 2 * px, py + 1, gacc1, gacc2, gf);
        }

        if (s >= z0) {
            const P2 phi = FORCING ? c2 : c1;
            const P2 lap = FORCING ? lapc : lapn;
            auto store = [&](auto I, int set, P2 v) {
                constexpr int i = decltype(I)::value;
                constexpr int ex = L::ex(i), ey = L::ey(i), ez = L::ez(i);
                const unsigned row = unsigned(set + i) * pitch + zr[1 + ez] + yr[1 + ey];
                const unsigned xa = ex == 0 ? xc : (ex == 1 ? xp1 : xm1), xb = ex == 0 ? xp1 : (ex == 1 ? xp2 : xc);
                LB_GUARD(zr[1 + ez] + yr[1 + ey] + xa < vol && zr[1 + ez] + yr[1 + ey] + xb < vol, BK_B3_STORE,
                         zr[1 + ez] + yr[1 + ey] + xa, return)
                if constexpr (AL && ex == 0) {
                    reinterpret_cast<float2*>(dst)[(row + xc) >> 1] = v.v;
                } else {
                    dst[row + xa] = v.v.x;
                    if (own1) dst[row + xb] = v.v.y;
                }
            };
            P2 rho, j[3] = {pp(0.f), pp(0.f), pp(0.f)};
            rho = f[0] + lbk::tree_sum<1, 19>(f);
            static_for<1, 19>([&](auto I) {
                constexpr int i = decltype(I)::value, o = lbk::opposite<L>(i);
                if constexpr (i < o) {
                    const P2 d = f[i] - f[o];
                    lbk::add_signed2<L::ex(i)>(j[0], d);
                    lbk::add_signed2<L::ey(i)>(j[1], d);
                    lbk::add_signed2<L::ez(i)>(j[2], d);
                }
            });
            bad |= (own && (!(rho.v.x > 0.f) || !isfinite(rho.v.x))) || (own1 && (!(rho.v.y > 0.f) || !isfinite(rho.v.y)));
            const P2 ir = pp(1.0f / rho.v.x, 1.0f / rho.v.y);
            P2 u[3], v[3], m[3];
#pragma unroll
            for (int c = 0; c < 3; ++c) {
                u[c] = j[c] * ir;
                v[c] = FORCING ? fma(pp(0.5f) * ir, gf[c], u[c]) : u[c];   // Eq. 40
                m[c] = phi * v[c];
            }
            const P2 phi2 = phi * phi;
            const P2 kl = pp(pk) * lap;
            // p0 - kappa phi lap(phi), p0 = rho/3 + A/2 phi^2 + 3B/4 phi^4
            const P2 iso = fma(phi2, fma(pp(0.75f * a.B), phi2, pp(0.5f * a.A)), fma(pp(1.0f / 3.0f), rho, -(phi * kl)));
            const P2 gmu = pp(a.Gamma) * fma(phi, fma(pp(a.B), phi2, pp(a.A)), -kl);
            Form K;
            K.prep<FORCING, !FORCING>(a.omega, j, u, iso, gf, pk, Gn);
            if (own) {
                static_for<1, 19>([&](auto I) {
                    constexpr int i = decltype(I)::value, o = lbk::opposite<L>(i);
                    if constexpr (i < o) {
                        P2 oi, on;
                        K.template out<i>(f[i], f[o], oi, on);
                        store(std::integral_constant<int, i>{}, 0, oi);
                        store(std::integral_constant<int, o>{}, 0, on);
                    }
                });
                store(std::integral_constant<int, 0>{}, 0, K.rest(f[0]));
            }
            P2 g[19];
#pragma unroll
            for (int i = 0; i < 19; ++i) g[i] = load(19 + i);
            K.prep<false, false>(a.omega_phi, m, v, gmu, gf, pk, Gn);
            if (own) {
                static_for<1, 19>([&](auto I) {
                    constexpr int i = decltype(I)::value, o = lbk::opposite<L>(i);
                    if constexpr (i < o) {
                        P2 oi, on;
                        K.template out<i>(g[i], g[o], oi, on);
                        store(std::integral_constant<int, i>{}, 19, oi);
                        store(std::integral_constant<int, o>{}, 19, on);
                    }
                });
                store(std::integral_constant<int, 0>{}, 19, K.rest(g[0]));
            }
            advance(zr[0]);
            advance(zr[1]);
            advance(zr[2]);
        }
        if (FORCING && assemble) {
#pragma unroll
            for (int c = 0; c < 3; ++c) Gc[c] = Gn[c];
            lapc = lapn;
        }
        c2 = c1;
        c1 = cn;
    }
    if (bad) atomicOr(a.status, 1u);
}

}  // namespace lbb

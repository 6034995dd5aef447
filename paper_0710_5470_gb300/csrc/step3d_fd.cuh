// D3Q19 forcing-scheme time step in two passes, two adjacent x sites per thread.
//
//   density_pairs      rho = sum_i f_i of every site into a field of the context;
//   step_kernel3d_fd   the marching step of step3d_pk.cuh, which reads that field
//                      on the tile and its halo instead of summing the halo's
//                      populations.
// The fused kernel recomputes the density of 1.69 sites per site and of four
// planes per z chunk, and for that keeps a plane of raw populations of the whole
// region in flight, the tile's in a stash of 20 to 38 words per pair, and 168
// (16-bit, three CTAs per SM) to 248 registers (float32, two).  Reading a field
// costs one more pass over the populations (16-bit: 44 bytes beside 84, float32: 80
// beside 156) and leaves a kernel that loads a site's populations once, in the turn
// that collides them, without a stash: 12 KB of shared memory, three CTAs per SM for
// either storage, 472 instructions per site where the fused form has 576 (fp16
// deviations).  Both are bound by latency and by the shared-memory pipe (M' of
// twelve sites per pair and plane), so the lighter kernel gains where the fused one
// has fewer CTAs (float32) and where the second pass reads from L2; kern_d3q19_fd.cu has the measurements
// and the lines.  Carries in thread-private shared memory allow four or five CTAs
// per SM but took 75 instead of 67 us (128^3, fp16 deviations).  The density sums
// keep their order: both forms give the same bits.
//
// Odd nx: one site per thread (step_kernel3d_fd1), since pairs would be split by the
// periodic wrap and by every second row's alignment.
#pragma once
#include "chain.cuh"
#include "step3d.cuh"
#include "step3d_pk.cuh"

namespace lbk {

// Density of two sites adjacent in memory per thread: the lattice as a row of
// sites, whatever its shape (the arrays are padded to whole 128-site rows).  MIXED:
// the sums of the step that follows (pair_rho).
template <class S, bool AOS, bool MIXED>
__global__ void __launch_bounds__(256) density_pairs(const StepArgs a, unsigned pairs) {
    chain_begin();
    using IO = PairIO<S>;
    const unsigned t = blockIdx.x * 256u + threadIdx.x;
    if (t >= pairs) return;
    const unsigned q = 2u * t;
    LB_GUARD((long long)q + 1 < a.pitch, BK_WORK, q, return)
    const float2 f0 = reinterpret_cast<const float2*>(a.src_base)[t];
    typename IO::W w[18];
    if constexpr (AOS) {
        const char* b = a.src[1] + size_t(q / AOS_SITES) * (2 * AOS_BLOCK_HALVES) + (q % AOS_SITES) * 2;
#pragma unroll
        for (int i = 0; i < 18; ++i) w[i] = *reinterpret_cast<const unsigned*>(b + i * 2 * AOS_SITES);
    } else {
        static_for<1, 19>([&](auto I) {
            constexpr int i = decltype(I)::value;
            w[i - 1] = IO::ld(a.src[i], q);
        });
    }
    reinterpret_cast<float2*>(a.rho32)[t] = pair_rho<S, MIXED>(f0, w, a.rsum).v;
}

template <int TX, int TY>
struct LayoutFD {
    using PK = LayoutPK<TX, TY, true>;
    static constexpr int NTH = PK::NTH, RX = PK::RX, RY = PK::RY, RN = PK::RN, SN = PK::SN;
    static constexpr size_t OFF_MPA = (size_t(2) * RN * 4 + 15) / 16 * 16;
    static constexpr size_t OFF_MPB = OFF_MPA + size_t(SN) * 16;
    static constexpr size_t BYTES = OFF_MPB + size_t(SN) * 8;
};

template <class S, int TX, int TY, int MINB, bool AOS>
__global__ void __launch_bounds__((TX / 2) * TY, MINB) step_kernel3d_fd(const StepArgs args) {
    chain_begin();
    using L = D3Q19;
    using IO = PairIO<S>;
    using Wd = typename IO::W;
    using Lay = LayoutPK<TX, TY, true>;
    using LF = LayoutFD<TX, TY>;
    constexpr bool RAW16 = IO::RAW16;
    constexpr int H = Lay::H, HX = Lay::HX, TXP = Lay::TXP, NTH = Lay::NTH;
    constexpr int RX = Lay::RX, SX = Lay::SX, NBR = Lay::NBR;
    static_assert(!AOS || RAW16, "interleaved layout: 16-bit storage, nx a multiple of 32");
    constexpr int ROWB = 2 * AOS_SITES;             // bytes of one population row of a block

    extern __shared__ __align__(16) unsigned char smem_raw[];
    float* rho_s = reinterpret_cast<float*>(smem_raw);
    float4* mpA = reinterpret_cast<float4*>(smem_raw + LF::OFF_MPA);   // (Mxx, Mxy, Mxz, Myy)
    float2* mpB = reinterpret_cast<float2*>(smem_raw + LF::OFF_MPB);   // (Myz, Mzz)

    const int nx = args.nx, ny = args.ny, nz = args.nz;
    const int tid = threadIdx.x;
    const int px = tid % TXP, py = tid / TXP;
    const int4 wk = args.work[blockIdx.x];
    const int x0 = wk.x, y0 = wk.y, z0 = wk.z, z1 = wk.w;
    const int plane = nx * ny;
#ifdef LB_DEBUG_BOUNDS
    const size_t nsites = size_t(plane) * nz;   // sites of the lattice
#endif
    const PairPhys ph{args.fa, args.fb, args.fT, args.fkappa, args.fomega, args.fnu, args.pref, args.rsum};
    const float pk = args.fkappa;
    const float* field = args.rho32;

    // ---- region pairs of the density: in-plane element index and place in the slot
    constexpr int NIT = Lay::NIT, NA = (NIT + NTH - 1) / NTH, RXP = Lay::RXP;
    unsigned a_in[NA];
#pragma unroll
    for (int m = 0; m < NA; ++m) {
        const int k = tid + m * NTH;
        a_in[m] = k < NIT ? unsigned(wrapi(y0 - H + k / RXP, ny) * nx + wrapi(x0 - HX + (k % RXP) * 2, nx)) : 0u;
    }
    const int xo = x0 + 2 * px, yo = y0 + py;
    const bool own = xo < nx && yo < ny;
    // ---- ring items of stage B: region index and M' index
    int b_rc[NBR], b_mp[NBR];
#pragma unroll
    for (int m = 0; m < NBR; ++m) {
        int sx = 0, sy = 0;
        const int r = tid + m * NTH;
        if (r < 2 * SX) {
            sx = r % SX;
            sy = r < SX ? 0 : Lay::SY - 1;
        } else {
            const int k = r - 2 * SX;
            sy = 1 + (k >> 1);
            sx = (k & 1) ? SX - 1 : 0;
        }
        b_rc[m] = r < Lay::NRING ? (sy + H - 1) * RX + (sx + HX - 1) : -1;
        b_mp[m] = Lay::mp_index(sx, sy);
    }
    const int rc = (py + H) * RX + 2 * px + HX;
    const int mp0 = Lay::mp_index(2 * px + 1, py + 1), mp1 = Lay::mp_index(2 * px + 2, py + 1);
    // push targets: x columns of the pair's neighbours, row offsets of the pair
    const unsigned xm1 = unsigned(wrapi(xo - 1, nx)), xc = unsigned(wrapi(xo, nx));
    const unsigned xp1 = xc + 1, xp2 = unsigned(wrapi(xo + 2, nx));
    const unsigned yr[3] = {unsigned(wrapi(yo - 1, ny) * nx), unsigned(wrapi(yo, ny) * nx),
                            unsigned(wrapi(yo + 1, ny) * nx)};
    const unsigned q_in = yr[1] + xc;

    const int pstart = z0 - 2, pend = z1 + 2;
    const int vol = nz * plane;
    int ld_off = wrapi(pstart, nz) * plane;
    int zr[3] = {wrapi(z0 - 1, nz) * plane, wrapi(z0, nz) * plane, wrapi(z0 + 1, nz) * plane};
    auto advance = [&](int& v) {
        v += plane;
        if (v == vol) v = 0;
    };
    // density of plane ld_off on the region, one plane ahead
    float2 rn[NA];
    auto issue = [&]() {
#pragma unroll
        for (int m = 0; m < NA; ++m) {
            if (tid + m * NTH < NIT) {
                const unsigned q = unsigned(ld_off) + a_in[m];
                LB_GUARD(size_t(q) + 1 < nsites, BK_WORK, q, rn[m] = make_float2(0.f, 0.f); continue)
                rn[m] = reinterpret_cast<const float2*>(field)[q >> 1];
            }
        }
        advance(ld_off);
    };
    issue();

    StencilAcc<float> acc[NBR];
#pragma unroll
    for (int m = 0; m < NBR; ++m) acc[m] = StencilAcc<float>{0, 0, 0, 0, 0, 0, 0};
    StencilAcc2 acc2{pp(0.f), pp(0.f), pp(0.f), pp(0.f), pp(0.f), pp(0.f), pp(0.f)};
    // body force carries of the own pair: -(U0(q-1) + U-(q-2)) and -U-(q-1)
    P2 gacc1[3] = {pp(0.f), pp(0.f), pp(0.f)}, gacc2[3] = {pp(0.f), pp(0.f), pp(0.f)};
    // G, lap and rho of the own pair one and (rho) two planes back
    P2 Gc[3] = {pp(0.f), pp(0.f), pp(0.f)}, lapc = pp(0.f), c1 = pp(0.f), c2 = pp(0.f);
    bool bad = false;

    for (int p = pstart; p < pend; ++p) {
        const int it = p - pstart;
        const int s = p - 2;
        // ---------------- density of plane p into its slot; loads of plane p + 1 and
        // of the own pair's populations of plane s, collided at the end of this turn
        float* rho_p = rho_s + (it & 1) * Lay::RN;
#pragma unroll
        for (int m = 0; m < NA; ++m) {
            const int k = tid + m * NTH;
            if (k < NIT) *reinterpret_cast<float2*>(rho_p + 2 * k) = rn[m];
        }
        if (p + 1 < pend) issue();
        float2 f0 = make_float2(0.f, 0.f);
        Wd w[18];
        if (s >= z0) {
            const unsigned q = unsigned(zr[1]) + q_in;
#ifdef LB_DEBUG_BOUNDS
            if (lbk::in_bounds(size_t(q) + 1 < nsites, BK_PK_LOAD, q))
#endif
            {
                f0 = reinterpret_cast<const float2*>(args.src_base)[q >> 1];
                if constexpr (AOS) {
                    const char* b = args.src[1] + size_t(q / AOS_SITES) * (2 * AOS_BLOCK_HALVES) + (q % AOS_SITES) * 2;
#pragma unroll
                    for (int i = 0; i < 18; ++i) w[i] = *reinterpret_cast<const unsigned*>(b + i * ROWB);
                } else {
                    static_for<1, 19>([&](auto I) {
                        constexpr int i = decltype(I)::value;
                        w[i - 1] = IO::ld(args.src[i], q);
                    });
                }
            }
        }
        __syncthreads();

        // ---------------- stage B: stencil parts of plane p; G, lap, M' of plane q = p - 1
        const bool assemble = it >= 2;
        P2 Gn[3], lapn, cn;
        {
            const PlaneParts2 cur = plane_parts2(rho_p, rc, RX);
            cn = cur.c;
            if (assemble) {
                finish2(acc2, cur, Gn, lapn);
#pragma unroll
                for (int m = 0; m < 2; ++m) {
                    const float G[3] = {m ? Gn[0].v.y : Gn[0].v.x, m ? Gn[1].v.y : Gn[1].v.x,
                                        m ? Gn[2].v.y : Gn[2].v.x};
                    const float g2 = G[0] * G[0] + G[1] * G[1] + G[2] * G[2];
                    const float hk = 0.5f * pk * g2;
                    const int at = m ? mp1 : mp0;
                    LB_GUARD(at >= 0 && at < Lay::SN, BK_PK_SHARED, at, continue)
                    mpA[at] = make_float4(pk * G[0] * G[0] - hk, pk * G[0] * G[1], pk * G[0] * G[2],
                                          pk * G[1] * G[1] - hk);
                    mpB[at] = make_float2(pk * G[1] * G[2], pk * G[2] * G[2] - hk);
                }
            }
            start2(acc2, cur);
#pragma unroll
            for (int m = 0; m < NBR; ++m) {
                if (b_rc[m] < 0) continue;
                const PlaneParts<float> cr = plane_parts(rho_p, b_rc[m], RX);
                if (assemble) {
                    float G[3], lap;
                    finish(acc[m], cr, G, lap);
                    const float g2 = G[0] * G[0] + G[1] * G[1] + G[2] * G[2];
                    const float hk = 0.5f * pk * g2;
                    LB_GUARD(b_mp[m] >= 0 && b_mp[m] < Lay::SN, BK_PK_SHARED, b_mp[m], continue)
                    mpA[b_mp[m]] = make_float4(pk * G[0] * G[0] - hk, pk * G[0] * G[1], pk * G[0] * G[2],
                                               pk * G[1] * G[1] - hk);
                    mpB[b_mp[m]] = make_float2(pk * G[1] * G[2], pk * G[2] * G[2] - hk);
                }
                start(acc[m], cr);
            }
        }
        __syncthreads();

        // ---------------- body force of the own pair: parts of plane q (Eq. 28)
        P2 gf[3] = {pp(0.f), pp(0.f), pp(0.f)};
        if (assemble) pair_force_parts<Lay>(mpA, mpB, 2 * px, py + 1, gacc1, gacc2, gf);

        // ---------------- stage C: collide and push plane s = p - 2
        if (s >= z0) {
            const P2 rho = c2;
            const P2 G[3] = {Gc[0], Gc[1], Gc[2]};
            bad |= own && (!(rho.v.x > 0.f) || !(rho.v.x < 1e30f) || !(rho.v.y > 0.f) || !(rho.v.y < 1e30f));
            P2 j[3];
            if constexpr (RAW16) pair_momentum_mixed<S>(w, j);
            else pair_momentum<S>(w, j);
            PairColl K;
            K.prep(rho, j, G, lapc, gf, ph);
            if (own) {
                // push f*_i(r) to r + e_i: populations with e_x = 0 as aligned pairs, the
                // others site by site (joined to aligned words by shuffles they took 75
                // instead of 67 us at 128^3, fp16 deviations)
                size_t zb[3] = {0, 0, 0};
                unsigned yb[3] = {0, 0, 0}, cb[4] = {0, 0, 0, 0};
                if constexpr (AOS) {
#pragma unroll
                    for (int k = 0; k < 3; ++k) {
                        zb[k] = size_t(unsigned(zr[k])) / AOS_SITES * (2 * AOS_BLOCK_HALVES);
                        yb[k] = yr[k] / AOS_SITES * (2 * AOS_BLOCK_HALVES);
                    }
                    cb[0] = aos_bytes(xm1);
                    cb[1] = aos_bytes(xc);
                    cb[2] = aos_bytes(xp1);
                    cb[3] = aos_bytes(xp2);
                }
                auto store = [&](auto I, P2 v) {
                    constexpr int i = decltype(I)::value;
                    constexpr int ex = L::ex(i), ey = L::ey(i), ez = L::ez(i);
                    [[maybe_unused]] const unsigned row = unsigned(zr[1 + ez]) + yr[1 + ey];
                    [[maybe_unused]] const unsigned xa = ex == 0 ? xc : (ex == 1 ? xp1 : xm1), xb = ex == 0 ? xp1 : (ex == 1 ? xp2 : xc);
                    LB_GUARD(size_t(row) + xa < nsites && size_t(row) + xb < nsites, BK_PK_STORE, row + xa, return)
                    if constexpr (AOS) {
                        char* b = args.dst[1] + zb[1 + ez] + yb[1 + ey] + (i - 1) * ROWB;
                        if constexpr (ex == 0) {
                            IO::st2p(b + cb[1], v);
                        } else if constexpr (ex == 1) {
                            IO::st1p(b + cb[2], v.v.x);
                            IO::st1p(b + cb[3], v.v.y);
                        } else {
                            IO::st1p(b + cb[0], v.v.x);
                            IO::st1p(b + cb[1], v.v.y);
                        }
                    } else if constexpr (ex == 0) {
                        IO::st2(args.dst[i], row + xc, v);
                    } else {
                        IO::st1(args.dst[i], row + xa, v.v.x);
                        IO::st1(args.dst[i], row + xb, v.v.y);
                    }
                };
                const P2 o0 = fma(K.omw, P2{f0}, K.c0);
                const unsigned q = unsigned(zr[1]) + q_in;
#ifdef LB_DEBUG_BOUNDS
                if (lbk::in_bounds(size_t(q) + 1 < nsites, BK_PK_STORE, q))
#endif
                    reinterpret_cast<float2*>(args.dst_base)[q >> 1] = o0.v;
                static_for<1, 19>([&](auto I) {
                    constexpr int i = decltype(I)::value;
                    constexpr int o = opposite<L>(i);
                    if constexpr (i < o) {
                        P2 oi, on;
                        K.template out<i>(IO::dec(w[i - 1]), IO::dec(w[o - 1]), oi, on);
                        store(std::integral_constant<int, i>{}, oi);
                        store(std::integral_constant<int, o>{}, on);
                    }
                });
            }
            advance(zr[0]);
            advance(zr[1]);
            advance(zr[2]);
        }
        if (assemble) {
#pragma unroll
            for (int c = 0; c < 3; ++c) Gc[c] = Gn[c];
            lapc = lapn;
        }
        c2 = c1;
        c1 = cn;
    }
    if (bad) atomicOr(args.status, 1u);
}

// The same step for an odd nx, one site per thread: the arithmetic of step_kernel3d
// (step3d.cuh) function by function, the density pass in its order too, so that both
// forms give the same bits; a last-bit difference would flip roundings to 16 bits.  A
// thread carries its own site's gradient and density in registers and takes at most one of
// the ring's sites; no stash, 6 KB of shared memory, four CTAs of 32 x 4 sites per SM (126
// registers).  Measured on a GB300, us per step at 101 x 75 x 53, bf16 deviations: one-site
// fused kernel 29.1, this 20.8, 32 x 8 tiles with two CTAs per SM 22.6, 32 x 4 with five
// 22.7, pairs split site by site 22.7.
template <class S, int TX, int TY, int MINB>
__global__ void __launch_bounds__(TX* TY, MINB) step_kernel3d_fd1(const StepArgs args) {
    chain_begin();
    using L = D3Q19;
    constexpr int Q = 19, H = 2, NT = TX * TY;
    constexpr int RX = TX + 2 * H, RY = TY + 2 * H, RN = RX * RY;
    constexpr int SX = TX + 2, SY = TY + 2, SN = SX * SY, NRING = SN - NT;
    constexpr int NA = (RN + NT - 1) / NT;
    static_assert(NRING <= NT, "one ring site per thread");
    __shared__ float rho_s[2 * RN];
    __shared__ __align__(16) float mpA[4 * SN];   // (Mxx, Mxy, Mxz, Myy) per ring-1 site
    __shared__ __align__(8) float mpB[2 * SN];    // (Myz, Mzz) per ring-1 site

    const int nx = args.nx, ny = args.ny, nz = args.nz;
    const int tid = threadIdx.x, tx = tid % TX, ty = tid / TX;
    const int4 wk = args.work[blockIdx.x];
    const int x0 = wk.x, y0 = wk.y, z0 = wk.z, z1 = wk.w;
    const int plane = nx * ny, vol = nz * plane;
    const float pk = args.fkappa;

    int a_in[NA];
#pragma unroll
    for (int m = 0; m < NA; ++m) {
        const int k = tid + m * NT;
        a_in[m] = k < RN ? wrapi(y0 - H + k / RX, ny) * nx + wrapi(x0 - H + k % RX, nx) : 0;
    }
    // stage-B sites: the own one and, for the first NRING threads, one of the ring
    const int rc = (ty + H) * RX + tx + H, kc = (ty + 1) * SX + tx + 1;
    int b_rc = -1, b_k = 0;
    if (tid < NRING) {
        int sx, sy;
        if (tid < 2 * SX) {
            sx = tid % SX;
            sy = tid < SX ? 0 : SY - 1;
        } else {
            const int k = tid - 2 * SX;
            sy = 1 + (k >> 1);
            sx = (k & 1) ? SX - 1 : 0;
        }
        b_rc = (sy + H - 1) * RX + (sx + H - 1);
        b_k = sy * SX + sx;
    }
    const int xs = x0 + tx, ys = y0 + ty;
    const bool own = xs < nx && ys < ny;
    const int xw[3] = {wrapi(xs - 1, nx), wrapi(xs, nx), wrapi(xs + 1, nx)};
    const int yr[3] = {wrapi(ys - 1, ny) * nx, wrapi(ys, ny) * nx, wrapi(ys + 1, ny) * nx};

    const int pstart = z0 - 2, pend = z1 + 2;
    int ld_off = wrapi(pstart, nz) * plane;
    int zr[3] = {wrapi(z0 - 1, nz) * plane, wrapi(z0, nz) * plane, wrapi(z0 + 1, nz) * plane};
    auto advance = [&](int& v) {
        v += plane;
        if (v == vol) v = 0;
    };
    float rn[NA];
    auto issue = [&]() {   // density of plane ld_off on the region
#pragma unroll
        for (int m = 0; m < NA; ++m) {
            if (tid + m * NT < RN) {
                const unsigned q = unsigned(ld_off + a_in[m]);
                LB_GUARD(q < unsigned(vol), BK_WORK, q, rn[m] = 0.f; continue)
                rn[m] = args.rho32[q];
            }
        }
        advance(ld_off);
    };
    issue();

    StencilAcc<float> acc{0, 0, 0, 0, 0, 0, 0}, accr{0, 0, 0, 0, 0, 0, 0};   // own site, ring site
    float gacc1[3] = {0, 0, 0}, gacc2[3] = {0, 0, 0};
    float Gc[3] = {0, 0, 0}, lapc = 0, c1 = 0, c2 = 0;   // G, lap one plane back, rho one and two
    bool bad = false;

    for (int p = pstart; p < pend; ++p) {
        const int it = p - pstart, s = p - 2;
        float* rho_p = rho_s + (it & 1) * RN;
#pragma unroll
        for (int m = 0; m < NA; ++m)
            if (tid + m * NT < RN) rho_p[tid + m * NT] = rn[m];
        if (p + 1 < pend) issue();
        typename S::raw0 r0{};
        typename S::rawi ri[Q - 1];
        if (s >= z0) {   // populations of the site collided at the end of this turn
            const unsigned q = unsigned(zr[1] + yr[1] + xw[1]);
#ifdef LB_DEBUG_BOUNDS
            if (lbk::in_bounds(q < unsigned(vol), BK_3D_LOAD, q))
#endif
            {
                r0 = S::ld0(args.src[0], q);
                static_for<1, Q>([&](auto I) {
                    constexpr int i = decltype(I)::value;
                    ri[i - 1] = S::ldi(args.src[i], q);
                });
            }
        }
        __syncthreads();

        // ---------------- stage B: stencil parts of plane p; G, lap and M' of plane p - 1
        const bool assemble = it >= 2;
        float Gn[3] = {0, 0, 0}, lapn = 0, cn;
        {
            auto put = [&](int k, const float (&G)[3]) {
                const float g2 = G[0] * G[0] + G[1] * G[1] + G[2] * G[2];
                const float hk = 0.5f * pk * g2;
                LB_GUARD(k >= 0 && k < SN, BK_PK_SHARED, k, return)
                st4(mpA + 4 * k, pk * G[0] * G[0] - hk, pk * G[0] * G[1], pk * G[0] * G[2], pk * G[1] * G[1] - hk);
                st_pair(mpB + 2 * k, pk * G[1] * G[2], pk * G[2] * G[2] - hk);
            };
            const PlaneParts<float> cur = plane_parts(rho_p, rc, RX);
            cn = cur.c;
            if (assemble) {
                finish(acc, cur, Gn, lapn);
                put(kc, Gn);
            }
            start(acc, cur);
            if (b_rc >= 0) {
                const PlaneParts<float> cr = plane_parts(rho_p, b_rc, RX);
                if (assemble) {
                    float G[3], lap;
                    finish(accr, cr, G, lap);
                    put(b_k, G);
                }
                start(accr, cr);
            }
        }
        __syncthreads();

        // ---------------- body force: parts of plane p - 1 (Eq. 28)
        float gf[3] = {0, 0, 0};
        if (assemble) site_force_parts(mpA, mpB, kc, SX, gacc1, gacc2, gf);

        // ---------------- stage C: collide and push plane s = p - 2
        if (s >= z0) {
            if (own) {
                float f[Q], out[Q];
                f[0] = S::dec0(r0);
                static_for<1, Q>([&](auto I) {
                    constexpr int i = decltype(I)::value;
                    f[i] = S::devi(ri[i - 1]);
                });
                bad |= !(c2 > 0.f) || !(c2 < 1e30f);
                collide<L, true, float>(f, c2, Gc, lapc, gf, args.fa, args.fb, args.fT, pk, args.fomega, args.fnu,
                                        args.pref, args.rsum, out);
                static_for<0, Q>([&](auto I) {
                    constexpr int i = decltype(I)::value;
                    const int idx = zr[1 + L::ez(i)] + yr[1 + L::ey(i)] + xw[1 + L::ex(i)];
                    LB_GUARD(idx >= 0 && idx < vol, BK_3D_STORE, idx, return)
                    if constexpr (i == 0) S::st0(args.dst[0], size_t(idx), out[0]);
                    else S::sti(args.dst[i], size_t(idx), out[i]);
                });
            }
            advance(zr[0]);
            advance(zr[1]);
            advance(zr[2]);
        }
        if (assemble) {
#pragma unroll
            for (int c = 0; c < 3; ++c) Gc[c] = Gn[c];
            lapc = lapn;
        }
        c2 = c1;
        c1 = cn;
    }
    if (bad) atomicOr(args.status, 1u);
}

}  // namespace lbk

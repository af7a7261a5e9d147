// step_d3q27.cuh -- fused pull-stream + FP central-moment collision of the coupled D3Q27 flow
// (Sec. 5.1-5.2) and D3Q15 energy (Appendix C) lattices, one node per thread.
//
// D3Q27: the 27 central moments kappa_abc are produced by three sweeps of 3-link lines (x, y, z),
// which on the tensor-product lattice equals P then F; the inverse sweeps map back.
// D3Q15: raw moments come from the six axis links in pairs and from an 8-point Walsh-Hadamard
// transform of the corner links (the structure of App. C Step 1); the central shift and its exact
// inverse are applied axis by axis (Steps 2 and 4, including the aliased moment 220).
//
// Deviation form: the kernel carries delta_a = f_a - w_a and gamma_b = g_b - w_b T_o.  The central
// moments of f are those of the rest populations at the velocity u, K_abc = W_a(ux) W_b(uy)
// W_c(uz) with W_0 = 1, W_1 = -u, W_2 = 1/3 + u^2, plus the central moments D_abc of delta; the
// flow relaxation is written for the deviations with the O(1) parts of K (the moments even in
// every direction) cancelled analytically, so the FP32 arithmetic resolves the small departures
// from rest.
#pragma once

#include "lattices.cuh"
#include "lbm_common.cuh"

#ifndef LBM_MAXREG3D
#define LBM_MAXREG3D Launch3D<S, kRates>::kMaxRegs
#endif

namespace lbm {

template <class R>
using Coeffs3D = Coeffs<R, 27, 15>;

// D3Q15 link b for D3Q27 link a, or -1.
__host__ __device__ constexpr int g15_of_27(int a)
{
    return a < 7 ? a : (a >= 19 ? a - 12 : -1);
}

template <class S, class Idx = size_t, int kPull = kPullDev>
__device__ __forceinline__ void pull_d3q27_d3q15(const typename S::T* __restrict__ fin,
                                                 const typename S::T* __restrict__ gin,
                                                 const Geometry& geo,
                                                 const NodeWalls<typename S::R>& w, int i,
                                                 typename S::R T_ref, typename S::R f[27],
                                                 typename S::R g[15])
{
    using R = typename S::R;
    static_for<27>([&](auto A) {
        constexpr int a = decltype(A)::value;
        constexpr int o = opp27(a);
        bool out, dir;
        R tw;
        const int s = link_source<e27(a, 0), e27(a, 1), e27(a, 2)>(geo, w, i, &out, &dir, &tw);
        const Idx off = out ? (Idx)o * geo.n + i : (Idx)a * geo.n + s;
        f[a] = load_link<S, kPull>(fin, off, R(w27(a)));
        constexpr int b = g15_of_27(a);
        if constexpr (b >= 0) {
            constexpr int ob = opp15(b);
            const Idx og = out ? (Idx)ob * geo.n + i : (Idx)b * geo.n + s;
            const R gv = load_link<S, kPull>(gin, og, R(w15(b)) * T_ref);
            g[b] = dir ? anti_bounce<S, kPull>(gv, w15(b), tw, T_ref) : gv;
        }
    });
}

// The same pull at a node whose 26 neighbours all lie inside the box (no wall, no wrap).
template <class S, class Idx = size_t, int kPull = kPullDev>
__device__ __forceinline__ void pull_d3q27_d3q15_interior(const typename S::T* __restrict__ fin,
                                                          const typename S::T* __restrict__ gin,
                                                          const Geometry& geo, int i,
                                                          typename S::R T_ref, typename S::R f[27],
                                                          typename S::R g[15])
{
    using R = typename S::R;
    static_for<27>([&](auto A) {
        constexpr int a = decltype(A)::value;
        const int s = i - (e27(a, 0) + e27(a, 1) * geo.nx + e27(a, 2) * geo.nxy);
        f[a] = load_link<S, kPull>(fin, (Idx)((Idx)a * geo.n + s), R(w27(a)));
        constexpr int b = g15_of_27(a);
        if constexpr (b >= 0) g[b] = load_link<S, kPull>(gin, (Idx)((Idx)b * geo.n + s), R(w15(b)) * T_ref);
    });
}

// Links of a node on an x wall (or x wrap) that leave the box through x, replaced by the wall
// rules (or the wrapped source) from global memory; the other links keep their staged values.
template <class S, class Idx, int kPull>
__device__ __forceinline__ void fix_x_edge_d3q27(const typename S::T* __restrict__ fin,
                                                 const typename S::T* __restrict__ gin,
                                                 const Geometry& geo, int x, int y, int z, int i,
                                                 typename S::R T_ref, typename S::R f[27],
                                                 typename S::R g[15])
{
    using R = typename S::R;
    const NodeWalls<R> w = node_walls_x<R>(geo, x, y, z);
    static_for<27>([&](auto A) {
        constexpr int a = decltype(A)::value;
        constexpr int ex = e27(a, 0);
        if constexpr (ex != 0) {
            const bool leaves = ex == 1 ? x == 0 : x == geo.nx - 1;
            if (leaves) {
                constexpr int o = opp27(a);
                bool out, dir;
                R tw;
                const int s = link_source<ex, e27(a, 1), e27(a, 2)>(geo, w, i, &out, &dir, &tw);
                const Idx off = out ? (Idx)o * geo.n + i : (Idx)a * geo.n + s;
                f[a] = load_link<S, kPull>(fin, off, R(w27(a)));
                constexpr int b = g15_of_27(a);
                if constexpr (b >= 0) {
                    constexpr int ob = opp15(b);
                    const Idx og = out ? (Idx)ob * geo.n + i : (Idx)b * geo.n + s;
                    const R gv = load_link<S, kPull>(gin, og, R(w15(b)) * T_ref);
                    g[b] = dir ? anti_bounce<S, kPull>(gv, w15(b), tw, T_ref) : gv;
                }
            }
        }
    });
}

// Flow collision (reading R6 of the oracle notes) on the deviations: D[c][b][a] = kappa_abc - K_abc
// on entry, kappa~_abc - K_abc on exit.  Rate slots follow the moment order of Sec. 5.2; slot 7
// relaxes the trace (bulk), slots 8 and 9 the deviators kappa_200 - kappa_020, kappa_200 - kappa_002.
// Sources (Eq. forcing:3D) use the full pre-collision moments kappa = K + D.
// kUnit: the rates are those of lbm_create (every rate 1 except the shear ones, slots 4-6, 8, 9;
// unit_flow_rates), which the host has checked.  A moment relaxed at rate 1 lands on its attractor
// plus half its source, so its pre-collision value drops out of its own update (order 6 drops out
// entirely).
template <bool kUnit = false, class R>
__device__ __forceinline__ void relax_f_d3q27(R D[3][3][3], R drho, R irho, R ux, R uy, R uz, R Fx,
                                              R Fy, R Fz, const Coeffs3D<R>& c)
{
    const R hu = R(0.5);   // 1 - omega / 2 at omega = 1
#define DD(a, b, cc) D[cc][b][a]
    const R* om = c.om_f;
    const R* h = c.hf;
    const R third = R(1.0 / 3.0);
    const R Fxr = Fx * irho, Fyr = Fy * irho, Fzr = Fz * irho;
    // rest moments at u: W_2 per axis, products of W_1
    const R A = third + ux * ux, B = third + uy * uy, C = third + uz * uz;
    const R xy = ux * uy, xz = ux * uz, yz = uy * uz;

    // pre-collision deviations
    const R d000 = DD(0, 0, 0), d100 = DD(1, 0, 0), d010 = DD(0, 1, 0), d001 = DD(0, 0, 1);
    const R d110 = DD(1, 1, 0), d101 = DD(1, 0, 1), d011 = DD(0, 1, 1);
    const R d200 = DD(2, 0, 0), d020 = DD(0, 2, 0), d002 = DD(0, 0, 2);
    const R d120 = DD(1, 2, 0), d102 = DD(1, 0, 2), d210 = DD(2, 1, 0), d012 = DD(0, 1, 2);
    const R d201 = DD(2, 0, 1), d021 = DD(0, 2, 1), d111 = DD(1, 1, 1);
    const R d220 = DD(2, 2, 0), d202 = DD(2, 0, 2), d022 = DD(0, 2, 2);
    const R d211 = DD(2, 1, 1), d121 = DD(1, 2, 1), d112 = DD(1, 1, 2);
    const R d122 = DD(1, 2, 2), d212 = DD(2, 1, 2), d221 = DD(2, 2, 1), d222 = DD(2, 2, 2);

    // full pre-collision moments needed by the sources
    const R k110 = xy + d110, k101 = xz + d101, k011 = yz + d011;
    const R k200 = A + d200, k020 = B + d020, k002 = C + d002;
    const R k120 = d120 - ux * B, k102 = d102 - ux * C, k210 = d210 - A * uy;
    const R k012 = d012 - uy * C, k201 = d201 - A * uz, k021 = d021 - B * uz;
    const R k111 = d111 - xy * uz;
    const R k220 = A * B + d220;
    const R k211 = A * yz + d211, k121 = B * xz + d121, k112 = C * xy + d112;
    const R k022 = B * C + d022, k202 = A * C + d202;
    const R k122 = d122 - ux * B * C, k212 = d212 - A * uy * C, k221 = d221 - A * B * uz;

    // orders 0 and 1 (K_000 = 1, K_100 = -ux, ...)
    const R t000 = kUnit ? drho : d000 + om[0] * (drho - d000);
    const R t100 = kUnit ? ux + hu * Fx : d100 - om[1] * (d100 - ux) + h[1] * Fx;
    const R t010 = kUnit ? uy + hu * Fy : d010 - om[2] * (d010 - uy) + h[2] * Fy;
    const R t001 = kUnit ? uz + hu * Fz : d001 - om[3] * (d001 - uz) + h[3] * Fz;

    // order 2: off-diagonal toward 0, trace toward rho, deviators toward 0
    const R t110 = d110 - om[4] * (d110 + xy);
    const R t101 = d101 - om[5] * (d101 + xz);
    const R t011 = d011 - om[6] * (d011 + yz);
    const R dtr = d200 + d020 + d002;
    const R dd1 = d200 - d020, dd2 = d200 - d002;
    const R ttr = kUnit ? drho - (ux * ux + uy * uy + uz * uz)
                        : dtr + om[7] * (drho - (ux * ux + uy * uy + uz * uz) - dtr);
    const R td1 = dd1 - om[8] * (dd1 + ux * ux - uy * uy);
    const R td2 = dd2 - om[9] * (dd2 + ux * ux - uz * uz);
    const R t200 = third * (ttr + td1 + td2);
    const R t020 = third * (ttr - R(2) * td1 + td2);
    const R t002 = third * (ttr + td1 - R(2) * td2);

    // order 3: attractors zero (at rate 1 the deviation is -K plus half the source)
    const R s120 = Fxr * k020 + R(2) * Fyr * k110, s102 = Fxr * k002 + R(2) * Fzr * k101;
    const R s210 = R(2) * Fxr * k110 + Fyr * k200, s012 = Fyr * k002 + R(2) * Fzr * k011;
    const R s201 = R(2) * Fxr * k101 + Fzr * k200, s021 = R(2) * Fyr * k011 + Fzr * k020;
    const R s111 = Fxr * k011 + Fyr * k101 + Fzr * k110;
    const R t120 = kUnit ? ux * B + hu * s120 : d120 - om[10] * k120 + h[10] * s120;
    const R t102 = kUnit ? ux * C + hu * s102 : d102 - om[11] * k102 + h[11] * s102;
    const R t210 = kUnit ? A * uy + hu * s210 : d210 - om[12] * k210 + h[12] * s210;
    const R t012 = kUnit ? uy * C + hu * s012 : d012 - om[13] * k012 + h[13] * s012;
    const R t201 = kUnit ? A * uz + hu * s201 : d201 - om[14] * k201 + h[14] * s201;
    const R t021 = kUnit ? B * uz + hu * s021 : d021 - om[15] * k021 + h[15] * s021;
    const R t111 = kUnit ? xy * uz + hu * s111 : d111 - om[16] * k111 + h[16] * s111;

    // full post-collision moments of orders 2-3 (small, or O(1) only through A, B, C)
    const R p110 = xy + t110, p101 = xz + t101, p011 = yz + t011;
    const R p120 = t120 - ux * B, p102 = t102 - ux * C, p210 = t210 - A * uy;
    const R p012 = t012 - uy * C, p201 = t201 - A * uz, p021 = t021 - B * uz;
    const R p111 = t111 - xy * uz;

    // order 4: attractor minus K, with the O(1) products cancelled
    const R M220 = (A * t020 + B * t200 + t200 * t020 + R(2) * p110 * p110 - A * B * drho) * irho;
    const R M202 = (A * t002 + C * t200 + t200 * t002 + R(2) * p101 * p101 - A * C * drho) * irho;
    const R M022 = (B * t002 + C * t020 + t020 * t002 + R(2) * p011 * p011 - B * C * drho) * irho;
    const R M211 = ((A + t200) * p011 + R(2) * p110 * p101) * irho - A * yz;
    const R M121 = ((B + t020) * p101 + R(2) * p110 * p011) * irho - B * xz;
    const R M112 = ((C + t002) * p110 + R(2) * p011 * p101) * irho - C * xy;
    const R s220 = R(2) * (Fxr * k120 + Fyr * k210), s202 = R(2) * (Fxr * k102 + Fzr * k201);
    const R s022 = R(2) * (Fyr * k012 + Fzr * k021);
    const R s211 = R(2) * Fxr * k111 + Fyr * k201 + Fzr * k210;
    const R s121 = Fxr * k021 + R(2) * Fyr * k111 + Fzr * k120;
    const R s112 = Fxr * k012 + Fyr * k102 + R(2) * Fzr * k111;
    const R t220 = kUnit ? M220 + hu * s220 : d220 + om[17] * (M220 - d220) + h[17] * s220;
    const R t202 = kUnit ? M202 + hu * s202 : d202 + om[18] * (M202 - d202) + h[18] * s202;
    const R t022 = kUnit ? M022 + hu * s022 : d022 + om[19] * (M022 - d022) + h[19] * s022;
    const R t211 = kUnit ? M211 + hu * s211 : d211 + om[20] * (M211 - d211) + h[20] * s211;
    const R t121 = kUnit ? M121 + hu * s121 : d121 + om[21] * (M121 - d121) + h[21] * s121;
    const R t112 = kUnit ? M112 + hu * s112 : d112 + om[22] * (M112 - d112) + h[22] * s112;

    // order 5: attractors from post-collision orders 2 and 3 (K_122 = -ux B C, ...)
    const R f25 = R(2.0 / 5.0) * irho;
    const R q200 = A + t200, q020 = B + t020, q002 = C + t002;
    const R M122 = f25 * (q020 * p102 + q002 * p120 + R(4) * p011 * p111
                          + R(2) * (p101 * p021 + p110 * p012)) + ux * B * C;
    const R M212 = f25 * (q200 * p012 + q002 * p210 + R(4) * p101 * p111
                          + R(2) * (p110 * p102 + p011 * p201)) + A * uy * C;
    const R M221 = f25 * (q200 * p021 + q020 * p201 + R(4) * p110 * p111
                          + R(2) * (p011 * p210 + p101 * p120)) + A * B * uz;
    const R s122 = Fxr * k022 + R(2) * (Fyr * k112 + Fzr * k121);
    const R s212 = Fyr * k202 + R(2) * (Fxr * k112 + Fzr * k211);
    const R s221 = Fzr * k220 + R(2) * (Fxr * k121 + Fyr * k211);
    const R t122 = kUnit ? M122 + hu * s122 : d122 + om[23] * (M122 - d122) + h[23] * s122;
    const R t212 = kUnit ? M212 + hu * s212 : d212 + om[24] * (M212 - d212) + h[24] * s212;
    const R t221 = kUnit ? M221 + hu * s221 : d221 + om[25] * (M221 - d221) + h[25] * s221;

    // order 6: attractor from post-collision orders 2 and 4, K_222 = A B C
    const R p112 = C * xy + t112, p121 = B * xz + t121, p211 = A * yz + t211;
    const R M222 = third * irho
                 * (A * t022 + B * t202 + C * t220 + B * C * t200 + A * C * t020 + A * B * t002
                    + t200 * t022 + t020 * t202 + t002 * t220
                    + R(4) * (p110 * p112 + p101 * p121 + p011 * p211) - R(3) * A * B * C * drho);
    const R s222 = R(2) * (Fxr * k122 + Fyr * k212 + Fzr * k221);
    const R t222 = kUnit ? M222 + hu * s222 : d222 + om[26] * (M222 - d222) + h[26] * s222;

    DD(0, 0, 0) = t000; DD(1, 0, 0) = t100; DD(0, 1, 0) = t010; DD(0, 0, 1) = t001;
    DD(1, 1, 0) = t110; DD(1, 0, 1) = t101; DD(0, 1, 1) = t011;
    DD(2, 0, 0) = t200; DD(0, 2, 0) = t020; DD(0, 0, 2) = t002;
    DD(1, 2, 0) = t120; DD(1, 0, 2) = t102; DD(2, 1, 0) = t210; DD(0, 1, 2) = t012;
    DD(2, 0, 1) = t201; DD(0, 2, 1) = t021; DD(1, 1, 1) = t111;
    DD(2, 2, 0) = t220; DD(2, 0, 2) = t202; DD(0, 2, 2) = t022;
    DD(2, 1, 1) = t211; DD(1, 2, 1) = t121; DD(1, 1, 2) = t112;
    DD(1, 2, 2) = t122; DD(2, 1, 2) = t212; DD(2, 2, 1) = t221; DD(2, 2, 2) = t222;
#undef DD
}

// The x sweep split at u: its raw part (independent of u) gives, per x-line (z, y), the sum a+b+c,
// the difference c-a and the sum c+a of the line's links.  The node's density and momentum are
// sums of these nine line values, so the step takes them from here (26 additions instead of 77).
template <class R>
__device__ __forceinline__ void xraw_d3q27(const R f[27], R p[3][3][3])
{
    static_for<27>([&](auto A) {
        constexpr int a = decltype(A)::value;
        p[e27(a, 2) + 1][e27(a, 1) + 1][e27(a, 0) + 1] = f[a];
    });
#pragma unroll
    for (int k = 0; k < 3; ++k)
#pragma unroll
        for (int j = 0; j < 3; ++j) {
            const R a = p[k][j][0], b = p[k][j][1], c = p[k][j][2];
            p[k][j][0] = a + b + c;
            p[k][j][1] = c - a;
            p[k][j][2] = c + a;
        }
}

// One y or z sweep over the nine lines of p: axis 1 sweeps j (lines (k, a)), axis 2 sweeps k
// (lines (j, a)); FP32 pairs the lines at a = 0 and a = 2.
template <bool kInverse, int kAxis, class R>
__device__ __forceinline__ void sweep_yz_d3q27(R p[3][3][3], R u)
{
#define LBM_P(l, m, a) (kAxis == 1 ? p[l][m][a] : p[m][l][a])
    if constexpr (std::is_same<R, float>::value) {
#pragma unroll
        for (int l = 0; l < 3; ++l) {
            float2 v0 = make_float2(LBM_P(l, 0, 0), LBM_P(l, 0, 2));
            float2 v1 = make_float2(LBM_P(l, 1, 0), LBM_P(l, 1, 2));
            float2 v2 = make_float2(LBM_P(l, 2, 0), LBM_P(l, 2, 2));
            if constexpr (kInverse) uncentral_line2(v0, v1, v2, u);
            else central_line2(v0, v1, v2, u);
            LBM_P(l, 0, 0) = v0.x; LBM_P(l, 0, 2) = v0.y;
            LBM_P(l, 1, 0) = v1.x; LBM_P(l, 1, 2) = v1.y;
            LBM_P(l, 2, 0) = v2.x; LBM_P(l, 2, 2) = v2.y;
            if constexpr (kInverse) uncentral_line(LBM_P(l, 0, 1), LBM_P(l, 1, 1), LBM_P(l, 2, 1), u);
            else central_line(LBM_P(l, 0, 1), LBM_P(l, 1, 1), LBM_P(l, 2, 1), u);
        }
    } else {
#pragma unroll
        for (int l = 0; l < 3; ++l)
#pragma unroll
            for (int a = 0; a < 3; ++a) {
                if constexpr (kInverse) uncentral_line(LBM_P(l, 0, a), LBM_P(l, 1, a), LBM_P(l, 2, a), u);
                else central_line(LBM_P(l, 0, a), LBM_P(l, 1, a), LBM_P(l, 2, a), u);
            }
    }
#undef LBM_P
}

// Central moments from the raw x-line values: the u part of the x sweep (the same operations as
// central_line), then the y and z sweeps.
template <class R>
__device__ __forceinline__ void central_from_xraw_d3q27(R p[3][3][3], R ux, R uy, R uz)
{
#pragma unroll
    for (int k = 0; k < 3; ++k)
#pragma unroll
        for (int j = 0; j < 3; ++j) {
            const R k0 = p[k][j][0], d = p[k][j][1], s = p[k][j][2];
            const R k1 = d - ux * k0;
            p[k][j][1] = k1;
            p[k][j][2] = s - ux * (d + k1);
        }
    sweep_yz_d3q27<false, 1>(p, uy);
    sweep_yz_d3q27<false, 2>(p, uz);
}

// Inverse transform; the populations come out multiplied by 2^L (L = 0 except for FP16 storage,
// whose scale is folded in here instead of at the store).
template <int L = 0, class R>
__device__ __forceinline__ void from_central_d3q27(R p[3][3][3], R f[27], R ux, R uy, R uz)
{
    sweep_yz_d3q27<true, 2>(p, uz);
    sweep_yz_d3q27<true, 1>(p, uy);
#pragma unroll
    for (int k = 0; k < 3; ++k)
#pragma unroll
        for (int j = 0; j < 3; ++j) uncentral_line_pow2<L>(p[k][j][0], p[k][j][1], p[k][j][2], ux);
    static_for<27>([&](auto A) {
        constexpr int a = decltype(A)::value;
        f[a] = p[e27(a, 2) + 1][e27(a, 1) + 1][e27(a, 0) + 1];
    });
}

// Raw moments of a D3Q15 population vector (App. C Step 1), in the moment order of the collision:
// (000, 100, 010, 001, 110, 101, 011, 200, 020, 002, 120, 012, 201, 111, 220).
template <class R>
struct G15Raw {
    R r000, r100, r010, r001, r110, r101, r011, r200, r020, r002, r120, r012, r201, r111, r220;
};

template <class R>
__device__ __forceinline__ G15Raw<R> raw_g_d3q15(const R g[15])
{
    // Axis pairs ...
    const R sx = g[1] + g[2], dx = g[1] - g[2];
    const R sy = g[3] + g[4], dy = g[3] - g[4];
    const R sz = g[5] + g[6], dz = g[5] - g[6];
    // ... and the corner links 7..14 = (+++), (-++), (+-+), (--+), (++-), (-+-), (+--), (---):
    // butterflies over x, then y, then z give sum, x, y, z, xy, xz, yz, xyz weighted sums.
    const R a0 = g[7] + g[8], a1 = g[7] - g[8];     // y+ z+
    const R b0 = g[9] + g[10], b1 = g[9] - g[10];   // y- z+
    const R c0 = g[11] + g[12], c1 = g[11] - g[12]; // y+ z-
    const R d0 = g[13] + g[14], d1 = g[13] - g[14]; // y- z-
    const R zp_s = a0 + b0, zp_y = a0 - b0, zp_x = a1 + b1, zp_xy = a1 - b1;
    const R zm_s = c0 + d0, zm_y = c0 - d0, zm_x = c1 + d1, zm_xy = c1 - d1;
    const R C1 = zp_s + zm_s, Cz = zp_s - zm_s;
    const R Cy = zp_y + zm_y, Cyz = zp_y - zm_y;
    const R Cx = zp_x + zm_x, Cxz = zp_x - zm_x;
    const R Cxy = zp_xy + zm_xy, Cxyz = zp_xy - zm_xy;
    G15Raw<R> r;
    r.r000 = g[0] + sx + sy + sz + C1;
    r.r100 = dx + Cx;
    r.r010 = dy + Cy;
    r.r001 = dz + Cz;
    r.r110 = Cxy;
    r.r101 = Cxz;
    r.r011 = Cyz;
    r.r200 = sx + C1;
    r.r020 = sy + C1;
    r.r002 = sz + C1;
    r.r120 = Cx;
    r.r012 = Cy;
    r.r201 = Cz;
    r.r111 = Cxyz;
    r.r220 = C1;
    return r;
}

// D3Q15 energy collision, App. C Steps 2-5 with option-A attractors (Eq. g-attractorsD3Q15optionA)
// or option B, in deviation form.  `d` holds the Step-1 raw moments of the deviations
// gamma = g - w T_o, and T = T_o + d.r000.  The rest state w T_o has the raw moments
// T_o (1, 1/3, 1/3, 1/3, 1/9) on (000, 200, 020, 002, 220) and none else: they are added before
// Step 2 and removed again after Step 4, so Step 5 writes the post-collision deviations to gd,
// multiplied by 2^L (exactly; L = 10 folds the FP16 storage scale into Step 5's own weights).
template <int L = 0, class R>
__device__ __forceinline__ void collide_g_d3q15(const G15Raw<R>& d, R T_ref, R T, R ux, R uy, R uz,
                                                const R om[15], int gopt, R gd[15])
{
    constexpr double cs2 = 1.0 / 3.0;
    const R rest2 = R(cs2) * T_ref, rest22 = R(1.0 / 9.0) * T_ref;
    const R r000 = T;
    const R r100 = d.r100, r010 = d.r010, r001 = d.r001;
    const R r110 = d.r110, r101 = d.r101, r011 = d.r011;
    const R r200 = d.r200 + rest2, r020 = d.r020 + rest2, r002 = d.r002 + rest2;
    const R r120 = d.r120, r012 = d.r012, r201 = d.r201, r111 = d.r111;
    const R r220 = d.r220 + rest22;

    // Step 2: central moments.
    const R n000 = r000;
    const R n100 = r100 - ux * r000;
    const R n010 = r010 - uy * r000;
    const R n001 = r001 - uz * r000;
    const R n110 = r110 - ux * r010 - uy * n100;
    const R n101 = r101 - ux * r001 - uz * n100;
    const R n011 = r011 - uy * r001 - uz * n010;
    const R n200 = r200 - ux * (r100 + n100);
    const R n020 = r020 - uy * (r010 + n010);
    const R n002 = r002 - uz * (r001 + n001);
    const R n120 = (r120 - uy * (R(2) * r110 - uy * r100)) - ux * n020;
    const R n012 = (r012 - uz * (R(2) * r011 - uz * r010)) - uy * n002;
    const R n201 = (r201 - ux * (R(2) * r101 - ux * r001)) - uz * n200;
    const R n111 = (r111 - ux * r011) - uy * (r101 - ux * r001) - uz * ((r110 - ux * r010) - uy * n100);
    // the raw moment e_x^2 e_y is r012 on D3Q15 (e_x^2 e_y = e_y e_z^2 on every link)
    const R Y1 = r012 - ux * (R(2) * r110 - ux * r010);
    const R Y2 = r220 - ux * (R(2) * r120 - ux * r020);
    const R n220 = Y2 - uy * (R(2) * Y1 - uy * n200);

    // Step 3: relaxation.
    const R t000 = n000 + om[0] * (T - n000);
    const R t100 = n100 - om[1] * n100;
    const R t010 = n010 - om[2] * n010;
    const R t001 = n001 - om[3] * n001;
    const R t110 = n110 - om[4] * n110;
    const R t101 = n101 - om[5] * n101;
    const R t011 = n011 - om[6] * n011;
    const R t200 = n200 + om[7] * (R(cs2) * T - n200);
    const R t020 = n020 + om[8] * (R(cs2) * T - n020);
    const R t002 = n002 + om[9] * (R(cs2) * T - n002);
    // attractors of orders 3-4 from the post-collision moments: option A or option B
    R M120, M012, M201, M111, M220;
    if (gopt == 0) {
        M120 = R(2.0 / 3.0 * cs2) * t100;
        M012 = R(2.0 / 3.0 * cs2) * t010;
        M201 = R(2.0 / 3.0 * cs2) * t001;
        M111 = R(0);
        M220 = R(0.5 * cs2) * (t200 + t020);
    } else {
        const R iT = R(1) / T;
        const R c23 = R(2.0 / 3.0) * iT;
        M120 = c23 * (t020 * t100 + R(2) * t110 * t010);
        M012 = c23 * (t002 * t010 + R(2) * t011 * t001);
        M201 = c23 * (t200 * t001 + R(2) * t101 * t100);
        M111 = c23 * (t110 * t001 + t011 * t100 + t101 * t010);
        M220 = iT * (t200 * t020 + R(2) * t110 * t110);
    }
    const R t120 = n120 + om[10] * (M120 - n120);
    const R t012 = n012 + om[11] * (M012 - n012);
    const R t201 = n201 + om[12] * (M201 - n201);
    const R t111 = n111 + om[13] * (M111 - n111);
    const R t220 = n220 + om[14] * (M220 - n220);

    // Step 4: raw moments from central moments (the inverse of Step 2 in reverse order).
    const R q000 = t000;
    const R q100 = t100 + ux * q000;
    const R q010 = t010 + uy * q000;
    const R q001 = t001 + uz * q000;
    const R q110 = t110 + ux * t010 + uy * q100;
    const R q101 = t101 + ux * t001 + uz * q100;
    const R q011 = t011 + uy * t001 + uz * q010;
    const R q200 = t200 + ux * (t100 + q100);
    const R q020 = t020 + uy * (t010 + q010);
    const R q002 = t002 + uz * (t001 + q001);
    const R q120 = (t120 + uy * (R(2) * t110 + uy * t100)) + ux * q020;
    const R q012 = (t012 + uz * (R(2) * t011 + uz * t010)) + uy * q002;
    const R q201 = (t201 + ux * (R(2) * t101 + ux * t001)) + uz * q200;
    const R q111 = (t111 + ux * t011) + uy * (t101 + ux * t001) + uz * q110;
    const R Z0 = t200;   // the x-central second moment at y-power 0
    const R Z1 = q012 - ux * (R(2) * q110 - ux * q010);
    const R Z2 = t220 + uy * (R(2) * Z1 - uy * Z0);
    const R q220 = Z2 + ux * (R(2) * q120 - ux * q020);

    // Step 5: populations of the deviations (the rest moments removed first).  Axis pairs and the
    // inverse corner transform.
    const R q000d = q000 - T_ref, q200d = q200 - rest2, q020d = q020 - rest2, q002d = q002 - rest2;
    const R q220d = q220 - rest22;
    const R Sx = q200d - q220d, Dx = q100 - q120;
    const R Sy = q020d - q220d, Dy = q010 - q012;
    const R Sz = q002d - q220d, Dz = q001 - q201;
    constexpr double s = double(1ull << L);
    const R g0 = q000d - q200d - q020d - q002d + R(2) * q220d;
    gd[0] = L == 0 ? g0 : R(s) * g0;
    const R hs = R(0.5 * s);
    gd[1] = hs * (Sx + Dx);
    gd[2] = hs * (Sx - Dx);
    gd[3] = hs * (Sy + Dy);
    gd[4] = hs * (Sy - Dy);
    gd[5] = hs * (Sz + Dz);
    gd[6] = hs * (Sz - Dz);
    const R e = R(0.125 * s);
    // z split
    const R P_s = q220d + q201, M_s = q220d - q201;   // sum part for z+ / z-
    const R P_y = q012 + q011, M_y = q012 - q011;
    const R P_x = q120 + q101, M_x = q120 - q101;
    const R P_xy = q110 + q111, M_xy = q110 - q111;
    // y split (z+)
    const R A0 = P_s + P_y, B0 = P_s - P_y, A1 = P_x + P_xy, B1 = P_x - P_xy;
    // y split (z-)
    const R C0 = M_s + M_y, D0 = M_s - M_y, C1_ = M_x + M_xy, D1_ = M_x - M_xy;
    gd[7] = e * (A0 + A1);
    gd[8] = e * (A0 - A1);
    gd[9] = e * (B0 + B1);
    gd[10] = e * (B0 - B1);
    gd[11] = e * (C0 + C1_);
    gd[12] = e * (C0 - C1_);
    gd[13] = e * (D0 + D1_);
    gd[14] = e * (D0 - D1_);
}

// D3Q15 energy collision for the rates lbm_create sets (option A; every rate 1 except those of the
// first-order moments, which carry alpha).  With those rates Step 3 leaves the post-collision
// central moments as T, the relaxed first-order moments t1 = (1 - omega) eta_1, the second-order
// c_s^2 T (diagonal) and 0 (mixed), the third-order (2/3) c_s^2 t1 and 0 (111), and
// eta~_220 = (c_s^2)^2 T: only T and the three first-order raw moments (r100, r010, r001) of the
// pulled populations enter.  Steps 4-5 are those of collide_g_d3q15 with these values (terms that
// vanish dropped), so the output is the same up to rounding; it is written to gd as deviations
// times 2^L.
template <int L = 0, class R>
__device__ __forceinline__ void collide_g_d3q15_unit(R T_ref, R T, R r100, R r010, R r001, R ux,
                                                     R uy, R uz, const R om[15], R gd[15])
{
    constexpr double cs2 = 1.0 / 3.0;
    const R rest2 = R(cs2) * T_ref, rest22 = R(1.0 / 9.0) * T_ref;
    // Steps 2-3: the first-order central moments, relaxed
    const R n100 = r100 - ux * T;
    const R n010 = r010 - uy * T;
    const R n001 = r001 - uz * T;
    const R t100 = n100 - om[1] * n100;
    const R t010 = n010 - om[2] * n010;
    const R t001 = n001 - om[3] * n001;
    const R t2 = R(cs2) * T;                       // t200 = t020 = t002
    const R c3 = R(2.0 / 3.0 * cs2);               // t120 = c3 t100, t012 = c3 t010, t201 = c3 t001
    const R t220 = R(cs2 * cs2) * T;
    // Step 4: raw moments (t110 = t101 = t011 = t111 = 0)
    const R q000 = T;
    const R q100 = t100 + ux * q000;
    const R q010 = t010 + uy * q000;
    const R q001 = t001 + uz * q000;
    const R q110 = ux * t010 + uy * q100;
    const R q101 = ux * t001 + uz * q100;
    const R q011 = uy * t001 + uz * q010;
    const R q200 = t2 + ux * (t100 + q100);
    const R q020 = t2 + uy * (t010 + q010);
    const R q002 = t2 + uz * (t001 + q001);
    const R q120 = (c3 * t100 + uy * (uy * t100)) + ux * q020;
    const R q012 = (c3 * t010 + uz * (uz * t010)) + uy * q002;
    const R q201 = (c3 * t001 + ux * (ux * t001)) + uz * q200;
    const R q111 = uy * (ux * t001) + uz * q110;
    const R Z1 = q012 - ux * (R(2) * q110 - ux * q010);
    const R Z2 = t220 + uy * (R(2) * Z1 - uy * t2);
    const R q220 = Z2 + ux * (R(2) * q120 - ux * q020);
    // Step 5: populations of the deviations
    const R q000d = q000 - T_ref, q200d = q200 - rest2, q020d = q020 - rest2, q002d = q002 - rest2;
    const R q220d = q220 - rest22;
    const R Sx = q200d - q220d, Dx = q100 - q120;
    const R Sy = q020d - q220d, Dy = q010 - q012;
    const R Sz = q002d - q220d, Dz = q001 - q201;
    constexpr double s = double(1ull << L);
    const R g0 = q000d - q200d - q020d - q002d + R(2) * q220d;
    gd[0] = L == 0 ? g0 : R(s) * g0;
    const R hs = R(0.5 * s);
    gd[1] = hs * (Sx + Dx);
    gd[2] = hs * (Sx - Dx);
    gd[3] = hs * (Sy + Dy);
    gd[4] = hs * (Sy - Dy);
    gd[5] = hs * (Sz + Dz);
    gd[6] = hs * (Sz - Dz);
    const R e = R(0.125 * s);
    const R P_s = q220d + q201, M_s = q220d - q201;
    const R P_y = q012 + q011, M_y = q012 - q011;
    const R P_x = q120 + q101, M_x = q120 - q101;
    const R P_xy = q110 + q111, M_xy = q110 - q111;
    const R A0 = P_s + P_y, B0 = P_s - P_y, A1 = P_x + P_xy, B1 = P_x - P_xy;
    const R C0 = M_s + M_y, D0 = M_s - M_y, C1_ = M_x + M_xy, D1_ = M_x - M_xy;
    gd[7] = e * (A0 + A1);
    gd[8] = e * (A0 - A1);
    gd[9] = e * (B0 + B1);
    gd[10] = e * (B0 - B1);
    gd[11] = e * (C0 + C1_);
    gd[12] = e * (C0 - C1_);
    gd[13] = e * (D0 + D1_);
    gd[14] = e * (D0 - D1_);
}

// Zeroth and first raw moments of the D3Q15 deviations (the part of raw_g_d3q15 that the
// unit-rate energy collision needs).
template <class R>
__device__ __forceinline__ void raw01_g_d3q15(const R g[15], R& r000, R& r100, R& r010, R& r001)
{
    const R a0 = g[7] + g[8], a1 = g[7] - g[8];     // y+ z+
    const R b0 = g[9] + g[10], b1 = g[9] - g[10];   // y- z+
    const R c0 = g[11] + g[12], c1 = g[11] - g[12]; // y+ z-
    const R d0 = g[13] + g[14], d1 = g[13] - g[14]; // y- z-
    const R zp_s = a0 + b0, zm_s = c0 + d0;
    const R C1 = zp_s + zm_s, Cz = zp_s - zm_s;
    const R Cy = (a0 - b0) + (c0 - d0);
    const R Cx = (a1 + b1) + (c1 + d1);
    r000 = g[0] + (g[1] + g[2]) + (g[3] + g[4]) + (g[5] + g[6]) + C1;
    r100 = (g[1] - g[2]) + Cx;
    r010 = (g[3] - g[4]) + Cy;
    r001 = (g[5] - g[6]) + Cz;
}

// Both collisions of one node at the rates lbm_create sets, option A and gravity along
// z (rate_class 3, checked by the host), from the stored numbers in f and g (raw); the 3D
// counterpart of collide_store_d2q9_unit, see there.  Of the flow's moments only those enter that
// relax with a rate of their own (rho, j and order 2) or that the force multiplies (orders 0-1 in z, up
// to 2 in x and y); t_210 and t_120 vanish.  The relaxed moments are held as deviations e from the
// rest state moving at u (1, 1/3, 1/9, 1/27 on the moments even in every direction, times kUnits) and
// halved once per axis of non-zero order, as the inverse sweeps want them.  606 FP64 instructions
// per node against 867 with the two reduced collisions above alone: 128^3 in FP64 2.40 ms against
// 3.36 per step; FP16 storage issues 1,012 instructions against 1,249: 79 us against 95 at 128^3, where
// half of it comes from L2.
// df, dg: the post-collision deviations, in storage units.
template <class S>
__device__ __forceinline__ void collide_d3q27_unit(const typename S::R f[27], const typename S::R g[15],
                                                   const UnitCoeffs<typename S::R>& c, unsigned* status,
                                                   typename S::R df[27], typename S::R dg[15])
{
    using R = typename S::R;
    constexpr double kS = S::kUnits;
    const R third = R(1.0 / 3.0), half = R(0.5), quarter = R(0.25), two = R(2);

    // raw moments: m[k][b][a] = sum e_x^a e_y^b over layer k (e_z = k - 1)
    R m[3][3][3];
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        R q[3][3];   // [j][a]
        static_for<3>([&](auto J) {
            constexpr int j = decltype(J)::value;
            // (the links of a layer's lines; k is unrolled, so the indices fold)
            const int la = k == 0 ? idx27(-1, j - 1, -1) : (k == 1 ? idx27(-1, j - 1, 0) : idx27(-1, j - 1, 1));
            const int lb = k == 0 ? idx27(0, j - 1, -1) : (k == 1 ? idx27(0, j - 1, 0) : idx27(0, j - 1, 1));
            const int lc = k == 0 ? idx27(1, j - 1, -1) : (k == 1 ? idx27(1, j - 1, 0) : idx27(1, j - 1, 1));
            const R a = f[la], b = f[lb], cc = f[lc];
            q[j][1] = cc - a;
            if constexpr (S::kFull) {   // the rest weights come off exactly
                q[j][2] = (a - R(2.0 * w27(la))) + cc;
                q[j][0] = q[j][2] + (b - R(w27(lb)));
            } else {
                q[j][2] = a + cc;
                q[j][0] = q[j][2] + b;
            }
        });
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            m[k][2][a] = q[0][a] + q[2][a];
            m[k][1][a] = q[2][a] - q[0][a];
            m[k][0][a] = m[k][2][a] + q[1][a];
        }
    }
    R z0[3][3], z1[3][3];   // [b][a]: orders 0 and 1 in z
#pragma unroll
    for (int b = 0; b < 3; ++b)
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            z0[b][a] = (m[0][b][a] + m[2][b][a]) + m[1][b][a];
            z1[b][a] = m[2][b][a] - m[0][b][a];
        }
    const R M002 = m[0][0][0] + m[2][0][0];
    const R drho = z0[0][0], jx = z0[0][1], jy = z0[1][0], jz = z1[0][0];

    // energy: T and the first-order moments.  g = dT + T0: stored populations lose their rest values here,
    // once per pair of opposite links ((a - 2 w T0) + b has no rounding near the rest state), and gain
    // them again in the store, so everything between is of the size of the deviations.  Against
    // 128 bits, T in [0, 1] about 0.5, an update's rounding is 6.5e-18 rms on a population and 2.7e-17 on
    // their sum, which the collision conserves; summed and written as stored (the better form in 2D) it
    // is 1.55e-17 and 5.9e-17, and with every link's deviation taken and the moments full, as in
    // collide_g_d3q15_unit, 1.17e-17 and 3.6e-17.
    const R T0 = S::kFull ? c.rest_T : R(kS) * c.T_ref;
    auto pair = [&](int a, int b, R rest) { return S::kFull ? (g[a] - two * rest) + g[b] : g[a] + g[b]; };
    const R w1 = c.rest_g[1], w7 = c.rest_g[2];
    const R dT = (((S::kFull ? g[0] - c.rest_g[0] : g[0])
                   + ((pair(7, 14, w7) + pair(8, 13, w7)) + (pair(9, 12, w7) + pair(10, 11, w7))))
                  + (pair(1, 2, w1) + pair(3, 4, w1))) + pair(5, 6, w1);
    R gx, gy, gz;
    {   // along the diagonals (+++), (-++), (+-+), (++-)
        const R d1 = g[7] - g[14], d2 = g[8] - g[13], d3 = g[9] - g[12], d4 = g[11] - g[10];
        const R a = d1 + d4, b = d3 - d2;
        gx = (g[1] - g[2]) + (a + b);
        gy = (g[3] - g[4]) + (a - b);
        gz = (g[5] - g[6]) + ((d1 - d4) + (d2 + d3));
    }
    const R T = T0 + dT, rho = R(kS) + drho;
    check_node_bits(status, rho, T);
    const R irho = recip(rho);
    const R Fz = c.gbeta * dT, hF = half * Fz;
    const R pz = jz + hF;                                  // rho u_z (u_x, u_y: no force)
    const R ux = jx * irho, uy = jy * irho, uz = pz * irho;
    const R uxh = half * ux, uyh = half * uy, uzh = half * uz;

    R p[3][3][3];   // z links, then orders in y and x (halved per axis of non-zero order)
    {
        // pre-collision central moments
        const R k110 = z0[1][1] - ux * jy;
        const R k101 = z1[0][1] - ux * jz;
        const R k011 = z1[1][0] - uy * jz;
        const R E200 = z0[0][2] - ux * jx, E020 = z0[2][0] - uy * jy, E002 = M002 - uz * (jz - hF);
        const R k200 = R(kS / 3.0) + E200, k020 = R(kS / 3.0) + E020;
        const R a21 = z0[1][2] - ux * (z0[1][1] + k110);                  // (e_x - u_x)^2 e_y
        const R m020 = R(kS / 3.0) + z0[2][0];
        const R a12 = z0[2][1] - ux * m020;                               // (e_x - u_x) e_y^2
        const R a22 = (R(kS / 9.0) + z0[2][2]) - ux * (z0[2][1] + a12);
        const R k120 = a12 - uy * (k110 + k110);
        const R k210 = a21 - uy * k200;
        const R k220 = a22 - uy * (a21 + k210);
        const R b20 = z1[0][2] - ux * (z1[0][1] + k101);                  // times e_z
        const R b11 = z1[1][1] - ux * z1[1][0];
        const R b21 = z1[1][2] - ux * (z1[1][1] + b11);
        const R b12 = z1[2][1] - ux * z1[2][0];
        const R b22 = z1[2][2] - ux * (z1[2][1] + b12);
        const R c02 = z1[2][0] - uy * (z1[1][0] + k011);
        const R c11 = b11 - uy * k101;
        const R c12 = b12 - uy * (b11 + c11);
        const R c21 = b21 - uy * b20;
        const R c22 = b22 - uy * (b21 + c21);
        const R k201 = b20 - uz * k200, k021 = c02 - uz * k020, k111 = c11 - uz * k110;
        const R k211 = c21 - uz * k210, k121 = c12 - uz * k120, k221 = c22 - uz * k220;

        // relaxation; x_abc = t_abc halved per axis of non-zero order
        const R G = Fz * irho, G4 = quarter * G, G8 = half * G4, G16 = half * G8;
        const R i4 = quarter * irho, i8 = half * i4, f5 = R(0.2) * irho, i6 = R(1.0 / 6.0) * irho;
        const R t110 = c.kf[0] * k110, t101 = c.kf[1] * k101, t011 = c.kf[2] * k011;
        const R td1 = c.kf[4] * (E200 - E020), td2 = c.kf[5] * (E200 - E002);
        const R e200 = third * (drho + td1 + td2), e020 = e200 - td1, e002 = e200 - td2;
        const R q200 = R(kS / 3.0) + e200, q020 = R(kS / 3.0) + e020, q002 = R(kS / 3.0) + e002;
        const R d110 = t110 + t110, d101 = t101 + t101, d011 = t011 + t011;
        const R x102 = G4 * k101, x012 = G4 * k011, x201 = G8 * k200, x021 = G8 * k020;
        const R y111 = G4 * k110, x111 = quarter * y111;
        const R l0 = R(kS * 2.0 / 9.0) * drho;
        const R x220 = i4 * (l0 - R(kS / 3.0) * e002 + e200 * e020 + d110 * t110);
        const R x202 = i4 * (l0 - R(kS / 3.0) * e020 + e200 * e002 + d101 * t101) + G4 * k201;
        const R x022 = i4 * (l0 - R(kS / 3.0) * e200 + e020 * e002 + d011 * t011) + G4 * k021;
        const R x211 = i8 * (q200 * t011 + d110 * t101) + G16 * k210;
        const R x121 = i8 * (q020 * t101 + d110 * t011) + G16 * k120;
        const R x112 = i8 * (q002 * t110 + d011 * t101) + G8 * k111;
        const R x122 = f5 * (q020 * x102 + d101 * x021 + d110 * x012 + d011 * y111) + G8 * k121;
        const R x212 = f5 * (q200 * x012 + d011 * x201 + d110 * x102 + d101 * y111) + G8 * k211;
        const R x221 = f5 * (q200 * x021 + q020 * x201 + d110 * y111) + G16 * k220;
        const R x222 = i6 * (q200 * x022 + q020 * x202 + q002 * x220
                             + R(4) * (d110 * x112 + d101 * x121 + d011 * x211)) + G8 * k221;

        // inverse sweep along z
        const R uz2 = uz + uz;
        unline(drho, rho, half * hF, half * e002, uz, uzh, p[0][0][0], p[1][0][0], p[2][0][0]);
        unline0(quarter * t101, x102, uz2, p[0][0][1], p[1][0][1], p[2][0][1]);
        unline0(quarter * t011, x012, uz2, p[0][1][0], p[1][1][0], p[2][1][0]);
        unline(half * e200, half * q200, x201, x202, uz, uzh, p[0][0][2], p[1][0][2], p[2][0][2]);
        unline(half * e020, half * q020, x021, x022, uz, uzh, p[0][2][0], p[1][2][0], p[2][2][0]);
        const R t110q = quarter * t110;
        unline(t110q, t110q, x111, x112, uz, uzh, p[0][1][1], p[1][1][1], p[2][1][1]);
        unline0(x211, x212, uz2, p[0][1][2], p[1][1][2], p[2][1][2]);
        unline0(x121, x122, uz2, p[0][2][1], p[1][2][1], p[2][2][1]);
        unline(x220, R(kS / 36.0) + x220, x221, x222, uz, uzh, p[0][2][2], p[1][2][2], p[2][2][2]);
    }
    // along y, then x; wz and wy are the rest weights of the links already formed
    static_for<3>([&](auto K) {
        constexpr int k = decltype(K)::value;
        constexpr double wz = kS * (k == 1 ? 2.0 / 3.0 : 1.0 / 6.0);
        unline(p[k][0][0], R(wz) + p[k][0][0], p[k][1][0], p[k][2][0], uy, uyh, p[k][0][0], p[k][1][0], p[k][2][0]);
        unline(p[k][0][1], p[k][0][1], p[k][1][1], p[k][2][1], uy, uyh, p[k][0][1], p[k][1][1], p[k][2][1]);
        unline(p[k][0][2], R(wz / 6.0) + p[k][0][2], p[k][1][2], p[k][2][2], uy, uyh, p[k][0][2], p[k][1][2], p[k][2][2]);
        static_for<3>([&](auto J) {
            constexpr int j = decltype(J)::value;
            constexpr double wy = wz * (j == 1 ? 2.0 / 3.0 : 1.0 / 6.0);
            unline(p[k][j][0], R(wy) + p[k][j][0], p[k][j][1], p[k][j][2], ux, uxh, df[idx27(-1, j - 1, k - 1)],
                   df[idx27(0, j - 1, k - 1)], df[idx27(1, j - 1, k - 1)]);
        });
    });

    // energy: the moments of collide_g_d3q15_unit as deviations from w T0
    {
        constexpr double c3 = 2.0 / 9.0;
        const R rest2 = third * T0;
        const R t100 = c.kg[0] * (gx - ux * T), t010 = c.kg[1] * (gy - uy * T), t001 = c.kg[2] * (gz - uz * T);
        const R q100 = t100 + ux * T, q010 = t010 + uy * T, q001 = t001 + uz * T;
        const R xt = ux * t001;
        const R q110 = ux * t010 + uy * q100, q101 = xt + uz * q100, q011 = uy * t001 + uz * q010;
        const R t2 = third * dT;
        const R q200 = t2 + ux * (t100 + q100), q020 = t2 + uy * (t010 + q010), q002 = t2 + uz * (t001 + q001);
        const R q020f = q020 + rest2;
        const R q120 = t100 * (R(c3) + uy * uy) + ux * q020f;
        const R q012 = t010 * (R(c3) + uz * uz) + uy * (q002 + rest2);
        const R q201 = t001 * (R(c3) + ux * ux) + uz * (q200 + rest2);
        const R q111 = uy * xt + uz * q110;
        const R Z1 = q012 - ux * (two * q110 - ux * q010);
        const R Z2 = R(1.0 / 9.0) * dT + uy * (two * Z1 - uy * (third * T));
        const R q220 = Z2 + ux * (two * q120 - ux * q020f);
        dg[0] = ((dT - q200) - q020) - q002 + two * q220;
        const R h220 = half * q220, h120 = half * q120, h012 = half * q012, h201 = half * q201;
        const R Sx = half * q200 - h220, Sy = half * q020 - h220, Sz = half * q002 - h220;
        const R Dx = half * q100 - h120, Dy = half * q010 - h012, Dz = half * q001 - h201;
        dg[1] = Sx + Dx;
        dg[2] = Sx - Dx;
        dg[3] = Sy + Dy;
        dg[4] = Sy - Dy;
        dg[5] = Sz + Dz;
        dg[6] = Sz - Dz;
        const R e = R(0.125);
        const R s0 = quarter * h220, sx = quarter * h120, sy = quarter * h012, sz = quarter * h201;
        const R sxy = e * q110, sxz = e * q101, syz = e * q011, sxyz = e * q111;
        const R P_s = s0 + sz, M_s = s0 - sz, P_y = sy + syz, M_y = sy - syz;
        const R P_x = sx + sxz, M_x = sx - sxz, P_xy = sxy + sxyz, M_xy = sxy - sxyz;
        const R A0 = P_s + P_y, B0 = P_s - P_y, A1 = P_x + P_xy, B1 = P_x - P_xy;
        const R C0 = M_s + M_y, D0 = M_s - M_y, C1 = M_x + M_xy, D1 = M_x - M_xy;
        dg[7] = A0 + A1;
        dg[8] = A0 - A1;
        dg[9] = B0 + B1;
        dg[10] = B0 - B1;
        dg[11] = C0 + C1;
        dg[12] = C0 - C1;
        dg[13] = D0 + D1;
        dg[14] = D0 - D1;
    }

}

template <class S, class Idx>
__device__ __forceinline__ void collide_store_d3q27_unit(const typename S::R f[27], const typename S::R g[15],
                                                         typename S::T* __restrict__ fout,
                                                         typename S::T* __restrict__ gout,
                                                         const Geometry& geo,
                                                         const UnitCoeffs<typename S::R>& c,
                                                         unsigned* status, int i)
{
    using R = typename S::R;
    R df[27], dg[15];
    collide_d3q27_unit<S>(f, g, c, status, df, dg);
    if constexpr (std::is_same<S, StoreF16S>::value) {
        store_node_f16s<27, 15, Idx, true>(fout, gout, (Idx)geo.n, i, df, dg, c.fp16_sr);
    } else {
        static_for<27>([&](auto A) {
            constexpr int a = decltype(A)::value;
            S::store_dev(fout, (Idx)a * geo.n + i, df[a], R(w27(a)));
        });
        static_for<15>([&](auto B) {
            constexpr int b = decltype(B)::value;
            S::store_dev(gout, (Idx)b * geo.n + i, dg[b], c.rest_g[b == 0 ? 0 : (b < 7 ? 1 : 2)]);
        });
    }
}

// The coefficients of collision instance kRates (rate_class).
template <class S, int kRates>
using StepCoeffs3D = typename std::conditional<kRates == 3, UnitCoeffs<typename S::R>, Coeffs3D<typename S::R>>::type;

// Macroscopic fields, both collisions and the store of one node whose pulled deviations are in
// f (flow) and g (energy); i is the node's linear index.  kRates (rate_class, checked by the host):
// 0 general rates; 1 the energy rates of lbm_create (collide_g_d3q15_unit); 2 the flow rates of
// lbm_create as well (relax_f_d3q27<true>).  (3, gravity along z too, is collide_store_d3q27_unit.)
template <class S, class Idx, int kRates = 0>
__device__ __forceinline__ void collide_store_d3q27(typename S::R f[27], typename S::R g[15],
                                                    typename S::T* __restrict__ fout,
                                                    typename S::T* __restrict__ gout,
                                                    const Geometry& geo,
                                                    const Coeffs3D<typename S::R>& c,
                                                    unsigned* status, int i);

template <class S, class Idx, int kRates = 0>
__device__ __forceinline__ void node_step_d3q27(const typename S::T* __restrict__ fin,
                                                const typename S::T* __restrict__ gin,
                                                typename S::T* __restrict__ fout,
                                                typename S::T* __restrict__ gout,
                                                const Geometry& geo, const StepCoeffs3D<S, kRates>& c,
                                                unsigned* status, int x, int y, int z)
{
    using R = typename S::R;
    const int i = x + geo.nx * y + geo.nxy * z;
    R f[27], g[15];
    // Which pull: decided per warp where possible, so that a warp holding an x-wall node of an
    // interior row runs one x-only pull instead of both the interior and the general pull.
    const bool yz_in = y > 0 && y < geo.ny - 1 && z > 0 && z < geo.nz - 1;
    const bool in = yz_in && x > 0 && x < geo.nx - 1;
    const unsigned lanes = __activemask();
    if (__all_sync(lanes, in)) {
        pull_d3q27_d3q15_interior<S, Idx, kRates == 3 ? kPullRaw : kPullDev>(fin, gin, geo, i, c.T_ref, f, g);
    } else if (__all_sync(lanes, yz_in)) {
        const NodeWalls<R> w = node_walls_x<R>(geo, x, y, z);
        pull_d3q27_d3q15<S, Idx, kRates == 3 ? kPullRaw : kPullDev>(fin, gin, geo, w, i, c.T_ref, f, g);
    } else if (in) {
        pull_d3q27_d3q15_interior<S, Idx, kRates == 3 ? kPullRaw : kPullDev>(fin, gin, geo, i, c.T_ref, f, g);
    } else {
        const NodeWalls<R> w = node_walls<R>(geo, x, y, z, 3);
        pull_d3q27_d3q15<S, Idx, kRates == 3 ? kPullRaw : kPullDev>(fin, gin, geo, w, i, c.T_ref, f, g);
    }
    if constexpr (kRates == 3) collide_store_d3q27_unit<S, Idx>(f, g, fout, gout, geo, c, status, i);
    else collide_store_d3q27<S, Idx, kRates>(f, g, fout, gout, geo, c, status, i);
}

template <class S, class Idx, int kRates>
__device__ __forceinline__ void collide_store_d3q27(typename S::R f[27], typename S::R g[15],
                                                    typename S::T* __restrict__ fout,
                                                    typename S::T* __restrict__ gout,
                                                    const Geometry& geo,
                                                    const Coeffs3D<typename S::R>& c,
                                                    unsigned* status, int i)
{
    using R = typename S::R;
    // rho = 1 + sum delta, rho u = sum delta e + F/2, T = T_o + sum gamma (the zeroth raw moment of
    // the energy deviations, which the energy collision starts from)
    constexpr bool kUnitG = kRates >= 1, kUnitF = kRates >= 2;
    G15Raw<R> gr;
    R dT;
    if constexpr (kUnitG) raw01_g_d3q15(g, dT, gr.r100, gr.r010, gr.r001);
    else {
        gr = raw_g_d3q15(g);
        dT = gr.r000;
    }
    // Density and momentum: from the raw x-line values for FP16 and FP64 storage, which are bound by
    // the instruction or FP64 rate (51 fewer additions; FP16S +1.2 %); directly from the links for
    // FP32 storage, where keeping the nine line values live adds spills (-0.6 % measured).
    // p[k][j] is the x-line at e_z = k - 1, e_y = j - 1.
    constexpr bool kLineSums = !std::is_same<S, StoreF32>::value;
    R p[3][3][3];
    R drho, jx, jy, jz;
    if constexpr (kLineSums) {
        xraw_d3q27(f, p);
        drho = p[0][0][0];
        jx = p[0][0][1];
#pragma unroll
        for (int l = 1; l < 9; ++l) {
            drho += p[l / 3][l % 3][0];
            jx += p[l / 3][l % 3][1];
        }
        jy = (p[0][2][0] + p[1][2][0] + p[2][2][0]) - (p[0][0][0] + p[1][0][0] + p[2][0][0]);
        jz = (p[2][0][0] + p[2][1][0] + p[2][2][0]) - (p[0][0][0] + p[0][1][0] + p[0][2][0]);
    } else {
        drho = f[0];
        jx = jy = jz = R(0);
        static_for<26>([&](auto A) {
            constexpr int a = decltype(A)::value + 1;
            drho += f[a];
            if (e27(a, 0) == 1) jx += f[a];
            if (e27(a, 0) == -1) jx -= f[a];
            if (e27(a, 1) == 1) jy += f[a];
            if (e27(a, 1) == -1) jy -= f[a];
            if (e27(a, 2) == 1) jz += f[a];
            if (e27(a, 2) == -1) jz -= f[a];
        });
    }
    const R Fb = c.gbeta * dT;
    const R Fx = c.gaxis == 0 ? Fb : R(0);
    const R Fy = c.gaxis == 1 ? Fb : R(0);
    const R Fz = c.gaxis == 2 ? Fb : R(0);
    const R rho = R(1) + drho;
    const R T = c.T_ref + dT;
    const R irho = R(1) / rho;
    const R ux = (jx + R(0.5) * Fx) * irho;
    const R uy = (jy + R(0.5) * Fy) * irho;
    const R uz = (jz + R(0.5) * Fz) * irho;
    check_node(status, rho, T);

    if constexpr (!kLineSums) xraw_d3q27(f, p);
    central_from_xraw_d3q27(p, ux, uy, uz);
    relax_f_d3q27<kUnitF>(p, drho, irho, ux, uy, uz, Fx, Fy, Fz, c);
    // FP16 storage keeps deviations times 2^10: both collisions return them already scaled
    constexpr bool kF16 = std::is_same<S, StoreF16S>::value;
    constexpr int kL = kF16 ? StoreF16S::kScaleLog2 : 0;
    from_central_d3q27<kL>(p, f, ux, uy, uz);
    // energy collision on the deviations: g receives the post-collision gamma
    if constexpr (kUnitG) collide_g_d3q15_unit<kL>(c.T_ref, T, gr.r100, gr.r010, gr.r001, ux, uy, uz, c.om_g, g);
    else collide_g_d3q15<kL>(gr, c.T_ref, T, ux, uy, uz, c.om_g, c.gopt, g);

    if constexpr (kF16) {
        if (c.fp16_sr) {
            store_node_f16s<27, 15, Idx, true>(fout, gout, (Idx)geo.n, i, f, g, 1);
        } else {
            static_for<27>([&](auto A) {
                constexpr int a = decltype(A)::value;
                StoreF16S::store_scaled(fout, (Idx)a * geo.n + i, f[a]);
            });
            static_for<15>([&](auto B) {
                constexpr int b = decltype(B)::value;
                StoreF16S::store_scaled(gout, (Idx)b * geo.n + i, g[b]);
            });
        }
        return;
    }
    static_for<27>([&](auto A) {
        constexpr int a = decltype(A)::value;
        S::store_dev(fout, (Idx)a * geo.n + i, f[a], R(w27(a)));
    });
    static_for<15>([&](auto B) {
        constexpr int b = decltype(B)::value;
        S::store_dev(gout, (Idx)b * geo.n + i, g[b], R(w15(b)) * c.T_ref);
    });
}

// Registers per thread of the plain step (sweeps on the 256^3 cavity): FP64 takes what its
// collision needs; FP32 with the reduced collisions of the default rates 72, so that 28 warps fit
// on an SM (+1.0 % against 80; 64 spills and is slower); every other form 80 (24 warps), where 72
// measured slower.
template <class S, int kRates>
struct Launch3D {
    static constexpr int kMaxRegs = sizeof(typename S::R) == 8 ? 255
                                    : (std::is_same<S, StoreF32>::value && kRates == 2 ? 72 : 80);
};

// kRows: each thread updates kRows consecutive rows (y) of its column, one after the other, so a
// block lives kRows times longer and the SM spends a smaller share of its slots on block
// turnover.  The grid's y extent is divided by kRows.
template <class S, class Idx, int kRows = 1, int kRates = 0>
__global__ void __maxnreg__(LBM_MAXREG3D)
    step_d3q27_kernel(const typename S::T* __restrict__ fin, const typename S::T* __restrict__ gin,
                      typename S::T* __restrict__ fout, typename S::T* __restrict__ gout,
                      Geometry geo, StepCoeffs3D<S, kRates> c, unsigned* status, bool flip)
{
    const int x = blockIdx.x * blockDim.x + threadIdx.x;
    const int y0 = ((flip ? gridDim.y - 1 - blockIdx.y : blockIdx.y) * blockDim.y + threadIdx.y) * kRows;
    const int z = flip ? gridDim.z - 1 - blockIdx.z : blockIdx.z;
    if (x >= geo.nx) return;
#pragma unroll 1
    for (int r = 0; r < kRows; ++r) {
        const int y = y0 + r;
        if (y >= geo.ny) return;
        node_step_d3q27<S, Idx, kRates>(fin, gin, fout, gout, geo, c, status, x, y, z);
    }
}

// ---------------------------------------------------------------------------------------------
// FP16 storage, reduced collision: two x-adjacent nodes per thread
// ---------------------------------------------------------------------------------------------

#ifndef LBM_MAXREG3D_PAIR
#define LBM_MAXREG3D_PAIR 96
#endif

// Both collisions of one node of a pair, rounded to packed storage.
__device__ __forceinline__ void pair_node(const float f[27], const float g[15], const UnitCoeffs<float>& c,
                                          unsigned* status, int i, unsigned h2[21])
{
    float df[27], dg[15];
    collide_d3q27_unit<StoreF16S>(f, g, c, status, df, dg);
    if (c.fp16_sr) pack_node_f16s<27, 15, true, true>(i, df, dg, h2);
    else pack_node_f16s<27, 15, false, true>(i, df, dg, h2);
}

// 32 consecutive FP16 values are only 64 bytes, so one node per thread makes twice the memory requests
// per byte of FP32, and at 256^3 the step ran at the FP32 step's node rate with DRAM 42 % busy and
// more warps or fewer instructions no help.  Here a thread updates nodes x0, x0 + 1 (x0 even): links
// without an x component load, and all links store, 32 bits at once; links along x are two 16-bit
// loads, the second a hit in L1.  The second node waits as packed halves (hold) while the first
// is computed, so registers stay near one node's (96, no spills; 80 and 112 measured slower).
// 256^3: 801 -> 680 us per step (52 % -> 61 % of the measured copy bandwidth); issue slots are then 59 %
// busy, and the first stalls are memory latency and the fetch of the two nodes' unrolled code (1.8 and 1.7
// warps per issue, ncu at 192^3).  Where L2 serves part of the loads the one-node kernel is faster (128^3 79
// against 96 us, 160^3 169 against 207), so boxes take this one from 6 million nodes on (192^3: 305
// against 328), if rows fill its warps (pairs_fill_rows).  Rows and planes start on 4 bytes.  The results are bitwise those of the
// one-node kernel.
template <class Idx>
__global__ void __maxnreg__(LBM_MAXREG3D_PAIR)
    step_d3q27_pair_f16s_kernel(const __half* __restrict__ fin, const __half* __restrict__ gin,
                                __half* __restrict__ fout, __half* __restrict__ gout, Geometry geo,
                                UnitCoeffs<float> c, unsigned* status, bool flip)
{
    using S = StoreF16S;
    const int x = 2 * (blockIdx.x * blockDim.x + threadIdx.x);
    // the two slices of wall rows, whose blocks take longest, first
    const int nz = geo.nz, bz = blockIdx.z;
    const int z = bz == 0 ? (flip ? nz - 1 : 0) : (bz == 1 ? (flip ? 0 : nz - 1) : (flip ? nz - bz : bz - 1));
    const int y = flip ? geo.ny - 1 - blockIdx.y : blockIdx.y;
    if (x >= geo.nx) return;
    const int i = x + geo.nx * y + geo.nxy * z;
    const Idx n = (Idx)geo.n;
    const bool yz_in = y > 0 && y < geo.ny - 1 && z > 0 && z < geo.nz - 1;   // uniform in the block
    unsigned out0[21];
    float f[27], g[15];
    if (yz_in) {
        unsigned hold[21];
        {
            // word a: the pair's values on link a (first node low)
            unsigned w[42];
            // an x link that would leave the row reads its partner's place instead (fix_x_edge_d3q27
            // replaces it): the row behind the last one may end the buffer
            const int lo = x > 0 ? i - 1 : i, hi = x + 2 < geo.nx ? i + 2 : i + 1;
            static_for<42>([&](auto A) {
                constexpr int a = decltype(A)::value;
                constexpr int l = a < 27 ? a : (a - 27 < 7 ? a - 27 : a - 27 + 12);   // D3Q27 link
                constexpr int ex = e27(l, 0);
                const __half* p = a < 27 ? fin + (Idx)a * n : gin + (Idx)(a < 27 ? 0 : a - 27) * n;
                const int row = e27(l, 1) * geo.nx + e27(l, 2) * geo.nxy;
                if constexpr (ex == 0) {
                    w[a] = ld_ro_pair(p + (i - row));
                } else {
                    const int s0 = (ex == 1 ? lo : i + 1) - row, s1 = (ex == 1 ? i : hi) - row;
                    w[a] = (unsigned)__half_as_ushort(ld_ro(p + s0)) | (unsigned)__half_as_ushort(ld_ro(p + s1)) << 16;
                }
            });
            static_for<21>([&](auto K) {
                constexpr int k = decltype(K)::value;
                hold[k] = __byte_perm(w[2 * k], w[2 * k + 1], 0x7632);
            });
            static_for<27>([&](auto A) { f[decltype(A)::value] = S::raw(low_half(w[decltype(A)::value])); });
            static_for<15>([&](auto B) { g[decltype(B)::value] = S::raw(low_half(w[27 + decltype(B)::value])); });
        }
        if (x == 0) fix_x_edge_d3q27<S, Idx, kPullRaw>(fin, gin, geo, x, y, z, i, c.T_ref, f, g);
        pair_node(f, g, c, status, i, out0);
        static_for<42>([&](auto A) {
            constexpr int a = decltype(A)::value;
            const __half h = (a & 1) ? high_half(hold[a / 2]) : low_half(hold[a / 2]);
            if constexpr (a < 27) f[a] = S::raw(h);
            else g[a - 27] = S::raw(h);
        });
        if (x + 2 == geo.nx) fix_x_edge_d3q27<S, Idx, kPullRaw>(fin, gin, geo, x + 1, y, z, i + 1, c.T_ref, f, g);
    } else {
        pull_d3q27_d3q15<S, Idx, kPullRaw>(fin, gin, geo, node_walls<float>(geo, x, y, z, 3), i, c.T_ref, f, g);
        pair_node(f, g, c, status, i, out0);
        pull_d3q27_d3q15<S, Idx, kPullRaw>(fin, gin, geo, node_walls<float>(geo, x + 1, y, z, 3), i + 1, c.T_ref, f, g);
    }
    unsigned out1[21];
    pair_node(f, g, c, status, i + 1, out1);
    static_for<42>([&](auto A) {
        constexpr int a = decltype(A)::value;
        const unsigned v = __byte_perm(out0[a / 2], out1[a / 2], (a & 1) ? 0x7632 : 0x5410);
        __half* p = a < 27 ? fout + (Idx)a * n : gout + (Idx)(a < 27 ? 0 : a - 27) * n;
        *reinterpret_cast<unsigned*>(p + i) = v;
    });
}

}  // namespace lbm
